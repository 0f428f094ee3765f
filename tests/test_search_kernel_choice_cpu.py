"""Which search kernel a call runs: the dispatch's rules, on the host alone."""
import numpy as np
import pytest

from paper_2510_18136_gb300 import build, synth

BARRIER, FREE, LONG, SHORT, MID, WIDE, TEAM, SERVE = range(1, 9)


@pytest.fixture(scope="module")
def native():
    build.build()
    from paper_2510_18136_gb300 import native as nat
    return nat


def kernel(native, n_t, dtype="f32", n_items=90601, n_sub=16, n_dm=64, out="candidates", noise="known", offset=0,
           new_blk=0, tile=0, tuned=False, dm_hi=2000.0):
    w = [1 << i for i in range(11) if (1 << i) <= n_t]
    cfg = synth.SearchConfig(ny=301, nx=301, n_sub=n_sub, n_t=n_t, freq_mhz=synth.band_centres(n_sub),
                             dm=np.linspace(0.0, dm_hi, n_dm), widths=np.array(w, np.int32), threshold=6.0)
    code = {"f32": native.F32, "bf16": native.BF16, "f16": native.F16}[dtype]
    with native.Plan(cfg, dtype=dtype, noise=noise, out=out) as plan:
        return native.lib.nsfrb_dbg_search_kernel(plan.handle, code, n_items, offset, new_blk, tile, int(tuned))


def test_kernels_by_window_length(native):
    for dtype in ("f32", "bf16", "f16"):
        got = [kernel(native, n, dtype) for n in (8, 25, 64, 65, 240, 607, 608, 1200, 1248, 2048)]
        assert got == [SHORT] * 3 + [MID] * 3 + [TEAM] * 2 + [WIDE] * 2
    assert kernel(native, 3000, "f32") == LONG and kernel(native, 3000, "bf16") == WIDE
    assert kernel(native, 1200, out="full") == FREE and kernel(native, 2048, out="full") == LONG
    assert kernel(native, 1199, noise="mad") == BARRIER and kernel(native, 1200, noise="mad") == TEAM
    assert kernel(native, 1200, offset=4) == BARRIER and kernel(native, 25, offset=4) == SHORT


def test_a_tile_kept_by_autotune_leaves_serving_blocks_their_kernel(native):
    for dtype in ("f32", "bf16"):
        assert kernel(native, 1200, dtype, new_blk=25) == SERVE
        assert kernel(native, 1200, dtype, new_blk=25, tile=21, tuned=True) == SERVE
        assert kernel(native, 1200, dtype, new_blk=25, tile=21) == FREE      # the caller's choice
        assert kernel(native, 1200, dtype, new_blk=40, tile=21, tuned=True) == FREE
        assert kernel(native, 1200, dtype, tile=21, tuned=True) == FREE
