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


@pytest.mark.parametrize("n_t,dtype,n_items,n_dm,want", [
    # few pixels: 16-bit rows and FP32 rows off 16 bytes stay with the barrier kernel
    (25, "bf16", 64, 64, BARRIER), (25, "bf16", 1672, 16, BARRIER), (25, "bf16", 1673, 16, SHORT),
    (25, "f32", 456, 16, BARRIER), (25, "f32", 457, 16, SHORT), (240, "bf16", 456, 64, BARRIER),
    (240, "bf16", 457, 64, MID), (640, "bf16", 152, 64, BARRIER), (640, "bf16", 153, 64, TEAM),
    # FP32 rows of whole 16 bytes: by pixels and rows
    (64, "f32", 90601, 1, FREE), (64, "f32", 90601, 64, SHORT), (32, "f32", 90601, 1, SHORT),
    (32, "f32", 456, 1, FREE), (240, "f32", 90601, 1, FREE), (240, "f32", 90601, 64, MID), (160, "f32", 64, 64, MID),
    (500, "f32", 90601, 12, FREE), (1200, "f32", 1, 1, TEAM), (1200, "bf16", 1, 1, TEAM), (1248, "f32", 1, 1, WIDE),
])
def test_few_pixels_and_few_rows(native, n_t, dtype, n_items, n_dm, want):
    """The general kernels keep the calls they are faster at; a test's switch passes the rule by."""
    hi = 0.0 if n_dm == 1 else 2000.0 if n_dm != 12 else 1500.0
    assert kernel(native, n_t, dtype, n_items=n_items, n_dm=n_dm, dm_hi=hi) == want
    assert kernel(native, n_t, dtype, n_items=n_items, n_dm=n_dm, dm_hi=hi, tile=-1) in (SHORT, MID, TEAM, WIDE)


def test_a_wide_field_of_many_subbands(native):
    """FP32 pixels too large for eight resident warps of the mid kernel, where the barrier-free kernel holds more."""
    assert kernel(native, 520, n_sub=24, n_items=9000) == FREE
    assert kernel(native, 600, n_sub=32, n_items=9000) == MID


def test_a_tile_kept_by_autotune_leaves_serving_blocks_their_kernel(native):
    for dtype in ("f32", "bf16"):
        assert kernel(native, 1200, dtype, new_blk=25) == SERVE
        assert kernel(native, 1200, dtype, new_blk=25, tile=21, tuned=True) == SERVE
        assert kernel(native, 1200, dtype, new_blk=25, tile=21) == FREE      # the caller's choice
        assert kernel(native, 1200, dtype, new_blk=40, tile=21, tuned=True) == FREE
        assert kernel(native, 1200, dtype, tile=21, tuned=True) == FREE


def test_bench_names_the_default_kernel(native):
    import os
    import sys

    sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    import bench

    def name(n_t, dtype, noise="known", n_sub=16, out="candidates"):
        cfg = synth.SearchConfig(ny=301, nx=301, n_t=n_t, n_sub=n_sub, freq_mhz=synth.band_centres(n_sub),
                                 widths=np.array([1, 8], np.int32), threshold=6.0)
        with native.Plan(cfg, dtype=dtype, noise=noise, out=out) as plan:
            return bench.search_kernel_name(n_t, dtype, noise, 0, out, bench.default_kernel(native, plan, dtype, noise))

    assert name(1200, "f32") == "search_kernel_team<38, 0, T, W>"
    assert name(1200, "bf16", "mad") == "mad_normalise_kernel + search_kernel_team<38, 0, T, W> (FP32 slabs)"
    assert name(240, "bf16") == "search_kernel_mid<34, 8, 1>" and name(25, "f32") == "search_kernel_short<26>"
    assert name(2048, "f32") == "search_kernel_wide<34, 2, 0>" and name(4096, "f32") == "search_kernel_long<0, 0>"
    assert name(1231, "f32").startswith("search_kernel_pipe<39") or name(1231, "f32").startswith("search_kernel<39")
    assert name(1200, "f32", out="full").startswith("search_kernel_pipe<38, 0")
