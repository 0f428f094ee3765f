"""The short-window search kernel (a lane per pixel, windows up to 64 samples) vs the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2510_18136_gb300 import synth
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    from paper_2510_18136_gb300 import build
    build.build()
    from paper_2510_18136_gb300 import native as nat
    assert torch.cuda.is_available()
    return nat


# window lengths at the edges of the compiled row lengths (16, 26, 32, 48, 64), pixel counts around a
# CTA's 32, DM grids with rows that leave few samples or none, every kind of width
@pytest.mark.parametrize("n_t,ny,nx,n_sub,n_dm,dm_hi,dtype", [
    (1, 3, 5, 16, 4, 500.0, "f32"), (2, 1, 1, 1, 3, 900.0, "f32"), (15, 4, 8, 16, 9, 6000.0, "f32"),
    (16, 5, 13, 7, 16, 2000.0, "bf16"), (17, 3, 11, 16, 33, 4000.0, "f32"), (25, 9, 11, 16, 16, 2000.0, "f32"),
    (25, 7, 5, 16, 40, 9000.0, "f16"), (26, 2, 16, 32, 16, 3000.0, "f32"), (27, 1, 33, 16, 2, 2000.0, "bf16"),
    (32, 6, 6, 16, 64, 12000.0, "f32"), (33, 5, 7, 16, 12, 2000.0, "f32"), (48, 4, 9, 16, 64, 4000.0, "f16"),
    (49, 3, 7, 9, 16, 2000.0, "f32"), (64, 5, 13, 16, 16, 4000.0, "f32"), (64, 2, 31, 27, 100, 30000.0, "bf16"),
])
def test_short_window_records(native, n_t, ny, nx, n_sub, n_dm, dm_hi, dtype):
    rng = np.random.default_rng(n_t + 100 * n_dm)
    every = [1, 2, 3, 4, 5, 7, 8, 11, 16, 21, 24, 32, 40, 47, 64, n_t]
    widths = sorted({w for w in every if w <= n_t})[:16]
    cfg = synth.SearchConfig(ny=ny, nx=nx, n_sub=n_sub, n_t=n_t, freq_mhz=synth.band_centres(n_sub),
                             dm=np.sort(rng.uniform(0, dm_hi, n_dm)), widths=np.array(widths, np.int32), threshold=4.0)
    cube = synth.plain_noise(cfg, n_t)
    sh = oracle.delay_table(cfg.freq_mhz, cfg.dm)
    for p in range(0, cfg.n_pix, 3):
        d = int(rng.integers(n_dm))
        synth.add_pulse(cube, cfg, p // nx, p % nx, int(rng.integers(n_t)), int(rng.integers(1, n_t + 1)), 2.0, sh[d])
    cube = cube.to({"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}[dtype])
    sig = rng.uniform(3.0, 6.0, cfg.n_pix).astype(np.float32)
    res, best, _ = oracle.search_cube(cube.float().numpy(), sh, cfg.widths, sigma=sig)
    with native.Plan(cfg, dtype=dtype) as plan:
        plan.search(cube.cuda(), torch.as_tensor(sig).cuda())
        snr, idx = plan.best()
        cand = plan.candidates()
        assert plan.get_tile(plan.dtype) == 0
    parity.compare_best(snr, idx, best)
    parity.compare_candidates(cand, best, cfg.threshold, np.arange(cfg.n_pix), cfg.nx)


def test_short_window_infinite_and_nan_samples(native):
    """Non-finite samples drop out of the trials that read them and of no others."""
    cfg = synth.SearchConfig(ny=1, nx=40, n_t=25, dm=np.array([0.0, 0.0]), widths=np.array([1, 4, 16], np.int32))
    cube = synth.plain_noise(cfg, 3)
    clean = cube.clone()
    cube[7, 5, 20] = float("nan")
    cube[9, 2, 24] = float("-inf")
    with native.Plan(cfg) as plan:
        plan.search(cube.cuda())
        snr, idx = plan.best()
    _, best, _ = oracle.search_cube(clean.numpy(), oracle.delay_table(cfg.freq_mhz, cfg.dm), cfg.widths)
    ok = np.ones(cfg.n_pix, bool)
    ok[[7, 9]] = False
    assert np.abs(snr[ok] - best["snr"][ok]).max() <= 1e-5 * np.abs(best["snr"][ok]).max()
    assert (idx[ok][:, 0] == 0).all()
    for p, end in ((7, 20), (9, 24)):      # prefix sums lose everything from the sample on
        _, b, _ = oracle.search_cube(clean[p:p + 1, :, :end].contiguous().numpy(),
                                     oracle.delay_table(cfg.freq_mhz, cfg.dm), cfg.widths)
        if not (idx[p, 1] == 0 and idx[p, 2] > end):
            assert abs(snr[p] - b["snr"][0]) <= 1e-5 * abs(b["snr"][0])


def test_short_window_autotune_keeps_results(native):
    """autotune on a window that both kernels take: whatever it keeps gives the same candidates."""
    cfg = synth.SearchConfig(ny=9, nx=21, n_t=32, dm=np.linspace(0.0, 2000.0, 16),
                             widths=np.array([1, 2, 4, 8, 16], np.int32), threshold=3.5)
    cube = synth.plain_noise(cfg, 8).cuda()
    with native.Plan(cfg) as plan:
        plan.search(cube)
        before = plan.candidates()
        chosen, ms = plan.autotune(cube, reps=1)
        assert chosen == 0 or chosen in ms
        assert plan.get_tile(native.F32) == chosen and len(ms) >= 2
        after = plan.candidates()
    for k in ("row", "col", "dm_idx", "w_idx", "t_idx"):
        assert (before[k] == after[k]).all()
    assert np.abs(before["snr"] - after["snr"]).max() <= 1e-5 * before["snr"].max()


def test_autotune_times_the_default_of_a_plan_with_a_tile(native):
    """A plan that holds a tile: autotune still times tile 0 (a lane per pixel, twice as fast here) and keeps it."""
    cfg = synth.SearchConfig(ny=64, nx=64, n_t=24, dm=np.linspace(0.0, 2000.0, 16),
                             widths=np.array([1, 2, 4, 8, 16], np.int32), threshold=9.0)
    cube = synth.plain_noise(cfg, 1).cuda()
    with native.Plan(cfg) as plan:
        plan.set_tile(native.F32, 41)
        tile, ms = plan.autotune(cube, reps=5)
        assert tile == 0 and plan.get_tile(native.F32) == 0
        assert 41 in ms
        # a storage type that was not searched keeps its tile
        plan.set_tile(native.BF16, 22)
        plan.autotune(cube, reps=1)
        assert plan.get_tile(native.BF16) == 22
