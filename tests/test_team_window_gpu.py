"""The team search kernel (608 to 1215 samples, candidate records) vs the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2510_18136_gb300 import synth
from tests import parity

pytestmark = pytest.mark.gpu

STORE = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


@pytest.fixture(scope="module")
def native():
    from paper_2510_18136_gb300 import build
    build.build()
    from paper_2510_18136_gb300 import native as nat
    assert torch.cuda.is_available()
    return nat


# windows at the edges of the compiled chunks (703, 831, 1087, 1215 samples) and of the kernel's range, odd
# lengths, pixels for several hand-overs per team, subband counts that leave other shapes, fewer DM
# rows than warps, rows with few samples or none, widths of every class
@pytest.mark.parametrize("n_t,n_pix,n_sub,n_dm,dm_hi,dtype", [
    (608, 1300, 16, 16, 2000.0, "f32"), (703, 5, 16, 40, 3000.0, "bf16"), (704, 3, 16, 2, 2000.0, "f32"),
    (831, 9, 16, 23, 90000.0, "f16"), (832, 700, 16, 12, 2000.0, "bf16"), (1001, 4, 16, 30, 4000.0, "f32"),
    (1087, 3, 16, 64, 2000.0, "f32"), (1088, 2, 16, 1, 0.0, "f16"), (1200, 1400, 16, 64, 2000.0, "bf16"),
    (1200, 650, 16, 64, 2000.0, "f32"), (1215, 3, 16, 200, 4000.0, "f32"), (1215, 4, 16, 12, 2000.0, "bf16"),
    (900, 3, 8, 9, 2000.0, "f32"), (1000, 3, 24, 9, 2000.0, "f32"), (1000, 3, 20, 9, 2000.0, "f32"),
    (1203, 3, 4, 9, 2000.0, "f32"), (1216, 3, 16, 9, 2000.0, "f32"),
])
def test_team_window_records(native, n_t, n_pix, n_sub, n_dm, dm_hi, dtype):
    rng = np.random.default_rng(n_t + n_dm)
    every = [1, 2, 3, 4, 8, 16, 32, 48, 64, 128, 200, 256, 512, 600, 1024, n_t]
    cfg = synth.SearchConfig(ny=1, nx=n_pix, n_sub=n_sub, n_t=n_t, freq_mhz=synth.band_centres(n_sub),
                             dm=np.sort(rng.uniform(0, dm_hi, n_dm)),
                             widths=np.array(sorted({w for w in every if w <= n_t}), np.int32), threshold=4.5)
    cube = synth.plain_noise(cfg, n_t)
    sh = oracle.delay_table(cfg.freq_mhz, cfg.dm)
    for p in range(0, n_pix, 7):
        d = int(rng.integers(n_dm))
        w = max(1, int(np.exp(rng.uniform(0, np.log(n_t)))))
        synth.add_pulse(cube, cfg, 0, p, int(rng.integers(n_t)), w, 10.0 / np.sqrt(16.0 * w), sh[d])
    cube = cube.to(STORE[dtype])
    sig = rng.uniform(3.0, 6.0, n_pix).astype(np.float32)
    pix = np.arange(n_pix) if n_pix < 10 else np.r_[0:12, n_pix // 2:n_pix // 2 + 6, n_pix - 12:n_pix]
    res, best, _ = oracle.search_cube(cube.float().numpy()[pix], sh, cfg.widths, sigma=sig[pix])
    dev, sg = cube.cuda(), torch.as_tensor(sig).cuda()
    with native.Plan(cfg, dtype=dtype) as plan:
        plan.search(dev, sg)
        snr, idx = plan.best()
        cand = plan.candidates()
        plan.search(dev, sg)          # the hand-overs race in another order: the same records
        snr2, idx2 = plan.best()
    assert (snr == snr2).all() and (idx == idx2).all()
    parity.compare_best(snr[pix], idx[pix], best)
    parity.compare_candidates(cand, best, cfg.threshold, pix, cfg.nx)


def test_team_window_ties_nan_and_rescore(native):
    """Exact ties on a zero cube; a NaN sample; re-scored pixels equal an FP32 search bit for bit."""
    cfg = synth.SearchConfig(ny=4, nx=9, n_t=1200, dm=np.linspace(0.0, 2000.0, 24),
                             widths=np.array([1, 2, 3, 8, 64, 1024], np.int32), threshold=4.0)
    with native.Plan(cfg) as plan:
        plan.search(torch.zeros((36, 16, 1200), device="cuda"))
        z, iz = plan.best()
    assert (z == 0.0).all() and (iz == 0).all()
    cube = synth.plain_noise(cfg, 6)
    bad = cube.clone()
    bad[5, 3, 700] = float("nan")
    with native.Plan(cfg) as plan:
        plan.search(cube.cuda())
        s32, i32 = plan.best()
        plan.search(bad.cuda())
        sn, jn = plan.best()
    keep = np.arange(36) != 5
    assert (sn[keep] == s32[keep]).all() and (jn[keep] == i32[keep]).all() and np.isfinite(sn[5])
    with native.Plan(cfg, dtype="bf16", rescore_eps=50.0) as plan:     # every pixel is re-scored
        plan.search(cube.to(torch.bfloat16).cuda(), None, cube.cuda())
        sr, ir = plan.best()
    assert (sr == s32).all() and (ir == i32).all()
