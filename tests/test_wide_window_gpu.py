"""The wide-window search kernel (several warps to a DM row, windows past 1247 samples) vs the FP64 oracle."""
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


# windows at the edges of the compiled tiles (1407, 1663, 2175, 2431, 3263, 4351 samples) and of what fits
# (FP32 past 2530 samples stays with the long-window kernel), odd lengths, more pixels than SMs
# (a CTA's second pixel), rows with few samples or none, widths of every class and across segments
@pytest.mark.parametrize("n_t,n_pix,n_sub,n_dm,dm_hi,dtype", [
    (1248, 170, 16, 16, 2000.0, "f32"), (1407, 3, 16, 40, 3000.0, "bf16"), (1408, 5, 16, 5, 2000.0, "f32"),
    (1663, 3, 16, 23, 90000.0, "f32"), (1664, 310, 16, 12, 2000.0, "f16"), (2048, 160, 16, 64, 2000.0, "f32"),
    (2175, 2, 16, 3, 2000.0, "f32"), (2176, 3, 8, 30, 9000.0, "bf16"), (2431, 4, 16, 12, 2000.0, "f32"),
    (2432, 4, 16, 12, 2000.0, "f32"), (2600, 3, 16, 9, 2000.0, "f32"), (3263, 3, 16, 12, 2000.0, "bf16"),
    (3264, 4, 16, 1, 0.0, "f16"), (4096, 157, 16, 12, 4000.0, "bf16"), (4095, 2, 16, 6, 2000.0, "f16"),
    (2000, 3, 4, 8, 2000.0, "f32"), (1501, 3, 3, 8, 2000.0, "f32"),
])
def test_wide_window_records(native, n_t, n_pix, n_sub, n_dm, dm_hi, dtype):
    rng = np.random.default_rng(n_t + n_dm)
    every = [1, 2, 3, 4, 8, 16, 32, 64, 100, 128, 256, 512, 1024, 1200, 2048, n_t]
    cfg = synth.SearchConfig(ny=1, nx=n_pix, n_sub=n_sub, n_t=n_t, freq_mhz=synth.band_centres(n_sub),
                             dm=np.sort(rng.uniform(0, dm_hi, n_dm)),
                             widths=np.array(sorted({w for w in every if w <= n_t}), np.int32), threshold=4.5)
    cube = synth.plain_noise(cfg, n_t)
    sh = oracle.delay_table(cfg.freq_mhz, cfg.dm)
    for p in range(0, n_pix, 2):
        d = int(rng.integers(n_dm))
        w = max(1, int(np.exp(rng.uniform(0, np.log(n_t)))))
        synth.add_pulse(cube, cfg, 0, p, int(rng.integers(n_t)), w, 12.0 / np.sqrt(16.0 * w), sh[d])
    cube = cube.to(STORE[dtype])
    sig = rng.uniform(3.0, 6.0, n_pix).astype(np.float32)
    pix = np.arange(n_pix) if n_pix < 10 else np.r_[0:3, n_pix - 3:n_pix]
    res, best, _ = oracle.search_cube(cube.float().numpy()[pix], sh, cfg.widths, sigma=sig[pix])
    with native.Plan(cfg, dtype=dtype) as plan:
        plan.search(cube.cuda(), torch.as_tensor(sig).cuda())
        snr, idx = plan.best()
        cand = plan.candidates()
    parity.compare_best(snr[pix], idx[pix], best)
    parity.compare_candidates(cand, best, cfg.threshold, pix, cfg.nx)


def test_wide_window_ties_and_flagged_pixels(native):
    """Exact ties on a zero cube (the smallest DM, width and sample win); MAD slabs with a constant row."""
    cfg = synth.SearchConfig(ny=2, nx=3, n_t=1600, dm=np.linspace(0.0, 2000.0, 12),
                             widths=np.array([1, 2, 3, 8, 64, 1024], np.int32), threshold=4.0)
    with native.Plan(cfg) as plan:
        plan.search(torch.zeros((6, 16, 1600), device="cuda"))
        z, iz = plan.best()
    assert (z == 0.0).all() and (iz == 0).all()
    cube = synth.plain_noise(cfg, 6)
    cube[4, 3] = 1.5
    with native.Plan(cfg, noise="mad") as plan:
        plan.search(cube.cuda())
        snr, idx = plan.best()
    keep = np.arange(6) != 4
    sh = oracle.delay_table(cfg.freq_mhz, cfg.dm)
    _, best, _ = oracle.search_cube(cube.numpy()[keep], sh, cfg.widths, mad=True)
    parity.compare_best(snr[keep], idx[keep], best)
    assert snr[4] == -np.inf and (idx[4] == -1).all()
