"""The mid-window search kernel (several pixels to a warp, 65 to 607 samples) vs the FP64 oracle."""
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


# window lengths at the edges of the compiled tiles (87, 103, 135, 175, 207, 271, 351, 415, 543, 607 samples) and
# of the kernel's range, pixel counts that leave a CTA's last set short, subband counts whose pixels are
# not whole 16-byte units, odd lengths, DM rows with few samples or none, every kind of width
@pytest.mark.parametrize("n_t,ny,nx,n_sub,n_dm,dm_hi,dtype", [
    (65, 3, 7, 16, 16, 2000.0, "f32"), (87, 2, 9, 16, 30, 9000.0, "bf16"), (88, 1, 1, 5, 7, 2000.0, "f32"),
    (103, 5, 5, 7, 20, 4000.0, "f32"), (104, 3, 3, 16, 16, 2000.0, "f16"), (135, 4, 5, 16, 64, 40000.0, "f32"),
    (136, 3, 3, 16, 16, 2000.0, "bf16"), (175, 2, 7, 13, 12, 3000.0, "f16"), (176, 5, 1, 16, 24, 2000.0, "f32"),
    (207, 3, 3, 3, 16, 2000.0, "f32"), (240, 3, 7, 16, 64, 10000.0, "f32"), (271, 2, 3, 32, 16, 2000.0, "f32"),
    (272, 1, 3, 16, 16, 2000.0, "bf16"), (351, 1, 5, 16, 2, 2000.0, "f32"), (415, 3, 1, 15, 16, 2000.0, "bf16"),
    (543, 1, 3, 16, 33, 5000.0, "f32"), (544, 3, 3, 16, 16, 2000.0, "f16"), (607, 1, 5, 16, 40, 2500.0, "f32"),
    (608, 1, 3, 16, 8, 2500.0, "f32"), (400, 3, 2, 16, 1, 0.0, "f32"),
])
def test_mid_window_records(native, n_t, ny, nx, n_sub, n_dm, dm_hi, dtype):
    rng = np.random.default_rng(n_t + 100 * n_dm)
    every = [1, 2, 3, 4, 8, 11, 16, 24, 32, 50, 64, 128, 200, 256, 512, n_t]
    cfg = synth.SearchConfig(ny=ny, nx=nx, n_sub=n_sub, n_t=n_t, freq_mhz=synth.band_centres(n_sub),
                             dm=np.sort(rng.uniform(0, dm_hi, n_dm)),
                             widths=np.array(sorted({w for w in every if w <= n_t}), np.int32), threshold=4.0)
    cube = synth.plain_noise(cfg, n_t)
    sh = oracle.delay_table(cfg.freq_mhz, cfg.dm)
    for p in range(0, cfg.n_pix, 2):
        d = int(rng.integers(n_dm))
        synth.add_pulse(cube, cfg, p // nx, p % nx, int(rng.integers(n_t)), int(rng.integers(1, n_t + 1)), 1.0, sh[d])
    cube = cube.to(STORE[dtype])
    sig = rng.uniform(3.0, 6.0, cfg.n_pix).astype(np.float32)
    res, best, _ = oracle.search_cube(cube.float().numpy(), sh, cfg.widths, sigma=sig)
    with native.Plan(cfg, dtype=dtype) as plan:
        plan.search(cube.cuda(), torch.as_tensor(sig).cuda())
        snr, idx = plan.best()
        cand = plan.candidates()
    parity.compare_best(snr, idx, best)
    parity.compare_candidates(cand, best, cfg.threshold, np.arange(cfg.n_pix), cfg.nx)


def test_mid_window_unaligned_cube_and_ties(native):
    """A cube that starts off a 16-byte boundary (plain loads), and exact ties on a constant cube: the
    smallest DM, width and sample win."""
    cfg = synth.SearchConfig(ny=3, nx=5, n_t=130, dm=np.linspace(0.0, 2000.0, 12),
                             widths=np.array([1, 2, 4, 8, 64], np.int32), threshold=3.0)
    cube = synth.plain_noise(cfg, 4)
    buf = torch.empty(cube.numel() + 1, device="cuda")
    off = buf[1:].view(cube.shape)
    off.copy_(cube)
    with native.Plan(cfg) as plan:
        plan.search(cube.cuda())
        a, ia = plan.best()
        plan.search(off)
        b, ib = plan.best()
        assert (a == b).all() and (ia == ib).all()
        plan.search(torch.zeros(cube.shape, device="cuda"))
        z, iz = plan.best()
    assert (z == 0.0).all() and (iz == 0).all()


def test_mid_window_mad_flags_pixels(native):
    """MAD slabs of a mid window, one pixel with a constant row."""
    cfg = synth.SearchConfig(ny=3, nx=4, n_t=240, dm=np.linspace(0.0, 4000.0, 16),
                             widths=np.array([1, 4, 32, 128], np.int32), threshold=4.0)
    cube = synth.plain_noise(cfg, 6)
    cube[5, 3] = 1.5
    with native.Plan(cfg, noise="mad") as plan:
        plan.search(cube.cuda())
        snr, idx = plan.best()
    keep = np.arange(cfg.n_pix) != 5
    sh = oracle.delay_table(cfg.freq_mhz, cfg.dm)
    _, best, _ = oracle.search_cube(cube.numpy()[keep], sh, cfg.widths, mad=True)
    parity.compare_best(snr[keep], idx[keep], best)
    assert snr[5] == -np.inf and (idx[5] == -1).all()
