"""Cutouts of every size and storage, tile by tile, against the oracle's definition."""
import numpy as np
import pytest
import torch

import oracle
from oracle import cnn
from paper_2510_18136_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    from paper_2510_18136_gb300 import build
    build.build()
    from paper_2510_18136_gb300 import native as nat
    assert torch.cuda.is_available()
    return nat


# time bins below, at and past a tile's 32 (with a remainder), odd sides and subbands, rows wider than a tile
@pytest.mark.parametrize("d,h,w,n_sub,dtype", [
    (2, 1, 1, 1, "f32"), (5, 3, 7, 3, "bf16"), (16, 16, 16, 16, "f32"), (32, 4, 32, 16, "f16"), (33, 2, 5, 7, "f32"),
    (40, 3, 33, 32, "bf16"), (64, 2, 20, 16, "f32"), (31, 5, 9, 27, "f16")])
def test_cutouts_sizes(native, d, h, w, n_sub, dtype):
    cfg = synth.SearchConfig(ny=11, nx=23, n_sub=n_sub, n_t=90, freq_mhz=synth.band_centres(n_sub),
                             dm=np.linspace(0, 3000, 7), widths=np.array([1, 3, 17, 60], np.int32))
    rng = np.random.default_rng(d * 100 + w)
    cube = torch.from_numpy(rng.standard_normal((cfg.n_pix, n_sub, 90)).astype(np.float32))
    cube = cube.to({"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}[dtype])
    sigma = torch.from_numpy(rng.uniform(2, 6, cfg.n_pix).astype(np.float32))
    cands = np.zeros(9, dtype=native.CANDIDATE_DTYPE)
    for i in range(9):
        cands[i] = (rng.integers(11), rng.integers(23), rng.integers(7), rng.integers(4), rng.integers(90), 7.0)
    with native.Plan(cfg, dtype=dtype) as plan:
        out = native.cutouts(plan, cube.cuda(), native.candidates_to_device(cands), d=d, h=h, w=w, sigma=sigma.cuda())
    smax = oracle.delay_table(cfg.freq_mhz, cfg.dm).max(axis=1)
    ref = cnn.cutouts_grid(cube.float().numpy(), 11, 23, cands, smax, cfg.widths, d, h, w, sigma=sigma.numpy())
    # one BF16 unit for an FP32 value on the other side of a rounding boundary
    np.testing.assert_allclose(out.float().cpu().numpy(), ref, rtol=2 ** -7, atol=1e-6)
