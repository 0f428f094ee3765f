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


@pytest.mark.parametrize("dtype,n_t,dm_hi,w_max", [("f32", 300, 2000.0, 64), ("bf16", 500, 4000.0, 128), ("f32", 200, 0.0, 1)])
def test_cutout_values_are_those_of_two_divisions(native, dtype, n_t, dm_hi, w_max):
    """Bit for bit (sum in sample order / bins) / (sigma / sqrt(n_sub)), rounded after each division and then to
    BF16, in FP32 on the device: the kernel multiplies by a reciprocal and divides only beside a midpoint of two
    BF16 values, one value in 4000, and without that about one in 20000 of these 8 million would differ."""
    d = h = w = 32
    n, n_sub = 16, 16
    widths = [v for v in (1, 2, 8, 32, 64, 128) if v <= w_max]
    cfg = synth.SearchConfig(ny=48, nx=48, n_t=n_t, dm=np.linspace(0.0, dm_hi, 8), widths=np.array(widths, np.int32),
                             threshold=6.0)
    store = torch.float32 if dtype == "f32" else torch.bfloat16
    cube = synth.plain_noise(cfg, 5, device="cuda").to(store)
    rng = np.random.default_rng(9)
    sig = torch.as_tensor(rng.uniform(3.0, 6.0, cfg.n_pix).astype(np.float32)).cuda()
    cand = np.zeros(n, native.CANDIDATE_DTYPE)
    for f, hi in (("row", 48), ("col", 48), ("dm_idx", 8), ("w_idx", len(widths)), ("t_idx", n_t - 20)):
        cand[f] = rng.integers(0, hi, n)
    with native.Plan(cfg, dtype=dtype) as plan:
        got = native.cutouts(plan, cube, native.candidates_to_device(cand), d=d, h=h, w=w, sigma=sig)
        smax = plan.info()[1]
    x = cube.view(48, 48, n_sub, n_t)
    for c in range(n):
        span = widths[cand["w_idx"][c]] + int(smax[cand["dm_idx"][c]])
        b = max(1, (span + d // 2 - 1) // (d // 2))
        t0 = int(cand["t_idx"][c]) + span // 2 - (d * b) // 2 + torch.arange(d, device="cuda") * b
        rows = int(cand["row"][c]) - h // 2 + torch.arange(h, device="cuda")
        cols = int(cand["col"][c]) - w // 2 + torch.arange(w, device="cuda")
        inside = ((rows >= 0) & (rows < 48))[:, None] & ((cols >= 0) & (cols < 48))[None, :]
        img = x[rows.clamp(0, 47)][:, cols.clamp(0, 47)].float()                    # [h, w, n_sub, n_t]
        acc = torch.zeros((d, h, w, n_sub), device="cuda")
        for j in range(b):
            t = t0 + j
            v = img[..., t.clamp(0, n_t - 1)].permute(3, 0, 1, 2)
            acc = torch.where(((t >= 0) & (t < n_t))[:, None, None, None], acc + v, acc)
        sg = sig[int(cand["row"][c]) * 48 + int(cand["col"][c])]
        want = acc / torch.tensor(float(b), device="cuda") / (sg / torch.tensor(float(n_sub), device="cuda").sqrt())
        want = torch.where(inside[None, :, :, None], want, torch.zeros_like(want)).to(torch.bfloat16)
        assert torch.equal(got[c], want)
