"""Binning through shared-memory tiles (factors from 32 up) against sums in 64 bits."""
import pytest
import torch

from paper_2510_18136_gb300 import synth  # noqa: F401  (the package builds the library)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def multiscale():
    from paper_2510_18136_gb300 import build
    build.build()
    from paper_2510_18136_gb300 import multiscale as ms
    assert torch.cuda.is_available()
    return ms


# rows of 1, 2, 4 and 8 to a 16-byte unit, factors with and without powers of two, one output a row, a
# remainder of samples, row counts that leave a tile short, rows as long as a stage and longer
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float16])
@pytest.mark.parametrize("n_pix,n_sub,n_t,factor", [
    (41, 16, 1200, 75), (7, 3, 1201, 64), (13, 5, 602, 150), (700, 16, 97, 33), (9, 7, 1200, 1200),
    (5, 2, 4096, 512), (3, 3, 5120, 96), (2, 3, 10243, 40), (300, 8, 64, 32), (1, 1, 33, 32)])
def test_bin_tiles(multiscale, dtype, n_pix, n_sub, n_t, factor):
    g = torch.Generator().manual_seed(factor + n_t)
    x = torch.randn((n_pix, n_sub, n_t), generator=g).to(dtype)
    n = n_t // factor
    ref = x[..., :n * factor].double().reshape(n_pix, n_sub, n, factor).sum(-1)
    # a sum of `factor` terms in FP32: at most factor roundings of 2^-24 of the sum of magnitudes
    tol = factor * 2.0 ** -24 * x[..., :n * factor].double().abs().reshape(n_pix, n_sub, n, factor).sum(-1)
    dev = x.cuda()
    got = multiscale.bin_time(dev, factor).cpu().double()
    assert ((got - ref).abs() <= tol).all()
    # off a 16-byte boundary: read in place
    buf = torch.empty(dev.numel() + 1, dtype=dtype, device="cuda")
    off = buf[1:].view(dev.shape)
    off.copy_(dev)
    got = multiscale.bin_time(off, factor).cpu().double()
    assert ((got - ref).abs() <= tol).all()


@pytest.fixture(scope="module")
def native(multiscale):
    from paper_2510_18136_gb300 import native as nat
    return nat


@pytest.mark.parametrize("give_up", [0, 1, 4, 7, 12])
@pytest.mark.parametrize("n_t,factor,dtype", [(1200, 75, torch.float32), (640, 32, torch.bfloat16), (1000, 1000, torch.float32)])
def test_a_wait_that_runs_out_leaves_the_sums(native, n_t, factor, dtype, give_up):
    """From a tile whose copy is given up the rows are read in place; enough rows for 13 tiles of each CTA."""
    row = n_t * (4 if dtype == torch.float32 else 2)
    n_rows = 13 * 304 * (20480 // row) + 5
    x = torch.randn((n_rows, n_t), generator=torch.Generator("cuda").manual_seed(1), device="cuda").to(dtype)
    want = torch.empty((n_rows, n_t // factor), device="cuda")
    got = torch.full_like(want, float("nan"))
    code = native.F32 if dtype == torch.float32 else native.BF16
    for k, out in ((-1, want), (give_up, got)):
        st = native.lib.nsfrb_dbg_bin_time(native._ptr(x), code, n_rows, n_t, factor, k, native._ptr(out),
                                           native._stream_handle(None))
        assert st == native.OK
    torch.cuda.synchronize()
    assert torch.equal(got, want)
