"""Served records of pixels with a very bright sample in or near the newest block, against 64-bit sums."""
import numpy as np
import pytest
import torch

import oracle
from paper_2510_18136_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    from paper_2510_18136_gb300 import build
    build.build()
    from paper_2510_18136_gb300 import native as nat
    assert torch.cuda.is_available()
    return nat


# A boxcar is the difference of two prefixes that hold the sample of -1e4, updated sample by sample: each rounding
# is uniform in half a unit u = 2^-10 (1e4 lies in [2^13, 2^14)), 0.29 u rms, and the few taken while the sample
# is in the sum add in squares: within 1 u rms.
@pytest.mark.parametrize("n_t,n_blk,n_dm,dm_hi,dtype", [(400, 25, 64, 2000.0, "f32"), (1200, 16, 200, 6000.0, "f32"),
                                                        (700, 8, 200, 6000.0, "bf16")])
def test_served_boxcars_beside_a_dip(native, n_t, n_blk, n_dm, dm_hi, dtype):
    cfg = synth.SearchConfig(ny=24, nx=24, n_t=n_t, dm=np.linspace(0.0, dm_hi, n_dm),
                             widths=np.array([1, 2, 4, 8, 16, 32], np.int32), threshold=2.0)
    total = n_t + n_blk - n_t % n_blk if n_t % n_blk else n_t
    x = np.random.default_rng(n_t).standard_normal((cfg.n_pix, 16, total)).astype(np.float32)
    for p in range(cfg.n_pix):
        x[p, p % 16, total - 1 - (p // 16) % 48] = -1e4
    blocks = torch.from_numpy(x).permute(2, 1, 0).reshape(total, 16, cfg.ny, cfg.nx).contiguous()
    with native.Plan(cfg, dtype=dtype) as plan:
        plan.stream_open(n_blk)
        for a in range(0, total, n_blk):
            plan.stream_push(blocks[a:a + n_blk])
            cand, _ = plan.stream_poll(timeout_ms=20000)
    store = torch.float32 if dtype == "f32" else torch.bfloat16
    win = torch.from_numpy(x[:, :, total - n_t:]).to(store).double().numpy()
    sh = oracle.delay_table(cfg.freq_mhz, cfg.dm)
    assert len(cand) > cfg.n_pix // 2
    err = []
    for c in cand:
        p, s = int(c["row"]) * cfg.nx + int(c["col"]), sh[int(c["dm_idx"])]
        w, t = int(cfg.widths[c["w_idx"]]), int(c["t_idx"])
        want = sum(win[p, k, t + s[k]:t + s[k] + w].sum() for k in range(16))
        err.append(float(c["snr"]) * 4.0 * np.sqrt(w) - want)
    u = 2.0 ** -10
    rms = float(np.sqrt(np.mean(np.square(err))))
    assert rms <= u, rms / u
