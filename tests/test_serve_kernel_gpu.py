"""The serving kernel (boxcars updated from DM row to DM row) vs the FP64 oracle's masked search."""
import numpy as np
import pytest
import torch

import oracle
from paper_2510_18136_gb300 import synth

pytestmark = pytest.mark.gpu

STORE = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


@pytest.fixture(scope="module")
def native():
    from paper_2510_18136_gb300 import build
    build.build()
    from paper_2510_18136_gb300 import native as nat
    assert torch.cuda.is_available()
    return nat


# blocks of one to 32 samples (32: the ends move out of the lanes whenever the delay grows), windows at the
# kernel's edges and of odd length, delays longer than the block and than the window, delays that grow
# by several samples per row, few rows, more pixels than teams
@pytest.mark.parametrize("n_t,n_pix,n_sub,n_dm,dm_hi,n_blk,dtype", [
    (1200, 5, 16, 64, 2000.0, 25, "bf16"), (1200, 3, 16, 64, 2000.0, 32, "f32"), (1215, 3, 16, 30, 4000.0, 31, "f16"),
    (704, 3, 16, 16, 9000.0, 7, "bf16"), (703, 4, 16, 16, 2000.0, 25, "f32"), (401, 3, 7, 12, 60000.0, 25, "bf16"),
    (60, 3, 16, 20, 20000.0, 30, "f32"), (33, 2, 16, 9, 20000.0, 32, "bf16"), (800, 3, 16, 1, 500.0, 1, "f32"),
    (1000, 1300, 8, 5, 2000.0, 25, "bf16"), (97, 3, 16, 200, 30000.0, 13, "f16"),
])
def test_serve_kernel(native, n_t, n_pix, n_sub, n_dm, dm_hi, n_blk, dtype):
    rng = np.random.default_rng(n_t + n_dm)
    every = [1, 2, 3, 4, 8, 16, 32, 64, 100, 128, 256, 512, 700, 1024, n_t]
    widths = np.array(sorted({w for w in every if w <= n_t}), np.int32)
    cfg = synth.SearchConfig(ny=1, nx=n_pix, n_sub=n_sub, n_t=n_t, freq_mhz=synth.band_centres(n_sub),
                             dm=np.sort(rng.uniform(0, dm_hi, n_dm)), widths=widths, threshold=-100.0)
    n_blocks = -(-n_t // n_blk) + 2
    x = rng.standard_normal((n_pix, n_sub, n_blocks * n_blk)).astype(np.float32)
    sh = oracle.delay_table(cfg.freq_mhz, cfg.dm)
    pix = np.arange(n_pix) if n_pix < 10 else np.r_[0:4, n_pix - 4:n_pix]
    with native.Plan(cfg, dtype=dtype) as plan:
        plan.stream_open(n_blk)
        view = plan.stream_block()
        for b in range(n_blocks):
            blk = torch.from_numpy(np.ascontiguousarray(x[:, :, b * n_blk:(b + 1) * n_blk].transpose(2, 1, 0)))
            view.copy_(blk.view(view.shape))
            plan.stream_push_device()
            cand, _ = plan.stream_poll(timeout_ms=20000)
            if b + 3 < n_blocks:
                continue
            end = (b + 1) * n_blk
            win = np.zeros((len(pix), n_sub, n_t), np.float32)
            lo = max(0, end - n_t)
            win[:, :, n_t - (end - lo):] = x[pix, :, lo:end]
            win = torch.from_numpy(win).to(STORE[dtype]).float().numpy().astype(np.float64)
            best = np.full(len(pix), -np.inf)
            for s in np.unique(sh, axis=0):
                length = n_t - int(s.max())
                if length < 1:
                    continue
                d = sum(win[:, k, s[k]:s[k] + length] for k in range(n_sub))
                sums = np.concatenate([np.zeros((len(pix), 1)), np.cumsum(d, axis=1)], axis=1)
                for w in (int(v) for v in widths):
                    t = np.arange(max(0, length - w - n_blk + 1), length - w + 1)
                    if t.size:
                        best = np.maximum(best, ((sums[:, t + w] - sums[:, t]) / (np.sqrt(n_sub * w))).max(axis=1))
            got = {int(c["col"]): c for c in cand}
            assert sorted(got) == list(range(n_pix))
            for q, p in enumerate(pix):
                c = got[int(p)]
                # FP32 sums: 1e-5 relative to the larger of 1 and the S/N, as everywhere
                assert abs(float(c["snr"]) - best[q]) <= 1e-5 * max(1.0, abs(best[q]))
                s, w, t = sh[c["dm_idx"]], int(widths[c["w_idx"]]), int(c["t_idx"])
                length = n_t - int(s.max())
                assert max(0, length - w - n_blk + 1) <= t <= length - w
                direct = sum(win[q, k, t + s[k]:t + s[k] + w].sum() for k in range(n_sub)) / np.sqrt(n_sub * w)
                assert abs(direct - best[q]) <= 2e-5 * max(1.0, abs(best[q]))
