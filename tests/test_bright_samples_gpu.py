"""Search records beside very bright, invalid and infinite samples, against the FP64 oracle.

A dirty image has deep negative sidelobes and, where data were flagged, samples that are not numbers.  The
record of a pixel is compared with the best trial that holds no such sample:

* S/N within parity's 1e-5.  A boxcar of the wide kernel and of the in-lane widths of the mid and short
  kernels is summed from its own samples, so its error is a few times 2^-24 of its own value whatever
  lies outside it; sums that ran over a sample of -1e4 would be off by 2^-24 x 1e4 = 6e-4, 1e-5
  to 4e-5 of an S/N of 4 to 14 at the widths used.
* the indices wherever the margin to the next trial is clear.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2510_18136_gb300 import synth
from tests import parity

pytestmark = pytest.mark.gpu

STORE = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
N_PIX = 48


@pytest.fixture(scope="module")
def native():
    from paper_2510_18136_gb300 import build
    build.build()
    from paper_2510_18136_gb300 import native as nat
    assert torch.cuda.is_available()
    return nat


def _config(n_t, widths, n_dm=12):
    return synth.SearchConfig(ny=1, nx=N_PIX, n_t=n_t, dm=np.linspace(0.0, 1500.0, n_dm),
                              widths=np.array(widths, np.int32), threshold=4.0)


def _search(native, cfg, cube, sig, dtype):
    with native.Plan(cfg, dtype=dtype) as plan:
        native.lib.nsfrb_dbg_plan_by_length(plan.handle, 1)   # few pixels: general kernels are faster
        plan.search(cube.cuda(), torch.as_tensor(sig).cuda())
        return plan.best()


# every width where no long prefix is differenced (wide; not 3 and 25 with 2400 FP32 samples, which the long-window
# kernel takes), the in-lane widths elsewhere
ALL = [1, 2, 3, 4, 8, 16, 25, 32, 64, 100, 128, 256, 512, 1024, 1200]


@pytest.mark.parametrize("n_t,dtype,widths", [
    (50, "f32", [1, 2]), (50, "bf16", [1, 2]), (64, "f32", [1, 2]),
    (80, "f32", [1, 2, 4, 8, 16]), (95, "bf16", [1, 2, 4, 8, 16]), (240, "f32", [1, 2, 4, 8, 16]),
    (287, "f16", [1, 4, 16]), (400, "bf16", [2, 8, 16]), (600, "f32", [1, 2, 4, 8, 16]),
    (1250, "f32", ALL), (1407, "bf16", ALL), (1664, "f32", ALL), (2048, "f32", ALL), (2048, "bf16", ALL + [2048]),
    (2175, "bf16", ALL), (2400, "f32", [v for v in ALL if v not in (3, 25)]), (3000, "bf16", ALL), (4096, "f16", ALL),
])
def test_deep_dips(native, n_t, dtype, widths):
    cfg = _config(n_t, widths)
    rng = np.random.default_rng(n_t)
    cube = synth.plain_noise(cfg, n_t)
    sh = oracle.delay_table(cfg.freq_mhz, cfg.dm)
    for p in range(N_PIX):
        at = int(rng.integers(n_t))
        if p % 2:       # a pulse of 8 to 12 sigma shortly after the dip
            d, w = int(rng.integers(cfg.dm.size)), int(rng.choice([v for v in widths if v <= 64]))
            t = min(at + int(rng.integers(1, 40)), n_t - int(sh[d].max()) - w)
            if t >= 0:
                synth.add_pulse(cube, cfg, 0, p, t, w, rng.uniform(8, 12) / np.sqrt(16.0 * w), sh[d])
        cube[p, int(rng.integers(16)), at] = -1e4
    cube = cube.to(STORE[dtype])
    sig = np.full(N_PIX, 4.0, np.float32)
    _, best, _ = oracle.search_cube(cube.float().numpy(), sh, cfg.widths, sigma=sig)
    snr, idx = _search(native, cfg, cube, sig, dtype)
    parity.compare_best(snr, idx, best)


def _direct(x, sh, w, t):
    return float(sum(x[k, t + s:t + s + w].astype(np.float64).sum() for k, s in enumerate(sh)))


@pytest.mark.parametrize("value", [float("nan"), float("-inf")])
@pytest.mark.parametrize("n_t,dtype,w", [(60, "f32", 2), (60, "bf16", 1), (80, "f32", 4), (240, "bf16", 4), (240, "f32", 8),
                                         (600, "f32", 16), (700, "f32", 8), (1200, "bf16", 16), (1250, "f32", 4),
                                         (2048, "f32", 16), (2048, "bf16", 2), (2048, "f32", 3), (4000, "bf16", 8)])
def test_pulse_after_an_invalid_sample(native, n_t, dtype, w, value):
    """A strong pulse of an in-lane width after (or before) an invalid sample is the record."""
    cfg = _config(n_t, sorted({1, w}), n_dm=4)
    cube = synth.plain_noise(cfg, n_t + 1)
    sh = oracle.delay_table(cfg.freq_mhz, cfg.dm)
    far = 40 if n_t >= 200 else 20        # further than a lane's samples and the delays
    for p in range(N_PIX):
        at = (p * n_t) // N_PIX
        t = at + far if at + far + w + 8 <= n_t else at - far - w
        synth.add_pulse(cube, cfg, 0, p, t, w, 30.0 / np.sqrt(16.0 * w), sh[1])
        cube[p, p % 16, at] = value
    cube = cube.to(STORE[dtype])
    snr, idx = _search(native, cfg, cube, np.full(N_PIX, 4.0, np.float32), dtype)
    x = cube.float().numpy()
    for p in range(N_PIX):
        d, wi, t = (int(v) for v in idx[p])
        assert t >= 0 and snr[p] > 20.0, (p, snr[p], idx[p])
        want = _direct(x[p], sh[d], int(cfg.widths[wi]), t) / (4.0 * np.sqrt(float(cfg.widths[wi])))
        assert abs(float(snr[p]) - want) <= parity.tol(want), (p, snr[p], want)


@pytest.mark.parametrize("n_t,dtype", [(1250, "f32"), (2048, "bf16"), (3000, "bf16")])
def test_infinite_samples_of_long_windows_are_left_out(native, n_t, dtype):
    """Past 1247 samples a trial that holds +inf is no trial: the record is the best of the others before it."""
    cfg = _config(n_t, [1, 2, 8, 64, 100])
    cube = synth.plain_noise(cfg, 3)
    sh = oracle.delay_table(cfg.freq_mhz, cfg.dm)
    for p in range(N_PIX):
        synth.add_pulse(cube, cfg, 0, p, 200 + 3 * p, 8, 20.0 / np.sqrt(16.0 * 8), sh[2])
        cube[p, p % 16, 700 + 2 * p] = float("inf")
    cube = cube.to(STORE[dtype])
    sig = np.full(N_PIX, 4.0, np.float32)
    clean = torch.where(torch.isinf(cube.float()), torch.tensor(-1e6), cube.float())
    _, best, _ = oracle.search_cube(clean.numpy(), sh, cfg.widths, sigma=sig)
    snr, idx = _search(native, cfg, cube, sig, dtype)
    parity.compare_best(snr, idx, best)


@pytest.mark.parametrize("n_t,dtype", [(100, "f32"), (300, "bf16"), (400, "f32"), (607, "f32")])
def test_records_of_other_widths_are_those_of_their_trial(native, n_t, dtype):
    """Mid windows, widths with a prefix: the record's S/N is its trial's within 1e-6 beside a wide deep dip (sums
    of the rebuilt row's samples alone: 16 subbands and the prefix's value and error, each a few times 2^-24)."""
    cfg = _config(n_t, sorted({3, 7, 11, 25, 32, 60, n_t // 3}))
    cube = synth.plain_noise(cfg, n_t + 2)
    sh = oracle.delay_table(cfg.freq_mhz, cfg.dm)
    for p in range(N_PIX):
        cube[p, :, (p * n_t) // N_PIX:(p * n_t) // N_PIX + n_t // 8] -= 300.0
    cube = cube.to(STORE[dtype])
    snr, idx = _search(native, cfg, cube, np.full(N_PIX, 4.0, np.float32), dtype)
    x = cube.float().numpy()
    for p in range(N_PIX):
        d, wi, t = (int(v) for v in idx[p])
        w = int(cfg.widths[wi])
        want = _direct(x[p], sh[d], w, t) / (4.0 * np.sqrt(float(w)))
        assert abs(float(snr[p]) - want) <= 1e-6 * max(1.0, abs(want)), (p, snr[p], want)


@pytest.mark.parametrize("n_t,dtype", [(1, "f32"), (25, "f32"), (62, "bf16"), (64, "f16"), (65, "f32"), (300, "bf16"),
                                       (607, "f32"), (1248, "f32"), (2400, "bf16"), (4096, "bf16")])
def test_record_is_its_boxcar_divided_once(native, n_t, dtype):
    """Short, mid and long windows: of integer samples every boxcar is exact, and what is left is the quotient
    box / (sigma sqrt(w)), rounded once: half a unit in the last place, 2^-24 of it at most (and its square)."""
    cfg = _config(n_t, sorted({w for w in (1, 2, 4, 7, 16, 50, 200, n_t) if w <= n_t}))
    rng = np.random.default_rng(n_t)
    x = rng.integers(-100, 101, (N_PIX, 16, n_t)).astype(np.float32)     # sums below 2^24
    sig = rng.uniform(0.7, 300.0, N_PIX).astype(np.float32)
    sh = oracle.delay_table(cfg.freq_mhz, cfg.dm)
    snr, idx = _search(native, cfg, torch.from_numpy(x).to(STORE[dtype]), sig, dtype)
    for p in range(N_PIX):
        d, wi, t = (int(v) for v in idx[p])
        w = int(cfg.widths[wi])
        want = _direct(x[p], sh[d], w, t) / (float(sig[p]) * np.sqrt(float(w)))
        assert abs(float(snr[p]) - want) <= 1.01 * 2.0 ** -24 * abs(want), (p, snr[p], want)
