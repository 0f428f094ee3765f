"""Plans of one kernel instance that need different shared memory, used from two host threads at once."""
import threading

import numpy as np
import pytest
import torch

from paper_2510_18136_gb300 import multiscale, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    from paper_2510_18136_gb300 import build
    build.build()
    from paper_2510_18136_gb300 import native as nat
    assert torch.cuda.is_available()
    return nat


def _in_two_threads(jobs):
    """Runs both jobs at once; raises what either of them raised."""
    raised = []

    def run(job):
        try:
            job()
        except Exception as e:
            raised.append(e)

    threads = [threading.Thread(target=run, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    if raised:
        raise raised[0]


# one window per kernel (several pixels to a warp, a warp per row, several warps per row, the MAD pass)
@pytest.mark.parametrize("n_t,noise", [(240, "known"), (1200, "known"), (2048, "known"), (240, "mad")])
def test_searches_of_two_plans(native, n_t, noise):
    def job(n_sub, got):
        cfg = synth.SearchConfig(ny=2, nx=4, n_sub=n_sub, n_t=n_t, freq_mhz=synth.band_centres(n_sub),
                                 dm=np.linspace(0.0, 500.0, 6), widths=np.array([1, 4, 16], np.int32), threshold=4.0)
        cube = synth.plain_noise(cfg, n_sub).cuda()
        torch.cuda.synchronize()

        def run():
            s = torch.cuda.Stream()
            with native.Plan(cfg, noise=noise) as plan:
                native.lib.nsfrb_dbg_plan_by_length(plan.handle, 1)   # few pixels: general kernels are faster
                for _ in range(400):
                    plan.search(cube, stream=s)
                got.append(plan.best()[0])
                plan.search(cube, stream=s)
                got.append(plan.best()[0])
        return run

    a, b = [], []
    _in_two_threads([job(6, a), job(16, b)])
    assert (a[0] == a[1]).all() and (b[0] == b[1]).all()


def test_binning_in_two_threads(native):
    def job(n_t):
        x = torch.ones((64, 4, n_t), device="cuda")
        torch.cuda.synchronize()

        def run():
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(400):
                    y = multiscale.bin_time(x, 32)
                assert (y == 32.0).all()
        return run

    _in_two_threads([job(640), job(4096)])


def test_serving_of_two_open_streams(native):
    """The smaller stream is opened after the larger one's graph was captured; both keep running."""
    plans = []
    for n_sub in (16, 6):
        cfg = synth.SearchConfig(ny=4, nx=4, n_sub=n_sub, n_t=300, freq_mhz=synth.band_centres(n_sub),
                                 dm=np.linspace(0.0, 500.0, 6), widths=np.array([1, 4, 16], np.int32), threshold=4.0)
        plan = native.Plan(cfg)
        plan.stream_open(20)
        plans.append((plan, torch.zeros((20, n_sub, 4, 4))))
    for _ in range(3):
        for plan, block in plans:
            plan.stream_push(block)
            cand, _ = plan.stream_poll(timeout_ms=10000)
            assert len(cand) == 0
    for plan, _ in plans:
        plan.close()


def test_two_imagers(native):
    """An imager of a smaller uv support made after a larger one; the larger one still images, same bits."""
    from paper_2510_18136_gb300 import synth_vis

    def make(n_ew, n_ns, n_grid):
        uv = synth_vis.baseline_uv(synth_vis.core_layout(0, n_ew, n_ns))
        chan = synth_vis.channel_freqs(4, 2)
        vis = synth_vis.visibilities(uv, chan, 1, [(3, -5, np.ones((1, 4)))], noise=1.0, seed=1, device="cuda")
        return native.Imager(uv, chan, n_grid=n_grid), vis

    large, vis = make(48, 34, 175)
    before = large.image(vis).clone()
    small, vis_small = make(12, 8, 64)
    small.image(vis_small)
    assert torch.equal(large.image(vis), before)
    large.status()
    small.close()
    large.close()
