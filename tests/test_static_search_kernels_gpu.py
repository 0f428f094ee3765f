"""nsfrb_search_static runs the kernel nsfrb_search would: the same candidates, byte for byte, at one window of each."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2510_18136_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    from paper_2510_18136_gb300 import build
    build.build()
    from paper_2510_18136_gb300 import native as nat
    assert torch.cuda.is_available()
    return nat


# short, mid, team and wide kernels; a general kernel (few pixels); the long-window kernel (pixels too large)
@pytest.mark.parametrize("n_t,ny,dtype", [(25, 40, "f32"), (240, 32, "f32"), (240, 32, "bf16"), (1200, 16, "f32"),
                                          (1200, 20, "bf16"), (2048, 8, "f32"), (240, 4, "bf16"), (3000, 5, "f32")])
def test_static_search_equals_search(native, n_t, ny, dtype):
    cfg = synth.SearchConfig(ny=ny, nx=ny, n_t=n_t, dm=np.linspace(0.0, 2000.0, 40),
                             widths=np.array([1, 2, 4, 8, 16], np.int32), threshold=3.0)
    cube = synth.plain_noise(cfg, n_t, device="cuda").to(torch.float32 if dtype == "f32" else torch.bfloat16)
    sig = torch.full((cfg.n_pix,), 4.0, device="cuda")
    out = torch.zeros((cfg.n_pix, 6), dtype=torch.int32, device="cuda")
    total = torch.full((1,), -5, dtype=torch.int32, device="cuda")
    with native.Plan(cfg, dtype=dtype) as plan:
        plan.search(cube, sig)
        want = plan.candidates()
        st = native.lib.nsfrb_search_static(plan.handle, ctypes.c_void_p(cube.data_ptr()), ctypes.c_void_p(sig.data_ptr()),
                                            ctypes.c_void_p(out.data_ptr()), cfg.n_pix, ctypes.c_void_p(total.data_ptr()),
                                            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert st == native.OK
        torch.cuda.synchronize()
    assert int(total) == len(want) > 0
    assert out[:len(want)].cpu().numpy().tobytes() == want.tobytes()
