"""Inference with batch norm, ReLU and pooling in the tcgen05 convolution's epilogue vs the FP64 oracle."""
import numpy as np
import pytest
import torch

from oracle import cnn
from tests.test_classifier_gpu import _as_oracle_params, _bf16, _init, _make, native  # noqa: F401

pytestmark = pytest.mark.gpu


# every channel pair with a fused kernel, in the first block or the second; sides of one and several bricks,
# batches of one and of an odd number
@pytest.mark.parametrize("b,d,h,w,c0,c", [
    (1, 16, 16, 16, 16, (16, 16, 8, 8)), (3, 32, 32, 32, 16, (16, 32, 16, 16)), (1, 32, 32, 32, 16, (32, 16, 16, 8)),
    (2, 32, 32, 32, 32, (32, 64, 16, 16)), (1, 32, 32, 32, 16, (64, 16, 16, 16)), (2, 16, 32, 48, 32, (16, 16, 16, 16)),
    (3, 32, 32, 64, 16, (32, 32, 32, 16)),
])
def test_fused_inference(native, b, d, h, w, c0, c):  # noqa: F811
    dims = cnn.CnnDims(B=b, D=d, H=h, W=w, C0=c0, C=c, F=8)
    rng = np.random.default_rng(d + w + c0)
    x = rng.standard_normal((b, d, h, w, c0)).astype(np.float32)
    p = _init(dims, 4)
    nc = sum(c)
    rm = rng.normal(0.0, 0.2, nc).astype(np.float32)
    rv = rng.uniform(0.5, 2.0, nc).astype(np.float32)
    clf = _make(native, dims)
    clf.set_params(p)
    clf.set_bn_stats(rm, rv)
    z = clf.infer(torch.from_numpy(x).to(torch.bfloat16).cuda()).cpu().numpy()
    clf.close()
    ref = cnn.forward_backward(dims, _as_oracle_params(dims, p), _bf16(x), train=False, run_mean=rm, run_var=rv,
                               grads=False, bf16_storage=True)
    # one BF16 unit of the storage network's logits plus 1e-3 for the FP32 sums of the head
    assert (np.abs(z - ref["logits"]) <= 2.0 ** -7 * np.abs(ref["logits"]) + 1e-3).all()
