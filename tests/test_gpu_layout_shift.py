"""NCHW -> NHWC of planes that are no multiple of 4 pixels, whose channel rows start on any 2-byte boundary:
every shift, planes shorter than a vector, channel chunks with missing channels, the end of the tensor,
both sides of the rules that pick the kernel.  Bit for bit against the oracle, padding included."""
import numpy as np
import pytest

from gpu_util import to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,c,h,w,c_pad", [
    (2, 64, 11, 13, 64), (3, 65, 9, 17, 72), (1, 130, 1, 131, 136), (5, 71, 2, 67, 72), (2, 64, 1, 3, 64), (1, 66, 5, 1, 72),
    (1, 64, 1, 2, 64), (2, 127, 43, 3, 128), (1, 60, 13, 10, 64), (16, 9, 89, 83, 16), (8, 3, 211, 213, 8), (3, 17, 45, 45, 24),
    (2, 72, 11, 11, 72), (1, 61, 7, 7, 64), (1, 257, 53, 67, 264), (20, 48, 33, 35, 48),
])
def test_nchw_to_nhwc_exact(oracle, n, c, h, w, c_pad):
    import torch
    from paper_1901_00858_b200 import binding as hgc
    rng = np.random.default_rng(n * 1000 + c + w)
    x = rng.uniform(-4, 4, (n, c, h, w)).astype(np.float16)
    want = oracle.nchw_to_nhwc(x, c_pad)
    out = torch.full((n, h, w, c_pad), float("nan"), dtype=torch.float16, device="cuda")
    hgc.layout_nchw_to_nhwc(to_dev(x), out, n, c, h, w, c_pad)
    torch.cuda.synchronize()
    assert np.array_equal(to_host(out).view(np.uint16), want.view(np.uint16))
