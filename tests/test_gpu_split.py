"""Tiles whose reduction a cluster of CTAs shares (plan_info k_slices): all cluster sizes, both stage
widths, the three epilogues, parts behind the ring and inside it, ragged channels, rows and images.
Against the oracle, every output; two runs give the same bits (the parts are added in a fixed order)."""
import numpy as np
import pytest

from paper_1901_00858_b200 import workloads
from gpu_util import attach_guarded_workspace, check_close, check_guards, guarded_output, params_dict, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hgc():
    import torch
    assert torch.cuda.is_available()
    from paper_1901_00858_b200 import binding
    binding.lib()
    return binding


# (n, c, h, w, k, kernel, stride, channels-last, CTAs per tile, parts behind the ring (1) or inside it (2))
CASES = [
    (1, 3392, 1, 1, 129, 1, 1, False, 8, 1),
    (8, 512, 13, 13, 320, 3, 1, False, 4, 2),   # copy epilogue, the last channel tile half empty
    (3, 512, 24, 24, 320, 3, 1, False, 4, 2),   # TMA-store epilogue
    (5, 1000, 28, 28, 130, 3, 1, False, 2, 1),   # 32-channel stages, two live channels in the second tile
    (8, 1000, 14, 14, 320, 3, 1, True, 2, 2),   # channels-last, staged
    (2, 1024, 16, 16, 130, 3, 1, True, 4, 1),   # channels-last, plain stores
    (3, 512, 24, 24, 130, 3, 1, False, 4, 2),
    (1, 512, 3, 3, 32, 3, 2, False, 4, 1),   # smallest: one tap per stage, 16 columns
    (2, 1000, 9, 9, 130, 3, 2, True, 4, 1),
    (3, 512, 7, 7, 96, 3, 1, False, 4, 1),
    (1, 25088, 1, 1, 129, 1, 1, False, 4, 1),   # inner products: one image, ragged channels
    (70, 4096, 1, 1, 200, 1, 1, False, 4, 1),
    (2, 8192, 3, 3, 40, 1, 1, False, 4, 1),
    (1, 1024, 7, 7, 64, 3, 1, False, 4, 1),
    (1, 2048, 16, 16, 100, 3, 1, False, 4, 1),
    (2, 3100, 7, 7, 32, 1, 1, False, 8, 1),   # copy epilogue of a cluster of eight
    (3, 1300, 16, 7, 129, (1, 3), 1, False, 8, 2),
    (3, 1100, 16, 16, 129, (1, 3), 1, False, 8, 2),   # TMA-store epilogue of a cluster of eight
    (1, 1100, 12, 16, 32, (3, 1), 1, False, 8, 1),
]


@pytest.mark.parametrize("n,c,h,w,k,kernel,stride,nhwc,slices,parts", CASES)
def test_split_reduction(hgc, oracle, n, c, h, w, k, kernel, stride, nhwc, slices, parts):
    import torch
    r, s = kernel if isinstance(kernel, tuple) else (kernel, kernel)
    rng = np.random.default_rng(n * 1000 + c + k)
    a = params_dict(n, c, h, w, k, r, s, r // 2, s // 2, stride, stride)
    x, wt, b = workloads.random_layer_tensors(rng, n, c, h, w, k, r, s, 1)
    d = hgc.ConvDesc(flags=hgc.HGC_FLAG_X_NHWC | hgc.HGC_FLAG_Y_NHWC if nhwc else 0, **a)
    assert d.plan_info()["k_slices"] == slices and d.plan_info()["parts"] == parts, d.plan_info()
    ws = attach_guarded_workspace(d)
    _, _, p, q = d.output_dims()
    xd, wd, bd = to_dev(np.ascontiguousarray(x.transpose(0, 2, 3, 1)) if nhwc else x), to_dev(wt), to_dev(b)
    d.set_weights(wd)
    for relu, bias in ((True, bd), (False, None)):
        ref = oracle.conv_fast(oracle.ConvParams(**a), x, wt, None if bias is None else b, relu)
        first = None
        for _ in range(2):
            y_whole, y = guarded_output((n, p, q, k) if nhwc else (n, k, p, q))
            hgc.conv_forward(d, xd, wd, bias, y, relu)
            torch.cuda.synchronize()
            assert d.last_device_status() == hgc.HGC_OK
            check_guards(y_whole, "y")
            check_guards(ws, "workspace")
            got = to_host(y)
            check_close(got.transpose(0, 3, 1, 2) if nhwc else got, ref, what=f"split relu={relu}")
            if first is None:
                first = got.copy()
        assert np.array_equal(first.view(np.uint16), got.view(np.uint16))
    d.close()
