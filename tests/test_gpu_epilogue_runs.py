"""How the epilogues walk through the accumulator columns, against the oracle, every output.
Channels-last layers with one tile per CTA: rows dealt out to the warps, also where they do not divide; without
junk columns (1x1) the rows of a unit are one run of pixels.  Shared reductions: the parts lie in pairs of columns,
and rows that begin in the middle of a pair (odd pitch) are read one by one."""
import numpy as np
import pytest

from paper_1901_00858_b200 import workloads
from gpu_util import attach_guarded_workspace, check_close, check_guards, guarded_output, max_ulp_error, params_dict, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hgc():
    import torch
    assert torch.cuda.is_available()
    from paper_1901_00858_b200 import binding
    binding.lib()
    return binding


# (layer, channels-last, what the plan has to be)
CASES = [
    (params_dict(16, 256, 14, 14, 256, 1, 1), True, {}),
    (params_dict(3, 64, 14, 14, 1024, 1, 1), True, {}),                # whole planes per tile
    (params_dict(9, 128, 7, 7, 512, 1, 1), True, {}),                  # several images per tile
    (params_dict(2, 64, 13, 11, 96, 1, 1), True, {}),                  # odd rows, rows that do not divide
    (params_dict(1, 64, 5, 31, 32, 1, 1), True, {}),
    (params_dict(1, 64, 9, 33, 32, 1, 1), True, {}),                   # rows of more than 32 pixels: one at a time
    (params_dict(2, 128, 14, 14, 128, 3, 3, 1, 1), True, {}),          # junk columns between the rows
    (params_dict(3, 96, 13, 13, 64, 3, 3, 1, 1, 2, 2), True, {}),
    (params_dict(1, 1024, 12, 9, 320, 2, 2), False, dict(k_slices=4, th=3, pitch=9)),     # TMA-store epilogue, odd rows of columns
    (params_dict(1, 1024, 12, 17, 320, 3, 2, 1, 0), False, dict(k_slices=4, th=2, pitch=17)),
    (params_dict(1, 1024, 12, 17, 320, 2, 2), True, dict(k_slices=4, th=2, pitch=17)),    # channels-last, staged
    (params_dict(1, 1024, 12, 9, 320, 3, 3, 1, 1), True, dict(k_slices=4, th=3, pitch=11)),
    (params_dict(1, 2048, 9, 12, 64, 2, 2), True, dict(k_slices=4)),
]


@pytest.mark.parametrize("a,nhwc,plan", CASES)
def test_epilogue_runs(hgc, oracle, a, nhwc, plan):
    import torch
    d = hgc.ConvDesc(flags=hgc.HGC_FLAG_X_NHWC | hgc.HGC_FLAG_Y_NHWC if nhwc else 0, **a)
    info = d.plan_info()
    assert info["k_slices"] > 1 or info["tiles"] <= info["grid"], info
    assert all(info[k] == v for k, v in plan.items()), info
    rng = np.random.default_rng(a["c"] + a["h"])
    x, w, b = workloads.random_layer_tensors(rng, a["n"], a["c"], a["h"], a["w"], a["k"], a["r"], a["s"], a["group"])
    ws = attach_guarded_workspace(d)
    n, k, p, q = d.output_dims()
    xd, wd, bd = to_dev(np.ascontiguousarray(x.transpose(0, 2, 3, 1)) if nhwc else x), to_dev(w), to_dev(b)
    d.set_weights(wd)
    for relu, bias in ((True, bd), (False, None)):
        ref = oracle.conv_fast(oracle.ConvParams(**a), x, w, None if bias is None else b, relu)
        y_whole, y = guarded_output((n, p, q, k) if nhwc else (n, k, p, q))
        hgc.conv_forward(d, xd, wd, bias, y, relu)
        torch.cuda.synchronize()
        assert d.last_device_status() == hgc.HGC_OK
        check_guards(y_whole, "y")
        check_guards(ws, "workspace")
        got = to_host(y)
        got = got.transpose(0, 3, 1, 2) if nhwc else got
        check_close(got, ref, what=str(a))
        assert max_ulp_error(np.ascontiguousarray(got), ref) <= 1, a
    d.close()
