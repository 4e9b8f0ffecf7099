"""1x1 layers that read x in place although no whole rows of theirs make a tile of a multiple of 8 pixels:
their planes are taken as rows of 8.  Against the oracle, every output; planes shorter than a
64-pixel box, a last tile of 8 pixels, odd channel counts, rows longer than a tile, the largest planes."""
import numpy as np
import pytest

from paper_1901_00858_b200 import workloads
from gpu_util import check_close, params_dict, run_layer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hgc():
    import torch
    assert torch.cuda.is_available()
    from paper_1901_00858_b200 import binding
    binding.lib()
    return binding


CASES = [
    params_dict(2, 325, 88, 43, 726, 1, 1),    # odd channels on both sides of a block
    params_dict(18, 208, 8, 33, 752, 1, 1),    # 264 pixels: one row of 8 more than a tile holds
    params_dict(3, 16, 8, 257, 9, 1, 1),       # rows longer than any tile, short reduction
    params_dict(2, 9, 1, 264, 130, 1, 1),      # one row
    params_dict(1, 48, 176, 210, 64, 1, 1),    # 64 channels: replicated weight rows
    params_dict(12, 64, 32, 45, 144, 1, 1),
    params_dict(1, 128, 12, 2002, 33, 1, 1),
]


@pytest.mark.parametrize("a", CASES)
def test_flat_planes(hgc, oracle, a):
    rng = np.random.default_rng(a["c"] * 1000 + a["h"])
    x, w, b = workloads.random_layer_tensors(rng, a["n"], a["c"], a["h"], a["w"], a["k"], a["r"], a["s"], a["group"])
    d = hgc.ConvDesc(**a)
    info = d.plan_info()
    dims = d.output_dims()
    d.close()
    assert info["path"] == hgc.HGC_PATH_IGEMM and info["x_source"] == 1 and info["flat"] == 1, info
    assert tuple(dims) == (a["n"], a["k"], a["h"], a["w"])
    for relu, bias in ((True, b), (False, None)):
        ref = oracle.conv_fast(oracle.ConvParams(**a), x, w, bias, relu)
        for registered in (True, False):
            got, _ = run_layer(hgc, a, x, w, bias, relu, register_weights=registered)
            check_close(got, ref, what=str(a))
