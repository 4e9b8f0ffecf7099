"""Layers whose weight tiles stay in the operand ring from its first lap on (several tiles per CTA, a whole
number of tiles' stages in the ring, a channel tile that does not change within a CTA), and
replicated weight rows with 16- and 32-pixel epilogue units.  Against the oracle, every output."""
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


# (layer, replicas)
CASES = [
    (params_dict(22, 64, 56, 56, 64, 3, 3, 1, 1), 1),          # three stages per tile, ring of three
    (params_dict(40, 256, 28, 28, 64, 1, 1), 1),              # four stages per tile, x in place
    (params_dict(24, 64, 56, 56, 256, 1, 1), 1),              # two channel tiles, one per CTA
    (params_dict(13, 128, 28, 28, 512, 1, 1), 1),             # four channel tiles, two stages
    (params_dict(30, 64, 28, 28, 128, 1, 1, 0, 0, 1, 1, 1, 1, 2), 1),   # two groups
    (params_dict(5, 3, 224, 224, 64, 7, 7, 3, 3, 2, 2), 2),   # stem: units of 16 pixels
    (params_dict(6, 3, 200, 192, 32, 3, 3, 1, 1, 2, 2), 4),   # 32 channels: four copies
    (params_dict(7, 3, 37, 208, 32, 3, 3, 1, 1), 4),
    (params_dict(8, 32, 61, 112, 64, 1, 1), 2),               # ragged last row tile
]


@pytest.mark.parametrize("a,replicas", CASES)
def test_resident_weights(hgc, oracle, a, replicas):
    rng = np.random.default_rng(a["c"] * 1000 + a["h"])
    x, w, b = workloads.random_layer_tensors(rng, a["n"], a["c"], a["h"], a["w"], a["k"], a["r"], a["s"], a["group"])
    d = hgc.ConvDesc(**a)
    info = d.plan_info()
    d.close()
    assert info["resident"] == 1 and info["replicas"] == replicas and info["tiles"] > info["grid"], info
    for relu, bias in ((True, b), (False, None)):
        ref = oracle.conv_fast(oracle.ConvParams(**a), x, w, bias, relu)
        got, _ = run_layer(hgc, a, x, w, bias, relu, register_weights=True)
        check_close(got, ref, what=str(a))
