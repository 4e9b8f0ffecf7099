"""3x3 layers of 65 to 96 channels per group: three 32-channel blocks.  Against the oracle, every output; the
ends of the range and their neighbours, odd channel counts, two groups."""
import numpy as np
import pytest

from paper_1901_00858_b200 import workloads
from gpu_util import check_close, params_dict, run_layer

pytestmark = pytest.mark.gpu

# (layer, channels per reduction block)
CASES = [
    (params_dict(9, 96, 56, 56, 96, 3, 3, 1, 1), 32),
    (params_dict(5, 65, 59, 58, 130, 3, 3, 1, 1), 32),
    (params_dict(4, 160, 56, 56, 160, 3, 3, 1, 1, 1, 1, 1, 1, 2), 32),
    (params_dict(3, 97, 56, 56, 96, 3, 3, 1, 1), 64),
    (params_dict(3, 96, 56, 56, 64, 3, 3, 1, 1), 64),
]


@pytest.mark.parametrize("a,kb", CASES)
def test_narrow_blocks(oracle, a, kb):
    from paper_1901_00858_b200 import binding as hgc
    rng = np.random.default_rng(a["c"] * 1000 + a["h"])
    x, w, b = workloads.random_layer_tensors(rng, a["n"], a["c"], a["h"], a["w"], a["k"], a["r"], a["s"], a["group"])
    d = hgc.ConvDesc(**a)
    info = d.plan_info()
    d.close()
    assert info["kb"] == kb, info
    for relu, bias in ((True, b), (False, None)):
        ref = oracle.conv_fast(oracle.ConvParams(**a), x, w, bias, relu)
        got, _ = run_layer(hgc, a, x, w, bias, relu, register_weights=True)
        check_close(got, ref, what=str(a))
