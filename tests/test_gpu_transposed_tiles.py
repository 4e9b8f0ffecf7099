"""Stride-1 layers whose kernel turns x (NCHW) channels-last itself, tile by tile (plan_info fused_layout 2):
against the oracle, every output.  Tiles that begin inside a group of 8 pixels (rows that are no multiple of 8 on
planes that are), blocks of 64 pixels that reach over the tile's input rows, borders wider than the kernel
needs, channel tails, groups, dilation, 64 output channels or fewer, shared reductions of both kinds, the
smallest planes.  The order of the sums is that of the separate pass: at most one unit in the last place from the
oracle."""
import numpy as np
import pytest

from paper_1901_00858_b200 import workloads
from gpu_util import check_close, max_ulp_error, params_dict, run_layer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hgc():
    import torch
    assert torch.cuda.is_available()
    from paper_1901_00858_b200 import binding
    binding.lib()
    return binding


# (layer, flags, what the plan has to be)
CASES = [
    (params_dict(2, 128, 56, 56, 256, 3, 3, 1, 1), "", dict(kb=32)),
    (params_dict(2, 64, 56, 56, 64, 3, 3, 1, 1), "", dict(kb=64)),                 # half of the staging tiles
    (params_dict(22, 64, 56, 56, 64, 3, 3, 1, 1), "", dict(kb=64, resident=1)),
    (params_dict(3, 128, 28, 28, 128, 3, 3, 1, 1), "", {}),                        # tiles begin 4 pixels into a group of 8
    (params_dict(2, 80, 16, 10, 40, 3, 3, 1, 1), "", {}),                          # rows of 10, copy epilogue, channel tail
    (params_dict(1, 49, 8, 15, 33, 3, 3, 1, 1), "", {}),                           # odd rows
    (params_dict(2, 64, 8, 8, 130, 3, 3, 1, 1), "", dict(tn=1)),                   # one block per tile
    (params_dict(1, 96, 40, 120, 72, 3, 3, 3, 4), "", {}),                         # wide borders
    (params_dict(2, 72, 24, 32, 100, 3, 3, 2, 2, 1, 1, 2, 2), "", {}),             # dilated
    (params_dict(1, 64, 24, 40, 96, 1, 7, 0, 3), "", {}),
    (params_dict(1, 64, 40, 24, 96, 7, 1, 3, 0), "", {}),                          # no border left and right
    (params_dict(2, 40, 16, 24, 20, 5, 5, 0, 0), "", {}),                          # unpadded
    (params_dict(2, 128, 24, 24, 256, 3, 3, 1, 1, 1, 1, 1, 1, 2), "", {}),         # groups of whole blocks
    (params_dict(1, 64, 112, 112, 128, 3, 3, 1, 1), "", dict(kb=32)),              # 64 channels as two blocks of 32
    (params_dict(1, 512, 28, 28, 512, 3, 3, 1, 1), "", dict(k_slices=4)),
    (params_dict(3, 512, 24, 24, 130, 3, 3, 1, 1), "", dict(k_slices=4)),
    (params_dict(2, 256, 56, 56, 256, 3, 3, 1, 1), "shared", dict(shared_tiles=1)),  # ranges that begin inside a channel block
]


@pytest.mark.parametrize("a,flag,plan", CASES)
def test_transposed_tiles(hgc, oracle, a, flag, plan):
    flags = hgc.HGC_FLAG_SHARED_TILES if flag else 0
    d = hgc.ConvDesc(flags=flags, **a)
    info = d.plan_info()
    d.close()
    assert info["fused_layout"] == 2 and all(info[k] == v for k, v in plan.items()), info
    rng = np.random.default_rng(a["c"] * 1000 + a["h"])
    x, w, b = workloads.random_layer_tensors(rng, a["n"], a["c"], a["h"], a["w"], a["k"], a["r"], a["s"], a["group"])
    for relu, bias in ((True, b), (False, None)):
        ref = oracle.conv_fast(oracle.ConvParams(**a), x, w, bias, relu)
        got, _ = run_layer(hgc, a, x, w, bias, relu, flags=flags, register_weights=relu)
        check_close(got, ref, what=str(a))
        assert max_ulp_error(got, ref) <= 1, a


def test_wait_for_a_block_of_x_runs_out(hgc, oracle):
    from test_gpu_timeouts import _runs_out_and_recovers
    a = params_dict(2, 128, 56, 56, 256, 3, 3, 1, 1)
    for drop in (0, 5, 11):
        _runs_out_and_recovers(hgc, oracle, f"block {drop} of x", a, 0, drop)
    _runs_out_and_recovers(hgc, oracle, "shared reduction, a block of x", params_dict(1, 512, 28, 28, 512, 3, 3, 1, 1), 0, 3)


def test_values_outside_a_channel_s_plane_do_not_reach_it(hgc):
    """Infinities in one channel's last row reach the outputs under the kernel only."""
    import torch
    d = hgc.ConvDesc(1, 40, 12, 10, 8, 3, 3, 1, 1)
    assert d.plan_info()["fused_layout"] == 2
    d.ensure_workspace()
    x = torch.ones((1, 40, 12, 10), dtype=torch.float16, device="cuda")
    x[0, 17, 11, 9] = float("inf")
    w = torch.ones((8, 40, 3, 3), dtype=torch.float16, device="cuda")
    y = torch.empty((1, 8, 12, 10), dtype=torch.float16, device="cuda")
    hgc.conv_forward(d, x, w, None, y, False)
    want = torch.zeros((12, 10), dtype=torch.bool, device="cuda")
    want[10:, 8:] = True
    assert bool(((~torch.isfinite(y[0])) == want).all())
    d.close()
