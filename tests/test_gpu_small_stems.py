"""Image stems of little work run as one launch (no copy of x): against the oracle, every output, at the edges
of its blocks (128 pixels, 8 channels), of its rule, and with strides, dilations, borders and channel counts it accepts.
Products of binary16 values are exact and at most 512 of them are summed in fp32, so a result is the oracle's
rounding or its neighbour."""
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


# (layer, launches of a forward with registered weights)
CASES = [
    (params_dict(1, 3, 32, 32, 16, 3, 3, 1, 1), 1),
    (params_dict(1, 1, 1, 127, 1, 1, 1), 1),                        # one pixel short of a block
    (params_dict(2, 2, 8, 16, 7, 1, 1), 1),                         # exactly a block
    (params_dict(1, 3, 3, 43, 9, 3, 3, 1, 1), 1),                   # one pixel more; one channel in the second block
    (params_dict(3, 6, 9, 11, 17, 3, 3, 1, 1), 1),                  # a block over all rows of a plane
    (params_dict(1, 1, 23, 19, 8, 5, 3, 2, 1, 2, 3), 1),            # strides, odd plane
    (params_dict(2, 2, 17, 21, 12, 3, 3, 4, 3, 1, 2, 2, 3), 1),     # dilated, border wider than the kernel
    (params_dict(1, 8, 11, 11, 5, 8, 8), 1),                        # 512 taps
    (params_dict(1, 1, 200, 1, 6, 7, 1, 3, 0), 1),                  # one column
    (params_dict(5, 3, 2, 2, 3, 2, 2), 1),                          # one output per image
    (params_dict(1, 3, 64, 64, 64, 3, 3, 1, 1), 1),                 # about the largest
    (params_dict(1, 3, 128, 128, 64, 3, 3, 1, 1), 2),               # too many products
    (params_dict(1, 3, 112, 112, 32, 3, 3, 1, 1, 2, 2), 2),         # too large an input tile
]


@pytest.mark.parametrize("a,launches", CASES)
def test_small_stem(hgc, oracle, a, launches):
    import torch
    rng = np.random.default_rng(a["h"] * 1000 + a["k"])
    x, w, b = workloads.random_layer_tensors(rng, a["n"], a["c"], a["h"], a["w"], a["k"], a["r"], a["s"], a["group"])
    for relu, bias in ((True, b), (False, None)):
        ref = oracle.conv_fast(oracle.ConvParams(**a), x, w, bias, relu)
        got, path = run_layer(hgc, a, x, w, bias, relu, register_weights=relu)
        assert path == hgc.HGC_PATH_IGEMM
        check_close(got, ref, what=str(a))
        assert max_ulp_error(got, ref) <= 1, a
    d = hgc.ConvDesc(**a)
    info = d.plan_info()
    assert (info["x_source"] == 5) == (launches == 1) and (info["tiles"] == 0) == (launches == 1), info
    d.ensure_workspace()
    xd, wd = (torch.from_numpy(t.view(np.int16)).cuda().view(torch.float16) for t in (x, w))
    d.set_weights(wd)
    y = torch.empty(d.output_dims(), dtype=torch.float16, device="cuda")
    before = hgc.kernel_launch_count()
    hgc.conv_forward(d, xd, wd, None, y, False)
    assert hgc.kernel_launch_count() - before == launches
    d.close()


def test_infinities_and_nans_go_where_the_definition_puts_them(hgc):
    """An infinity reaches the outputs under the kernel and no others, also across the zero border; a NaN passes the ReLU."""
    import torch
    d = hgc.ConvDesc(1, 3, 8, 10, 4, 3, 3, 1, 1)
    d.ensure_workspace()
    w = torch.ones((4, 3, 3, 3), dtype=torch.float16, device="cuda")
    for value in (float("inf"), float("nan")):
        x = torch.ones((1, 3, 8, 10), dtype=torch.float16, device="cuda")
        x[0, 1, 0, 9] = value
        y = torch.empty((1, 4, 8, 10), dtype=torch.float16, device="cuda")
        hgc.conv_forward(d, x, w, None, y, True)
        odd = ~torch.isfinite(y[0])
        want = torch.zeros((8, 10), dtype=torch.bool, device="cuda")
        want[:2, 8:] = True
        assert bool((odd == want).all()), value
    d.close()


def test_registered_weights_are_the_ones_that_were_registered(hgc):
    """A buffer may be reused after it has been registered; also by the chunks of a host call, which read what they were given."""
    import torch
    d = hgc.ConvDesc(1, 2, 9, 9, 5, 3, 3, 1, 1)
    d.ensure_workspace()
    x = torch.randn((1, 2, 9, 9), device="cuda").half()
    w = torch.randn((5, 2, 3, 3), device="cuda").half()
    y, z = (torch.empty((1, 5, 9, 9), dtype=torch.float16, device="cuda") for _ in range(2))
    hgc.conv_forward(d, x, w, None, y, False)
    d.set_weights(w)
    w.zero_()
    hgc.conv_forward(d, x, w, None, z, False)
    assert bool((y == z).all()) and float(y.abs().max()) > 0
    d.close()
    d = hgc.ConvDesc(64, 1, 192, 192, 1, 1, 1)
    assert d.plan_info()["host_chunks"] == 2
    d.ensure_workspace(host=True)
    x = torch.randn((64, 1, 192, 192)).half().pin_memory()
    for factor in (2.0, -3.0):
        w = torch.full((1, 1, 1, 1), factor).half().pin_memory()
        y = torch.empty((64, 1, 192, 192), dtype=torch.float16).pin_memory()
        hgc.conv_forward_host(d, x, w, None, y, False)
        torch.cuda.synchronize()
        assert bool((y == x * factor).all())
    d.close()
