"""Failure detection without a fault: every device-side wait of the TMA-fed kernels is bounded.
The tests shorten the bound to a few milliseconds and make one copy never arrive (the first CTA
announces it and does not issue it), then check what a caller sees: the launch ends by itself,
the status reads HGC_DEVICE_TIMEOUT once, forwards are skipped until it has been read, and the
next forward on the same descriptor is correct again.  Nothing here traps, faults or waits
without bound."""
import time

import numpy as np
import pytest

from paper_1901_00858_b200 import workloads
from gpu_util import check_close, params_dict, to_dev, to_host

pytestmark = pytest.mark.gpu
LIMIT_NS = 2_000_000     # 2 ms per wait


@pytest.fixture(scope="module")
def hgc():
    import torch
    assert torch.cuda.is_available()
    from paper_1901_00858_b200 import binding
    binding.lib()
    return binding


def _forward(hgc, d, xd, wd, bd, shape, relu=True):
    import torch
    y = torch.full(shape, float("nan"), dtype=torch.float16, device="cuda")
    hgc.conv_forward(d, xd, wd, bd, y, relu)
    torch.cuda.synchronize()
    return y


@pytest.mark.parametrize("name,a,flags_name,drop", [
    ("one tile on one CTA, second ring stage", params_dict(1, 32, 8, 8, 32, 3, 3, 1, 1), "", 1),
    ("several CTAs, first stage of the first CTA", params_dict(4, 64, 16, 16, 256, 3, 3, 1, 1), "", 0),
    ("CTA pairs: the first CTA's copies of a stage", params_dict(2, 64, 12, 12, 256, 3, 3, 1, 1), "pairs", 2),
    ("tiles shared between CTAs: a part that is never handed over", params_dict(2, 256, 24, 24, 256, 3, 3, 1, 1), "shared", 0),
    ("layout pass inside the kernel", params_dict(2, 64, 24, 24, 64, 3, 3, 1, 1), "fused", 1),
    ("whole-plane epilogue (the warps of a lane quarter meet on a bounded barrier)", params_dict(40, 64, 14, 14, 256, 1, 1), "", 0),
    ("x gathered by the kernel's own warps: the weight copy of a later stage", params_dict(20, 256, 14, 14, 256, 1, 1), "gather", 1),
])
def test_tensor_core_wait_runs_out_and_the_descriptor_recovers(hgc, oracle, name, a, flags_name, drop):
    import torch
    flags = {"": 0, "pairs": hgc.HGC_FLAG_CTA_PAIRS, "shared": hgc.HGC_FLAG_SHARED_TILES,
             "fused": hgc.HGC_FLAG_FUSED_LAYOUT, "gather": hgc.HGC_FLAG_GATHER_X}[flags_name]
    _runs_out_and_recovers(hgc, oracle, name, a, flags, drop)


DROP_SLAB = 1 << 20

NEWER_FORMS = [
    # (name, layer, flags, stage whose copies never arrive, what the plan has to be)
    ("cluster of four, parts behind the ring", params_dict(1, 1024, 7, 7, 64, 3, 3, 1, 1), "", 3, dict(k_slices=4, parts=1)),
    ("cluster of four, parts inside the ring", params_dict(3, 512, 24, 24, 320, 3, 3, 1, 1), "", 1, dict(k_slices=4, parts=2)),
    ("cluster of two, channels-last", params_dict(8, 1000, 14, 14, 320, 3, 3, 1, 1), "nhwc", 0, dict(k_slices=2, parts=2)),
    ("cluster of eight, inner product", params_dict(1, 3392, 1, 1, 129, 1, 1), "", 2, dict(k_slices=8, parts=1)),
    ("cluster of eight, parts inside the ring", params_dict(3, 1300, 16, 7, 129, 1, 3, 0, 1), "", 1, dict(k_slices=8, parts=2)),
    ("row pairs beside their weight slabs", params_dict(1, 64, 32, 128, 64, 3, 3, 1, 1), "", 2, dict(weight_slabs=1)),
    ("row pairs, a weight slab", params_dict(1, 64, 32, 128, 64, 3, 3, 1, 1), "", DROP_SLAB, dict(weight_slabs=1)),
    ("resident weights, second lap of the ring", params_dict(22, 64, 56, 56, 64, 3, 3, 1, 1), "", 4, dict(resident=1, stages=3)),
    ("flat planes", params_dict(2, 325, 88, 43, 726, 1, 1), "", 1, dict(flat=1)),
]


@pytest.mark.parametrize("name,a,flags_name,drop,plan", NEWER_FORMS, ids=[c[0] for c in NEWER_FORMS])
def test_every_form_of_the_kernel_gives_up_and_recovers(hgc, oracle, name, a, flags_name, drop, plan):
    flags = {"": 0, "nhwc": hgc.HGC_FLAG_X_NHWC | hgc.HGC_FLAG_Y_NHWC}[flags_name]
    info = hgc.ConvDesc(flags=flags, **a).plan_info()
    assert all(info[k] == v for k, v in plan.items()), info
    _runs_out_and_recovers(hgc, oracle, name, a, flags, drop)


def _runs_out_and_recovers(hgc, oracle, name, a, flags, drop):
    import torch
    rng = np.random.default_rng(3)
    x, w, b = workloads.random_layer_tensors(rng, a["n"], a["c"], a["h"], a["w"], a["k"], a["r"], a["s"], a["group"])
    ref = oracle.conv_fast(oracle.ConvParams(**a), x, w, b, True)
    d = hgc.ConvDesc(flags=flags, **a)
    assert d.path() == hgc.HGC_PATH_IGEMM
    if flags & hgc.HGC_FLAG_X_NHWC:
        x, ref = (np.ascontiguousarray(t.transpose(0, 2, 3, 1)) for t in (x, ref))
    d.ensure_workspace()
    shape = ref.shape
    xd, wd, bd = to_dev(x), to_dev(w), to_dev(b)
    d.set_weights(wd)
    check_close(to_host(_forward(hgc, d, xd, wd, bd, shape)), ref, what=name + " (before)")
    assert d.last_device_status() == hgc.HGC_OK
    try:
        hgc.debug_set_wait_limit_ns(LIMIT_NS)
        hgc.debug_drop_copies(drop)
        t0 = time.time()
        _forward(hgc, d, xd, wd, bd, shape)
        assert time.time() - t0 < 2.0, "the launch must end within a few wait limits"
        hgc.debug_drop_copies(-1)
        # the word is still raised: this forward is skipped and leaves y as it was
        y_skipped = _forward(hgc, d, xd, wd, bd, shape)
        assert bool(torch.isnan(y_skipped).all())
        assert d.last_device_status() == hgc.HGC_DEVICE_TIMEOUT
        assert d.last_device_status() == hgc.HGC_OK          # reading it cleared it
    finally:
        hgc.debug_drop_copies(-1)
        hgc.debug_set_wait_limit_ns(0)
    for rep in range(2):
        check_close(to_host(_forward(hgc, d, xd, wd, bd, shape)), ref, what=f"{name} (after, {rep})")
    assert d.last_device_status() == hgc.HGC_OK
    d.close()


def test_depthwise_copy_never_arrives(hgc, oracle):
    """The TMA-fed channels-last depthwise kernel: same form."""
    import torch
    a = params_dict(2, 64, 20, 20, 64, 3, 3, 1, 1, 1, 1, 1, 1, 64)
    rng = np.random.default_rng(4)
    x, w, b = workloads.random_layer_tensors(rng, a["n"], a["c"], a["h"], a["w"], a["k"], 3, 3, 64)
    ref = oracle.conv_fast(oracle.ConvParams(**a), x, w, b, True)
    d = hgc.ConvDesc(flags=hgc.HGC_FLAG_X_NHWC | hgc.HGC_FLAG_Y_NHWC, **a)
    assert d.path() == hgc.HGC_PATH_DEPTHWISE
    n, k, p, q = d.output_dims()
    xd = to_dev(np.ascontiguousarray(x.transpose(0, 2, 3, 1)))
    wd, bd = to_dev(w), to_dev(b)

    def run():
        return to_host(_forward(hgc, d, xd, wd, bd, (n, p, q, k))).transpose(0, 3, 1, 2)

    check_close(run(), ref, what="depthwise channels-last (before)")
    assert d.last_device_status() == hgc.HGC_OK
    try:
        hgc.debug_set_wait_limit_ns(LIMIT_NS)
        hgc.debug_drop_copies(0)
        t0 = time.time()
        run()
        assert time.time() - t0 < 2.0
        assert d.last_device_status() == hgc.HGC_DEVICE_TIMEOUT
        assert d.last_device_status() == hgc.HGC_OK
    finally:
        hgc.debug_drop_copies(-1)
        hgc.debug_set_wait_limit_ns(0)
    check_close(run(), ref, what="depthwise channels-last (after)")
    assert d.last_device_status() == hgc.HGC_OK
    d.close()


def test_block_with_teams_gives_up_and_recovers(hgc, oracle):
    """Depthwise + pointwise block whose depthwise warps form teams: the weight copy of a later stage."""
    import torch
    from test_gpu_dwpw import _block_tensors, _oracle_block
    n, c, h, w, k = 1, 712, 7, 7, 1000
    rng = np.random.default_rng(6)
    t = _block_tensors(rng, n, c, h, w, k)
    ref = _oracle_block(oracle, n, c, h, w, k, 1, *t, True, True)
    d = hgc.DwPwDesc(n, c, h, w, k, 1)
    assert d.plan_info()["dw_teams"] == 4
    d.ensure_workspace()
    xd = to_dev(np.ascontiguousarray(t[0].transpose(0, 2, 3, 1)))
    wd, bd, wp, bp = (to_dev(v) for v in t[1:])
    d.set_weights(wd, wp)

    def run():
        y = torch.full(ref.shape, float("nan"), dtype=torch.float16, device="cuda")
        hgc.dwpw_forward(d, xd, wd, bd, wp, bp, y, True, True)
        torch.cuda.synchronize()
        return y

    check_close(to_host(run()), ref, what="block (before)")
    for drop in (0, 5):
        try:
            hgc.debug_set_wait_limit_ns(LIMIT_NS)
            hgc.debug_drop_copies(drop)
            t0 = time.time()
            run()
            assert time.time() - t0 < 2.0
            hgc.debug_drop_copies(-1)
            assert bool(torch.isnan(run()).all())   # skipped
            assert d.last_device_status() == hgc.HGC_DEVICE_TIMEOUT
            assert d.last_device_status() == hgc.HGC_OK
        finally:
            hgc.debug_drop_copies(-1)
            hgc.debug_set_wait_limit_ns(0)
        for rep in range(2):
            check_close(to_host(run()), ref, what=f"block (after {drop}, {rep})")
    d.close()


def test_host_call_in_chunks_reports_a_timeout(hgc, oracle):
    """The chunks of a host call are descriptors of their own: their status is read through the caller's."""
    import torch
    a = params_dict(5, 32, 149, 151, 32, 3, 3, 1, 1)
    rng = np.random.default_rng(8)
    x, w, b = workloads.random_layer_tensors(rng, a["n"], a["c"], a["h"], a["w"], a["k"], 3, 3, 1)
    ref = oracle.conv_fast(oracle.ConvParams(**a), x, w, b, True)
    d = hgc.ConvDesc(**a)
    assert d.plan_info()["host_chunks"] == 3
    d.ensure_workspace(host=True)
    pinned = [torch.from_numpy(t.view(np.int16)).pin_memory() for t in (x, w, b)]

    def run():
        y = torch.full(ref.shape, float("nan"), dtype=torch.float16).pin_memory()
        hgc.conv_forward_host(d, *pinned, y, True)
        torch.cuda.synchronize()
        return y.numpy()

    check_close(run(), ref, what="host chunks (before)")
    try:
        hgc.debug_set_wait_limit_ns(LIMIT_NS)
        hgc.debug_drop_copies(1)
        t0 = time.time()
        run()
        assert time.time() - t0 < 2.0
        hgc.debug_drop_copies(-1)
        assert d.last_device_status() == hgc.HGC_DEVICE_TIMEOUT
        assert d.last_device_status() == hgc.HGC_OK
    finally:
        hgc.debug_drop_copies(-1)
        hgc.debug_set_wait_limit_ns(0)
    for rep in range(2):
        check_close(run(), ref, what=f"host chunks (after, {rep})")
    d.close()
