"""hgc_conv_forward_host with enough images to be cut into chunks (copies in, kernels and copies out on
streams of their own): results against the oracle for chunks that do and do not divide the batch,
for planes whose bytes are not a multiple of the staging alignment, on the paths that read x in
place, through a layout pass and without tensor cores."""
import numpy as np
import pytest

from paper_1901_00858_b200 import workloads
from gpu_util import check_close, params_dict, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hgc():
    import torch
    assert torch.cuda.is_available()
    from paper_1901_00858_b200 import binding
    binding.lib()
    return binding


# (name, layer, chunks): 2 MB of x and of y per chunk at least
CASES = [
    ("3x3, five images in chunks of two and a last one of one", params_dict(5, 32, 149, 151, 32, 3, 3, 1, 1), 3),
    ("1x1 read in place, chunks of one", params_dict(3, 128, 96, 96, 128, 1, 1), 3),
    ("depthwise, four chunks", params_dict(10, 24, 160, 160, 24, 3, 3, 1, 1, 1, 1, 1, 1, 24), 4),
    ("grouped, generic kernel", params_dict(4, 63, 131, 127, 63, 3, 3, 1, 1, 1, 1, 1, 1, 3), 2),
    ("below two chunks: one piece", params_dict(3, 16, 100, 100, 16, 3, 3, 1, 1), 1),
]


@pytest.mark.parametrize("name,a,chunks", CASES, ids=[c[0] for c in CASES])
def test_host_forward_in_chunks(hgc, oracle, name, a, chunks):
    import torch
    d = hgc.ConvDesc(**a)
    assert d.plan_info()["host_chunks"] == chunks
    d.ensure_workspace(host=True)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    shape = d.output_dims()
    calls = []
    for i in range(4):   # new tensors on every call, alternating streams; nothing waits in between
        rng = np.random.default_rng(70 + i)
        x, w, b = workloads.random_layer_tensors(rng, a["n"], a["c"], a["h"], a["w"], a["k"], a["r"], a["s"], a["group"])
        bias = b if i % 2 == 0 else None
        pin = lambda t: None if t is None else torch.from_numpy(t.view(np.int16)).pin_memory()
        xh, wh, bh = pin(x), pin(w), pin(bias)
        yh = torch.full(shape, 0x7e00, dtype=torch.int16).pin_memory()   # binary16 NaN
        if i > 0:
            streams[i % 2].wait_stream(streams[(i - 1) % 2])
        hgc.conv_forward_host(d, xh, wh, bh, yh, True, streams[i % 2])
        calls.append((x, w, bias, xh, wh, bh, yh))
    streams[1].synchronize()
    assert d.last_device_status() == hgc.HGC_OK
    for x, w, bias, _, _, _, yh in calls:
        ref = oracle.conv_fast(oracle.ConvParams(**a), x, w, bias, True)
        check_close(yh.numpy().view(np.float16), ref, what=name)
    # the descriptor still serves device tensors from the same workspace
    x, w, bias = calls[0][:3]
    y = torch.empty(shape, dtype=torch.float16, device="cuda")
    hgc.conv_forward(d, to_dev(x), to_dev(w), to_dev(bias), y, True)
    torch.cuda.synchronize()
    check_close(to_host(y), oracle.conv_fast(oracle.ConvParams(**a), x, w, bias, True), what=name + " (device)")
    d.close()


# (name, layer, flags, chunks): layers for which the planner, asked for a chunk's few images, would take the sums in
# another order than for the whole batch: other reduction blocks, tiles shared by CTAs or not
SAME_BITS = [
    ("blocks of 32 channels, a chunk alone would take 64", params_dict(4, 128, 112, 112, 128, 3, 3, 1, 1), "", 4),
    ("the same, chunks of two and one", params_dict(5, 256, 56, 56, 256, 3, 3, 1, 1), "", 3),
    ("a chunk alone would be split over clusters", params_dict(8, 512, 28, 28, 512, 3, 3, 1, 1), "", 3),
    ("tiles shared by CTAs in the whole batch", params_dict(16, 256, 56, 56, 256, 3, 3, 1, 1), "", 1),
    ("row pairs", params_dict(4, 64, 224, 224, 64, 3, 3, 1, 1), "", 4),
    ("stem", params_dict(33, 3, 224, 224, 64, 7, 7, 3, 3, 2, 2), "", 4),
    ("stem whose chunks are of little work (1x3)", params_dict(64, 2, 128, 128, 2, 1, 3, 0, 1), "", 2),
    ("the same, 1x7", params_dict(128, 1, 128, 128, 1, 1, 7, 0, 3), "", 2),
    ("the same, 2x2", params_dict(128, 1, 192, 192, 1, 2, 2), "", 4),
    ("the same, 1x1, last chunk smaller", params_dict(200, 3, 128, 128, 1, 1, 1), "", 3),
    ("the same, 1x1", params_dict(400, 3, 96, 96, 2, 1, 1), "", 4),
    ("1x1 read in place", params_dict(8, 256, 56, 56, 512, 1, 1), "", 4),
    ("CTA pairs whose chunks would take other blocks", params_dict(6, 128, 56, 56, 256, 3, 3, 1, 1), "pairs", 1),
    ("depthwise", params_dict(32, 32, 112, 112, 32, 3, 3, 1, 1, 1, 1, 1, 1, 32), "", 4),
    ("depthwise channels-last", params_dict(32, 64, 112, 112, 64, 3, 3, 1, 1, 1, 1, 1, 1, 64), "nhwc", 4),
]


@pytest.mark.parametrize("name,a,how,chunks", SAME_BITS, ids=[c[0] for c in SAME_BITS])
def test_host_forward_gives_the_bits_of_the_device_forward(hgc, name, a, how, chunks):
    import torch
    flags = {"": 0, "pairs": hgc.HGC_FLAG_CTA_PAIRS, "nhwc": hgc.HGC_FLAG_X_NHWC | hgc.HGC_FLAG_Y_NHWC}[how]
    g = torch.Generator(device="cuda").manual_seed(a["c"] * 100 + a["n"])
    d = hgc.ConvDesc(flags=flags, **a)
    assert d.plan_info()["host_chunks"] == chunks, d.plan_info()
    d.ensure_workspace(host=True)
    n, k, p, q = d.output_dims()
    rand = lambda *s: (torch.rand(s, generator=g, device="cuda") * 2 - 1).half()   # noqa: E731
    x = rand(*((n, a["h"], a["w"], a["c"]) if how == "nhwc" else (n, a["c"], a["h"], a["w"])))
    w, b = rand(k, a["c"] // a["group"], a["r"], a["s"]), rand(k)
    y = torch.full((n, p, q, k) if how == "nhwc" else (n, k, p, q), float("nan"), dtype=torch.float16, device="cuda")
    hgc.conv_forward(d, x, w, b, y, False)
    yh = torch.full(tuple(y.shape), float("nan"), dtype=torch.float16).pin_memory()
    hgc.conv_forward_host(d, *(t.cpu().pin_memory() for t in (x, w, b)), yh, False)
    torch.cuda.synchronize()
    assert d.last_device_status() == hgc.HGC_OK
    assert bool(torch.isfinite(yh).all())
    different = int((yh.view(torch.int16) != y.cpu().view(torch.int16)).sum())
    assert different == 0, f"{name}: {different} of {yh.numel()} values differ"
    d.close()


@pytest.mark.parametrize("shift", [0, 2 * 64 * 224 * 224], ids=["y is x", "y begins two images into x"])
def test_host_forward_in_place(hgc, shift):
    """y may lie over x in host memory: all of x is read before any of y is written, however large the batch."""
    import torch
    a = params_dict(4, 64, 224, 224, 64, 3, 3, 1, 1)
    g = torch.Generator().manual_seed(5)
    d = hgc.ConvDesc(**a)
    d.ensure_workspace(host=True)
    rand = lambda *s: (torch.rand(s, generator=g) * 2 - 1).half().pin_memory()   # noqa: E731
    x, w, b = rand(4, 64, 224, 224), rand(64, 64, 3, 3), rand(64)
    y = torch.empty((4, 64, 224, 224), dtype=torch.float16).pin_memory()
    hgc.conv_forward_host(d, x, w, b, y, True)
    torch.cuda.synchronize()
    for _ in range(3):
        both = torch.zeros(x.numel() + shift, dtype=torch.float16).pin_memory()
        both[:x.numel()] = x.flatten()
        hgc.conv_forward_host(d, both.data_ptr(), w, b, both.data_ptr() + 2 * shift, True)
        torch.cuda.synchronize()
        got = both[shift:shift + y.numel()]
        assert torch.equal(got.view(torch.int16), y.flatten().view(torch.int16))
    d.close()


@pytest.mark.parametrize("a", [params_dict(1, 32, 20, 20, 32, 3, 3, 1, 1), params_dict(4, 64, 112, 112, 64, 3, 3, 1, 1)],
                         ids=["in one piece", "in chunks"])
def test_host_forward_forgets_registered_weights(hgc, oracle, a):
    """After a host call device weights are laid out anew on every call, however the host call went."""
    import torch
    rng = np.random.default_rng(21)
    x, w, b = workloads.random_layer_tensors(rng, a["n"], a["c"], a["h"], a["w"], a["k"], 3, 3, 1)
    w2 = workloads.random_layer_tensors(rng, a["n"], a["c"], a["h"], a["w"], a["k"], 3, 3, 1)[1]
    d = hgc.ConvDesc(**a)
    d.ensure_workspace(host=True)
    xd, wd, bd = to_dev(x), to_dev(w), to_dev(b)
    d.set_weights(wd)
    pin = lambda t: torch.from_numpy(t.view(np.int16)).pin_memory()   # noqa: E731
    hgc.conv_forward_host(d, pin(x), pin(w), pin(b), torch.empty(d.output_dims(), dtype=torch.float16).pin_memory(), True)
    wd.copy_(to_dev(w2))
    y = torch.empty(d.output_dims(), dtype=torch.float16, device="cuda")
    hgc.conv_forward(d, xd, wd, bd, y, True)
    torch.cuda.synchronize()
    check_close(to_host(y), oracle.conv_fast(oracle.ConvParams(**a), x, w2, b, True), what=str(a))
    d.close()


def test_host_forwards_of_other_streams_are_not_waited_for(hgc):
    """Calls on a stream that is held up, more of them than the library has internal streams, do not hold up a
    call on another stream.  Calls on more streams than that, all held up, come out right (they are not
    timed: so many streams share the device's hardware queues, which make them wait for one another)."""
    import time
    import torch
    a = params_dict(4, 64, 112, 112, 64, 3, 3, 1, 1)
    tensors = lambda: tuple(torch.rand(s).half().pin_memory() for s in   # noqa: E731
                            ((4, 64, 112, 112), (64, 64, 3, 3), (64,), (4, 64, 112, 112)))
    descs = [hgc.ConvDesc(**a) for _ in range(10)]
    sets = [tensors() for _ in descs]
    for d in descs:
        d.ensure_workspace(host=True)
    streams = [torch.cuda.Stream() for _ in descs]
    for d, t, s in zip(descs, sets, streams):   # (the first calls make streams)
        hgc.conv_forward_host(d, *t, True, s)
    torch.cuda.synchronize()
    want = sets[-1][3].clone()
    for held in ([streams[0]] * 9, streams[:9]):
        sets[-1][3].zero_()
        with torch.cuda.stream(streams[0]):
            torch.cuda._sleep(1_500_000_000)   # most of a second
        for s in set(held) - {streams[0]}:
            s.wait_stream(streams[0])
        for d, t, s in zip(descs, sets, held):
            hgc.conv_forward_host(d, *t, True, s)
        hgc.conv_forward_host(descs[-1], *sets[-1], True, streams[-1])
        t0 = time.time()
        streams[-1].synchronize()
        took = time.time() - t0
        if held[0] is held[1]:
            assert not streams[0].query(), "the held stream is still held"
            assert took < 0.2, took
        assert torch.equal(sets[-1][3], want)
        torch.cuda.synchronize()
        for d in descs:
            assert d.last_device_status() == hgc.HGC_OK
    for d in descs:
        d.close()


def test_host_forward_of_pageable_memory(hgc, oracle):
    import torch
    a = params_dict(5, 32, 149, 151, 32, 3, 3, 1, 1)
    rng = np.random.default_rng(12)
    x, w, b = workloads.random_layer_tensors(rng, a["n"], a["c"], a["h"], a["w"], a["k"], 3, 3, 1)
    d = hgc.ConvDesc(**a)
    d.ensure_workspace(host=True)
    y = np.full(d.output_dims(), np.nan, np.float16)
    hgc.conv_forward_host(d, x, w, b, y, True)
    torch.cuda.synchronize()
    check_close(y, oracle.conv_fast(oracle.ConvParams(**a), x, w, b, True), what="pageable")
    d.close()
