"""GPU: the ways a start reaches the device.  A launch of one op carries its descriptor by value,
a start of several launches replays a graph on the buffers bound at init and launches them one by one
on others, graph=0 and pooled launches read descriptors in device memory (rewritten by a rebind, or
by the first batch after one).  Every way writes the oracle's bytes into the buffers bound at that
moment, whether the start is completed by the host, on the request's own stream or on another."""
import gc

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2309_07337_gb300 as gbx  # noqa: E402
from paper_2309_07337_gb300 import patterns as pt  # noqa: E402
from gpu_util import assert_bytes_equal, dev_bytes, payload  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.fixture(autouse=True)
def no_collection():
    """Requests of earlier tests that a collection frees inside a capture would invalidate it."""
    gc.collect()
    gc.disable()
    yield
    gc.enable()


def _complete(how, r, side):
    if how == "host":
        r.wait()
    elif how == "own":
        r.wait_stream()
    else:
        r.wait_stream(side)


@pytest.mark.parametrize("alg", ["standard", "locality"])
@pytest.mark.parametrize("info", ["", "graph=0"])
@pytest.mark.parametrize("how", ["host", "own", "other"])
def test_rebinds_between_starts(alg, info, how):
    p = pt.stencil((20, 15, 12), (4, 3, 3), ppn=5, comps=3)
    xs = [payload(p, 60 + k) for k in range(3)]
    want = [oracle.standard(p, x) for x in xs]
    sends = [dev_bytes(x) for x in xs]
    outs = [torch.zeros(p.recvbuf_bytes, dtype=torch.uint8, device="cuda") for _ in range(3)]
    ex = gbx.Exchange(p, sends[0], outs[0], alg, info=info)
    other = gbx.Exchange(p, sends[0], torch.empty_like(outs[0]), alg, dp=ex.dp, graph=ex.graph)
    side = torch.cuda.Stream()
    bound = 0
    for k in (0, 0, 1, 2, 0, 1):         # the first two starts run on the buffers bound at init
        if k != bound:
            ex.request.bind(sends[k], outs[k])
            bound = k
        outs[k].fill_(0xA5)
        ex.start()
        _complete(how, ex.request, side)
        with torch.cuda.stream(side if how == "other" else torch.cuda.current_stream()):
            got = outs[k].cpu().numpy()
        assert_bytes_equal(got, want[k], f"{alg} {info} {how} buffers {k}")
    # a batch built after the last rebind runs on those buffers, and again after one more
    for k in (1, 2):
        if k == 2:
            ex.request.bind(sends[k], outs[k])
        outs[k].fill_(0xA5)
        gbx.startall([ex.request, other.request])
        _complete(how, ex.request, side)
        other.request.wait()
        torch.cuda.synchronize()
        assert_bytes_equal(outs[k].cpu().numpy(), want[k], f"{alg} {info} {how} batch, buffers {k}")


@pytest.mark.parametrize("info", ["", "graph=0"])
def test_rebinds_between_batch_starts(info):
    """A batch of a forward and its backward exchange: launches of one op each, by value."""
    p = pt.stencil((24, 20, 16), (3, 2, 2), ppn=4, comps=8)
    xs = [payload(p, 70 + k) for k in range(2)]
    rng = np.random.default_rng(7)
    ws = [rng.standard_normal(p.recvbuf_bytes // 8) for _ in range(2)]
    sends, grads = [dev_bytes(x) for x in xs], [torch.from_numpy(w).cuda() for w in ws]
    halo = [torch.zeros(p.recvbuf_bytes, dtype=torch.uint8, device="cuda") for _ in range(2)]
    gx = [torch.zeros(p.sendbuf_bytes // 8, dtype=torch.float64, device="cuda") for _ in range(2)]
    ex = gbx.Exchange(p, sends[0], halo[0], "standard", info=info)
    bwd = gbx.backward_init(ex.request, grads[0], gx[0], info=info)
    for k, rebind in ((0, 0), (0, 0), (1, 1), (1, 0), (0, 1)):
        if rebind:
            ex.request.bind(sends[k], halo[k])
            bwd.bind(grads[k], gx[k])
        halo[k].fill_(0xA5)
        gx[k].zero_()
        gbx.startall([ex.request, bwd])
        gbx.waitall([ex.request, bwd])
        assert_bytes_equal(halo[k].cpu().numpy(), oracle.standard(p, xs[k], np.full(p.recvbuf_bytes, 0xA5, np.uint8)), "forward")
        assert_bytes_equal(gx[k].cpu().numpy(), oracle.backward(p, ws[k], form=0), "backward")


@pytest.mark.parametrize("comps", [1, 5, 2046, 2048, 2050, 6144])
@pytest.mark.parametrize("info", ["form=1", "form=5", "form=10", "form=14", "flat=0", "graph=0", "vec=8;form=5"])
def test_chunks_per_element(comps, info):
    """Elements of less, exactly and more than a tile (1024 chunks of 16 bytes; of 8 with vec=8)."""
    p = pt.stencil((8, 6, 4), (2, 2, 2), ppn=3, comps=comps)
    x = payload(p, 9)
    recv = torch.full((p.recvbuf_bytes,), 0xA5, dtype=torch.uint8, device="cuda")
    ex = gbx.Exchange(p, dev_bytes(x), recv, "standard", info=info)
    ex.start()
    ex.wait()
    want = oracle.standard(p, x, np.full(p.recvbuf_bytes, 0xA5, np.uint8))
    assert_bytes_equal(recv.cpu().numpy(), want, f"{comps} {info}")


@pytest.mark.parametrize("alg", ["standard", "locality"])
@pytest.mark.parametrize("info", ["", "graph=0"])
@pytest.mark.parametrize("other_stream", [False, True])
def test_exchange_stream(alg, info, other_stream):
    """One call on buffers of its own: the same bytes, the gaps zero or as they were, the request's own
    binding (and its graph) unchanged, errors as from the calls it stands for."""
    p = pt.random_pattern(91, P=24, dtype="f64", max_count=60)
    xs = [payload(p, k) for k in range(3)]
    own, out = (torch.full((p.recvbuf_bytes,), 0xA5, dtype=torch.uint8, device="cuda") for _ in range(2))
    ex = gbx.Exchange(p, dev_bytes(xs[0]), own, alg, info=info)
    side = torch.cuda.Stream()
    init = np.full(p.recvbuf_bytes, 0xA5, np.uint8)
    for k, zero in ((1, False), (2, True), (1, True)):
        send = dev_bytes(xs[k])
        out.fill_(0xA5)
        ex.request.exchange_stream(send, out, zero_dst=zero, stream=side if other_stream else None)
        with torch.cuda.stream(side if other_stream else torch.cuda.current_stream()):
            got = out.cpu().numpy()
        assert_bytes_equal(got, oracle.standard(p, xs[k], None if zero else init), f"{alg} {info} {k} {zero}")
    ex.start()
    with pytest.raises(gbx.GbxError) as e:
        ex.request.exchange_stream(send, out)
    assert e.value.code == gbx.ERR_ACTIVE
    ex.wait()
    assert_bytes_equal(own.cpu().numpy(), oracle.standard(p, xs[0], init), "own binding")


def test_start_under_capture_is_refused():
    """A graph=1 start launches with the buffers bound now, which a caller's graph would keep: it
    returns ERR_CUDA inside a stream capture and works again after it."""
    p = pt.config1()
    x = payload(p, 3)
    recv = torch.zeros(p.recvbuf_bytes, dtype=torch.uint8, device="cuda")
    s = torch.cuda.Stream()
    ex = gbx.Exchange(p, dev_bytes(x), recv, stream=s)
    s.synchronize()
    torch.cuda.synchronize()
    probe = torch.zeros(4, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        probe.add_(1)
        with pytest.raises(gbx.GbxError) as e:
            ex.start()
    assert e.value.code == gbx.ERR_CUDA
    ex.start()
    ex.wait()
    assert_bytes_equal(recv.cpu().numpy(), oracle.standard(p, x), "after the capture")


@pytest.mark.parametrize("alg", ["standard", "locality"])
@pytest.mark.parametrize("zero", [False, True])
@pytest.mark.parametrize("joins", [False, True])
def test_exchange_stream_under_capture_is_refused(alg, zero, joins):
    """graph=1, on the capturing stream or with the request's own stream outside the capture: nothing
    stays bound, nothing enters the caller's graph, the request's own stream joins no capture."""
    p = pt.random_pattern(92, P=24, dtype="f64", max_count=60)
    xs = [payload(p, k) for k in range(2)]
    init = np.full(p.recvbuf_bytes, 0xA5, np.uint8)
    own, other = (torch.full((p.recvbuf_bytes,), 0xA5, dtype=torch.uint8, device="cuda") for _ in range(2))
    s, own_stream = torch.cuda.Stream(), torch.cuda.Stream()
    send = dev_bytes(xs[1])
    ex = gbx.Exchange(p, dev_bytes(xs[0]), own, alg, stream=own_stream if joins else s)
    own.fill_(0xA5)
    torch.cuda.synchronize()
    probe = torch.zeros(4, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        probe.add_(1)
        with pytest.raises(gbx.GbxError) as e:
            ex.request.exchange_stream(send, other, zero_dst=zero, stream=s)
    assert e.value.code == gbx.ERR_CUDA
    g.replay()
    ex.start()
    ex.wait()
    torch.cuda.synchronize()
    assert probe.tolist() == [1.0] * 4
    assert_bytes_equal(other.cpu().numpy(), init, "the refused call's destination")
    assert_bytes_equal(own.cpu().numpy(), oracle.standard(p, xs[0], init), "the request's own buffers")


def _smallest_limit(make):
    """The smallest power of two as wait_limit with which five starts of a request succeed."""
    for k in range(23):
        r = make(1 << k)
        try:
            for _ in range(5):
                r.start()
                r.wait()
            return 1 << k
        except gbx.GbxError as e:
            assert e.code == gbx.ERR_DEVICE_WAIT
    raise AssertionError("no limit is enough")


def test_capped_launches_do_not_wait_for_each_other():
    """Two blocks per launch walk hundreds of tiles each: a launch that started beside its predecessor
    would fill its stages and then spend its bounded wait on the predecessor's whole run.  A
    limit well above what one launch needs by itself is enough for a chain of three."""
    p = pt.spmv_halo(200003, 64, 8, 12, 5, "f64")
    x, g = payload(p, 1), np.random.default_rng(2).standard_normal(p.recvbuf_bytes // 8)
    send, grad = dev_bytes(x), torch.from_numpy(g).cuda()
    recv = torch.zeros(p.recvbuf_bytes, dtype=torch.uint8, device="cuda")
    gx = torch.zeros(p.sendbuf_bytes // 8, dtype=torch.float64, device="cuda")
    dp, keep = gbx.DevicePattern(p), []

    def forward(alg, limit):
        keep.append(gbx.Exchange(p, send, recv, alg, info=f"stream=2;autotune=0;max_ctas=2;wait_limit={limit}", dp=dp))
        assert keep[-1].info()["copy_forms"] == 1 << 10
        return keep[-1].request

    def backward(alg, limit):
        r = gbx.backward_init(forward(alg, 1 << 22), grad, gx, info=f"stream=2;autotune=0;max_ctas=2;wait_limit={limit};"
                                                                    "single_split=0")
        assert r.info()["copy_forms"] & 1 << 12
        return r

    for make, out, want in ((forward, recv, oracle.standard(p, x)), (backward, gx, oracle.backward(p, g, form=1))):
        limit = 16 * _smallest_limit(lambda n: make("standard", n))
        r = make("locality", limit)
        for _ in range(5):
            out.zero_()
            r.start()
            r.wait()
            assert_bytes_equal(out.cpu().numpy(), want, f"{make.__name__} {limit}")
    gbx.device_status()


def _us(r, n=9):
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    t = []
    for _ in range(n + 2):
        ev[0].record()
        r.start()
        r.wait_stream()
        ev[1].record()
        ev[1].synchronize()
        t.append(ev[0].elapsed_time(ev[1]) * 1e3)
    return sorted(t[2:])[n // 2]


def test_capped_requests_have_shapes_of_their_own():
    """Shapes are tuned once per process and kind of op: the whole GPU's shapes of a form take up to
    twice the time of its best one on a few blocks, so a capped request is tuned under its cap."""
    p = pt.stencil((256,) * 3, (8,) * 3, 64, comps=8)
    x = torch.zeros(p.sendbuf_bytes, dtype=torch.uint8, device="cuda")
    y = torch.zeros(p.recvbuf_bytes, dtype=torch.uint8, device="cuda")
    ex = gbx.Exchange(p, x, y)
    dp, graph = ex.dp, ex.graph
    us = {}
    for form in ("", "form=1", "form=5", "form=14"):
        gbx.Exchange(p, x, y, info=form, dp=dp, graph=graph)
        us[form] = _us(gbx.Exchange(p, x, y, info="max_ctas=16;" + form, dp=dp, graph=graph).request)
    assert max(us[""], us["form=5"], us["form=14"]) <= 1.6 * min(us.values()), us
