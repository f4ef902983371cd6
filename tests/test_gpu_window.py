"""GPU: the window form of the flat gather (source windows and 16-bit indices through shared
memory, forced with info form=15), at the edges of its pieces (2048 slots) and windows (1024 or 2048
elements), on buffers whose ends and starts are not 16-byte aligned, through both sources
(locality form), rebound to unaligned and to host memory, and pooled in batches."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2309_07337_gb300 as gbx  # noqa: E402
from paper_2309_07337_gb300 import patterns as pt  # noqa: E402
from gpu_util import assert_bytes_equal, dev_bytes, forward  # noqa: E402

FORM = 1 << 15


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    gbx.device_status()


@pytest.fixture(autouse=True)
def status_clean():
    yield
    assert gbx.device_status() == 0


def ring(P, n, region, s, seed, deg=4, dtype="bytes"):
    """Every rank sends n ascending random elements of its region to each of the next deg ranks."""
    rng = np.random.default_rng(seed)
    deg = min(deg, P - 1)
    src = np.repeat(np.arange(P), deg)
    dst = (src + np.tile(np.arange(1, deg + 1), P)) % P
    o = np.lexsort((dst, src))
    src, dst = src[o], dst[o]
    el = np.sort(rng.integers(0, region, (P * deg, n)), axis=1)
    i = np.lexsort((src, dst))
    g = src[:, None] * region + el
    return pt._assemble(f"ring_{P}_{n}_{s}", P, 2, src, dst, np.full(P * deg, n), el.ravel(), g.ravel(), dst[i], src[i],
                        np.full(P * deg, n), g[i].ravel(), s, dtype, np.full(P, region), {})


# runs of 12 and 20 elements (windows of 2048 source elements) up to whole pieces (of 1024)
CASES = [(130, 4, 200, 129), (90, 9, 701, 89), (8, 2048, 1024, 4), (5, 4097, 1025, 4), (16, 1500, 999, 4),
         (3, 40000, 300, 2), (33, 700, 4099, 4), (40, 512, 2048, 4)]


@pytest.mark.parametrize("s", [4, 8])
@pytest.mark.parametrize("P,n,region,deg", CASES)
def test_edges(P, n, region, deg, s):
    p = ring(P, n, region, s, n + s, deg)
    assert oracle.validate(p) == 0
    x = pt.random_bytes(p.sendbuf_bytes, n)
    init = pt.random_bytes(p.recvbuf_bytes, 1)
    want = oracle.standard(p, x, init)
    for alg in ("standard", "locality"):
        for info in ("block=128", "block=256;max_ctas=1", "block=512;max_ctas=3;graph=0", "autotune=1"):
            got, ex = forward(p, x, alg, info="form=15;" + info, recv_init=init)
            if alg == "standard":   # (an aggregate read by few ranks may cost too much in whole windows)
                assert ex.info()["copy_forms"] & FORM, (p.name, alg, info)
            assert_bytes_equal(got, want, f"{p.name} {alg} {info}")


@pytest.mark.parametrize("s", [4, 8])
def test_rebind_and_batch(s):
    """Sources one element past a 16-byte boundary and in host memory (lane copies for ends or all of
    the windows), destinations in host memory, then a batch of two patterns in one launch."""
    p, q = ring(16, 1500, 999, s, 3), ring(5, 4097, 1025, s, 4)
    xs = [pt.random_bytes(p.sendbuf_bytes, k) for k in range(3)]
    y = pt.random_bytes(q.sendbuf_bytes, 9)
    recv = torch.zeros(p.recvbuf_bytes, dtype=torch.uint8, device="cuda")
    ex = gbx.Exchange(p, dev_bytes(xs[0]), recv, info="form=15;block=256")
    off = torch.zeros(p.sendbuf_bytes + s, dtype=torch.uint8, device="cuda")
    off[s:].copy_(dev_bytes(xs[1]))
    host = torch.from_numpy(xs[2].copy()).pin_memory()
    hout = torch.zeros(p.recvbuf_bytes, dtype=torch.uint8).pin_memory()
    qout = torch.zeros(q.recvbuf_bytes, dtype=torch.uint8, device="cuda")
    other = gbx.Exchange(q, dev_bytes(y), qout, info="form=15;block=256")
    assert ex.info()["copy_forms"] & other.info()["copy_forms"] & FORM
    for send, out, x in ((None, None, xs[0]), (off[s:], recv, xs[1]), (host, recv, xs[2]), (host, hout, xs[2]),
                         (off[s:], recv, xs[1])):
        if send is not None:
            ex.request.bind(send, out)
        out = recv if out is None else out
        for batch in (False, True):
            out.zero_()
            qout.zero_()
            if batch:
                gbx.startall([ex.request, other.request])
                gbx.waitall([ex.request, other.request])
                assert_bytes_equal(qout.cpu().numpy(), oracle.standard(q, y), "batch partner")
            else:
                ex.start()
                ex.wait()
            assert_bytes_equal(out.cpu().numpy(), oracle.standard(p, x), f"batch={batch}")


def _kernels(fn):
    """Names of the kernels that run in fn ([] where the profiler records none)."""
    from torch.profiler import ProfilerActivity, profile
    prof = profile(activities=[ProfilerActivity.CUDA])
    try:
        prof.start()
    except RuntimeError:     # (another profiler holds the device)
        fn()
        return []
    fn()
    torch.cuda.synchronize()
    prof.stop()
    return [e.name for e in prof.events() if "gbx_" in e.name]


@pytest.mark.parametrize("s", [4, 8])
@pytest.mark.parametrize("sizes", [("wide",), ("narrow",), ("wide", "narrow"), ("narrow", "other"), ("wide", "narrow", "other"),
                                   ("narrow", "other", "other")])
def test_batch_of_both_window_sizes(s, sizes):
    """One launch takes windows of 1024 and of 2048 elements, and an op tuned to another form where most
    elements were tuned to windows; where they were not, none runs in windows."""
    make = {"wide": (ring(130, 4, 200, s, 3, 129), 2048, "form=15"), "narrow": (ring(16, 1500, 999, s, 4), 1024, "form=15"),
            "other": (ring(12, 1500, 999, s, 5), 1024, "form=1")}
    items = []
    for k, w in enumerate(sizes):
        p, _, info = make[w]
        x = pt.random_bytes(p.sendbuf_bytes, k)
        out = torch.zeros(p.recvbuf_bytes, dtype=torch.uint8, device="cuda")
        ex = gbx.Exchange(p, dev_bytes(x), out, info=info)
        assert ex.info()["copy_forms"] == (FORM if w != "other" else 2)
        items.append((p, x, out, ex))
    reqs = [i[3].request for i in items]

    def start():
        gbx.startall(reqs)
        gbx.waitall(reqs)

    start()                                          # (builds and tunes the batch)
    for _, _, out, _ in items:
        out.zero_()
    names = _kernels(start)
    for p, x, out, _ in items:
        assert_bytes_equal(out.cpu().numpy(), oracle.standard(p, x), f"{p.name} {sizes}")
    tuned = sum(p.volume if w != "other" else -p.volume for w, (p, _, _, _) in zip(sizes, items))
    if names and tuned >= 0:
        assert len(names) == 1 and "gbx_window_kernel" in names[0], names
        assert f"<{s}, {2048 if 'wide' in sizes else 1024}," in names[0], names
    elif names:
        assert not any("gbx_window_kernel" in k for k in names), names


@pytest.mark.parametrize("s,off", [(4, 4), (4, 8), (4, 12), (8, 8)])
def test_sources_off_a_16_byte_boundary(s, off):
    """At init and after a bind: windows whose first and last 16-byte units are partly theirs, down to
    single elements, in the first and last window of the buffer, in both window sizes and a batch."""
    for P, n, region, deg in CASES:
        p = ring(P, n, region, s, n + s, deg)
        x = pt.random_bytes(p.sendbuf_bytes, n)
        want = oracle.standard(p, x)
        room = torch.zeros(p.sendbuf_bytes + 16, dtype=torch.uint8, device="cuda")
        src = room[off:off + p.sendbuf_bytes]
        src.copy_(dev_bytes(x))
        recv = torch.zeros(p.recvbuf_bytes, dtype=torch.uint8, device="cuda")
        late = torch.zeros_like(recv)
        ex = gbx.Exchange(p, src, recv, info="form=15")
        assert ex.info()["copy_forms"] & FORM
        other = gbx.Exchange(p, dev_bytes(x), late, info="form=15;block=128", dp=ex.dp, graph=ex.graph)
        other.request.bind(src, late)
        for start in (lambda: (ex.start(), other.start()), lambda: gbx.startall([ex.request, other.request])):
            recv.zero_()
            late.zero_()
            start()
            gbx.waitall([ex.request, other.request])
            assert_bytes_equal(recv.cpu().numpy(), want, f"{p.name} +{off}")
            assert_bytes_equal(late.cpu().numpy(), want, f"{p.name} +{off} bound later")


def test_time_off_a_16_byte_boundary():
    """Windows copied by the lanes alone took three times as long."""
    p = pt.spmv_halo_torch(1 << 19, 512, 32, 20, 5, "f64")
    n = p.sendbuf_bytes // 8
    x = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
    y = torch.zeros(p.recvbuf_bytes // 8, dtype=torch.float64, device="cuda")
    ex = gbx.Exchange(p, x[:n], y, info="form=15")
    assert ex.info()["copy_forms"] & FORM
    us = []
    for src in (x[:n], x[1:]):
        ex.request.bind(src, y)
        t = []
        for _ in range(12):
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            ev[0].record()
            for _ in range(10):
                ex.start()
                ex.request.wait_stream()
            ev[1].record()
            ev[1].synchronize()
            t.append(ev[0].elapsed_time(ev[1]) * 100)
        us.append(sorted(t)[6])
    assert us[1] <= 1.5 * us[0], us


@pytest.mark.parametrize("s", [4, 8])
def test_algorithmic_bytes(s):
    """Every window counts once, however many elements and pieces read it."""
    for (P, n, region, deg), we in ((CASES[4], 1024), (CASES[0], 2048)):
        p = ring(P, n, region, s, n, deg)
        _, ex = forward(p, pt.random_bytes(p.sendbuf_bytes, n), info="form=15")
        rank = np.repeat(np.arange(p.P), np.diff(p.send_slot_ptr))
        windows = len(np.unique((np.asarray(p.send_base)[rank] // s + p.send_idx) // we))
        low = windows * we * s + p.volume * (s + 2)
        assert ex.info()["copy_forms"] == FORM
        assert low < ex.info()["algo_bytes"] < low + p.volume * 9 // 4 + 32 * (windows + p.volume // 2048 + 1)


def _host(n, dtype=torch.uint8):
    return torch.zeros(n, dtype=dtype).pin_memory()


@pytest.mark.parametrize("info", ["", "graph=0", "max_ctas=5"])
@pytest.mark.parametrize("alg", ["standard", "locality"])
def test_host_destinations(alg, info):
    """Forward and reverse requests tuned on device memory and bound to host memory later, one after the
    other and with requests that stay on the device in one batch, then back on the device."""
    items, want = [], []
    for k, n in enumerate((60007, 50021, 41011)):
        p = pt.spmv_halo(n, 97, 11, 13, k, "f64")
        x, g = pt.spmv_x(p, k), np.random.default_rng(k).standard_normal(p.recvbuf_bytes // 8)
        send, grad = dev_bytes(x), torch.from_numpy(g).cuda()
        ex = gbx.Exchange(p, send, torch.zeros(p.recvbuf_bytes, dtype=torch.uint8, device="cuda"), alg, info="form=15;" + info)
        bw = gbx.backward_init(ex.request, grad, torch.zeros(p.sendbuf_bytes // 8, dtype=torch.float64, device="cuda"),
                               info="form=2;" + info)
        assert ex.info()["copy_forms"] & FORM and bw.info()["copy_forms"] & 1 << 13
        items += [(ex.request, send, p.recvbuf_bytes), (bw, grad, p.sendbuf_bytes)]
        want += [oracle.standard(p, x, np.full(p.recvbuf_bytes, 0x5A, np.uint8)),
                 oracle.backward(p, g, grad_send=np.full(p.sendbuf_bytes, 0x5A, np.uint8), form=int(alg == "locality"))]
    for host in ((True,) * 6, (True, False, False, True, False, True), (False,) * 6):
        outs = [_host(n) if h else torch.zeros(n, dtype=torch.uint8, device="cuda") for h, (_, _, n) in zip(host, items)]
        for (r, src, _), out in zip(items, outs):
            r.bind(src, out)
        reqs = [i[0] for i in items]
        for start in (lambda: [r.start() for r in reqs], lambda: gbx.startall(reqs)):
            for out in outs:
                out.fill_(0x5A)
            start()
            gbx.waitall(reqs)
            for k, (out, w) in enumerate(zip(outs, want)):
                assert_bytes_equal(out.cpu().numpy(), w, f"{alg} {info} {host} {k}")


def test_time_into_host_memory():
    """Window forms store runs and single values, which go to host memory one by one: bound or built
    there, a request takes no longer than in the stream forms (1.6 and 2 times as long before)."""
    p = pt.spmv_halo_torch(1 << 20, 1024, 32, 20, 2311, "f64")
    n, m = p.sendbuf_bytes // 8, p.recvbuf_bytes // 8
    x, y = (torch.zeros(k, dtype=torch.float64, device="cuda") for k in (n, m))
    hx, hy = _host(n, torch.float64), _host(m, torch.float64)
    late = gbx.Exchange(p, x, y, info="form=15")
    now = gbx.Exchange(p, x, hy, dp=late.dp, graph=late.graph)
    stream = gbx.Exchange(p, x, hy, info="stream=2", dp=late.dp, graph=late.graph)
    late.request.bind(x, hy)
    late_b, now_b, stream_b = (gbx.backward_init(late.request, y, b, info=i)
                               for b, i in ((x, ""), (hx, ""), (hx, "stream=2;single_split=0")))
    assert late_b.info()["copy_forms"] & 1 << 13
    late_b.bind(y, hx)
    us = []
    for r in (late.request, now.request, stream.request, late_b, now_b, stream_b):
        t = []
        for _ in range(9):
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            ev[0].record()
            r.start()
            r.wait_stream()
            ev[1].record()
            ev[1].synchronize()
            t.append(ev[0].elapsed_time(ev[1]) * 1e3)
        us.append(sorted(t)[4])
    assert max(us[:2]) <= 1.3 * us[2] and max(us[3:5]) <= 1.3 * us[5], us


@pytest.mark.parametrize("captured", ["aligned", "off", "host"])
def test_replays_after_a_rebind(captured):
    """graph=0: a caller's graph keeps the kernel that suited the buffers bound when it was captured, and
    reads the descriptors of those bound now: aligned, off a 16-byte boundary, into host memory."""
    import gc
    gc.collect()
    p = ring(16, 1500, 999, 8, 3)
    x = pt.random_bytes(p.sendbuf_bytes, 5)
    want = oracle.standard(p, x)
    room = torch.zeros(p.sendbuf_bytes + 8, dtype=torch.uint8, device="cuda")
    room[8:].copy_(dev_bytes(x))
    dev, host = torch.zeros(p.recvbuf_bytes, dtype=torch.uint8, device="cuda"), _host(p.recvbuf_bytes)
    bound = {"aligned": (dev_bytes(x), dev), "off": (room[8:], dev), "host": (room[8:], host)}
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    ex = gbx.Exchange(p, dev_bytes(x), dev, info="form=15;graph=0", stream=s)
    assert ex.info()["copy_forms"] & FORM
    ex.request.bind(*bound[captured])
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        ex.start()
        ex.request.wait_stream(s)
    for now in ("aligned", "off", "host", captured):
        ex.request.bind(*bound[now])
        out = bound[now][1]
        out.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            g.replay()
        torch.cuda.synchronize()
        assert_bytes_equal(out.cpu().numpy(), want, f"captured {captured}, bound {now}")


@pytest.mark.parametrize("what", ["forward", "backward"])
def test_too_little_memory_for_the_tables(what):
    """With just the memory that a request needs without window forms it is built without them."""
    p = ring(1000, 2000, 1900, 8, 3, 4, "f64")
    x, g = pt.random_bytes(p.sendbuf_bytes, 1), np.random.default_rng(2).standard_normal(p.recvbuf_bytes // 8)
    send, grad = dev_bytes(x), torch.from_numpy(g).cuda()
    recv = torch.zeros(p.recvbuf_bytes, dtype=torch.uint8, device="cuda")
    gx = torch.zeros(p.sendbuf_bytes // 8, dtype=torch.float64, device="cuda")
    fwd = gbx.Exchange(p, send, recv, info="stream=0;min_run=0")

    def make(info):
        if what == "forward":
            return gbx.Exchange(p, send, recv, info="min_run=0;" + info, dp=fwd.dp, graph=fwd.graph).request
        return gbx.backward_init(fwd.request, grad, gx, accumulate=True, info=info)

    bit = 1 << (15 if what == "forward" else 13)
    for info in ("", "stream=0", "form=15" if what == "forward" else "form=2"):   # (loads the kernels)
        r = make(info)
        assert info == "" or bool(r.info()["copy_forms"] & bit) == (info != "stream=0")
        r.free()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    block, keep = 16 << 20, []
    try:
        free = torch.cuda.mem_get_info()[0]
        keep = [torch.empty(free - (4 << 30), dtype=torch.uint8, device="cuda")]
        while torch.cuda.mem_get_info()[0] > 5 * block:
            keep.append(torch.empty(block, dtype=torch.uint8, device="cuda"))
        r = None
        while r is None:
            assert len(keep) > 1
            keep.pop()
            torch.cuda.empty_cache()
            try:
                r = make("stream=0")
            except gbx.GbxError as e:
                assert e.code == gbx.ERR_NOMEM
        r.free()
        r = make("")
    finally:
        del keep
        torch.cuda.empty_cache()
    assert not r.info()["copy_forms"] & bit
    gx.zero_()
    r.start()
    r.wait()
    if what == "forward":
        assert_bytes_equal(recv.cpu().numpy(), oracle.standard(p, x), what)
    else:
        assert_bytes_equal(gx.cpu().numpy(), oracle.backward(p, g, form=0), what)


def test_wait_gives_up():
    p = ring(16, 1500, 999, 8, 7)
    x = pt.random_bytes(p.sendbuf_bytes, 7)
    recv = torch.zeros(p.recvbuf_bytes, dtype=torch.uint8, device="cuda")
    ex = gbx.Exchange(p, dev_bytes(x), recv, info="form=15;autotune=0;wait_limit=0")
    assert ex.info()["copy_forms"] & FORM
    ex.start()
    with pytest.raises(gbx.GbxError) as e:
        ex.wait()
    assert e.value.code == gbx.ERR_DEVICE_WAIT
    assert gbx.device_status() == 1


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_spmv_halo(dtype):
    p = pt.spmv_halo(60007, 97, 11, 13, 5, dtype)
    x = pt.spmv_x(p, 3)
    want = oracle.standard(p, x)
    for alg in ("standard", "locality"):
        got, ex = forward(p, x, alg, info="form=15")
        assert ex.info()["copy_forms"] & FORM
        assert_bytes_equal(got, want, f"{dtype} {alg}")
