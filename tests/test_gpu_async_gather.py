"""GPU: the async gather (cp.async into per-warp rings, bulk stores), forced with info form=14, at
the edges of its units (128 or 256 chunks of 16 bytes), of the tiles (1024 chunks) and of the
rings (one thread block walking many units), for chunks per element of 1, 3, 4, 5 and 64, through
both sources (locality form), and with the destination in host memory (lane stores)."""
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

FORM = 1 << 14


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def two_ranks(n, s, seed, region=97):
    """Rank 0 sends n indexed elements to rank 1 and rank 1 n // 3 to rank 0 (one rank per node)."""
    rng = np.random.default_rng(seed)
    m = n // 3
    el = np.concatenate([rng.integers(0, region, n), rng.integers(0, region, m)])
    g = np.concatenate([el[:n], el[n:] + region])
    src, dst, cnt = ([0, 1], [1, 0], [n, m]) if m else ([0], [1], [n])
    order = np.argsort(dst)
    rg = np.concatenate([g[n:], g[:n]])
    return pt._assemble(f"two_{n}_{s}", 2, 1, src, dst, np.array(cnt), el, g, np.array(dst)[order],
                        np.array(src)[order], np.array(cnt)[order], rg, s, "bytes", np.full(2, region), {})


@pytest.mark.parametrize("cpe", [1, 3, 4, 5, 64])
@pytest.mark.parametrize("chunks", [1, 127, 128, 129, 257, 1023, 1024, 1025, 40001])
def test_edges(cpe, chunks):
    n = max(1, -(-chunks // cpe))
    p = two_ranks(n, 16 * cpe, chunks)
    x = pt.random_bytes(p.sendbuf_bytes, chunks + cpe)
    init = pt.random_bytes(p.recvbuf_bytes, 1)
    want = oracle.standard(p, x, init)
    for alg in ("standard", "locality"):
        for info in ("block=128", "block=256;max_ctas=1", "block=512;max_ctas=2", "graph=0"):
            got, ex = forward(p, x, alg, info="form=14;" + info, recv_init=init)
            assert ex.info()["copy_forms"] & FORM
            assert_bytes_equal(got, want, f"{p.name} {alg} {info}")


def test_host_destination_and_batch():
    p, q = two_ranks(5000, 48, 1), two_ranks(777, 64, 2)
    x, y = pt.random_bytes(p.sendbuf_bytes, 5), pt.random_bytes(q.sendbuf_bytes, 6)
    recv = torch.zeros(p.recvbuf_bytes, dtype=torch.uint8).pin_memory()
    ex = gbx.Exchange(p, dev_bytes(x), recv, info="form=14;block=256")
    ex.start()
    ex.wait()
    assert_bytes_equal(recv.numpy(), oracle.standard(p, x), "host destination")
    dev = torch.zeros(p.recvbuf_bytes, dtype=torch.uint8, device="cuda")
    ex.request.bind(None, dev)
    out = torch.zeros(q.recvbuf_bytes, dtype=torch.uint8, device="cuda")
    other = gbx.Exchange(q, dev_bytes(y), out, info="form=14;block=128")
    gbx.startall([ex.request, other.request])
    gbx.waitall([ex.request, other.request])
    assert_bytes_equal(dev.cpu().numpy(), oracle.standard(p, x), "batch, rebound to the device")
    assert_bytes_equal(out.cpu().numpy(), oracle.standard(q, y), "batch")
