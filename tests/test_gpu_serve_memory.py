"""Small arrowheads solved in merged passes are charged the device memory of one
solved alone and the pass's tables: three lists of pairs of integers (24 bytes an
eigenpair), a descriptor (a page with its alignment).  The charge lasts until a
request is released, so that it bounds how many results a caller may keep."""
import pytest

from paper_1302_7203_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ae():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1302_7203_gb300 import arrowhead, build
    build.build()
    return arrowhead


@pytest.mark.parametrize("n, count", [(1000, 2), (1000, 8), (64, 40)])
def test_merged_requests_are_charged_as_single_ones(ae, n, count):
    to = lambda x: torch.as_tensor(x, device="cuda")
    d, z, a = W.uniform_arrow(n, seed=1)
    dt, zt = to(d), to(z)
    D, Z, A = W.graded_arrow(8000, seed=2)
    Dt, Zt = to(D), to(Z)
    torch.cuda.synchronize()
    # one slot: the small requests wait behind a large one, and go together
    srv = ae.Server(budget_bytes=64 << 30, max_inflight=1)
    tk = srv.submit(0, dt, zt, a)
    srv.wait(tk)
    alone = srv.stats()["bytes_in_use"]
    srv.release(tk)
    for _ in range(5):                       # (the large one may end before all are queued)
        before = srv.stats()["merged"]
        big = srv.submit(0, Dt, Zt, A, vectors=False)
        small = [srv.submit(0, dt, zt, a) for _ in range(count)]
        for tk in [big] + small:
            assert srv.wait(tk)[0] == ae.REQ_DONE
        srv.release(big)
        used, merged = srv.stats()["bytes_in_use"], srv.stats()["merged"] - before
        for tk in small:
            srv.release(tk)
        if merged == count:
            break
    assert merged == count
    assert alone > 0 and used <= count * (alone + 24 * n + 4096)
    assert srv.stats()["bytes_in_use"] == 0
    srv.close()
