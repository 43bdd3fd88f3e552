"""A search workspace sized for the largest batch serves every smaller one, although the
default path may screen every row at some of these sizes only (more scratch per query):
by the caller's own workspace, by a server without graphs (which searches at the batch's
real size), and by the library's allocation when the larger one fails."""
import numpy as np
import pytest

from helpers import to_dev, to_np
from test_gpu_failures import _FailingAllocator, _search_lib_ws

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def osann():
    import paper_1509_03453_gb300 as m
    from paper_1509_03453_gb300 import build
    build.build()
    m.load()
    return m


def same(a, b):
    assert np.array_equal(to_np(a[0]), to_np(b[0]))
    assert np.array_equal(to_np(a[1]).view(np.uint32), to_np(b[1]).view(np.uint32))


# N, d, L, P, k, largest batch: batches between two powers of two take the dense screen
# where both of these do not
@pytest.mark.parametrize("N,d,L,P,k,most", [(500_000, 128, 1, 8, 4, 256), (200_000, 100, 2, 96, 1, 2048)])
def test_smaller_batches_fit(osann, N, d, L, P, k, most):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(d)
    idx = osann.Index(torch.randn((N, d), generator=g, device="cuda"), L)
    Y = torch.randn((most, d), generator=g, device="cuda")
    ref = idx.search(Y, P, k, path="plain")
    dense = [q for q in range(most // 2 + 1, most + 1)
             if idx.workspace_size(q, P, k) not in [idx.workspace_size(q, P, k, p) for p in ("plain", "fp16")]]
    assert dense and dense[-1] < most
    sizes = sorted({most // 2 + 1, dense[0] - 1, dense[0], dense[len(dense) // 2], dense[-1], most})
    ws = torch.empty(idx.workspace_size(most, P, k), dtype=torch.uint8, device="cuda")
    for q in sizes:
        same(idx.search(Y[:q], P, k, workspace=ws), [t[:q] for t in ref])
    srv = osann.Server([idx], P=[P], k=[k], slots=1, max_batch=most, graphs=False)
    for q in sizes:
        t = srv.submit(0, Y[:q])
        srv.drain()
        same(srv.result(t), [r[:q] for r in ref])
    srv.close()
    assert idx.status() == 0
    idx.close()


def test_failed_dense_workspace_takes_the_smaller_form(osann):
    import torch
    from paper_1509_03453_gb300 import _lib
    L = _lib.load()
    rng = np.random.default_rng(2)
    idx = osann.Index(to_dev(rng.standard_normal((30_011, 32)).astype(np.float32)), 3)
    Y = to_dev(rng.standard_normal((1700, 32)).astype(np.float32))
    auto, plain, fp16 = (idx.workspace_size(1700, 1500, 1, p) for p in ("auto", "plain", "fp16"))
    assert auto not in (plain, fp16)
    with _FailingAllocator(L, fail_at=1) as a:
        rc, ids, d2 = _search_lib_ws(L, idx, Y, 1500, 1, "auto")
        torch.cuda.synchronize()
        assert rc == 0 and a.calls == 2 and a.live == {}
    same((ids, d2), idx.search(Y, 1500, 1, path="plain"))
    idx.close()


@pytest.mark.parametrize("graphs", [True, False])
def test_tuner_can_choose_the_dense_screen(osann, graphs):
    """Thin cones and k = 10: screening every row is several times faster than cone by cone,
    and only the default path does it; batches of all sizes give the per-query scan's bits."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    idx = osann.Index(torch.randn((200_000, 32), generator=g, device="cuda"), 3)
    Y = torch.randn((2048, 32), generator=g, device="cuda")
    P, k = 6000, 10
    srv = osann.Server([idx], P=[P], k=[k], slots=1, max_batch=2048, graphs=graphs)
    choices = srv.tune(reps=2, queries=[Y])
    assert choices[0][-1] == ("auto", 0, "default")
    ref = idx.search(Y, P, k, path="plain")
    for q in (2048, 1999, 1100, 300, 31, 1):
        t = srv.submit(0, Y[:q])
        srv.drain()
        same(srv.result(t), [r[:q] for r in ref])
    srv.close()
    idx.close()
