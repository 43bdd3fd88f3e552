"""The per-query scan where one cone is far larger than the others: a query that meets it is
left to a second launch, in which all its warps share the cone.  The same bits as the
batched fp32 scan over its classes of warps per query, and no batch held up by one warp."""
import numpy as np
import pytest

from helpers import to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def osann():
    import paper_1509_03453_gb300 as m
    from paper_1509_03453_gb300 import build
    build.build()
    m.load()
    return m


def skewed(N, big, d, seed):
    """big of the N rows share the cone of their first components."""
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((N, d)).astype(np.float32)
    X[:big] *= 0.2
    X[:big, :3] = [9.0, 7.0, 5.0] + 0.3 * np.abs(X[:big, :3])
    return rng, X


# thin cones (1.7 rows) and fat ones (25), the query counts of their classes
@pytest.mark.parametrize("N,d,L,Qs", [(30_000, 128, 2, (3, 40, 200, 400, 1000, 2100)),
                                      (30_000, 24, 3, (9, 300, 2100, 3700)),
                                      (220_000, 64, 2, (100, 700, 2100, 6200))])
def test_one_large_cone(osann, N, d, L, Qs):
    import torch
    rng, X = skewed(N, 20_000, d, d)
    idx = osann.Index(to_dev(X), L)
    assert idx.max_bucket >= 20_000
    for Q in Qs:
        Y = rng.standard_normal((Q, d)).astype(np.float32)
        Y[1::7] = X[rng.integers(0, 20_000, len(Y[1::7]))] + np.float32(0.05)
        Yd = to_dev(Y)
        ex = dict(query_src=to_dev(rng.integers(0, N, Q)), grid_w=61, radius=4)
        for P, k, kw in ((5, 3, {}), (64, 10, ex), (300, 32, {})):
            ref = idx.search(Yd, P, k, path="batched", **kw)
            ids, d2 = idx.search(Yd, P, k, path="plain", **kw)
            assert torch.equal(ids, ref[0]) and torch.equal(d2.view(torch.int32), ref[1].view(torch.int32))
    # its largest cone not read yet: an asynchronous build
    late, ids, d2 = osann.build_search(to_dev(X), L, Yd, 300, 32, path="plain", sync=False)
    ref = idx.search(Yd, 300, 32, path="batched")
    for _ in range(2):
        assert torch.equal(ids, ref[0]) and torch.equal(d2.view(torch.int32), ref[1].view(torch.int32))
        ids, d2 = late.search(Yd, 300, 32, path="plain")
    late.close()
    assert idx.status() == 0
    idx.close()


def test_many_large_cones(osann):
    """Nothing but large cones: eight of 11 000 rows, the other rows thin."""
    import torch
    rng = np.random.default_rng(8)
    N, d, P = 100_000, 24, 5000
    X = rng.standard_normal((N, d)).astype(np.float32)
    X[:90_000] = np.sign(X[:90_000])                           # ties: one set of components,
    X[:90_000] *= (1.0 + 0.01 * rng.random((90_000, 1))).astype(np.float32)  # eight signs
    idx = osann.Index(to_dev(X), 3)
    Y = to_dev(np.sign(rng.standard_normal((30, d))).astype(np.float32))
    for k in (1, 10):
        ref = idx.search(Y, P, k, path="batched")
        ids, d2 = idx.search(Y, P, k, path="plain")
        assert torch.equal(ids, ref[0]) and torch.equal(d2.view(torch.int32), ref[1].view(torch.int32))
    assert idx.status() == 0
    idx.close()


def test_one_warp_does_not_hold_a_batch(osann):
    """8 of 3000 queries have a cone of 400 000 rows of 512 bytes among their thin ones: a
    warp alone took 98 ms for it (the staged scan 12 ms)."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    X = torch.randn((1_000_000, 128), generator=g, device="cuda")
    X[:400_000] *= 0.2
    X[:400_000, :3] = 5 + 0.3 * X[:400_000, :3].abs()
    idx = osann.Index(X, 3)
    del X
    for Q, P in ((300, 400), (3000, 300), (4000, 64)):
        Y = torch.randn((Q, 128), generator=g, device="cuda")
        Y[:8] = torch.cat([5 + 0.1 * torch.rand((8, 3), generator=g, device="cuda"), 0.2 * Y[:8, 3:]], 1)
        times = []
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            idx.search(Y, P, 4, path="plain")
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        assert min(times) < 25.0, (Q, times)
    idx.close()


def test_screen_over_a_large_cone(osann):
    """k > 4 on the 16-bit screen, one cone of 6000 rows among thin ones: a long seed and
    items of one query tile (by the average cone a tenth of a seed, and 5 ms)."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(1241)
    X = torch.randn((31_318, 128), generator=g, device="cuda")
    X[:6263] *= 0.2
    X[:6263, :3] = 5 + 0.3 * X[:6263, :3].abs()
    Y = torch.randn((4334, 128), generator=g, device="cuda")
    Y[:433] = X[:433]
    idx = osann.Index(X, 2)
    for P, k in ((122, 32), (30, 5)):
        ref = idx.search(Y, P, k, path="plain")
        times = []
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            ids, d2 = idx.search(Y, P, k, path="fp16")
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        assert torch.equal(ids, ref[0]) and torch.equal(d2.view(torch.int32), ref[1].view(torch.int32))
        if k == 32:
            assert min(times) < 3.6, times
    assert idx.status() == 0
    idx.close()
