"""The per-query scan (warps reading rows straight from global memory), over thin
and fat cones: the same bits as the batched fp32 scan over padded widths, query counts
around its warps-per-query classes, k up to 32, budgets around its 32-cone
look-ups, exclusion, ties by id, missing results and mixed cone sizes."""
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


@pytest.mark.parametrize("d,L", [(10, 3), (16, 3), (24, 3), (50, 2), (64, 2), (100, 2), (128, 2), (200, 2),
                                 (10, 1), (32, 1), (64, 1), (128, 1)])
@pytest.mark.parametrize("Q", [1, 255, 256, 700, 2050])
def test_query_scan_matches_batched(osann, d, L, Q):
    rng = np.random.default_rng(d + Q)
    N = 4003
    X = rng.standard_normal((N, d)).astype(np.float32)
    X[:900] = X[rng.integers(0, 30, 900)]     # equal rows: ties by id, and a few full cones
    Y = rng.standard_normal((Q, d)).astype(np.float32)
    Y[: min(Q, 20)] = X[: min(Q, 20)]
    idx = osann.Index(to_dev(X), L)
    assert (N / idx.occupied() < 24) == (L > 1 or d == 128)
    Yd = to_dev(Y)
    kw = dict(query_src=to_dev(rng.integers(0, N, Q)), grid_w=61, radius=4)
    for P, k in ((1, 3), (31, 1), (33, 10), (400, 32)):
        for extra in ({}, kw):
            a = idx.search(Yd, P, k, path="plain", **extra)
            b = idx.search(Yd, P, k, path="batched", **extra)
            assert np.array_equal(to_np(a[0]), to_np(b[0]))
            assert np.array_equal(to_np(a[1]).view(np.uint32), to_np(b[1]).view(np.uint32))
    assert idx.status() == 0
    idx.close()


@pytest.mark.parametrize("L", [1, 2])
@pytest.mark.parametrize("Q", [2, 38, 39, 76, 77, 152, 153])
def test_query_scan_clusters_and_teams(osann, L, Q):
    """One to eight blocks per query (more than two per SM never), and budgets that
    leave teams of 1, 2, ... all of a query's warps per 32 probes."""
    rng = np.random.default_rng(L + Q)
    N, d = 6007, 48
    X = rng.standard_normal((N, d)).astype(np.float32)
    Y = rng.standard_normal((Q, d)).astype(np.float32)
    idx = osann.Index(to_dev(X), L)
    Yd = to_dev(Y)
    for P, k in ((5, 4), (64, 32), (65, 1), (515, 10), (4512, 17)):
        a = idx.search(Yd, P, k, path="plain")
        b = idx.search(Yd, P, k, path="batched")
        assert np.array_equal(to_np(a[0]), to_np(b[0]))
        assert np.array_equal(to_np(a[1]).view(np.uint32), to_np(b[1]).view(np.uint32))
    assert idx.status() == 0
    idx.close()


@pytest.mark.parametrize("L", [1, 2])
@pytest.mark.parametrize("n", [1, 37, 39, 300])
def test_overflowed_queries(osann, L, n):
    """n of 500 queries whose survivor lists overflow (2000 equal rows at their
    distance): the exact scan of the listed queries by clusters in turns."""
    rng = np.random.default_rng(L + n)
    d = 32
    X = rng.standard_normal((20_000, d)).astype(np.float32)
    X[5000:7000] = X[5000]
    Y = rng.standard_normal((500, d)).astype(np.float32)
    Y[::500 // n if n < 500 else 1][:n] = X[5000]
    idx = osann.Index(to_dev(X), L)
    Yd = to_dev(Y)
    idx.screen_stats()
    for P, k in ((60, 3), (60, 20), (idx.NC, 8)):
        a = idx.search(Yd, P, k, path="fp16")
        assert idx.screen_stats()["fallbacks"] >= n
        b = idx.search(Yd, P, k, path="batched")
        assert np.array_equal(to_np(a[0]), to_np(b[0]))
        assert np.array_equal(to_np(a[1]).view(np.uint32), to_np(b[1]).view(np.uint32))
    assert idx.status() == 0
    idx.close()
