"""Linear search through the tensor-core screen (every row against every query in
phases, the survivors evaluated exactly): the same bits as the per-query scan of
all cones, which evaluates every row in fp32, over widths, odd sizes, query
counts around the tile sizes, k, exclusion, equal rows (survivor lists that
overflow) and vectors out of the 16-bit range."""
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


def same(a, b):
    assert np.array_equal(to_np(a[0]), to_np(b[0]))
    assert np.array_equal(to_np(a[1]).view(np.uint32), to_np(b[1]).view(np.uint32))


def check(osann, X, Y, ks, **kw):
    idx = osann.Index(to_dev(X), 1)
    Yd = to_dev(Y)
    for k in ks:
        same(idx.bruteforce(Yd, k, **kw), idx.search(Yd, idx.NC, k, path="plain", **kw))
    assert idx.status() == 0
    idx.close()


@pytest.mark.parametrize("d", [10, 32, 50, 64, 100, 128])
@pytest.mark.parametrize("N,Q", [(8192, 1), (8191, 3), (20_011, 129), (70_003, 300), (300_007, 77)])
def test_linear_matches_scan(osann, d, N, Q):
    rng = np.random.default_rng(d * 7 + Q)
    X = rng.standard_normal((N, d)).astype(np.float32)
    Y = rng.standard_normal((Q, d)).astype(np.float32)
    check(osann, X, Y, (1, 5, 32))


@pytest.mark.parametrize("d", [24, 128])
def test_linear_equal_rows_and_exclusion(osann, d):
    rng = np.random.default_rng(d)
    base = np.round(2 * rng.standard_normal((40, d))).astype(np.float32)
    X = base[rng.integers(0, 40, 30_000)]          # 750 copies of each row: ties by id
    X[:12_000] = X[0]                                # and a list that overflows
    Y = np.concatenate([X[:5], X[-60:], base[:20] + 0.25]).astype(np.float32)
    check(osann, X, Y, (1, 10))
    src = to_dev(rng.integers(0, len(X), len(Y)))
    Z = rng.standard_normal((30_000, d)).astype(np.float32)
    check(osann, Z, Z[:85] + 0.01 * rng.standard_normal((85, d)).astype(np.float32), (4,), query_src=src, grid_w=173,
          radius=8)


def test_linear_ranges(osann):
    rng = np.random.default_rng(5)
    X = rng.standard_normal((9000, 32)).astype(np.float32)
    Y = rng.standard_normal((40, 32)).astype(np.float32)
    Y[3] *= 1e9      # out of the scaled 16-bit range
    Y[7] = 0
    Y[9] *= 1e-20
    check(osann, X, Y, (3,))
    check(osann, X * 1e-12, Y * 1e-12, (3,))
    check(osann, X * 1e12, Y[10:] * 1e12, (3,))
    check(osann, np.zeros((9000, 32), np.float32), Y, (2,))
    big = X.copy()
    big[17] = 1e19   # its squared norm passes the fp32 range
    check(osann, big, Y, (3,))


# L, d, P (up to past all unflipped profiles), Q: sizes at which the automatic
# path screens every row and keeps the survivors of probed cones
@pytest.mark.parametrize("L,d,m,P,Q", [(3, 32, 0, 1500, 1700), (3, 32, 0, 6000, 700), (2, 100, 0, 2600, 1501),
                                       (2, 100, 0, 9000, 513), (4, 20, 0, 9000, 700), (1, 128, 0, 140, 4500),
                                       (3, 64, 40, 11_000, 600)])
def test_thin_cones_match_scan(osann, L, d, m, P, Q):
    rng = np.random.default_rng(L * 1000 + d + P)
    N = 30_011 if L > 1 else 9_001
    X = rng.standard_normal((N, d)).astype(np.float32)
    X[:, : d // 2] = np.abs(X[:, : d // 2])
    Y = rng.standard_normal((Q, d)).astype(np.float32)
    Y[5] *= 1e9          # left to the exact scan
    Y[6] = 0
    kw = {}
    if m:
        q, _ = np.linalg.qr(rng.standard_normal((d, d)))
        kw = dict(rot=to_dev(q[:m].astype(np.float32)), rot_offset=to_dev(q[:m].sum(1).astype(np.float32)))
    idx = osann.Index(to_dev(X), L, **kw)
    Yd = to_dev(Y)
    src = to_dev(rng.integers(0, N, Q))
    for k in (1, 10):
        if L > 1:  # the dense route: neither the per-query scan nor the cone-major list
            sizes = {p: idx.workspace_size(Q, P, k, p) for p in ("auto", "plain", "fp16")}
            assert sizes["auto"] not in (sizes["plain"], sizes["fp16"])
        same(idx.search(Yd, P, k), idx.search(Yd, P, k, path="plain"))
        ex = dict(query_src=src, grid_w=173, radius=6)
        same(idx.search(Yd, P, k, **ex), idx.search(Yd, P, k, path="plain", **ex))
    assert idx.status() == 0
    idx.close()


def test_thin_cones_overflow(osann):
    rng = np.random.default_rng(11)
    base = np.round(3 * rng.standard_normal((300, 32))).astype(np.float32)
    X = rng.standard_normal((30_000, 32)).astype(np.float32)
    X[:20_000] = base[rng.integers(0, 6, 20_000)]   # thousands of equal rows: lists overflow
    Y = np.concatenate([X[:300], rng.standard_normal((1400, 32))]).astype(np.float32)
    idx = osann.Index(to_dev(X), 3)
    Yd = to_dev(Y)
    idx.screen_stats()
    same(idx.search(Yd, 1500, 4), idx.search(Yd, 1500, 4, path="plain"))
    assert idx.status() == 0
    idx.close()


@pytest.mark.parametrize("k", [2, 5, 16, 32])
def test_many_candidates_match_scan(osann, k):
    """Fat cones, k > 1 and so many candidates that survivor lists would overflow cone
    by cone: the default path screens every row; the same bits as the per-query scan."""
    rng = np.random.default_rng(k)
    N, d, Q, P = 400_003, 32, 301, 40
    X = rng.standard_normal((N, d)).astype(np.float32)
    Y = rng.standard_normal((Q, d)).astype(np.float32)
    idx = osann.Index(to_dev(X), 1)
    Yd = to_dev(Y)
    same(idx.search(Yd, P, k, path="fp16"), idx.search(Yd, P, k, path="plain"))
    over = idx.screen_stats()["fallbacks"]
    kw = dict(query_src=to_dev(rng.integers(0, N, Q)), grid_w=700, radius=5)
    for extra in ({}, kw):
        same(idx.search(Yd, P, k, **extra), idx.search(Yd, P, k, path="plain", **extra))
    if k == 32:
        assert over > 0 and idx.screen_stats()["fallbacks"] == 0
    assert idx.status() == 0
    idx.close()
