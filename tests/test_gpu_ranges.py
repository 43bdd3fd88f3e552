"""Vectors at the ends of what the 16-bit screen can scale: large norms and rows of very
different norms.  Linear search, the cone screen and the screen over all rows return
the bits of the per-query fp32 scan, which scales nothing."""
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


def check(osann, X, Y, L, P, k, dense):
    """dense: the default path screens every row (its workspace is neither the per-query
    scan's nor the cone screen's)."""
    idx = osann.Index(to_dev(X), L)
    Yd = to_dev(Y)
    sizes = {p: idx.workspace_size(len(Y), P, k, p) for p in ("auto", "plain", "fp16")}
    assert (sizes["auto"] not in (sizes["plain"], sizes["fp16"])) == dense
    ref = idx.search(Yd, P, k, path="plain")
    assert (to_np(ref[0]) >= 0).any()
    same(idx.search(Yd, P, k), ref)
    same(idx.search(Yd, P, k, path="fp16"), ref)
    same(idx.search(Yd, P, k, path="bf16"), ref)
    if L == 1:
        same(idx.bruteforce(Yd, k), idx.search(Yd, idx.NC, k, path="plain"))
    assert idx.status() == 0
    idx.close()


@pytest.mark.parametrize("d", [32, 100])
@pytest.mark.parametrize("sx,sy", [(1e13, 1e13), (1e14, 1e11), (1e15, 1e12), (1e17, 1e13), (5e17, 5e17)])
def test_large_norms(osann, d, sx, sy):
    rng = np.random.default_rng(3)
    X = rng.standard_normal((9000, d)).astype(np.float32) * np.float32(sx)
    Y = rng.standard_normal((1600, d)).astype(np.float32) * np.float32(sy)
    Y[7] = 0
    Y[9] *= np.float32(1e-20)
    check(osann, X, Y[:60], 1, 2 * d, 3, False)
    X = rng.standard_normal((30_011, d)).astype(np.float32) * np.float32(sx)
    check(osann, X, Y, *((3, 1500, 4) if d == 32 else (2, 2600, 4)), True)


@pytest.mark.parametrize("norm", [3e5, 1e6, 3e6, 1e8])
def test_one_row_of_large_norm(osann, norm):
    """The scale follows the largest norm; the others' squares are then around the fp16
    subnormal spacing, whose rounding the screen's bound has to cover."""
    rng = np.random.default_rng(4)
    X = rng.standard_normal((30_011, 32)).astype(np.float32)
    X[17] *= np.float32(norm / np.linalg.norm(X[17]))
    Y = rng.standard_normal((1600, 32)).astype(np.float32)
    Y[7] = 0
    check(osann, X, Y[:300], 1, 40, 2, False)
    check(osann, X, Y, 3, 1500, 2, True)


@pytest.mark.parametrize("scale", [1e-13, 3e-15, 1e-16])
def test_small_norms(osann, scale):
    rng = np.random.default_rng(6)
    X = rng.standard_normal((30_011, 32)).astype(np.float32) * np.float32(scale)
    Y = rng.standard_normal((1600, 32)).astype(np.float32) * np.float32(scale)
    check(osann, X, Y[:300], 1, 40, 2, False)
    check(osann, X, Y, 3, 1500, 2, True)


@pytest.mark.parametrize("d,L,N,k", [(64, 1, 11_028, 2), (32, 2, 40_011, 5), (100, 1, 20_003, 32), (16, 1, 20_003, 1)])
def test_uneven_norms(osann, d, L, N, k):
    """Norms over a factor of 100 and more: a candidate bounds the k-th best by its own norm
    (by the largest, most bounds say nothing and four times as many rows survive)."""
    rng = np.random.default_rng(d)
    X = (rng.standard_normal((N, d)) * np.exp(1.2 * rng.standard_normal((N, 1)))).astype(np.float32)
    Q = 8000 if k == 2 else 2000
    Y = (rng.standard_normal((Q, d)) * np.exp(1.2 * rng.standard_normal((Q, 1)))).astype(np.float32)
    idx = osann.Index(to_dev(X), L)
    Yd = to_dev(Y)
    ex = dict(query_src=to_dev(rng.integers(0, N, Q)), grid_w=141, radius=3)
    for P in (7, 120):
        idx.screen_stats()
        same(idx.search(Yd, P, k, path="fp16"), idx.search(Yd, P, k, path="plain"))
        if P == 120 and k == 2:
            assert idx.screen_stats()["survivors"] < 60 * Q
        same(idx.search(Yd, P, k, path="fp16", **ex), idx.search(Yd, P, k, path="plain", **ex))
        same(idx.search(Yd, P, k, path="bf16"), idx.search(Yd, P, k, path="plain"))
    assert idx.status() == 0
    idx.close()


@pytest.mark.parametrize("scale,outlier", [(1e14, 3e4), (1e16, 3e2), (3e9, 1.0), (4e9, 1.0), (1e18, 1.0)])
def test_bf16_near_the_limit(osann, scale, outlier):
    """bf16 columns hold fp32's range but the sums of the screen do not: norms up to fp32's
    limit, on both sides of the line from which they are scaled, and queries beyond."""
    rng = np.random.default_rng(9)
    X = rng.standard_normal((9000, 32)).astype(np.float32) * np.float32(scale)
    X[17] *= np.float32(outlier)
    Y = rng.standard_normal((200, 32)).astype(np.float32) * np.float32(scale)
    Y[3] *= np.float32(outlier)
    Y[5:8] *= np.float32(1e6)
    Y[7] = 0
    Y[9] *= np.float32(1e-20)
    check(osann, X, Y, 1, 40, 3, False)
