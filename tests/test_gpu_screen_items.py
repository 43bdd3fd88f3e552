"""Work items of the tensor-core screen: an item is a cone and up to 256
queries in two query tiles, whose two halves of the kernel meet on every cone
tile.  Cones of one row up to many times the tile ring, query counts around
the tile and item sizes (items of one tile and of two mixed), every padded
width, exclusion on and off: the same bits as the per-query scan."""
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


def skewed_rows(d, sizes, seed):
    """Rows of L = 1 cones with the given sizes (cone j: component j // 2, sign j % 2)."""
    rng = np.random.default_rng(seed)
    rows = []
    for j, n in enumerate(sizes):
        x = 0.1 * rng.standard_normal((n, d))
        x[:, j // 2] = (1.0 if j % 2 else -1.0) * (1.0 + rng.random(n))
        rows.append(x)
    X = np.concatenate(rows).astype(np.float32)
    return X[rng.permutation(len(X))]


@pytest.mark.parametrize("d", [10, 32, 50, 64, 100, 128])
@pytest.mark.parametrize("Q", [1, 127, 129, 255, 300, 513])
def test_item_shapes(osann, d, Q):
    sizes = [1, 63, 64, 65, 127, 128, 129, 1, 2000, 3, 1500, 257, 1, 900, 0, 640, 511, 2, 1, 385]
    X = skewed_rows(d, sizes, d)
    rng = np.random.default_rng(100 + Q)
    Y = (0.5 * rng.standard_normal((Q, d))).astype(np.float32)
    idx = osann.Index(to_dev(X), 1)
    Yd = to_dev(Y)
    for k in (1, 7):
        for P in (3, 2 * d):
            a = idx.search(Yd, P, k, path="plain")
            for group in (0, 40):
                b = idx.search(Yd, P, k, path="fp16", group=group)
                assert np.array_equal(to_np(a[0]), to_np(b[0]))
                assert np.array_equal(to_np(a[1]).view(np.uint32), to_np(b[1]).view(np.uint32))
    src = to_dev(rng.integers(0, len(X), Q))
    kw = dict(query_src=src, grid_w=101, radius=5)
    a, b = (idx.search(Yd, 6, 3, path=p, **kw) for p in ("plain", "fp16"))
    assert np.array_equal(to_np(a[0]), to_np(b[0]))
    assert np.array_equal(to_np(a[1]).view(np.uint32), to_np(b[1]).view(np.uint32))
    assert idx.status() == 0
    idx.close()
