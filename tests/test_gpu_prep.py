"""Query preparation of the 16-bit screen around the batch sizes at which a warp per query
replaces a block per query: the same bits as the per-query scan on both sides."""
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


@pytest.mark.parametrize("d,L,k,line,rot", [(12, 2, 1, 128, False), (16, 2, 10, 512, False), (32, 2, 4, 1024, False),
                                            (50, 2, 1, 512, True), (64, 1, 5, 900, True), (64, 2, 5, 1024, True),
                                            (100, 1, 1, 900, True), (128, 2, 2, 1024, False)])
def test_both_sides_of_the_line(osann, d, L, k, line, rot):
    rng = np.random.default_rng(d + k)
    N = 40_003
    kw = {}
    if rot:
        q, _ = np.linalg.qr(rng.standard_normal((d, d)))
        kw = dict(rot=to_dev(q.astype(np.float32)))
    idx = osann.Index(to_dev(rng.standard_normal((N, d)).astype(np.float32)), L, **kw)
    Y = to_dev(rng.standard_normal((line, d)).astype(np.float32))
    ex = dict(query_src=to_dev(rng.integers(0, N, line)), grid_w=211, radius=3)
    for P, kw in ((3, {}), (60, ex)):
        for Q in (line - 1, line):
            kq = {n: (v[:Q] if n == "query_src" else v) for n, v in kw.items()}
            a, b = (idx.search(Y[:Q], P, k, path=p, **kq) for p in ("fp16", "plain"))
            assert np.array_equal(to_np(a[0]), to_np(b[0]))
            assert np.array_equal(to_np(a[1]).view(np.uint32), to_np(b[1]).view(np.uint32))
    assert idx.status() == 0
    idx.close()
