"""The staged per-query scan, which runs while a wait budget is set: with a budget that no
wait reaches, the bits of the unstaged scan, on the plain path and as the exact rescan of
queries whose survivor lists overflow."""
import numpy as np
import pytest

from helpers import to_dev, to_np

pytestmark = pytest.mark.gpu

AMPLE = 4_000_000_000  # cycles: about two seconds


@pytest.fixture(scope="module")
def osann():
    import paper_1509_03453_gb300 as m
    from paper_1509_03453_gb300 import build
    build.build()
    m.load()
    return m


@pytest.mark.parametrize("d,L", [(16, 2), (50, 1), (128, 2), (200, 1)])
def test_staged_scan_matches(osann, d, L):
    from paper_1509_03453_gb300 import _lib
    lib = _lib.load()
    rng = np.random.default_rng(d)
    N, Q = 12_007, 301
    X = rng.standard_normal((N, d)).astype(np.float32)
    X[3000:5000] = X[3000]
    Y = rng.standard_normal((Q, d)).astype(np.float32)
    Y[::10] = X[3000]
    idx = osann.Index(to_dev(X), L)
    Yd = to_dev(Y)
    ex = dict(query_src=to_dev(rng.integers(0, N, Q)), grid_w=109, radius=4)
    runs = [(P, k, path, kw) for P, k in ((3, 1), (70, 5), (300, 32)) for kw in ({}, ex)
            for path in (("plain", "fp16") if d <= 128 else ("plain",))]
    ref = [idx.search(Yd, P, k, path="plain", **kw) for P, k, _, kw in runs]
    assert lib.osann_debug_wait_budget(AMPLE) == 0
    try:
        got = [idx.search(Yd, P, k, path=path, **kw) for P, k, path, kw in runs]
        assert idx.status() == 0
    finally:
        assert lib.osann_debug_wait_budget(0) == 0
    if d <= 128:
        assert idx.screen_stats()["fallbacks"] > 0
    for a, b in zip(got, ref):
        assert np.array_equal(to_np(a[0]), to_np(b[0]))
        assert np.array_equal(to_np(a[1]).view(np.uint32), to_np(b[1]).view(np.uint32))
    idx.close()
