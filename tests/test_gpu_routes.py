"""Which route the default path takes, told by its workspace size (the dense screen's is
neither the per-query scan's nor the cone screen's), where results alone would not show
that another ran; the results are compared all the same."""
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


def route(idx, Q, P, k):
    auto, plain, fp16 = (idx.workspace_size(Q, P, k, p) for p in ("auto", "plain", "fp16"))
    return "plain" if auto == plain else "fp16" if auto == fp16 else "dense"


def test_dense_route_with_overflowing_lists(osann):
    rng = np.random.default_rng(11)
    base = np.round(3 * rng.standard_normal((300, 32))).astype(np.float32)
    X = rng.standard_normal((30_000, 32)).astype(np.float32)
    X[:20_000] = base[rng.integers(0, 6, 20_000)]   # thousands of equal rows: lists overflow
    Y = to_dev(np.concatenate([X[:300], rng.standard_normal((1400, 32))]).astype(np.float32))
    idx = osann.Index(to_dev(X), 3)
    assert route(idx, 1700, 1500, 4) == "dense"
    idx.screen_stats()
    got = idx.search(Y, 1500, 4)
    assert idx.screen_stats()["fallbacks"] > 0
    same(got, idx.search(Y, 1500, 4, path="plain"))
    idx.close()


@pytest.mark.parametrize("k,want", [(2, "fp16"), (5, "fp16"), (16, "dense"), (32, "dense")])
def test_many_candidates(osann, k, want):
    rng = np.random.default_rng(k)
    N, d, Q, P = 400_003, 32, 301, 40
    idx = osann.Index(to_dev(rng.standard_normal((N, d)).astype(np.float32)), 1)
    Y = to_dev(rng.standard_normal((Q, d)).astype(np.float32))
    assert route(idx, Q, P, k) == want
    same(idx.search(Y, P, k), idx.search(Y, P, k, path="plain"))
    assert idx.status() == 0
    idx.close()


def test_few_rows_per_query_take_the_scan(osann):
    rng = np.random.default_rng(1)
    idx = osann.Index(to_dev(rng.standard_normal((30_000, 64)).astype(np.float32)), 3)
    assert route(idx, 500, 20, 4) == "plain" and route(idx, 70_000, 20, 4) != "dense"
    idx.close()


@pytest.mark.parametrize("N,d,L,Q,P,k,sigma", [(13_000, 64, 3, 4000, 330, 5, 1.2), (75_000, 128, 3, 5000, 300, 1, 0.0)])
def test_scan_where_it_beats_both_screens(osann, N, d, L, Q, P, k, sigma):
    """Few candidates per query over thin cones: neither screen runs (no survivors counted),
    although enough queries share a cone for one."""
    rng = np.random.default_rng(d)
    X = rng.standard_normal((N, d)) * np.exp(sigma * rng.standard_normal((N, 1)))
    Y = rng.standard_normal((Q, d)) * np.exp(sigma * rng.standard_normal((Q, 1)))
    if sigma == 0.0:
        X, Y = np.abs(X), np.abs(Y)
    idx = osann.Index(to_dev(X.astype(np.float32)), L)
    Y = to_dev(Y.astype(np.float32))
    assert Q * P / idx.occupied() > 8
    idx.screen_stats()
    got = idx.search(Y, P, k)
    assert idx.screen_stats()["survivors"] == 0
    same(got, idx.search(Y, P, k, path="fp16"))
    for q in (1, 777):  # and a workspace for all of them serves fewer
        import torch
        ws = torch.empty(idx.workspace_size(Q, P, k), dtype=torch.uint8, device="cuda")
        same(idx.search(Y[:q], P, k, workspace=ws), [t[:q] for t in got])
    idx.close()
