"""Performance cases: the calls that users of this package make, at the sizes of its
benchmark, tests and named workloads, and a generator of more cases of the same ranges.

A case is a dict of plain values:

    kind   "search"   Index.search on a prebuilt index
           "excl"     Index.search with the self/near exclusion of the patch workload
           "rebuild"  Index.rebuild_search: index rebuilt in place, then searched
           "build"    Index(data, L) and its exported table
           "linear"   Index.bruteforce: exact linear search (ground truth, recall checks)
           "multi"    MultiIndex.search over R bases
           "serve"    one closed-loop window of requests through the tuned Server
    data   "gauss" (iid N(0,1)), "desc" (the descriptor recipe), "patch" (8 x 8 patches of a 1/f^2 image)
    N, d   rows and components; L: components hashed; axes: PCA axes that key the rows (0: none)
    Q, P, k   queries, cones visited, neighbours

`exact` restates the search in 64-bit torch arithmetic: magnitude orders, the neighbouring-cone
list by plain enumeration, and the k smallest distances over the points of the listed cones.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

import paper_1509_03453_gb300 as osann

PATCH, RADIUS = 8, 8  # patch side; exclusion within Chebyshev distance 8

# the three resident indexes of the serving benchmark, their budgets and requests of 1..4096 queries
SERVE = (dict(data="gauss", N=1_000_000, d=32, L=2, axes=0, P=256),
         dict(data="gauss", N=4_000_000, d=64, L=2, axes=0, P=3072),
         dict(data="desc", N=2_000_000, d=128, L=3, axes=16, P=2048))
SERVE_POOL = 8192


def _case(name, kind, data, N, d, L, Q, P, k, axes=0, R=1):
    return dict(name=name, kind=kind, data=data, N=N, d=d, L=L, Q=Q, P=P, k=k, axes=axes, R=R)


def listed():
    return [
        # one query at a time against a resident index (an interactive caller): latency and launches
        _case("one_query_gauss32", "search", "gauss", 1_000_000, 32, 2, 1, 256, 1),
        # a small request on the largest resident index
        _case("small_batch_gauss64", "search", "gauss", 4_000_000, 64, 2, 77, 3072, 1),
        # a full serving batch on the d = 64 index
        _case("batch_gauss64", "search", "gauss", 4_000_000, 64, 2, 4096, 3072, 1),
        # a full serving batch on the descriptor index keyed on 16 PCA axes (Sec. 4-B)
        _case("batch_desc128_pca", "search", "desc", 2_000_000, 128, 3, 4096, 2048, 1, axes=16),
        # k = 10 descriptor search with one basis at recall@1 >= 0.9: thin cones, many of them
        _case("desc128_k10", "search", "desc", 2_000_000, 128, 3, 10_000, 12_288, 10),
        # the same index at a small budget: few rows per query (the per-query scan)
        _case("desc128_thin", "search", "desc", 2_000_000, 128, 3, 10_000, 128, 10),
        # copy-move search (Sec. 4-C): all patches of an image, near matches excluded
        _case("patch64_excl", "excl", "patch", 0, 64, 3, 20_000, 64, 4),
        # data that change every step: index rebuilt in place and searched
        _case("rebuild_search_gauss32", "rebuild", "gauss", 1_000_000, 32, 2, 10_000, 224, 1),
        # loading an index
        _case("build_gauss64", "build", "gauss", 4_000_000, 64, 2, 0, 0, 0),
        # ground truth for a recall check
        _case("linear_desc128_k10", "linear", "desc", 2_000_000, 128, 3, 1000, 0, 10),
        # several bases (Sec. 3-D) on vectors of an odd width, k between the template sizes
        _case("multibasis_d100", "multi", "gauss", 500_003, 100, 2, 3001, 96, 5, R=2),
        # the serving step: 1000 requests of 1..4096 queries over three resident indexes
        _case("serving_window", "serve", "mixed", 0, 0, 0, 1000, 0, 1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "search", "pca", "desc", "excl", "rebuild", "build", "linear", "multi",
                       "serve"])
    k = rng.choice([1, 1, 1, 2, 4, 5, 10, 16, 32])
    if kind == "serve":
        return _unnamed("serve", "mixed", 0, 0, 0, _log_int(rng, 20, 1000), 0, 1)
    if kind == "excl":
        return _unnamed("excl", "patch", 0, 64, 3, _log_int(rng, 100, 20_000), _log_int(rng, 4, 64), min(k, 10))
    if kind == "desc":
        Q = _log_int(rng, 1, 10_000)
        return _unnamed("search", "desc", _log_int(rng, 50_000, 2_000_000), 128, 3, Q, _log_int(rng, 8, 12_288), k)
    if kind == "pca":
        return _unnamed("search", "desc", _log_int(rng, 50_000, 2_000_000), 128, 3, _log_int(rng, 1, 4096),
                        _log_int(rng, 64, 2048), k, axes=16)
    d = rng.choice([16, 24, 32, 48, 50, 64, 96, 100, 128, rng.randint(10, 128)])
    N = _log_int(rng, 20_000, 4_000_000 * 64 // max(64, d))
    if kind == "build":
        return _unnamed("build", "gauss", N, d, rng.choice([1, 2, 2, 3]), 0, 0, 0)
    if kind == "linear":
        return _unnamed("linear", "gauss", min(N, 2_000_000), d, 2, _log_int(rng, 1, 1000), 0, min(k, 10))
    Q = _log_int(rng, 1, 10_000)
    nc = 4 * math.comb(d, 2)
    # a budget of about 1/10 to 4/10 of the cones (recall on iid data), at most 3072, or far below
    P = min(nc, 3072, max(1, int(nc * rng.choice([0.01, 0.11, 0.2, 0.38]))))
    while Q * P * (N / nc) * d > 4.0e11:  # no more than a full batch on the largest index
        Q = max(1, Q // 2)
    if kind == "multi":
        return _unnamed("multi", "gauss", min(N, 1_000_000), d, 2, max(1, Q // 2), max(1, P // 2), k, R=2)
    return _unnamed(kind, "gauss", N, d, 2, Q, P, k)


def _unnamed(*a, **kw):
    c = _case("", *a, **kw)
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs

def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1_000_003 + salt) % (1 << 62))
    return g


def _desc_rows(n, d, g):
    """Descriptor-like rows: Gamma(0.5, scale 20) (= 10 Z^2) clipped to [0, 255], L2-normalised to
    512, rounded half to even."""
    out = torch.empty((n, d), device="cuda")
    for s in range(0, n, 1 << 19):
        z = torch.randn((min(n - s, 1 << 19), d), generator=g, device="cuda")
        z = (10.0 * z * z).clamp_(0.0, 255.0)
        nrm = z.norm(dim=1, keepdim=True)
        out[s:s + z.shape[0]] = torch.round(z * torch.where(nrm > 0, 512.0 / nrm, torch.zeros_like(nrm)))
    return out


def _patches(seed):
    """All 8 x 8 patches (mean removed) of a 1024 x 1024 image with a 1/f^2 power spectrum plus
    uniform noise, row-major by position; grid_w positions per row."""
    n = 1024
    rng = np.random.default_rng(seed)
    spec = np.fft.fft2(rng.standard_normal((n, n)))
    f = np.hypot(np.fft.fftfreq(n)[:, None], np.fft.fftfreq(n)[None, :])
    f[0, 0] = np.inf
    img = np.real(np.fft.ifft2(spec / f))
    img = (img - img.min()) / (img.max() - img.min())
    img = (img + rng.uniform(-0.0346, 0.0346, img.shape)).astype(np.float32)
    t = torch.from_numpy(img).cuda()
    x = t.unfold(0, PATCH, 1).unfold(1, PATCH, 1).reshape(-1, PATCH * PATCH)
    return (x - x.mean(1, keepdim=True)).contiguous(), n - PATCH + 1


def _data(c, seed):
    """Rows and queries of one index (exclusion cases: also the sources and the grid width)."""
    if c["data"] == "patch":
        X, w = _patches(seed)
        src = torch.randperm(X.shape[0], generator=_gen(seed, 3), device="cuda")[:c["Q"]].sort().values
        return X, X[src].contiguous(), src, w
    g = _gen(seed, 1)
    if c["data"] == "desc":
        X = _desc_rows(c["N"], c["d"], g)
        Y = _desc_rows(c["Q"], c["d"], _gen(seed, 2))
        Y = (Y + 2.0 * torch.randn(Y.shape, generator=_gen(seed, 4), device="cuda")).clamp_(0.0, 512.0)
    else:
        X = torch.randn((c["N"], c["d"]), generator=g, device="cuda")
        Y = torch.randn((c["Q"], c["d"]), generator=_gen(seed, 2), device="cuda")
    return X, Y, None, 0


def _axes(X, m):
    """m principal axes of a sample of the rows (fp64, largest entry positive) and the projected mean."""
    S = X[:16384].cpu().numpy().astype(np.float64)
    mu = S.mean(0)
    w, V = np.linalg.eigh((S - mu).T @ (S - mu))
    A = V[:, np.argsort(w)[::-1][:m]].T
    A = A * np.sign(A[np.arange(m), np.abs(A).argmax(1)])[:, None]
    A = A.astype(np.float32)
    return torch.from_numpy(A).cuda(), torch.from_numpy((A.astype(np.float64) @ mu).astype(np.float32)).cuda()


def _bases(c, seed):
    """R orthonormal bases: the identity, then random rotations."""
    rng = np.random.default_rng(seed + 17)
    out = [np.eye(c["d"], dtype=np.float32)]
    for _ in range(1, c["R"]):
        q, t = np.linalg.qr(rng.standard_normal((c["d"], c["d"])))
        out.append((q * np.sign(np.diag(t))[None, :]).T.astype(np.float32))
    return torch.from_numpy(np.stack(out)).cuda()


def _index(c, X):
    if c["axes"]:
        A, off = _axes(X, c["axes"])
        return osann.Index(X, c["L"], rot=A, rot_offset=off)
    return osann.Index(X, c["L"])


def _trace(seed, n):
    """Request sizes (log-uniform 1..4096, the benchmark's trace), index and offset in the index's query pool."""
    sizes = np.floor(np.exp(np.random.default_rng(5000).uniform(0.0, np.log(4096.0), n))).astype(np.int64).clip(1, 4096)
    rng = np.random.default_rng(seed)
    which = rng.integers(0, len(SERVE), n)
    return [(int(s), int(w), int(rng.integers(0, SERVE_POOL - s + 1))) for s, w in zip(sizes, which)]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        idx, pools = [], []
        for i, s in enumerate(SERVE):
            X, Y, _, _ = _data(dict(s, Q=SERVE_POOL), seed * 8 + i)
            idx.append(_index(s, X))
            pools.append(Y)
            del X
        srv = osann.Server(idx, P=[s["P"] for s in SERVE], k=[1] * len(SERVE), slots=4, max_batch=4096)
        srv.tune(reps=2, queries=pools)
        srv.warmup()
        trace = _trace(seed, case["Q"])
        total = sum(s for s, _, _ in trace)
        ids = torch.empty((total, 1), dtype=torch.int64, device="cuda")
        d2 = torch.empty((total, 1), dtype=torch.float32, device="cuda")
        reqs, at = [], 0
        for s, w, o in trace:
            reqs.append((w, pools[w][o:o + s], (ids[at:at + s], d2[at:at + s])))
            at += s
        return dict(kind=kind, idx=idx, srv=srv, reqs=reqs, ids=ids, d2=d2)
    X, Y, src, w = _data(case, seed)
    st = dict(kind=kind, X=X, Y=Y, src=src, w=w, L=case["L"], P=case["P"], k=case["k"])
    if kind == "multi":
        st["ix"] = osann.MultiIndex(X, case["L"], _bases(case, seed))
    elif kind != "build":
        st["ix"] = _index(case, X)
    if kind not in ("rebuild", "build"):
        st["X"] = None  # the index holds its own copy
    return st


def run(st):
    kind = st["kind"]
    if kind == "serve":
        srv = st["srv"]
        for w, q, out in st["reqs"]:
            srv.submit(w, q, out=out)
        for t in srv.drain():
            srv.result(t)
        return {"ids": st["ids"], "d2": st["d2"]}
    if kind == "build":
        ix = osann.Index(st["X"], st["L"])
        keys, offsets, perm = ix.export()
        ix.close()
        return {"keys": keys, "offsets": offsets, "perm": perm}
    ix, Y, P, k = st["ix"], st["Y"], st["P"], st["k"]
    if kind == "rebuild":
        ids, d2 = ix.rebuild_search(st["X"], Y, P, k)
    elif kind == "linear":
        ids, d2 = ix.bruteforce(Y, k)
    elif kind == "excl":
        ids, d2 = ix.search(Y, P, k, query_src=st["src"], grid_w=st["w"], radius=RADIUS)
    else:
        ids, d2 = ix.search(Y, P, k)
    return {"ids": ids, "d2": d2}


# ---------------------------------------------------------------- work

def _rows_per_cone(c):
    """Rows of a probed cone, on average: N / N_C for iid data; nonnegative descriptors use one sign
    pattern of 2^L; image patches crowd the cones next to each other's (measured: about 14 times N / N_C)."""
    if c["data"] == "patch":
        return 14.0 * 1017 * 1017 / (math.comb(64, c["L"]) * 2 ** c["L"])
    if c["data"] == "desc" and not c["axes"]:
        return c["N"] / math.comb(c["d"], c["L"])
    m = c["axes"] or c["d"]
    return c["N"] / (math.comb(m, c["L"]) * 2 ** c["L"])


def work(case):
    if case["kind"] == "serve":
        f = b = 0.0
        q = 480.0 * case["Q"] / len(SERVE)  # mean request: 4095 / ln 4096 queries
        for s in SERVE:
            f += 2.0 * s["d"] * q * s["P"] * _rows_per_cone(s)
            b += 4.0 * s["d"] * (s["N"] + q) + 12.0 * q
        return {"bytes": b, "flops": f}
    c = dict(case, N=1017 * 1017) if case["data"] == "patch" else case
    N, d, Q, k = c["N"], c["d"], c["Q"], c["k"]
    if c["kind"] == "build":
        nc = math.comb(d, c["L"]) * 2 ** c["L"]
        return {"bytes": 4.0 * N * d + 24.0 * N + 8.0 * nc, "flops": 2.0 * N * d}
    m = c["axes"] or d
    nc = math.comb(m, c["L"]) * 2 ** c["L"]
    cand = N if c["kind"] == "linear" else min(N, min(c["P"], nc) * _rows_per_cone(c)) * c["R"]
    rows = min(N, Q * cand)
    byt = 4.0 * d * (rows + Q) + 12.0 * Q * k
    if c["kind"] == "rebuild":
        byt = 4.0 * d * (N + Q) + 12.0 * Q * k
    return {"bytes": byt, "flops": 2.0 * d * Q * cand}


# ---------------------------------------------------------------- 64-bit values

def _coords(A, off, X):
    """Coordinates of the rows on the axes A, by fp32 fused multiply-adds in component order (each
    product exact and each sum rounded once from 64 bits): they only decide which cone a row is in."""
    out = torch.empty((X.shape[0], A.shape[0]), device="cuda")
    for s in range(0, X.shape[0], 1 << 19):
        x = X[s:s + (1 << 19)]
        acc = torch.zeros((x.shape[0], A.shape[0]), device="cuda")
        for j in range(X.shape[1]):
            acc = torch.addcmul(acc.double(), x[:, j:j + 1].double(), A[None, :, j].double()).float()
        out[s:s + x.shape[0]] = acc if off is None else acc - off
    return out


def _binom(d, L):
    return torch.tensor([[math.comb(n, j) for j in range(L + 1)] for n in range(d + 1)], device="cuda")


def _ids(members, signs, L, binom):
    """Cone ids from member components and their sign bits (last axis of length L, any order)."""
    members, at = members.sort(dim=-1)
    signs = signs.gather(-1, at)
    key = torch.zeros(members.shape[:-1], dtype=torch.int64, device="cuda")
    code = torch.zeros_like(key)
    for j in range(L):
        key += binom[members[..., j], j + 1]
        code |= signs[..., j].long() << (L - 1 - j)
    return (key << L) | code


def _row_keys(V, L, binom):
    out = []
    for s in range(0, V.shape[0], 1 << 20):
        v = V[s:s + (1 << 20)]
        top = v.abs().sort(dim=1, descending=True, stable=True).indices[:, :L]
        out.append(_ids(top, v.gather(1, top) >= 0, L, binom))
    return torch.cat(out)


def _positions(d, L, P):
    """The first P list positions as (magnitude ranks of the members, sign flips)."""
    profiles = []
    for delta in range(L + 1):
        keep = L - delta
        for t in ([()] if delta == 0 else itertools.combinations(range(keep + 1, d), delta)):
            profiles.append(tuple(range(keep)) + t)
            if len(profiles) >= P:
                break
        if len(profiles) >= P:
            break
    pos = [(p, (0,) * L) for p in profiles[:P]]
    for h in range(1, L + 1):
        for p in profiles if len(pos) < P else ():
            for flipped in itertools.combinations(range(L), h):  # 0: the member of smallest magnitude
                pos.append((p, tuple(1 if L - 1 - j in flipped else 0 for j in range(L))))
            if len(pos) >= P:
                break
    pos = pos[:P]
    return (torch.tensor([p for p, _ in pos], device="cuda"), torch.tensor([f for _, f in pos], device="cuda"))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("serve", "build"):
        return None  # whole numbers, or too long
    X, Y, src, w = _data(case, seed)
    N, Q, k, L = X.shape[0], Y.shape[0], case["k"], case["L"]
    tables = []
    if kind != "linear":
        if case["axes"]:
            A, off = _axes(X, case["axes"])
            views = [(_coords(A, off, X), _coords(A, off, Y))]
        elif case["R"] > 1:
            views = [(_coords(b, None, X), _coords(b, None, Y)) for b in _bases(case, seed)]
        else:
            views = [(X, Y)]
        m = views[0][0].shape[1]
        binom = _binom(m, L)
        nc = math.comb(m, L) << L
        ranks, flips = _positions(m, L, min(case["P"], nc))
        for V, U in views:
            order = U.abs().sort(dim=1, descending=True, stable=True).indices
            tables.append((_row_keys(V, L, binom), order, U >= 0))
        del views
    Xd = X.double()
    xn = (Xd * Xd).sum(1)
    d2 = torch.full((Q, k), float("inf"), dtype=torch.float64, device="cuda")
    ident = torch.arange(N, device="cuda")
    step = max(1, min(256, int(4e8 // N)))
    for s in range(0, Q, step):
        y = Y[s:s + step].double()
        D = (y * y).sum(1)[:, None] + xn[None, :] - 2.0 * (y @ Xd.T)
        if tables:
            seen = torch.zeros(D.shape, dtype=torch.bool, device="cuda")
            for keys, order, pos in tables:
                members = order[s:s + step][:, ranks]
                signs = pos[s:s + step].gather(1, members.flatten(1)).view(members.shape) ^ flips.bool()
                mask = torch.zeros((y.shape[0], nc), dtype=torch.bool, device="cuda")
                mask.scatter_(1, _ids(members, signs, L, binom), True)
                seen |= mask[:, keys]
            D.masked_fill_(~seen, float("inf"))
        if src is not None:
            t = src[s:s + step, None]
            near = torch.maximum((ident[None] // w - t // w).abs(), (ident[None] % w - t % w).abs()) <= RADIUS
            D.masked_fill_(near, float("inf"))
        v, at = D.topk(min(k, N), dim=1, largest=False)
        # the selected pairs again as direct differences
        again = (Xd[at] - y[:, None, :]).square().sum(2)
        d2[s:s + step, :v.shape[1]] = torch.where(torch.isinf(v), v, again).sort(dim=1).values
    return {"ids": None, "d2": d2}
