"""The work a user of the library has it do, as cases to be timed: whole FastWalk
calls on small graphs, the tree samplers over their range of sizes, the pivot
solve with the recovery, the gradient, the batch of small graphs and the rank
comparison of two centrality vectors.

``listed`` gives the fixed cases, ``draw`` more of the same ranges; ``prepare``
makes a case's inputs and handles, ``run`` is one pass through the public entry
points, ``work`` the bytes and operations a pass cannot do without and ``exact``
its outputs in 64 bits, without the library.
"""
import math

import numpy as np
import torch

import paper_2510_20604_gb300 as rwc

DEV = "cuda"


# ------------------------------------------------------------------- graphs
class Csr:
    """Host CSR of an undirected graph, both arc directions, rows sorted."""

    def __init__(self, row_ptr, col, w):
        self.row_ptr, self.col, self.w = row_ptr, col, w
        self.n = len(row_ptr) - 1
        self.nnz = int(row_ptr[-1])

    def degrees(self):
        if self.w is None:
            return np.diff(self.row_ptr).astype(np.float64)
        src = np.repeat(np.arange(self.n), np.diff(self.row_ptr))
        return np.bincount(src, self.w.astype(np.float64), self.n)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _ints(high, size, gen):
    return torch.randint(0, high, (size,), generator=gen, device=DEV)


def _csr(n, u, v, sigma, gen):
    """CSR from undirected edges: self-loops and copies dropped, lognormal(0,
    sigma) weights per edge (unit weights for sigma = 0)."""
    lo, hi = torch.minimum(u, v), torch.maximum(u, v)
    key = torch.unique((lo * n + hi)[lo != hi])
    lo, hi = key // n, key % n
    arc, order = torch.sort(torch.cat([lo * n + hi, hi * n + lo]))
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    row_ptr[1:] = torch.cumsum(torch.bincount(arc // n, minlength=n), 0)
    w = None
    if sigma:
        we = torch.exp(sigma * torch.randn(len(key), generator=gen, device=DEV))
        w = torch.cat([we, we])[order].float().cpu().numpy()
    return Csr(row_ptr.cpu().numpy(), (arc % n).int().cpu().numpy(), w)


def _with_path(n, u, v, gen):
    """The edges plus those of a random Hamiltonian path (connectivity)."""
    perm = torch.randperm(n, generator=gen, device=DEV)
    return torch.cat([u, perm[:-1]]), torch.cat([v, perm[1:]])


def _er(n, kbar, gen):
    m = max(1, round(kbar * n / 2))
    return _ints(n, m, gen), _ints(n, m, gen)


def _ba(n, m, gen):
    """Preferential attachment: every edge end is drawn from the earlier edge
    ends, an even position naming a new node and an odd one an earlier draw
    (resolved by pointer jumping)."""
    e = torch.arange(n * m, device=DEV)
    pos = (torch.rand(n * m, generator=gen, device=DEV, dtype=torch.float64) * (2 * (e - e % m) + 1)).long()
    while True:
        odd = pos % 2 == 1
        if not bool(odd.any()):
            break
        pos = torch.where(odd, pos[pos // 2], pos)
    return e // m, (pos // 2) // m


def _rgg(n, kbar, gen):
    """Uniform points in the unit square, an edge below the radius that gives
    average degree kbar (no boundary correction)."""
    p = torch.rand(n, 2, generator=gen, device=DEV)
    r2 = kbar / (math.pi * (n - 1))
    us, vs = [], []
    step = max(1, (1 << 27) // n)
    for a in range(0, n, step):
        q = p[a:a + step]
        d2 = (q[:, 0, None] - p[None, :, 0]).square_().add_((q[:, 1, None] - p[None, :, 1]).square_())
        i, j = torch.nonzero(d2 < r2, as_tuple=True)
        us.append(i + a)
        vs.append(j)
    return torch.cat(us), torch.cat(vs)


def _rmat(n, ef, gen):
    """R-MAT with quadrants (0.57, 0.19, 0.19, 0.05); ids beyond n fold back."""
    scale, m = max(1, (n - 1).bit_length()), ef * n // 2
    u = torch.zeros(m, dtype=torch.int64, device=DEV)
    v = torch.zeros_like(u)
    for _ in range(scale):
        r = torch.rand(m, generator=gen, device=DEV)
        u = 2 * u + (r >= 0.76)
        v = 2 * v + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    return u % n, v % n


def _grid(rows, cols):
    i = torch.arange(rows * cols, device=DEV).reshape(rows, cols)
    return (torch.cat([i[:, :-1].reshape(-1), i[:-1].reshape(-1)]),
            torch.cat([i[:, 1:].reshape(-1), i[1:].reshape(-1)]))


def graph(case, seed):
    # a gradient has one value per edge: its graph is the case's own, so that
    # every seed gives as many, and the weights and the objective are the seed's
    gen = _gen(case["n"] if case.get("kind") == "grad" else seed)
    f = case["family"]
    if f == "grid":
        n = case["rows"] * case["cols"]
        return _csr(n, *_grid(case["rows"], case["cols"]), 0.0, gen)
    n = case["n"]
    if f == "er":
        e = _er(n, 8.0, gen)
    elif f == "ba":
        e = _ba(n, case.get("m", 3), gen)
    elif f == "rgg":
        e = _rgg(n, case.get("kbar", 12.0), gen)
    else:
        e = _rmat(n, 16, gen)
    return _csr(n, *_with_path(n, *e, gen), case.get("sigma", 0.0), _gen(seed + 2))


def handle(g, case):
    flags = rwc.GRAPH_INT64_OFFSETS if case.get("int64") else 0
    return rwc.Graph(g.row_ptr, g.col, g.w, flags=flags)


def _vertices(case):
    return case["rows"] * case["cols"] if case["family"] == "grid" else case["n"]


def batch_specs(case):
    """Sizes log-uniform in [50, 20000], kinds drawn equally; the sizes are the
    case's own (quantiles of the law, so that its work is the same for every
    seed), the graphs and the trees the seed's."""
    G = case["graphs"]
    q = (np.arange(G) + 0.5) / G
    sizes = np.floor(np.exp(math.log(50) + q * (math.log(20000) - math.log(50)))).astype(int)
    sizes = np.random.default_rng(G).permutation(sizes)
    return [(int(n), ("er", "ba", "rgg")[i % 3]) for i, n in enumerate(sizes)]


# -------------------------------------------------------------------- cases
def listed():
    return [
        # one small network, a few trees: what an interactive call costs
        {"name": "fastwalk_er100", "kind": "fastwalk", "family": "er", "n": 100, "trees": 64},
        # the small reference configuration: BA, 2000 vertices, 1000 trees
        {"name": "fastwalk_ba2000", "kind": "fastwalk", "family": "ba", "n": 2000, "trees": 1000},
        # FastWalk to 1% predicted error, trees added by the stopping rule
        {"name": "target_ba2000", "kind": "target", "family": "ba", "n": 2000, "eps": 0.01},
        # the largest graphs whose tree fits one SM, weighted, trees returned
        {"name": "trees_rgg19999w", "kind": "trees", "family": "rgg", "n": 19999, "sigma": 0.5,
         "trees": 304, "want": True},
        # high diameter, long walks: a grid, 1000 trees
        {"name": "trees_grid240", "kind": "trees", "family": "grid", "rows": 224, "cols": 240,
         "trees": 1000, "want": False},
        # social-network shape at scale 20, 2000 trees
        {"name": "trees_rmat20", "kind": "trees", "family": "rmat", "n": 1 << 20, "trees": 2000,
         "want": False},
        # the paper-size configuration's shape: lognormal weights, int64 offsets, 500 trees
        {"name": "trees_rmat20w", "kind": "trees", "family": "rmat", "n": 1 << 20, "sigma": 1.0,
         "int64": True, "trees": 500, "want": False},
        # pivot solve and recovery, ill-conditioned (large diameter)
        {"name": "estimate_grid1024", "kind": "estimate", "family": "grid", "rows": 1024,
         "cols": 1024, "trees": 2000},
        # pivot solve and recovery, power-law degrees
        {"name": "estimate_rmat20", "kind": "estimate", "family": "rmat", "n": 1 << 20,
         "trees": 2000},
        # backward of the centrality: sketched gradient, 64 columns
        {"name": "grad_rgg100k", "kind": "grad", "family": "rgg", "n": 100000, "sigma": 0.5,
         "k": 64},
        # many small graphs in one launch
        {"name": "batch512", "kind": "batch", "family": "batch", "graphs": 512, "trees": 64},
        # comparing two centrality vectors: mean relative error and Kendall distance
        {"name": "rank_262144", "kind": "rank", "family": "vector", "n": 1 << 18, "ties": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fastwalk", "target", "trees", "trees", "trees", "estimate", "grad", "batch", "rank"])
    if kind == "fastwalk":
        return {"kind": kind, "family": rng.choice(["er", "ba", "rgg"]), "n": _log_int(rng, 50, 4000),
                "sigma": rng.choice([0.0, 0.5]), "trees": _log_int(rng, 16, 2000)}
    if kind == "target":
        return {"kind": kind, "family": rng.choice(["er", "ba", "rgg"]), "n": _log_int(rng, 300, 4000),
                "eps": round(math.exp(rng.uniform(math.log(0.01), math.log(0.1))), 4)}
    if kind == "trees":
        f = rng.choice(["grid", "rmat", "rgg", "small"])
        if f == "grid":
            return {"kind": kind, "family": f, "rows": rng.randint(143, 220), "cols": rng.randint(143, 220),
                    "trees": _log_int(rng, 16, 900), "want": False}
        if f == "small":
            return {"kind": kind, "family": rng.choice(["er", "ba", "rgg"]), "n": _log_int(rng, 1000, 20000),
                    "sigma": rng.choice([0.0, 0.5]), "trees": _log_int(rng, 64, 600),
                    "want": rng.random() < 0.5}
        c = {"kind": kind, "family": f, "sigma": rng.choice([0.0, 0.5, 1.0]), "int64": rng.random() < 0.3,
             "want": False}
        c["n"] = _log_int(rng, 20001, 1000000) if f == "rmat" else _log_int(rng, 20001, 60000)
        c["trees"] = _log_int(rng, 16, 1000)
        c["want"] = c["n"] * c["trees"] < 20_000_000 and rng.random() < 0.5
        return c
    if kind == "estimate":
        f = rng.choice(["grid", "rmat", "rgg"])
        if f == "grid":
            return {"kind": kind, "family": f, "rows": rng.randint(100, 900), "cols": rng.randint(100, 900),
                    "trees": 2000}
        return {"kind": kind, "family": f, "sigma": rng.choice([0.0, 0.5]), "trees": 2000,
                "n": _log_int(rng, 5000, 1000000 if f == "rmat" else 100000)}
    if kind == "grad":
        return {"kind": kind, "family": rng.choice(["rgg", "ba"]), "n": _log_int(rng, 1000, 100000),
                "sigma": rng.choice([0.0, 0.5]), "k": rng.choice([8, 16, 33, 64])}
    if kind == "batch":
        return {"kind": kind, "family": "batch", "graphs": _log_int(rng, 32, 400), "trees": _log_int(rng, 16, 128)}
    return {"kind": kind, "family": "vector", "n": _log_int(rng, 2000, 250000), "ties": rng.random() < 0.5}


# ------------------------------------------------------------------ one pass
def _estimate_sums(g, case, seed):
    """Visit totals with the spread tree sampling gives: at least one visit per
    tree, a long tail, 0 at the pivot."""
    gen = _gen(seed + 1)
    t = 1.0 + torch.exp(torch.randn(g.n, generator=gen, device=DEV, dtype=torch.float64))
    s = torch.floor(t * case["trees"])
    s[int(np.argmax(g.degrees()))] = 0.0
    return s


def _grad_c(case, seed):
    return torch.rand(case["n"], generator=_gen(seed + 1), device=DEV, dtype=torch.float64)


def _rank_vectors(case, seed):
    """A centrality vector and an estimate of it with 2% error; with ties, both
    rounded as a degree ranking or a printed table is."""
    gen = _gen(seed)
    H = case["n"] * torch.exp(0.5 * torch.randn(case["n"], generator=gen, device=DEV, dtype=torch.float64))
    E = H * (1.0 + 0.02 * torch.randn(case["n"], generator=gen, device=DEV, dtype=torch.float64))
    if case["ties"]:
        unit = case["n"] / 20.0
        H, E = torch.ceil(H / unit) * unit, torch.ceil(E.clamp_min(unit) / unit) * unit
    return H, E


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "seed": seed}
    if kind == "rank":
        s["H"], s["E"] = _rank_vectors(case, seed)
        return s
    if kind == "batch":
        s["batch"] = rwc.Batch([graph({"family": f, "n": n, "m": 2, "kbar": 10.0}, seed * 4096 + i)
                                for i, (n, f) in enumerate(batch_specs(case))])
        return s
    g = graph(case, seed)
    s["G"] = handle(g, case)
    if kind == "estimate":
        s["sums"] = _estimate_sums(g, case, seed)
    if kind == "grad":
        s["c"] = _grad_c(case, seed)
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "fastwalk":
        H, _ = rwc.fastwalk(s["G"], case["trees"], seed=s["seed"])
        return {"H": H}
    if kind == "target":
        H, T, mre = rwc.fastwalk_to_target(s["G"], case["eps"], seed=s["seed"])
        return {"H": H, "trees": T, "mre": mre}
    if kind == "trees":
        sums, _, par, vis = s["G"].sample(case["trees"], seed=s["seed"], want_trees=case["want"])
        return {"sums": sums, "parents": par, "visits": vis} if case["want"] else {"sums": sums}
    if kind == "estimate":
        return {"H": s["G"].estimate(s["sums"], case["trees"])}
    if kind == "grad":
        return {"grad": s["G"].grad(s["c"], k=case["k"], sketch_seed=s["seed"])}
    if kind == "batch":
        sums, _ = s["batch"].sample(case["trees"], seed=s["seed"])
        return {"sums": sums}
    mre = rwc.rwc_mre(s["H"], s["E"])
    tau, diff = rwc.rwc_kendall(s["H"], s["E"])
    return {"mre": mre, "tau": tau, "diff": diff}


# ----------------------------------------------------------------- the floor
#: mean successor draws per vertex and tree of the families, from sampled trees
DRAWS = {"er": 1.2, "ba": 1.3, "rgg": 1.4, "rmat": 1.6}
OPS_PER_DRAW = 60.0          # Philox-4x32-10: 20 multiplies, 40 xors and adds


def _arcs(case):
    if case["family"] == "grid":
        return 4 * _vertices(case) - 2 * (case["rows"] + case["cols"])
    n = case["n"]
    k = {"er": 8.0, "ba": 2.0 * case.get("m", 3), "rgg": case.get("kbar", 12.0), "rmat": 15.3}[case["family"]]
    return int((k + 2.0) * n)


def _sampler_work(case, trees):
    """Each draw reads its row's bounds and one arc (head; threshold and alias
    of a weighted one); each tree and vertex has a parent and a visit count."""
    n = _vertices(case)
    per = 2.93 * math.log(math.sqrt(n)) if case["family"] == "grid" else DRAWS[case["family"]] * (
        1.7 if case.get("sigma", 0.0) >= 1.0 else 1.1 if case.get("sigma") else 1.0)
    draws = per * n * trees
    arc = (16 if case.get("int64") else 8) + (12 if case.get("sigma") else 4)
    return {"bytes": draws * arc + 8.0 * n * trees + 8.0 * n, "flops": OPS_PER_DRAW * draws}


def _solve_work(case, k):
    """The graph, the right-hand sides and the result once; two operations per
    arc and column for each iteration, iterations growing with the diameter."""
    n, nnz = _vertices(case), _arcs(case)
    iters = 8.0 * max(case["rows"], case["cols"]) if case["family"] == "grid" else 60.0
    return {"bytes": nnz * (8.0 if case.get("sigma") else 4.0) + n * (4.0 + 16.0 * k),
            "flops": iters * k * (2.0 * nnz + 12.0 * n)}


def work(case):
    kind = case["kind"]
    if kind == "trees":
        return _sampler_work(case, case["trees"])
    if kind in ("fastwalk", "target"):
        T = case["trees"] if kind == "fastwalk" else max(256.0, 0.14 / case["eps"] ** 2)
        a, b = _sampler_work(case, T), _solve_work(case, 1)
        return {m: a[m] + b[m] for m in a}
    if kind == "estimate":
        return _solve_work(case, 1)
    if kind == "grad":
        w = _solve_work(case, case["k"] + 2)
        return {"bytes": w["bytes"] + 4.0 * _arcs(case) / 2, "flops": w["flops"] + 3.0 * case["k"] * _arcs(case) / 2}
    if kind == "batch":
        parts = [_sampler_work({"family": f, "n": n}, case["trees"]) for n, f in batch_specs(case)]
        return {m: sum(p[m] for p in parts) for m in ("bytes", "flops")}
    n = case["n"]
    return {"bytes": 16.0 * n, "flops": 4.0 * n * math.log2(n)}


# --------------------------------------------------------------- in 64 bits
def _philox(c0, c1, c2, c3, seed):
    """Word 0 and 1 of Philox-4x32-10 (Salmon et al., SC'11) on uint64 arrays."""
    M = np.uint64(0xFFFFFFFF)
    S = np.uint64(32)
    c = [np.asarray(x, np.uint64) for x in (c0, c1, c2, c3)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        a, b = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(b >> S) ^ c[1] ^ np.uint64(k0), b & M, (a >> S) ^ c[3] ^ np.uint64(k1), a & M]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c[0], c[1]


def _visits(g, root, seed, tree0, trees):
    """Visit totals of Wilson's algorithm (unit weights), all trees in step:
    each is at one vertex of its walk or of the path it adds to its tree."""
    n = g.n
    deg = np.diff(g.row_ptr).astype(np.uint64)
    nxt = np.zeros((trees, n), np.int64)
    cnt = np.zeros((trees, n), np.int64)
    done = np.zeros((trees, n), bool)
    done[:, root] = True
    start = np.zeros(trees, np.int64)
    x = np.zeros(trees, np.int64)
    settle = np.zeros(trees, bool)
    live = np.arange(trees)
    while len(live):
        xs = x[live]
        tree = done[live, xs]
        adding = settle[live]
        walk = live[~tree & ~adding]
        if len(walk):
            u = x[walk]
            o, _ = _philox(cnt[walk, u], u, walk + tree0, np.zeros_like(u), seed)
            j = ((o * deg[u]) >> np.uint64(32)).astype(np.int64)
            v = g.col[g.row_ptr[u] + j].astype(np.int64)
            cnt[walk, u] += 1
            nxt[walk, u] = v
            x[walk] = v
        add = live[~tree & adding]
        if len(add):
            u = x[add]
            done[add, u] = True
            x[add] = nxt[add, u]
        back = live[tree & ~adding]          # the walk met the tree: add its path
        settle[back] = True
        x[back] = start[back]
        fresh = live[tree & adding]          # the path is in: next start
        settle[fresh] = False
        start[fresh] += 1
        x[fresh] = np.minimum(start[fresh], n - 1)
        live = live[start[live] < n]
    return cnt.sum(0).astype(np.float64)


def _laplacian(g):
    d = torch.tensor(g.degrees(), device=DEV)
    vals = torch.ones(g.nnz, dtype=torch.float64, device=DEV) if g.w is None else torch.tensor(g.w, device=DEV).double()
    A = torch.sparse_csr_tensor(torch.tensor(g.row_ptr, device=DEV), torch.tensor(g.col, device=DEV).long(), vals,
                                (g.n, g.n))
    return A, d


def _pinv_times(g, B):
    """L^+ B by conjugate gradients in 64 bits, columns together, two rounds."""
    A, d = _laplacian(g)

    def mul(X):
        return d[:, None] * X - A @ X

    B = B - B.mean(0)
    X = torch.zeros_like(B)
    for _ in range(2):
        R = B - mul(X)
        R = R - R.mean(0)
        Z = R / d[:, None]
        P, rz = Z.clone(), (R * Z).sum(0)
        stop = torch.maximum(1e-26 * (R * R).sum(0), 1e-31 * (B * B).sum(0))
        for it in range(20000):
            Q = mul(P)
            a = rz / (P * Q).sum(0).clamp_min(1e-300)
            X = X + a * P
            R = R - a * Q
            Z = R / d[:, None]
            new = (R * Z).sum(0)
            if it % 8 == 7 and bool(((R * R).sum(0) <= stop).all()):
                break
            P = Z + (new / rz.clamp_min(1e-300)) * P
            rz = new
        X = X - X.mean(0)
    return X


def _grid_pinv(case, b):
    """L^+ b on a grid: its cosine eigenvectors through the even extension."""
    R, C = case["rows"], case["cols"]
    f = b.reshape(R, C)
    f = torch.cat([f, f.flip(0)], 0)
    f = torch.cat([f, f.flip(1)], 1)
    lam = (2 - 2 * torch.cos(math.pi * torch.arange(2 * R, device=DEV, dtype=torch.float64) / R))[:, None] + (
        2 - 2 * torch.cos(math.pi * torch.arange(2 * C, device=DEV, dtype=torch.float64) / C))[None, :]
    F = torch.fft.fft2(f.to(torch.complex128))
    lam[0, 0] = 1.0
    F = F / lam
    F[0, 0] = 0.0
    return torch.fft.ifft2(F).real[:R, :C].reshape(-1)


def _recover(g, case, sums, trees):
    """Algorithm 1: H from the visit totals."""
    d = torch.tensor(g.degrees(), device=DEV)
    v, vol = int(np.argmax(g.degrees())), float(g.degrees().sum())
    b = -(math.sqrt(float(d[v])) / vol) * d
    b[v] += math.sqrt(float(d[v]))
    z = _grid_pinv(case, b - b.mean()) if case["family"] == "grid" else _pinv_times(g, b[:, None])[:, 0]
    y = torch.sqrt(d) * z - torch.sqrt(d) * ((d * z).sum() / vol)
    r, pi = d / d[v], d / vol
    H = (sums / trees - r * y[v] + 2.0 * torch.sqrt(r) * y) / pi
    H[v] = y[v] / pi[v]
    return H


def _predicted(g, sums, T, H):
    d = torch.tensor(g.degrees(), device=DEV)
    v = int(np.argmax(g.degrees()))
    t = sums / T
    e = math.sqrt(2.0 / math.pi) * torch.sqrt((t * (t - 1.0)).clamp_min(0.0) / T) / ((d / d.sum()) * H.abs())
    e[v] = 0.0
    return float(e.mean())


def exact(case, seed):
    kind = case["kind"]
    if kind == "rank":
        H, E = _rank_vectors(case, seed)
        mre = ((H - E).abs() / H).mean()
        n, diff = case["n"], 0
        step = max(1, (1 << 28) // n)
        for a in range(0, n, step):
            sa = (H[a:a + step, None] > H[None, :]).to(torch.int8) - (H[a:a + step, None] < H[None, :]).to(torch.int8)
            sb = (E[a:a + step, None] > E[None, :]).to(torch.int8) - (E[a:a + step, None] < E[None, :]).to(torch.int8)
            diff += int((sa * sb).sum(dtype=torch.int64))
        diff //= 2
        return {"mre": mre, "tau": 2.0 * diff / (n * (n - 1.0)), "diff": diff}
    if kind == "estimate":
        g = graph(case, seed)
        return {"H": _recover(g, case, _estimate_sums(g, case, seed), case["trees"])}
    if kind == "grad":
        g, c, k = graph(case, seed), _grad_c(case, seed), case["k"]
        d = torch.tensor(g.degrees(), device=DEV)
        vol, csum = float(d.sum()), float(c.sum())
        i, u = np.meshgrid(np.arange(k), np.arange(g.n))
        o, _ = _philox(i, u, np.full_like(u, 0xFFFFFFFF), np.zeros_like(u), seed)
        q = torch.tensor(np.where(o >> np.uint64(31), -1.0, 1.0) / math.sqrt(k), device=DEV)
        S = torch.sqrt(c)[:, None] * q
        X = _pinv_times(g, torch.cat([S, c[:, None], d[:, None]], 1))
        tr, dTy = float((X[:, :k] * S).sum()), float((d * X[:, k + 1]).sum())
        src = torch.repeat_interleave(torch.arange(g.n, device=DEV), torch.tensor(np.diff(g.row_ptr), device=DEV))
        dst = torch.tensor(g.col, device=DEV).long()
        a, b = src[src < dst], dst[src < dst]
        D = X[a] - X[b]
        x, y = X[:, k], X[:, k + 1]
        J = (2 * tr - vol * D[:, :k].square().sum(1) + 2 * D[:, k] * D[:, k + 1] - 2 * (x[a] + x[b])
             + csum * ((2 * (y[a] + y[b]) - D[:, k + 1].square()) / vol - 2 * dTy / vol ** 2))
        return {"grad": J}
    if kind in ("fastwalk", "target") and not case.get("sigma") and case["n"] <= 2500:
        g = graph(case, seed)
        v = int(np.argmax(g.degrees()))
        T = case["trees"] if kind == "fastwalk" else 256
        total = _visits(g, v, seed, 0, T)
        while True:
            sums = torch.tensor(total, device=DEV)
            H = _recover(g, case, sums, T)
            if kind == "fastwalk":
                return {"H": H}
            mre = _predicted(g, sums, T, H)
            if mre <= case["eps"]:
                return {"H": H, "trees": T, "mre": mre}
            need = max(math.ceil(T * (mre / case["eps"]) ** 2), T + 1)
            if need > 8000:
                return None
            total = total + _visits(g, v, seed, T, need - T)
            T = need
    return None
