"""The work a user of this library has it do, as measurable cases.

A case is a dict of plain values.  `job` says what a program does with a
graph:

* decompose: one graph, from its CSR to every kappa asked for (build the
  incidence, iterate to convergence, free the handle), on device arrays or,
  with host = True, on numpy arrays in and out as the serving loop does;
* batch: many small graphs as one disjoint union, build to convergence;
* sweeps: a handle the program keeps, and on it the early-stopped iterates
  with their quality against kappa, and AND without notification;
* ego: PartialAnd queries on a kept handle (Section 5.4 of the paper);
* otf: k-truss with no stored incidence, for inputs whose incidence does not
  fit the memory at hand;
* normalize: a raw list of vertex pairs to the CSR the builds take.

Graphs are drawn on the GPU from the seed: R-MAT (0.57, 0.19, 0.19, 0.05),
Chung-Lu power laws with or without planted cliques, and uniform random
pairs, with scrambled vertex ids, as in paper_1704_00386_gb300/graphs.py.
AND's pass and evaluation counts depend on the schedule of the GPU's blocks,
so the results of AND are its tau alone; SND's pass count is exact and is
returned with its tau.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1704_00386_gb300 import nd

ABC = (0.57, 0.19, 0.19)   # R-MAT quadrants


def listed():
    return [
        # the smallest workload of bench.py: a 2,000-vertex k-core, where launches and host waits count
        dict(name="core_chunglu_2k", job="decompose", family="chunglu", n=2000, degree=10.0, gamma=2.5, cliques=0,
             r=1, modes="snd,and", host=False),
        # a small request as the serving loop gets it: numpy in, k-truss by AND, numpy out
        dict(name="truss_request_11k", job="decompose", family="chunglu", n=2811, degree=8.0, gamma=2.2, cliques=0,
             r=2, modes="and", host=True),
        # a mid-sized (3,4) request on device arrays, the third job of the serving mix
        dict(name="nucleus_request_300k", job="decompose", family="rmat", n=37501, degree=16.0, gamma=0.0, cliques=0,
             r=3, modes="and", host=False),
        # an ordinary k-truss, a vertex count that is no power of two, both algorithms
        dict(name="truss_rmat_100k", job="decompose", family="rmat", n=100003, degree=32.0, gamma=0.0, cliques=0,
             r=2, modes="snd,and", host=False),
        # bench.py's headline workload: k-truss of R-MAT scale 20, edge factor 16
        dict(name="truss_rmat_s20", job="decompose", family="rmat", n=1 << 20, degree=32.0, gamma=0.0, cliques=0,
             r=2, modes="snd,and", host=False),
        # deep (3,4) nuclei: Chung-Lu of 100,000 vertices with 200 planted cliques
        dict(name="nucleus_planted_100k", job="decompose", family="chunglu", n=100000, degree=20.0, gamma=2.1,
             cliques=200, r=3, modes="snd,and", host=False),
        # a large k-core: R-MAT scale 24, edge factor 16
        dict(name="core_rmat_s24", job="decompose", family="rmat", n=1 << 24, degree=32.0, gamma=0.0, cliques=0,
             r=1, modes="snd,and", host=False),
        # many small graphs at once: the batched k-truss of 256 mixed graphs
        dict(name="batch_truss_256", job="batch", graphs=256, n_lo=100, n_hi=50000, r=2, modes="snd"),
        # the evaluation of Section 5.2 on a kept handle: early-stopped iterates, their quality, AND-nn
        dict(name="sweeps_truss_131k", job="sweeps", family="rmat", n=131071, degree=32.0, gamma=0.0, cliques=0,
             r=2, early=3),
        # ego-network queries on a kept k-truss handle
        dict(name="ego_truss_262k", job="ego", family="rmat", n=262144, degree=32.0, gamma=0.0, cliques=0, r=2,
             centres=16),
        # k-truss without a stored incidence
        dict(name="otf_truss_50k", job="otf", family="rmat", n=50021, degree=32.0, gamma=0.0, cliques=0, r=2,
             modes="snd"),
        # raw pairs of an R-MAT scale 20 edge list to the simple CSR
        dict(name="normalize_16m", job="normalize", family="rmat", n=1 << 20, degree=32.0, gamma=0.0, cliques=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the jobs of the list in the proportions a user meets them, sizes over their whole range."""
    job = rng.choice(["decompose"] * 6 + ["batch", "sweeps", "ego", "otf", "normalize"])
    if job == "batch":
        hi = _log(rng, 1000, 50000)
        r = rng.choice([1, 2])
        return dict(job=job, graphs=rng.randint(17, 256), n_lo=100, n_hi=hi, r=r, modes=rng.choice(["snd", "and"]))
    family = rng.choice(["rmat", "chunglu"])
    degree = round(rng.uniform(8.0, 32.0), 2)
    gamma = round(rng.uniform(2.1, 2.5), 2) if family == "chunglu" else 0.0
    graph = dict(family=family, degree=degree, gamma=gamma, cliques=0)
    if job == "normalize":
        return dict(job=job, n=_log(rng, 1000, 1 << 20), **graph)
    if job == "otf":
        return dict(job=job, n=_log(rng, 1000, 60000), r=2, modes=rng.choice(["snd", "and"]), **graph)
    if job == "ego":
        return dict(job=job, n=_log(rng, 2000, 262144), r=2, centres=rng.randint(1, 32), **graph)
    if job == "sweeps":
        return dict(job=job, n=_log(rng, 2000, 131072), r=rng.choice([1, 2]), early=rng.randint(1, 9), **graph)
    r = rng.choice([1, 2, 3])
    n = _log(rng, 500, {1: 1 << 23, 2: 700000, 3: 50000}[r])
    if r == 3:
        graph["degree"] = min(degree, 20.0)
        if family == "chunglu":
            graph["cliques"] = min(rng.randint(0, 200), n // 500)
    modes = rng.choice(["snd", "and", "snd,and", "and_nn"])
    return dict(job=job, n=n, r=r, modes=modes, host=n < 20000 and rng.random() < 0.5, **graph)


# ---- graphs -----------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _rmat_pairs(n, pairs, g):
    """R-MAT samples with both ends below n (the first n ids of the next power of two)."""
    scale = max(1, math.ceil(math.log2(n)))
    a, b, c = ABC
    out = []
    for lo in range(0, pairs, 1 << 26):
        k = min(1 << 26, pairs - lo)
        s = torch.zeros(k, dtype=torch.int64, device="cuda")
        d = torch.zeros(k, dtype=torch.int64, device="cuda")
        for level in range(scale):
            x = torch.rand(k, generator=g, device="cuda")
            s += (x >= a + b).to(torch.int64) << level
            d += (((x >= a) & (x < a + b)) | (x >= a + b + c)).to(torch.int64) << level
        if n < 1 << scale:
            keep = (s < n) & (d < n)
            s, d = s[keep], d[keep]
        out.append((s, d))
    return torch.cat([s for s, _ in out]), torch.cat([d for _, d in out])


def _chunglu_pairs(n, pairs, gamma, degree, g):
    w = torch.arange(1, n + 1, dtype=torch.float64, device="cuda") ** (-1.0 / (gamma - 1.0))
    w *= n * degree / w.sum()
    cdf = torch.cumsum(torch.clamp(w, max=float(w.sum()) ** 0.5), 0)
    top = float(cdf[-1])
    ends = [torch.searchsorted(cdf, torch.rand(pairs, generator=g, device="cuda", dtype=torch.float64) * top)
            for _ in range(2)]
    return ends[0].clamp_(max=n - 1), ends[1].clamp_(max=n - 1)


def _clique_pairs(n, count, seed):
    """Pairs of count cliques of 20 to 60 vertices on random vertex sets."""
    rng = np.random.default_rng(seed)
    src, dst = [], []
    for _ in range(count):
        k = int(rng.integers(20, 61))
        vs = rng.choice(n, size=k, replace=False)
        i, j = np.triu_indices(k, 1)
        src.append(vs[i])
        dst.append(vs[j])
    return [torch.from_numpy(np.concatenate(x).astype(np.int64)).cuda() for x in (src, dst)]


def _edges(case):
    """The distinct edges of a case's graph, cliques left out: a tenth below the pairs of its mean degree."""
    return int(case["n"] * case["degree"] * 0.45)


def _pairs(case, seed):
    """Raw pairs of a case's graph, repeats and self-loops as drawn, up to the one that completes its edges; and
    which of them are the first of their edge."""
    g = _gen(seed)
    n, edges = case["n"], _edges(case)
    s = d = torch.zeros(0, dtype=torch.int64, device="cuda")
    while True:
        pairs = edges // 8 + 1000 if s.numel() else int(edges * 1.12) + 1000
        if case["family"] == "rmat":
            a, b = _rmat_pairs(n, pairs, g)
        elif case["family"] == "chunglu":
            a, b = _chunglu_pairs(n, pairs, case["gamma"], case["degree"], g)
        else:
            a, b = (torch.randint(n, (pairs,), generator=g, device="cuda") for _ in range(2))
        s, d = torch.cat([s, a]), torch.cat([d, b])
        del a, b
        key, at = torch.sort(torch.minimum(s, d) * n + torch.maximum(s, d), stable=True)
        new = torch.ones_like(key, dtype=torch.bool)
        new[1:] = key[1:] != key[:-1]
        del key
        first = torch.zeros_like(new)
        first[at[new]] = True
        del at, new
        first &= s != d
        seen = torch.cumsum(first, 0)
        if int(seen[-1]) >= edges:
            break
    cut = int(torch.searchsorted(seen, edges)) + 1
    perm = torch.randperm(n, generator=g, device="cuda")
    return perm[s[:cut]], perm[d[:cut]], first[:cut]


def _csr(n, s, d):
    """Symmetric sorted CSR of distinct edges."""
    key = torch.sort(torch.cat([s * n + d, d * n + s]))[0]
    rows = torch.arange(n + 1, dtype=torch.int64, device="cuda") * n
    return torch.searchsorted(key, rows), (key % n).to(torch.int32)


def _graph(case, seed):
    n = case["n"]
    s, d, first = _pairs(case, seed)
    s, d = s[first], d[first]
    if case.get("cliques"):
        a, b = _clique_pairs(n, case["cliques"], seed)
        s, d = torch.cat([s, a]), torch.cat([d, b])
        key = torch.unique(torch.minimum(s, d) * n + torch.maximum(s, d))
        s, d = key // n, key % n
    return _csr(n, s, d)


def _batch(case, seed):
    """n uniform in [n_lo, n_hi]; uniform pairs, Chung-Lu or R-MAT by chance.  The sizes are the case's, so that the
    results of every seed have one layout; the edges are the seed's."""
    rng = np.random.default_rng([case["graphs"], case["n_hi"]])
    out = []
    for i in range(case["graphs"]):
        n = int(rng.integers(case["n_lo"], case["n_hi"] + 1))
        family = ("uniform", "chunglu", "rmat")[int(rng.integers(3))]
        one = dict(family=family, n=n, degree=16.0 if family == "rmat" else 8.0, gamma=2.2)
        out.append(_graph(one, seed * 100003 + i))
    return out


def _results(case):
    """A result buffer of a (3,4) decomposition, whose number of triangles is only known after the build: a program
    that decomposes graph after graph keeps one that is long enough."""
    size = 32 * _edges(case) + 50000 * case["cliques"]
    return np.zeros(size, np.int32) if case["host"] else torch.zeros(size, dtype=torch.int32, device="cuda")


def _upper_edges(rp, col):
    """The canonical edges (u < v), in order."""
    n = rp.numel() - 1
    u = torch.repeat_interleave(torch.arange(n, device=rp.device), rp[1:] - rp[:-1])
    v = col.to(torch.int64)
    up = u < v
    return u[up], v[up]


def _ego_members(case, rp, col, seed):
    """Edge ids inside the closed neighbourhoods of a few random vertices of positive degree."""
    rng = np.random.default_rng(seed + 77)
    inside = torch.zeros(case["n"], dtype=torch.bool, device="cuda")
    rph = rp.cpu().numpy()
    some = np.flatnonzero(np.diff(rph))
    for c in rng.choice(some, size=min(case["centres"], some.size), replace=False):
        inside[int(c)] = True
        inside[col[rph[c]:rph[c + 1]].to(torch.int64)] = True
    u, v = _upper_edges(rp, col)
    return torch.nonzero(inside[u] & inside[v]).flatten().to(torch.int32)


# ---- the work -----------------------------------------------------------------

def prepare(case, seed):
    job = case["job"]
    if job == "normalize":
        s, d, _ = _pairs(case, seed)
        return dict(case=case, src=s, dst=d)
    if job == "batch":
        return dict(case=case, graphs=_batch(case, seed))
    rp, col = _graph(case, seed)
    state = dict(case=case, rp=rp, col=col)
    if case.get("host"):
        state.update(rp=rp.cpu().numpy(), col=col.cpu().numpy())
    if job == "decompose" and case["r"] == 3:
        state["out"] = {mode: _results(case) for mode in case["modes"].split(",")}
    if job in ("sweeps", "ego"):
        state["inc"] = nd.build_incidence(rp, col, case["r"], case["r"] + 1)
    if job == "sweeps":
        state["kappa"] = state["inc"].snd()[0]
    if job == "ego":
        state["members"] = _ego_members(case, rp, col, seed)
    return state


def _iterate(inc, modes, results=None):
    out = {}
    for mode in modes.split(","):
        into = results[mode] if results and len(results[mode]) >= inc.num_r else None
        if mode == "snd":
            out["snd"], out["passes"] = inc.snd(out=into)
        else:
            out[mode] = inc.and_(notify=mode == "and", out=into)[0]
    return out


def run(state):
    case = state["case"]
    job = case["job"]
    if job == "normalize":
        return nd.normalize(state["src"], state["dst"], case["n"])
    if job == "sweeps":
        inc, kappa = state["inc"], state["kappa"]
        early, passes = inc.iterate_k("snd", case["early"])
        later, more = inc.iterate_k("snd", 2, tau=early)
        return dict(early=early, passes=passes, later=later, more=more, equal=nd.count_equal(later, kappa),
                    order=nd.kendall_tau_b(later, kappa), and_nn=inc.and_(notify=False)[0])
    if job == "ego":
        return state["inc"].and_partial(state["members"])[0]
    if job == "batch":
        inc, offsets = nd.build_incidence_batch(state["graphs"], case["r"], case["r"] + 1)
        out = _iterate(inc, case["modes"])
        out.pop("passes", None)
        out["offsets"] = offsets
    else:
        inc = nd.build_incidence(state["rp"], state["col"], case["r"], case["r"] + 1, on_the_fly=job == "otf")
        out = _iterate(inc, case["modes"], state.get("out"))
    inc.free()
    return out


def work(case):
    """The input read once and the outputs written once; sizes as expected from the recipe."""
    job = case["job"]
    if job == "batch":
        n = case["graphs"] * (case["n_lo"] + case["n_hi"]) / 2.0
        m, results = n * 5.0, 1
    else:
        n, m = case["n"], _edges(case) + 800.0 * case["cliques"]
        results = len(case["modes"].split(",")) if "modes" in case else {"sweeps": 3, "ego": 1}.get(job, 0)
    if job == "normalize":
        return {"bytes": 16.0 * m + 8.0 * n + 8.0 * m, "flops": 0}
    r_cliques = {1: n, 2: m, 3: m + 13000.0 * case.get("cliques", 0)}[case["r"]]
    return {"bytes": 8.0 * n + 8.0 * m + 4.0 * r_cliques * results, "flops": 0}


# ---- the same results in plain torch --------------------------------------------

def _ranges(start, length):
    """Concatenated start[i] .. start[i] + length[i] - 1, and i for each."""
    owner = torch.repeat_interleave(torch.arange(length.numel(), device=length.device), length)
    base = torch.cumsum(length, 0) - length
    return start[owner] + torch.arange(owner.numel(), device=length.device) - base[owner], owner


def _incidence(rp, col, r):
    """(N_R, rows, others): per (R, S) pair the r-clique R and the other r-cliques of S; None if it is too large."""
    n = rp.numel() - 1
    deg = rp[1:] - rp[:-1]
    if r == 1:
        if col.numel() > 1 << 27:
            return None
        return n, torch.repeat_interleave(torch.arange(n, device=rp.device), deg), col.to(torch.int64)[:, None]
    u, v = _upper_edges(rp, col)
    m = u.numel()
    if m > 1 << 22:
        return None
    edge = u * n + v
    before = (deg[u] < deg[v]) | ((deg[u] == deg[v]) & (u < v))
    a, b = torch.where(before, u, v), torch.where(before, v, u)
    order = torch.argsort(a * n + b)
    a, b = a[order], b[order]
    first = torch.searchsorted(a, torch.arange(n + 1, device=rp.device))
    outs = first[1:] - first[:-1]

    def edge_id(x, y):
        key = torch.minimum(x, y) * n + torch.maximum(x, y)
        at = torch.searchsorted(edge, key).clamp_(max=m - 1)
        return torch.where(edge[at] == key, at, -1)

    tris = []
    step = max(1, int((1 << 26) / max(1, int(outs.max()) if n else 1)))
    for lo in range(0, m, step):
        aa, bb = a[lo:lo + step], b[lo:lo + step]
        j, i = _ranges(first[bb], outs[bb])
        w = b[j]
        ok = edge_id(aa[i], w) >= 0
        tris.append(torch.stack([aa[i][ok], bb[i][ok], w[ok]], 1))
    tri = torch.cat(tris) if tris else torch.zeros((0, 3), dtype=torch.int64, device=rp.device)
    del tris
    if tri.shape[0] > 1 << 26:
        return None
    if r == 2:
        e = [edge_id(tri[:, 0], tri[:, 1]), edge_id(tri[:, 0], tri[:, 2]), edge_id(tri[:, 1], tri[:, 2])]
        return m, torch.cat(e), torch.cat([torch.stack([e[1], e[2]], 1), torch.stack([e[0], e[2]], 1),
                                           torch.stack([e[0], e[1]], 1)])
    if n > 1 << 20:
        return None
    key = torch.sort(tri, 1)[0]
    key = (key[:, 0] * n + key[:, 1]) * n + key[:, 2]
    names = torch.sort(key)[0]

    def tri_id(x, y, z):
        t = torch.sort(torch.stack([x, y, z], 1), 1)[0]
        return torch.searchsorted(names, (t[:, 0] * n + t[:, 1]) * n + t[:, 2])

    quads = []
    for lo in range(0, tri.shape[0], step):
        t = tri[lo:lo + step]
        j, i = _ranges(first[t[:, 2]], outs[t[:, 2]])
        x = b[j]
        ok = (edge_id(t[i, 0], x) >= 0) & (edge_id(t[i, 1], x) >= 0)
        quads.append(torch.cat([t[i[ok]], x[ok][:, None]], 1))
    q = torch.cat(quads) if quads else torch.zeros((0, 4), dtype=torch.int64, device=rp.device)
    if q.shape[0] > 1 << 26:
        return None
    ids = torch.stack([tri_id(q[:, 0], q[:, 1], q[:, 2]), tri_id(q[:, 0], q[:, 1], q[:, 3]),
                       tri_id(q[:, 0], q[:, 2], q[:, 3]), tri_id(q[:, 1], q[:, 2], q[:, 3])], 1)
    rest = [torch.cat([ids[:, :k], ids[:, k + 1:]], 1) for k in range(4)]
    return names.numel(), ids.t().reshape(-1), torch.cat(rest)


class _Exact:
    """SND by sorting every row, Definition 4 as it stands."""

    def __init__(self, incidence):
        self.n, rows, others = incidence
        order = torch.argsort(rows)
        self.rows, self.others = rows[order], others[order]
        self.ds = torch.bincount(self.rows, minlength=self.n)
        self.start = torch.cumsum(self.ds, 0) - self.ds

    def update(self, tau):
        rho = tau[self.others].amin(1) if self.others.numel() else self.rows
        big = int(tau.max()) + 1 if tau.numel() else 1
        order = torch.sort(self.rows * big + (big - 1 - rho))[0]
        rho = big - 1 - order % big
        rank = torch.arange(1, rho.numel() + 1, device=rho.device) - self.start[self.rows]
        h = torch.zeros_like(tau)
        return h.scatter_reduce_(0, self.rows, torch.minimum(rho, rank), "amax")

    def snd(self, most=1 << 30, tau=None, members=None):
        """(tau, updating passes) of at most `most` passes; members: every other r-clique keeps d_s."""
        tau, passes = self.ds.clone() if tau is None else tau, 0
        for _ in range(most):
            new = self.update(tau)
            if members is not None:
                new = torch.where(members, new, tau)
            if torch.equal(new, tau):
                break
            tau, passes = new, passes + 1
        return tau, passes


def _tau_b(x, y):
    """Kendall's tau-b of two integer sequences."""
    n = x.numel()
    x, y = x - x.min(), y - y.min()
    h = torch.bincount(x * (int(y.max()) + 1) + y, minlength=(int(x.max()) + 1) * (int(y.max()) + 1))
    h = h.reshape(int(x.max()) + 1, int(y.max()) + 1).to(torch.float64)
    if h.numel() > 1 << 24 or h.shape[0] < 2 or h.shape[1] < 2:
        return None
    pad = torch.zeros((h.shape[0] + 1, h.shape[1] + 1), dtype=torch.float64, device=h.device)
    pad[:-1, :-1] = h.flip(0, 1).cumsum(0).cumsum(1).flip(0, 1)   # at or above (a, b)
    above = pad[1:, 1:]
    discordant = pad[1:, :1] - pad[1:, :-1]
    s = float((h * (above - discordant)).sum())
    ties = [float((t * (t - 1) / 2).sum()) for t in (h.sum(1), h.sum(0))]
    all_pairs = n * (n - 1) / 2
    return s / math.sqrt((all_pairs - ties[0]) * (all_pairs - ties[1]))


def exact(case, seed):
    job = case["job"]
    if job == "batch":
        return None
    if job == "normalize":
        return _graph(case, seed)
    rp, col = _graph(case, seed)
    if (case["r"] == 2 and case["n"] > 150000) or (case["r"] == 1 and case["n"] > 1 << 21):
        return None
    incidence = _incidence(rp, col, case["r"])
    if incidence is None:
        return None
    e = _Exact(incidence)
    del incidence
    i32 = lambda t: t.to(torch.int32)  # noqa: E731
    if job == "ego":
        members = torch.zeros(e.n, dtype=torch.bool, device="cuda")
        members[_ego_members(case, rp, col, seed).to(torch.int64)] = True
        return i32(e.snd(members=members)[0])
    kappa, passes = e.snd()
    if job == "sweeps":
        early, p0 = e.snd(case["early"])
        later, p1 = e.snd(2, tau=early)
        return dict(early=i32(early), passes=p0, later=i32(later), more=p1, equal=int((later == kappa).sum()),
                    order=_tau_b(later, kappa), and_nn=i32(kappa))
    out = {mode: i32(kappa) for mode in case["modes"].split(",")}
    if "snd" in out:
        out["passes"] = passes
    if case["r"] == 3 and job == "decompose":
        for mode in case["modes"].split(","):
            out[mode] = torch.as_tensor(_results(case)).to(out[mode])
            if out[mode].numel() < kappa.numel():
                return None
            out[mode][:kappa.numel()] = i32(kappa)
    if case.get("host"):
        out = {k: v.cpu().numpy() if torch.is_tensor(v) else v for k, v in out.items()}
    return out
