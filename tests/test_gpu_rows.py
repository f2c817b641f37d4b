"""GPU rows at the edges of the h-index kernels, against the CPU oracle.

A power-law background gives tau many values; hub vertices (for (1,2)) and
pairs of adjacent hubs (for (2,3)) get rows of exactly the lengths where the
evaluation changes: the lane-group, warp and CTA buckets, blocks of 64 and
128 streamed entries, and histograms that hold one value per bin, several
values per bin, or need a second sweep.  Integers: every comparison is exact.
"""
import numpy as np
import pytest

import oracle
from paper_1704_00386_gb300 import graphs as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LENGTHS = (7, 8, 9, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1024, 2047, 2048, 2049, 4095, 4097, 5900)


@pytest.fixture(scope="module")
def nd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_00386_gb300 import nd as _nd
    _nd.load()
    return _nd


def _rows_graph(pairs: bool, pad: int = 0):
    n0 = 6000
    rng = np.random.default_rng(31)
    src, dst = [x.tolist() for x in G.chung_lu(n0, 2.1, 60.0 if not pairs else 24.0, seed=33)]
    n = n0
    for k in LENGTHS:
        nb = rng.choice(n0, size=k, replace=False).tolist()
        for h in ((n, n + 1) if pairs else (n,)):
            src += [h] * k
            dst += nb
        if pairs:
            src.append(n)
            dst.append(n + 1)
        n += 2 if pairs else 1
    return G.to_csr(n + pad, src, dst)


# 60,000 isolated vertices more: the build renumbers by degree class, and the
# rows of a k-core come in the order that lets a pass stop early
@pytest.mark.parametrize("r,pad", [(1, 0), (2, 0), (1, 60000), (2, 60000)])
def test_rows_at_the_edges(nd, r, pad):
    rp, col = _rows_graph(pairs=r == 2, pad=pad)
    g = oracle.Graph(rp, col, r, r + 1)
    inc = nd.build_incidence(torch.from_numpy(rp).cuda(), torch.from_numpy(col).cuda(), r, r + 1)
    ds = inc.s_degree().cpu().numpy()
    np.testing.assert_array_equal(ds, g.s_degree())
    assert set(LENGTHS) <= set(ds.tolist())
    kap = g.peel()
    tau, iters = inc.snd()
    assert iters == g.snd()[2]
    np.testing.assert_array_equal(tau.cpu().numpy(), kap)
    for k in (1, 2, 3, 4):
        tk, _ = inc.iterate_k("snd", k)
        np.testing.assert_array_equal(tk.cpu().numpy(), g.snd(max_sweeps=k)[0])
    # from a given tau the first pass counts before it searches
    t1, _ = inc.iterate_k("snd", 1)
    t3, _ = inc.iterate_k("snd", 2, tau=t1)
    np.testing.assert_array_equal(t3.cpu().numpy(), g.snd(max_sweeps=3)[0])
    for notify in (True, False):
        np.testing.assert_array_equal(inc.and_(notify=notify)[0].cpu().numpy(), kap)
    ta, _ = inc.iterate_k("and", 1 << 20, tau=t1)
    np.testing.assert_array_equal(ta.cpu().numpy(), kap)


# builds that keep the count pass's triangles as records: warps with thousands
# of triangles (whole blocks of two per lane), and with none, one or a few
@pytest.mark.parametrize("n,m", [(700, 70_000), (9000, 90_000), (40_000, 68_000)])
def test_fill_from_records(nd, n, m):
    rng = np.random.default_rng(n)
    key = np.unique(rng.integers(0, n, 3 * m) * n + rng.integers(0, n, 3 * m))
    u, v = key // n, key % n
    rp, col = G.to_csr(n, u[u < v][:m], v[u < v][:m])
    assert rp[-1] // 2 >= 1 << 16
    g = oracle.Graph(rp, col, 2, 3)
    inc = nd.build_incidence(torch.from_numpy(rp).cuda(), torch.from_numpy(col).cuda(), 2, 3)
    np.testing.assert_array_equal(inc.s_degree().cpu().numpy(), g.s_degree())
    for k in (1, 2, 3):
        np.testing.assert_array_equal(inc.iterate_k("snd", k)[0].cpu().numpy(), g.snd(max_sweeps=k)[0])
    np.testing.assert_array_equal(inc.snd()[0].cpu().numpy(), g.peel())


def test_no_storage_rows_with_hub_tables(nd):
    """The no-storage passes of a graph large enough for hub tables: lists by
    degree class, their bound, and the lists below the tables' degree."""
    n, s, d = G.rmat(14, 16, seed=61)
    rp, col = G.to_csr(n, s, d)
    assert rp[-1] >= 1 << 18
    g = oracle.ParallelSND(rp, col, 2, threads=8)
    inc = nd.build_incidence(torch.from_numpy(rp).cuda(), torch.from_numpy(col).cuda(), 2, 3, on_the_fly=True)
    for k in (1, 2, 5):
        tk, _ = inc.iterate_k("snd", k)
        np.testing.assert_array_equal(tk.cpu().numpy(), g.snd(max_sweeps=k)[0])
    t1, _ = inc.iterate_k("snd", 1)
    t3, _ = inc.iterate_k("snd", 2, tau=t1)
    np.testing.assert_array_equal(t3.cpu().numpy(), g.snd(max_sweeps=3)[0])
    kap, passes = inc.snd()
    kap = kap.cpu().numpy()
    want = g.snd()
    np.testing.assert_array_equal(kap, want[0])
    for notify in (True, False):
        np.testing.assert_array_equal(inc.and_(notify=notify)[0].cpu().numpy(), kap)
    stored = nd.build_incidence(torch.from_numpy(rp).cuda(), torch.from_numpy(col).cuda(), 2, 3)
    members = torch.arange(0, inc.num_r, 3, dtype=torch.int32, device="cuda")
    np.testing.assert_array_equal(inc.and_partial(members)[0].cpu().numpy(),
                                  stored.and_partial(members)[0].cpu().numpy())


def test_nuclei_by_triangle_ids(nd):
    """A (3,4) handle whose memory limit leaves no room for the list slots
    keeps triangle ids in its rows: the same results, fewer bytes."""
    rp, col = G.hub_graph(2000, 5, seed=71)
    drp, dcol = torch.from_numpy(rp).cuda(), torch.from_numpy(col).cuda()

    def results(inc):
        kap, passes = inc.snd()
        t2, _ = inc.iterate_k("snd", 2)
        members = torch.arange(0, inc.num_r, 5, dtype=torch.int32, device="cuda")
        out = [kap, t2, inc.and_()[0], inc.and_(notify=False)[0], inc.and_partial(members)[0], inc.s_degree()]
        return [x.cpu().numpy() for x in out], passes, inc.incidence_bytes()

    want, passes, held = results(nd.build_incidence(drp, dcol, 3, 4))
    g = oracle.Graph(rp, col, 3, 4)
    np.testing.assert_array_equal(want[0], g.peel())
    try:
        nd.set_handle_memory_limit(held - 20 * len(want[0]))
        got, passes_ids, held_ids = results(nd.build_incidence(drp, dcol, 3, 4))
    finally:
        nd.set_handle_memory_limit(0)
    assert held_ids < held - 20 * len(want[0]) and passes_ids == passes
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("r", [1, 2, 3])
def test_active_list_in_parts(nd, r):
    """AND with notification whose handle has no room for the list of active
    rows makes every pass in parts, from a sixteenth of it."""
    n, s, d = G.rmat(13 if r < 3 else 11, 12, seed=83)
    rp, col = G.to_csr(n, s, d)
    drp, dcol = torch.from_numpy(rp).cuda(), torch.from_numpy(col).cuda()
    inc = nd.build_incidence(drp, dcol, r, r + 1)
    want = inc.and_()[0].cpu().numpy()
    np.testing.assert_array_equal(want, oracle.Graph(rp, col, r, r + 1).peel())
    held = inc.incidence_bytes()
    members = torch.arange(0, inc.num_r, 7, dtype=torch.int32, device="cuda")
    part = inc.and_partial(members)[0].cpu().numpy()
    try:
        nd.set_handle_memory_limit(held - 4)
        tight = nd.build_incidence(drp, dcol, r, r + 1)
        for _ in range(3):  # the second run of a mode would take a graph
            tau, _, evals = tight.and_()
            np.testing.assert_array_equal(tau.cpu().numpy(), want)
            assert evals >= len(want)
        np.testing.assert_array_equal(tight.and_partial(members)[0].cpu().numpy(), part)
        assert tight.incidence_bytes() < held
    finally:
        nd.set_handle_memory_limit(0)
