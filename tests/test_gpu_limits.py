"""Handles at their memory limit: the library does without what it only keeps to
be faster, and what ran without those arrays still runs."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1704_00386_gb300 import graphs as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_00386_gb300 import nd as _nd
    _nd.load()
    return _nd


def _cycle(n):
    v = np.arange(n)
    return G.to_csr(n, v, np.roll(v, -1))


@pytest.mark.parametrize("r,mode", [(1, "snd"), (1, "and_nn"), (2, "snd"), (2, "and_nn")])
def test_list_of_one_tile_is_the_run_s_own(nd, r, mode):
    """A batch whose rows all lie in one bucket and fit one tile: a run without
    room for the list on the handle has all of it as scratch.  Later runs must
    not use that scratch again."""
    graphs = [_cycle(n) if r == 1 else G.complete_graph(n % 4 + 4) for n in range(9, 60)]
    graphs = [tuple(torch.from_numpy(x).cuda() for x in g) for g in graphs]

    def run(inc):
        return (inc.snd()[0] if mode == "snd" else inc.and_(notify=False)[0]).cpu().numpy()

    inc, _ = nd.build_incidence_batch(graphs, r, r + 1)
    assert inc.num_r <= 2048
    want = run(inc)
    np.testing.assert_array_equal(want, inc.s_degree().cpu().numpy())  # cycles and cliques are their own nuclei
    held = inc.incidence_bytes()
    other = G.hub_graph(3000, 6, seed=205)
    core = oracle.decompose(*other, 1, 2)
    try:
        nd.set_handle_memory_limit(held - 4)
        tight, _ = nd.build_incidence_batch(graphs, r, r + 1)
        for _ in range(4):
            np.testing.assert_array_equal(run(tight), want)
            nd.set_handle_memory_limit(0)
            between = nd.build_incidence(*other, 1, 2)  # takes the memory that runs have given back
            np.testing.assert_array_equal(between.snd()[0], core)
            nd.set_handle_memory_limit(held - 4)
        assert tight.incidence_bytes() <= held - 4
    finally:
        nd.set_handle_memory_limit(0)


@pytest.mark.parametrize("r,scale", [(1, 16), (1, 9), (2, 13), (2, 8), (3, 10), (3, 6)])
def test_and_leaves_room_for_the_other_modes(nd, r, scale):
    """The list of active rows, and the frontiers of a small handle, give way to
    what another mode cannot do without, in whatever order the modes come."""
    n, s, d = G.rmat(scale, 8, seed=17 + r)
    g = [torch.from_numpy(x).cuda() for x in G.to_csr(n, s, d)]
    inc = nd.build_incidence(*g, r, r + 1)
    kap = inc.snd()[0]
    one = inc.iterate_k("snd", 1)[0]
    inc.and_(notify=False)
    held = inc.incidence_bytes()  # with all that SND and AND need
    try:
        nd.set_handle_memory_limit(held)
        for order in (("and", "snd", "and_nn", "and"), ("and_nn", "and", "snd"), ("snd", "and", "snd", "and")):
            tight = nd.build_incidence(*g, r, r + 1)
            for mode in order:
                for _ in range(3):  # the later runs take graphs
                    assert torch.equal(tight.iterate_k(mode, 1 << 20)[0], kap), (order, mode)
            assert torch.equal(tight.iterate_k("snd", 1)[0], one)
            assert tight.incidence_bytes() <= held
            nd.set_handle_memory_limit(0)  # room for the spare arrays again
            assert torch.equal(tight.and_()[0], kap)
            nd.set_handle_memory_limit(held)
            assert torch.equal(tight.and_()[0], kap) and torch.equal(tight.snd()[0], kap)
            tight.free()
    finally:
        nd.set_handle_memory_limit(0)


def test_hub_tables_are_counted_and_give_way(nd):
    """A handle without storage keeps the hub tables that its first long run
    builds; they count in its bytes, are left out where its limit has no room,
    and go where another mode needs theirs.  Short questions build none."""
    n, s, d = G.rmat(14, 16, seed=61)
    rp, col = G.to_csr(n, s, d)
    g = [torch.from_numpy(x).cuda() for x in (rp, col)]
    new = lambda: nd.build_incidence(*g, 2, 3, on_the_fly=True)  # noqa: E731
    inc = new()
    few = torch.arange(0, 10, dtype=torch.int32, device="cuda")
    part = inc.and_partial(few)[0]
    bare = inc.incidence_bytes()  # what AND needs
    snd_more = 4 * inc.num_r + 2 * int(rp[-1])  # and SND: the second tau and its copy
    kap, passes = inc.snd()
    tables = inc.incidence_bytes() - bare - snd_more
    assert 8 * rp[-1] < tables <= 8 * rp[-1] + 4 * n + (128 << 20)
    assert torch.equal(inc.and_()[0], kap) and torch.equal(inc.and_partial(few)[0], part)
    assert inc.incidence_bytes() == bare + snd_more + tables  # built once
    try:
        for room in (bare + snd_more, bare + tables, bare + tables + snd_more // 2, bare + tables + snd_more):
            nd.set_handle_memory_limit(room)
            tight = new()
            for _ in range(2):
                assert torch.equal(tight.and_()[0], kap)
                assert torch.equal(tight.and_partial(few)[0], part)
                tau, it = tight.snd()
                assert torch.equal(tau, kap) and it == passes
            assert tight.incidence_bytes() == (room if room == bare + tables + snd_more else bare + snd_more)
            tight.free()
    finally:
        nd.set_handle_memory_limit(0)
    # rows of few triangles: none either
    rng = np.random.default_rng(5)
    rp, col = G.to_csr(20000, rng.integers(0, 20000, 300_000), rng.integers(0, 20000, 300_000))
    grown = []
    for otf in (True, False):
        inc = nd.build_incidence(rp, col, 2, 3, on_the_fly=otf)
        bare = inc.incidence_bytes()
        np.testing.assert_array_equal(inc.snd()[0], oracle.decompose(rp, col, 2, 3))
        grown.append(inc.incidence_bytes() - bare)
    assert grown[0] == grown[1]  # the state of SND alone


def _pool_bytes():
    """Bytes in use in the memory pool that the library allocates from."""
    cu = ctypes.CDLL("libcuda.so.1")
    dev, pool, used = ctypes.c_int(), ctypes.c_void_p(), ctypes.c_uint64()
    torch.cuda.synchronize()
    assert cu.cuDeviceGet(ctypes.byref(dev), torch.cuda.current_device()) == 0
    assert cu.cuDeviceGetMemPool(ctypes.byref(pool), dev) == 0
    assert cu.cuMemPoolGetAttribute(pool, 7, ctypes.byref(used)) == 0  # CU_MEMPOOL_ATTR_USED_MEM_CURRENT
    return used.value


@pytest.mark.parametrize("r", [1, 2, 3])
def test_a_refused_build_frees_what_it_took(nd, r):
    """Builds under limits from nothing to what the handle holds, so that they
    fail at one allocation after the other; 65,536 vertices are renumbered."""
    n, s, d = G.rmat(16, 4, seed=29)
    g = [torch.from_numpy(x).cuda() for x in G.to_csr(n, s, d)]
    before = _pool_bytes()
    inc = nd.build_incidence(*g, r, r + 1)
    held = inc.incidence_bytes()
    inc.free()
    assert _pool_bytes() == before
    refused = 0
    try:
        for k in range(1, 65):
            nd.set_handle_memory_limit(held * k // 64)
            try:
                nd.build_incidence(*g, r, r + 1).free()
            except nd.NDError as e:
                assert e.status == nd.ND_E_NOMEM
                refused += 1
            assert _pool_bytes() == before, k
    finally:
        nd.set_handle_memory_limit(0)
    assert 32 <= refused < 64


class _PoolProps(ctypes.Structure):
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int), ("location_type", ctypes.c_int),
                ("location_id", ctypes.c_int), ("security", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


class _small_pool:
    """The library's allocations come from a pool of at most max_size bytes:
    a device without memory, as the library sees it."""

    def __init__(self, max_size):
        self.cu, self.dev, self.pool = ctypes.CDLL("libcuda.so.1"), ctypes.c_int(), ctypes.c_void_p()
        torch.cuda.synchronize()
        assert self.cu.cuDeviceGet(ctypes.byref(self.dev), torch.cuda.current_device()) == 0
        props = _PoolProps(alloc_type=1, location_type=1, location_id=self.dev.value, max_size=max_size)
        assert self.cu.cuMemPoolCreate(ctypes.byref(self.pool), ctypes.byref(props)) == 0

    def __enter__(self):
        self.old = ctypes.c_void_p()
        assert self.cu.cuDeviceGetMemPool(ctypes.byref(self.old), self.dev) == 0
        assert self.cu.cuDeviceSetMemPool(self.dev, self.pool) == 0

    def __exit__(self, *exc):
        torch.cuda.synchronize()
        assert self.cu.cuDeviceSetMemPool(self.dev, self.old) == 0
        assert self.cu.cuMemPoolDestroy(self.pool) == 0


def test_nuclei_without_memory_for_the_slots(nd):
    """A (3,4) build on a device with room for triangle ids, but not for list
    slots, keeps ids.  3.4M triangles of a complete tripartite graph, in no
    4-clique, and ten cliques of 20."""
    a, k = 150, 20
    part = [np.arange(a) + i * a for i in range(3)]
    pairs = [np.meshgrid(part[i], part[j]) for i, j in ((0, 1), (0, 2), (1, 2))]
    up = np.triu_indices(k, 1)
    src = np.concatenate([p[0].ravel() for p in pairs] + [3 * a + c * k + up[0] for c in range(10)])
    dst = np.concatenate([p[1].ravel() for p in pairs] + [3 * a + c * k + up[1] for c in range(10)])
    g = [torch.from_numpy(x).cuda() for x in G.to_csr(3 * a + 10 * k, src, dst)]
    inc = nd.build_incidence(*g, 3, 4)
    want = np.concatenate([np.zeros(a ** 3, np.int32), np.full(10 * k * (k - 1) * (k - 2) // 6, k - 3, np.int32)])
    np.testing.assert_array_equal(inc.snd()[0].cpu().numpy(), want)
    held = inc.incidence_bytes()
    inc.free()
    outcomes = []
    for mb in range(384, 64, -8):
        with _small_pool(mb << 20):
            try:
                inc = nd.build_incidence(*g, 3, 4)
            except nd.NDError as e:
                assert e.status == nd.ND_E_NOMEM
                outcomes.append("refused")
                assert _pool_bytes() == 0
                continue
            try:
                for tau in (inc.and_()[0], inc.snd()[0]):
                    np.testing.assert_array_equal(tau.cpu().numpy(), want)
                # ids hold neither the slots (24 B a triangle) nor their 16-bit copies
                outcomes.append("ids" if inc.incidence_bytes() < held - 24 * len(want) else "slots")
            except nd.NDError as e:
                assert e.status == nd.ND_E_NOMEM
                outcomes.append("built only")
            inc.free()
    assert outcomes[0] == "slots" and outcomes[-1] == "refused"
    assert "ids" in outcomes, outcomes
