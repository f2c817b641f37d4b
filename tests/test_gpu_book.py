"""A (3,4) row past 65,535 entries, whose values do not fit the 16-bit copies:
three adjacent hubs with 70,000 common neighbours.  The hub triangle is in
70,000 4-cliques and every other triangle in one, so kappa is 1 throughout."""
import numpy as np
import pytest

from paper_1704_00386_gb300 import graphs as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PAGES = 70_000


def test_nucleus_book():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_00386_gb300 import nd
    z = np.arange(3, PAGES + 3)
    src = np.concatenate([[0, 0, 1]] + [np.full(PAGES, h) for h in range(3)])
    dst = np.concatenate([[1, 2, 2], z, z, z])
    rp, col = G.to_csr(PAGES + 3, src, dst)
    inc = nd.build_incidence(torch.from_numpy(rp).cuda(), torch.from_numpy(col).cuda(), 3, 4)
    assert inc.num_r == 3 * PAGES + 1 and inc.num_incidences == 4 * PAGES
    ds = torch.ones(inc.num_r, dtype=torch.int32, device="cuda")
    kap = ds.clone()
    ds[0] = PAGES
    assert torch.equal(inc.s_degree(), ds)
    assert torch.equal(inc.iterate_k("snd", 1)[0], kap)
    for mode in ("snd", "and", "and_nn"):
        assert torch.equal(inc.iterate_k(mode, 1 << 20)[0], kap)
    # from tau = 70,000 everywhere the hub triangle keeps it for a pass: every
    # one of its 70,000 entries is read as 70,000, not as 65,535
    given = torch.full_like(ds, PAGES)
    assert torch.equal(inc.iterate_k("snd", 1, tau=given)[0], ds)
    # one entry less at 70,000: 69,999 values of 70,000 and one of 69,998
    given[1] = PAGES - 2
    want = ds.clone()
    want[0] = PAGES - 1
    assert torch.equal(inc.iterate_k("snd", 1, tau=given)[0], want)
    for mode in ("snd", "and", "and_nn"):
        assert torch.equal(inc.iterate_k(mode, 1 << 20, tau=given)[0], kap)
