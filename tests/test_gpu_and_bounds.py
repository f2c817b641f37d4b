"""AND between kappa and SND, pass by pass, on rows that need several readings.

AND lowers tau in place, so after k passes kappa <= tau_AND_k <= tau_SND_k
(Thm. 1 and the remark after Alg. 3), whatever the schedule of the blocks; and
its result is a fixed point, which one more pass of SND leaves as it is.
Integers: every comparison is exact."""
import numpy as np
import pytest

import oracle
from paper_1704_00386_gb300 import graphs as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# k-core rows up to the CTA's, renumbered by degree class; k-truss and nucleus
# rows up to the warp's
@pytest.mark.parametrize("r,scale,otf", [(1, 17, False), (2, 14, False), (2, 14, True), (3, 11, False)])
def test_and_stays_between_kappa_and_snd(r, scale, otf):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_00386_gb300 import nd
    n, s, d = G.rmat(scale, 16, seed=91 + r)
    rp, col = G.to_csr(n, s, d)
    inc = nd.build_incidence(torch.from_numpy(rp).cuda(), torch.from_numpy(col).cuda(), r, r + 1, on_the_fly=otf)
    assert int(inc.s_degree().max()) > (2048 if r == 1 else 64)
    kap, _ = inc.snd()
    np.testing.assert_array_equal(kap.cpu().numpy(), oracle.decompose(rp, col, r, r + 1))
    for k in range(1, 9):
        top, _ = inc.iterate_k("snd", k)
        for mode in ("and", "and_nn"):
            tau, _ = inc.iterate_k(mode, k)
            assert bool((kap <= tau).all()) and bool((tau <= top).all()), (mode, k)
    for _ in range(10):
        tau, _, _ = inc.and_()
        assert torch.equal(tau, kap)
    assert torch.equal(inc.iterate_k("snd", 1, tau=tau)[0], tau)
