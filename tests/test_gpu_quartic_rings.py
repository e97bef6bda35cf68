"""The FP64 ring products of the trispectrum in both layouts: many maps at once take eight lanes along the rings, a map
alone 32, so that a batch equals its maps one by one up to the order of FP64 sums."""
import numpy as np
import pytest
import torch

import simgen

pytestmark = pytest.mark.gpu


# 1, 2, 5, 6, 10 and 17 groups of eight pairs, the last one whole or ragged; 17 rings (a remainder of one), 24 and 37
@pytest.mark.parametrize("P,maps", [(2, 1500), (3, 1500), (5, 1500), (8, 1500), (9, 64), (12, 64), (16, 64)])
@pytest.mark.parametrize("nrings", [17, 24, 37])
def test_many_maps_equal_single_maps(P, maps, nrings):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1105_2791_gb300 as M
    L, nphi = 16, 64
    cl = simgen.cl_model(L)
    plan = M.Plan(L, P, simgen.shifted_legendre_basis(L, P), cl, nrings, nphi)
    plan.set_chunk(maps)
    plan.set_linear_mode("ring")
    alm = torch.from_numpy(simgen.gaussian_alm(cl, maps, seed=P).astype(np.complex64)).cuda()
    plan.linear_term(alm[:7].contiguous(), finalize=True)
    whole, bare = plan.quartic(alm, use_linear=True), plan.quartic(alm)
    for b in (0, 1, maps // 2, maps - 1):
        one = alm[b:b + 1].contiguous()
        assert torch.equal(plan.quartic(one)[0], bare[b])
        # nine FP64 sums of at most 37 terms, each of the size of the quartic sums: below 1e-13 of these
        assert float((plan.quartic(one, use_linear=True)[0] - whole[b]).abs().max()) <= 1e-13 * float(bare[b].abs().max())
    plan.sync()
    plan.close()
