"""The forward FP32 Legendre sums in every launch shape (one or two maps per thread, one, two or four warps along the maps)
give each map what it gives alone, bit for bit."""
import numpy as np
import pytest
import torch

import simgen

pytestmark = pytest.mark.gpu


# few warps (one map per thread), then enough for two: 2 maps; 3, 4, 9, 12 (two warps along the maps); 5, 8, 13, 16 (four)
@pytest.mark.parametrize("lmax,nrings,nphi,batches", [(20, 33, 64, (2, 3, 9)), (90, 513, 256, (2, 3, 4, 5, 8, 9, 12, 13, 16)),
                                                      (150, 160, 512, (9, 12))])
@pytest.mark.parametrize("P", [2, 7, 12, 16])
def test_every_shape_equals_single_maps(lmax, nrings, nphi, batches, P):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1105_2791_gb300 as M
    cl = simgen.cl_model(lmax)
    plan = M.Plan(lmax, P, simgen.shifted_legendre_basis(lmax, P), cl, nrings, nphi)
    alm = torch.from_numpy(simgen.gaussian_alm(cl, max(batches), seed=P).astype(np.complex64)).cuda()
    single = torch.cat([plan.synthesize(alm[b:b + 1].contiguous()) for b in range(max(batches))])
    for n in batches:
        assert torch.equal(plan.synthesize(alm[:n].contiguous()), single[:n])
    plan.sync()
    plan.close()
