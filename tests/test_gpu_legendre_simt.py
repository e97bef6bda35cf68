"""Forward FP32 Legendre sums: every split of a block over maps and ring pairs gives each map the same chain of
operations (a batch equals its maps one by one, bit for bit), and the maps agree with the oracle."""
import numpy as np
import pytest
import torch

import simgen
from oracle import sht as osh

pytestmark = pytest.mark.gpu


# rings: fewer than a warp, one and a half warps; orders of 1 .. 131 rows: shorter than eight, around the 64-row chunk
@pytest.mark.parametrize("lmax,nrings,nphi", [(2, 3, 16), (64, 65, 256), (130, 150, 512)])
@pytest.mark.parametrize("P", [1, 4, 6, 9, 12, 13, 16])
def test_batches_equal_single_maps_and_oracle(lmax, nrings, nphi, P):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1105_2791_gb300 as M
    basis, cl = simgen.shifted_legendre_basis(lmax, P), simgen.cl_model(lmax)
    plan = M.Plan(lmax, P, basis, cl, nrings, nphi)
    plan.set_chunk(9)
    alm = simgen.gaussian_alm(cl, 9, seed=lmax + P).astype(np.complex64)
    a = torch.from_numpy(alm).cuda()
    single = torch.cat([plan.synthesize(a[b:b + 1].contiguous()) for b in range(9)])
    for n in (2, 3, 4, 5, 9):
        assert torch.equal(plan.synthesize(a[:n].contiguous()), single[:n])
    mu, _ = osh.gl_nodes(nrings)
    filt = osh.filter_table(basis, cl)
    for b in (0, 8):
        ref = osh.synthesize(alm[b].astype(np.complex128), lmax, filt, mu, nphi)
        assert np.max(np.abs(single[b].cpu().numpy() - ref)) <= 1e-5 * np.max(np.abs(ref))
    plan.close()
