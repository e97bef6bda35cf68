"""The synthesis ring transform with tiled copies: one, two and the most row tiles per parity, ring counts that leave a
partial block of ring pairs, odd and even, against the 8192-point transform (which fetches its rows itself) at the
shared longitudes."""
import numpy as np
import pytest
import torch

import simgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nphi,lmax", [(256, 7), (256, 127), (512, 254), (512, 255), (1024, 256), (1024, 511), (2048, 300),
                                       (2048, 1023), (4096, 255), (4096, 511)])
@pytest.mark.parametrize("extra", [1, 2, 37])
def test_tiled_rows_match_the_longest_transform(nphi, lmax, extra):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1105_2791_gb300 as M
    P, R = 2, lmax + extra
    basis, cl = simgen.shifted_legendre_basis(lmax, P), simgen.cl_model(lmax)
    alm = torch.from_numpy(simgen.gaussian_alm(cl, 2, seed=lmax).astype(np.complex64)).cuda()
    out = []
    for n in (nphi, 8192):
        plan = M.Plan(lmax, P, basis, cl, R, n)
        out.append(plan.synthesize(alm)[..., :: n // nphi].clone())
        plan.sync()
        plan.close()
    # two FP32 transforms of the same coefficients: the accepted error of a map
    assert float((out[0] - out[1]).abs().max()) <= 1e-5 * float(out[1].abs().max())
