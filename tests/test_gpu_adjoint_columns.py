"""Tensor-core adjoint pixel weights with 8, 12 and 16 columns per mode: the gradient of every number of modes against
the oracle, with 1, 4 and 5 maps (a quad of maps, a partial one) and a ragged last pixel tile."""
import numpy as np
import pytest
import torch

import simgen
from oracle import modal as om, sht as osh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", list(range(1, 17)))
@pytest.mark.parametrize("maps", [1, 5])
@pytest.mark.parametrize("prec", ["fp16x3", "3xtf32"])
def test_gradient_of_every_mode_count_matches_oracle(P, maps, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1105_2791_gb300 as M
    L, R, nphi = 14, 17, 64                                # 1088 pixels: eight and a half tiles
    basis, cl = simgen.shifted_legendre_basis(L, P), simgen.cl_model(L)
    plan = M.Plan(L, P, basis, cl, R, nphi, prec=prec)
    alm = simgen.gaussian_alm(cl, maps, seed=P).astype(np.complex64)
    g = simgen.standard_normals((maps, plan.n_max), seed=9)
    grad = plan.backward(torch.from_numpy(alm).cuda(), torch.from_numpy(g).cuda()).cpu().numpy()
    plan.sync()
    mu, w = osh.gl_nodes(R)
    filt = osh.filter_table(basis, cl)
    for b in range(maps):
        ref = om.adjoint_grad(alm[b].astype(np.complex128), g[b], L, filt, mu, w, nphi)
        assert np.linalg.norm(grad[b] - ref) <= 1e-5 * np.linalg.norm(ref)
    plan.close()
