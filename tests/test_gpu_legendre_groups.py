"""Tensor-core Legendre sums in groups of equally many maps: ragged batches (groups of fewer maps than the plan's
largest, columns padded to the MMA's width) give each map what it gives alone, and the FP32 plan's sums."""
import numpy as np
import pytest
import torch

import simgen

pytestmark = pytest.mark.gpu


# batches of one, two and three groups of up to eight maps; 2 P G a multiple of 16 or not, and the widest (16 modes)
@pytest.mark.parametrize("P,maps", [(1, 1), (1, 11), (2, 3), (3, 9), (5, 7), (7, 5), (9, 13), (10, 9), (12, 17), (16, 8), (16, 12)])
@pytest.mark.parametrize("prec", ["fp16x3", "bf16x3", "3xtf32"])
def test_ragged_groups(P, maps, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1105_2791_gb300 as M
    L, R, nphi = 45, 47, 256
    basis, cl = simgen.shifted_legendre_basis(L, P), simgen.cl_model(L)
    plans = [M.Plan(L, P, basis, cl, R, nphi, prec=p) for p in (prec, "fp32")]
    for plan in plans:
        plan.set_chunk(maps)
    alm = torch.from_numpy(simgen.gaussian_alm(cl, maps, seed=P).astype(np.complex64)).cuda()
    g = torch.from_numpy(simgen.standard_normals((maps, plans[0].n_max), seed=9)).cuda()
    whole, ref = (plan.synthesize(alm) for plan in plans)
    grad, grad_ref = (plan.backward(alm, g) for plan in plans)
    for b in range(maps):
        one = alm[b:b + 1].contiguous()
        assert torch.equal(plans[0].synthesize(one)[0], whole[b])
        assert torch.equal(plans[0].backward(one, g[b:b + 1].contiguous())[0], grad[b])
        # three products of bf16 leave 2^-16 of each term, of fp16 or tf32 2^-21, and the FP32 sums a few 1e-7
        tol = 1e-4 if prec == "bf16x3" else 1e-5
        for x, y in ((whole[b], ref[b]), (grad[b], grad_ref[b])):
            assert float((x - y).abs().max()) <= tol * float(y.abs().max())
    for plan in plans:
        plan.sync()
        plan.close()
