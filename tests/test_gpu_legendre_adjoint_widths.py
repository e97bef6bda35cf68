"""Transposed FP32 Legendre sums at sizes where every channel tile is taken (from l_max = 150 on the tile goes by padded
cost alone): each width whole, ragged and one channel past its edge, without and with the filter, against the oracle;
a batch equals its maps one by one, which take other tiles, bit for bit."""
import numpy as np
import pytest
import torch

import simgen
from oracle import modal as om, sht as osh

pytestmark = pytest.mark.gpu

L, R, NPHI = 160, 163, 512


def _module():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1105_2791_gb300 as M
    return M


def _rel(a, b):
    return float(np.linalg.norm(np.ravel(a - b)) / np.linalg.norm(np.ravel(b)))


# tiles of 2 (1, 2), 8 (3, 8, 17), 16 (9, 15, 16) and 32 channels (25, 31, 32; 49 and 63 in two tiles, the second ragged)
@pytest.mark.parametrize("maps", [1, 2, 3, 8, 9, 15, 16, 17, 25, 31, 32, 49, 63])
def test_analysis_widths(maps):
    M = _module()
    plan = M.Plan(L, 1, simgen.shifted_legendre_basis(L, 1), simgen.cl_model(L), R, NPHI)
    plan.set_chunk(64)
    xi = simgen.pixel_normals(R, NPHI, maps, seed=5).astype(np.float32)
    x = torch.from_numpy(xi).cuda()
    got = plan.analyze(x)
    for b in {0, maps // 2, maps - 1}:
        assert torch.equal(plan.analyze(x[b:b + 1].contiguous())[0], got[b])
    mu, w = osh.gl_nodes(R)
    ref = osh.analyze_many(xi[-1:].astype(np.float64), L, mu, w, NPHI)
    assert _rel(got[-1].cpu().numpy(), ref[0]) <= 1e-5
    plan.close()


# whole maps fill 30, 28, 27, 22, 26, 30 and 32 channels of the widest tile (the last tile of the first three and of 5 modes
# holds fewer maps), and 14 and 16 of the next
@pytest.mark.parametrize("P,maps", [(6, 14), (7, 11), (9, 5), (11, 6), (13, 4), (5, 11), (16, 6), (7, 9), (16, 5)])
def test_filtered_gradient_widths(P, maps):
    M = _module()
    basis, cl = simgen.shifted_legendre_basis(L, P), simgen.cl_model(L)
    plan = M.Plan(L, P, basis, cl, R, NPHI)
    alm = simgen.gaussian_alm(cl, maps, seed=2).astype(np.complex64)
    g = simgen.standard_normals((maps, plan.n_max), seed=3)
    a, gd = torch.from_numpy(alm).cuda(), torch.from_numpy(g).cuda()
    got = plan.backward(a, gd)
    for b in range(maps):
        assert torch.equal(plan.backward(a[b:b + 1].contiguous(), gd[b:b + 1].contiguous())[0], got[b])
    mu, w = osh.gl_nodes(R)
    ref = om.adjoint_grad(alm[-1].astype(np.complex128), g[-1], L, osh.filter_table(basis, cl), mu, w, NPHI)
    assert _rel(got[-1].cpu().numpy(), ref) <= 1e-5
    plan.close()
