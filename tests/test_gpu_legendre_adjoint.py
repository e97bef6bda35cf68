"""Transposed Legendre sums in channel tiles: every tile width and its edges (channels per block, rows of one
parity, ring pairs per stage) against the oracle, and the pair-mean table built in several groups of rows."""
import numpy as np
import pytest
import torch

import simgen
from oracle import modal as om, sht as osh

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.linalg.norm(np.ravel(a - b)) / np.linalg.norm(np.ravel(b)))


def _module():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1105_2791_gb300 as M
    return M


# lmax 2 (fewer rows than a tile), 127 and 128 (63 / 64 / 65 rows of one parity), ring pairs 2, 64 and 65;
# 1, 2 | 3, 8 | 9, 32, 33 channels: one, the edge and one past the edge of each tile width
@pytest.mark.parametrize("lmax,nrings,nphi", [(2, 3, 16), (127, 128, 256), (128, 129, 512)])
@pytest.mark.parametrize("maps", [1, 2, 3, 8, 9, 32, 33])
def test_analysis_tiles_match_oracle(lmax, nrings, nphi, maps):
    M = _module()
    plan = M.Plan(lmax, 1, simgen.shifted_legendre_basis(lmax, 1), simgen.cl_model(lmax), nrings, nphi)
    plan.set_chunk(maps)
    xi = simgen.pixel_normals(nrings, nphi, maps, seed=5).astype(np.float32)
    got = plan.analyze(torch.from_numpy(xi).cuda()).cpu().numpy()
    mu, w = osh.gl_nodes(nrings)
    ref = osh.analyze_many(xi.astype(np.float64), lmax, mu, w, nphi)
    for b in range(maps):
        assert _rel(got[b], ref[b]) <= 1e-5
    plan.close()


@pytest.mark.parametrize("P,maps", [(1, 1), (2, 1), (3, 2), (8, 1), (9, 1), (6, 6), (16, 3)])
def test_fp32_gradient_tiles_match_oracle(P, maps):
    """The filtered form: the P channels of each map are summed inside a block (several maps per block)."""
    M = _module()
    L, R, nphi = 20, 22, 64
    basis, cl = simgen.shifted_legendre_basis(L, P), simgen.cl_model(L)
    plan = M.Plan(L, P, basis, cl, R, nphi)
    alm = simgen.gaussian_alm(cl, maps, seed=2).astype(np.complex64)
    g = simgen.standard_normals((maps, plan.n_max), seed=3)
    got = plan.backward(torch.from_numpy(alm).cuda(), torch.from_numpy(g).cuda()).cpu().numpy()
    mu, w = osh.gl_nodes(R)
    filt = osh.filter_table(basis, cl)
    for b in range(maps):
        ref = om.adjoint_grad(alm[b].astype(np.complex128), g[b], L, filt, mu, w, nphi)
        assert _rel(got[b], ref) <= 1e-5
    plan.close()


def test_pair_mean_table_in_groups_of_rows():
    """A workspace of one map holds P of the P (P + 1) / 2 pair-mean rows: the table is built in groups and equals
    the one built at once, bit for bit."""
    M = _module()
    L, P, R, nphi = 40, 7, 41, 128
    basis, cl = simgen.shifted_legendre_basis(L, P), simgen.cl_model(L)
    sims = torch.from_numpy(simgen.gaussian_alm(cl, 4, seed=7).astype(np.complex64)).cuda()
    alm = torch.from_numpy(simgen.gaussian_alm(cl, 1, seed=8).astype(np.complex64)).cuda()
    out = []
    for chunk in (1, 8):
        plan = M.Plan(L, P, basis, cl, R, nphi, prec="fp16x3")
        plan.linear_term(sims)
        plan.set_chunk(chunk)
        plan.linear_term(None, finalize=True)
        beta = plan.cubic(alm, use_linear=True)
        grad = plan.backward(alm, torch.ones_like(beta), use_linear=True)
        out.append((beta.cpu(), grad.cpu()))
        plan.close()
    assert torch.equal(out[0][0], out[1][0])
    assert torch.equal(out[0][1], out[1][1])
