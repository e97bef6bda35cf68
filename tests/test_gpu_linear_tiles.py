"""The FP32 plan's linear-term sums: every tile of the product (64 x 64, 32 x 32 and the chain kernel's 16 x 16) forms
each output by the same chain of multiply-adds, so a batch equals its maps one by one, bit for bit; and the sums
against float64 on the library's own maps and pair means."""
import numpy as np
import pytest
import torch

import simgen

pytestmark = pytest.mark.gpu


def _plan(L, P, R, nphi, maps, seed):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1105_2791_gb300 as M
    basis, cl = simgen.shifted_legendre_basis(L, P), simgen.cl_model(L)
    plan = M.Plan(L, P, basis, cl, R, nphi)
    plan.set_chunk(maps)
    sims = torch.from_numpy(simgen.gaussian_alm(cl, 3, seed=seed).astype(np.complex64)).cuda()
    plan.linear_term(sims, finalize=True)
    alm = torch.from_numpy(simgen.gaussian_alm(cl, maps, seed=seed + 1).astype(np.complex64)).cuda()
    return plan, alm


# (16 modes, 8 maps: 64 x 64 against 32 x 32 for one map), (3 modes, 60 maps: 32 x 32 against the chain kernel),
# and small grids on the chain kernel alone with ragged row and column tiles, one and several splits
@pytest.mark.parametrize("L,P,R,nphi,maps", [(20, 16, 260, 8192, 8), (20, 3, 260, 8192, 60), (20, 7, 23, 64, 5),
                                             (30, 1, 33, 1024, 3), (30, 16, 70, 1024, 2)])
def test_linear_term_tiles_agree_bit_for_bit(L, P, R, nphi, maps):
    plan, alm = _plan(L, P, R, nphi, maps, seed=31)
    whole = plan.cubic(alm, use_linear=True)
    single = torch.cat([plan.cubic(alm[b:b + 1].contiguous(), use_linear=True) for b in range(maps)])
    assert torch.equal(whole, single)
    plan.close()


@pytest.mark.parametrize("L,P,R,nphi,maps", [(20, 16, 260, 8192, 8), (20, 3, 260, 8192, 60), (20, 7, 23, 64, 5)])
def test_linear_term_matches_float64(L, P, R, nphi, maps):
    plan, alm = _plan(L, P, R, nphi, maps, seed=41)
    lin = plan.cubic(alm) - plan.cubic(alm, use_linear=True)
    M = plan.synthesize(alm).reshape(maps, P, -1).double()
    mean = plan.pair_mean().double()
    _, w = plan.rings()
    W = torch.from_numpy(np.repeat(w * 2 * np.pi / nphi, nphi)).cuda()
    G = torch.einsum("cx,bpx->bcp", mean * W, M)
    A = torch.einsum("cx,bpx->bcp", (mean * W).abs(), M.abs())
    order = [(a, b) for a in range(P) for b in range(a, P)]
    num = {ab: i for i, ab in enumerate(order)}
    at = lambda T, a, b, c: T[:, num[min(a, b), max(a, b)], c]
    trip = [(p, r, s) for p in range(P) for r in range(p, P) for s in range(r, P)]
    ref = torch.stack([at(G, p, r, s) + at(G, p, s, r) + at(G, r, s, p) for p, r, s in trip], 1)
    bound = torch.stack([at(A, p, r, s) + at(A, p, s, r) + at(A, r, s, p) for p, r, s in trip], 1)
    # a chain of K rounded FP32 additions errs by about sqrt(K) 2^-24 of the sum of magnitudes; K <= 16,448 pixels a split
    assert bool(((lin - ref).abs() <= 8 * 128.3 * 2.0 ** -24 * bound).all())
    plan.close()
