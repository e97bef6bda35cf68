"""The harmonic linear term of split-precision plans: its sum over l in blocks of pairs, for one block and several, whole
and ragged blocks and l ranges: a batch equals its maps one by one bit for bit, and the sums against float64 on the
library's own maps and pair means (the same finite sum, taken over the pixels)."""
import numpy as np
import pytest
import torch

import simgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,P,B", [(30, 1, 3), (31, 2, 2), (32, 7, 5), (63, 8, 2), (64, 10, 3), (95, 15, 2), (33, 16, 4)])
def test_harmonic_linear_sums(L, P, B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1105_2791_gb300 as M
    basis, cl = simgen.shifted_legendre_basis(L, P), simgen.cl_model(L)
    R, nphi = 3 * L // 2 + 1, 256 if 3 * L < 256 else 512
    plan = M.Plan(L, P, basis, cl, R, nphi, prec="fp16x3")
    plan.set_chunk(B)
    sims = torch.from_numpy(simgen.gaussian_alm(cl, 3, seed=P).astype(np.complex64)).cuda()
    plan.linear_term(sims, finalize=True)
    alm = torch.from_numpy(simgen.gaussian_alm(cl, B, seed=P + 1).astype(np.complex64)).cuda()
    whole = plan.cubic(alm, use_linear=True)
    assert torch.equal(whole, torch.cat([plan.cubic(alm[b:b + 1].contiguous(), use_linear=True) for b in range(B)]))

    lin = plan.cubic(alm) - whole
    X = plan.synthesize(alm).reshape(B, P, -1).double()
    _, w = plan.rings()
    mean = plan.pair_mean().double() * torch.from_numpy(np.repeat(w * 2 * np.pi / nphi, nphi)).cuda()
    G, A = torch.einsum("cx,bpx->bcp", mean, X), torch.einsum("cx,bpx->bcp", mean.abs(), X.abs())
    num = {ab: i for i, ab in enumerate((a, b) for a in range(P) for b in range(a, P))}
    trip = [(p, r, s) for p in range(P) for r in range(p, P) for s in range(r, P)]
    take = lambda T: torch.stack([T[:, num[p, r], s] + T[:, num[p, s], r] + T[:, num[r, s], p] for p, r, s in trip], 1)
    # a split-precision sum errs by about 1e-6 of its terms' size in the maps and again in the table: 1e-5 of the magnitudes
    assert bool(((lin - take(G)).abs() <= 1e-5 * take(A)).all())
    plan.close()
