"""Cubic sums in boxes of modes: every number of modes (whole and half last blocks, one to twenty boxes), pixel
ranges that end inside a stage, an odd number of ranges, and a pass over several plans, against float64 sums over the
library's own maps."""
import numpy as np
import pytest
import torch

import simgen

pytestmark = pytest.mark.gpu


def _module():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1105_2791_gb300 as M
    return M


def _reference(plan, alm, P):
    """(beta, sum of magnitudes) in float64."""
    X = plan.synthesize(alm).reshape(alm.shape[0], P, -1).double()
    _, w = plan.rings()
    W = torch.from_numpy(np.repeat(w * 2 * np.pi / plan.nphi, plan.nphi)).cuda()
    p, r, s = torch.tensor([(a, b, c) for a in range(P) for b in range(a, P) for c in range(b, P)], device="cuda").T
    out, mag = [], []
    for x in X:
        pr = torch.einsum("ax,bx,cx->abc", x * W, x, x)
        ab = torch.einsum("ax,bx,cx->abc", x.abs() * W, x.abs(), x.abs())
        out.append(pr[p, r, s])
        mag.append(ab[p, r, s])
    return torch.stack(out), torch.stack(mag)


# 17 x 64 = 1088 pixels: eight and a half stages; ranges of 1, 3 and 8 per map leave one range without a partner, end
# one inside a stage and leave the last ranges empty
@pytest.mark.parametrize("P", list(range(1, 17)))
@pytest.mark.parametrize("ctas", [1, 3, 8])
def test_every_mode_count_matches_float64(P, ctas):
    M = _module()
    L, R, nphi, maps = 16, 17, 64, 3
    basis, cl = simgen.shifted_legendre_basis(L, P), simgen.cl_model(L)
    plan = M.Plan(L, P, basis, cl, R, nphi)
    plan.set_tuning({"cubic_ctas": ctas})
    alm = torch.from_numpy(simgen.gaussian_alm(cl, maps, seed=P).astype(np.complex64)).cuda()
    beta = plan.cubic(alm)
    ref, mag = _reference(plan, alm, P)
    # chains of at most 8 + 9 + 16 rounded FP32 additions after two rounded products and the FP32 weights
    assert bool(((beta - ref).abs() <= 36 * 2.0 ** -24 * mag).all())
    plan.sync()
    plan.close()


@pytest.mark.parametrize("P", [3, 6, 10, 12, 13, 16])
def test_shared_launch_equals_each_plan(P):
    M = _module()
    plans, alms = [], []
    for L, R, nphi, maps in ((16, 17, 64, 3), (30, 33, 128, 2), (20, 21, 64, 1)):
        basis, cl = simgen.shifted_legendre_basis(L, P), simgen.cl_model(L)
        plans.append(M.Plan(L, P, basis, cl, R, nphi))
        alms.append(torch.from_numpy(simgen.gaussian_alm(cl, maps, seed=L).astype(np.complex64)).cuda())
    plans[1].set_tuning({"cubic_ctas": 5})
    batch = M.Batch(plans, schedule="shared_cubic")
    got = [b.clone() for b in batch.cubic(alms, graph=False)]
    for plan, alm, b in zip(plans, alms, got):
        assert torch.equal(plan.cubic(alm), b)
    batch.close()
    for plan in plans:
        plan.close()
