"""Kernels compiled per even number of modes: quartic sums with the per-ring Monte Carlo terms, and pair means per pixel
and per ring, for every number of modes, against float64 on the library's own maps."""
import numpy as np
import pytest
import torch

import simgen

pytestmark = pytest.mark.gpu

L, R, NPHI = 16, 37, 64             # 37 rings: more than one warp of rings, and a remainder


def _setup(P, mode):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1105_2791_gb300 as M
    basis, cl = simgen.shifted_legendre_basis(L, P), simgen.cl_model(L)
    plan = M.Plan(L, P, basis, cl, R, NPHI)
    if mode == "ring":
        plan.set_linear_mode("ring")
    sims = torch.from_numpy(simgen.gaussian_alm(cl, 7, seed=P).astype(np.complex64)).cuda()
    plan.linear_term(sims, finalize=True)
    X = plan.synthesize(sims).reshape(7, P, -1).double()
    pairs = torch.tensor([(a, b) for a in range(P) for b in range(a, P)], device="cuda").T
    return plan, sims, X, pairs


@pytest.mark.parametrize("P", list(range(1, 17)))
@pytest.mark.parametrize("mode", ["pixel", "ring"])
def test_pair_means_match_float64(P, mode):
    plan, _, X, (pa, pb) = _setup(P, mode)
    prod = X[:, pa] * X[:, pb]
    ref, mag = prod.mean(0), prod.abs().mean(0)
    if mode == "ring":
        ref, mag = (t.reshape(len(pa), R, NPHI).mean(2) for t in (ref, mag))
    # FP32 sums of at most 7 maps and 64 longitudes, rounded to FP32 once more
    assert bool(((plan.pair_mean() - ref).abs() <= (7 + 64 + 2) * 2.0 ** -24 * mag).all())
    plan.close()


@pytest.mark.parametrize("P", list(range(1, 17)))
def test_quartic_with_ring_terms_matches_float64(P):
    plan, sims, X, (pa, pb) = _setup(P, "ring")
    tau = plan.quartic(sims[:2].contiguous(), use_linear=True)
    num = torch.zeros((P, P), dtype=torch.long, device="cuda")
    num[pa, pb] = num[pb, pa] = torch.arange(len(pa), device="cuda")
    q = torch.tensor([(a, b, c, d) for a in range(P) for b in range(a, P) for c in range(b, P) for d in range(c, P)],
                     device="cuda").T
    _, w = plan.rings()
    W = torch.from_numpy(np.repeat(w * 2 * np.pi / NPHI, NPHI)).cuda()
    mean = (X[:, pa] * X[:, pb]).mean(0).reshape(len(pa), R, NPHI).mean(2, keepdim=True)
    mean = mean.expand(-1, R, NPHI).reshape(len(pa), -1)
    for b in range(2):
        Q = X[b][pa] * X[b][pb]
        T, H, K = (Q * W) @ Q.T, (mean * W) @ Q.T, (mean * W) @ mean.T
        at = lambda M, i, j, k, o: M[num[q[i], q[j]], num[q[k], q[o]]]
        ref, size = at(T, 0, 1, 2, 3), (Q.abs() * W) @ Q.abs().T
        size = at(size, 0, 1, 2, 3) + 6 * at((mean.abs() * W) @ Q.abs().T, 0, 1, 2, 3) + 3 * at((mean.abs() * W) @ mean.abs().T, 0, 1, 2, 3)
        ref = ref - sum(at(H, *i) for i in ((0, 1, 2, 3), (0, 2, 1, 3), (0, 3, 1, 2), (1, 2, 0, 3), (1, 3, 0, 2), (2, 3, 0, 1)))
        ref = ref + sum(at(K, *i) for i in ((0, 1, 2, 3), (0, 2, 1, 3), (0, 3, 1, 2)))
        # three rounded products, chains of up to 32 FP32 additions and the FP32 pair means and ring sums behind H and K;
        # the magnitudes of every mode are within a factor of the largest
        assert bool(((tau[b] - ref).abs() <= 128 * 2.0 ** -24 * size.max()).all())
    plan.close()
