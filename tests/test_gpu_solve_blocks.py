"""The panelled Cholesky with carried rows and the blocked back substitution: every number of modes from 1 to 816
(all remainders of the 32-column panels that occur), few and many right-hand sides, against float64 on the host, and
a pivot that fails in a later panel."""
import numpy as np
import pytest
import torch

import simgen

pytestmark = pytest.mark.gpu


def _plan(P):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1105_2791_gb300 as M
    L = 8
    return M, M.Plan(L, P, simgen.shifted_legendre_basis(L, P), simgen.cl_model(L), L + 1, 32)


@pytest.mark.parametrize("P", list(range(1, 17)))
@pytest.mark.parametrize("B", [0, 1, 31, 300])
def test_solve_and_weights_match_float64(P, B):
    M, plan = _plan(P)
    n = plan.n_max
    mix = simgen.random_modes_matrix(n, seed=P)
    sims = simgen.standard_normals((2 * n + 10, n), seed=50 + P) @ mix.T
    alpha, beta = simgen.standard_normals(n, seed=3), simgen.standard_normals((max(B, 1), n), seed=4) @ mix.T
    plan.cov_accumulate(torch.from_numpy(sims).cuda())
    zeta = np.atleast_2d(np.cov(sims.T)) / 6.0
    fnl, sigma = plan.solve(alpha, torch.from_numpy(beta).cuda() if B else None)
    w, sigma_w = plan.fnl_weights(alpha)
    x = np.linalg.solve(zeta, alpha)
    norm = alpha @ x
    # condition numbers stay below 1e4 here: rounding of n-term FP64 sums times that is under 1e-10
    assert np.linalg.cond(zeta) < 1e4
    assert abs(sigma - np.sqrt(6.0 / norm)) <= 1e-10 * sigma and sigma_w == sigma
    assert np.linalg.norm(w.cpu().numpy() - x / norm) <= 1e-10 * np.linalg.norm(x / norm)
    if len(fnl):
        ref = beta[:len(fnl)] @ x / norm
        assert np.linalg.norm(fnl - ref) <= 1e-10 * np.linalg.norm(ref)
    plan.close()


@pytest.mark.parametrize("bad", [0, 31, 32, 70, 83])
def test_failing_pivot_in_any_panel_is_reported_and_cleared(bad):
    M, plan = _plan(7)                                     # 84 modes: three panels, the last of 20 columns
    n = plan.n_max
    bt, x = np.zeros(n), torch.ones((2, n), dtype=torch.float64, device="cuda")
    zeta0 = np.diag(1.0 + np.arange(n))
    broken = zeta0.copy()
    broken[bad, bad] = -1.0
    with pytest.raises(M.ModalError) as e:
        plan.bivector_rotate(broken, bt, x)
    assert e.value.status == M.MODAL_ENOTPD
    out = plan.bivector_rotate(zeta0, bt, x)
    ref = 1.0 / np.sqrt(1.0 + np.arange(n))
    assert np.allclose(out.cpu().numpy(), ref, rtol=1e-14, atol=0)
    plan.close()
