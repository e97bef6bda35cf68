"""The solve's own division and square root (corrected products, k_solve.cu) against IEEE division and square root, bit
for bit: each is within 2^-85 of the exact value before its one rounding, so a different last bit has odds of 2^-32
per value.  Random, extreme and subnormal operands, and the paths that fall back to `/` and sqrt."""
import numpy as np
import pytest
import torch

import simgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def plan():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1105_2791_gb300 as M
    L, P = 8, 16
    p = M.Plan(L, P, simgen.shifted_legendre_basis(L, P), simgen.cl_model(L), L + 1, 32)
    yield p
    p.close()


# scales at which squares and their sums stay exact, and one (2^511) at which they are infinite
@pytest.mark.parametrize("sims", [2, 3, 7, 10, 1000])
@pytest.mark.parametrize("exponent", [0, -480, 480, 511])
def test_covariance_divisions(plan, sims, exponent):
    """zeta = ((S2 - S1 S1^T / N) / (N - 1)) / 6 of whole numbers times a power of two: both sums are exact."""
    rng = np.random.default_rng(sims)
    low = 0 if exponent == 511 else -1000                  # no infinities of both signs
    beta = np.ldexp(rng.integers(low, 1001, (sims, plan.n_max)).astype(np.float64), exponent)
    plan.reset()
    plan.cov_accumulate(torch.from_numpy(beta).cuda())
    with np.errstate(over="ignore", invalid="ignore"):
        S1, S2 = beta.sum(0), beta.T @ beta
        ref = ((S2 - S1[:, None] * S1[None, :] / sims) / (sims - 1.0)) / 6.0
    assert np.array_equal(plan.zeta(), ref, equal_nan=True)
    plan.reset()


def _rotated(plan, zeta0, x):
    return plan.bivector_rotate(zeta0, np.zeros(plan.n_max), torch.from_numpy(x[None, :]).cuda()).cpu().numpy()[0]


@pytest.mark.parametrize("kind", ["near one", "any exponent", "even and odd exponents", "largest and smallest", "subnormal"])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_pivot_roots(plan, kind, seed):
    """A diagonal covariance: L^-1 x = x / sqrt(d), the division by `/`."""
    n, rng = plan.n_max, np.random.default_rng(seed)
    m = 1.0 + rng.random(n)
    d = {"near one": 1.0 + (rng.integers(-40, 41, n) * 2.0 ** -52),
         "any exponent": np.ldexp(m, rng.integers(-1021, 1023, n)),
         "even and odd exponents": np.ldexp(np.nextafter(np.where(rng.random(n) < 0.5, 1.0, 2.0), rng.choice([0.0, 4.0], n)), rng.integers(-3, 4, n)),
         "largest and smallest": rng.choice([np.finfo(float).max, np.finfo(float).tiny, np.nextafter(np.finfo(float).tiny, 1.0)], n),
         "subnormal": np.ldexp(m, rng.integers(-1073, -1022, n))}[kind]
    assert np.array_equal(_rotated(plan, np.diag(d), np.ones(n)), 1.0 / np.sqrt(d))


@pytest.mark.parametrize("exponent", [0, -900, 400])
@pytest.mark.parametrize("d0", [2.0, 3.0, 1.0 / 3.0, 1e300, 1e-300, 1.0 - 2.0 ** -53])
def test_column_divisions(plan, exponent, d0):
    """First column v over a pivot d0, the other pivots so large that nothing else reaches a result: with x = (sqrt(d0),
    0, ...) row r of L^-1 x is -(v_r / sqrt(d0)) / 2^k.  Rows 1 to 31 are the diagonal block's, the others the panel's."""
    n, rng = plan.n_max, np.random.default_rng(exponent + 1000)
    v = np.ldexp(rng.standard_normal(n), exponent)
    v[[5, 40]] = 0.0
    root = np.sqrt(d0)
    k = max(0, int(np.ceil(np.log2(max(np.abs(v / root).max(), 1e-300)))) + 80)
    if k > 500:
        pytest.skip("the other pivots would leave the range")
    zeta0 = np.diag(np.full(n, np.ldexp(1.0, 2 * k)))
    zeta0[:, 0] = zeta0[0, :] = v
    zeta0[0, 0] = d0
    x = np.zeros(n)
    x[0] = root
    got = _rotated(plan, zeta0, x)
    assert got[0] == 1.0
    assert np.array_equal(-np.ldexp(got[1:], k), (v / root)[1:])
