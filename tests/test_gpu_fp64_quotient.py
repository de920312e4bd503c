"""The FP64 smoother's quotient (a reciprocal approximation refined by two Newton
steps) against division: within one ulp, over random significands, both signs
and divisors over many exponents, powers of two and their neighbours among them.

It is read off single cell updates.  With every value of theta zero but the one
above an isolated cell, A = I + H theta is diag(a, 1, 1) there, its determinant
a, the sum of its diagonal cofactors S = (1 + a) + a, and the update's step is
(h^2 / 2) tau, tau = (a - g) / S; at h = 2 the factor is exactly 2."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _divisors(kind, n, rng):
    if kind == "powers":
        S = 2.0 ** rng.integers(-30, 40, n)
        return np.where(np.arange(n) % 3 == 0, S, np.where(np.arange(n) % 3 == 1, np.nextafter(S, 0), np.nextafter(S, 1e300)))
    lo, hi = {"small": (-30, 0), "near 3": (1, 2), "large": (0, 45)}[kind]
    return rng.uniform(1.0, 2.0, n) * 2.0 ** rng.uniform(lo, hi, n).astype(int)


@pytest.mark.parametrize("kind", ["powers", "small", "near 3", "large"])
def test_quotient_is_within_an_ulp(kind):
    from paper_1709_06350_gb300 import recon as R
    N, h = 64, 2.0
    assert 3.0 * (h * h / 6.0) == 2.0
    at = np.arange(0, N, 4)                       # red cells whose stencils do not meet
    cells = np.ix_(at, at, at)
    above = np.ix_(at + 1, at, at)
    rng = np.random.default_rng(11)
    n = at.size ** 3
    S = _divisors(kind, n, rng)
    # the kernel's own roundings of a and S from theta
    theta_up = 4.0 * ((S - 1.0) * 0.5 - 1.0)
    a = theta_up * 0.25 + 1.0
    S = (1.0 + a) + a
    assert np.all(S > 0) and np.all(a + 2.0 > 0)
    # |tau| (s - tau) <= S, s = a + 2: the step is kept
    tau = rng.uniform(0.05, 0.4, n) * np.where(rng.random(n) < 0.5, -1.0, 1.0) * np.minimum(S / (a + 2.0), 1.0)
    g = a - S * tau
    F = a - g
    theta, rhs = np.zeros((N, N, N)), np.ones((N, N, N))
    theta[above] = theta_up.reshape((at.size,) * 3)
    rhs[cells] = g.reshape((at.size,) * 3)
    t = torch.from_numpy(theta).cuda()
    R.recon_step_sweep(t, torch.from_numpy(rhs).cuda(), 0.0, h)
    got = t.cpu().numpy()[cells].ravel() / 2.0
    want = F / S
    assert np.all(np.abs(got - want) <= np.spacing(np.abs(want)))
    assert np.mean(got == want) > 0.5
