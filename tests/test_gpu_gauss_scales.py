"""Gaussianisation of fields in any unit: scaled fields give scaled outputs, over
both ways of ranking, as long as their variance is a normal number."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# 48^3: 82% of the ranks lie beyond the direct tails (16384 at either end) and take the series
@pytest.mark.parametrize("scale", [1e-150, 1e-60, 1e-30, 1.0, 1e30, 1e60, 1e100, 1e145])
@pytest.mark.parametrize("ties", [False, True])
def test_values_follow_the_scale(O, scale, ties):
    from paper_1709_06350_gb300 import recon as R
    N = 48
    v = np.random.default_rng(5).standard_normal((N,) * 3)
    v = scale * (np.round(3.0 * v) if ties else v)   # ties: the radix sort
    s = R.Solver(N, float(N))
    g = s.gaussianise(torch.from_numpy(v).cuda()).cpu().numpy()
    s.close()
    ref, rank = O.gaussianise(v)
    assert np.max(np.abs(g - ref)) <= 1e-11 * v.std()   # the oracle's quantile of a probability near 1
    # the lower half: both quantiles have a few ulp, the series leaves 2^-58, and
    # the moments of 1e5 values in another order a few ulp more
    low = (rank < rank.size // 2).reshape(v.shape)
    assert np.max(np.abs(g - ref)[low]) <= 1e-13 * v.std()
    assert np.all(np.diff(g.ravel()[np.argsort(v, axis=None, kind="stable")]) > 0)
