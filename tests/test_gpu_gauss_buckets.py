"""Gaussianisation's bucket ranks and the device's choice between them and the
radix sort, over the fields that decide it: the output orders like a stable
sort's ranks on all of them, and its values are the quantiles' (the bound of
the repository's parity test)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def fields(N):
    rng = np.random.default_rng(N)
    v = rng.standard_normal((N,) * 3)
    out = {
        "normal": v,
        "fp32 digits": v.astype(np.float32).astype(np.float64),
        "sorted": np.sort(v, axis=None).reshape(v.shape),
        "skewed": 3.0 - 3.0 * np.exp(-v),
        "heavy tails": np.tan(1.5 * np.tanh(v)),
        "half zeros": np.maximum(v, 0.0),          # one bucket of half the cells
        "rounded": np.round(3.0 * v),              # a dozen values
        "constant": np.full_like(v, 2.5),
        "outlier": np.where(v == v.max(), 1e30, v),
        "offset": v + 1e9,
        "tiny": v * 1e-300,
    }
    out["signed zeros"] = np.where(v < 0, -0.0, np.where(v < 0.5, 0.0, v))
    return out


@pytest.mark.parametrize("N", [4, 10, 48, 96])   # 96: the quantiles' series and their direct tails
@pytest.mark.parametrize("kind", list(fields(4)))
def test_ranks_and_quantiles(O, N, kind):
    from paper_1709_06350_gb300 import recon as R
    v = fields(N)[kind]
    s = R.Solver(N, float(N))
    g = s.gaussianise(torch.from_numpy(v).cuda()).cpu().numpy()
    again = s.gaussianise(torch.from_numpy(v).cuda()).cpu().numpy()
    s.close()
    assert np.array_equal(g, again)
    order = np.argsort(v, axis=None, kind="stable")
    assert np.all(np.diff(g.ravel()[order]) >= 0)
    if kind in ("offset", "outlier", "tiny"):      # the moments' own rounding or underflow dominates the values
        return
    ref, _ = O.gaussianise(v)
    assert np.max(np.abs(g - ref)) <= 1e-11 * v.std()
    if v.std() > 0:
        assert np.all(np.diff(g.ravel()[order]) > 0)
