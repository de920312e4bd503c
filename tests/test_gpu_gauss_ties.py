"""Gaussianisation of fields whose equal values are neighbours: a warp takes their
places in a bucket together.  Runs that stay with the buckets and runs that go to
the radix sort, on sides around the scans' sizes in one launch (64: both; 80:
neither) and on one whose last warp is partial."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [10, 48, 64, 80])
@pytest.mark.parametrize("run", [2, 5, 33, 300])
def test_runs_rank_by_position(O, N, run):
    from paper_1709_06350_gb300 import recon as R
    n = N ** 3
    v = np.repeat(np.random.default_rng(N + run).standard_normal(-(-n // run)), run)[:n].reshape((N,) * 3)
    s = R.Solver(N, float(N))
    g = s.gaussianise(torch.from_numpy(v).cuda()).cpu().numpy()
    s.close()
    ref, _ = O.gaussianise(v)
    assert np.all(np.diff(g.ravel()[np.argsort(v, axis=None, kind="stable")]) > 0)
    assert np.max(np.abs(g - ref)) <= 1e-11 * v.std()   # the bound of tests/test_gpu_gauss_buckets.py
