"""The V-cycle's level-to-level kernels and the sweeps' alternating arrays: odd
and even sweep counts before and after the coarse correction (none among them),
sweeps that start from e = 0, restrictions to several levels in one launch."""
import numpy as np
import pytest

from workloads import smooth_density, zeldovich_density

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# 64: tail below the first level; 80, 96: plane-pair sweeps and partial tiles;
# 128: all its levels in one restriction; 160: one level restricted by itself
@pytest.mark.parametrize("N", [64, 80, 96, 128, 160])
@pytest.mark.parametrize("nu1,nu2", [(2, 1), (0, 3)])
def test_fp64_iterates(O, N, nu1, nu2):
    """The iterate after two cycles is the oracle's: the same steps, only sums
    in another order (the bound of the repository's FP64 solve parity)."""
    from paper_1709_06350_gb300 import recon as R
    L = 2.0 * N
    b, _, _ = zeldovich_density(O, N, L, 0.6, 4.0, 300 + N)
    ref, _ = O.solve(b, L, tol=1e-30, max_cycles=2, nu1=nu1, nu2=nu2)
    s = R.Solver(N, L, nu1=nu1, nu2=nu2)
    phi, _ = s.solve(torch.from_numpy(b).cuda(), tol=1e-30, max_cycles=2, raise_on_noconv=False)
    assert np.linalg.norm(phi.cpu().numpy() - ref) < 1e-10 * np.linalg.norm(ref)
    s.close()


# 64, 128, 192: register-blocked sweeps (192 with a side that is no power of
# two); 160: plane-pair sweeps above a 80^3 level of two passes
@pytest.mark.parametrize("N", [64, 128, 160, 192])
@pytest.mark.parametrize("nu1,nu2", [(1, 1), (1, 2), (2, 1), (2, 2), (3, 2), (0, 3), (3, 0)])
def test_mixed_solution(N, nu1, nu2):
    """A mixed solve against the FP64 solver with the same sweeps.  Solutions
    at tolerance t agree to 20 t, and FP32 corrections cost no cycles: a
    linear V-cycle contracts as a FAS cycle of the same sweeps does, and a
    defect correction takes two, so at most the hand-over's one is added."""
    from paper_1709_06350_gb300 import recon as R
    L = 2.0 * N
    b = torch.from_numpy(smooth_density(N, 500 + N, amp=0.4)).cuda()
    s = R.Solver(N, L, nu1=nu1, nu2=nu2)
    ref, st64 = s.solve(b, tol=1e-10, max_cycles=80)
    s.close()
    s = R.Solver(N, L, R.RECON_MIXED, nu1=nu1, nu2=nu2)
    phi, st = s.solve(b, tol=1e-10, max_cycles=80)
    assert float((phi - ref).norm()) < 20e-10 * float(ref.norm())
    assert st["cycles"] <= st64["cycles"] + 1
    again, _ = s.solve(b, tol=1e-10, max_cycles=80)   # from whichever array the last one left
    assert torch.equal(again, phi)
    s.close()
