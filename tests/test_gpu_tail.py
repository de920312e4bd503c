"""The small levels of a V-cycle in one thread-block cluster (recon_tail.cu):
solves whose hierarchies start a tail at every side it takes, among them the
sides that split unevenly over the cluster and the single-level grids."""
import numpy as np
import pytest

from workloads import smooth_density, zeldovich_density

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# 10, 14: coarsest grid alone; 40, 48, 56: a tail from 20^3, 24^3, 28^3
SIDES = [8, 10, 12, 14, 16, 20, 24, 28, 32, 40, 48, 56]


@pytest.mark.parametrize("N", SIDES)
def test_fp64_iterates(O, N):
    """The iterate after three cycles is the oracle's: the same steps, only
    sums in another order (the bound of the repository's FP64 solve parity)."""
    from paper_1709_06350_gb300 import recon as R
    L = 2.0 * N
    b, _, _ = zeldovich_density(O, N, L, 0.6, 4.0, 900 + N)
    ref, info = O.solve(b, L, tol=1e-30, max_cycles=3)
    s = R.Solver(N, L)
    phi, st = s.solve(torch.from_numpy(b).cuda(), tol=1e-30, max_cycles=3, raise_on_noconv=False)
    assert np.linalg.norm(phi.cpu().numpy() - ref) < 1e-10 * np.linalg.norm(ref)
    assert st["compat_c"] == pytest.approx(info["c"], rel=1e-6, abs=1e-13)
    # the scaled-defect factors reach the handle from inside the tail
    assert all(0.0 <= x <= 1.0 for x in s.level_scales())
    s.close()


# (28 and 56 are left out: FAS does not reach 1e-10 there in 80 cycles, in the
# oracle either)
@pytest.mark.parametrize("N", [n for n in SIDES if n % 28])
def test_mixed_solution(O, N):
    """FP32 tails (FAS and linear) inside a converged solve.  A residual of
    relative size t leaves |phi - phi*| of at most about 10 t |phi| on smooth
    fields, so two solutions at tolerance t agree to 20 t."""
    from paper_1709_06350_gb300 import recon as R
    L = 2.0 * N
    b = smooth_density(N, 700 + N, amp=0.4)
    ref, info = O.solve(b, L, tol=1e-10, max_cycles=80)
    assert info["status"] == 0
    s = R.Solver(N, L, R.RECON_MIXED)
    phi, st = s.solve(torch.from_numpy(b).cuda(), tol=1e-10, max_cycles=60)
    assert np.linalg.norm(phi.cpu().numpy() - ref) < 20e-10 * np.linalg.norm(ref)
    s.close()


def test_unaligned_top_level(O):
    """A tail that starts on the caller's own arrays at an odd 8-byte offset."""
    from paper_1709_06350_gb300 import recon as R
    N, L = 16, 32.0
    b, _, _ = zeldovich_density(O, N, L, 0.6, 4.0, 7)
    ref, _ = O.solve(b, L, tol=1e-30, max_cycles=3)
    room = torch.zeros(2 * N ** 3 + 2, dtype=torch.float64, device="cuda")
    bd, phi = room[1:N ** 3 + 1].view(N, N, N), room[N ** 3 + 1:2 * N ** 3 + 1].view(N, N, N)
    bd.copy_(torch.from_numpy(b))
    s = R.Solver(N, L)
    s.solve(bd, phi=phi, tol=1e-30, max_cycles=3, raise_on_noconv=False)
    assert np.linalg.norm(phi.cpu().numpy() - ref) < 1e-10 * np.linalg.norm(ref)
    s.close()
