"""The adjoint's mixed-precision solve (grids above 32^3): the residual of
J^T lam + mu 1 = g, evaluated independently in FP64, meets the solver's 1e-12
(2e-12 here: the null-space fix and this evaluation round too), for formed
(side 64, 128) and stored cofactors, on FP64 and MIXED handles."""
import numpy as np
import pytest

from workloads import zeldovich_density

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _at(a, *shift):
    return np.roll(a, [-x for x in shift], (0, 1, 2))


def _jt(phi, lam, h):
    """J^T lam = sum_ab D_ab (adj(I + H phi)_ab lam)."""
    def second(a, d):
        e = [0, 0, 0]
        e[d] = 1
        return (_at(a, *e) + _at(a, *[-x for x in e]) - 2 * a) / h ** 2

    def cross(a, d, f):
        def e(x, y):
            v = [0, 0, 0]
            v[d], v[f] = x, y
            return _at(a, *v)
        return ((e(1, 1) + e(-1, -1)) - (e(1, -1) + e(-1, 1))) / (4 * h ** 2)
    xx, yy, zz = (1 + second(phi, d) for d in range(3))
    xy, yz, xz = cross(phi, 0, 1), cross(phi, 1, 2), cross(phi, 0, 2)
    out = second((yy * zz - yz * yz) * lam, 0) + second((xx * zz - xz * xz) * lam, 1)
    out += second((xx * yy - xy * xy) * lam, 2)
    return out + 2 * (cross((xz * yz - xy * zz) * lam, 0, 1) + cross((xy * xz - xx * yz) * lam, 1, 2) +
                      cross((xy * yz - xz * yy) * lam, 0, 2))


@pytest.mark.parametrize("N,store", [(48, 0), (64, 0), (64, 1), (80, 0), (128, 0)])
@pytest.mark.parametrize("mixed", [False, True])
def test_residual(O, N, store, mixed):
    from paper_1709_06350_gb300 import recon as R
    L = 2.0 * N
    b, _, _ = zeldovich_density(O, N, L, 0.8, 4.0, 300 + N)
    s = R.Solver(N, L, R.RECON_MIXED if mixed else R.RECON_F64, adjoint_store_cofactors=store)
    phi, _ = s.solve(torch.from_numpy(b).cuda(), tol=1e-8, max_cycles=60)
    # tiny and large right sides: the corrections are scaled
    for scale in (1.0, 1e-100, 1e100):
        g = scale * np.random.default_rng(N).standard_normal((N,) * 3)
        lam = s.adjoint(torch.from_numpy(g).cuda()).cpu().numpy()
        r = (g - _jt(phi.cpu().numpy(), lam, 2.0)) / scale
        r -= r.mean()
        assert np.linalg.norm(r) < 2e-12 * np.linalg.norm(g / scale)
        assert abs((lam / scale).sum()) < 1e-9 * np.abs(lam / scale).sum()
    s.close()
