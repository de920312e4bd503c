"""The tiles and plane chunks of the displacement kernel: sides below a tile,
ragged in both of its directions, one plane a chunk (below 96) and several with
a shorter last one, with displacements of a few cells across the box edge."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [4, 6, 10, 28, 64, 96, 112, 128])
@pytest.mark.parametrize("rough", [0.0, 0.03])
def test_displace_tiles(O, N, rough):
    """Against the FP64 oracle.  psi: one rounding of the scale.  delta_r: the
    CIC coordinate and H carry FP32 roundings of differences of up to 20
    (1.2e-6), the sums ~8 contributions of |b v| < 3: within the 1e-5 of the
    repository's parity.  rough: white noise, so that neighbours' targets do
    not line up and nothing can be merged."""
    from paper_1709_06350_gb300 import recon as R
    L, h = 1.7 * N, 1.7
    x = (np.arange(N) + 0.5) * 2.0 * np.pi / N
    X, Y, Z = np.meshgrid(x, x, x, indexing="ij")
    k = 2.0 * np.pi / L
    amp = min(4.0 * h / k, 0.1 / k ** 2)   # up to 4 cells, |H| <= 0.1 per mode
    phi = amp * (np.sin(X + 0.3) + np.cos(Y + Z) / 2 + np.sin(Z - X + 1.0) / 2)
    phi += rough * h * h * np.random.default_rng(N).standard_normal(phi.shape)
    b = 1.0 + 0.5 * np.sin(X) * np.cos(Y - Z)
    psi_ref, dl_ref = O.displace(phi, b, L)
    s = R.Solver(N, L)
    psi, dl = s.displace(torch.from_numpy(phi).cuda(), torch.from_numpy(b).cuda())
    assert np.abs(psi.cpu().numpy() - psi_ref).max() < 1e-13 * np.abs(psi_ref).max()
    assert np.abs(dl.cpu().numpy() - dl_ref).max() < 1e-5
    s.close()
