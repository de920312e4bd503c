"""The adjoint when its workspace does not fit: a build of the library whose
recon_adjoint.cu allocates through a fake that refuses what exceeds a limit."""
import json
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#include <cuda_runtime.h>
#include <map>
static std::map<void *, size_t> held;
extern "C" {
double recon_test_left = 1e18;
cudaError_t recon_test_malloc(void **p, size_t n)
{
    *p = nullptr;
    if ((double)n > recon_test_left) return cudaErrorMemoryAllocation;
    const cudaError_t e = cudaMalloc(p, n);
    if (e != cudaSuccess) return e;
    held[*p] = n;
    recon_test_left -= (double)n;
    return e;
}
cudaError_t recon_test_free(void *p)
{
    if (held.count(p)) recon_test_left += (double)held[p];
    held.erase(p);
    return cudaFree(p);
}
}
"""

CASE = r"""
import ctypes, json, sys
import numpy as np, torch
sys.path[:0] = [{root!r}, {tests!r}]
from paper_1709_06350_gb300 import recon as R
from test_gpu_adjoint_mixed import _jt
R.LIB_PATH = {lib!r}
N, L, limit = {N}, {L}, {limit}
rng = np.random.default_rng(3)
b = np.exp(0.3 * np.sin(2 * np.pi * (np.arange(N)[:, None, None] + 2 * np.arange(N)[:, None]) / N)
           * np.cos(2 * np.pi * np.arange(N) / N))
s = R.Solver(N, L)
phi, _ = s.solve(torch.from_numpy(b / b.mean()).cuda(), tol=1e-11, max_cycles=60)
g = rng.standard_normal((N,) * 3)
left = ctypes.c_double.in_dll(R.load(), "recon_test_left")
left.value = limit * N ** 3
try:
    lam = s.adjoint(torch.from_numpy(g).cuda()).cpu().numpy()
    r = g - _jt(phi.cpu().numpy() * (N / L) ** 2, lam * (N / L) ** 2, 1.0)
    r -= r.mean()
    print(json.dumps(dict(status=0, rel=float(np.linalg.norm(r) / np.linalg.norm(g)), left=left.value / N ** 3)))
except R.ReconError as e:
    print(json.dumps(dict(status=e.status, left=left.value / N ** 3)))
"""


@pytest.fixture(scope="module")
def faked(tmp_path_factory):
    from paper_1709_06350_gb300 import build as B
    B.build()
    d = tmp_path_factory.mktemp("faked")
    with open(d / "fake.cu", "w") as f:
        f.write(FAKE)
    jobs = [[B.nvcc(), *B._flags(False), "-DcudaMalloc=recon_test_malloc", "-DcudaFree=recon_test_free", "-c",
             os.path.join(B.CSRC, "recon_adjoint.cu"), "-o", str(d / "adjoint.o")],
            [B.nvcc(), *B._flags(False), "-c", str(d / "fake.cu"), "-o", str(d / "fake.o")]]
    objs = [os.path.join(B.OUT, s.replace(".cu", ".o")) for s in B.SOURCES if s != "recon_adjoint.cu"]
    lib = str(d / "librecon_faked.so")
    jobs.append([B.nvcc(), "-shared", *B.ARCH, "-o", lib, *objs, str(d / "adjoint.o"), str(d / "fake.o")])
    for j in jobs:
        p = subprocess.run(j, capture_output=True, text=True)
        assert p.returncode == 0, p.stderr
    return lib


# Bytes per cell on a side of 48 (stored cofactors): FP64 64 + 10.3 for the
# coarse levels, FP32 corrections 28.6.  In a box of 1e25, 1/h^2 is 0 in FP32,
# so the corrections come to nothing and the FP64 V-cycles run.
@pytest.mark.parametrize("L,limit,status", [(96.0, 1e9, 0), (96.0, 93.0, 0), (96.0, 75.0, 0), (96.0, 70.0, 6),
                                            (96.0, 50.0, 6), (1e25, 1e9, 0), (1e25, 95.0, 0), (1e25, 70.0, 6)])
def test_workspace_limits(faked, L, limit, status):
    code = CASE.format(root=ROOT, tests=os.path.join(ROOT, "tests"), lib=faked, N=48, L=L, limit=limit)
    p = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    got = json.loads(p.stdout.splitlines()[-1])
    assert got["status"] == status
    if status == 0:
        assert got["rel"] < 2e-12
    else:
        assert got["left"] == pytest.approx(limit)   # everything given back
