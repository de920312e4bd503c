"""Mixed solves follow their recorded iterates.

FP32 cycles amplify a single flipped digit (of a mean, of a cell's update) to
1e-7 of phi, which moves the last digits of a solve's result and, where the
corrections converge slowly, their number.  The residual norms of every cycle
and correction are therefore recorded (tests/golden/mixed_history.txt) and
compared to 1e-12: the norms are FP64 sums of FP32 values, equal as long as no
FP32 value changes.  Sides: 64 (its levels below 32^3 in one launch), 112 (sums
over more groups of rows than one wave of blocks; ends in 14^3), 128
(register-blocked sweeps, a first sweep from zero).
"""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "mixed_history.txt")


def density(N):
    """Smoothed integers as dyadic fractions: the same bits on every machine."""
    x = np.random.Generator(np.random.PCG64(N)).integers(0, 1 << 16, (N, N, N))
    for axis in range(3):
        for _ in range(3):
            x = sum(np.roll(x, s, axis) for s in range(-2, 3))
    p = int(np.floor(np.log2(np.std(x.astype(np.float64))))) + 1   # rms between 1/2 and 1
    return np.maximum(1.0 + (x - int(np.sum(x) // x.size)) * 2.0 ** -p, 2.0 ** -4)


def history(N):
    """(norms of the FP32 cycles, norms before each correction)"""
    from paper_1709_06350_gb300 import recon as R
    s = R.Solver(N, 1.75 * N, R.RECON_MIXED)
    _, st = s.solve(torch.from_numpy(density(N)).cuda(), tol=1e-8, max_cycles=40)
    s.close()
    return st["history"][:st["cycles"]], st["history"][st["cycles"]:]


def recorded(N):
    with open(GOLDEN) as f:
        rows = [line.split() for line in f if not line.startswith("#")]
    return [[float.fromhex(v) for v in r[2:]] for part in ("cycles", "corrections") for r in rows
            if r[:2] == [str(N), part]]


@pytest.mark.parametrize("N", [64, 112, 128])
def test_fp32_cycles(N):
    got, want = history(N)[0], recorded(N)[0]
    assert len(got) == len(want)
    np.testing.assert_allclose(got, want, rtol=1e-12)


@pytest.mark.parametrize("N", [64, 112, 128])
def test_corrections(N):
    got, want = history(N)[1], recorded(N)[1]
    assert len(got) == len(want)
    np.testing.assert_allclose(got, want, rtol=1e-12)
