"""Every transform length with a compile-time plan, along each axis, against the CPU FP64 oracle.

A length is put on one axis of a small grid at a time: along x the rows of a batch do not fill their block
(48 rows), along y and z the tile of 11 spectral columns has a full part and a ragged one.  A batched
solver runs the same kernels with a medium per item.  Three evaluations from u = 0.  Lengths without a
plan, and one with a plan in FP32 only, run the run-time plan in FP64.

Tolerances are those of the parity tests: FP64 1e-10 relative L2 on the fields, FP32 1e-5 (rounding of
the transforms and of sums over some 10^2 terms).
"""
import numpy as np
import pytest

import synth
from oracle import tetra as T

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

E_MIX = np.array([1e-3, -2e-4, 5e-4, 3e-4, -1e-4, 2e-3])
LENGTHS = [32, 40, 44, 48, 56, 64, 72, 80, 88, 96, 112, 120, 128, 144, 160, 176, 192, 224, 240, 256, 384, 512]


@pytest.fixture(scope="module")
def hs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_11168_gb300 import build, hs as _hs

    build.build()
    _hs.load()
    return _hs


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("axis", ["x", "y", "z"])
@pytest.mark.parametrize("length", LENGTHS)
def test_length_along_axis(hs, length, axis):
    grid = {"x": (length, 8, 6), "y": (20, length, 6), "z": (20, 6, length)}[axis]
    ids = synth.random_phase_map(grid, 2, seed=length)
    table = synth.two_phase_table(1.0, 0.3, 4.0, 0.2)
    C0 = synth.isotropic_voigt(2.5, 0.25)
    ref = T.solve_alg1(ids, table, T.stiffness_tensor(C0), T.strain_tensor_from_voigt(E_MIX), tol=0.0, max_iter=3)
    eps, sig = T.voigt_from_tensor(ref.eps), T.voigt_from_tensor(ref.sig)
    for prec, tol in ((hs.HS_FP64, 1e-10), (hs.HS_FP32, 1e-5)):
        for threads in (0, 64):  # 64: the column passes' run-time plan
            s = hs.Solver(ids, table, C0=C0, precision=prec, col_threads=threads)
            out = s.solve(E_MIX, tol=0.0, max_iter=3)
            assert rel(np.asarray(out["eps"].cpu(), dtype=np.float64), eps) < tol, (prec, threads)
            assert rel(np.asarray(out["sig"].cpu(), dtype=np.float64), sig) < tol, (prec, threads)
            s.close()


@pytest.mark.parametrize("length", [32, 44, 80, 112, 160, 192])
def test_length_in_a_batch(hs, length):
    """The items of a batch against single solves, which check the same lengths above."""
    grid = (length, 6, 8)
    rves = [(synth.random_phase_map(grid, 2, seed=k), synth.two_phase_table(1.0, 0.3, e, 0.2)) for k, e in ((1, 4.0), (2, 0.2))]
    batch = hs.Batch(rves, [0, 1, 0], precision=hs.HS_FP32, stream=torch.cuda.Stream())
    E = np.stack([E_MIX, E_MIX, E_MIX[::-1]])
    got = batch.solve(E, tol=0.0, max_iter=3)
    for k, rve in enumerate((0, 1, 0)):
        s = hs.Solver(*rves[rve], precision=hs.HS_FP32)
        want = s.solve(E[k], tol=0.0, max_iter=3, fields=False)["sig_eff"]
        np.testing.assert_allclose(got["sig_eff"][k], want, rtol=0, atol=1e-5 * np.abs(want).max())
        s.close()
    batch.close()
