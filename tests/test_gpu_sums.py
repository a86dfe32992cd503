"""Accuracy of the FP32 real-space pass's sums over the voxels, whatever its chunk.

A homogeneous cell with lambda = 0 and mu = 1 under a shear strain v (an FP32 number) is in equilibrium at u = 0:
every voxel has the stress 2 v exactly, so the mean stress differs from it by the rounding of the sums alone.
A thread adds at most 16 equal values in FP32 before the sum goes on in two floats; the k-th partial sum of
n = 16 equal values is rounded by at most 2^-24 of itself, hence (n + 1) / 2 2^-24 = 5.1e-7 of the mean.  (One
chain over a chunk of 64 planes of 4 rows: up to 3.8e-6.)
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

BOUND = 17 / 2 * 2.0**-24


@pytest.fixture(scope="module")
def hs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_11168_gb300 import build, hs as _hs

    build.build()
    _hs.load()
    return _hs


# chunks: one plane, shorter and longer than the register chains, the longest; bulk and element copies; every row tile
@pytest.mark.parametrize("grid,kw", [
    ((16, 16, 64), {"zchunk": 64}), ((30, 20, 50), {"zchunk": 50}), ((16, 16, 64), {"zchunk": 3}),
    ((512, 8, 64), {"zchunk": 64}), ((16, 16, 64), {"zchunk": 64, "ytile": 8}), ((16, 16, 64), {"zchunk": 64, "ytile": 2}),
    ((64, 64, 64), {}), ((192, 192, 192), {}), ((256, 256, 256), {}),
])
def test_mean_stress_of_a_uniform_field(hs, grid, kw):
    s = hs.Solver(np.zeros(grid[::-1], np.uint16), synth.isotropic_voigt(2.0, 0.0)[None], precision=hs.HS_FP32, **kw)
    for v in (1 + np.random.default_rng(0).random(20)).astype(np.float32):
        out = s.solve([0, 0, 0, 0, 0, float(v)], tol=1e-8, max_iter=3, fields=False)
        assert out["iters"] == 1 and out["err"] == 0
        assert abs(out["sig_eff"][5] / (2 * float(v)) - 1) <= BOUND, float(v)
    s.close()


@pytest.mark.parametrize("grid", [(16, 16, 16), (64, 64, 64)])
def test_overflowing_residual_is_infinite(hs, grid):
    """|F|^2 beyond the FP32 range: the error is infinite, not undefined."""
    s = hs.Solver(synth.random_phase_map(grid, 2, seed=1), synth.two_phase_table(1.0, 0.3, 4.0, 0.3), precision=hs.HS_FP32,
                  zchunk=grid[2])
    with pytest.raises(hs.HSError) as e:
        s.solve([1e25, 0, 0, 0, 0, 0], tol=1e-8, max_iter=3, fields=False)
    assert e.value.status == hs.HS_DIVERGED
    assert s.err_history()[0] == np.inf
    s.close()
