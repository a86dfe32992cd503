"""The real-space pass at the edges of its tiles, against the CPU FP64 oracle.

x extents around the warp and row-pitch limits (a partial warp, a last column alone in its warp, rows
that bulk copies cannot take, the largest), every row tile, both laws, with and without an
eigenstrain (its own kernel variant), and a chunk length that leaves a short last chunk.  Three
evaluations from u = 0, so that the strain, the adjoint and the stores of every column enter.

Tolerances are those of the parity tests: FP64 1e-10 relative L2 on the fields, FP32 1e-5 (rounding of
the transforms and of sums over some 10^2 terms).  The output fields lie between guard bands that the
pass must leave alone.
"""
import numpy as np
import pytest

import synth
from oracle import tetra as T

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

E_MIX = np.array([1e-3, -2e-4, 5e-4, 3e-4, -1e-4, 2e-3])
GUARD = 4096


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


def guarded(shape, dtype):
    n = int(np.prod(shape))
    buf = torch.full((n + 2 * GUARD,), -7.0, dtype=dtype, device="cuda")
    return buf, buf[GUARD:GUARD + n].view(shape)


@pytest.mark.parametrize("ytile", [0, 2, 4, 8])
@pytest.mark.parametrize("n1", [4, 30, 32, 44, 64, 66, 96, 128, 132, 160, 256])
def test_row_extents_and_tiles(hs, n1, ytile):
    check(hs, (n1, 8, 6), ytile, eigen=(n1 % 4 == 0))


@pytest.mark.parametrize("n1", [264, 352, 512])
def test_wide_rows(hs, n1):
    check(hs, (n1, 8, 6), 0, eigen=True)


@pytest.mark.parametrize("n1", [288, 320, 352])
def test_wide_rows_in_halves(hs, n1):
    """Tiles of 8 FP64 rows of more than 256 columns run as two blocks of a cluster (partial warps at 288 to 352):
    the FP64 sweep of the refined precision, with a wrapped first row and tiles on both sides.  (An explicit
    tile of 8 rows at 512 columns is refused: the FP32 pass has no room for it.)"""
    check(hs, (n1, 16, 6), 8, eigen=(n1 == 320), precisions=(hs.HS_FP32_REFINED,))


def check(hs, grid, ytile, eigen, precisions=None):
    n1, n2, n3 = grid
    for law in ("iso", "aniso"):
        ids = synth.random_phase_map(grid, 3, seed=n1 + ytile)
        if law == "iso":
            table = np.stack([synth.isotropic_voigt(E, nu) for E, nu in ((1.0, 0.3), (4.0, 0.2), (0.0, 0.3))])
        else:
            table = synth.polycrystal_table(168.4, 121.4, 75.4, synth.random_rotations(3, seed=6))
        C0 = synth.isotropic_voigt(0.6 * float(table[:, 0, 0].max()), 0.25)
        lam0 = T.stiffness_tensor(C0)
        eps0 = 1e-4 * np.random.default_rng(n1).standard_normal((3, 6)) if eigen else None
        e0 = None if eps0 is None else np.stack([T.strain_tensor_from_voigt(e) for e in eps0])
        ref = T.solve_alg1(ids, table, lam0, T.strain_tensor_from_voigt(E_MIX), tol=0.0, max_iter=3, eigen=e0)
        want = T.voigt_from_tensor(ref.eps), T.voigt_from_tensor(ref.sig)
        for prec, tol, dtype in ((hs.HS_FP64, 1e-10, torch.float64), (hs.HS_FP32, 1e-5, torch.float32),
                                 (hs.HS_FP32_REFINED, 1e-5, torch.float32)):
            if precisions is not None and prec not in precisions:
                continue
            kw = dict(C0=C0, precision=prec, ytile=ytile, zchunk=4, out_f32=int(dtype == torch.float32))
            if prec == hs.HS_FP64 and ytile == 8 and n1 == 256:
                with pytest.raises(hs.HSError):  # a tile that is too large stays refused
                    hs.Solver(ids, table, **kw)
                continue
            s = hs.Solver(ids, table, **kw)
            if eigen:
                s.set_eigenstrain(eps0)
            shape = (6, n3, n2, n1)
            bufs = [guarded(shape, dtype) for _ in range(2)]
            # a refined solve repeats its last evaluation in FP64
            out = s.solve(E_MIX, tol=0.0, max_iter=4 if prec == hs.HS_FP32_REFINED else 3, out=[v for _, v in bufs])
            assert out["status"] == hs.HS_NOT_CONVERGED
            for (buf, view), w in zip(bufs, want):
                assert rel(view.cpu().double().numpy(), w) < tol, (law, prec)
                assert bool((buf[:GUARD] == -7.0).all()) and bool((buf[-GUARD:] == -7.0).all())
            np.testing.assert_allclose(out["sig_eff"], T.voigt_from_tensor(ref.sig_mean),
                                       rtol=0, atol=tol * np.abs(ref.sig_mean).max())
            s.close()
