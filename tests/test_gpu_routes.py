"""Kernel variants that the other tests do not reach, against the oracle or against the variant they replace.

* FP64 rows of more than 256 columns in two halves (clusters of two blocks): chosen by the tile model on grids
  with enough blocks (512 x 16 x 24 and 320 x 32 x 32 among them), in FP64 solves (force and fields), in
  batches and in the residual call, whose unaligned inputs take the whole-row pass;
* graph replay of FP32 passes that start before the kernel in front of them has ended (2^17 voxels and more);
* persistent column passes of every length that has them, in FP64 with either kind of tile load;
* FP64 run-time column plans of the short lengths that also have a compile-time one.

Tolerances are those of the parity tests: 1e-10 relative L2 in FP64; the rest is bit for bit.
"""
import ctypes

import numpy as np
import pytest

import synth
from oracle import tetra as T

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

E_MIX = np.array([1e-3, -2e-4, 5e-4, 3e-4, -1e-4, 2e-3])
HALVES = [(512, 16, 24), (320, 32, 32)]


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


def material(law, grid):
    ids = synth.random_phase_map(grid, 3, seed=grid[0])
    if law == "iso":
        return ids, np.stack([synth.isotropic_voigt(E, nu) for E, nu in ((1.0, 0.3), (4.0, 0.2), (0.0, 0.3))])
    return ids, synth.polycrystal_table(168.4, 121.4, 75.4, synth.random_rotations(3, seed=6))


@pytest.mark.parametrize("law", ["iso", "aniso"])
@pytest.mark.parametrize("grid", HALVES)
def test_fp64_halves_follow_the_oracle(hs, grid, law):
    ids, table = material(law, grid)
    C0 = synth.isotropic_voigt(0.6 * float(table[:, 0, 0].max()), 0.25)
    eps0 = 1e-4 * np.random.default_rng(1).standard_normal((3, 6)) if law == "aniso" else None
    e0 = None if eps0 is None else np.stack([T.strain_tensor_from_voigt(e) for e in eps0])
    ref = T.solve_alg1(ids, table, T.stiffness_tensor(C0), T.strain_tensor_from_voigt(E_MIX), tol=0.0, max_iter=3, eigen=e0)
    s = hs.Solver(ids, table, C0=C0, precision=hs.HS_FP64)
    if eps0 is not None:
        s.set_eigenstrain(eps0)
    out = s.solve(E_MIX, tol=0.0, max_iter=3)
    assert rel(out["eps"].cpu().numpy(), T.voigt_from_tensor(ref.eps)) < 1e-10
    assert rel(out["sig"].cpu().numpy(), T.voigt_from_tensor(ref.sig)) < 1e-10
    assert rel(out["sig_eff"], T.voigt_from_tensor(ref.sig_mean)) < 1e-10
    s.close()


@pytest.mark.parametrize("precision", ["HS_FP64", "HS_FP32_REFINED"])
def test_batched_halves_equal_single_solves(hs, precision):
    grid, prec = HALVES[0], getattr(hs, precision)
    rves = [(synth.random_phase_map(grid, 2, seed=k), synth.two_phase_table(1.0, 0.3, e, 0.3)) for k, e in ((1, 4.0), (2, 0.2))]
    batch = hs.Batch(rves, [0, 1], precision=prec, stream=torch.cuda.Stream(), inner_max=6)
    got = batch.solve(np.stack([E_MIX, E_MIX[::-1]]), tol=0.0, max_iter=12)
    for k, E in enumerate((E_MIX, E_MIX[::-1])):
        s = hs.Solver(*rves[k], precision=prec, inner_max=6)
        want = s.solve(E, tol=0.0, max_iter=12, fields=False)
        np.testing.assert_array_equal(got["sig_eff"][k], want["sig_eff"])
        # a refined batch's history holds the FP64 sweeps only
        n = len(batch.err_history(k)) if precision == "HS_FP64" else 1
        np.testing.assert_array_equal(batch.err_history(k)[-n:], s.err_history()[-n:])
        s.close()
    batch.close()


@pytest.mark.parametrize("grid", HALVES)
def test_residual_call_in_halves_and_on_unaligned_inputs(hs, grid):
    """u 8 bytes and ids 2 bytes off a 16-byte boundary rule out bulk copies, and with them the halves."""
    ids, table = material("aniso", grid)
    shape = (3,) + grid[::-1]
    u_r = 1e-3 * np.random.default_rng(3).standard_normal(shape)
    q1, q2, q3 = T.q_vectors(grid)
    u_q = np.fft.rfftn(u_r, axes=(1, 2, 3)) / np.prod(grid) * np.exp(-0.5j * (q1 + q2 + q3))[None]
    _, _, _, _, _, L2, sm = T.evaluate(u_q, T.D_of_q(grid), T.Material(ids, table), T.strain_tensor_from_voigt(E_MIX), grid)
    sig_ref = T.voigt_from_tensor(sm)
    lib, forces = hs.load(), []
    table = np.ascontiguousarray(table, dtype=np.float64).reshape(-1, 36)
    for off in (0, 1):
        u = torch.zeros(u_r.size + 2, dtype=torch.float64, device="cuda")[off:off + u_r.size].view(shape)
        d = torch.zeros(ids.size + 8, dtype=torch.int16, device="cuda")[off:off + ids.size].view(grid[::-1])
        u.copy_(torch.from_numpy(u_r))
        d.copy_(torch.from_numpy(ids.astype(np.int16)))
        force = torch.full(shape, float("nan"), dtype=torch.float32, device="cuda")
        sig, l2 = np.zeros(6), ctypes.c_double()
        st = lib.hs_residual_noalloc((ctypes.c_int * 3)(*grid), ctypes.c_void_p(d.data_ptr()), hs._dp(table), 3, hs._dp(E_MIX),
                                     ctypes.c_void_p(u.data_ptr()), ctypes.c_void_p(force.data_ptr()), hs._dp(sig),
                                     ctypes.byref(l2), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert st == hs.HS_OK
        np.testing.assert_allclose(sig, sig_ref, rtol=0, atol=1e-10 * np.abs(sig_ref).max())
        assert abs(l2.value - L2) <= 1e-10 * L2
        forces.append(force.double().cpu().numpy())
    # FP64 arithmetic in another order, stored as float
    np.testing.assert_allclose(forces[0], forces[1], rtol=0, atol=2e-7 * np.abs(forces[1]).max())


@pytest.mark.parametrize("precision", ["HS_FP32", "HS_FP32_REFINED"])
@pytest.mark.parametrize("grid", [(64, 64, 64), (80, 64, 48), (128, 40, 44)])
def test_replay_of_dependent_passes_matches_plain_launches(hs, grid, precision):
    """Budgets and tolerances that end a solve inside a chunk of four evaluations, and at its end."""
    ids = synth.random_phase_map(grid, 2, seed=3)
    table = synth.two_phase_table(1.0, 0.3, 4.0, 0.3)
    runs = []
    for graphs in (0, 1):
        s = hs.Solver(ids, table, precision=getattr(hs, precision), check_every=4, use_graphs=graphs, stream=torch.cuda.Stream())
        res = []
        for E, tol, budget in ((E_MIX, 0.0, 23), (E_MIX[::-1], 3e-3, 60), (E_MIX, 0.0, 24), (E_MIX[::-1], 1e-4, 60)):
            out = s.solve(E, tol=tol, max_iter=budget)
            res += [out["iters"], out["err"], out["sig_eff"], out["eps"].cpu().numpy(), out["sig"].cpu().numpy(), s.err_history()]
        s.close()
        runs.append(res)
    for a, b in zip(*runs):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("precision", ["HS_FP64", "HS_FP32"])
@pytest.mark.parametrize("grid", [(20, 128, 512), (22, 192, 384), (24, 384, 192), (20, 256, 128), (18, 512, 256)])
def test_persistent_column_passes_match_one_tile_per_block(hs, grid, precision):
    ids = synth.random_phase_map(grid, 2, seed=7)
    table = synth.two_phase_table(1.0, 0.3, 6.0, 0.3)
    runs = []
    for pipe, copy in ((1, 1), (2, 1), (2, 2)):
        s = hs.Solver(ids, table, precision=getattr(hs, precision), col_pipe=pipe, col_copy=copy)
        out = s.solve(E_MIX, tol=0.0, max_iter=6)
        runs.append([out["sig_eff"], out["eps"].cpu().numpy(), out["sig"].cpu().numpy(), s.err_history()])
        s.close()
    for run in runs[1:]:
        for a, b in zip(runs[0], run):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("length", [32, 48, 96])
def test_fp64_run_time_plans_of_short_lengths(hs, length):
    """Blocks of 128 threads are not the compile-time plans' (64), so the run-time plan runs."""
    for grid in ((20, length, 6), (20, 6, length)):
        ids = synth.random_phase_map(grid, 2, seed=length)
        table = synth.two_phase_table(1.0, 0.3, 4.0, 0.2)
        C0 = synth.isotropic_voigt(2.5, 0.25)
        ref = T.solve_alg1(ids, table, T.stiffness_tensor(C0), T.strain_tensor_from_voigt(E_MIX), tol=0.0, max_iter=3)
        s = hs.Solver(ids, table, C0=C0, precision=hs.HS_FP64, col_threads=128)
        out = s.solve(E_MIX, tol=0.0, max_iter=3)
        assert rel(out["eps"].cpu().numpy(), T.voigt_from_tensor(ref.eps)) < 1e-10
        assert rel(out["sig"].cpu().numpy(), T.voigt_from_tensor(ref.sig)) < 1e-10
        s.close()
