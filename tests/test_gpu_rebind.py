"""A context bound to another material gives what a context created with that material gives, bit for bit,
also when the constitutive law changes (other kernels, and with them the tiling they choose).

The iteration chunks replay as graphs; a change of law has to capture them again.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

E_MIX = np.array([1e-3, -2e-4, 5e-4, 3e-4, -1e-4, 2e-3])


@pytest.fixture(scope="module")
def hs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_11168_gb300 import build, hs as _hs

    build.build()
    _hs.load()
    return _hs


@pytest.mark.parametrize("precision", ["HS_FP64", "HS_FP32", "HS_FP32_REFINED"])
@pytest.mark.parametrize("grid", [(24, 20, 16), (64, 64, 64), (256, 24, 40)])
def test_rebinding_across_laws_equals_a_fresh_solver(hs, grid, precision):
    prec, stream = getattr(hs, precision), torch.cuda.Stream()
    ids = [synth.random_phase_map(grid, 2, seed=k) for k in range(2)]
    tables = {"iso": synth.two_phase_table(1.0, 0.3, 3.0, 0.25),
              "aniso": synth.polycrystal_table(168.4, 121.4, 75.4, synth.random_rotations(2, seed=6))}

    def solve(s):
        out = s.solve(E_MIX, tol=0.0, max_iter=24)
        return [out["sig_eff"], np.array(s.err_history()), out["eps"].cpu().numpy(), out["sig"].cpu().numpy()]

    want = {}
    for law, table in tables.items():
        for k in range(2):
            s = hs.Solver(ids[k], table, precision=prec, stream=stream)
            want[law, k] = solve(s)
            s.close()
    s = hs.Solver(ids[0], tables["iso"], precision=prec, stream=stream)
    solve(s)
    for law, k in (("aniso", 1), ("aniso", 0), ("iso", 1), ("iso", 0), ("aniso", 0)):
        s.set_material(ids[k], tables[law])
        for got, ref in zip(solve(s), want[law, k]):
            np.testing.assert_array_equal(got, ref)
    s.close()
