"""The autotuner does not return a slower plan than the automatic choice.

The automatic tiling is one of the timed plans, and another one replaces it only when 2% faster, so a tuned
solver may take 1.02 of the automatic one's time, and 1.03 with the spread of a median of solves (below 1%).
"""
import time

import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def hs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_11168_gb300 import build, hs as _hs

    build.build()
    _hs.load()
    return _hs


@pytest.mark.parametrize("precision,n", [("HS_FP32", 128), ("HS_FP32", 192), ("HS_FP64", 64), ("HS_FP64", 128)])
def test_tuned_plan_is_not_slower(hs, precision, n):
    ids = synth.random_phase_map((n, n, n), 2, seed=3)
    table = synth.two_phase_table(1.0, 0.3, 0.1, 0.3)
    prec, stream = getattr(hs, precision), torch.cuda.Stream()
    opts, _ = hs.autotune(ids, table, precision=prec, iters=16, stream=stream)
    opts.pop("precision")
    E = [1e-3, 0, 0, 0, 0, 0]

    def median(kw):
        s = hs.Solver(ids, table, precision=prec, stream=stream, **kw)
        times = []
        for _ in range(9):
            torch.cuda.synchronize()
            t = time.perf_counter()
            s.solve(E, tol=0.0, max_iter=32, fields=False)
            times.append(time.perf_counter() - t)
        s.close()
        return sorted(times)[4]

    default = min(median({}), median({}))
    assert min(median(opts), median(opts)) <= 1.03 * default, opts
