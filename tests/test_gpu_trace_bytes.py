"""Traced bytes of a plain FP64 solve, which launches sweeps ahead: those that the device skips move nothing."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1504_07499_gb300 import hmg, inputs as I


@pytest.mark.parametrize("N", [32, 96])   # x inverse and next x forward in one kernel, and in two
def test_skipped_sweeps_count_no_bytes(N):
    ph, k = I.random_phase_grid(1, N), (0.2, 0.25, 0.3)
    with hmg.Context(0) as ctx:
        hmg.hmg_trace_enable(ctx.handle, 1)

        def fp64_bytes(max_iter):
            a = hmg.hmg_trace_read(ctx.handle)["fp64"][2]
            _, info, _ = hmg.hmg_solve(ctx.handle, ph, N, k, 0.9, hmg.HMG_FP64, max_iter,
                                       allow=(hmg.HMG_OK, hmg.HMG_NOT_CONVERGED))
            assert info["iters"] == [1, 1, 1]
            return hmg.hmg_trace_read(ctx.handle)["fp64"][2] - a

        one = fp64_bytes(1)       # one sweep and an equilibrium test, as the last iterate's
        many = fp64_bytes(50)     # one sweep that meets the tolerance, and its equilibrium test; the chained
        assert 0 < one <= many < 1.2 * one   # form also writes the next spectrum, a twelfth of a sweep
