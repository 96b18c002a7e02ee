"""The resident-grid kernel over windows of a 2-D grid that does not fit the SMs.

Per node the arithmetic is the one-step kernel's, so outputs are equal bit for bit:
grids cut along either axis, ragged last windows and tiles, several passes with a
shorter last one, the three read-outs, and the run's first state at rest after an
earlier run left other states behind.
"""
import numpy as np
import pytest

from paper_2006_16861_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2006_16861_gb300 import htd  # noqa: E402
from test_gpu_parity import dev, het_problem, host  # noqa: E402

SIZES = [(1303, 1301), (2207, 703), (611, 2503), (1501, 2001)]


@pytest.mark.parametrize("n", SIZES, ids=lambda n: "x".join(map(str, n)))
@pytest.mark.parametrize("mode", ["table1", "exact", "project"])
def test_windows_equal_the_one_step_kernel(n, mode):
    p = het_problem(2, n, T=26, layer=20, seed=3)
    forcings = [dev(W.random_rhs(2, n)), dev(p.F)]
    out = []
    for kw in (dict(tblock=1), dict(tb_form=htd.TB_RESIDENT)):
        s = htd.Solver(p, precision="mixed", mode=mode, **kw)
        prm = s.params
        out.append([host(s.precond(f)) for f in forcings])
        s.close()
    assert prm["step_kernel"] == 4 and 1 < prm["steps_per_launch"] < prm["steps"]
    for a, b in zip(*out):
        assert np.isfinite(a).all() and np.abs(a).max() > 0
        assert np.array_equal(a, b)


def test_window_wait_runs_out_then_the_handle_applies():
    p = het_problem(2, (1301, 1303), T=6, layer=20, seed=3)
    F = dev(p.F)
    s = htd.Solver(p, precision="mixed", tb_form=htd.TB_RESIDENT)
    want = host(s.precond(F))
    htd.htd_set_wait_limit(s.handle, 1_000_000, stall_test=True)     # 1 ms, stalled
    with pytest.raises(htd.HtdError):
        htd.htd_gmres_solve(s.handle, F, s.zeros(), 1e-6, 2)
    htd.htd_set_wait_limit(s.handle, 0, stall_test=False)
    assert np.array_equal(host(s.precond(F)), want)
    s.close()
