"""A grid that the resident kernel runs window by window, where the windows' own
tables (step coefficients, exchange words, projection weights) find no memory.

The blocked kernel needs none of them and gives the same bits, so the handle is made
with it; every other allocation of create that fails is out of memory (status 3).
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


@pytest.mark.parametrize("mode,tables", [("table1", 2), ("project", 3)])
def test_no_memory_for_the_windows_leaves_the_blocked_kernel(mode, tables):
    n = (1301, 1303)
    p = het_problem(2, n, T=26, layer=20, seed=3)
    F = dev(W.random_rhs(2, n))
    kw = dict(precision="mixed", mode=mode, tb_form=htd.TB_RESIDENT, restart=2)
    s = htd.Solver(p, **kw)
    assert s.params["step_kernel"] == 4 and s.params["steps_per_launch"] < s.params["steps"]
    want = host(s.precond(F))
    s.close()
    blocked = refused = 0
    for k in range(60):
        htd.htd_test_fail_alloc(k)
        try:
            s = htd.Solver(p, **kw)
        except htd.HtdError as e:
            assert e.status == 3
            refused += 1
            continue
        finally:
            htd.htd_test_fail_alloc(-1)
        form = s.params["step_kernel"]
        if form == 1:
            blocked += 1
            assert np.array_equal(host(s.precond(F)), want)
        s.close()
        if form == 4:                       # allocation k was never reached
            break
    assert form == 4 and refused > 10 and blocked == tables
