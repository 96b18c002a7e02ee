"""The 2-D I_abd step with one, two and four rows per thread against the FP64 oracle.

The launcher takes the most rows that leave two blocks per SM, so the grids are sized
around that rule, with a last row that ends inside a thread's rows.  Tolerances of
test_gpu_abd: 1e-10 (FP64), 5e-5 (mixed).
"""
import pytest

import oracle
from paper_2006_16861_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2006_16861_gb300 import htd  # noqa: E402
from test_gpu_abd import abd_problem  # noqa: E402
from test_gpu_parity import dev, host, rel_l2  # noqa: E402


@pytest.mark.parametrize("n", [(1, 5), (9, 33), (333, 417), (631, 650)],
                         ids=lambda n: "x".join(map(str, n)))
@pytest.mark.parametrize("damping", ["node", "cell"])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_abd_rows_match_the_oracle(n, damping, precision):
    p = abd_problem(2, n, T=1)
    s = htd.Solver(p, precision=precision, integrator="abd", damping=damping)
    o = oracle.Oracle(p, integrator="abd", damping=damping)
    F = W.random_rhs(12, p.n)
    tol = 1e-10 if precision == "fp64" else 5e-5
    assert rel_l2(host(s.precond(dev(F))).reshape(-1), o.precond(F, "table1").reshape(-1)) <= tol
    s.close()
