"""Every row count of the 2-D I_abd step against the FP64 oracle, at sizes made from the
device's SM count.

The launcher takes the most of 4, 2 and 1 rows per thread that leave two blocks (32
columns, 8 threads of rows) per SM; in FP64 the one of those whose SM with the most blocks
has the least to do, a node costing 1, 0.83, 0.8 with 1, 2, 4 rows.  For each count one
grid just inside the rule, with a last row that ends inside a thread's rows.  Tolerances
of test_gpu_abd: 1e-10 (FP64), 5e-5 (mixed).
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

NX = 401


def blocks(ny, rows):
    return -(-NX // 32) * -(-ny // (8 * rows))


def rule(ny, precision):
    """The row count that the launcher takes for ny x NX nodes."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = next((r for r in (4, 2) if blocks(ny, r) >= 2 * sms), 1)
    if precision == "fp64":
        node = {1: 1.0, 2: 0.83, 4: 0.8}
        rows = min((r for r in (4, 2, 1) if r <= rows),
                   key=lambda r: -(-blocks(ny, r) // sms) * r * node[r])
    return rows


def grid_rows(rows, rest, precision):
    """The fewest grid rows for which the rule takes `rows`, `rest` more than whole threads."""
    ny = rest
    while rule(ny, precision) != rows:
        ny += rows
    return ny


@pytest.mark.parametrize("rows,rest", [(1, 0), (2, 1), (4, 1), (4, 3)])
@pytest.mark.parametrize("damping", ["node", "cell"])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_abd_rows_match_the_oracle(rows, rest, damping, precision):
    ny = grid_rows(rows, rest, precision) if rows > 1 else 37
    assert rule(ny, precision) == rows and ny % rows == rest
    p = abd_problem(2, (ny, NX), T=1)
    s = htd.Solver(p, precision=precision, integrator="abd", damping=damping, restart=2)
    assert s.params["step_kernel"] == 3
    o = oracle.Oracle(p, integrator="abd", damping=damping)
    F = W.random_rhs(12, p.n)
    tol = 1e-10 if precision == "fp64" else 5e-5
    assert rel_l2(host(s.precond(dev(F))).reshape(-1), o.precond(F, "table1").reshape(-1)) <= tol
    s.close()
