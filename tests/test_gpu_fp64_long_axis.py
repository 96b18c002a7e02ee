"""FP64 3-D grids whose y axis needs more than 65535 tiles of the step's four rows.

A launch may have 65535 blocks along y and z and 2^31 - 1 along x, where the excess
goes.  262141 rows are one tile more than four-row tiles reach along y; the
eight-row kernels (split, operator) go to 524280.  Tolerance: the FP64 parity
tolerance 1e-10.
"""
import pytest

import oracle
from paper_2006_16861_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2006_16861_gb300 import htd  # noqa: E402
from test_gpu_parity import dev, het_problem, host, rel_l2  # noqa: E402


@pytest.mark.parametrize("n", [(1, 262141, 2), (2, 300001, 1)], ids=lambda n: "x".join(map(str, n)))
def test_fp64_3d_step_on_a_long_y_axis(n):
    p = het_problem(3, n, T=1, layer=2, seed=5)
    s = htd.Solver(p, precision="fp64", restart=2)
    F = W.random_rhs(8, n)
    want = oracle.Oracle(p).precond(F, "table1")
    assert rel_l2(host(s.precond(dev(F))).reshape(-1), want.reshape(-1)) <= 1e-10
    s.close()
