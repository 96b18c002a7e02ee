"""FP64 I_acd handles hold no per-cell recurrence plane.

Their steps read the assembled operator; I_abd steps read q kappa per cell and keep a
third state plane.  With the same grid, I_abd therefore makes two allocations more.
"""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2006_16861_gb300 import htd  # noqa: E402
from test_gpu_abd import abd_problem  # noqa: E402


def allocations(p, **kw):
    """Allocations of a handle's create: the first number whose failure it does not see."""
    for k in range(100):
        htd.htd_test_fail_alloc(k)
        try:
            htd.Solver(p, precision="fp64", restart=2, **kw).close()
            return k
        except htd.HtdError as e:
            assert e.status == 3
        finally:
            htd.htd_test_fail_alloc(-1)
    raise AssertionError("no end")


def test_fp64_acd_makes_two_allocations_fewer_than_abd():
    p = abd_problem(3, (9, 12, 35))
    assert allocations(p, integrator="abd") == allocations(p) + 2
