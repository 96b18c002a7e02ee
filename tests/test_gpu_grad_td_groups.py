"""htd_grad_td over groups of sources, and its form without room for a group.

Sources run together in the step launches; the gradient is the sum over them, so a
call with several sources equals the sum of calls with one each.  The misfit and the
states are the same bits; the sums over sources and terms are FP64, added in another
order: 1e-12 relative.  A workspace that cannot be had (allocation failure injected)
falls back to one source and fewer planes with the same result.
"""
import numpy as np
import pytest

from paper_2006_16861_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2006_16861_gb300 import htd  # noqa: E402
from test_gpu_parity import dev, het_problem  # noqa: E402

CASES = [((37, 70), "mixed", "table1", 3), ((37, 70), "fp64", "exact", 3),
         ((130, 257), "mixed", "exact", 2), ((9, 12, 35), "mixed", "table1", 3),
         ((9, 12, 35), "fp64", "table1", 2), ((900, 640), "mixed", "table1", 4)]


def _setup(n, precision, mode, nsrc):
    p = het_problem(len(n), n, T=2, layer=2, seed=31)
    s = htd.Solver(p, precision=precision, mode=mode)
    F = dev(np.stack([W.random_rhs(60 + k, n) for k in range(nsrc)]))
    rec = np.arange(3, int(np.prod(n)), 7, dtype=np.int64)[:50]
    d = dev(W.random_rhs(70, (nsrc, rec.size)))
    return s, F, rec, d


def _close(a, b):
    return float((a - b).norm()) <= 1e-12 * float(b.norm())


@pytest.mark.parametrize("n,precision,mode,nsrc", CASES)
def test_sources_together_equal_the_sum_of_sources(n, precision, mode, nsrc):
    s, F, rec, d = _setup(n, precision, mode, nsrc)
    J, gm, gR = s.grad_td(F, rec, d)
    again = s.grad_td(F, rec, d)                    # replays the captured passes
    assert again[0] == J and torch.equal(again[1], gm) and torch.equal(again[2], gR)
    parts = [s.grad_td(F[k:k + 1].contiguous(), rec, d[k:k + 1].contiguous())
             for k in range(nsrc)]
    assert abs(sum(x[0] for x in parts) / J - 1) <= 1e-13
    assert _close(gm, sum(x[1] for x in parts)) and _close(gR, sum(x[2] for x in parts))
    s.close()


@pytest.mark.parametrize("n,precision,mode,nsrc", CASES[:5])
def test_without_room_one_source_and_fewer_planes(n, precision, mode, nsrc):
    s, F, rec, d = _setup(n, precision, mode, 1)
    try:
        htd.htd_test_fail_alloc(2)                  # after the two receiver buffers
        lean = s.grad_td(F, rec, d)
    finally:
        htd.htd_test_fail_alloc(-1)
    s.close()
    s, F, rec, d = _setup(n, precision, mode, 1)
    ref = s.grad_td(F, rec, d)
    assert lean[0] == ref[0] and _close(lean[1], ref[1]) and _close(lean[2], ref[2])
    s.close()
