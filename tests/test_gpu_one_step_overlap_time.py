"""Overlapped one-step launches do not cost time.

Where a step's blocks fill between half of the device and all of it, letting the next
step in early puts several of its blocks on one SM while others idle; where steps were
let in before their wait, that also happened on small grids.  Such forms took up to 2.3
times as long as in plain stream order.  Bound: 1.2 times (a whole application replayed
from a graph, median of nine, both in this process).
"""
import pytest

from paper_2006_16861_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2006_16861_gb300 import htd  # noqa: E402
from test_gpu_abd import abd_problem  # noqa: E402
from test_gpu_parity import dev, het_problem  # noqa: E402

NODE, CELL = (dict(integrator="abd", damping=d) for d in ("node", "cell"))
CASES = [((333, 127), "fp64", dict(tblock=1)), ((350, 350), "fp64", dict(tblock=1)),
         ((401, 401), "mixed", dict(tblock=1)), ((333, 127), "fp64", NODE),
         ((350, 350), "fp64", CELL), ((401, 401), "mixed", NODE), ((48, 48, 48), "mixed", NODE),
         ((90, 80, 70), "mixed", dict(s3_kernel=htd.S3_ZMARCH)), ((30, 40, 50), "fp64", {}),
         # one of eight right-hand sides active: most blocks of a launch are idle
         ((170, 150), "fp64", dict(CELL, max_rhs=8)), ((300, 200), "fp64", dict(max_rhs=8))]


@pytest.mark.parametrize("n,precision,kw", CASES,
                         ids=["%s-%s-%s" % ("x".join(map(str, n)), p,
                                            "-".join(map(str, kw.values())) or "acd")
                              for n, p, kw in CASES])
def test_overlap_costs_no_time(n, precision, kw):
    p = (abd_problem if "integrator" in kw else het_problem)(len(n), n, T=20)
    F = dev(W.random_rhs(5, n))
    solvers = [htd.Solver(p, precision=precision, launch=launch, restart=2, **kw)
               for launch in (0, htd.LAUNCH_NO_OVERLAP)]
    ms = [[], []]
    for k in range(12):
        for s, t in zip(solvers, ms):
            U = s.zeros()
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            s.precond(F, U)
            e1.record()
            e1.synchronize()
            if k >= 3:
                t.append(e0.elapsed_time(e1))
    with_overlap, plain = (sorted(t)[len(t) // 2] for t in ms)
    assert with_overlap <= 1.2 * plain
    for s in solvers:
        s.close()
