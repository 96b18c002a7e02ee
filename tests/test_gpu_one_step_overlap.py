"""The one-step kernels with overlapped launches against plain stream order.

A launch of these kernels may start while the one before it drains and waits for it
before it touches a state (the 2-D I_abd step reads its coefficients before that wait).
The outputs equal those of HTD_LAUNCH_NO_OVERLAP bit for bit, from the captured graph
and launch by launch.
"""
import numpy as np
import pytest

from paper_2006_16861_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2006_16861_gb300 import htd  # noqa: E402
from test_gpu_abd import abd_problem  # noqa: E402
from test_gpu_parity import dev, het_problem, host  # noqa: E402

ACD2, ACD3 = dict(tblock=1), dict(s3_kernel=htd.S3_ZMARCH)
NODE, CELL = (dict(integrator="abd", damping=d) for d in ("node", "cell"))
CASES = [  # (grid, precision, options): one and several rows per thread, 2-D and 3-D
    ((37, 70), "mixed", ACD2), ((801, 701), "mixed", ACD2), ((37, 70), "fp64", ACD2),
    ((301, 257), "fp64", ACD2), ((21, 34, 45), "mixed", ACD3), ((21, 34, 45), "fp64", {}),
    ((37, 70), "mixed", NODE), ((37, 70), "fp64", CELL), ((401, 401), "mixed", CELL),
    ((801, 701), "mixed", NODE), ((801, 701), "mixed", CELL), ((12, 17, 34), "mixed", CELL),
    ((12, 17, 34), "fp64", NODE),
]


@pytest.mark.parametrize("n,precision,kw", CASES,
                         ids=["%s-%s-%s" % ("x".join(map(str, n)), p,
                                            "-".join(map(str, kw.values())) or "acd")
                              for n, p, kw in CASES])
@pytest.mark.parametrize("mode", ["table1", "project"])
def test_overlapped_one_step_launches_change_nothing(n, precision, kw, mode):
    p = (abd_problem if "integrator" in kw else het_problem)(len(n), n, T=3)
    kw = dict(kw, precision=precision, mode=mode, restart=2, max_rhs=2)
    forcings = [dev(W.random_rhs(k, n)) for k in (5, 6)]
    s = htd.Solver(p, launch=htd.LAUNCH_NO_OVERLAP, **kw)
    assert s.params["step_kernel"] == (3 if "integrator" in kw else 0)
    want = [host(s.precond(f)) for f in forcings]
    s.close()
    for launch in (0, htd.LAUNCH_NO_GRAPH):
        s = htd.Solver(p, launch=launch, **kw)
        for _ in range(3):
            for f, w in zip(forcings, want):
                assert np.isfinite(w).all() and np.abs(w).max() > 0
                assert np.array_equal(host(s.precond(f)), w)
        s.close()
