"""The captured passes of htd_grad_td stay while only the receivers change.

Nothing that is captured reads the receivers: their residuals enter the adjoint
forcing before the captured backward pass.  Calls with other receivers replay the same
graphs, with the result of a handle that has seen nothing else.
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


@pytest.mark.parametrize("n,precision,mode,nsrc", [((37, 70), "mixed", "table1", 3),
                                                   ((37, 70), "fp64", "exact", 1),
                                                   ((9, 12, 35), "mixed", "table1", 2)])
def test_other_receivers_replay_the_captured_passes(n, precision, mode, nsrc):
    p = het_problem(len(n), n, T=2, layer=2, seed=31)
    F = dev(np.stack([W.random_rhs(60 + k, n) for k in range(nsrc)]))

    def call(s, nrec):
        rec = np.arange(3, int(np.prod(n)), 2, dtype=np.int64)[:nrec]
        return s.grad_td(F, rec, dev(W.random_rhs(70 + nrec, (nsrc, max(1, rec.size)))))

    s = htd.Solver(p, precision=precision, mode=mode)
    call(s, 50)
    d = htd.htd_grad_td_describe(s.handle)
    assert d["group"] == nsrc and d["lean"] == 0
    assert d["captures"] == (3 if mode == "exact" else 2)     # forward, a backward per run
    for nrec in (7, 400, 51, 50):
        J, gm, gR = call(s, nrec)
        assert htd.htd_grad_td_describe(s.handle) == d
        fresh = htd.Solver(p, precision=precision, mode=mode)
        J1, gm1, gR1 = call(fresh, nrec)
        assert J == J1 and torch.equal(gm, gm1) and torch.equal(gR, gR1)
        fresh.close()
    s.close()
