"""htd_grad_td where one source's workspace is beyond the bound of a group (1 GiB).

Such a source keeps eight multipliers at a time instead of a segment's, with the same bits:
every checkpoint interval gives the same gradient.
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

GIB = 1 << 30


@pytest.mark.parametrize("n,mode,intervals", [((100, 120, 140), "table1", (55, 64)),
                                              ((1400, 1500), "exact", (70, 96))])
def test_few_multipliers_give_the_same_gradient(n, mode, intervals):
    p = het_problem(len(n), n, T=12, layer=6, seed=31)
    s = htd.Solver(p, precision="mixed", mode=mode, restart=2)
    steps = s.params["steps"]
    F = dev(W.random_rhs(60, n)[None])
    rec = np.arange(3, int(np.prod(n)), 1001, dtype=np.int64)
    d = dev(W.random_rhs(70, (1, rec.size)))
    want = s.grad_td(F, rec, d, checkpoint_every=12)
    assert htd.htd_grad_td_describe(s.handle)["workspace_bytes"] <= GIB
    pitch = (32 + n[-1] + 1 + 31) // 32 * 32
    plane = 4 * pitch * np.prod([m + 2 for m in n[:-1]])
    for c in intervals:
        assert 8 < c <= steps and (2 * -(-steps // c) + 2 * c + 8) * plane > GIB
        got = s.grad_td(F, rec, d, checkpoint_every=c)
        ws = htd.htd_grad_td_describe(s.handle)
        assert ws["lean"] == 0 and ws["workspace_bytes"] > 0
        # 2 ceil(steps / c) + c + 8 + 8 planes, the sums and U; a segment's multipliers
        # would be c - 8 planes more
        planes = 2 * -(-steps // c) + c + 16
        rest = 8 * (np.prod([m + 1 for m in n]) + 3 * np.prod(n))
        assert ws["workspace_bytes"] <= 1.01 * (planes * plane + rest)
        assert got[0] == want[0] and torch.equal(got[1], want[1]) and torch.equal(got[2], want[2])
    s.close()
