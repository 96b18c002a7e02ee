"""The plain form of a batch whose 2-D handles fit the SMs together: one resident-grid
launch, each rhs slot on its own share of the SMs.

Every output equals the handle's own application bit for bit (the kernels evaluate
the same expression), for tiny and ragged grids, several rhs slots with some idle,
both read-outs, beside a 3-D handle, and where the grids do not fit together (then
every handle runs its own sequence).
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

BATCHES = {
    "tiny": [((1, 7), 1, 1), ((3, 2), 1, 1), ((2, 40), 1, 1)],
    "slots": [((65, 70), 3, 2), ((33, 129), 2, 2), ((64, 64), 1, 1)],
    "large": [((401, 389), 1, 1), ((613, 300), 1, 1), ((97, 211), 1, 1)],
    "beside_3d": [((120, 90), 2, 1), ((40, 40, 40), 4, 3), ((77, 201), 1, 1)],
    "one": [((130, 257), 1, 1)],
    "no_fit": [((1101, 1101), 1, 1), ((700, 700), 1, 1)],
}


@pytest.mark.parametrize("name", BATCHES)
@pytest.mark.parametrize("mode", ["table1", "exact"])
def test_batch_equals_single_handles(name, mode):
    solvers, F, nrhs = [], [], []
    for k, (n, cap, r) in enumerate(BATCHES[name]):
        p = het_problem(len(n), n, T=2 + k % 2, layer=2, seed=20 + k)
        solvers.append(htd.Solver(p, precision="mixed", mode=mode, max_rhs=cap))
        F.append(dev(np.stack([W.random_rhs(50 + 7 * k + q, n) for q in range(r)])))
        nrhs.append(r)
    b = htd.Batch(solvers, nrhs)
    b.set_form(1)
    for _ in range(2):                              # a second run starts from rest again
        U = [host(u) for u in b.precond(F)]
    b.close()
    for s, f, u in zip(solvers, F, U):
        for q in range(f.shape[0]):
            assert np.isfinite(u[q]).all() and np.abs(u[q]).max() > 0
            assert np.array_equal(u[q], host(s.precond(f[q])))
        s.close()


def test_no_memory_for_the_resident_launch_leaves_the_handles_sequences():
    """An allocation that fails while a batch is built is reported (3: out of memory),
    except those of the resident launch, which the handles' own sequences replace: same
    outputs."""
    solvers, F = [], []
    for k, n in enumerate([(65, 70), (120, 33)]):
        solvers.append(htd.Solver(het_problem(2, n, T=2, layer=2, seed=30 + k), precision="mixed"))
        F.append(dev(W.random_rhs(60 + k, n)[None]))
    want = [host(s.precond(f[0])) for s, f in zip(solvers, F)]
    built = 0
    for k in range(24):
        b = None
        htd.htd_test_fail_alloc(k)
        try:
            b = htd.Batch(solvers, [1, 1])
            b.set_form(1)
        except htd.HtdError as e:
            assert e.status == 3
            if b:
                b.close()
            continue
        finally:
            htd.htd_test_fail_alloc(-1)
        built += 1
        for u, w in zip(b.precond(F), want):
            assert np.array_equal(host(u)[0], w)
        b.close()
    assert built >= 4                       # the three of the resident launch, and none
    for s in solvers:
        s.close()
