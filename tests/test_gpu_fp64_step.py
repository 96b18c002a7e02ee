"""The FP64 step from the assembled stencil against the FP64 oracle.

Sizes lie at the edges of the kernel's 32 x 4 tiles and z columns, with one-node
axes (every neighbour a ghost, every negative offset's index clamped) and odd
lengths; a handle with several right-hand sides puts them beyond the first
plane stack.  Tolerance: the FP64 parity tolerance 1e-10 of the other tests
(the recurrence sums 3^d products per node in another order than the oracle;
a run of a few hundred steps keeps that within some hundred ulps).
"""
import numpy as np
import pytest

import oracle
from paper_2006_16861_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2006_16861_gb300 import htd  # noqa: E402
from test_gpu_parity import dev, het_problem, host, rel_l2  # noqa: E402

SIZES_3D = [(1, 1, 1), (1, 1, 40), (40, 1, 1), (1, 9, 1), (5, 4, 32), (3, 5, 33), (17, 3, 31),
            (33, 8, 65)]


@pytest.mark.parametrize("n", SIZES_3D, ids=lambda n: "x".join(map(str, n)))
@pytest.mark.parametrize("mode", ["table1", "exact"])
def test_fp64_3d_step_matches_the_oracle(n, mode):
    p = het_problem(3, n, T=2, layer=2, seed=5)
    s = htd.Solver(p, precision="fp64", mode=mode)
    assert s.params["step_kernel"] == 0
    o = oracle.Oracle(p)
    F = W.random_rhs(8, n)
    assert rel_l2(host(s.precond(dev(F))).reshape(-1), o.precond(F, mode).reshape(-1)) <= 1e-10
    X = W.random_rhs(9, n)                       # apply_H reads the same (scaled) planes
    assert rel_l2(host(s.apply_H(dev(X))).reshape(-1), o.apply_H(X).reshape(-1)) <= 1e-12
    s.close()


def test_fp64_3d_step_in_a_batch_equals_single():
    p = het_problem(3, (6, 9, 34), T=2, layer=2, seed=6)
    s = htd.Solver(p, precision="fp64", max_rhs=3)
    F = np.stack([W.random_rhs(k, p.n) for k in (1, 2)])
    b = htd.Batch([s], [2])
    U = host(b.precond([dev(F)])[0])
    for r in range(2):
        assert np.array_equal(U[r], host(s.precond(dev(F[r]))))
    b.close()
    s.close()


# one tile, one tile row or column, tiles two nodes wide or high, last tiles of one
# node, the ring reaching past the domain, and tiles of many nodes per thread
SIZES_2D = [(1, 1), (1, 7), (2, 3), (5, 5), (3, 400), (400, 3), (305, 5), (31, 33), (153, 77),
            (97, 613), (500, 501)]


@pytest.mark.parametrize("n", SIZES_2D, ids=lambda n: "x".join(map(str, n)))
@pytest.mark.parametrize("mode", ["table1", "project"])
def test_fp64_2d_resident_and_one_step_match_the_oracle(n, mode):
    p = het_problem(2, n, T=2, layer=2, seed=5)
    o = oracle.Oracle(p)
    F = W.random_rhs(8, n)
    want = o.precond(F, mode).reshape(-1)
    got = []
    for kw in (dict(tblock=1), dict(tb_form=htd.TB_RESIDENT)):
        s = htd.Solver(p, precision="fp64", mode=mode, **kw)
        assert s.params["step_kernel"] == (0 if "tblock" in kw else 4)
        U = host(s.precond(dev(F)))
        assert rel_l2(U.reshape(-1), want) <= 1e-10
        got.append(U)
        s.close()
    if mode == "table1":
        assert np.array_equal(got[0], got[1])
