"""The two ways of a batch's plain run: the handles' own sequences, and the resident
launch of the 2-D handles that fit the SMs together.

The launch is planned for the right-hand sides that the batch carries, not for the
slots that its handles could hold; both ways give the same bits; both are timed and
the faster one runs; and where the launch finds no memory there is none.
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

OWN, RESIDENT = 1, 2                     # htd_batch_set_resident
LAST_OWN, LAST_RESIDENT = 1, 3           # describe_resident()["last"]


def _batch(shapes, max_rhs, nrhs, T=2):
    solvers, F = [], []
    for k, (n, cap, r) in enumerate(zip(shapes, max_rhs, nrhs)):
        p = het_problem(len(n), n, T=T + k % 2, layer=2, seed=40 + k)
        solvers.append(htd.Solver(p, precision="mixed", max_rhs=cap))
        F.append(dev(np.stack([W.random_rhs(90 + 7 * k + q, n) for q in range(r)])))
    return solvers, htd.Batch(solvers, nrhs), F


SHAPES = [(401, 389), (200, 301), (97, 211)]


@pytest.mark.parametrize("nrhs", [[1, 1, 1], [2, 1, 3]], ids=["one", "several"])
def test_the_launch_is_planned_for_the_rhs_of_the_batch(nrhs):
    found = []
    for cap in (nrhs, [8, 8, 8]):
        solvers, b, F = _batch(SHAPES, cap, nrhs)
        b.set_resident(RESIDENT)
        U = [host(u) for u in b.precond(F)]
        d = b.describe_resident()
        assert d["systems"] == sum(nrhs) and d["last"] == LAST_RESIDENT
        found.append((d["ctas"], U))
        b.close()
        for s in solvers:
            s.close()
    assert found[0][0] == found[1][0] > 0
    for a, c in zip(found[0][1], found[1][1]):
        assert np.array_equal(a, c)


def test_a_3d_handle_beside_it_is_judged_by_the_rhs_of_the_batch():
    """A 3-D handle whose launches fill the GPU with all its slots, but not with the one
    that the batch carries: nothing is gained by running the 2-D handles after it."""
    shapes = [(12, 16, 64), (120, 90)]
    systems = []
    for r in (64, 1):
        solvers, b, F = _batch(shapes, [64, 1], [r, 1])
        b.set_form(1)
        systems.append(b.describe_resident()["systems"])
        b.close()
        for s in solvers:
            s.close()
    assert systems == [1, 0]


@pytest.mark.parametrize("solve", [False, True], ids=["applications", "solve"])
def test_both_ways_are_timed_and_the_faster_runs(solve):
    solvers, b, F = _batch(SHAPES, [1, 1, 1], [1, 1, 1], T=20)
    b.set_form(1)
    first = None
    for k in range(4):
        if solve:
            out = b.solve(F, tol=1e-6, max_iters=6, allow_not_converged=True)[0]
        else:
            out = b.precond(F)
        out = [host(u) for u in out]
        first = first or out
        for u, w in zip(out, first):
            assert np.array_equal(u, w)
        if k == 0 and not solve:
            assert b.describe_resident()["last"] == LAST_RESIDENT
    d = b.describe_resident()
    own, res = d["ns_per_update_own"], d["ns_per_update_resident"]
    assert own > 0 and res > 0
    assert d["last"] == (LAST_OWN if own < res else LAST_RESIDENT)
    for pick, last in ((OWN, LAST_OWN), (RESIDENT, LAST_RESIDENT)):
        b.set_resident(pick)
        got = [host(u) for u in b.precond(F)]
        assert b.describe_resident()["last"] == last
        for s, f, u in zip(solvers, F, got):
            assert np.array_equal(u[0], host(s.precond(f[0])))
    b.close()
    for s in solvers:
        s.close()


def test_own_sequences_from_the_first_run():
    solvers, b, F = _batch(SHAPES, [1, 1, 1], [1, 1, 1])
    b.set_resident(OWN)
    U = b.precond(F)
    assert b.describe_resident()["last"] == LAST_OWN
    for s, f, u in zip(solvers, F, U):
        assert np.array_equal(host(u)[0], host(s.precond(f[0])))
    b.close()
    for s in solvers:
        s.close()


def test_grids_that_do_not_fit_have_no_resident_launch():
    solvers, b, F = _batch([(1101, 1101), (700, 700)], [1, 1], [1, 1])
    with pytest.raises(htd.HtdError) as e:
        b.set_resident(RESIDENT)
    assert e.value.status == 1
    b.set_resident(OWN)
    for s, f, u in zip(solvers, F, b.precond(F)):
        assert np.array_equal(host(u)[0], host(s.precond(f[0])))
    d = b.describe_resident()
    assert d["systems"] == 0 and d["ctas"] == 0
    b.close()
    for s in solvers:
        s.close()


def test_only_the_launchs_own_allocations_may_fail():
    """The resident launch's three allocations are a batch's last ones: with one of them
    failing there is no such launch, with an earlier one the batch reports it."""
    solvers = [htd.Solver(het_problem(2, n, T=2, layer=2, seed=30 + k), precision="mixed")
               for k, n in enumerate([(65, 70), (120, 33)])]
    F = [dev(W.random_rhs(60 + k, s.n)[None]) for k, s in enumerate(solvers)]
    want = [host(s.precond(f[0])) for s, f in zip(solvers, F)]
    outcome = []
    while not outcome or outcome[-1] != 2:
        assert len(outcome) < 60
        b = None
        htd.htd_test_fail_alloc(len(outcome))
        try:
            b = htd.Batch(solvers, [1, 1])
            b.set_form(1)
            htd.htd_test_fail_alloc(-1)
            for u, w in zip(b.precond(F), want):
                assert np.array_equal(host(u)[0], w)
            outcome.append(b.describe_resident()["systems"])
        except htd.HtdError as e:
            assert e.status == 3
            outcome.append(None)
        finally:
            htd.htd_test_fail_alloc(-1)
            if b:
                b.close()
    assert outcome[-4:] == [0, 0, 0, 2]
    assert len(outcome) > 8 and all(o is None for o in outcome[:-4])
    for s in solvers:
        s.close()
