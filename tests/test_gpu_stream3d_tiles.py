"""The streamed 3-D pair kernel's tile widths and z chunks against the z-march kernel.

The pair kernel covers a grid with 64 x 8 or 32 x 16 column tiles, whichever covers
fewer columns, two node rows per thread, and chunks of one plane up.  Sizes lie at
the tiles' edges: widths just over 32 and 64, an odd last row of a thread, chunks
whose last one has a single plane, grids of one plane.  Tolerance: every variant
evaluates the same sum per node in FP32; the z-march kernel leaves contraction to
the compiler, so as in the other kernel-variant tests they agree to 2e-6 relative
L2, while the pair kernel's own variants are bit-identical.
"""
import numpy as np
import pytest

from paper_2006_16861_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2006_16861_gb300 import htd  # noqa: E402
from test_gpu_parity import dev, het_problem, host, rel_l2  # noqa: E402

SIZES = [(1, 3, 5), (2, 17, 33), (5, 16, 32), (7, 15, 31), (9, 33, 97), (6, 8, 64), (5, 7, 65),
         (12, 9, 130), (3, 40, 96), (4, 1, 40), (33, 2, 2)]


@pytest.mark.parametrize("n", SIZES, ids=lambda n: "x".join(map(str, n)))
def test_tiles_and_chunks_agree(n):
    p = het_problem(3, n, T=2, layer=2, seed=9)
    F = dev(W.random_rhs(4, n))
    s0 = htd.Solver(p, precision="mixed", s3_kernel=htd.S3_ZMARCH)
    want = host(s0.precond(F))
    s0.close()
    got = []
    for kw in (dict(), dict(s3_zchunk=1), dict(s3_zchunk=2, s3_stages=4), dict(s3_zchunk=n[0]),
               dict(s3_zchunk=max(1, n[0] - 1), s3_stages=6), dict(max_rhs=2, s3_rhs_per_cta=2)):
        s = htd.Solver(p, precision="mixed", **kw)
        assert s.params["step_kernel"] == 2
        tx = s.params["tile"][0]
        cover = {w: -(-n[2] // w) * w * (-(-n[1] // (512 // w)) * (512 // w)) for w in (32, 64)}
        assert tx == (32 if cover[32] < cover[64] else 64) and s.params["tile"][1] == 512 // tx
        got.append(host(s.precond(F)))
        s.close()
    assert rel_l2(got[0].reshape(-1), want.reshape(-1)) <= 2e-6
    for g in got[1:]:
        assert np.array_equal(g, got[0])
