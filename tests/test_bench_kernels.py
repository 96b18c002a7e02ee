"""The benchmark's kernel names and FLOP counts against the library's sources (CPU).

The FP64 steps compute asm2d_step (2-D) and the sum over 26 neighbours of
step3d_asm_kernel; a multiply-add counts two.  The fraction of the FP64 pipe is a
fraction: at the step times that the kernels' comments give it stays below one.
"""
import glob
import os
import re
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)
import bench  # noqa: E402

CSRC = os.path.join(ROOT, "paper_2006_16861_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def body(text, start):
    """The braces' block that follows `start`."""
    i = text.index("{", text.index(start))
    depth = 0
    for j in range(i, len(text)):
        depth += (text[j] == "{") - (text[j] == "}")
        if depth == 0:
            return text[i:j + 1]
    raise AssertionError(start)


def test_fp64_flops_2d_are_those_of_the_step():
    b = body(source("htd_internal.h"), "double asm2d_step(")
    flops = 2 * b.count("__fma_rn(") + b.count("__dmul_rn(") + b.count("__dadd_rn(")
    assert bench.FP64_FLOPS_PER_UPDATE[2] == flops


def test_fp64_flops_3d_are_those_of_the_step():
    b = body(source("htd_kernels.cu"), "step3d_asm_kernel(const double")
    # own node: a product and four multiply-adds; neighbours: a product, then one
    # multiply-add in the loop over the other 25; their sum; the update
    assert b.count("fma(") == 6 and b.count("-b * fim[i]") == 1 and b.count("acc += own") == 1
    assert bench.FP64_FLOPS_PER_UPDATE[3] == (1 + 4 * 2) + (1 + 25 * 2) + 1 + 2


@pytest.mark.parametrize("ndim,nodes,us", [(3, 96 ** 3, 58.0), (2, 801 ** 2, 19.6)])
def test_fp64_fraction_is_below_one_at_the_measured_times(ndim, nodes, us):
    tflops = bench.FP64_FLOPS_PER_UPDATE[ndim] * nodes / (us * 1e-6) / 1e12
    assert 0.5 < tflops / bench.peaks(152)["fp64_tflops"] <= 1.0


def params(sk, **kw):
    return dict(dict(step_kernel=sk, tile=[64, 8, 16], steps=120, steps_per_launch=1), **kw)


NAMES = [(params(0), n, p) for n in (2, 3) for p in ("float", "double")] + \
        [(params(3), n, p) for n in (2, 3) for p in ("float", "double")] + \
        [(params(4, steps_per_launch=120), 2, p) for p in ("float", "double")] + \
        [(params(4, steps_per_launch=64), 2, "float"), (params(1, tile=[48, 144, 2]), 2, "float"),
         (params(1, tile=[48, 144, 1]), 2, "float"), (params(2), 3, "float"),
         (params(2, tile=[32, 16, 16]), 3, "float"), (params(2, tile=[32, 8, 64]), 3, "float")]


def test_every_kernel_name_is_a_kernel():
    text = "".join(source(os.path.basename(f)) for f in glob.glob(os.path.join(CSRC, "*.cu")))
    kernels = set(re.findall(r"\b(\w+_kernel)\(const|\b(\w+_kernel)\(", text))
    kernels = {a or b for a, b in kernels}
    names = [bench.step_kernel_name(*x)[0].split("<")[0] for x in NAMES]
    assert set(names) <= kernels, set(names) - kernels
    # each form of the resident kernel and each precision of the one-step one its own
    assert len({bench.step_kernel_name(*x)[0].split("<")[0] for x in NAMES[8:11]}) == 3
    assert bench.step_kernel_name(*NAMES[0])[0] != bench.step_kernel_name(*NAMES[1])[0]
