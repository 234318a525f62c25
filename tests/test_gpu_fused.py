"""Fused batches whose problems finish in another order than their dependency levels.

A fused application runs the union of the problems' levels, so the levels past those of the
smaller problems belong to the largest alone.  When that one has converged (or its source is
zero), these levels hold only CTAs of a problem that is left out, and the lane sums of the
others, launched after the last level, must still wait for the smaller problems' own last
levels.  Solutions and iteration counts equal those of the batch over streams bit for bit.
"""
import math
import os

import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1909_01467_gb300 import build, lsweep
    if not os.path.exists(lsweep._LIB_PATH):
        build.build()
    return lsweep


@pytest.mark.parametrize("kernel", [0, 2])
@pytest.mark.parametrize("first", ["loose", "zero source"])
def test_largest_problem_finishes_first(L, kernel, first):
    """128^2 on 4 x 4 subdomains and 512^2 on 16 x 16, which has about four times as many levels,
    both on lines of 50 and 52 nodes; the larger one stops after a few applications or at once."""
    sizes = [(128, 1e-12), (512, 0.5 if first == "loose" else 1e-8), (128, 1e-6)]
    out = {}
    for fused in (False, True):
        hs, fs, us = [], [], []
        for k, (n, tol) in enumerate(sizes):
            m = torch.tensor(synth.medium_smooth_bump(n, seed=2 + k), device="cuda")
            h = L.Handle(2, n, 8, (n // 32, n // 32), 2 * math.pi * 0.6 * n / 10, m, tol=tol,
                         precision=L.LSWEEP_C64, schedule=2, front_kernel=kernel)
            L.lsweep_factor(h.h)
            f = h.ext_zeros()
            if n == 128 or first == "loose":
                L.lsweep_extend_source(h.h, torch.tensor(
                    synth.source_gaussian(n, 2, (0.3, 0.6), 2.0 / n), device="cuda"), f)
            hs.append(h)
            fs.append(f)
            us.append(h.ext_zeros())
        torch.cuda.synchronize()
        infos = L.lsweep_solve_batch([h.h for h in hs], fs, us, fused=fused)
        torch.cuda.synchronize()
        out[fused] = us, [i.iterations for i in infos]
        for h in hs:
            h.close()
    its = out[True][1]
    assert its == out[False][1]
    assert its[1] < its[0], its                     # the order this test is about
    for a, b in zip(out[True][0], out[False][0]):
        assert torch.equal(a, b)
