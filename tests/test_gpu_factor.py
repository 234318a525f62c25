"""The blocked factorisation in shared memory where its form changes: lines of up to 64, 96, 128
and 158 nodes take 2, 3, 4 and 6 register rows per lane (64 / 65 and 96 / 97 are among the sizes
of the twisted sweep kernels' tests), beyond 158 the column by column form takes over; the last
panel of 8 columns is whole or has 1, 2, 6 or 7.

Applications on 3 x 3 subdomains (lines of the named width inside, two nodes less at the border)
are compared with the oracle's L-sweeps within 1e-4 as at other sizes, and above 150 nodes, where
the column by column form itself is up to 1.3e-4 off, within four times that; blocks stored whole
(front_kernel 1) take the same factorisation through another store."""
import math
import os

import numpy as np
import pytest

import synth
from oracle.lsweeps import LSweeps
from oracle.problem import Problem

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

_oracle = {}


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1909_01467_gb300 import build, lsweep
    if not os.path.exists(lsweep._LIB_PATH):
        build.build()
    return lsweep


@pytest.mark.parametrize("width", [18, 23, 128, 129, 158, 159])
@pytest.mark.parametrize("kernel", [0, 1])
def test_apply_at_factor_edges(L, width, kernel):
    npml = 20 if width > 100 else 4
    n = 3 * (width - 4 - 2 * npml)
    m = synth.medium_smooth_bump(n, seed=3)
    omega = 2 * math.pi * 0.6 * n / 10
    prob = Problem(m, omega, npml)
    rng = np.random.default_rng(width)
    f = rng.standard_normal(prob.shape) + 1j * rng.standard_normal(prob.shape)
    if width not in _oracle:
        _oracle[width] = LSweeps(prob, 3, 3).apply(f.ravel())
    h = L.Handle(2, n, npml, (3, 3), omega, torch.tensor(m, device="cuda"),
                 precision=L.LSWEEP_C64, front_kernel=kernel)
    L.lsweep_factor(h.h)
    z = h.ext_zeros()
    L.lsweep_apply(h.h, torch.tensor(f, device="cuda"), z)
    L.lsweep_sync(h.h)
    err = np.linalg.norm(z.cpu().numpy().ravel() - _oracle[width]) / np.linalg.norm(_oracle[width])
    assert err < (1e-4 if width < 150 else 5e-4)
    h.close()
