"""Half-row factor storage and its sweep kernel (3D planes too wide for a row slab per CTA) where
the geometry changes: even and odd planes (an even one has an antipodal pair in every row), the
last plane of each width of the column window (529, 576, 1089 nodes for complex64; 441, 484 for
complex128), line vectors in shared and in global memory, clusters of 2, 4 and 8 CTAs, and beams of
unequal sizes in one plan.

Local solves of one box are compared with a sparse direct solve, applications with the oracle's,
within the bounds of the other 3D sizes: 1e-4 (complex64) and 1e-10 (complex128) relative.
"""
import math
import os

import numpy as np
import pytest
from scipy.sparse.linalg import splu

import synth
from oracle.cdd import CDD
from oracle.lsweeps import LSweeps
from oracle.problem import Problem

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


def rel(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b)))


def setup(L, n, npml, q, r, precision):
    m = synth.medium_layered_3d(n, seed=3)
    omega = 2 * math.pi * 1.5 * n / 8
    h = L.Handle(3, n, npml, (q, r), omega, torch.tensor(m, device="cuda"),
                 precision=getattr(L, "LSWEEP_" + precision))
    L.lsweep_factor(h.h)
    return Problem(m, omega, npml), h


# planes of (n + 2 npml)^2 nodes
SIDES = [("C64", s, 1e-4) for s in (18, 23, 24, 28, 32, 33, 34)] + \
        [("C128", s, 1e-10) for s in (15, 18, 21, 22, 23, 24)]


@pytest.mark.parametrize("precision,side,tol", SIDES)
def test_local_solve_at_plane_edges(L, precision, side, tol):
    prob, h = setup(L, side - 4, 2, 1, 1, precision)
    lp = CDD(prob, 1, 1).local(0, 0)
    rng = np.random.default_rng(side)
    g = rng.standard_normal(lp.shape) + 1j * rng.standard_normal(lp.shape)
    x = torch.zeros(lp.shape, dtype=torch.complex128, device="cuda")
    L.lsweep_local_solve(h.h, 0, 0, torch.tensor(g, device="cuda"), x)
    want = splu(lp.A.tocsc()).solve(g.ravel())
    assert rel(x.cpu().numpy(), want) < tol
    h.close()


@pytest.mark.parametrize("precision,tol", [("C64", 1e-4), ("C128", 1e-10)])
def test_apply_unequal_beams(L, precision, tol):
    """27 cells in 3 x 1 beams: planes of 465 and 527 nodes in one plan."""
    prob, h = setup(L, 27, 2, 3, 1, precision)
    rng = np.random.default_rng(5)
    f = rng.standard_normal(prob.shape) + 1j * rng.standard_normal(prob.shape)
    want = LSweeps(prob, 3, 1).apply(f.ravel())
    z = h.ext_zeros()
    for _ in range(2):                              # launched directly, then from a graph
        z.fill_(complex(np.nan, np.nan))
        L.lsweep_apply(h.h, torch.tensor(f, device="cuda"), z)
        L.lsweep_sync(h.h)
        assert rel(z.cpu().numpy(), want) < tol
    h.close()
