"""The twisted sweep kernels on triangular factor storage at the sizes where their geometry
changes: lines at the edges of the 4 x 4 and 6 x 6 tiles (padded and whole last tile row), of
one and two CTAs per half (96 / 97 nodes), of the small and large thread counts (64 / 65), the
widest line that fits (145, 146) and the fallback beyond it (147); complex128 at the edges of
its row and column split; more lines than nodes per line and the reverse.

Local solves are compared with the oracle's banded LU.  How far a single-precision solve may
be off depends on the problem's conditioning (a whole domain without local PML is the worst
case), so the bound is the error of the general path, the cluster-split kernel on the plain
whole-block factor (front_kernel 1), on the same input: at most four times that, a factor of two
for eliminating from both ends (each half's Schur complements belong to a problem with one more
Dirichlet end) and one for storing the symmetric part.  Whole applications are compared with the
oracle's L-sweeps within 1e-4 (FP32) and 1e-10 (FP64), as at other sizes.
"""
import math
import os

import numpy as np
import pytest

import synth
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


def setup(L, n, npml, q, r, precision, **kw):
    m = synth.medium_smooth_bump(n, seed=3)
    omega = 2 * math.pi * 0.6 * n / 10
    prob = Problem(m, omega, npml)
    h = L.Handle(2, n, npml, (q, r), omega, torch.tensor(m, device="cuda"),
                 precision=getattr(L, "LSWEEP_" + precision), **kw)
    L.lsweep_factor(h.h)
    return prob, h


# (n, npml, q, r): lines of n / r + 2 npml (+ 2 or 4 at interior sides) nodes
WIDTHS = [(5, 2, 1, 1), (12, 2, 1, 1), (13, 2, 1, 1), (44, 10, 1, 1), (45, 10, 1, 1),
          (72, 10, 1, 1), (73, 10, 1, 1), (76, 10, 1, 1), (77, 10, 1, 1), (78, 10, 1, 1),
          (125, 10, 1, 1), (126, 10, 1, 1), (127, 10, 1, 1), (60, 6, 1, 3), (60, 6, 3, 1)]


@pytest.mark.parametrize("n,npml,q,r", WIDTHS)
@pytest.mark.parametrize("precision", ["C64", "C128"])
def test_local_solve_at_tile_edges(L, n, npml, q, r, precision):
    prob, h = setup(L, n, npml, q, r, precision)
    _, general = setup(L, n, npml, q, r, precision, front_kernel=1)
    ls = LSweeps(prob, q, r)
    rng = np.random.default_rng(n)
    for i, j in {(0, 0), (q - 1, r - 1), (q // 2, r // 2)}:
        shape = ls.loc[i, j].shape
        g = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
        err = []
        for hh in (h, general):
            x = torch.zeros(shape, dtype=torch.complex128, device="cuda")
            L.lsweep_local_solve(hh.h, i, j, torch.tensor(g, device="cuda"), x)
            err.append(rel(x.cpu().numpy(), ls.solve_local(i, j, g)))
        assert err[0] <= 4 * err[1], (i, j, err)
    h.close()
    general.close()


# every sweep family on lines of 58 / 60, 89 / 91, 97 / 99, 143 / 145 and (not square) 70 nodes
APPLIES = [(96, 12, 3, 3), (129, 22, 3, 3), (129, 26, 3, 3), (303, 20, 3, 3), (96, 10, 4, 2)]


@pytest.mark.parametrize("n,npml,q,r", APPLIES)
@pytest.mark.parametrize("precision,tol", [("C64", 1e-4), ("C128", 1e-10)])
def test_apply_at_tile_edges(L, n, npml, q, r, precision, tol):
    prob, h = setup(L, n, npml, q, r, precision)
    rng = np.random.default_rng(n)
    f = rng.standard_normal(prob.shape) + 1j * rng.standard_normal(prob.shape)
    z = h.ext_zeros()
    for _ in range(2):                              # launched directly, then from a graph
        z.fill_(complex(np.nan, np.nan))
        L.lsweep_apply(h.h, torch.tensor(f, device="cuda"), z)
        L.lsweep_sync(h.h)
        assert rel(z.cpu().numpy(), LSweeps(prob, q, r).apply(f.ravel())) < tol
    h.close()


@pytest.mark.parametrize("k", [1, 3, 5, 8])
def test_block_apply_wide_lines(L, k):
    """Block applications on lines above 64 nodes (four right-hand sides between two barriers)
    equal the single ones bit for bit, with the rounds full, partial and of one."""
    _, h = setup(L, 96, 20, 2, 2, "C64")            # lines of 90 nodes
    rng = np.random.default_rng(k)
    R = torch.tensor(rng.standard_normal((k,) + (h.Ne,) * 2)
                     + 1j * rng.standard_normal((k,) + (h.Ne,) * 2), device="cuda")
    Z = torch.full_like(R, complex(np.nan, np.nan))
    L.lsweep_apply_multi(h.h, R, Z)
    L.lsweep_sync(h.h)
    for c in range(k):
        z = h.ext_zeros()
        L.lsweep_apply(h.h, R[c].contiguous(), z)
        torch.cuda.synchronize()
        assert torch.equal(z, Z[c]), c
    h.close()
