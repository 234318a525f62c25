"""complex128 twisted solves on short lines, which take fewer warps per CTA and more CTAs per SM: up to
36 nodes 3 warps, up to 54 nodes 6, above 12.

The host test counts the local solves that one launch may hold (38 with one CTA per SM).  On the GPU,
local solves on both sides of each edge, and on lines so short that threads have one column or none,
are at most four times as far from the oracle's banded LU as the general path (front_kernel 1) on the
same input: a factor of two for eliminating from both ends and one for storing the symmetric part;
applications on subdomains of these widths match the oracle's L-sweeps within 1e-10.
"""
import math
import os

import numpy as np
import pytest

import synth


def library():
    from paper_1909_01467_gb300 import build, lsweep
    if not os.path.exists(lsweep._LIB_PATH):
        build.build()
    return lsweep


@pytest.mark.parametrize("n,npml,least", [(128, 4, 150), (256, 8, 150), (512, 8, 70)])
def test_solves_per_launch(n, npml, least):
    """16 x 16 subdomains on lines of 20, 36 and 52 nodes."""
    L = library()
    p = L.lsweep_default_params()
    p.n, p.npml, p.cdd_q, p.cdd_r, p.omega = n, npml, 16, 16, 40.0
    p.precision = L.LSWEEP_C128
    assert L.lsweep_plan_info(p)[2] >= least


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return library()


def setup(L, n, npml, q, r, **kw):
    import torch
    from oracle.problem import Problem
    m = synth.medium_smooth_bump(n, seed=3)
    omega = 2 * math.pi * 0.6 * n / 10
    h = L.Handle(2, n, npml, (q, r), omega, torch.tensor(m, device="cuda"),
                 precision=L.LSWEEP_C128, **kw)
    L.lsweep_factor(h.h)
    return Problem(m, omega, npml), h


def rel(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b)))


@pytest.mark.gpu
@pytest.mark.parametrize("n,npml", [(2, 1), (3, 1), (6, 1), (15, 2), (31, 2), (32, 2), (33, 2),
                                    (46, 4), (47, 4)])
def test_local_solve_at_warp_edges(L, n, npml):
    import torch
    from oracle.lsweeps import LSweeps
    prob, h = setup(L, n, npml, 1, 1)
    _, general = setup(L, n, npml, 1, 1, front_kernel=1)
    ls = LSweeps(prob, 1, 1)
    rng = np.random.default_rng(n)
    g = rng.standard_normal(prob.shape) + 1j * rng.standard_normal(prob.shape)
    err = []
    for hh in (h, general):
        x = torch.zeros(prob.shape, dtype=torch.complex128, device="cuda")
        L.lsweep_local_solve(hh.h, 0, 0, torch.tensor(g, device="cuda"), x)
        err.append(rel(x.cpu().numpy(), ls.solve_local(0, 0, g)))
        hh.close()
    assert err[0] <= 4 * err[1], err


@pytest.mark.gpu
@pytest.mark.parametrize("n,npml,q,r", [(64, 4, 8, 8), (64, 8, 4, 4), (68, 8, 4, 4),
                                        (78, 12, 3, 3), (81, 12, 3, 3), (120, 4, 3, 12)])
def test_apply_at_warp_edges(L, n, npml, q, r):
    """Widest lines of 20, 36, 37, 54, 55 and (more lines than nodes per line) 22 nodes; narrower
    ones at the borders."""
    import torch
    from oracle.lsweeps import LSweeps
    prob, h = setup(L, n, npml, q, r)
    rng = np.random.default_rng(n)
    f = rng.standard_normal(prob.shape) + 1j * rng.standard_normal(prob.shape)
    want = LSweeps(prob, q, r).apply(f.ravel())
    z = h.ext_zeros()
    for _ in range(2):                              # launched directly, then from a graph
        z.fill_(complex(np.nan, np.nan))
        L.lsweep_apply(h.h, torch.tensor(f, device="cuda"), z)
        L.lsweep_sync(h.h)
        assert rel(z.cpu().numpy(), want) < 1e-10
    h.close()
