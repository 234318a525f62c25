"""complex128 twisted solves whose line vectors do not fit shared memory, and the widest that do:
subdomains of many lines, lines of 99 to 108 nodes, and 3D planes of up to 92 nodes (all of whose sources are built in global memory).

Each plan stores fewer factor bytes than for the cluster split (it is twisted: triangles instead of
whole blocks); its applications match the oracle's within 1e-10, directly and
from a graph, and its local solves are at most four times as far from a sparse direct solve as the
cluster split's (as in the tests of the other twisted sizes).
"""
import math
import os

import numpy as np
import pytest

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


def setup(L, dim, n, npml, q, r, **kw):
    m = synth.medium_smooth_bump(n, seed=3) if dim == 2 else synth.medium_layered_3d(n, seed=3)
    omega = 2 * math.pi * (0.6 * n / 10 if dim == 2 else 1.5 * n / 8)
    h = L.Handle(dim, n, npml, (q, r), omega, torch.tensor(m, device="cuda"),
                 precision=L.LSWEEP_C128, **kw)
    L.lsweep_factor(h.h)
    return Problem(m, omega, npml), h


# lines x nodes: 228 x 90 (12 warps), 176 x 36 (3 warps), 312 x 52 (6 warps), 108 x 108; in shared
# memory still 99 x 99 and 100 x 100 (the widest); 198 x 92 just past it; planes of 36 to 81 nodes
PLANS = [(2, 420, 8, 2, 6), (2, 160, 8, 1, 10), (2, 288, 12, 1, 12), (2, 240, 12, 3, 3),
         (2, 213, 12, 3, 3), (2, 216, 12, 3, 3), (2, 360, 8, 2, 5),
         (3, 9, 1, 3, 3), (3, 6, 1, 2, 2), (3, 5, 2, 1, 1)]


@pytest.mark.parametrize("dim,n,npml,q,r", PLANS)
def test_apply_and_local_solves(L, dim, n, npml, q, r):
    prob, h = setup(L, dim, n, npml, q, r)
    _, general = setup(L, dim, n, npml, q, r, front_kernel=1)
    assert L.lsweep_factor_bytes(h.h)[0] < L.lsweep_factor_bytes(general.h)[0]
    rng = np.random.default_rng(n)
    f = rng.standard_normal(prob.shape) + 1j * rng.standard_normal(prob.shape)
    want = LSweeps(prob, q, r).apply(f.ravel())
    z = h.ext_zeros()
    for _ in range(2):                              # launched directly, then from a graph
        z.fill_(complex(np.nan, np.nan))
        L.lsweep_apply(h.h, torch.tensor(f, device="cuda"), z)
        L.lsweep_sync(h.h)
        assert rel(z.cpu().numpy(), want) < 1e-10
    from scipy.sparse.linalg import splu
    for i, j in {(0, 0), (q // 2, r // 2)}:
        lp = CDD(prob, q, r).local(i, j)
        g = rng.standard_normal(lp.shape) + 1j * rng.standard_normal(lp.shape)
        exact = splu(lp.A.tocsc()).solve(g.ravel())
        err = []
        for hh in (h, general):
            x = torch.zeros(lp.shape, dtype=torch.complex128, device="cuda")
            L.lsweep_local_solve(hh.h, i, j, torch.tensor(g, device="cuda"), x)
            err.append(rel(x.cpu().numpy(), exact))
        assert err[0] <= 4 * err[1], (i, j, err)
    h.close()
    general.close()


def test_autotune_reaches_the_twisted_kernel(L):
    """A plan set up with the cluster split has room for the line vectors too: tuning may move to the
    twisted kernel, and the application it leaves selected still matches."""
    prob, h = setup(L, 2, 160, 8, 1, 10, front_kernel=1)
    rng = np.random.default_rng(2)
    f = torch.tensor(rng.standard_normal(prob.shape) + 0j, device="cuda")
    before, after = h.ext_zeros(), h.ext_zeros()
    L.lsweep_apply(h.h, f, before)
    L.lsweep_autotune(h.h, 2)
    L.lsweep_apply(h.h, f, after)
    L.lsweep_sync(h.h)
    assert rel(after.cpu().numpy(), before.cpu().numpy()) < 1e-10
    h.close()
