"""complex128 lines of 109 to 128 nodes with too many lines for a row slab per CTA: the wide sweep
kernel on whole blocks (from 129 nodes on it streams half rows).  Stored bytes show the form;
applications match the oracle's L-sweeps within 1e-10, directly and from a graph, and local solves a
sparse direct solve."""
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


@pytest.mark.parametrize("n,whole", [(404, True), (480, True), (484, False)])
def test_apply_and_local_solve(L, n, whole):
    """Lines of up to 109, 128 and 129 nodes (two nodes less at the border) on 1 x 4 subdomains."""
    npml, q, r = 2, 1, 4
    m = synth.medium_smooth_bump(n, seed=3)
    omega = 2 * math.pi * 0.6 * n / 10
    prob = Problem(m, omega, npml)
    h = L.Handle(2, n, npml, (q, r), omega, torch.tensor(m, device="cuda"), precision=L.LSWEEP_C128)
    L.lsweep_factor(h.h)
    entries = sum((n // r + 2 * npml + (2 if j in (0, r - 1) else 4)) ** 2 for j in range(r))
    stored = L.lsweep_factor_bytes(h.h)[0] / (16 * (n + 2 * npml))
    assert (stored > entries) == whole
    rng = np.random.default_rng(n)
    f = rng.standard_normal(prob.shape) + 1j * rng.standard_normal(prob.shape)
    want = LSweeps(prob, q, r).apply(f.ravel())
    z = h.ext_zeros()
    for _ in range(2):
        z.fill_(complex(np.nan, np.nan))
        L.lsweep_apply(h.h, torch.tensor(f, device="cuda"), z)
        L.lsweep_sync(h.h)
        assert rel(z.cpu().numpy(), want) < 1e-10
    from scipy.sparse.linalg import splu
    lp = CDD(prob, q, r).local(0, 1)
    g = rng.standard_normal(lp.shape) + 1j * rng.standard_normal(lp.shape)
    x = torch.zeros(lp.shape, dtype=torch.complex128, device="cuda")
    L.lsweep_local_solve(h.h, 0, 1, torch.tensor(g, device="cuda"), x)
    assert rel(x.cpu().numpy(), splu(lp.A.tocsc()).solve(g.ravel())) < 1e-10
    h.close()
