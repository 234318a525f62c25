"""Block applications on lines of 65 to 92 nodes, where two threads own a row, each for every second
right-hand side: equal to the single applications bit for bit on both sides of the steps of the thread
count (136 to 253 tiles; the fewest threads per row are at 68, 72 and 80 nodes) and with the last round
of four full or not, and faster than applying one after another."""
import math
import os

import numpy as np
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


def setup(L, n, npml, q, k):
    m = torch.tensor(synth.medium_smooth_bump(n, seed=3), device="cuda")
    h = L.Handle(2, n, npml, (q, q), 2 * math.pi * 0.6 * n / 10, m, precision=L.LSWEEP_C64)
    L.lsweep_factor(h.h)
    rng = np.random.default_rng(n + k)
    R = torch.tensor(rng.standard_normal((k,) + (h.Ne,) * 2)
                     + 1j * rng.standard_normal((k,) + (h.Ne,) * 2), device="cuda")
    return h, R


@pytest.mark.parametrize("width", [65, 68, 69, 72, 80, 81, 92])
@pytest.mark.parametrize("k", [2, 5, 8])
def test_block_equals_singles(L, width, k):
    h, R = setup(L, 3 * (width - 28), 12, 3, k)
    Z = torch.full_like(R, complex(np.nan, np.nan))
    L.lsweep_apply_multi(h.h, R, Z)
    for c in range(k):
        z = h.ext_zeros()
        L.lsweep_apply(h.h, R[c].contiguous(), z)
        L.lsweep_sync(h.h)
        assert torch.equal(z, Z[c]), c
    h.close()


@pytest.mark.parametrize("width", [68, 92])
def test_block_of_eight_is_faster(L, width):
    """Measured 0.71 of the time of eight single applications (0.94 and 0.98 with one owner per row)."""
    h, R = setup(L, 8 * (width - 28), 12, 8, 8)
    Z = torch.zeros_like(R)
    rows = [R[c].contiguous() for c in range(8)]
    zs = [h.ext_zeros() for _ in range(8)]

    def block():
        L.lsweep_apply_multi(h.h, R, Z)

    def singles():
        for r, z in zip(rows, zs):
            L.lsweep_apply(h.h, r, z)

    def ms(fn):
        t = []
        for _ in range(9):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            fn()
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        return sorted(t[2:])[3]

    block(), singles()
    assert ms(block) < 0.88 * ms(singles)
    h.close()
