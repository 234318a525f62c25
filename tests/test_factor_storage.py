"""Storage of the twisted factors, checked on the host: the room that setup takes for the factors,
and the map of a block's entries to its triangle's tiles (csrc/internal.h).

The map is compiled from the header as host code.  Every pair of a row and a column of a block has
one place, the same for its mirror image; places are in range, distinct, and apart from the
couplings' and the padding's; the worker threads' tiles are the stored ones, each once.
"""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1909_01467_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <vector>
#include "internal.h"
using namespace lsw;
static int check(int b, TileStore s, int es) {
  const int n = block_elems(b, s), G = tile_rows(b, s.T), bs = (b + 1) & ~1;
  std::vector<int> used(n, 0);
  for (int q = 0; q < s.NQ; ++q) {
    const int part = q ? part_elems(b, s, 0) : 0, c0 = part + part_cpl(b, s, q);
    if (c0 % 2 || part % 2 || c0 + 2 * bs != part + part_elems(b, s, q)) return 1;
    for (int p = 0; p < 2 * bs; ++p) used[c0 + p] += 1;
    for (int o = 0; o < tile_count(G, s.NQ, q); ++o) {
      int I = -1, J = -1;
      const bool has = s.NQ == 1 ? worker_tile<1>(o, G, q, I, J) : worker_tile<2>(o, G, q, I, J);
      if (!has || !(0 <= J && J < I && I < G) || (s.NQ == 2 && ((I + J) & 1) != q) ||
          tile_number(I, J, s.NQ) != o) return 2;
    }
    int I, J;
    if (s.NQ == 1 ? worker_tile<1>(tile_count(G, 1, q), G, q, I, J)
                  : worker_tile<2>(tile_count(G, 2, q), G, q, I, J)) return 3;
  }
  for (int r = 0; r < G * s.T; ++r)
    for (int c = 0; c <= r; ++c) {
      const int at = tile_index(b, s, es, r, c);
      if (at < 0 || at >= n || at != tile_index(b, s, es, c, r) || used[at]++) return 4;
    }
  return 0;
}
int main() {
  int bad = 0;
  for (int b = 1; b <= 160; ++b)
    for (int es = 8; es <= 16; es += 8)
      for (int nq = 1; nq <= 2; ++nq)
        if (int rc = check(b, TileStore{nq == 1 ? 4 : 6, nq}, es)) {
          printf("b %d NQ %d es %d: %d\n", b, nq, es, rc);
          bad = 1;
        }
  for (int b = 1; b <= 160; ++b) {
    const long long whole = (b + 2LL) * (b + ((2 - b % 4) + 4) % 4);
    for (int nq = 1; nq <= 2; ++nq) {
      const TileStore s{nq == 1 ? 4 : 6, nq};
      const long long room = block_room(b, (int)whole, s);
      if (room < whole || room < block_elems(b, s) || room % 2) {
        printf("b %d NQ %d: room %lld\n", b, nq, room);
        bad = 1;
      }
    }
    if (block_room(b, (int)whole, TileStore{0, 1}) != whole) bad = 1;
  }
  puts(bad ? "bad" : "ok");
  return bad;
}
"""


def test_tile_map_and_room(tmp_path):
    from paper_1909_01467_gb300 import build
    src, exe = tmp_path / "storage.cu", tmp_path / "storage"
    src.write_text(HARNESS)
    subprocess.run([build._nvcc(), "-std=c++17", "-I" + CSRC, "-I" + os.path.join(ROOT, "include"),
                    str(src), "-o", str(exe)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout


@pytest.mark.parametrize("n,npml,precision,block", [
    (3, 1, "C64", 48),      # 5-node lines: a triangle's tiles (48 entries) are more than the whole
    (3, 1, "C128", 48),     # block with its couplings (42)
    (4, 1, "C64", 48),      # 6 nodes: as large; wider ones are smaller
    (12, 2, "C64", 324)])   # 16 nodes: whole blocks, which the plain kernels may be tuned to
def test_factor_room_of_setup(n, npml, precision, block):
    """The factor array holds every block of the form that is stored, ahead of the zero slack: here
    from the sizes that setup asks the allocator for (which then refuses, so nothing runs)."""
    from paper_1909_01467_gb300 import build
    from paper_1909_01467_gb300 import lsweep as L
    if not os.path.exists(L._LIB_PATH):
        build.build()
    sizes = []

    def alloc(nbytes, ctx):
        sizes.append(int(nbytes))
        return 0x1000 * len(sizes) if len(sizes) < 7 else None   # addresses nobody uses

    L.lsweep_set_allocator(alloc, lambda p, c: None)
    try:
        p = L.lsweep_default_params()
        p.n, p.npml, p.cdd_q, p.cdd_r, p.omega = n, npml, 1, 1, 10.0
        p.precision = getattr(L, "LSWEEP_" + precision)
        h = ctypes.c_void_p()
        rc = L.library().lsweep_setup(ctypes.byref(p), ctypes.c_void_p(0x1000), ctypes.byref(h))
        assert rc == L.LSWEEP_ENOMEM and not h.value
    finally:
        L.lsweep_set_allocator()
    es = 8 if precision == "C64" else 16
    assert (n + 2 * npml) * block * es + 4096 in sizes, sizes


@pytest.mark.gpu
@pytest.mark.parametrize("n", [2, 3, 4])
@pytest.mark.parametrize("precision,tol", [("C64", 1e-4), ("C128", 1e-10)])
def test_smallest_lines(n, precision, tol):
    """Lines of 4, 5 and 6 nodes: the twisted solve against the general path (front_kernel 1), within
    the bounds of applications at other sizes."""
    import numpy as np
    import synth
    torch = pytest.importorskip("torch")
    from paper_1909_01467_gb300 import build
    from paper_1909_01467_gb300 import lsweep as L
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(L._LIB_PATH):
        build.build()
    m = torch.tensor(synth.medium_smooth_bump(n, seed=3), device="cuda")
    g = torch.tensor(np.random.default_rng(n).standard_normal((n + 2,) * 2) + 0j, device="cuda")
    x = []
    for kernel in (0, 1):
        h = L.Handle(2, n, 1, (1, 1), 2.0, m, precision=getattr(L, "LSWEEP_" + precision),
                     front_kernel=kernel)
        L.lsweep_factor(h.h)
        z = torch.zeros_like(g)
        L.lsweep_local_solve(h.h, 0, 0, g, z)
        L.lsweep_sync(h.h)
        x.append(z)
        h.close()
    assert (x[0] - x[1]).norm() / x[1].norm() < tol
