// Phase 2 "Factorize" (Sec. 3): block-tridiagonal LU of every local matrix A_ij over its
// grid lines (2D) or planes (3D).  With A_kk the block of line k and the diagonal
// couplings L_k = U_{k-1} = diag(l_k) between lines k-1 and k (A is complex symmetric),
//   D_0 = A_00,  D_k = A_kk - diag(l_k) D_{k-1}^-1 diag(l_k),
// and the dense inverses D_k^-1 are stored row-major (row stride bp, zero padding) so that
// any range of rows is contiguous for the substitutions of the sweeps.  Two more rows
// follow each block: the couplings l_k (line k to k + 1) and l_{k-1}, which the forward and
// the backward substitution step of block k use, so that one contiguous copy brings a step
// everything it reads.  One CTA per
// subdomain; each D_k is inverted in shared memory by Gauss-Jordan elimination with
// partial (row) pivoting.
#include <math.h>

#include <type_traits>

#include "gj.cuh"

namespace lsw {

// Block-tridiagonal LU of one local problem per CTA, the Schur complement of each line
// built and inverted in shared memory.  Lines are eliminated in the order 0, 1, .., L-1
// (D_k = A_kk - c_{k-1} D_{k-1}^-1 c_{k-1}, c_k the diagonal coupling of lines k and k+1),
// or, for a factor twisted at m = twist_line(L), first 0 .. m-1 as above, then L-1 down to
// m+1 (E_k = A_kk - c_k E_{k+1}^-1 c_k), and last the middle line, whose Schur complement
// takes both neighbours' updates: T_m = A_mm - c_{m-1} D_{m-1}^-1 c_{m-1} - c_m E_{m+1}^-1 c_m.
// Stored block k holds the inverse of line k's Schur complement and the couplings c_k, c_{k-1}.
// RPL > 0: the blocked inverse for lines of up to 32 RPL nodes (threads and CTAs per SM:
// simt_threads); 0: the column by column one (complex128, and lines of more than 158 nodes, whose
// block leaves no room for the scratch).  Up to 96 nodes two CTAs of 256 threads share an SM, so
// that one's tiles fill the other's steps; wider blocks are alone on theirs and take more warps,
// as many as leave warp 0 its rows in registers (a scheduler's 16384 over its warps).
// The column by column form also has to leave room for a second CTA (64 registers a thread; with 105
// there was one per SM, and 16 x 16 subdomains of 36-node lines in complex128 took 15.1 ms instead
// of 13.2).
__host__ __device__ constexpr int simt_threads(int rpl) {
  return rpl == 0 || rpl == 4 ? 512 : rpl == 6 ? 384 : 256;
}
template <typename C, int RPL>
__global__ void __launch_bounds__(simt_threads(RPL), RPL == 4 || RPL == 6 ? 1 : 2)
k_factor_simt(const SubGeom* __restrict__ subs, const C* __restrict__ lcoef,
                              long long cstride, C* __restrict__ fac, int dim, TileStore ts,
                              int* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SubGeom g = subs[blockIdx.x];
  const int b = g.b, bp = g.bp, L = g.L, Lx = g.Lx;
  C* M = reinterpret_cast<C*>(smem_raw);
  // column by column: the column and the row of a step, the interchanges; blocked: its scratch,
  // the pivot rows and the step of each
  C* f = M + (size_t)bp * b;
  C* prow = f + b;
  int* perm = reinterpret_cast<int*>(RPL ? f + gj_scratch(b, bp) : prow + b);
  int* step_of = perm + b;
  // entry (r, c) of the inverse
  auto inverse = [&](int r, int c) -> C& {
    if constexpr (RPL > 0) return M[step_of[c] * bp + perm[r]];
    else return M[(size_t)c * bp + r];
  };
  const C* d = lcoef + g.node_off;
  const C* cx = d + cstride;
  const C* cy = d + 2 * cstride;
  const C* cl = dim == 3 ? d + 3 * cstride : cy;   // coupling between consecutive lines
  const int tid = threadIdx.x, nth = blockDim.x;
  const bool twisted = ts.T > 0;
  const int m = twisted ? twist_line(L) : L;
  for (int st = 0; st < L; ++st) {
    // line k; coupling line ci of the update by the inverse held in M (the previous line's),
    // and cg of the update by D_{m-1}^-1 read back from the stored factor (middle line only)
    int k, ci = -1, cg = -1;
    if (st < m) {
      k = st;
      if (k > 0) ci = k - 1;
    } else if (st < L - 1) {
      k = L - 1 - (st - m);
      if (k < L - 1) ci = k;
    } else {
      k = m;
      if (m < L - 1) ci = m;
      if (m > 0) cg = m - 1;
    }
    const long long bstr = twisted ? block_elems(b, ts) : g.bs;
    const C* Dg = fac + g.fac_off + (cg < 0 ? 0 : cg) * bstr;
    const C* Di = fac + g.fac_off + (ci < 0 ? 0 : ci) * bstr;
    // Schur complement of line k, built in place over the previous inverse
    for (int idx = tid; idx < b * b; idx += nth) {
      int col = idx / b, row = idx - col * b;
      size_t kb = (size_t)k * b;
      C v = czero<C>();
      if (row == col) v = d[kb + row];
      else if (col == row + 1) v = cx[kb + row];
      else if (row == col + 1) v = cx[kb + col];
      else if (dim == 3 && col == row + Lx) v = cy[kb + row];
      else if (dim == 3 && row == col + Lx) v = cy[kb + col];
      if (ci >= 0) {
        C lr = cl[(size_t)ci * b + row], lc = cl[(size_t)ci * b + col];
        // (the blocked inverse of a block stored whole stands permuted in M)
        const C x = RPL == 0 || twisted ? M[(size_t)col * bp + row] : Di[(size_t)row * bp + col];
        v = v - cmul(cmul(lr, x), lc);
      }
      if (cg >= 0) {
        C lr = cl[(size_t)cg * b + row], lc = cl[(size_t)cg * b + col];
        v = v - cmul(cmul(lr, Dg[tile_index(b, ts, (int)sizeof(C), row, col)]), lc);
      }
      M[(size_t)col * bp + row] = v;
    }
    __syncthreads();
    if constexpr (RPL > 0) gj_block_inverse<RPL>(M, b, bp, f, perm, step_of, status);
    else gauss_jordan_inverse<C>(M, b, bp, f, prow, perm, status);
    C* Dk = fac + g.fac_off + k * bstr;
    if (twisted) {
      // the tiles of the symmetric part, which replaces the inverse in M as well: the next
      // line's Schur complement is then that of the stored block.  n: b padded to whole tiles
      const int n = tile_rows(b, ts.T) * ts.T, pairs = n * (n + 1) / 2;
      auto pair = [&](int idx, int& row, int& col) {
        // pair idx of the triangle, two columns of it folded into one of n + 1 entries
        const int j = idx / (n + 1), i = idx - j * (n + 1);
        row = i > j ? i - 1 : n / 2 + j;
        col = i > j ? j : n / 2 + i;
      };
      auto store = [&](int idx) {
        int row, col;
        pair(idx, row, col);
        C v = czero<C>();
        if (row < b) {
          const C u = inverse(row, col), t = inverse(col, row);
          v = mk((u.x + t.x) / 2, (u.y + t.y) / 2);
        }
        Dk[tile_index(b, ts, (int)sizeof(C), row, col)] = v;
        return v;
      };
      auto put = [&](int idx, C v) {
        int row, col;
        pair(idx, row, col);
        if (row < b) M[(size_t)col * bp + row] = M[(size_t)row * bp + col] = v;
      };
      if constexpr (RPL > 0) {
        // the pairs leave their permuted places in registers before any is written in its own
        constexpr int NM = RPL == 6 ? 168 : 32 * RPL + 5;
        constexpr int NP = (NM * (NM + 1) / 2 + simt_threads(RPL) - 1) / simt_threads(RPL);
        C v[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i)
          if (tid + i * nth < pairs) v[i] = store(tid + i * nth);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < NP; ++i)
          if (tid + i * nth < pairs) put(tid + i * nth, v[i]);
      } else {
        for (int idx = tid; idx < pairs; idx += nth) put(idx, store(idx));
      }
      const int bs = (b + 1) & ~1;
      for (int q = 0; q < ts.NQ; ++q) {
        C* part = Dk + (q ? part_elems(b, ts, 0) : 0);
        const int c0 = part_cpl(b, ts, q);
        for (int p = tid; p < 2 * bs; p += nth) {
          const int up = p >= bs, col = up ? p - bs : p, kk = k - up;   // c_k, then c_{k-1}
          part[c0 + p] = col < b && kk >= 0 ? cl[(size_t)kk * b + col] : czero<C>();
        }
      }
      __syncthreads();
      continue;
    }
    for (int idx = tid; idx < g.bs; idx += nth) {
      int row = idx / bp, col = idx - row * bp;
      C v = czero<C>();
      if (col < b) {
        if (row < b) v = inverse(row, col);
        else if (row == b) v = cl[(size_t)k * b + col];                       // c_k
        else if (k > 0) v = cl[(size_t)(k - 1) * b + col];                   // c_{k-1}
      }
      Dk[idx] = v;
    }
    __syncthreads();
  }
}

// ---- planes wider than shared memory: blocked Gauss-Jordan in global memory -------------
//
// For each plane k (in order) the stored block k of every subdomain is first set to
// D_k = A_kk - diag(l_{k-1}) D_{k-1}^-1 diag(l_{k-1}) (rows 0..b-1, row-major, stride bp,
// zero padding) plus the coupling rows l_k, l_{k-1}, and then inverted in place panel by
// panel (J = the nb columns of a panel, R = the other b - nb; four launches per panel):
//   A_JJ <- A_JJ^-1 (partial pivoting inside the nb x nb block),  A_JR <- A_JJ^-1 A_JR,
//   A_RR <- A_RR - A_RJ A_JR,  A_RJ <- -A_RJ A_JJ^-1,
// after which the block holds D_k^-1.  Pivoting stays inside the diagonal block; on the
// Schur complements of the PML Helmholtz planes this keeps the complex64 inverse within
// ~1e-6 of the exact one (checked against LAPACK on 1024-node planes).
constexpr int kPanel = 32;

template <typename C>
__global__ void k_plane_schur(const SubGeom* __restrict__ subs, const C* __restrict__ lcoef,
                              long long cstride, C* __restrict__ fac, int dim, int k) {
  const SubGeom g = subs[blockIdx.y];
  const int b = g.b, bp = g.bp, L = g.L, Lx = g.Lx;
  if (k >= L) return;
  const C* d = lcoef + g.node_off;
  const C* cx = d + cstride;
  const C* cy = d + 2 * cstride;
  const C* cl = dim == 3 ? d + 3 * cstride : cy;
  C* Dk = fac + g.fac_off + (long long)k * g.bs;
  const C* Dp = fac + g.fac_off + (long long)(k - 1) * g.bs;
  const long long kb = (long long)k * b;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < g.bs;
       idx += (long long)gridDim.x * blockDim.x) {
    const int row = (int)(idx / bp), col = (int)(idx - (long long)row * bp);
    C v = czero<C>();
    if (col < b) {
      if (row < b) {
        if (row == col) v = d[kb + row];
        else if (col == row + 1) v = cx[kb + row];
        else if (row == col + 1) v = cx[kb + col];
        else if (dim == 3 && col == row + Lx) v = cy[kb + row];
        else if (dim == 3 && row == col + Lx) v = cy[kb + col];
        if (k > 0) {
          const C lr = cl[kb - b + row], lc = cl[kb - b + col];
          v = v - cmul(cmul(lr, Dp[(long long)row * bp + col]), lc);
        }
      } else if (row == b) {
        v = cl[kb + col];                                    // l_k
      } else if (k > 0) {
        v = cl[kb - b + col];                                // l_{k-1}
      }
    }
    Dk[idx] = v;
  }
}

// Half rows: between two planes the inverse of plane k in the workspace (subs: offsets without
// a stride per line) is stored as half rows of its symmetric part in fac (dst: the plan's
// geometry) and replaced by the Schur complement of plane k + 1 formed from that part,
//   A_{k+1,k+1} - diag(l_k) D_k^-1 diag(l_k)   (k = -1: the first plane).
// One CTA of 256 threads per pair of mirrored 32 x 32 tiles (tile row blockIdx.y >= tile
// column blockIdx.x), so that both entries of a pair are read before either is written.
template <typename C>
__global__ void __launch_bounds__(256) k_plane_half(const SubGeom* __restrict__ subs,
                                                    const SubGeom* __restrict__ dst,
                                                    const C* __restrict__ lcoef, long long cstride,
                                                    C* __restrict__ W, C* __restrict__ fac, int dim,
                                                    int k) {
  __shared__ C lo[32][33], up[32][33];
  if (blockIdx.x > blockIdx.y) return;
  const SubGeom g = subs[blockIdx.z];
  const int b = g.b, bp = g.bp, L = g.L, Lx = g.Lx;
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  if (k >= L || r0 >= b) return;
  const C* d = lcoef + g.node_off;
  const C* cx = d + cstride;
  const C* cy = d + 2 * cstride;
  const C* cl = dim == 3 ? d + 3 * cstride : cy;
  C* M = W + g.fac_off;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const SubGeom gd = dst[blockIdx.z];
  C* S = fac + gd.fac_off + (long long)k * gd.bs;
  if (k >= 0) {
    for (int i = ty; i < 32; i += 8) {
      const int r = r0 + i, c = c0 + tx;                  // lower tile, and its mirror image
      lo[i][tx] = r < b && c < b ? M[(long long)r * bp + c] : czero<C>();
      const int r2 = c0 + i, c2 = r0 + tx;
      up[i][tx] = r2 < b && c2 < b ? M[(long long)r2 * bp + c2] : czero<C>();
    }
    __syncthreads();
    const int hw = b / 2, hp = half_row(b);
    for (int i = ty; i < 32; i += 8) {
      // entry (r, c) of the lower tile, read along its row, and (r2, c2) of the upper one
      const int r = r0 + i, c = c0 + tx, r2 = c0 + i, c2 = r0 + tx;
      if (r < b && c < b) {
        const C u = lo[i][tx], t = up[tx][i];
        const int j = c >= r ? c - r : c - r + b;
        const bool twice = 2 * j == b && r >= hw;         // (its pair is in row r - b / 2)
        if (j <= hw)
          S[(long long)r * hp + j] = twice ? czero<C>() : mk((u.x + t.x) / 2, (u.y + t.y) / 2);
      }
      if (r2 < b && c2 < b && r0 != c0) {
        const C u = lo[tx][i], t = up[i][tx];
        const int j = c2 - r2;
        if (j <= hw) S[(long long)r2 * hp + j] = mk((u.x + t.x) / 2, (u.y + t.y) / 2);
      }
    }
    if (c0 == 0) {
      // couplings c_k and c_{k-1} of this tile row's nodes
      const int bs = (b + 1) & ~1;
      for (int t = threadIdx.x; t < 64; t += 256) {
        const int p = r0 + (t & 31), kk = k - (t >> 5);
        if (p < b) S[half_cpl(b) + (t >> 5) * bs + p] = kk >= 0 ? cl[(long long)kk * b + p] : czero<C>();
      }
    }
  }
  if (k + 1 >= L) return;
  const long long kb = (long long)(k + 1) * b;
  auto entry = [&](int r, int c, C s) -> C {
    const int lw = min(r, c), df = abs(r - c);
    C v = czero<C>();
    if (df == 0) v = d[kb + r];
    else if (df == 1) v = cx[kb + lw];
    else if (dim == 3 && df == Lx) v = cy[kb + lw];
    if (k >= 0) v = v - cmul(cmul(cl[kb - b + r], s), cl[kb - b + c]);
    return v;
  };
  for (int i = ty; i < 32; i += 8) {
    const int r = r0 + i, c = c0 + tx, r2 = c0 + i, c2 = r0 + tx;
    if (r < b && c < b) {
      C s = czero<C>();
      if (k >= 0) s = mk((lo[i][tx].x + up[tx][i].x) / 2, (lo[i][tx].y + up[tx][i].y) / 2);
      M[(long long)r * bp + c] = entry(r, c, s);
    }
    if (r2 < b && c2 < b && r0 != c0) {
      C s = czero<C>();
      if (k >= 0) s = mk((lo[tx][i].x + up[i][tx].x) / 2, (lo[tx][i].y + up[i][tx].y) / 2);
      M[(long long)r2 * bp + c2] = entry(r2, c2, s);
    }
  }
}

// A_JJ <- A_JJ^-1 (one CTA per subdomain)
template <typename C>
__global__ void k_gj_panel(const SubGeom* __restrict__ subs, C* __restrict__ fac, int k, int j0,
                           int* status) {
  __shared__ C A[kPanel * kPanel];
  __shared__ C f[kPanel];
  __shared__ C prow[kPanel];
  __shared__ int perm[kPanel];
  const SubGeom g = subs[blockIdx.x];
  const int b = g.b, bp = g.bp;
  if (k >= g.L || j0 >= b) return;
  const int nb = min(kPanel, b - j0);
  C* M = fac + g.fac_off + (long long)k * g.bs;
  for (int t = threadIdx.x; t < nb * nb; t += blockDim.x) {
    const int r = t / nb, cc = t - r * nb;
    A[cc * kPanel + r] = M[(long long)(j0 + r) * bp + j0 + cc];   // column-major
  }
  __syncthreads();
  gauss_jordan_inverse<C>(A, nb, kPanel, f, prow, perm, status);
  __syncthreads();
  for (int t = threadIdx.x; t < nb * nb; t += blockDim.x) {
    const int r = t / nb, cc = t - r * nb;
    M[(long long)(j0 + r) * bp + j0 + cc] = A[cc * kPanel + r];
  }
}

// A_JR <- A_JJ^-1 A_JR: one thread per column outside the panel, many CTAs per subdomain
template <typename C>
__global__ void k_gj_rows(const SubGeom* __restrict__ subs, C* __restrict__ fac, int k, int j0) {
  __shared__ C Ainv[kPanel * kPanel];
  const SubGeom g = subs[blockIdx.y];
  const int b = g.b, bp = g.bp;
  if (k >= g.L || j0 >= b) return;
  const int nb = min(kPanel, b - j0);
  C* M = fac + g.fac_off + (long long)k * g.bs;
  for (int t = threadIdx.x; t < nb * nb; t += blockDim.x) {
    const int r = t / nb, cc = t - r * nb;
    Ainv[r * kPanel + cc] = M[(long long)(j0 + r) * bp + j0 + cc];   // row-major
  }
  __syncthreads();
  const int col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= b || (col >= j0 && col < j0 + nb)) return;
  C x[kPanel];
#pragma unroll
  for (int t = 0; t < kPanel; ++t) x[t] = t < nb ? M[(long long)(j0 + t) * bp + col] : czero<C>();
  for (int r = 0; r < nb; ++r) {
    C s = czero<C>();
#pragma unroll
    for (int t = 0; t < kPanel; ++t)
      if (t < nb) s = cfma(Ainv[r * kPanel + t], x[t], s);
    M[(long long)(j0 + r) * bp + col] = s;
  }
}

// A_RR <- A_RR - A_RJ A_JR on T x T tiles (16 x 16 threads, (T/16)^2 outputs each; T = 64
// for complex64, 32 for complex128 to stay within 48 KB of static shared memory)
template <typename C, int T>
__global__ void __launch_bounds__(256) k_gj_update(const SubGeom* __restrict__ subs,
                                                   C* __restrict__ fac, int k, int j0) {
  constexpr int U = T / 16;
  __shared__ C As[T][kPanel + 1];
  __shared__ C Bs[kPanel][T];
  const SubGeom g = subs[blockIdx.z];
  const int b = g.b, bp = g.bp;
  if (k >= g.L || j0 >= b) return;
  const int nb = min(kPanel, b - j0);
  const int i0 = blockIdx.y * T, c0 = blockIdx.x * T;
  if (i0 >= b || c0 >= b) return;
  C* M = fac + g.fac_off + (long long)k * g.bs;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  for (int t = threadIdx.x; t < T * kPanel; t += 256) {
    const int r = t / kPanel, q = t - r * kPanel;
    const int i = i0 + r;
    As[r][q] = (i < b && q < nb) ? M[(long long)i * bp + j0 + q] : czero<C>();
    const int qq = t / T, cc = t - qq * T;
    const int col = c0 + cc;
    Bs[qq][cc] = (col < b && qq < nb) ? M[(long long)(j0 + qq) * bp + col] : czero<C>();
  }
  __syncthreads();
  C acc[U][U];
#pragma unroll
  for (int a = 0; a < U; ++a)
#pragma unroll
    for (int e = 0; e < U; ++e) acc[a][e] = czero<C>();
  for (int q = 0; q < nb; ++q) {
    C av[U], bv[U];
#pragma unroll
    for (int a = 0; a < U; ++a) av[a] = As[ty + 16 * a][q];
#pragma unroll
    for (int e = 0; e < U; ++e) bv[e] = Bs[q][tx + 16 * e];
#pragma unroll
    for (int a = 0; a < U; ++a)
#pragma unroll
      for (int e = 0; e < U; ++e) acc[a][e] = cfma(av[a], bv[e], acc[a][e]);
  }
#pragma unroll
  for (int a = 0; a < U; ++a) {
    const int i = i0 + ty + 16 * a;
    if (i >= b || (i >= j0 && i < j0 + nb)) continue;
#pragma unroll
    for (int e = 0; e < U; ++e) {
      const int col = c0 + tx + 16 * e;
      if (col >= b || (col >= j0 && col < j0 + nb)) continue;
      C* o = M + (long long)i * bp + col;
      *o = *o - acc[a][e];
    }
  }
}

// A_RJ <- -A_RJ A_JJ^-1 (one thread per row outside the panel)
template <typename C>
__global__ void k_gj_cols(const SubGeom* __restrict__ subs, C* __restrict__ fac, int k, int j0) {
  __shared__ C Ainv[kPanel * kPanel];
  const SubGeom g = subs[blockIdx.y];
  const int b = g.b, bp = g.bp;
  if (k >= g.L || j0 >= b) return;
  const int nb = min(kPanel, b - j0);
  C* M = fac + g.fac_off + (long long)k * g.bs;
  for (int t = threadIdx.x; t < nb * nb; t += blockDim.x) {
    const int r = t / nb, cc = t - r * nb;
    Ainv[r * kPanel + cc] = M[(long long)(j0 + r) * bp + j0 + cc];   // row-major
  }
  __syncthreads();
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= b || (row >= j0 && row < j0 + nb)) return;
  C x[kPanel];
#pragma unroll
  for (int t = 0; t < kPanel; ++t) x[t] = t < nb ? M[(long long)row * bp + j0 + t] : czero<C>();
  for (int cc = 0; cc < nb; ++cc) {
    C s = czero<C>();
#pragma unroll
    for (int t = 0; t < kPanel; ++t)
      if (t < nb) s = cfma(x[t], Ainv[t * kPanel + cc], s);
    M[(long long)row * bp + j0 + cc] = mk(-s.x, -s.y);
  }
}

template <typename C>
static cudaError_t launch_factor_wide(Ctx& c) {
  const int nsub = (int)c.subs.size();
  const C* lc = reinterpret_cast<const C*>(c.d_lcoef);
  const long long bs_max = (long long)(c.bmax + 2) * c.bpmax;
  const dim3 gs((unsigned)std::min<long long>(1024, (bs_max + 255) / 256), (unsigned)nsub);
  // complex64: 128-column panels with the products on the tensor cores (three TF32 terms
  // per operand: FP32-level; one for LSWEEP_C64_TF32; three BF16 terms for
  // LSWEEP_C64_BF16X3); complex128: 32-column panels on the CUDA cores in FP64
  constexpr bool tc = std::is_same<C, float2>::value;
  if (tc) {
    cudaError_t e = prepare_gj_panel_tc();
    if (e != cudaSuccess) return e;
  }
  // whole blocks are inverted where they are stored; half rows are made from one whole block
  // per subdomain in a workspace, which every plane passes through
  void* W = nullptr;
  void* fac_at = c.d_fac;
  if (c.half_rows) {
    W = c.mem.get((size_t)nsub * c.bmax * c.bpmax * sizeof(C));
    if (!W) return cudaErrorMemoryAllocation;
    fac_at = W;
  }
  c.f_subs = c.half_rows ? c.d_wsubs : c.d_subs;
  c.f_fac = fac_at;
  C* fac = reinterpret_cast<C*>(c.f_fac);
  const SubGeom* subs = c.f_subs;
  const unsigned t32 = (unsigned)((c.bmax + 31) / 32);
  // the Schur complement of plane k (half rows: plane k - 1 is stored on the way)
  auto next_plane = [&](int k) {
    if (c.half_rows)
      k_plane_half<C><<<dim3(t32, t32, (unsigned)nsub), 256, 0, c.stream>>>(
          subs, c.d_subs, lc, c.node_elems, fac, reinterpret_cast<C*>(c.d_fac), c.dim, k - 1);
    else
      k_plane_schur<C><<<gs, 256, 0, c.stream>>>(subs, lc, c.node_elems, fac, c.dim, k);
  };
  const int panel = tc ? gj_panel_width_tc() : kPanel;
  cudaError_t e = cudaSuccess;
  constexpr int T = 32;
  const int tiles = (c.bmax + T - 1) / T;
  const int npan = (c.bmax + panel - 1) / panel;
  if constexpr (tc) {
    // look-ahead: the products of panel step j update the next panel's column tile first;
    // that panel's inverse (which reads and writes only its diagonal block, final after
    // that update) then runs on a second stream beside the rest of step j's products, and
    // the streams join before step j + 1's products.  Panels and column tiles are both 128
    // columns, so column tile j + 1 is panel j + 1.
    cudaStream_t aux = nullptr;
    cudaEvent_t ev_a = nullptr, ev_b = nullptr;
    e = cudaStreamCreateWithFlags(&aux, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev_a, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev_b, cudaEventDisableTiming);
    const int prec = c.p.precision;
    // the operands of a panel step split once into their terms (left: row tiles, right:
    // column tiles; tile J of both holds the panel inverse P), read by the products
    size_t lb = 0, rb = 0;
    split_tile_bytes(c, prec, lb, rb);
    void* Lbuf = e == cudaSuccess ? c.mem.get(lb * nsub) : nullptr;
    void* Rbuf = e == cudaSuccess ? c.mem.get(rb * nsub) : nullptr;
    if (e == cudaSuccess && (!Lbuf || !Rbuf)) e = cudaErrorMemoryAllocation;
    const int tiles_t = (c.bmax + 127) / 128;
    auto split = [&](int k, int j0, const SplitJobs& jobs) {
      return launch_split_panel(c, k, j0, jobs, Lbuf, Rbuf, (long long)lb, (long long)rb, prec,
                                c.stream);
    };
    auto prod = [&](int k, int j0, int mode, int x0, int ncols, int x_skip) {
      return launch_gj_panel_product_tma(c, k, j0, mode, x0, ncols, x_skip, Lbuf, Rbuf,
                                         (long long)lb, (long long)rb, prec, c.stream);
    };
    for (int k = 0; e == cudaSuccess && k < c.Lmax; ++k) {
      next_plane(k);
      e = launch_gj_panel_inverse(c, k, 0, c.stream);
      for (int j = 0; e == cudaSuccess && j < npan; ++j) {
        const int j0 = j * panel;
        // P on both sides and A_JR before mode 0 updates it
        const SplitJobs pre{3, {0, 1, 1}, {j, j, 0}, {1, 1, tiles_t}, {-1, -1, j}};
        e = split(k, j0, pre);
        if (e == cudaSuccess) e = prod(k, j0, 0, 0, -1, -1);
        // A_JR after mode 0, and A_RJ (unchanged until mode 2 writes it)
        const SplitJobs post{2, {1, 0, 0}, {0, 0, 0}, {tiles_t, tiles_t, 0}, {j, j, -1}};
        if (e == cudaSuccess) e = split(k, j0, post);
        if (e != cudaSuccess) break;
        if (j + 1 < npan) {
          e = prod(k, j0, 1, j + 1, 1, -1);
          if (e == cudaSuccess) e = cudaEventRecord(ev_a, c.stream);
          if (e == cudaSuccess) e = cudaStreamWaitEvent(aux, ev_a, 0);
          if (e == cudaSuccess) e = launch_gj_panel_inverse(c, k, j0 + panel, aux);
          if (e == cudaSuccess) e = cudaEventRecord(ev_b, aux);
          if (e == cudaSuccess) e = prod(k, j0, 1, 0, -1, j + 1);
          if (e == cudaSuccess) e = prod(k, j0, 2, 0, -1, -1);
          if (e == cudaSuccess) e = cudaStreamWaitEvent(c.stream, ev_b, 0);
        } else {
          e = prod(k, j0, 1, 0, -1, -1);
          if (e == cudaSuccess) e = prod(k, j0, 2, 0, -1, -1);
        }
      }
    }
    if (e == cudaSuccess && c.half_rows) next_plane(c.Lmax);   // the last plane's half rows
    if (e == cudaSuccess) e = cudaGetLastError();
    // the buffers are released once the factor's work has completed, on both streams: after an
    // error the last work of aux may not have been joined into c.stream
    cudaStreamSynchronize(c.stream);
    if (aux) cudaStreamSynchronize(aux);
    c.mem.put(Lbuf);
    c.mem.put(Rbuf);
    if (ev_a) cudaEventDestroy(ev_a);
    if (ev_b) cudaEventDestroy(ev_b);
    if (aux) cudaStreamDestroy(aux);
  } else {
    for (int k = 0; e == cudaSuccess && k < c.Lmax; ++k) {
      next_plane(k);
      for (int j0 = 0; j0 < c.bmax; j0 += panel) {
        k_gj_panel<C><<<nsub, 256, 0, c.stream>>>(subs, fac, k, j0, c.d_status);
        k_gj_rows<C><<<dim3((c.bmax + 127) / 128, nsub), 128, 0, c.stream>>>(subs, fac, k, j0);
        k_gj_update<C, T><<<dim3(tiles, tiles, nsub), 256, 0, c.stream>>>(subs, fac, k, j0);
        k_gj_cols<C><<<dim3((c.bmax + 127) / 128, nsub), 128, 0, c.stream>>>(subs, fac, k, j0);
      }
      e = cudaGetLastError();
    }
    if (c.half_rows) {
      if (e == cudaSuccess) next_plane(c.Lmax);
      if (e == cudaSuccess) e = cudaGetLastError();
      cudaStreamSynchronize(c.stream);
    }
  }
  c.mem.put(W);
  c.f_subs = nullptr;
  c.f_fac = nullptr;
  if (e != cudaSuccess) return e;
  c.kernels += (long long)c.Lmax * (1 + 4 * ((c.bmax + panel - 1) / panel));
  return cudaSuccess;
}

// planes whose Gauss-Jordan block fits in shared memory use k_factor_simt
static size_t simt_smem(const Ctx& c, int rpl) {
  const size_t es = c.c64() ? sizeof(float2) : sizeof(double2);
  const size_t work = rpl ? gj_scratch(c.bmax, c.bpmax) * es + 2 * c.bmax * sizeof(int)
                          : 2 * c.bmax * es + c.bmax * sizeof(int);
  return (size_t)c.bpmax * c.bmax * es + work + 16;
}
bool factor_fits_smem(const Ctx& c) { return simt_smem(c, 0) <= 227 * 1024; }

cudaError_t launch_factor(Ctx& c) {
  // (planes of the wide sweep kernel that would fit are inverted faster in panels: complex128 lines of
  // 112 nodes, 462 of them on 2 x 10 subdomains, 1270 -> 860 ms)
  if (c.wide || !factor_fits_smem(c))
    return c.c64() ? launch_factor_wide<float2>(c) : launch_factor_wide<double2>(c);
  const TileStore ts = c.fac_twisted ? tile_store(c) : TileStore{0, 1};
  auto launch = [&](auto kern, auto zero, int rpl) {
    using C = decltype(zero);
    const size_t smem = simt_smem(c, rpl);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)c.subs.size(), simt_threads(rpl), smem, c.stream>>>(
        c.d_subs, (const C*)c.d_lcoef, c.node_elems, (C*)c.d_fac, c.dim, ts, c.d_status);
    return cudaGetLastError();
  };
  if (!c.c64()) return launch(k_factor_simt<double2, 0>, double2(), 0);
  if (simt_smem(c, 6) > 227 * 1024) return launch(k_factor_simt<float2, 0>, float2(), 0);
  if (c.bmax <= 64) return launch(k_factor_simt<float2, 2>, float2(), 2);
  if (c.bmax <= 96) return launch(k_factor_simt<float2, 3>, float2(), 3);
  if (c.bmax <= 128) return launch(k_factor_simt<float2, 4>, float2(), 4);
  return launch(k_factor_simt<float2, 6>, float2(), 6);
}

}  // namespace lsw
