// In-place dense complex inverse by Gauss-Jordan elimination with row pivoting, shared by
// the factorisation kernels (Phase 2 "Factorize", Sec. 3).  Not part of the C ABI.
#pragma once

#include <math.h>

#include "internal.h"

namespace lsw {

__device__ inline float cabs1(float2 a) { return fabsf(a.x) + fabsf(a.y); }
__device__ inline double cabs1(double2 a) { return fabs(a.x) + fabs(a.y); }
__device__ inline bool finite_c(float2 a) { return isfinite(a.x) && isfinite(a.y); }
__device__ inline bool finite_c(double2 a) { return isfinite(a.x) && isfinite(a.y); }

// In-place inverse of the b x b column-major matrix M (leading dimension ld) by
// Gauss-Jordan elimination with row pivoting; the row interchanges are undone on the
// columns of the result at the end (in reverse order).  f and prow are b-entry scratch
// vectors in shared memory: the pivot column before the step and the scaled pivot row.
// Each column step: the pivot search (one warp), the row interchange, then f and prow,
// then the rank-one update, in which every thread keeps one row and a fixed set of
// columns (no index division per element).
template <typename C>
__device__ void gauss_jordan_inverse(C* M, int b, int ld, C* f, C* prow, int* perm,
                                     int* status) {
  using R = decltype(M->x);
  __shared__ int s_piv;
  const int tid = threadIdx.x, nth = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5;
  // update mapping: row ur, columns uc0, uc0 + ncg, ... (threads beyond ncg * b idle);
  // blocks wider than the thread count fall back to a flat element loop
  const bool mapped = nth >= b;
  const int ncg = mapped ? nth / b : 1;
  const int ur = mapped ? tid % b : 0, uc0 = mapped ? tid / b : 0;
  for (int c = 0; c < b; ++c) {
    if (warp == 0) {
      R best = (R)-1;
      int bi = c;
      for (int r = c + lane; r < b; r += 32) {
        R m = cabs1(M[(size_t)c * ld + r]);
        if (m > best) { best = m; bi = r; }
      }
      for (int o = 16; o > 0; o >>= 1) {
        R ob = __shfl_down_sync(0xffffffffu, best, o);
        int oi = __shfl_down_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
      }
      if (lane == 0) {
        s_piv = bi;
        perm[c] = bi;
        if (!(best > (R)0) || !isfinite(best)) atomicOr(status, 1);
      }
    }
    __syncthreads();
    const int p = s_piv;
    if (p != c) {                                        // the same p in every thread
      for (int col = tid; col < b; col += nth) {
        C t = M[(size_t)col * ld + c];
        M[(size_t)col * ld + c] = M[(size_t)col * ld + p];
        M[(size_t)col * ld + p] = t;
      }
      __syncthreads();
    }
    const C pv = M[(size_t)c * ld + c];
    const C inv = (cabs1(pv) > (R)0 && finite_c(pv)) ? cdiv(mk((R)1, (R)0), pv) : czero<C>();
    for (int r = tid; r < b; r += nth) f[r] = M[(size_t)c * ld + r];
    for (int col = tid; col < b; col += nth)
      prow[col] = (col == c) ? inv : cmul(M[(size_t)col * ld + c], inv);
    __syncthreads();
    auto update = [&](int r, int col) {
      if (r == c) {
        M[(size_t)col * ld + c] = prow[col];
      } else if (col == c) {
        const C t = cmul(f[r], inv);
        M[(size_t)c * ld + r] = mk(-t.x, -t.y);
      } else {
        const C t = cmul(f[r], prow[col]);
        M[(size_t)col * ld + r] = M[(size_t)col * ld + r] - t;
      }
    };
    if (mapped) {
      if (uc0 < ncg)
        for (int col = uc0; col < b; col += ncg) update(ur, col);
    } else {
      for (int idx = tid; idx < b * b; idx += nth) {
        const int col = idx / b;
        update(idx - col * b, col);
      }
    }
    __syncthreads();
  }
  for (int c = b - 1; c >= 0; --c) {
    const int p = perm[c];
    if (p != c) {                                        // the same p in every thread
      for (int r = tid; r < b; r += nth) {
        C t = M[(size_t)c * ld + r];
        M[(size_t)c * ld + r] = M[(size_t)p * ld + r];
        M[(size_t)p * ld + r] = t;
      }
      __syncthreads();
    }
  }
}

// ---- blocked form in shared memory (complex64) --------------------------------------------
//
// The same elimination, bit for bit, in panels of 8 columns and without moving rows: the pivot of
// column c is the row p_c that the interchanges would bring there (the largest |re| + |im| among
// the rows not yet used, on ties the first in interchanged order, which pos tracks).  The steps of
// a panel touch its own columns alone and leave the columns F_c before each step and the inverse
// pivots; for a column outside, its 8 pivot entries are then taken through the panel's steps in
// one thread, which gives the scaled pivot rows P_c, and every other entry follows as
//   a <- (..((a - F_0 P_0) - F_1 P_1) ..) - F_7 P_7
// in the order and with the roundings of the single steps.  After the last panel entry (r, c) of
// the inverse stands at row p_r of column step_of[c] (step_of[p_c] = c); whoever reads the result
// applies that permutation.
//
// Warp 0 runs the steps of a panel: lane l holds rows l, l + 32, .. of it in registers, so that a
// step is two warp reductions, one row through shared memory, a reciprocal and one rank-one
// update, with no CTA barrier.  Meanwhile the other warps apply the previous panel to the columns
// outside, in tiles of 4 rows x 4 columns per thread: an entry is read and written once per 8
// steps (row pairs 2 t and 2 (t + G), so that a warp's 16-byte reads are consecutive).  The next
// panel's columns come first, by all warps.  Four CTA barriers per panel instead of three per
// column.  What bounds it: the chain of warp 0's steps (about 600 clocks each).  Measured, clocks of
// one block (column by column -> here): 54 nodes 180 -> 67 k, 92 nodes 537 -> 137 k, 145 nodes
// 1686 -> 400 k; all lines of 16 x 16 subdomains of 92 nodes 31.3 -> 12.1 ms.  Panels of 8: wider
// ones would not leave warp 0 its registers.
constexpr int kGjPanel = 8;

// Entries of scratch for a block of b columns and leading dimension ld: two panels' columns F,
// the pivot rows P, warp 0's rows, the pivot entries of F, the inverse pivots
__host__ __device__ constexpr int gj_scratch(int b, int ld) {
  return kGjPanel * (2 * ld + (b + 3) / 4 * 4 + 2 + kGjPanel + 1);
}

// The row v to shared memory where `on`: predicated, never a branch
__device__ __forceinline__ void store_row_if(bool on, float2* at, const float2 (&v)[kGjPanel]) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %0, 0;\n"
      " @p st.shared.v4.f32 [%1], {%2, %3, %4, %5};\n"
      " @p st.shared.v4.f32 [%1 + 16], {%6, %7, %8, %9};\n"
      " @p st.shared.v4.f32 [%1 + 32], {%10, %11, %12, %13};\n"
      " @p st.shared.v4.f32 [%1 + 48], {%14, %15, %16, %17};\n}\n" ::"r"((int)on),
      "r"((uint32_t)__cvta_generic_to_shared(at)), "f"(v[0].x), "f"(v[0].y), "f"(v[1].x),
      "f"(v[1].y), "f"(v[2].x), "f"(v[2].y), "f"(v[3].x), "f"(v[3].y), "f"(v[4].x), "f"(v[4].y),
      "f"(v[5].x), "f"(v[5].y), "f"(v[6].x), "f"(v[6].y), "f"(v[7].x), "f"(v[7].y)
      : "memory");
}

// A panel's steps j0 .. j0 + nb - 1 on warp 0's registers (y[i][c]: row lane + 32 i); pos: the
// place of each row in interchanged order (used rows: -1).  The columns rotate through the
// registers, the step's own always first.  F: the columns before their steps.
template <int RPL>
__device__ __forceinline__ void gj_panel_steps(float2 (&y)[RPL][kGjPanel], int b, int ld, int j0,
                                               int nb, int (&pos)[RPL], float2* prow, float2* F,
                                               float2* inv_out, int* piv, int* step_of,
                                               int* status) {
  const int lane = threadIdx.x & 31;
  bool singular = false;
#pragma unroll 1
  for (int c = 0; c < nb; ++c) {
    // (an entry that is not finite counts as zero)
    unsigned mag[RPL], best = 0;
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
      const float m = cabs1(y[i][0]);
      mag[i] = m <= 3.4028234e38f ? __float_as_uint(m) : 0u;
      best = max(best, pos[i] >= 0 ? mag[i] : 0u);
    }
    best = __reduce_max_sync(0xffffffffu, best);
    unsigned key = 0xffffffffu;
#pragma unroll
    for (int i = 0; i < RPL; ++i)
      if (pos[i] >= 0 && mag[i] == best) key = min(key, (unsigned)(pos[i] << 8 | (lane + 32 * i)));
    key = __reduce_min_sync(0xffffffffu, key);
    const int p = (int)(key & 255u), pp = (int)(key >> 8), pi = p >> 5;
    const bool mine = lane == (p & 31);
    singular |= best == 0u;                              // zero or non-finite pivot
    float2* row = prow + (c & 1) * kGjPanel;             // (the last one may still be read)
#pragma unroll
    for (int i = 0; i < RPL; ++i) store_row_if(mine && i == pi, row, y[i]);
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
      if (lane + 32 * i < b) F[c * ld + lane + 32 * i] = y[i][0];
      if (pos[i] == j0 + c) pos[i] = pp;
      if (mine && i == pi) pos[i] = -1;
    }
    __syncwarp();
    float2 pr[kGjPanel];
#pragma unroll
    for (int j = 0; j < kGjPanel; j += 2) {
      const float4 v = reinterpret_cast<const float4*>(row)[j / 2];
      pr[j] = make_float2(v.x, v.y);
      pr[j + 1] = make_float2(v.z, v.w);
    }
    const float2 inv = cabs1(pr[0]) > 0.f && finite_c(pr[0]) ? cdiv(make_float2(1.f, 0.f), pr[0])
                                                             : make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 1; j < kGjPanel; ++j) pr[j] = cmul(pr[j], inv);
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
      const float2 f = y[i][0];
      const float2 t = cmul(f, inv);
#pragma unroll
      for (int j = 1; j < kGjPanel; ++j) y[i][j - 1] = y[i][j] - cmul(f, pr[j]);
      y[i][kGjPanel - 1] = make_float2(-t.x, -t.y);
      if (mine && i == pi) {
#pragma unroll
        for (int j = 1; j < kGjPanel; ++j) y[i][j - 1] = pr[j];
        y[i][kGjPanel - 1] = inv;
      }
    }
    if (lane == 0) {
      piv[j0 + c] = p;
      step_of[p] = j0 + c;
      inv_out[c] = inv;
    }
  }
#pragma unroll 1
  for (int c = nb; c < kGjPanel; ++c)                    // the columns back to their places
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
      const float2 t = y[i][0];
#pragma unroll
      for (int j = 1; j < kGjPanel; ++j) y[i][j - 1] = y[i][j];
      y[i][kGjPanel - 1] = t;
    }
  if (singular && lane == 0) atomicOr(status, 1);
}

// The inverse of the b x b column-major block M (leading dimension ld, even), permuted as above,
// by a whole CTA of at least 64 threads; b <= 32 RPL.  scratch: gj_scratch(b, ld) entries, 16-byte
// aligned; piv, step_of: b entries each.  The block is complete after the last barrier.
template <int RPL>
__device__ void gj_block_inverse(float2* M, int b, int ld, float2* scratch, int* piv, int* step_of,
                                 int* status) {
  constexpr int NB = kGjPanel;
  const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31;
  const int ldp = (b + 3) / 4 * 4;
  float2* FF = scratch;                                  // two panels' F[c][row]
  float2* P = FF + 2 * NB * ld;                          // P[c][column]
  float2* prow = P + NB * ldp;
  float2* FP = prow + 2 * NB;                            // F_c at the panel's pivot rows
  float2* inv = FP + NB * NB;
  const int G = (b + 3) / 4, CT = G;                     // row and column tiles
  const int npan = (b + NB - 1) / NB;
  int pos[RPL];
#pragma unroll
  for (int i = 0; i < RPL; ++i) pos[i] = lane + 32 * i < b ? lane + 32 * i : -1;
  auto panel = [&](int j) {                              // warp 0: the steps of panel j
    float2 y[RPL][NB];
    const int j0 = j * NB, nb = min(NB, b - j0);
    float2* F = FF + (j & 1) * NB * ld;
#pragma unroll
    for (int i = 0; i < RPL; ++i)
#pragma unroll
      for (int c = 0; c < NB; ++c)                       // (a copy past the last row or column is
        y[i][c] = M[(j0 + min(c, nb - 1)) * ld + min(lane + 32 * i, b - 1)];   // never stored)
    gj_panel_steps<RPL>(y, b, ld, j0, nb, pos, prow, F, inv, piv, step_of, status);
#pragma unroll
    for (int i = 0; i < RPL; ++i)
#pragma unroll
      for (int c = 0; c < NB; ++c) {
        const int r = lane + 32 * i;
        if (r < b && c < nb) M[(j0 + c) * ld + r] = y[i][c];
      }
    __syncwarp();
    // the pivot rows' entries of F move to FP: the tiles leave those rows alone
    for (int e = lane; e < NB * NB; e += 32) {
      const int c = e / NB, q = e % NB;
      if (c < nb && q < nb) {
        float2* f = F + c * ld + piv[j0 + q];
        FP[e] = *f;
        *f = make_float2(0.f, 0.f);
      }
    }
  };
  for (int j = -1; j < npan; ++j) {
    const int j0 = max(j, 0) * NB, nb = min(NB, b - j0);
    const float2* F = FF + (j & 1) * NB * ld;
    if (j >= 0) {
      // the pivot rows of the columns outside, one thread a column
      for (int col = tid; col < b; col += nth) {
        if (col >= j0 && col < j0 + nb) continue;
        float2 x[NB];
#pragma unroll
        for (int c = 0; c < NB; ++c) x[c] = M[col * ld + piv[j0 + min(c, nb - 1)]];
#pragma unroll
        for (int c = 0; c < NB; ++c) {
          if (c >= nb) break;
          const float2 v = cmul(x[c], inv[c]);
#pragma unroll
          for (int q = 0; q < NB; ++q)
            if (q != c) x[q] = x[q] - cmul(FP[c * NB + q], v);
          x[c] = v;
          P[c * ldp + col] = v;
        }
#pragma unroll
        for (int c = 0; c < NB; ++c)
          if (c < nb) M[col * ld + piv[j0 + c]] = x[c];
      }
      __syncthreads();
      if (j + 1 < npan) {
        // the next panel's columns first (panel j is then a whole one)
        for (int idx = tid; idx < 32 * RPL * NB; idx += nth) {
          const int r = idx % (32 * RPL), col = j0 + NB + idx / (32 * RPL);
          if (r >= b || col >= b) continue;
          float2 a = M[col * ld + r];
#pragma unroll
          for (int c = 0; c < NB; ++c) a = a - cmul(F[c * ld + r], P[c * ldp + col]);
          M[col * ld + r] = a;
        }
        __syncthreads();
      }
    }
    if (tid < 32) {
      if (j + 1 < npan) panel(j + 1);
    } else if (j >= 0) {
      // column tiles but those of panels j and j + 1
      const int skip = min(NB / 2, CT - j * (NB / 4)), tiles = G * (CT - skip);
      for (int t = tid - 32; t < tiles; t += nth - 32) {
        const int u = t / G, ti = t - u * G;
        const int c0 = 4 * (u < j * (NB / 4) ? u : u + skip);
        const int ra = 2 * ti, rb = 2 * (ti + G);        // row pairs ra, ra + 1 and rb, rb + 1
        const bool hi = rb < ld;
        const int rs = hi ? rb : ra;
        float2 a[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2* m = M + min(c0 + q, b - 1) * ld;
          const float4 lo = *reinterpret_cast<const float4*>(m + ra);
          const float4 up = *reinterpret_cast<const float4*>(m + rs);
          a[q][0] = make_float2(lo.x, lo.y);
          a[q][1] = make_float2(lo.z, lo.w);
          a[q][2] = make_float2(up.x, up.y);
          a[q][3] = make_float2(up.z, up.w);
        }
        // the operands of a step are read one step ahead of their use
        float4 w0, w1, p0, p1;
        auto read = [&](int c) {
          w0 = *reinterpret_cast<const float4*>(F + c * ld + ra);
          w1 = *reinterpret_cast<const float4*>(F + c * ld + rs);
          p0 = *reinterpret_cast<const float4*>(P + c * ldp + c0);
          p1 = *reinterpret_cast<const float4*>(P + c * ldp + c0 + 2);
        };
        read(0);
#pragma unroll
        for (int c = 0; c < NB; ++c) {
          if (c >= nb) break;
          const float2 wv[4] = {make_float2(w0.x, w0.y), make_float2(w0.z, w0.w),
                                make_float2(w1.x, w1.y), make_float2(w1.z, w1.w)};
          const float2 p[4] = {make_float2(p0.x, p0.y), make_float2(p0.z, p0.w),
                               make_float2(p1.x, p1.y), make_float2(p1.z, p1.w)};
          if (c + 1 < NB) read(c + 1);
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int i = 0; i < 4; ++i) a[q][i] = a[q][i] - cmul(wv[i], p[q]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float2* m = M + (c0 + q) * ld;
          if (c0 + q < b)
            *reinterpret_cast<float4*>(m + ra) =
                make_float4(a[q][0].x, a[q][0].y, a[q][1].x, a[q][1].y);
          if (c0 + q < b && hi)
            *reinterpret_cast<float4*>(m + rb) =
                make_float4(a[q][2].x, a[q][2].y, a[q][3].x, a[q][3].y);
        }
      }
    }
    __syncthreads();
  }
}

}  // namespace lsw
