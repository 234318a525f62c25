// Geometry of the sweep kernel for planes too wide for a row slab per ring slot (k_front_wide in
// wide.cuh).
#pragma once

#include <algorithm>

#include "front.cuh"

namespace lsw {

struct Wide {
  int NS, RB, CH, NSLOT, Lmax, bmax, NW;
  unsigned slot_bytes;
  int PA;   // chunks between a ring copy and the L2 prefetch it issues (0: none)
  int gl;   // 1: the line vectors in global memory (`lines`, Lmax x RB per CTA)
  void* lines;
};

// default of Wide::PA (48^3 on 3 x 3 x 3 boxes: 18.6 ms with 3, 18.4 with 6)
constexpr int kWideL2Ahead = 6;

template <typename C>
__host__ __device__ constexpr int wide_halves() { return sizeof(C) == 8 ? 2 : 1; }
// columns that a thread completes at most (complex128: every plane that fits has no more than
// 768 rows and half columns per CTA, also with a narrow window)
template <typename C>
__host__ __device__ constexpr int wide_my_cols(int NW) {
  constexpr int HV = wide_halves<C>(), ncons = 8 * HV * 32;
  const int n = (32 * (NW * HV + 8) + ncons - 1) / ncons;
  return HV == 1 && n < 3 ? 3 : n;
}

// Register groups of the window for a plane that spans nw of them per warp, out of the compiled
// ones (more windows mean more code to compile: those of cube boxes start at their smallest planes).
// A group past the last one needed costs its multiply-adds per row and its share of the exchange all
// the same.  Complex128 is bound by the FP64 pipe (a warp's multiply-add takes an SM 16 clocks), so
// there nearly every count has a window of its own.  Measured with windows of 8 and 15 groups only,
// then with these, ms per application: lines of 200 nodes (5 groups; 480^2 on 3 x 3) 78.9 -> 46.0,
// 40^3 on 4 x 4 beams (planes of 484 nodes, 9 groups) 66.4 -> 39.8, 16^3 in one box (484 nodes) 12.7 ->
// 7.5 (whole rows: 8.2).  Complex64, lines of 302 nodes (3 groups instead of 5): 512^2 on 2 x 2
// 11.0 -> 8.5, 516^2 on 1 x 2 9.8 -> 7.7 (whole rows: 11.8 and 9.1).
template <typename C>
inline int wide_window(int nw, bool cube) {
  if (wide_halves<C>() == 1)
    return cube && nw <= 5 ? 5 : nw <= 3 ? 3 : nw <= 11 ? nw : nw <= 13 ? 13 : 15;
  return nw <= 3 && !cube ? 3 : nw <= 5 ? 5 : nw <= 9 ? 9 : 14;
}

// Blocks stored and streamed whole (NW = 0): complex128 lines of up to 128 nodes.  A step is then two
// chunks of rows per CTA (clusters of 8), a half row's 58 to 65 entries take up to three groups of its
// window (24 multiply-adds a lane where the whole row has 16), and a step of so few rows does not pay
// for the exchange of column sums.  ms per application, half -> whole rows: 114 nodes (2 x 10
// subdomains) 85.7 -> 64.5, 128 nodes (2 x 8) 72.7 -> 51.1; from 129 nodes on, with a third chunk, half
// rows are faster: 130 nodes (2 x 7) 63.8 against 73.4, 140 nodes (2 x 8) 101 against 127.
inline bool wide_whole_rows(const Ctx& c) { return !c.c64() && c.dim == 2 && c.bmax <= 128; }

// Geometry of k_front_wide: NS CTAs per solve (the smallest of 2, 4, 8, 16 whose rows and line
// vectors fit beside a ring of at least 2 chunks of 8 whole rows: the planes that fit so were
// taken before the rows were halved, and the ring has twice the depth for it).  The window of
// columns must fit NW register groups.
template <typename C>
inline bool choose_wide(const Ctx& c, Wide& wp, size_t& smem) {
  const size_t limit = 227 * 1024;
  wp.CH = 8;
  wp.PA = c.p.prefetch_steps < 0 ? kWideL2Ahead : c.p.prefetch_steps;
  wp.Lmax = c.Lmax;
  wp.bmax = c.bmax;
  wp.gl = 0;
  wp.lines = nullptr;
  const size_t whole = ((size_t)wp.CH * c.bpmax * sizeof(C) + 127) / 128 * 128;
  const bool half = !wide_whole_rows(c);
  wp.slot_bytes = half ? (unsigned)(((size_t)wp.CH * half_row(c.bmax) * sizeof(C) + 127) / 128 * 128)
                       : (unsigned)whole;
  constexpr int HV = wide_halves<C>(), ncons = 8 * HV * 32;
  for (int ns : {2, 4, 8, 16}) {
    const int rb = ((c.bmax + ns - 1) / ns + 1) / 2 * 2;
    // groups of 32 columns a row's 32-row window spans, per warp of the row
    const int nw = (c.bmax / 2 / 32 + 2 + HV - 1) / HV;
    wp.NW = half ? wide_window<C>(nw, c.cube) : 0;
    // (a thread completes at most wide_my_cols of the columns)
    const int cols = HV == 2 ? 32 * (wp.NW * HV + 8) : wide_my_cols<C>(wp.NW) * ncons;
    if (half && (nw > wp.NW || rb + c.bmax / 2 > cols)) continue;
    const size_t lines = (size_t)c.Lmax * rb * sizeof(C);
    const size_t old_vec = 24 * sizeof(uint64_t) + ((size_t)rb + 2 * (size_t)c.bmax) * sizeof(C);
    const size_t vec = 24 * sizeof(uint64_t) +
                       ((size_t)HV * rb + 2 * (size_t)(c.bmax + 3) +
                        (half ? (size_t)(1 + ns) * rb +
                                    (size_t)wp.CH * HV * 32 * ((rb + 31) / 32 + wp.NW)
                              : 0)) * sizeof(C);
    // the line vectors in shared memory, or in global memory (the handle's d_lines): clusters
    // of 8 CTAs whose rows the consumer threads cover one each (two clusters per GPC instead
    // of one of 16; fewer CTAs per solve would lengthen each solve's dependent chain)
    const bool in_smem = old_vec + lines + 2 * whole <= limit;
    const bool in_global = ns == 8 && rb <= 256 && old_vec + 2 * whole <= limit;
    if (!in_smem && !in_global) continue;
    const bool gl = !in_smem || vec + lines + 2 * (size_t)wp.slot_bytes > limit;
    if (gl && rb > ncons) continue;
    const size_t fixed = vec + (gl ? 0 : lines);
    if (fixed + 2 * (size_t)wp.slot_bytes > limit) continue;
    wp.NS = ns;
    wp.RB = rb;
    wp.gl = gl;
    wp.NSLOT = (int)std::min<size_t>(8, (limit - fixed) / wp.slot_bytes);
    smem = fixed + (size_t)wp.NSLOT * wp.slot_bytes;
    return true;
  }
  return false;
}

using WideKernel = void (*)(FrontArgs, Wide, int*);
template <typename C, bool kCube>
WideKernel wide_kernel(const Wide& wp);

}  // namespace lsw
