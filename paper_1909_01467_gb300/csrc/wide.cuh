// The sweep kernel for planes too wide for a row slab per ring slot; its instantiations are in
// wide_c64.cu, wide_c128.cu and wide_c128_cube.cu, which compile side by side.
#pragma once

#include <type_traits>

#include "wide.h"

namespace lsw {

// ---- planes too wide for a row slab per slot: a cluster streaming chunks of rows ---------
//
// For 3D beams (b = Lx Ly up to ~1000 nodes per plane) one block is several MB and a solve
// streams its factor from HBM twice, so its bytes are what the solve costs.  The block
// inverses are symmetric: of each unordered pair of entries one is stored, row r holding the
// columns r, r + 1, .., r + b / 2 (mod b) (half_row entries; for even b the antipodal pair has a
// place in both rows, zero in the later one).  All rows have the same length, so any range of rows
// is contiguous and as long as any other of its size.  An entry d = D[r][c] is used twice: d v_c
// for row r's sum, and d v_r for row c's.
// A solve runs on a cluster of NS CTAs (up to 16); CTA q owns rows [q RB, (q+1) RB) of every
// block, and its producer warp streams them in chunks of CH rows through a ring of NSLOT
// shared-memory slots (one bulk copy per chunk).  Two warps (complex128, bound by the FP64
// pipe: one) take each row of a chunk, NW groups of 32 columns each, so that four warps per
// scheduler hide one another's waits.  A warp's lanes hold the columns
// that the next 32 rows touch (counted from the row's own position): their vector entries and
// column sums stay in registers, and a row costs one
// shared-memory read per entry (32 consecutive ones, conflict-free) and eight multiply-adds,
// without a branch.  Every 32 rows the window moves on by one group, whose column sums are then
// complete for the warp.  After the step's chunks the warps' column sums are added through
// shared memory and sent to the CTAs that own the columns (st.async completing on the
// receiver's mbarrier); the row owners add them to their row sums in a fixed order, update the
// line vectors, and each CTA sends its rows of the next right-hand vector to the others as one
// bulk copy each.
// Blocks that stay whole (NW = 0, wide_whole_rows) take the same path without column sums.
// Measured against whole rows, one application: 96^3 on 6 x 6 beams (planes of up to 1024 nodes)
// 66.1 -> 49.1 ms, 48^3 on 3 x 3 x 3 boxes 21.9 -> 18.4 ms.  A step of 16 chunks takes 24.6 k
// clocks, 20.1 k of them in the chunks (19.2 k at the measured copy bandwidth with 120 SMs
// streaming) and the rest in the exchange of sums and vectors.

// Row sums of four rows over the warp: lanes 16-31 keep rows 2, 3, lanes with bit 3 the odd
// row, then a 3-level sum; lane 8q returns row q's sum.
template <typename C>
__device__ __forceinline__ C warp_rows4(const C (&r)[4], int lane) {
  const bool h16 = lane & 16, h8 = lane & 8;
  C k0 = h16 ? r[2] : r[0], k1 = h16 ? r[3] : r[1];
  const C o0 = h16 ? r[0] : r[2], o1 = h16 ? r[1] : r[3];
  auto add = [&](C& v, C o, int m) {
    v.x += __shfl_xor_sync(0xffffffffu, o.x, m);
    v.y += __shfl_xor_sync(0xffffffffu, o.y, m);
  };
  add(k0, o0, 16);
  add(k1, o1, 16);
  C v = h8 ? k1 : k0;
  add(v, h8 ? k0 : k1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) add(v, v, o);
  return v;
}

// Entry `off` past shared address `at`, or zero when off > last: a predicated read, never a
// branch (the lanes at the ends of a row's window differ).
template <typename C> __device__ __forceinline__ C entry_or_zero(uint32_t at, int off, int last);
template <>
__device__ __forceinline__ float2 entry_or_zero<float2>(uint32_t at, int off, int last) {
  float2 v;
  asm volatile(
      "{\n .reg .pred p;\n setp.le.s32 p, %3, %4;\n mov.f32 %0, 0f00000000;\n"
      " mov.f32 %1, 0f00000000;\n @p ld.shared.v2.f32 {%0, %1}, [%2];\n}\n"
      : "=&f"(v.x), "=&f"(v.y)
      : "r"(at + (uint32_t)off * 8), "r"(off), "r"(last)
      : "memory");
  return v;
}
template <>
__device__ __forceinline__ double2 entry_or_zero<double2>(uint32_t at, int off, int last) {
  double2 v;
  asm volatile(
      "{\n .reg .pred p;\n setp.le.s32 p, %3, %4;\n mov.f64 %0, 0d0000000000000000;\n"
      " mov.f64 %1, 0d0000000000000000;\n @p ld.shared.v2.f64 {%0, %1}, [%2];\n}\n"
      : "=&d"(v.x), "=&d"(v.y)
      : "r"(at + (uint32_t)off * 16), "r"(off), "r"(last)
      : "memory");
  return v;
}

template <typename C, bool kCube, int NW>
__global__ void __launch_bounds__(8 * wide_halves<C>() * 32 + 32, 1)
k_front_wide(FrontArgs a, Wide wp, int* status) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int NS = wp.NS;
  const int rank = NS > 1 ? (int)cluster_rank() : 0;
  const Task task = a.tasks[a.task_off + blockIdx.x / NS];
  const int sub = task.sub, kind = task.kind;
  const SubGeom g = a.subs[sub];
  constexpr bool kHalf = NW > 0;                        // blocks stored as half rows, or whole
  const int b = g.b, hp = kHalf ? half_row(b) : g.bp, hw = b / 2, L = g.L;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  constexpr int CH = 8, HV = wide_halves<C>();          // rows per chunk, warps per row
  constexpr int ncw = CH * HV, ncons = ncw * 32;         // consumer warps and threads
  // rows per CTA of this box (boundary boxes have smaller planes)
  const int RB = ((b + NS - 1) / NS + 1) / 2 * 2;
  Rows R;
  R.RB = RB;
  R.r0 = min(b, rank * RB);
  R.r1 = min(b, R.r0 + RB);
  const int nr = R.r1 - R.r0;
  const int nch = (nr + CH - 1) / CH;             // chunks per step
  // CTAs that have rows (a small box may leave the last ones without: they take no part in the
  // exchanges, so nothing is sent to them either)
  const int NA = (b + RB - 1) / RB;
  const int ncol = kHalf && nr > 0 ? nr + hw : 0;        // columns this CTA's rows touch
  // shared memory: ring | full[8] | empty[8] | vbar[2] | rbar (+pad) | ysum[HV][RB] | own[RB] |
  // recv[NS][RB] | vk[2][bmax + 2] | part[ncw][PW] | yl[Lmax][RB]
  unsigned char* ring = smem_raw;
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + (size_t)wp.NSLOT * wp.slot_bytes);
  uint64_t* empty = full + 8;
  uint64_t* vbar = empty + 8;
  uint64_t* rbar = vbar + 2;                             // the other CTAs' column sums
  C* ysum = reinterpret_cast<C*>(vbar + 8);
  C* own = ysum + HV * wp.RB;
  C* recv = own + wp.RB;
  C* vk = kHalf ? recv + NS * wp.RB : own;               // (whole rows: no column sums)
  const int vs = (wp.bmax + 3) & ~1;                     // (a rounded copy may pass row b)
  C* part = vk + 2 * vs;
  const int PW = kHalf ? 32 * ((wp.RB + 31) / 32 + NW) : 0;   // columns of a warp's sums
  // line vectors: shared memory, or (when they do not fit beside the ring: smaller clusters
  // of more rows per CTA) one global region per CTA; a thread then owns at most one row and
  // loads its next line entry at the start of each step
  C* yl = wp.lines ? reinterpret_cast<C*>(wp.lines) + (size_t)blockIdx.x * wp.Lmax * wp.RB
                   : part + (size_t)ncw * PW;
  const C* fac = reinterpret_cast<const C*>(a.fac) + g.fac_off;
  const int nsteps = 2 * L - 1;
  // rows of the vector that CTA q sends as one copy: its own, rounded up to even (16 bytes)
  auto sent_rows = [&](int q) {
    const int q0 = min(b, q * RB), qn = min(b, q0 + RB) - q0;
    return (qn + 1) & ~1;
  };
  uint32_t peer_bytes = 0;
  for (int q = 0; q < NS; ++q)
    if (q != rank) peer_bytes += (uint32_t)(sent_rows(q) * (int)sizeof(C));
  // column sums this CTA receives per step: of every other CTA, the columns of its window
  // that fall on this CTA's rows
  auto overlap = [&](int q) {
    const int q0 = min(b, q * RB), qn = min(b, q0 + RB) - q0;
    int n = 0;
    if (qn > 0 && q != rank)
      for (int wrap = 0; wrap <= b; wrap += b)           // columns [q0 + qn, q0 + qn + hw) mod b
        n += max(0, min(R.r1 + wrap, q0 + qn + hw) - max(R.r0 + wrap, q0 + qn));
    return n;
  };
  uint32_t recv_bytes = 0;
  for (int q = 0; kHalf && q < NS; ++q) recv_bytes += (uint32_t)(overlap(q) * (int)sizeof(C));
  bool timed_out = false;
  auto blk = [&](int s) { return s < L ? s : 2 * L - 2 - s; };
  const int total = nsteps * nch;                        // chunk copies of the whole solve
  // chunk c of step s: its rows of the step's block
  auto chunk = [&](int s, int c, uint32_t& bytes) {
    const int rr0 = R.r0 + c * CH, rows = min(CH, R.r1 - rr0);
    bytes = (uint32_t)((size_t)rows * hp * sizeof(C));
    return fac + (size_t)blk(s) * g.bs + (size_t)rr0 * hp;
  };
  auto issue = [&](int s, int c, int slot) {
    uint32_t bytes;
    const C* src = chunk(s, c, bytes);
    mbar_expect_tx(&full[slot], bytes);
    bulk_g2s(ring + (size_t)slot * wp.slot_bytes, src, bytes, &full[slot]);
    // a chunk a few copies ahead is brought into L2 now, so that its copy into the ring
    // does not wait on DRAM latency (the ring holds only a few chunks); the distance is
    // short so that the prefetched rows of all resident CTAs stay in L2
    int ps = s, pc = c + wp.PA;
    while (pc >= nch) {
      pc -= nch;
      ++ps;
    }
    if (wp.PA > 0 && ps < nsteps) {
      uint32_t pb;
      const C* p = chunk(ps, pc, pb);
      bulk_prefetch_l2(p, pb);
    }
  };

  if (tid == 0) {
    for (int i = 0; i < wp.NSLOT; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], (uint32_t)ncw);
    }
    mbar_init(&vbar[0], 1);
    mbar_init(&vbar[1], 1);
    mbar_init(rbar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (NS > 1) {
      mbar_expect_tx(&vbar[0], peer_bytes);
      if (nsteps > 1) mbar_expect_tx(&vbar[1], peer_bytes);
      if (kHalf) mbar_expect_tx(rbar, recv_bytes);
    }
  }
  for (int t = tid; kHalf && t < NS * wp.RB; t += blockDim.x) recv[t] = czero<C>();
  if (NS > 1) cluster_sync_all();
  else __syncthreads();
  const bool producer = tid == ncons;                    // lane 0 of the last warp
  int is = 0, ic = 0;                                    // step and chunk of its next copy
  auto copy_next = [&](int slot) {
    issue(is, ic, slot);
    if (++ic == nch) {
      ic = 0;
      ++is;
    }
  };
  if (producer && nr > 0)
    for (int t = 0; t < min(wp.NSLOT, total); ++t) copy_next(t);
  build_source<C, kCube>(a, g, kind, yl, R);
  __syncthreads();
  // this CTA's rows of vector s to the other CTAs of the cluster (lane q of a warp: CTA q), one
  // bulk copy each that completes on the receiver's barrier; the rows were written and fenced by
  // their owners before a barrier
  auto send = [&](int s, int q) {
    const int n = sent_rows(rank);
    if (q >= NA || q == rank || n == 0) return;
    const uint32_t src = smem_u32(vk + (size_t)(s & 1) * vs + R.r0);
    asm volatile(
        "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(mapa(src, (uint32_t)q)),
        "r"(src), "r"(n * (int)sizeof(C)), "r"(mapa(smem_u32(&vbar[s & 1]), (uint32_t)q))
        : "memory");
  };
  auto fence_rows = [] { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); };
  // v_0 = g_0
  for (int rl = tid; rl < nr; rl += blockDim.x) vk[R.r0 + rl] = yl[rl];
  fence_rows();
  __syncthreads();
  if (w == 0) send(0, lane);

  int s_end = nsteps;
  if (w < ncw && nr > 0) {
    // ---- consumers -------------------------------------------------------------------
    int slot = 0;                                        // ring position of chunk t
    uint32_t phase = 0;
    const int rw = w % CH, first = w / CH * 32 * NW + lane;   // row of a chunk, first column
    const uint32_t ring_at = smem_u32(ring);
    int cfirst = R.r0 + first;                           // that column's position
    while (cfirst >= b) cfirst -= b;
    constexpr int kMyCols = wide_my_cols<C>(NW);
    for (int s = 0; s < nsteps; ++s) {
      const bool fwd = s < L;
      const int k = blk(s);
      const int buf = s & 1;
      // this thread's coupling and (global line vectors) row entry that the step's update
      // reads, in flight during the step's chunks (rows rl = tid < nr; with global line vectors
      // RB <= ncons)
      C line_pre = czero<C>(), cpl_pre = line_pre;
      // couplings l_k, then l_{k-1}: the one towards the line of the next vector
      const C* cpl = fac + (size_t)k * g.bs + b * hp +
                     (fwd && k + 1 < L ? 0 : kHalf ? (b + 1) & ~1 : hp) + R.r0;
      if (tid < nr) {
        cpl_pre = cpl[tid];
        if (wp.lines) {
          if (fwd) {
            if (k + 1 < L) line_pre = yl[(size_t)(k + 1) * RB + tid];
          } else {
            line_pre = yl[(size_t)k * RB + tid];
          }
        }
      }
      if (NS > 1) {
        mbar_wait(&vbar[buf], (uint32_t)((s >> 1) & 1), status, timed_out);  // peers' parts
        consumer_sync(ncons);
        if (tid == 0 && s + 2 < nsteps) mbar_expect_tx(&vbar[buf], peer_bytes);
      }
      const C* v = vk + (size_t)buf * vs;
      // entries of the window's columns, 32 apart (past the last column touched any finite
      // value does: its factor entries read as zero)
      int cnext = cfirst;
      auto entry = [&]() -> C {
        const C x = v[cnext];
        cnext += 32;
        cnext = cnext >= b ? cnext - b : cnext;
        return x;
      };
      C vc[kHalf ? NW : 1], yc[kHalf ? NW : 1];
#pragma unroll
      for (int u = 0; u < NW; ++u) {
        vc[u] = entry();
        yc[u] = czero<C>();
      }
      C* mine = part + (size_t)w * PW + lane;
      for (int g32 = 0; g32 * 32 < nr; ++g32) {          // rows 32 g32 .. + 31: four chunks
        C acc[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          acc[q] = czero<C>();
          const int chn = 4 * g32 + q;
          if (chn >= nch) continue;
          mbar_wait<false>(&full[slot], phase, status, timed_out);
          const int rr = CH * q + rw, rl = 32 * g32 + rr;   // this warp's row of the chunk
          // entry j of the row, for column `first` + 32 u of the window: j = j0 + 32 u, there
          // for 0 <= j <= b / 2 (no entry of a row past the CTA's last one)
          const int j0 = first - rr, last = rl < nr ? hw - j0 : -1;
          const uint32_t row = ring_at + (uint32_t)slot * wp.slot_bytes +
                               (uint32_t)((rw * hp + j0) * (int)sizeof(C));
          if constexpr (!kHalf) {
            // the whole row, columns 32 apart, in four sums
            const C* d = reinterpret_cast<const C*>(ring + (size_t)slot * wp.slot_bytes) + rw * hp;
            C p[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) p[u] = czero<C>();
            if (rl < nr)
              for (int c0 = lane; c0 < b; c0 += 128)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                  if (c0 + 32 * u < b) p[u] = cfma(d[c0 + 32 * u], v[c0 + 32 * u], p[u]);
            acc[q] = (p[0] + p[1]) + (p[2] + p[3]);
          }
          const C vr = v[min(R.r0 + rl, b - 1)];
          // n groups of the window: the last one holds no entry of the first rows of a group of 32,
          // which complex128, bound by these multiply-adds, leaves out (a body of its own: where the
          // group is only predicated off it costs as much)
          auto products = [&](auto groups) {
            constexpr int n = decltype(groups)::value;
            C d[n];
#pragma unroll
            for (int u = 0; u < n; ++u)
              d[u] = entry_or_zero<C>(row, 32 * u, u == 0 && j0 < 0 ? -1 : last);
            C A = czero<C>(), B = czero<C>();
#pragma unroll
            for (int u = 0; u < n; ++u) {
              if (u & 1) B = cfma(d[u], vc[u], B);
              else A = cfma(d[u], vc[u], A);
              // the diagonal entry (u = 0, j = 0) is used once
              yc[u] = cfma(d[u], u == 0 && j0 == 0 ? czero<C>() : vr, yc[u]);
            }
            acc[q] = A + B;
          };
          if constexpr (kHalf) {
            if (HV == 1 && 32 * (NW - 1) > rr + hw) products(std::integral_constant<int, NW - 1>());
            else products(std::integral_constant<int, NW>());
          }
          __syncwarp();
          // (a warp whose wait gave up never releases the slot: the copy may still be landing)
          if (lane == 0 && !timed_out) mbar_arrive(&empty[slot]);
          if (++slot == wp.NSLOT) {
            slot = 0;
            phase ^= 1u;
          }
        }
        const C sum = warp_rows4<C>(acc, lane);          // lane 8 q: the row of chunk q
        const int rl = 32 * g32 + lane + rw;
        if ((lane & 7) == 0 && rl < nr) ysum[w / CH * wp.RB + rl] = sum;
        if constexpr (kHalf) {
          mine[32 * g32] = yc[0];                        // the window moves on
#pragma unroll
          for (int u = 0; u + 1 < NW; ++u) {
            vc[u] = vc[u + 1];
            yc[u] = yc[u + 1];
          }
          vc[NW - 1] = entry();
          yc[NW - 1] = czero<C>();
        }
      }
#pragma unroll
      for (int u = 0; u < NW; ++u) mine[32 * ((nr + 31) / 32 + u)] = yc[u];
      consumer_sync(ncons);                              // row and column sums are complete
      if constexpr (kHalf) {
#pragma unroll
        for (int i = 0; i < kMyCols; ++i) {
          const int cidx = tid + i * ncons;
          if (cidx >= ncol) break;
          C sum = czero<C>();
#pragma unroll
          for (int hv = 0; hv < HV; ++hv) {
            const int rel = cidx - hv * 32 * NW;           // in the windows of these warps
            if (rel < 0 || rel >= 32 * ((nr + 31) / 32 + NW)) continue;
            const C* p = part + (size_t)hv * CH * PW + rel;
            C s0 = czero<C>(), s1 = czero<C>();
#pragma unroll
            for (int ww = 0; ww < CH; ww += 2) {
              s0 = s0 + p[ww * PW];
              s1 = s1 + p[(ww + 1) * PW];
            }
            sum = sum + (s0 + s1);
          }
          if (cidx < nr) {
            own[cidx] = sum;
          } else {
            int c = R.r0 + cidx;
            while (c >= b) c -= b;
            const int q = c / RB;
            C* dst = recv + rank * wp.RB + c - q * RB;
            if (q == rank) *dst = sum;
            else st_async(mapa(smem_u32(dst), (uint32_t)q), sum, mapa(smem_u32(rbar), (uint32_t)q));
          }
        }
        if (NS > 1 && tid < nr) mbar_wait(rbar, (uint32_t)(s & 1), status, timed_out);
        consumer_sync(ncons);
        // the next step's column sums are sent after the vector that this CTA's rows are part
        // of, so the barrier is re-armed before any can arrive
        if (NS > 1 && tid == 0 && s + 1 < nsteps) mbar_expect_tx(rbar, recv_bytes);
      }
      for (int rl = tid; rl < nr; rl += ncons) {
        C sum = ysum[rl];
        if constexpr (kHalf) {
          sum = sum + own[rl];
          if (HV == 2) sum = sum + ysum[wp.RB + rl];
          for (int q = 0; q < NA; ++q) sum = sum + recv[q * wp.RB + rl];
        }
        const C cc = rl == tid ? cpl_pre : cpl[rl];
        C nv = czero<C>(), ynew;
        if (fwd) {
          // y_k = D_k^-1 (g_k - l_k y_{k-1}); next right-hand vector (x_{L-1} = y_{L-1})
          if (k + 1 < L)
            nv = (wp.lines ? line_pre : yl[(size_t)(k + 1) * RB + rl]) - cmul(cc, sum);
          else if (L > 1) nv = cmul(cc, sum);
          ynew = sum;
        } else {
          // x_k = y_k - D_k^-1 (l_{k+1} x_{k+1})
          ynew = (wp.lines ? line_pre : yl[(size_t)k * RB + rl]) - sum;
          if (k > 0) nv = cmul(cc, ynew);
        }
        yl[(size_t)k * RB + rl] = ynew;
        if (s + 1 < nsteps) vk[(size_t)((s + 1) & 1) * vs + R.r0 + rl] = nv;
      }
      if (tid < nr) fence_rows();
      if (bar_red_or(timed_out, ncons)) {                // a wait gave up: leave together
        s_end = s;
        break;
      }
      if (w == 0 && s + 1 < nsteps) send(s + 1, lane);
    }
    if (s_end < nsteps && tid == 0) {
      // give the remote stores of CTAs that have sent them the time to land
      const long long c0 = clock64();
      while (clock64() - c0 < 200000) {}
    }
  } else if (producer && nr > 0) {
    // ---- producer: refill each slot once every consumer warp has released it; before the CTA
    // may exit, wait for every copy it issued ----------------------------------------------
    int issued = min(wp.NSLOT, total), slot = 0;
    uint32_t phase = 0;
    for (int t = wp.NSLOT; t < total; ++t) {
      mbar_wait<false>(&empty[slot], phase, status, timed_out);
      if (timed_out) break;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      copy_next(slot);
      issued = t + 1;
      if (++slot == wp.NSLOT) {
        slot = 0;
        phase ^= 1u;
      }
    }
    drain_ring(full, wp.NSLOT, issued, status);
  }
  __syncthreads();
  if (NS > 1) cluster_sync_all();                      // no remote stores into exited CTAs
  front_epilogue<C, kCube>(a, g, kind, sub, yl, R);
}

// the instantiation of the plan's window, out of those listed
template <typename C, bool kCube, int NW, int... More>
static WideKernel pick_window(const Wide& wp) {
  if constexpr (sizeof...(More) > 0)
    if (wp.NW != NW) return pick_window<C, kCube, More...>(wp);
  return k_front_wide<C, kCube, NW>;
}

}  // namespace lsw
