// One front of the L-sweeps application (Alg. computeScenario3).  Every task of a front is
// one local solve on one subdomain; all tasks of the front run in the same launch.
//
//   1. source: stage 1 restricts the residual to the owned nodes (Alg. computeLocSol); the
//      sweeps build the equivalent interface source of Eq. DiscPol,
//      g = A_ij(chi_Q w) - chi_Q(A_ij w), from the incoming traces (half-plane Q for the
//      cardinal sweeps, quadrant Q with an L-shaped trace for the diagonal ones);
//   2. block forward / backward substitution with the stored inverse Schur blocks:
//      y_k = D_k^-1 (g_k - l_k y_{k-1}),  x_k = y_k - D_k^-1 (l_{k+1} x_{k+1});
//   3. epilogue: the owned part of the local field is added to the sweep's accumulation
//      lane and the traces on the faces are set or accumulated as the algorithms of App. C
//      state (Alg. extractTraces: the two lines either side of each interior face).
//
// GB300 mapping.  The substitution is a chain of 2L-1 dependent b x b complex block-vector
// products whose blocks are streamed from HBM once per solve, so a solve is split over a
// thread-block cluster of NS CTAs (NS = 1, 2, 4, 8 chosen per front so that the front fills
// the GPU).  CTA q of a cluster owns rows [q RB, (q+1) RB) of every block: the factor
// blocks are stored row-major, so its rows of D_k are one contiguous TMA bulk copy, issued
// by a producer warp into a shared-memory ring of PF slots (mbarrier completion), refilled
// one step after each slot is consumed.  One thread per (row, column chunk) forms partial
// products that are summed per row through shared memory; the row's senders then write
// the next right-hand-side entry to this CTA's vector and send it to the other CTAs of the
// cluster with st.async remote stores that complete on the receiver's mbarrier
// (distributed shared memory), so a step needs no cluster-wide barrier.  The line vectors
// (source, y, x) and the line couplings of the CTA's rows stay in shared memory for the whole
// solve.  The kernels on twisted factors are in twist.cu, the one for planes too wide for a row
// slab per slot in wide.cuh.
#include <algorithm>
#include <type_traits>

#include "front.cuh"
#include "wide.h"

namespace lsw {

constexpr int kMaxCC = 16;   // columns per thread in a block product (at most)
constexpr int kMaxNC = 16;   // column chunks per row (at most)

// kCube: the instantiation cube-CDD plans launch (with the cube tasks' source and trace
// code); beam and 2D plans launch the one without it.
template <typename C, bool kCube>
__global__ void __launch_bounds__(768, 1) k_front(FrontArgs a, Pipe pp, int* status) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int NS = pp.NS;
  const int rank = NS > 1 ? (int)cluster_rank() : 0;
  const Task task = a.tasks[a.task_off + blockIdx.x / NS];
  const int sub = task.sub, kind = task.kind;
  const SubGeom g = a.subs[sub];
  const int b = g.b, bp = g.bp, L = g.L;
  const int tid = threadIdx.x;
  Rows R;
  R.RB = pp.RB;
  R.r0 = min(b, rank * pp.RB);
  R.r1 = min(b, R.r0 + pp.RB);
  const int nr = R.r1 - R.r0;
  // shared memory: D ring | full[8] | vbar[2] (+pad) | vk[2][bmax] | part[NC][RB] |
  // yl[Lmax][RB] | cll[Lmax][RB]
  unsigned char* ring = smem_raw;
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + (size_t)pp.PF * pp.slot_bytes);
  uint64_t* vbar = full + 8;
  C* vk = reinterpret_cast<C*>(vbar + 8);
  C* part = vk + 2 * pp.bmax;
  C* yl = part + (size_t)pp.NC * pp.RB;
  C* cll = yl + (size_t)pp.Lmax * pp.RB;
  const C* lc = reinterpret_cast<const C*>(a.lcoef);
  const C* cl = (a.dim == 3 ? lc + 3 * a.cstride : lc + 2 * a.cstride) + g.node_off;
  const C* fac = reinterpret_cast<const C*>(a.fac) + g.fac_off;
  const int nsteps = 2 * L - 1;                       // forward 0..L-1, backward L-2..0
  const uint32_t peer_bytes = (uint32_t)((b - nr) * sizeof(C));   // the peers' rows of v
  bool timed_out = false;
  auto blk = [&](int s) { return s < L ? s : 2 * L - 2 - s; };
  auto issue = [&](int s) {                           // this CTA's rows of D_blk(s)
    const int slot = s % pp.PF;
    const uint32_t bytes = (uint32_t)((size_t)nr * bp * sizeof(C));
    mbar_expect_tx(&full[slot], bytes);
    bulk_g2s(ring + (size_t)slot * pp.slot_bytes, fac + (size_t)blk(s) * g.bs + (size_t)R.r0 * bp,
             bytes, &full[slot]);
  };

  if (tid == 0) {
    for (int s = 0; s < pp.PF; ++s) mbar_init(&full[s], 1);
    mbar_init(&vbar[0], 1);
    mbar_init(&vbar[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (NS > 1) {
      mbar_expect_tx(&vbar[0], peer_bytes);           // the peers' parts of v_0 and v_1
      if (nsteps > 1) mbar_expect_tx(&vbar[1], peer_bytes);
    }
  }
  if (NS > 1) cluster_sync_all();                      // peers' barriers exist before use
  else __syncthreads();
  // the last warp of the CTA is the producer of the factor stream
  const int producer = (int)blockDim.x - 32;
  if (tid == producer && nr > 0)
    for (int s = 0; s < min(pp.PF, nsteps); ++s) issue(s);
  // couplings of this CTA's rows for every line: cll[k][rl] = coupling of lines k and k+1
  for (size_t t = tid; t < (size_t)(L - 1) * pp.RB; t += blockDim.x) {
    size_t k = t / pp.RB;
    int rl = (int)(t - k * pp.RB);
    if (rl < nr) cll[t] = cl[k * b + R.r0 + rl];
  }
  build_source<C, kCube>(a, g, kind, yl, R);
  __syncthreads();

  // the right-hand vector v_s of step s lives in vk[s & 1]; v_0 = g_0.  Publishing v_{s}
  // entries: thread (rl, q) writes row R.r0 + rl into CTA q of the cluster (q == rank: a
  // local store; otherwise an st.async completing on q's vector barrier).
  const int rl_s = tid % pp.RB, q_s = tid / pp.RB;
  const bool sender = q_s < NS && rl_s < nr;
  auto send = [&](int s_next, C val) {
    const int buf = s_next & 1;
    C* dst = vk + (size_t)buf * pp.bmax + R.r0 + rl_s;
    if (q_s == rank) *dst = val;
    else st_async(mapa(smem_u32(dst), (uint32_t)q_s), val, mapa(smem_u32(&vbar[buf]), (uint32_t)q_s));
  };
  if (sender) send(0, yl[rl_s]);
  __syncthreads();

  // block product roles: row r_w of this CTA's rows, columns [c0, c1) of chunk ch_w
  const int r_w = tid % pp.RB, ch_w = tid / pp.RB;
  const int c0 = ch_w * pp.CC, c1 = min(b, c0 + pp.CC);
  const bool worker = ch_w < pp.NC && r_w < nr && c0 < b;
  int s_end = nsteps;                                  // first step not completed
  for (int s = 0; s < nsteps; ++s) {
    const bool fwd = s < L;
    const int k = blk(s);
    const int buf = s & 1;
    if (NS > 1) {
      mbar_wait(&vbar[buf], (uint32_t)((s >> 1) & 1), status, timed_out);  // peers' parts of v_s
      __syncthreads();
      if (tid == 0 && s + 2 < nsteps) mbar_expect_tx(&vbar[buf], peer_bytes);  // arm v_{s+2}
    }
    if (tid == producer && nr > 0 && s > 0 && s - 1 + pp.PF < nsteps) {
      // the slot of step s-1 was released at its mid-step barrier: refill it while the
      // consumers work on step s
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      issue(s - 1 + pp.PF);
    }
    const C* v = vk + (size_t)buf * pp.bmax;
    if (nr > 0 && worker) {
      const int slot = s % pp.PF;
      mbar_wait<false>(&full[slot], (uint32_t)((s / pp.PF) & 1), status, timed_out);
      const C* row = reinterpret_cast<const C*>(ring + (size_t)slot * pp.slot_bytes) +
                     (size_t)r_w * bp;
      C acc0 = czero<C>(), acc1 = czero<C>();
#pragma unroll
      for (int j = 0; j < kMaxCC; j += 2) {
        if (c0 + j < c1) acc0 = cfma(row[c0 + j], v[c0 + j], acc0);
        if (c0 + j + 1 < c1) acc1 = cfma(row[c0 + j + 1], v[c0 + j + 1], acc1);
      }
      part[(size_t)ch_w * pp.RB + r_w] = acc0 + acc1;
    }
    __syncthreads();
    C yk_new = czero<C>();
    if (sender) {
      const int rl = rl_s;
      C s0 = part[rl], s1 = czero<C>(), s2 = czero<C>(), s3 = czero<C>();
#pragma unroll
      for (int ch = 1; ch < kMaxNC; ch += 4) {
        if (ch < pp.NC && ch * pp.CC < b) s1 = s1 + part[(size_t)ch * pp.RB + rl];
        if (ch + 1 < pp.NC && (ch + 1) * pp.CC < b) s2 = s2 + part[(size_t)(ch + 1) * pp.RB + rl];
        if (ch + 2 < pp.NC && (ch + 2) * pp.CC < b) s3 = s3 + part[(size_t)(ch + 2) * pp.RB + rl];
        if (ch + 3 < pp.NC && (ch + 3) * pp.CC < b) s0 = s0 + part[(size_t)(ch + 3) * pp.RB + rl];
      }
      const C sum = (s0 + s1) + (s2 + s3);
      C nv = czero<C>();
      if (fwd) {
        // y_k = D_k^-1 (g_k - l_k y_{k-1}); next right-hand vector
        if (k + 1 < L) nv = yl[(size_t)(k + 1) * pp.RB + rl] - cmul(cll[(size_t)k * pp.RB + rl], sum);
        else if (L > 1) nv = cmul(cll[(size_t)(L - 2) * pp.RB + rl], sum);   // x_{L-1} = y_{L-1}
        yk_new = sum;
      } else {
        // x_k = y_k - D_k^-1 (l_{k+1} x_{k+1})
        yk_new = yl[(size_t)k * pp.RB + rl] - sum;
        if (k > 0) nv = cmul(cll[(size_t)(k - 1) * pp.RB + rl], yk_new);
      }
      if (s + 1 < nsteps) send(s + 1, nv);
    }
    const bool stop = __syncthreads_or(timed_out);   // a wait gave up: leave together
    // line k of this CTA's rows is overwritten only after every sender has read it
    if (sender && q_s == rank) yl[(size_t)k * pp.RB + rl_s] = yk_new;
    if (stop) {
      s_end = s;
      break;
    }
  }
  __syncthreads();
  if (s_end < nsteps && tid == producer && nr > 0) {
    // drain the bulk copies still in flight into the ring before the CTA can exit: the
    // last step issued into each slot is in (imax - PF, imax]
    bool t2 = false;
    const int imax = min(nsteps - 1, s_end + pp.PF - 1);
    for (int t = max(0, imax - pp.PF + 1); t <= imax; ++t)
      mbar_wait<false>(&full[t % pp.PF], (uint32_t)((t / pp.PF) & 1), status, t2);
  }
  if (NS > 1) cluster_sync_all();                      // no remote stores into exited CTAs

  front_epilogue<C, kCube>(a, g, kind, sub, yl, R);
}


// ---- one CTA per solve: full factor blocks through a TMA ring (complex64, b <= 92) -----
//
// A CTA of W = ceil(b/4) consumer warps and one producer warp solves one task.  The
// producer streams whole stored blocks (the b rows of D_k^-1 and the two coupling rows l_k,
// l_{k-1}: one bulk copy each) into a ring of NSLOT shared-memory slots, NSLOT - 1 steps
// ahead; a slot is released by one arrival per consumer warp on its "empty" barrier.
// Consumer warp w owns rows 4w..4w+3; lane l owns columns l, l + 32, l + 64, so each entry
// of the right-hand vector is read once from shared memory per warp and used for four rows
// (packed FP32 products P += a (vr, vr), Q += a (vi, vi)), the factor is read
// conflict-free (32 consecutive entries per access), and the four row sums are reduced over
// the warp by a 12-shuffle transpose.  The row's owner lane (lane 8q) updates the line
// vectors (shared memory) and publishes the next right-hand entry; one named barrier per
// step orders the double-buffered vector.  No global memory is touched inside the loop.
// kFused: as for k_twist.
template <bool kFused>
__global__ void __launch_bounds__(768, 1) k_front_solo(FrontArgs a_, int Lmax, int bmax, int nslot,
                                                       unsigned slot_bytes, int PD,
                                                       const FrontArgs* __restrict__ table,
                                                       int* status) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  griddep_launch_dependents();                          // the next level may start its setup
  const Task task = a_.tasks[a_.task_off + blockIdx.x];
  const FrontArgs& a = kFused ? table[task.kind >> 8] : a_;
  if (kFused && a.skip) {                               // (waits: as in k_twist)
    griddep_wait();
    return;
  }
  const int sub = task.sub, kind = kFused ? (task.kind & 0xff) : task.kind;
  const SubGeom g = a.subs[sub];
  const int b = g.b, bp = g.bp, L = g.L;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int ncw = (int)(blockDim.x >> 5) - 1;          // consumer warps; the last is the producer
  const int ncons = ncw * 32;
  Rows R;
  R.RB = b;
  R.r0 = 0;
  R.r1 = b;
  // shared memory: ring[nslot][slot_bytes] | full[8] | empty[8] | vb[2][128] | yl[Lmax][bmax]
  unsigned char* ring = smem_raw;
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + (size_t)nslot * slot_bytes);
  uint64_t* empty = full + kSoloMaxSlots;
  float2* vb = reinterpret_cast<float2*>(empty + kSoloMaxSlots);
  float2* yl = vb + 2 * kSoloNV;                        // line vectors [L][b]
  const float2* fac = reinterpret_cast<const float2*>(a.fac) + g.fac_off;
  const int nsteps = 2 * L - 1;
  // forward steps over lines whose right-hand side is zero give exact zeros: skip them
  int slo, shi;
  source_lines(g, kind, a.dim, slo, shi);
  const int f0 = min(slo, L - 1);
  const int nit = nsteps - f0;                         // steps run: s = f0 + it
  const uint32_t blk_bytes = (uint32_t)((size_t)g.bs * sizeof(float2));
  auto blk = [&](int s) { return s < L ? s : 2 * L - 2 - s; };
  auto src = [&](int it) { return fac + (size_t)blk(f0 + it) * g.bs; };
  bool timed_out = false;

  if (tid == 0) {
    for (int i = 0; i < nslot; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], (uint32_t)ncw);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int t = tid; t < 2 * kSoloNV; t += blockDim.x) vb[t] = make_float2(0.f, 0.f);
  __syncthreads();
  if (w == ncw && lane == 0) {
    // first copies, in flight while the source is built
    for (int t = 0; t < min(PD, nit); ++t) bulk_prefetch_l2(src(t), blk_bytes);
    for (int t = 0; t < min(nslot, nit); ++t) {
      mbar_expect_tx(&full[t], blk_bytes);
      bulk_g2s(ring + (size_t)t * slot_bytes, src(t), blk_bytes, &full[t]);
    }
  }
  griddep_wait();                                       // traces of the previous level
  build_source<float2>(a, g, kind, yl, R);
  __syncthreads();

  if (w == ncw) {
    // ---- producer: refill each slot once every consumer warp has released it; before the
    // CTA may exit, wait for every copy it issued -----------------------------------------
    if (lane == 0) {
      int issued = min(nslot, nit);
      for (int t = nslot; t < nit; ++t) {
        const int slot = t % nslot;
        mbar_wait<false>(&empty[slot], (uint32_t)((t / nslot - 1) & 1), status, timed_out, a.spin);
        if (timed_out) break;
        if (PD > 0 && t + PD < nit) bulk_prefetch_l2(src(t + PD), blk_bytes);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(&full[slot], blk_bytes);
        bulk_g2s(ring + (size_t)slot * slot_bytes, src(t), blk_bytes, &full[slot]);
        issued = t + 1;
      }
      drain_ring(full, nslot, issued, status);
    }
  } else {
    // ---- consumers ---------------------------------------------------------------------
    const int r0 = 4 * w;
    const int orow = r0 + (lane >> 3);                  // row of this lane after the reduction
    const bool owner = (lane & 7) == 0 && orow < b;
    if (tid < b) vb[tid] = yl[(size_t)f0 * b + tid];    // v = g of the first nonzero line
    bar_red_or(false, ncons);
    int slot = 0;
    uint32_t phase = 0;
    for (int it = 0; it < nit; ++it) {
      const int s = f0 + it;
      const bool fwd = s < L;
      const int k = blk(s);
      mbar_wait<false>(&full[slot], phase, status, timed_out, a.spin);
      const float2* D = reinterpret_cast<const float2*>(ring + (size_t)slot * slot_bytes);
      const float2* Dw = D + (size_t)r0 * bp + lane;
      const float2* v = vb + (size_t)(it & 1) * kSoloNV;
      // the owner's operands that do not depend on this step's sums, read first
      float2* yk = yl + (size_t)k * b + orow;
      float2 Aval = make_float2(0.f, 0.f), cpl = Aval;
      if (owner) {
        // forward: g_{k+1} and l_k (row b); at the last forward step l_{L-2} (row b + 1),
        // which starts the backward sweep; backward: y_k and l_{k-1} (row b + 1)
        if (fwd) {
          if (k + 1 < L) Aval = yk[b];
          cpl = D[(size_t)(k + 1 < L ? b : b + 1) * bp + orow];
        } else {
          Aval = *yk;
          cpl = D[(size_t)(b + 1) * bp + orow];
        }
      }
      // columns past b have v = 0 and rows past b are discarded, so the reads need no
      // bounds tests: they stay inside the slot (its size covers 4 W rows of bp + 96) and
      // read finite copied data wherever v is nonzero
      float2 vr[3], vi[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float2 x = v[lane + 32 * c];
        vr[c] = make_float2(x.x, x.x);
        vi[c] = make_float2(x.y, x.y);
      }
      float re[4], im[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float2 P = make_float2(0.f, 0.f), Q = P;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float2 d = Dw[q * bp + 32 * c];
          P = __ffma2_rn(d, vr[c], P);
          Q = __ffma2_rn(d, vi[c], Q);
        }
        re[q] = P.x - Q.y;
        im[q] = Q.x + P.y;
      }
      __syncwarp();
      // this warp is done with the slot; a warp whose wait gave up never releases it (the
      // copy may still be landing), so the producer refills no slot with a copy in flight
      if (lane == 0 && !timed_out) mbar_arrive(&empty[slot]);
      if (++slot == nslot) {
        slot = 0;
        phase ^= 1u;
      }
      // transpose-reduce the four rows over the warp: lanes 16-31 keep rows 2, 3 and lanes
      // 0-15 rows 0, 1; then lanes with bit 3 set keep the odd row; then a 3-level sum
      const bool h16 = lane & 16, h8 = lane & 8;
      float kr0 = h16 ? re[2] : re[0], ki0 = h16 ? im[2] : im[0];
      float kr1 = h16 ? re[3] : re[1], ki1 = h16 ? im[3] : im[1];
      const float or0 = h16 ? re[0] : re[2], oi0 = h16 ? im[0] : im[2];
      const float or1 = h16 ? re[1] : re[3], oi1 = h16 ? im[1] : im[3];
      kr0 += __shfl_xor_sync(0xffffffffu, or0, 16);
      ki0 += __shfl_xor_sync(0xffffffffu, oi0, 16);
      kr1 += __shfl_xor_sync(0xffffffffu, or1, 16);
      ki1 += __shfl_xor_sync(0xffffffffu, oi1, 16);
      float kr = h8 ? kr1 : kr0, ki = h8 ? ki1 : ki0;
      const float orr = h8 ? kr0 : kr1, oii = h8 ? ki0 : ki1;
      kr += __shfl_xor_sync(0xffffffffu, orr, 8);
      ki += __shfl_xor_sync(0xffffffffu, oii, 8);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        kr += __shfl_xor_sync(0xffffffffu, kr, o);
        ki += __shfl_xor_sync(0xffffffffu, ki, o);
      }
      if (owner) {
        const float2 sum = make_float2(kr, ki);
        float2 nv = make_float2(0.f, 0.f);
        if (fwd) {
          // y_k = D_k^-1 (g_k - l_k y_{k-1}); next right-hand vector (x_{L-1} = y_{L-1})
          if (k + 1 < L) nv = Aval - cmul(cpl, sum);
          else if (L > 1) nv = cmul(cpl, sum);
          *yk = sum;
        } else {
          // x_k = y_k - D_k^-1 (l_{k+1} x_{k+1})
          const float2 x = Aval - sum;
          if (k > 0) nv = cmul(cpl, x);
          *yk = x;
        }
        vb[(size_t)((it + 1) & 1) * kSoloNV + orow] = nv;
      }
      if (bar_red_or(timed_out, ncons)) break;          // a wait gave up: leave together
    }
  }
  __syncthreads();
  front_epilogue<float2>(a, g, kind, sub, yl, R);
}

// Geometry of the one-CTA-per-solve kernel: ring slots of one stored block, as many as fit
// beside the line vectors (at least 2, at most kSoloMaxSlots).  False when it does not apply.
// `extra` bytes of fixed shared memory are added.
static bool solo_geometry(const Ctx& c, size_t extra, int& threads, int& nslot,
                          unsigned& slot_bytes, size_t& smem) {
  if (!c.c64() || c.bmax > 92 || c.cube) return false;   // cube plans: k_front / k_front_wide
  const int ncw = (c.bmax + 3) / 4;
  threads = (ncw + 1) * 32;
  // a slot holds one stored block (b + 2 rows) and covers the unguarded reads of the
  // consumers: rows up to 4 ncw - 1, columns up to 95
  const size_t rows_read = (size_t)4 * ncw * c.bpmax + 96;
  const size_t slot_elems = std::max((size_t)(c.bmax + 2) * c.bpmax, rows_read);
  slot_bytes = (unsigned)((slot_elems * sizeof(float2) + 127) / 128 * 128);
  const size_t fixed = 2 * kSoloMaxSlots * sizeof(uint64_t) + 2 * kSoloNV * sizeof(float2) +
                       (size_t)c.Lmax * c.bmax * sizeof(float2) + extra;
  const size_t limit = 227 * 1024;
  if (fixed + 2 * (size_t)slot_bytes > limit) return false;
  nslot = (int)std::min<size_t>(kSoloMaxSlots, (limit - fixed) / slot_bytes);
  nslot = std::min(nslot, 4);
  smem = (size_t)nslot * slot_bytes + fixed;
  return threads <= 768;
}
static bool choose_solo(const Ctx& c, int& threads, int& nslot, unsigned& slot_bytes,
                        size_t& smem) {
  return solo_geometry(c, 0, threads, nslot, slot_bytes, smem);
}
// Launch geometry for a front of `tasks` solves: the smallest cluster that fits shared
// memory (ring of at least 2 row slabs beside the line vectors) and gives at least ~128
// CTAs, at most 8 (portable cluster size); NC column chunks (at most 16 columns each) so
// that one thread per row and chunk fills up to 736 threads, plus one producer warp.
template <typename C>
static bool choose_pipe(const Ctx& c, int tasks, Pipe& pp, int& threads, size_t& smem) {
  const size_t limit = 227 * 1024;
  const int b = c.bmax, bp = c.bpmax, L = c.Lmax;
  auto geom = [&](int ns, int& rb, int& nc, int& cc, size_t& slot, size_t& fixed) {
    rb = (b + ns - 1) / ns;
    nc = std::max(1, std::min(kMaxNC, 736 / rb));
    cc = (b + nc - 1) / nc;
    nc = (b + cc - 1) / cc;
    slot = ((size_t)rb * bp * sizeof(C) + 127) / 128 * 128;
    fixed = 16 * sizeof(uint64_t) + (size_t)(2 * b + nc * rb + 2 * (size_t)L * rb) * sizeof(C);
  };
  int ns_fit = 0, rb, nc, cc;
  size_t slot, fixed;
  for (int ns : {1, 2, 4, 8}) {
    geom(ns, rb, nc, cc, slot, fixed);
    if (fixed + 2 * slot <= limit && cc <= kMaxCC) { ns_fit = ns; break; }
  }
  if (!ns_fit) return false;
  int ns = ns_fit;
  while (ns < 8 && (long long)tasks * ns < 128) ns *= 2;
  geom(ns, rb, nc, cc, slot, fixed);
  pp.NS = ns;
  pp.RB = rb;
  pp.NC = nc;
  pp.CC = cc;
  pp.Lmax = L;
  pp.bmax = b;
  pp.slot_bytes = (unsigned)slot;
  pp.PF = (int)std::min<size_t>(6, (limit - fixed) / slot);
  if (pp.PF < 2) return false;
  threads = (std::max(rb * nc, rb * ns) + 31) / 32 * 32 + 32;   // + producer warp
  smem = (size_t)pp.PF * slot + fixed;
  return threads <= 768 && cc <= kMaxCC && nc <= kMaxNC;
}

// ---- launches ---------------------------------------------------------------------------
template <typename C>
static unsigned wide_threads() { return (8 * wide_halves<C>() + 1) * 32; }

template <typename C>
static cudaError_t launch_front_wide(Ctx& c, const FrontArgs& a, int count) {
  Wide wp;
  size_t smem = 0;
  if (!choose_wide<C>(c, wp, smem)) return cudaErrorInvalidConfiguration;
  if (wp.gl) {
    if (!c.d_lines) return cudaErrorInvalidConfiguration;
    wp.lines = c.d_lines;
  }
  const WideKernel kern = c.cube ? wide_kernel<C, true>(wp) : wide_kernel<C, false>(wp);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e == cudaSuccess && wp.NS > 8)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(count * wp.NS));
  cfg.blockDim = dim3(wide_threads<C>());
  cfg.dynamicSmemBytes = smem;
  cfg.stream = c.stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)wp.NS;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a, wp, c.d_status);
}

// solves (clusters) that the device runs at once (0: the kernel does not apply)
template <typename C>
static int wide_clusters(const Ctx& c) {
  Wide wp;
  size_t smem = 0;
  if (!choose_wide<C>(c, wp, smem)) return 0;
  int ncl = 0;
  const WideKernel kern = c.cube ? wide_kernel<C, true>(wp) : wide_kernel<C, false>(wp);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e == cudaSuccess && wp.NS > 8)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(wp.NS * 64));
    cfg.blockDim = dim3(wide_threads<C>());
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)wp.NS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&ncl, kern, &cfg) != cudaSuccess) ncl = 0;
  }
  cudaGetLastError();
  return ncl;
}

template <typename C>
static cudaError_t launch_front_t(Ctx& c, const Task* tasks, int off, int count,
                                  const double2* rin, const double2* g_raw, double2* x_raw) {
  FrontArgs a;
  a.subs = c.d_subs;
  a.tasks = tasks;
  a.task_off = off;
  a.lcoef = c.d_lcoef;
  a.cstride = c.node_elems;
  a.fac = c.d_fac;
  a.lane = c.d_lane;
  a.Next = c.Next;
  a.trace = c.d_trace;
  a.W = c.trace_W;
  a.nsub = (int)c.subs.size();
  a.q = c.q;
  a.r = c.r;
  a.pz = c.pz;
  a.dim = c.dim;
  a.Ne = c.Ne;
  a.rin = rin;
  a.g_raw = g_raw;
  a.x_raw = x_raw;
  a.spin = c.spin();
  a.skip = 0;
  if (c.twisted()) return launch_twist(c, a, count, nullptr, c.stream);
  if constexpr (std::is_same<C, float2>::value) {
    int th, nslot;
    unsigned slot_bytes;
    size_t smem;
    if (c.p.front_kernel == 3) return cudaErrorInvalidConfiguration;   // not factored twisted
    if (c.p.front_kernel != 1 && choose_solo(c, th, nslot, slot_bytes, smem)) {
      const int PD = c.p.prefetch_steps < 0 ? 0 : c.p.prefetch_steps;
      cudaError_t e = cudaFuncSetAttribute(k_front_solo<false>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)count);
      cfg.blockDim = dim3((unsigned)th);
      cfg.dynamicSmemBytes = smem;
      cfg.stream = c.stream;
      cudaLaunchAttribute at[2];
      at[0].id = cudaLaunchAttributeClusterDimension;   // a cluster of one CTA (bulk copies
      at[0].val.clusterDim.x = 1;                         // address shared::cluster)
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      at[1].val.programmaticStreamSerializationAllowed = 1;
      cfg.attrs = at;
      cfg.numAttrs = c.p.pdl ? 2 : 1;
      return cudaLaunchKernelEx(&cfg, k_front_solo<false>, a, c.Lmax, c.bmax, nslot, slot_bytes,
                                PD, (const FrontArgs*)nullptr, c.d_status);
    }
    if (c.p.front_kernel == 2) return cudaErrorInvalidConfiguration;
  }
  Pipe pp;
  int th = 0;
  size_t smem = 0;
  if (c.wide) return launch_front_wide<C>(c, a, count);
  if (!choose_pipe<C>(c, count, pp, th, smem)) return cudaErrorInvalidConfiguration;
  auto kern = c.cube ? k_front<C, true> : k_front<C, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(count * pp.NS));
  cfg.blockDim = dim3((unsigned)th);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = c.stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)pp.NS;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a, pp, c.d_status);
}

// One level of a fused application over several problems (k_twist on twisted factors,
// k_front_solo on plain ones): `count` tasks from tasks[off..], each naming its problem
// (kind >> 8) in `table`; the geometry is c's, which every problem shares.
cudaError_t launch_front_fused(Ctx& c, const Task* tasks, int off, int count,
                               const FrontArgs* table, cudaStream_t stream) {
  FrontArgs a{};
  a.tasks = tasks;
  a.task_off = off;
  if (c.twisted()) return launch_twist(c, a, count, table, stream);
  int th, nslot;
  unsigned slot_bytes;
  size_t smem;
  if (!choose_solo(c, th, nslot, slot_bytes, smem)) return cudaErrorInvalidConfiguration;
  const int PD = c.p.prefetch_steps < 0 ? 0 : c.p.prefetch_steps;
  cudaError_t e = cudaFuncSetAttribute(k_front_solo<true>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)count);
  cfg.blockDim = dim3((unsigned)th);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = c.p.pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, k_front_solo<true>, a, c.Lmax, c.bmax, nslot, slot_bytes, PD,
                            table, c.d_status);
}

// solves of k_front_wide the device runs at once (0 if it does not apply): a dependency level of
// at most that many runs as one wave
template <typename C>
static int wide_capacity(const Ctx& c) {
  Pipe pp;
  int th = 0;
  size_t smem = 0;
  return choose_pipe<C>(c, 1, pp, th, smem) ? 0 : wide_clusters<C>(c);
}

// bytes of line-vector scratch the plan's sweep kernels need in global memory (d_lines): the
// wide kernel (NS CTAs per solve, Lmax x RB each) and complex128 twisted solves (four CTAs, their
// half's lines and rows), for the largest level
size_t lines_bytes(const Ctx& c) {
  // (also when the plan is set up with another kernel that lsweep_autotune may change from)
  size_t need = c.wide ? 0 : twist_lines_bytes(c);
  const size_t tasks = (size_t)std::max(1, c.max_tasks);
  Pipe pp;
  int th = 0;
  size_t smem = 0;
  Wide wp;
  if (c.c64()) {
    if (!choose_pipe<float2>(c, 1, pp, th, smem) && choose_wide<float2>(c, wp, smem) && wp.gl)
      need = std::max(need, tasks * wp.NS * wp.Lmax * wp.RB * sizeof(float2));
  } else {
    if (!choose_pipe<double2>(c, 1, pp, th, smem) && choose_wide<double2>(c, wp, smem) && wp.gl)
      need = std::max(need, tasks * wp.NS * wp.Lmax * wp.RB * sizeof(double2));
  }
  return need;
}

// true when the plan's whole-factor sweeps run on k_front_wide, which streams half rows
bool uses_wide(const Ctx& c) {
  Pipe pp;
  int th, nslot;
  unsigned slot;
  size_t smem;
  if (wants_twisted(c)) return false;
  if (c.c64()) {
    if (c.p.front_kernel != 1 && choose_solo(c, th, nslot, slot, smem)) return false;
    return !choose_pipe<float2>(c, 1, pp, th, smem);
  }
  return !choose_pipe<double2>(c, 1, pp, th, smem);
}

bool wide_whole(const Ctx& c) { return wide_whole_rows(c); }

bool front_pipeline_fits(const Ctx& c) {
  Pipe pp;
  int th, nslot;
  unsigned slot;
  size_t smem;
  Wide wp;
  if (c.p.front_kernel == 2) return choose_solo(c, th, nslot, slot, smem);
  if (c.p.front_kernel == 3) return wants_twisted(c);
  if (c.c64())
    return choose_solo(c, th, nslot, slot, smem) || choose_pipe<float2>(c, 1, pp, th, smem) ||
           choose_wide<float2>(c, wp, smem);
  return choose_pipe<double2>(c, 1, pp, th, smem) || choose_wide<double2>(c, wp, smem);
}

bool wants_twisted(const Ctx& c) {
  if (!factor_fits_smem(c) || !twist_fits(c)) return false;
  if (c.p.front_kernel == 0) return true;
  // front_kernel 3 asked for by name: the plans whose whole line vectors fit shared memory
  int th, nslot;
  unsigned slot;
  size_t smem;
  return c.p.front_kernel == 3 && solo_geometry(c, 1040, th, nslot, slot, smem);
}

int front_form(const Ctx& c) {
  int th, nslot;
  unsigned slot;
  size_t smem;
  if (c.twisted()) return 2;
  if (!c.c64()) return 0;
  return c.p.front_kernel != 1 && c.p.front_kernel != 3 && choose_solo(c, th, nslot, slot, smem)
             ? 1
             : 0;
}

int front_concurrency(const Ctx& c) {
  int th, nslot;
  unsigned slot;
  size_t smem;
  if (wants_twisted(c)) return twist_concurrency(c);
  // planes too wide for a row slab (3D beams): levels of at most the co-resident clusters
  // fill whole waves; other cluster-split plans take no limit
  if (!c.c64()) return c.dim == 3 ? wide_capacity<double2>(c) : 0;
  if (c.p.front_kernel == 1 || !choose_solo(c, th, nslot, slot, smem))
    return c.dim == 3 ? wide_capacity<float2>(c) : 0;
  int dev = 0, sms = 0, nb = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
    cudaGetLastError();
    return 152;
  }
  if (cudaFuncSetAttribute(k_front_solo<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)smem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_front_solo<false>, th, smem) != cudaSuccess)
    nb = 1;
  cudaGetLastError();
  return std::max(1, nb) * sms;
}

cudaError_t launch_front(Ctx& c, int li, const double2* r, const double2* g_raw, double2* x_raw,
                         const Task* raw_task) {
  const Task* tasks = raw_task ? raw_task : c.d_tasks;
  int off = raw_task ? 0 : c.launches[li].off;
  int count = raw_task ? 1 : c.launches[li].count;
  if (c.c64())
    return launch_front_t<float2>(c, tasks, off, count, r, g_raw, x_raw);
  return launch_front_t<double2>(c, tasks, off, count, r, g_raw, x_raw);
}

template <typename C>
__global__ void k_sum_lanes(const C* __restrict__ lane, double2* __restrict__ z, long long N,
                            int accumulate) {
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= N) return;
  double2 s = widen(lane[t]);
  s = s + widen(lane[N + t]);
#pragma unroll
  for (int l = 2; l < kLanes; ++l) s = s + widen(lane[(size_t)l * N + t]);
  z[t] = accumulate ? z[t] + s : s;
}

cudaError_t launch_sum_lanes(Ctx& c, double2* z, bool accumulate) {
  long long nb = (c.Next + 255) / 256;
  const int acc = accumulate ? 1 : 0;
  if (c.c64())
    k_sum_lanes<float2><<<(unsigned)nb, 256, 0, c.stream>>>((const float2*)c.d_lane, z, c.Next, acc);
  else
    k_sum_lanes<double2><<<(unsigned)nb, 256, 0, c.stream>>>((const double2*)c.d_lane, z, c.Next, acc);
  return cudaGetLastError();
}

}  // namespace lsw
