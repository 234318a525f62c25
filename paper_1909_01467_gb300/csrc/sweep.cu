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
// (distributed shared memory), so a step needs no cluster-wide barrier.  The line vectors (source, y, x) and the line couplings
// of the CTA's rows stay in shared memory for the whole solve.
#include <algorithm>
#include <type_traits>

#include "front.cuh"

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
// ---- planes too wide for a row slab per slot: a cluster streaming chunks of rows ---------
//
// For 3D beams (b = Lx Ly up to ~1000 nodes per plane) one block is several MB and a solve
// streams its factor from HBM twice, so its bytes are what the solve costs.  The block
// inverses are symmetric: of each unordered pair of entries one is stored, row r holding the
// columns r, r + 1, .., r + b / 2 (mod b) (half_row entries; for even b the antipodal pair has a
// place in both rows, zero in the later one).  All rows have the same length, so any range of rows is contiguous and
// as long as any other of its size.  An entry d = D[r][c] is used twice: d v_c for row r's
// sum, and d v_r for row c's.
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
// Measured against whole rows, one application: 96^3 on 6 x 6 beams (planes of up to 1024 nodes)
// 66.1 -> 49.1 ms, 48^3 on 3 x 3 x 3 boxes 21.9 -> 18.4 ms.  A step of 16 chunks takes 24.6 k
// clocks, 20.1 k of them in the chunks (19.2 k at the measured copy bandwidth with 120 SMs
// streaming) and the rest in the exchange of sums and vectors.
struct Wide {
  int NS, RB, CH, NSLOT, Lmax, bmax, NW;
  unsigned slot_bytes;
  int PA;   // chunks between a ring copy and the L2 prefetch it issues (0: none)
  int gl;   // 1: the line vectors in global memory (`lines`, Lmax x RB per CTA)
  void* lines;
};

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

// default of Wide::PA (48^3 on 3 x 3 x 3 boxes: 18.6 ms with 3, 18.4 with 6)
constexpr int kWideL2Ahead = 6;

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

template <typename C>
__host__ __device__ constexpr int wide_halves() { return sizeof(C) == 8 ? 2 : 1; }

template <typename C, bool kCube, int NW>
__global__ void __launch_bounds__(8 * wide_halves<C>() * 32 + 32, 1)
k_front_wide(FrontArgs a, Wide wp, int* status) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int NS = wp.NS;
  const int rank = NS > 1 ? (int)cluster_rank() : 0;
  const Task task = a.tasks[a.task_off + blockIdx.x / NS];
  const int sub = task.sub, kind = task.kind;
  const SubGeom g = a.subs[sub];
  const int b = g.b, hp = half_row(b), hw = b / 2, L = g.L;
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
  const int ncol = nr > 0 ? nr + hw : 0;                 // columns this CTA's rows touch
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
  C* vk = recv + NS * wp.RB;
  const int vs = (wp.bmax + 3) & ~1;                     // (a rounded copy may pass row b)
  C* part = vk + 2 * vs;
  const int PW = 32 * ((wp.RB + 31) / 32 + NW);          // columns of a warp's sums
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
  for (int q = 0; q < NS; ++q) recv_bytes += (uint32_t)(overlap(q) * (int)sizeof(C));
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
      mbar_expect_tx(rbar, recv_bytes);
    }
  }
  for (int t = tid; t < NS * wp.RB; t += blockDim.x) recv[t] = czero<C>();
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
    constexpr int kMyCols = (32 * (NW * HV + 8) + ncons - 1) / ncons;   // columns per thread
    for (int s = 0; s < nsteps; ++s) {
      const bool fwd = s < L;
      const int k = blk(s);
      const int buf = s & 1;
      // this thread's coupling and (global line vectors) row entry that the step's update
      // reads, in flight during the step's chunks (rows rl = tid < nr; with global line vectors
      // RB <= ncons)
      C line_pre = czero<C>(), cpl_pre = line_pre;
      // couplings l_k, then l_{k-1}: the one towards the line of the next vector
      const C* cpl = fac + (size_t)k * g.bs + half_cpl(b) +
                     (fwd && k + 1 < L ? 0 : (b + 1) & ~1) + R.r0;
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
      C vc[NW], yc[NW];
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
          const C vr = v[min(R.r0 + rl, b - 1)];
          C d[NW];
#pragma unroll
          for (int u = 0; u < NW; ++u) d[u] = entry_or_zero<C>(row, 32 * u, u == 0 && j0 < 0 ? -1 : last);
          C A = czero<C>(), B = czero<C>();
#pragma unroll
          for (int u = 0; u < NW; ++u) {
            if (u & 1) B = cfma(d[u], vc[u], B);
            else A = cfma(d[u], vc[u], A);
            // the diagonal entry (u = 0, j = 0) is used once
            yc[u] = cfma(d[u], u == 0 && j0 == 0 ? czero<C>() : vr, yc[u]);
          }
          acc[q] = A + B;
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
        mine[32 * g32] = yc[0];                          // the window moves on
#pragma unroll
        for (int u = 0; u + 1 < NW; ++u) {
          vc[u] = vc[u + 1];
          yc[u] = yc[u + 1];
        }
        vc[NW - 1] = entry();
        yc[NW - 1] = czero<C>();
      }
#pragma unroll
      for (int u = 0; u < NW; ++u) mine[32 * ((nr + 31) / 32 + u)] = yc[u];
      consumer_sync(ncons);                              // row and column sums are complete
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
      for (int rl = tid; rl < nr; rl += ncons) {
        C sum = ysum[rl] + own[rl];
        if (HV == 2) sum = sum + ysum[wp.RB + rl];
        for (int q = 0; q < NA; ++q) sum = sum + recv[q * wp.RB + rl];
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

// Geometry of k_front_wide: NS CTAs per solve (the smallest of 2, 4, 8, 16 whose rows and line
// vectors fit beside a ring of at least 2 chunks of 8 whole rows: the planes that fit so were
// taken before the rows were halved, and the ring has twice the depth for it).  The window of
// columns must fit NW register groups.
template <typename C>
static bool choose_wide(const Ctx& c, Wide& wp, size_t& smem) {
  const size_t limit = 227 * 1024;
  wp.CH = 8;
  wp.PA = c.p.prefetch_steps < 0 ? kWideL2Ahead : c.p.prefetch_steps;
  wp.Lmax = c.Lmax;
  wp.bmax = c.bmax;
  wp.gl = 0;
  wp.lines = nullptr;
  wp.slot_bytes = (unsigned)(((size_t)wp.CH * half_row(c.bmax) * sizeof(C) + 127) / 128 * 128);
  const size_t whole = ((size_t)wp.CH * c.bpmax * sizeof(C) + 127) / 128 * 128;
  constexpr int HV = wide_halves<C>(), ncons = 8 * HV * 32;
  for (int ns : {2, 4, 8, 16}) {
    const int rb = ((c.bmax + ns - 1) / ns + 1) / 2 * 2;
    // groups of 32 columns a row's 32-row window spans, per warp of the row
    const int nw = (c.bmax / 2 / 32 + 2 + HV - 1) / HV;
    wp.NW = HV == 2 ? (nw <= 5 ? 5 : nw <= 9 ? 9 : 14) : nw <= 8 ? 8 : 15;
    // (a thread completes at most kMyCols of the columns)
    if (nw > wp.NW || rb + c.bmax / 2 > 32 * (wp.NW * HV + 8)) continue;
    const size_t lines = (size_t)c.Lmax * rb * sizeof(C);
    const size_t old_vec = 24 * sizeof(uint64_t) + ((size_t)rb + 2 * (size_t)c.bmax) * sizeof(C);
    const size_t vec = 24 * sizeof(uint64_t) +
                       ((size_t)(1 + HV + ns) * rb + 2 * (size_t)(c.bmax + 3) +
                        (size_t)wp.CH * HV * 32 * ((rb + 31) / 32 + wp.NW)) * sizeof(C);
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
template <typename C>
static WideKernel wide_kernel(const Ctx& c, const Wide& wp) {
  if constexpr (wide_halves<C>() == 2) {
    if (c.cube)
      return wp.NW == 5 ? k_front_wide<C, true, 5>
             : wp.NW == 9 ? k_front_wide<C, true, 9> : k_front_wide<C, true, 14>;
    return wp.NW == 5 ? k_front_wide<C, false, 5>
           : wp.NW == 9 ? k_front_wide<C, false, 9> : k_front_wide<C, false, 14>;
  } else {
    if (c.cube) return wp.NW == 8 ? k_front_wide<C, true, 8> : k_front_wide<C, true, 15>;
    return wp.NW == 8 ? k_front_wide<C, false, 8> : k_front_wide<C, false, 15>;
  }
}
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
  auto kern = wide_kernel<C>(c, wp);
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
  if (c.half_rows) return launch_front_wide<C>(c, a, count);
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

// clusters of k_front_wide the device runs at once (0 if it does not apply): a dependency
// level of at most that many solves runs as one wave
template <typename C>
static int wide_capacity(const Ctx& c) {
  Pipe pp;
  int th = 0;
  size_t smem = 0;
  Wide wp;
  if (choose_pipe<C>(c, 1, pp, th, smem) || !choose_wide<C>(c, wp, smem)) return 0;
  int ncl = 0;
  auto kern = wide_kernel<C>(c, wp);
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

// bytes of line-vector scratch the plan's sweep kernels need in global memory (d_lines): the
// wide kernel with global line vectors (NS CTAs per solve, Lmax x RB each), for the largest
// level
size_t lines_bytes(const Ctx& c) {
  size_t need = 0;
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
