// Sweep-front kernels on twisted factors stored as triangles (2D lines, and the few 3D
// planes that are as small): one dependency level of Alg. computeScenario3 per launch, for
// one right-hand side (k_twist) or for a block of up to eight (k_twist_multi).
//
// Twisted solve.  A factor twisted at m = twist_line(L) holds, for the lines above m, the
// inverses D_k^-1 of the elimination from line 0, for the lines below m the inverses E_k^-1
// of the elimination from line L - 1, and at m the inverse of T_m = A_mm - c_{m-1} D_{m-1}^-1
// c_{m-1} - c_m E_{m+1}^-1 c_m (c_k: diagonal coupling of lines k and k + 1).  The
// substitution is two chains of about L steps that meet once, run side by side by the two
// halves of a cluster:
//   half 0:  y_k = D_k^-1 (g_k - c_{k-1} y_{k-1}),  k = 0 .. m-1;
//   half 1:  z_k = E_k^-1 (g_k - c_k z_{k+1}),      k = L-1 .. m+1;
// each sends its part of line m's right-hand side to the other (st.async on the receiver's
// mbarrier), both form x_m = T_m^-1 (g_m - c_{m-1} y_{m-1} - c_m z_{m+1}) and return outwards:
//   x_k = y_k - D_k^-1 (c_k x_{k+1})  (k < m),   x_k = z_k - E_k^-1 (c_{k-1} x_{k-1})  (k > m).
//
// Storage.  The local operator is complex symmetric, so every inverse is too, and only its
// lower triangle is stored, in T x T tiles (TileStore).  Full levels are bound by the factor
// stream, so half the bytes is what counts there.
//
// Step.  A producer thread streams the stored blocks (one bulk copy each) into a ring.  A
// worker thread holds one off-diagonal tile (I, J) of the block in registers and uses it for
// the rows of I (with the vector's part J) and, transposed, for the rows of J (with part I);
// the owner thread of a row adds its row of the diagonal tile.  What limits a step is the
// shared-memory pipe (it returns 128 bytes a clock, a broadcast costs as much as any read):
// the tile form reads every entry once, and 2 T vector entries and 2 T partial sums per T^2
// entries.  The tiles of step s + 1 are read into the registers column by column as step s
// finishes with them, since they do not depend on the vector.  On the chain of dependent
// steps there are then only the reads of the vector, the products, the partial sums through
// shared memory, the row owner's update and two barriers.
//
// Measured, ms per application, against whole blocks in two- and four-CTA kernels (complex64 up
// to 92 nodes, complex128) or cluster-split ones (wider lines): 1024^2 on 16 x 16 subdomains of
// 92-node lines 4.24 -> 2.71, 404^2 on 4 x 4 of 145-node lines 4.6 -> 1.5, complex128 330^2 on
// 6 x 5 of 81-node lines 7.4 -> 5.4, a block of 8 at 512^2 (60-node lines) 10.4 -> 7.1.
#include <algorithm>
#include <type_traits>

#include "front.cuh"

namespace lsw {

// ---- geometry of a twisted kernel ---------------------------------------------------------
struct Twist {
  TileStore ts;
  int Lh, bs;            // lines per half at most; bmax rounded up to even
  int nslot, PD;         // ring slots; steps between a copy and the L2 prefetch it issues
  int W, gl;             // k_twist_rows: consumer warps; line vectors in global memory
  unsigned slot_bytes;
};

// threads of a CTA at most: a thread per tile and the producer warp
__host__ __device__ constexpr int twist_threads(int T, int GM, int NQ) {
  return (GM * (GM - 1) / 2 / NQ + T * GM / 8 + 31) / 32 * 32 + 32;
}
constexpr int kTwistBars = 22;                 // 8-byte words of barriers: see the layouts below

// Stride (entries) of the partial sums of one tile index: T GM rows, padded so that the
// stores of neighbouring tiles (one stride apart) fall on different banks.
__host__ __device__ constexpr int part_stride(int T, int GM) { return (T * GM + 15) / 16 * 16 + 2; }

// A += (dr vr, di vi), B += (dr vi, di vr): d v = (A.x - A.y, B.x + B.y).  Plain multiply-adds:
// the packed FP32 form runs at half their rate and needs the vector's entries swapped into
// register pairs (a 6 x 6 tile: 287 clocks against 472).
__device__ inline void mac(float2 d, float2 v, float2& A, float2& B) {
  A.x = fmaf(d.x, v.x, A.x);
  A.y = fmaf(d.y, v.y, A.y);
  B.x = fmaf(d.x, v.y, B.x);
  B.y = fmaf(d.y, v.x, B.y);
}
// T consecutive entries between registers and shared memory, 16 bytes at a time
template <int T>
__device__ inline void load_run(const float2* p, float2 (&v)[T]) {
#pragma unroll
  for (int i = 0; i < T; i += 2) {
    const float4 x = *reinterpret_cast<const float4*>(p + i);
    v[i] = make_float2(x.x, x.y);
    v[i + 1] = make_float2(x.z, x.w);
  }
}
__device__ inline void store_pair(float2* p, float2 a, float2 b) {
  *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
}
// Rows i, i + 1 of this thread's tile from a ring slot.
template <int T>
__device__ __forceinline__ void load_rows(float2 (&D)[T * T], const unsigned char* tile,
                                          unsigned unit, int i) {
#pragma unroll
  for (int e = i * T; e < (i + 2) * T; e += 2) {
    const float4 x = *reinterpret_cast<const float4*>(tile + (unsigned)(e / 2) * unit);
    D[e] = make_float2(x.x, x.y);
    D[e + 1] = make_float2(x.z, x.w);
  }
}

// Products of one tile (I, J) with one vector: the rows' partial sums to rowp (from part J of
// the vector), the columns' to colp (from part I).  The tile's last two rows come from the
// current block here (`early`, after the reads of the vector), the others were read during the
// previous step: with kRefill two rows are replaced by the next block's as soon as the last
// product that uses them is done, so that the reads of a tile are spread over the products.
// The next block's barrier is tested first and, where that block has not landed, waited for
// (`wait`) before the first refill.  One basic block otherwise: threads without a tile compute
// on tile 0 and store to a dump.
template <int T, bool kRefill, typename Early, typename Wait>
__device__ __forceinline__ void tile_products(float2 (&D)[T * T], const float2* pI,
                                              const float2* pJ, float2* rowp, float2* colp,
                                              Early early, uint64_t* full, uint32_t phase,
                                              Wait wait, const unsigned char* tile,
                                              unsigned unit) {
  using C = float2;
  C vI[T], vJ[T], cA[T], cB[T];
  load_run<T>(pJ, vJ);
  load_run<T>(pI, vI);
  early();
  const bool landed = !kRefill || mbar_try_wait_cta(full, phase);
#pragma unroll
  for (int j = 0; j < T; ++j) cA[j] = cB[j] = czero<C>();
#pragma unroll
  for (int i = 0; i < T; i += 2) {
    C rA[2], rB[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) rA[u] = rB[u] = czero<C>();
#pragma unroll
    for (int j = 0; j < T; ++j)
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        mac(D[(i + u) * T + j], vJ[j], rA[u], rB[u]);
        mac(D[(i + u) * T + j], vI[i + u], cA[j], cB[j]);
      }
    store_pair(rowp + i, mk(rA[0].x - rA[0].y, rB[0].x + rB[0].y),
               mk(rA[1].x - rA[1].y, rB[1].x + rB[1].y));
    if (kRefill && i + 2 < T) {
      if (i == 0 && !landed) wait();
      load_rows<T>(D, tile, unit, i);
    }
  }
#pragma unroll
  for (int j = 0; j < T; j += 2)
    store_pair(colp + j, mk(cA[j].x - cA[j].y, cB[j].x + cB[j].y),
               mk(cA[j + 1].x - cA[j + 1].y, cB[j + 1].x + cB[j + 1].y));
}

// A step that a wait gave up in, shared by the consumer warps: every thread that gave up
// writes the step before the step's last barrier; after it all threads read the same verdict
// for that step (a later step's entry is larger) and leave together in the next one.
__device__ inline void stop_at(int* stop, int it) { atomicMin(stop, it); }

// Row sum over the tile partials of one row (p: the row's entry of part 0) and the diagonal
// tile's row product `diag`, in a fixed order.  NQ = 2: the partials of CTA q.
template <int T, int GM, int NQ>
__device__ inline float2 row_sum(const float2* p, int G, int I, int q, float2 diag) {
  using C = float2;
  constexpr int SP = part_stride(T, GM);
  C s[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) s[u] = czero<C>();
  const int g0 = NQ == 1 ? 0 : (I + q) & 1;
#pragma unroll
  for (int u = 0; u < GM / NQ; ++u) {
    const int g = g0 + NQ * u;
    if (g < G) s[u & 3] = s[u & 3] + p[g * SP];
  }
  return ((s[0] + s[1]) + (s[2] + s[3])) + diag;
}

__device__ inline void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ inline void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// ---- sources and results of a 2D solve ----------------------------------------------------
// The Eq. DiscPol source of a sweep lives on the two lines across the horizontal side of Q
// (lines ra, ra + 1) and on the two columns across its vertical side (cb, cb + 1): H[2][hs]
// and V[2][vs] (indexed by line) hold it, zero where it is.  hl, vl: the incoming traces.
struct Sides {
  int rc, cc, ra, cb;
  __device__ Sides(const SubGeom& g, int kind) {
    rc = row_cond(kind);
    cc = col_cond(kind);
    ra = rc == 1 ? g.oy0 - 1 : g.oy1 - 1;
    cb = cc == 1 ? g.ox0 - 1 : g.ox1 - 1;
  }
};

// incoming traces of a sweep: across the horizontal (h) and the vertical (v) side of Q
template <typename C>
__device__ inline void incoming(const FrontArgs& a, const SubGeom& g, int kind, const C*& h,
                                const C*& v) {
  const int up = (g.i + 1) * a.r + g.j, dn = (g.i - 1) * a.r + g.j;
  const int lf = g.i * a.r + g.j - 1, rt = g.i * a.r + g.j + 1;
  h = v = nullptr;
  switch (kind) {
    case K_UP: h = trace_ptr<C>(a, T_LOC, dn); break;
    case K_DOWN: h = trace_ptr<C>(a, B_LOC, up); break;
    case K_RIGHT: v = trace_ptr<C>(a, R_LOC, lf); break;
    case K_LEFT: v = trace_ptr<C>(a, L_LOC, rt); break;
    case K_BL2TR: h = trace_ptr<C>(a, T_RIGHT, dn); v = trace_ptr<C>(a, R_UP, lf); break;
    case K_TR2BL: h = trace_ptr<C>(a, B_LEFT, up); v = trace_ptr<C>(a, L_DOWN, rt); break;
    case K_BR2TL: h = trace_ptr<C>(a, T_LEFT, dn); v = trace_ptr<C>(a, L_UP, rt); break;
    case K_TL2BR: h = trace_ptr<C>(a, B_RIGHT, up); v = trace_ptr<C>(a, R_DOWN, lf); break;
    default: break;
  }
}

// The two entries of the source on either side of Q's boundary.
template <typename C>
struct SideSource {
  const C *h, *v, *cx, *cy;
  int rc, cc, ra, cb, qr0, qr1, qc0, qc1, Lx, W;
  __device__ SideSource(const FrontArgs& a, const SubGeom& g, int kind, const Sides& S)
      : rc(S.rc), cc(S.cc), ra(S.ra), cb(S.cb), Lx(g.Lx), W(a.W) {
    incoming<C>(a, g, kind, h, v);
    const C* lc = reinterpret_cast<const C*>(a.lcoef) + g.node_off;
    cx = lc + a.cstride;
    cy = lc + 2 * a.cstride;
    qr0 = rc == 1 ? g.oy0 : 0;
    qr1 = rc == 2 ? g.oy1 - 1 : g.Ly - 1;
    qc0 = cc == 1 ? g.ox0 : 0;
    qc1 = cc == 2 ? g.ox1 - 1 : Lx - 1;
  }
  __device__ void pair(int cond, C c, C w0, C w1, C& lo, C& hi) const {
    const C m0 = cmul(c, w0), m1 = cmul(c, w1);
    if (cond == 1) { hi = mk(-m0.x, -m0.y); lo = m1; }
    else { lo = mk(-m1.x, -m1.y); hi = m0; }
  }
  // lines ra and ra + 1 at position x
  __device__ void across_row(int x, C& lo, C& hi) const {
    lo = hi = czero<C>();
    if (x >= qc0 && x <= qc1) pair(rc, cy[ra * Lx + x], h[x], h[W + x], lo, hi);
  }
  // columns cb and cb + 1 of line y; on the horizontal lines the L-shaped trace takes the
  // horizontal neighbour's values
  __device__ void across_column(int y, C& lo, C& hi) const {
    lo = hi = czero<C>();
    if (y < qr0 || y > qr1) return;
    C w0 = v[y], w1 = v[W + y];
    if (rc && (y == ra || y == ra + 1)) {
      const C* hl = h + (y - ra) * W;
      if (cb >= qc0 && cb <= qc1) w0 = hl[cb];
      if (cb + 1 >= qc0 && cb + 1 <= qc1) w1 = hl[cb + 1];
    }
    pair(cc, cx[y * Lx + cb], w0, w1, lo, hi);
  }
};

// H and V of a sweep for the positions [0, b) and the lines [ka, kb); called by all threads
template <typename C>
__device__ void side_sources(const FrontArgs& a, const SubGeom& g, int kind, const Sides& S,
                             int ka, int kb, C* H, int hs, C* V, int vs, int tid, int nth) {
  const SideSource<C> src(a, g, kind, S);
  const int nh = S.rc ? g.Lx : 0, nv = S.cc ? kb - ka : 0;
  for (int t = tid; t < nh + nv; t += nth) {
    C lo, hi;
    if (t < nh) {
      src.across_row(t, lo, hi);
      H[t] = lo;
      H[hs + t] = hi;
    } else {
      src.across_column(ka + t - nh, lo, hi);
      V[t - nh] = lo;
      V[vs + t - nh] = hi;
    }
  }
}

// source entry of line k, position p
template <typename C>
__device__ inline C side_entry(const Sides& S, const C* H, int hs, const C* V, int vs, int ka,
                               int k, int p) {
  C v = czero<C>();
  if (S.rc && (unsigned)(k - S.ra) < 2u) v = H[(k - S.ra) * hs + p];
  if (S.cc && (unsigned)(p - S.cb) < 2u) v = v + V[(p - S.cb) * vs + k - ka];
  return v;
}
// right-hand side of the local solve of stage 1: the input on the owned nodes
template <typename C>
__device__ inline C local_entry(const FrontArgs& a, const SubGeom& g, int k, int p) {
  if (k < g.oy0 || k >= g.oy1 || p < g.ox0 || p >= g.ox1) return czero<C>();
  return to<C>(a.rin[(size_t)(g.gy0 + k) * a.Ne + g.gx0 + p]);
}

// One outgoing face: trace array, and whether the values are added to it
struct Face { char side; int arr; bool add; };
__device__ inline int outgoing(const FrontArgs& a, const SubGeom& g, int kind, Face* f) {
  const bool T = g.i < a.q - 1, B = g.i > 0, Rr = g.j < a.r - 1, Lf = g.j > 0;
  int n = 0;
  auto put = [&](bool has, char s, int arr, bool add) {
    if (has) f[n++] = Face{s, arr, add};
  };
  switch (kind) {
    case K_LOCAL:
      put(T, 'T', T_LOC, false);
      put(B, 'B', B_LOC, false);
      put(Lf, 'L', L_LOC, false);
      put(Rr, 'R', R_LOC, false);
      break;
    case K_UP: put(T, 'T', T_LOC, true); put(Rr, 'R', R_UP, false); put(Lf, 'L', L_UP, false); break;
    case K_DOWN: put(B, 'B', B_LOC, true); put(Rr, 'R', R_DOWN, false); put(Lf, 'L', L_DOWN, false); break;
    case K_RIGHT: put(Rr, 'R', R_LOC, true); put(B, 'B', B_RIGHT, false); put(T, 'T', T_RIGHT, false); break;
    case K_LEFT: put(Lf, 'L', L_LOC, true); put(B, 'B', B_LEFT, false); put(T, 'T', T_LEFT, false); break;
    case K_BL2TR: put(Rr, 'R', R_UP, true); put(T, 'T', T_RIGHT, true); break;
    case K_TR2BL: put(Lf, 'L', L_DOWN, true); put(B, 'B', B_LEFT, true); break;
    case K_BR2TL: put(Lf, 'L', L_UP, true); put(T, 'T', T_LEFT, true); break;
    case K_TL2BR: put(Rr, 'R', R_DOWN, true); put(B, 'B', B_RIGHT, true); break;
    default: break;
  }
  return n;
}

// Epilogue of a 2D solve for K right-hand sides: lines [k0, k1) and rows [r0, r1) of the
// solution (entry (k, p) of right-hand side c at yl[k * ls + c * cs + p]).  The owned part
// goes to the sweep's accumulation lane, the face values to the outgoing traces.  A thread
// loads the old values of kBatch entries together: few threads share the work, so what counts
// is how often each waits for memory.
template <typename C, int kBatch, typename LaneOf, typename ArgsOf>
__device__ void twist_epilogue(const FrontArgs& a, const SubGeom& g, int kind, int sub, const C* yl,
                               int ls, int cs, int K, int k0, int k1, int r0, int r1,
                               LaneOf lane_ptr, ArgsOf trace_base) {
  const int tid = threadIdx.x, nth = blockDim.x;
  const int ya = max(k0, g.oy0), yb = min(k1, g.oy1), xa = max(r0, g.ox0), xb = min(r1, g.ox1);
  const int ow = xb - xa, per = ow > 0 && yb > ya ? (yb - ya) * ow : 0, n0 = per * K;
  const size_t off = kind == K_LOCAL ? 0 : (size_t)lane_of(kind) * a.Next;
  Face f[4];
  const int nf = outgoing(a, g, kind, f);
  const int nl = max(0, k1 - k0), nr = max(0, r1 - r0);
  // entries of the faces: horizontal ones first the two lines over [r0, r1), vertical ones the
  // two columns over [k0, k1)
  int end[4];
  int n = n0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (q < nf) n += 2 * K * (f[q].side == 'T' || f[q].side == 'B' ? nr : nl);
    end[q] = n;
  }
  for (int t0 = tid; t0 < n; t0 += kBatch * nth) {
    C v[kBatch], old[kBatch];
    C* dst[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int t = t0 + u * nth;
      dst[u] = nullptr;
      old[u] = czero<C>();
      if (t < n0) {
        const int c = K == 1 ? 0 : t / per, rem = K == 1 ? t : t - c * per;
        const int row = rem / ow, y = ya + row, x = xa + rem - row * ow;
        v[u] = yl[y * ls + c * cs + x];
        dst[u] = lane_ptr(c) + off + (size_t)(g.gy0 + y) * a.Ne + g.gx0 + x;
        if (kind != K_LOCAL) old[u] = *dst[u];
      } else if (t < n) {
        const int q = (t >= end[0]) + (t >= end[1]) + (t >= end[2]);
        const Face fc = q == 0 ? f[0] : q == 1 ? f[1] : q == 2 ? f[2] : f[3];
        const int e = t - (q == 0 ? n0 : q == 1 ? end[0] : q == 2 ? end[1] : end[2]);
        const bool horiz = fc.side == 'T' || fc.side == 'B';
        const int at = fc.side == 'T' ? g.oy1 - 1 : fc.side == 'B' ? g.oy0 - 1
                       : fc.side == 'R' ? g.ox1 - 1 : g.ox0 - 1;   // lower of the two lines
        const int s0 = horiz ? r0 : k0, len = horiz ? nr : nl;
        const int ln = e / len, s = s0 + e - ln * len, c = ln >> 1, tt = ln & 1;
        const int y = horiz ? at + tt : s, x = horiz ? s : at + tt;
        if (y >= k0 && y < k1 && x >= r0 && x < r1) {
          v[u] = yl[y * ls + c * cs + x];
          dst[u] = trace_base(c) + ((size_t)fc.arr * a.nsub + sub) * 2 * a.W + (size_t)tt * a.W + s;
          if (fc.add) old[u] = *dst[u];
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      if (!dst[u]) continue;
      const int t = t0 + u * nth;
      *dst[u] = old[u] + v[u];
      if (kind == K_LOCAL && t < n0)
#pragma unroll
        for (int l = 1; l < kLanes; ++l) dst[u][(size_t)l * a.Next] = czero<C>();
    }
  }
}

// Right-hand side of a 2D solve into the line vectors of the lines [ka, kb), yl[(k - ka) b + p],
// which are zero; every entry is written by one thread.
template <typename C>
__device__ void dense_source(const FrontArgs& a, const SubGeom& g, int kind, C* yl, int ka, int kb) {
  const int tid = threadIdx.x, nth = blockDim.x, b = g.b;
  if (kind == K_RAW) {
    for (int t = tid; t < (kb - ka) * b; t += nth) yl[t] = to<C>(a.g_raw[(size_t)ka * b + t]);
    return;
  }
  if (kind == K_LOCAL) {
    constexpr int kBatch = 8;
    const int ya = max(ka, g.oy0), yb = min(kb, g.oy1), ow = g.ox1 - g.ox0, n = (yb - ya) * ow;
    for (int t0 = tid; t0 < n; t0 += kBatch * nth) {
      double2 v[kBatch];
      int at[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int t = t0 + u * nth, row = t / ow, y = ya + row, x = g.ox0 + t - row * ow;
        at[u] = t < n ? (y - ka) * b + x : -1;
        if (t < n) v[u] = a.rin[(size_t)(g.gy0 + y) * a.Ne + g.gx0 + x];
      }
#pragma unroll
      for (int u = 0; u < kBatch; ++u)
        if (at[u] >= 0) yl[at[u]] = to<C>(v[u]);
    }
    return;
  }
  const Sides S(g, kind);
  const SideSource<C> src(a, g, kind, S);
  const int nh = S.rc ? b : 0, nv = S.cc ? kb - ka : 0;
  for (int t = tid; t < nh + nv; t += nth) {
    C lo, hi;
    if (t < nh) {
      // the lines ra, ra + 1 at position t, with the vertical side's share of them
      src.across_row(t, lo, hi);
      C w0, w1;
      if (S.cc && (unsigned)(t - S.cb) < 2u) {
        src.across_column(S.ra, w0, w1);
        lo = lo + (t == S.cb ? w0 : w1);
        src.across_column(S.ra + 1, w0, w1);
        hi = hi + (t == S.cb ? w0 : w1);
      }
      if (S.ra >= ka && S.ra < kb) yl[(S.ra - ka) * b + t] = lo;
      if (S.ra + 1 >= ka && S.ra + 1 < kb) yl[(S.ra + 1 - ka) * b + t] = hi;
    } else {
      const int y = ka + t - nh;
      if (S.rc && (unsigned)(y - S.ra) < 2u) continue;
      src.across_column(y, lo, hi);
      yl[(y - ka) * b + S.cb] = lo;
      yl[(y - ka) * b + S.cb + 1] = hi;
    }
  }
}

// ---- one right-hand side ---------------------------------------------------------------
// NQ CTAs per half: CTA (h, q) has rank h NQ + q.  With NQ = 2 each CTA of a half forms its
// tiles' partial sums of every row, sends them to its mate (st.async, two barriers by step
// parity, re-armed one step ahead) and adds the mate's, so that both hold all rows of the line
// vectors and one exchange per step is enough; CTA q writes half of the rows out.  At the last
// step before the middle line CTA (h, q) sends its half's part of the right-hand side to CTA
// (1 - h, q).
// kFused: one launch over the solves of several problems (fused applications): the task's
// kind carries its problem in bits 8.., whose arguments come from `table`; a problem marked
// skip is not applied (its CTAs wait for the previous level and exit).
template <int T, int GM, int NQ, bool kFused>
__global__ void __launch_bounds__(twist_threads(T, GM, NQ), 1)
k_twist(FrontArgs a_, Twist tg, const FrontArgs* __restrict__ table, int* status) {
  static_assert(NQ == 1 || NQ == 2, "one mate per CTA at most");
  using C = float2;
  constexpr int VN = T * GM, SP = part_stride(T, GM);
  extern __shared__ __align__(128) unsigned char smem_raw[];
  griddep_launch_dependents();                          // the next level may start its setup
  const Task task = a_.tasks[a_.task_off + blockIdx.x / (2 * NQ)];
  const FrontArgs& a = kFused ? table[task.kind >> 8] : a_;
  if (kFused && a.skip) {
    // (a level is complete only with the levels before it: a launch of nothing but such CTAs must
    // not finish while an earlier one still runs, as the next launch waits for this one alone)
    griddep_wait();
    return;
  }
  const int sub = task.sub, kind = kFused ? (task.kind & 0xff) : task.kind;
  const SubGeom g = a.subs[sub];
  const int b = g.b, L = g.L, G = tile_rows(b, T);
  const int rank = (int)cluster_rank();
  const int h = rank / NQ, q = rank % NQ;              // half (0: from line 0), part of the tiles
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int ncw = (int)(blockDim.x >> 5) - 1;          // consumer warps; the last is the producer
  const int ncons = ncw * 32;
  const int m = twist_line(L);
  const int nf = h ? L - 1 - m : m;                    // steps before the middle line
  // forward steps over lines whose right-hand side is zero give exact zeros, and backward
  // steps past the last line whose values anyone reads are not needed: skip both
  int slo, shi, nlo, nhi;
  source_lines(g, kind, a.dim, slo, shi);
  needed_lines(g, kind, a.dim, nlo, nhi);
  const int f0 = h ? min(L - 1 - shi, nf) : min(slo, nf);
  const int nsteps = nf + 1 + (h ? nhi - m : m - nlo);
  const int nit = nsteps - f0;                         // steps this CTA runs: s = f0 + it
  const int ka = h ? m : 0, kb = h ? L : m + 1;        // lines of this half (m in both)
  // shared memory: ring[nslot][slot_bytes] | full[8] | empty[8] | pbar[2] | xbar[2] | flags[4]
  // (32-bit) | vb[2][VN] | part[GM][SP] | dump[8] | pm[2][bs] (NQ 2) | xb[bs] | yl[Lh][b]
  unsigned char* ring = smem_raw;
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + (size_t)tg.nslot * tg.slot_bytes);
  uint64_t* empty = full + kSoloMaxSlots;
  uint64_t* pbar = empty + kSoloMaxSlots;              // the mate's partial sums
  uint64_t* xbar = pbar + 2;                           // the other half's part of line m
  // flags[0]: this CTA sent its part of line m (all rows or none); flags[1]: partial sums sent
  // to the mate (steps); flags[2]: the step a wait gave up in (stop_at)
  volatile uint32_t* flags = reinterpret_cast<volatile uint32_t*>(xbar + 2);
  int* stop = reinterpret_cast<int*>(xbar + 3);
  const int bs = tg.bs;
  C* vb = reinterpret_cast<C*>(full + kTwistBars);
  C* part = vb + 2 * VN;
  C* dump = part + GM * SP;
  C* pm = dump + 8;
  C* xb = pm + (NQ == 2 ? 2 * bs : 0);
  C* yl = xb + bs;
  auto line = [&](int k) { return yl + (k - ka) * b; };
  const TileStore ts{T, NQ};
  const C* fac = reinterpret_cast<const C*>(a.fac) + g.fac_off + (q ? part_elems(b, ts, 0) : 0);
  const int stride = block_elems(b, ts);
  const uint32_t blk_bytes = (uint32_t)(part_elems(b, ts, q) * (int)sizeof(C));
  auto blk = [&](int s) {
    if (s < nf) return h ? L - 1 - s : s;
    return h ? m + (s - nf) : m - (s - nf);
  };
  auto src = [&](int it) { return fac + (size_t)blk(f0 + it) * stride; };
  auto issue = [&](int it, int slot) {
    mbar_expect_tx(&full[slot], blk_bytes);
    bulk_g2s(ring + (size_t)slot * tg.slot_bytes, src(it), blk_bytes, &full[slot]);
  };
  bool timed_out = false;

  if (tid == 0) {
    for (int i = 0; i < tg.nslot; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], (uint32_t)ncw);
    }
    mbar_init(&pbar[0], 1);
    mbar_init(&pbar[1], 1);
    mbar_init(&xbar[0], 1);
    flags[0] = flags[1] = 0;
    *stop = 0x7fffffff;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(&xbar[0], (uint32_t)(b * sizeof(C)));   // one entry per row
    if (NQ == 2) {                                      // one partial sum per row, steps 0 and 1
      mbar_expect_tx(&pbar[0], (uint32_t)(b * sizeof(C)));
      if (nit > 1) mbar_expect_tx(&pbar[1], (uint32_t)(b * sizeof(C)));
    }
  }
  {
    // vectors, partial sums and line vectors start as zeros
    const int nz = (int)(yl - vb) + (kb - ka) * b;
    for (int t = tid; t < (nz + 1) / 2; t += blockDim.x)
      reinterpret_cast<float4*>(vb)[t] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncthreads();
  cluster_sync_all();                                  // every CTA's barriers are armed
  if (w == ncw && lane == 0) {
    for (int t = 0; t < min(tg.PD, nit); ++t) bulk_prefetch_l2(src(t), blk_bytes);
    for (int t = 0; t < min(tg.nslot, nit); ++t) issue(t, t);
  }
  griddep_wait();                                       // traces of the previous level
  if (a.dim == 2) {
    dense_source<C>(a, g, kind, yl, ka, kb);
  } else {
    Rows R;
    R.RB = b;
    R.r0 = 0;
    R.r1 = b;
    R.ls = b;
    R.k0 = ka;
    R.k1 = kb;
    build_source<C>(a, g, kind, yl - (long long)ka * b, R);
  }
  __syncthreads();

  int parmed = min(nit, 2) - 1, pok = -1;               // (tid 0) last step armed / received
  if (w == ncw) {
    // ---- producer: refill each slot once every consumer warp has released it; before the
    // CTA may exit, wait for every copy it issued -----------------------------------------
    if (lane == 0) {
      int issued = min(tg.nslot, nit);
      for (int t = tg.nslot; t < nit; ++t) {
        const int slot = t % tg.nslot;
        mbar_wait<false>(&empty[slot], (uint32_t)((t / tg.nslot - 1) & 1), status, timed_out, a.spin);
        if (timed_out) break;
        if (tg.PD > 0 && t + tg.PD < nit) bulk_prefetch_l2(src(t + tg.PD), blk_bytes);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        issue(t, slot);
        issued = t + 1;
      }
      drain_ring(full, tg.nslot, issued, status);
    }
  } else {
    // ---- workers (thread o: tile o of this CTA) and owners (thread p: row p) ---------------
    int I, J;
    const bool worker = worker_tile<NQ>(tid, G, q, I, J);
    const unsigned unit = (unsigned)tile_count(G, NQ, q) * 16;
    const unsigned tile_off = worker ? (unsigned)tid * 16 : 0;
    C* rowp = worker ? part + J * SP + I * T : dump;
    C* colp = worker ? part + I * SP + J * T : dump;
    const bool owner = tid < b;                         // owns row tid of the vectors
    const bool owner_warp = w * 32 < b;
    const int OI = owner ? tid / T : 0, oi = owner ? tid - OI * T : 0;
    const bool odiag = owner && (NQ == 1 || (OI & 1) == q);   // its diagonal tile is here
    // offsets (entries) of the couplings and of this row's entries of the diagonal tile
    const int cpl_off = part_cpl(b, ts, q), nd = diag_count(G, NQ, q);
    int doff[T];
#pragma unroll
    for (int j = 0; j < T; ++j)
      doff[j] = odiag ? tile_count(G, NQ, q) * T * T + (NQ == 1 ? OI : OI >> 1) +
                            (oi >= j ? oi * (oi + 1) / 2 + j : j * (j + 1) / 2 + oi) * nd
                      : 0;
    const uint32_t peer = (uint32_t)((h ^ 1) * NQ + q), mate = (uint32_t)(h * NQ + (q ^ 1));
    auto send_middle = [&](C v) {                       // this row's part of line m
      st_async(mapa(smem_u32(xb + tid), peer), v, mapa(smem_u32(xbar), peer));
      flags[0] = 1;
    };
    int slot = 0, nslot = 0;                            // slots of this block and the next
    uint32_t phase = 0;                                 // of slot nslot
    C D[T * T];
    auto ready = [&]() { mbar_wait<false>(&full[nslot], phase, status, timed_out, a.spin); };
    const int lrow = owner ? tid : 0;
    if (owner) {
      C v = line(blk(f0))[tid];                         // the first right-hand side
      if (f0 >= nf) {
        // the middle line comes first: this half adds nothing to its right-hand side (no
        // lines before it, or zero right-hand sides on all of them)
        send_middle(czero<C>());
        mbar_wait<true>(xbar, 0, status, timed_out, a.spin);
        v = v + xb[tid];
      }
      vb[tid] = v;
    }
    ready();
#pragma unroll
    for (int i = 0; i + 2 < T; i += 2) load_rows<T>(D, ring + tile_off, unit, i);
    if (timed_out) stop_at(stop, -1);
    consumer_sync(ncons);
    int halt = *(volatile int*)stop;
    for (int it = 0; it < nit; ++it) {
      const int s = f0 + it;
      const int k = blk(s);
      const bool more = it + 1 < nit;
      const C* v = vb + (it & 1) * VN;
      const unsigned char* tile = ring + (size_t)slot * tg.slot_bytes + tile_off;
      // the owner's operands.  Forward: the source of the next line inwards and the coupling
      // towards it; middle and backward: y_k (backward only) and the coupling towards the next
      // line outwards (a block's couplings: c_k, then c_{k-1}); its row of the diagonal tile
      C Ac = czero<C>(), cc = Ac, dr[T], vO[T];
      auto early = [&]() {
        load_rows<T>(D, tile, unit, T - 2);
        if (owner_warp) {
          const C* sl = reinterpret_cast<const C*>(ring + (size_t)slot * tg.slot_bytes);
          load_run<T>(v + OI * T, vO);
#pragma unroll
          for (int j = 0; j < T; ++j) dr[j] = sl[doff[j]];
          Ac = line(s < nf ? (h ? k - 1 : k + 1) : k)[lrow];
          cc = sl[cpl_off + ((s < nf) == (h != 0) ? (b + 1) & ~1 : 0) + lrow];
        }
      };
      if (more) {
        if (++nslot == tg.nslot) {
          nslot = 0;
          phase ^= 1u;
        }
        tile_products<T, true>(D, v + I * T, v + J * T, rowp, colp, early, &full[nslot], phase,
                               ready, ring + (size_t)nslot * tg.slot_bytes + tile_off, unit);
      } else {
        tile_products<T, false>(D, v + I * T, v + J * T, rowp, colp, early, full, 0, ready,
                                nullptr, 0);
      }
      if (halt < it) break;                             // a wait gave up: leave together
      consumer_sync(ncons);                             // the partial sums are there
      // this warp is done with the slot; a warp whose wait gave up never releases it (the copy
      // may still be landing), so the producer refills no slot with a copy in flight
      if (lane == 0 && !timed_out) mbar_arrive(&empty[slot]);
      if (owner) {
        C dA = czero<C>(), dB = dA;
#pragma unroll
        for (int j = 0; j < T; ++j) mac(dr[j], vO[j], dA, dB);
        C sum = row_sum<T, GM, NQ>(part + tid, G, OI, q,
                                   odiag ? mk(dA.x - dA.y, dB.x + dB.y) : czero<C>());
        if (NQ == 2) {
          C* in = pm + (it & 1) * bs + tid;
          st_async(mapa(smem_u32(in), mate), sum, mapa(smem_u32(&pbar[it & 1]), mate));
          if (tid == 0) flags[1] = (uint32_t)(it + 1);
          mbar_wait<true>(&pbar[it & 1], (uint32_t)((it >> 1) & 1), status, timed_out, a.spin);
          // re-arm for step it + 2: the mate sends it only after it received this CTA's step
          // it + 1, which is sent after this step's last barrier, and only if no wait of this
          // step gave up
          if (tid == 0 && !timed_out) {
            pok = it;
            if (it + 2 < nit) {
              mbar_expect_tx(&pbar[it & 1], (uint32_t)(b * sizeof(C)));
              parmed = it + 2;
            }
          }
          sum = sum + *in;
        }
        C nv = czero<C>();
        C* yk = line(k) + tid;
        if (s < nf) {
          *yk = sum;                                    // y_k (z_k)
          const C t = cmul(cc, sum);
          nv = Ac - t;
          if (s + 1 == nf) {
            // next is the middle line: exchange the halves' parts of its right-hand side
            // (every owner of this CTA sends in this step, timed out or not: all or none)
            send_middle(mk(-t.x, -t.y));
            mbar_wait<true>(xbar, 0, status, timed_out, a.spin);
            nv = nv + xb[tid];
          }
        } else {
          const C x = s == nf ? sum : Ac - sum;         // x_m, or x_k = y_k - D_k^-1 (c x)
          *yk = x;
          nv = cmul(cc, x);
        }
        vb[((it + 1) & 1) * VN + tid] = nv;
      }
      if (timed_out) stop_at(stop, it);
      consumer_sync(ncons);                             // the next vector is there
      halt = *(volatile int*)stop;
      slot = nslot;
    }
  }
  const bool gave_up = __syncthreads_or(timed_out) != 0;
  cluster_sync_all();                                   // every CTA has left its loop
  if (gave_up && tid == 0) {
    // A CTA that did not give up has seen everything sent to it land.  After a timeout wait
    // (bounded) for what may still be in flight to this CTA before it exits: the mate's partial
    // sums of the steps after the last one received, up to the last one it sent (never beyond
    // the last one armed here), and the other half's part of line m if it was sent.
    if (NQ == 2) {
      const uint32_t mate = (uint32_t)(h * NQ + (q ^ 1));
      const int sent = (int)ld_cluster_u32(mapa(smem_u32((const void*)&flags[1]), mate));
      for (int t = pok + 1; t < sent && t <= parmed; ++t)
        mbar_drain<true>(&pbar[t & 1], (uint32_t)((t >> 1) & 1), status);
    }
    const uint32_t peer = (uint32_t)((h ^ 1) * NQ + q);
    if (ld_cluster_u32(mapa(smem_u32((const void*)&flags[0]), peer)) != 0)
      mbar_drain<true>(xbar, 0, status);
  }
  cluster_arrive();                                     // the others' flags have been read
  // this half's lines of the solution that were computed: within [0, m] or [m + 1, L)
  const int o0 = h ? m + 1 : nlo, o1 = h ? nhi + 1 : m + 1;
  const int rb = (b + NQ - 1) / NQ, r0 = q * rb, r1 = min(b, r0 + rb);   // and this CTA's rows
  if (a.dim == 2 && kind != K_RAW) {
    twist_epilogue<C, 8>(
        a, g, kind, sub, yl - (long long)ka * b, b, 0, 1, o0, o1, r0, r1,
        [&](int) { return reinterpret_cast<C*>(a.lane); },
        [&](int) { return reinterpret_cast<C*>(a.trace); });
  } else {
    Rows R;
    R.RB = b;
    R.r0 = r0;
    R.r1 = r1;
    R.ls = b;
    R.k0 = o0;
    R.k1 = o1;
    front_epilogue<C>(a, g, kind, sub, yl - (long long)ka * b + r0, R);
  }
  cluster_wait();                                       // this CTA's flags have been read
}

// ---- complex128 -------------------------------------------------------------------------
// The same solve with FP64 products, which two lanes a clock per SM bound (a warp's multiply-
// add keeps its scheduler's FP64 unit busy for 64 clocks however many lanes are active).  So a
// block's rows are split over two CTAs per half, and the row and column split inside a CTA is
// chosen to fill its W warps with as few idle lanes as possible: thread t has row t mod nr and
// column chunk t / nr, CH = 32 W / nr chunks (W = 12: three warps per scheduler; shorter lines take
// 6 warps and two CTAs per SM or 3 and four, see rows_warps).  Every CTA copies whole
// stored blocks; a thread's entries have fixed offsets in the slot, and those of step s + 1
// are read while step s is finished.  CTA (h, q) owns rows [q RB, q RB + nr) of its half's
// line vectors; the owners send their entries of the next vector to the mate (st.async, two
// barriers by step parity, re-armed one step ahead), and at the last step before the middle
// line their part of its right-hand side to both CTAs of the other half.
// kGlobal: the line vectors and their sources in global memory (L2-resident, a region per CTA),
// where they do not fit beside two slots: many lines per subdomain, and the 3D planes of up to 92
// nodes.  An owner's next entry is loaded a step ahead.  ms per application, four-CTA kernel on whole
// blocks / cluster split on the plain factor / this: 512^2 on 2 x 8 (92-node lines, 282 of them) 23.3 /
// 35.3 / 16.9, 1024^2 on 4 x 16 49.8 / 135 / 36.0, 24^3 on 8 x 8 beams of 81-node planes 3.8 / 7.7 /
// 2.8; 640^2 on 8 x 8 (108-node lines) - / 46.4 / 16.0.
constexpr int kRowsMaxCH = 32;
template <int W, int NC, bool kGlobal>
__global__ void __launch_bounds__(W * 32 + 32, 12 / W)
k_twist_rows(FrontArgs a, Twist tg, double2* lines, int* status) {
  using C = double2;
  constexpr int ncons = W * 32;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  griddep_launch_dependents();                          // the next level may start its setup
  const Task task = a.tasks[a.task_off + blockIdx.x / 4];
  const int sub = task.sub, kind = task.kind;
  const SubGeom g = a.subs[sub];
  const int b = g.b, L = g.L;
  const int rank = (int)cluster_rank();
  const int h = rank >> 1, q = rank & 1;               // half (0: from line 0), row group
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int m = twist_line(L);
  const int nf = h ? L - 1 - m : m;
  int slo, shi, nlo, nhi;
  const int dim = kGlobal ? a.dim : 2;
  source_lines(g, kind, dim, slo, shi);
  needed_lines(g, kind, dim, nlo, nhi);
  const int f0 = h ? min(L - 1 - shi, nf) : min(slo, nf);
  const int nsteps = nf + 1 + (h ? nhi - m : m - nlo);
  const int nit = nsteps - f0;                         // steps this CTA runs: s = f0 + it
  const int RB = (b + 1) / 2, r0 = q * RB, nr = q ? b - RB : RB;
  const int ka = h ? m : 0, kb = h ? L : m + 1;        // lines of this half (m in both)
  const int CH = min(kRowsMaxCH, ncons / RB), nc = (b + CH - 1) / CH;
  // shared memory: ring[nslot][slot_bytes] | full[8] | empty[8] | vbar[2] | xbar[2] | flags[4]
  // (32-bit) | vb[2][bs] | part[32 W] | xb[bs] | H[2][bs] | V[2][Lh] | yl[Lh][RB]; kGlobal: H, V
  // and yl are not there, yl is this CTA's region of `lines`
  unsigned char* ring = smem_raw;
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + (size_t)tg.nslot * tg.slot_bytes);
  uint64_t* empty = full + kSoloMaxSlots;
  uint64_t* vbar = empty + kSoloMaxSlots;              // the mate's entries of the next vector
  uint64_t* xbar = vbar + 2;                           // [qq]: part of line m of CTA (1 - h, qq)
  // flags[0]: this CTA sent its part of line m (all rows or none); flags[1]: the last step
  // whose vector entries it sent to its mate; flags[2]: the step a wait gave up in (stop_at);
  // flags[3]: the last step whose barrier for the step after next is armed, plus one
  volatile uint32_t* flags = reinterpret_cast<volatile uint32_t*>(xbar + 2);
  int* stop = reinterpret_cast<int*>(xbar + 3);
  const int bs = tg.bs;
  C* vb = reinterpret_cast<C*>(full + kTwistBars);
  C* part = vb + 2 * bs;
  C* xb = part + ncons;
  C* H = xb + bs;
  C* Vs = H + 2 * bs;
  C* yl = kGlobal ? lines + (size_t)blockIdx.x * tg.Lh * (bs / 2) : Vs + 2 * tg.Lh;
  auto line = [&](int k) { return yl + (k - ka) * nr; };
  const TileStore ts = tg.ts;
  const C* fac = reinterpret_cast<const C*>(a.fac) + g.fac_off;
  const int stride = block_elems(b, ts);
  const uint32_t blk_bytes = (uint32_t)(stride * (int)sizeof(C));
  const uint32_t mate_bytes = (uint32_t)((b - nr) * sizeof(C));
  auto blk = [&](int s) {
    if (s < nf) return h ? L - 1 - s : s;
    return h ? m + (s - nf) : m - (s - nf);
  };
  auto src = [&](int it) { return fac + (size_t)blk(f0 + it) * stride; };
  auto issue = [&](int it, int slot) {
    mbar_expect_tx(&full[slot], blk_bytes);
    bulk_g2s(ring + (size_t)slot * tg.slot_bytes, src(it), blk_bytes, &full[slot]);
  };
  auto vparity = [](int it) { return (uint32_t)(((it - 1) >> 1) & 1); };
  bool timed_out = false;

  if (tid == 0) {
    for (int i = 0; i < tg.nslot; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], W);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&vbar[i], 1);
      mbar_init(&xbar[i], 1);
    }
    flags[0] = flags[1] = 0;
    flags[3] = 1;                                       // steps 1 and 2 are armed below
    *stop = 0x7fffffff;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(&xbar[0], (uint32_t)(RB * sizeof(C)));
    mbar_expect_tx(&xbar[1], (uint32_t)((b - RB) * sizeof(C)));
    if (nit > 1) mbar_expect_tx(&vbar[1], mate_bytes);  // it = 1
    if (nit > 2) mbar_expect_tx(&vbar[0], mate_bytes);  // it = 2
  }
  __syncthreads();
  cluster_sync_all();                                  // every CTA's barriers are armed
  if (w == W && lane == 0) {
    for (int t = 0; t < min(tg.PD, nit); ++t) bulk_prefetch_l2(src(t), blk_bytes);
    for (int t = 0; t < min(tg.nslot, nit); ++t) issue(t, t);
  }
  griddep_wait();                                       // traces of the previous level
  const Sides S(g, kind);
  const bool sweep = kind != K_RAW && kind != K_LOCAL;
  if (!kGlobal && sweep) {
    side_sources<C>(a, g, kind, S, ka, kb, H, bs, Vs, tg.Lh, tid, blockDim.x);
    __syncthreads();
  }
  auto source = [&](int k, int p) -> C {
    return sweep ? side_entry<C>(S, H, bs, Vs, tg.Lh, ka, k, p)
                 : kind == K_LOCAL ? local_entry<C>(a, g, k, p) : to<C>(a.g_raw[(size_t)k * b + p]);
  };
  // this CTA's rows of the solution: line vectors of nr entries
  auto rows = [&](int lo, int hi) {
    Rows R;
    R.RB = R.ls = nr;
    R.r0 = r0;
    R.r1 = r0 + nr;
    R.k0 = lo;
    R.k1 = hi;
    return R;
  };
  if constexpr (kGlobal) {
    build_source<C>(a, g, kind, yl - (long long)ka * nr, rows(ka, kb));
    Rows R;                                             // the first vector, every row of it
    R.RB = R.r1 = R.ls = b;
    R.r0 = 0;
    R.k0 = blk(f0);
    R.k1 = R.k0 + 1;
    build_source<C>(a, g, kind, vb - (long long)R.k0 * b, R);
  } else {
    for (int t = tid; t < (kb - ka) * nr; t += blockDim.x) {
      const int kk = t / nr;
      yl[t] = source(ka + kk, r0 + t - kk * nr);
    }
  }
  __syncthreads();

  int varmed = nit > 2 ? 2 : nit - 1, vok = 0;          // (tid 0) last step armed / received
  if (w == W) {
    // ---- producer (as k_twist) ---------------------------------------------------------
    if (lane == 0) {
      int issued = min(tg.nslot, nit);
      for (int t = tg.nslot; t < nit; ++t) {
        const int slot = t % tg.nslot;
        mbar_wait<false>(&empty[slot], (uint32_t)((t / tg.nslot - 1) & 1), status, timed_out, a.spin);
        if (timed_out) break;
        if (tg.PD > 0 && t + tg.PD < nit) bulk_prefetch_l2(src(t + tg.PD), blk_bytes);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        issue(t, slot);
        issued = t + 1;
      }
      drain_ring(full, tg.nslot, issued, status);
    }
  } else {
    const int ch = tid / nr, row = tid - ch * nr;
    const bool worker = ch < CH;
    const bool owner = tid < nr;                        // owns row r0 + tid of the vectors
    const int orow = r0 + tid, c0 = worker ? min(b, ch * nc) : 0;
    const int cn = worker ? min(nc, b - c0) : 0;        // columns of this thread
    uint32_t off[NC];                                   // byte offsets in a slot
#pragma unroll
    for (int t = 0; t < NC; ++t)
      off[t] = t < cn ? (uint32_t)(tile_index(b, ts, 16, r0 + row, c0 + t) * 16) : 0u;
    const int cpl_off = part_cpl(b, ts, 0), lrow = owner ? tid : 0;
    const uint32_t mate = (uint32_t)(rank ^ 1), oth = (uint32_t)(2 * (h ^ 1));
    auto send_middle = [&](C v) {                       // this row's part of line m
#pragma unroll
      for (uint32_t j = 0; j < 2; ++j)
        st_async(mapa(smem_u32(xb + orow), oth + j), v, mapa(smem_u32(&xbar[q]), oth + j));
      flags[0] = 1;
    };
    auto wait_middle = [&]() {                          // the other half's CTAs' parts
      mbar_wait<true>(&xbar[0], 0, status, timed_out, a.spin);
      mbar_wait<true>(&xbar[1], 0, status, timed_out, a.spin);
    };
    if (f0 >= nf) {
      // the middle line comes first: this half adds nothing to its right-hand side
      if (owner) send_middle(czero<C>());
      wait_middle();
    }
    for (int p = tid; p < b; p += ncons) {              // the first vector, every row of it
      const C v = kGlobal ? vb[p] : source(blk(f0), p);
      vb[p] = f0 >= nf ? v + xb[p] : v;
    }
    int nslot = 0;
    uint32_t phase = 0;
    C D[NC], cpl, Aval;
    auto load_block = [&](int it) {                     // entries and owner's operands of step it
      const int s = f0 + it, k = blk(s);
      mbar_wait<false>(&full[nslot], phase, status, timed_out, a.spin);
      const unsigned char* sp = ring + (size_t)nslot * tg.slot_bytes;
#pragma unroll
      for (int t = 0; t < NC; ++t) D[t] = *reinterpret_cast<const C*>(sp + off[t]);
      Aval = line(s < nf ? (h ? k - 1 : k + 1) : k)[lrow];
      cpl = reinterpret_cast<const C*>(sp)[cpl_off + ((s < nf) == (h != 0) ? (b + 1) & ~1 : 0) +
                                           (owner ? orow : 0)];
      __syncwarp();
      if (lane == 0 && !timed_out) mbar_arrive(&empty[nslot]);   // see k_twist
    };
    load_block(0);
    if (timed_out) stop_at(stop, -1);
    consumer_sync(ncons);
    int halt = *(volatile int*)stop;
    for (int it = 0; it < nit; ++it) {
      const int s = f0 + it;
      const int k = blk(s);
      C* v = vb + (it & 1) * bs;
      if (it > 0) {
        // the mate's rows of this step's vector; then re-arm the barrier for step it + 2: the
        // mate sends step it + 2 only after it received this CTA's step it + 1, which is sent
        // after this point and only if the barrier was armed
        mbar_wait<true>(&vbar[it & 1], vparity(it), status, timed_out, a.spin);
        if (tid == 0 && !timed_out) {
          vok = it;
          if (it + 2 < nit) {
            mbar_expect_tx(&vbar[it & 1], mate_bytes);
            varmed = it + 2;
          }
          flags[3] = (uint32_t)(it + 1);
        }
        if (s == nf) {
          // middle line: add the other half's part of its right-hand side
          wait_middle();
          consumer_sync(ncons);
          for (int p = tid; p < b; p += ncons) v[p] = v[p] + xb[p];
          consumer_sync(ncons);
        }
      }
      C sum = czero<C>();
#pragma unroll
      for (int t = 0; t < NC; ++t)
        if (t < cn) sum = cfma(D[t], v[c0 + t], sum);
      if (worker) part[tid] = sum;
      const C Ac = Aval, cc = cpl;
      if (it + 1 < nit) {
        if (++nslot == tg.nslot) {
          nslot = 0;
          phase ^= 1u;
        }
        load_block(it + 1);
      }
      if (halt < it) break;                             // a wait gave up: leave together
      consumer_sync(ncons);                             // the partial sums are there
      if (owner) {
        C s0 = part[tid], s1 = part[nr + tid];          // (CH >= 2)
        for (int c = 2; c + 1 < CH; c += 2) {
          s0 = s0 + part[c * nr + tid];
          s1 = s1 + part[(c + 1) * nr + tid];
        }
        if (CH & 1) s0 = s0 + part[(CH - 1) * nr + tid];
        sum = s0 + s1;
        C nv = czero<C>();
        C* yk = line(k) + tid;
        if (s < nf) {
          *yk = sum;                                    // y_k (z_k)
          const C t = cmul(cc, sum);
          nv = Ac - t;
          // next is the middle line: every owner of this CTA sends in this step, timed out or
          // not (all rows or none)
          if (s + 1 == nf) send_middle(mk(-t.x, -t.y));
        } else {
          const C x = s == nf ? sum : Ac - sum;         // x_m, or x_k = y_k - D_k^-1 (c x)
          *yk = x;
          nv = cmul(cc, x);
        }
        if (it + 1 < nit) {
          C* dst = vb + ((it + 1) & 1) * bs + orow;
          *dst = nv;
          if (flags[3] == (uint32_t)(it + 1)) {
            st_async(mapa(smem_u32(dst), mate), nv, mapa(smem_u32(&vbar[(it + 1) & 1]), mate));
            if (tid == 0) flags[1] = (uint32_t)(it + 1);
          }
        }
      }
      if (timed_out) stop_at(stop, it);
      consumer_sync(ncons);                             // this CTA's rows of the next vector
      halt = *(volatile int*)stop;
    }
  }
  const bool gave_up = __syncthreads_or(timed_out) != 0;
  cluster_sync_all();                                   // every CTA has left its loop
  if (gave_up && tid == 0) {
    // as k_twist: wait for what may still be in flight to this CTA (the mate's vector entries
    // of the steps after the last one received, up to the last one sent and armed)
    const int sent = (int)ld_cluster_u32(mapa(smem_u32((const void*)&flags[1]), (uint32_t)(rank ^ 1)));
    for (int t = vok + 1; t <= min(sent, varmed); ++t)
      mbar_drain<true>(&vbar[t & 1], vparity(t), status);
    for (uint32_t j = 0; j < 2; ++j)
      if (ld_cluster_u32(mapa(smem_u32((const void*)&flags[0]), (uint32_t)(2 * (h ^ 1)) + j)) != 0)
        mbar_drain<true>(&xbar[j], 0, status);
  }
  cluster_arrive();                                     // the others' flags have been read
  const int o0 = h ? m + 1 : nlo, o1 = h ? nhi + 1 : m + 1;
  if (kGlobal && dim != 2) {
    front_epilogue<C>(a, g, kind, sub, yl - (long long)ka * nr, rows(o0, o1));
  } else if (kind != K_RAW) {
    twist_epilogue<C, 4>(
        a, g, kind, sub, yl - (long long)ka * nr - r0, nr, 0, 1, o0, o1, r0, r0 + nr,
        [&](int) { return reinterpret_cast<C*>(a.lane); },
        [&](int) { return reinterpret_cast<C*>(a.trace); });
  } else {
    for (int t = tid; t < (o1 - o0) * nr; t += blockDim.x) {
      const int kk = t / nr, p = t - kk * nr;
      a.x_raw[(size_t)(o0 + kk) * b + r0 + p] = line(o0 + kk)[p];
    }
  }
  cluster_wait();                                       // this CTA's flags have been read
}

// ---- several right-hand sides ------------------------------------------------------------
// The same solve for a block of K right-hand sides (the pipelining over right-hand sides that
// Sec. 1 and Sec. 6 point to for many sources): a tile in registers is used for all of them,
// with the products and sums of k_twist in the same order, so each one's result is bit for bit
// the single application's.  The workers form NG groups that hold the same tiles; group e does
// the right-hand sides e, e + NG, ..., ER of them between two barriers (what the partial sums
// leave room for).  The line vectors do not fit beside the ring:
// they live in a global scratch per CTA ([line][K][b], L2-resident), and the source stays in
// its compact form (H, V of every right-hand side) or is read from the input when it is needed.
// An owner's next operands are loaded one step ahead.
struct MultiArgs {
  FrontArgs a;                  // plan, factors, coefficients (rin / lane / trace unused)
  const double2* rin[kMaxRHS];  // stage-1 input of each right-hand side
  void* lane[kMaxRHS];          // accumulation lanes of each right-hand side
  void* trace[kMaxRHS];         // trace arrays of each right-hand side
  float2* line;                 // line vectors, per CTA [Lmax][K][bmax]
  long long line_stride;        // elements per CTA
  int K;
};

__device__ inline FrontArgs rhs_args(const MultiArgs& m, int c) {
  FrontArgs a = m.a;
  a.rin = m.rin[c];
  a.lane = m.lane[c];
  a.trace = m.trace[c];
  return a;
}

// KG: right-hand sides per group at most.  OG: owners per row.  A group on lines of more than 64 nodes has
// at least two threads per row (160 to 256 for 136 to 253 tiles), and each owns its row for every second
// right-hand side; with one owner the others waited while it walked a round's four.  ms per block with
// one owner -> two (the kernel on whole blocks): 1024^2 of 92-node lines, 8 right-hand sides 20.4 ->
// 15.5 (19.6), 4 9.9 -> 8.4 (11.4); 1008^2 of 64- to 66-node lines, 8 28.3 -> 20.5 (25.1).
template <int T, int GM, int NG, int ER, int KG>
__global__ void __launch_bounds__(320, 1)
k_twist_multi(const __grid_constant__ MultiArgs ma, Twist tg, int* status) {
  using C = float2;
  constexpr int VN = T * GM, SP = part_stride(T, GM);
  constexpr int OG = NG == 1 && KG > 1 ? 2 : 1, KO = (KG + OG - 1) / OG;   // owners per row, share
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const FrontArgs& a = ma.a;
  const int K = ma.K;
  griddep_launch_dependents();                          // the next level may start its setup
  const Task task = a.tasks[a.task_off + blockIdx.x / 2];
  const int sub = task.sub, kind = task.kind;
  const SubGeom g = a.subs[sub];
  const int b = g.b, L = g.L, G = tile_rows(b, T);
  const int h = (int)cluster_rank();
  const uint32_t peer = (uint32_t)(h ^ 1);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int ncw = (int)(blockDim.x >> 5) - 1;          // consumer warps; the last is the producer
  const int ncons = ncw * 32;
  const int m = twist_line(L);
  const int nf = h ? L - 1 - m : m;
  int slo, shi, nlo, nhi;
  source_lines(g, kind, 2, slo, shi);
  needed_lines(g, kind, 2, nlo, nhi);
  const int f0 = h ? min(L - 1 - shi, nf) : min(slo, nf);
  const int nsteps = nf + 1 + (h ? nhi - m : m - nlo);
  const int nit = nsteps - f0;                         // steps this CTA runs: s = f0 + it
  const int ka = h ? m : 0, kb = h ? L : m + 1;        // lines of this half (m in both)
  // shared memory: ring[nslot][slot_bytes] | full[8] | empty[8] | - [2] | xbar[2] | flags[4]
  // (32-bit) | vb[K][2][VN] | part[NG ER][GM][SP] | dump[8] | xb[K][bs] | H[K][2][bs] | V[K][2][Lh]
  unsigned char* ring = smem_raw;
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + (size_t)tg.nslot * tg.slot_bytes);
  uint64_t* empty = full + kSoloMaxSlots;
  uint64_t* xbar = empty + kSoloMaxSlots + 2;          // the other half's parts of line m
  volatile uint32_t* flags = reinterpret_cast<volatile uint32_t*>(xbar + 2);   // [0]: sent
  int* stop = reinterpret_cast<int*>(xbar + 3);
  const int bs = tg.bs;
  C* vb = reinterpret_cast<C*>(full + kTwistBars);
  C* part = vb + K * 2 * VN;
  constexpr int NP = NG * (ER < KG ? ER : KG);          // partial-sum buffers
  C* dump = part + NP * GM * SP;
  C* xb = dump + 8;
  C* H = xb + K * bs;
  C* Vs = H + K * 2 * bs;
  C* yl = ma.line + (size_t)blockIdx.x * ma.line_stride;   // [L][K][b], global
  const int LS = K * b;
  const TileStore ts{T, 1};
  const C* fac = reinterpret_cast<const C*>(a.fac) + g.fac_off;
  const int stride = block_elems(b, ts);
  const uint32_t blk_bytes = (uint32_t)(stride * (int)sizeof(C));
  auto blk = [&](int s) {
    if (s < nf) return h ? L - 1 - s : s;
    return h ? m + (s - nf) : m - (s - nf);
  };
  auto src = [&](int it) { return fac + (size_t)blk(f0 + it) * stride; };
  auto issue = [&](int it, int slot) {
    mbar_expect_tx(&full[slot], blk_bytes);
    bulk_g2s(ring + (size_t)slot * tg.slot_bytes, src(it), blk_bytes, &full[slot]);
  };
  bool timed_out = false;

  if (tid == 0) {
    for (int i = 0; i < tg.nslot; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], (uint32_t)ncw);
    }
    mbar_init(&xbar[0], 1);
    flags[0] = 0;
    *stop = 0x7fffffff;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(&xbar[0], (uint32_t)(K * b * sizeof(C)));   // K entries per row
  }
  for (int t = tid; t < K * 2 * VN + NP * GM * SP; t += blockDim.x) vb[t] = czero<C>();
  __syncthreads();
  cluster_sync_all();                                  // the partner's xbar is armed
  if (w == ncw && lane == 0) {
    for (int t = 0; t < min(tg.PD, nit); ++t) bulk_prefetch_l2(src(t), blk_bytes);
    for (int t = 0; t < min(tg.nslot, nit); ++t) issue(t, t);
  }
  griddep_wait();                                       // traces of the previous level
  const Sides S(g, kind);
  const bool sweep = kind != K_LOCAL;
  if (sweep)
    for (int c = 0; c < K; ++c)
      side_sources<C>(rhs_args(ma, c), g, kind, S, ka, kb, H + c * 2 * bs, bs, Vs + c * 2 * tg.Lh,
                      tg.Lh, tid, blockDim.x);
  __syncthreads();

  if (w == ncw) {
    // ---- producer (as k_twist) ---------------------------------------------------------
    if (lane == 0) {
      int issued = min(tg.nslot, nit);
      for (int t = tg.nslot; t < nit; ++t) {
        const int slot = t % tg.nslot;
        mbar_wait<false>(&empty[slot], (uint32_t)((t / tg.nslot - 1) & 1), status, timed_out, a.spin);
        if (timed_out) break;
        if (tg.PD > 0 && t + tg.PD < nit) bulk_prefetch_l2(src(t + tg.PD), blk_bytes);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        issue(t, slot);
        issued = t + 1;
      }
      drain_ring(full, tg.nslot, issued, status);
    }
  } else {
    // ---- workers and owners as in k_twist, in every group ---------------------------------
    const int gth = ncons / NG, grp = tid / gth, gt = tid - grp * gth;
    const int kg = K > grp ? (K - grp + NG - 1) / NG : 0;   // right-hand sides here
    auto rhs = [&](int e) { return grp + NG * e; };
    int I, J;
    const bool worker = worker_tile<1>(gt, G, 0, I, J);
    const unsigned unit = (unsigned)tile_count(G, 1, 0) * 16;
    const unsigned tile_off = worker ? (unsigned)gt * 16 : 0;
    const int og = OG == 1 ? 0 : gt / (gth / OG);         // owner: row ot, right-hand sides og + OG i
    const int ot = OG == 1 ? gt : gt - og * (gth / OG);
    const bool owner = ot < b;
    const int OI = owner ? ot / T : 0, oi = owner ? ot - OI * T : 0;
    const int cpl_off = part_cpl(b, ts, 0);
    int doff[T];
#pragma unroll
    for (int j = 0; j < T; ++j)
      doff[j] = owner ? tile_count(G, 1, 0) * T * T + OI +
                            (oi >= j ? oi * (oi + 1) / 2 + j : j * (j + 1) / 2 + oi) * G
                      : 0;
    const uint32_t rbar = mapa(smem_u32(xbar), peer);
    auto source = [&](int c, int k, int p) -> C {
      if (sweep) return side_entry<C>(S, H + c * 2 * bs, bs, Vs + c * 2 * tg.Lh, tg.Lh, ka, k, p);
      if (k < g.oy0 || k >= g.oy1 || p < g.ox0 || p >= g.ox1) return czero<C>();
      return to<C>(ma.rin[c][(size_t)(g.gy0 + k) * a.Ne + g.gx0 + p]);
    };
    auto send_middle = [&](int c, C v) {
      st_async(mapa(smem_u32(xb + c * bs + ot), peer), v, rbar);
      flags[0] = 1;
    };
    // operands of step it: the next line's source (forward), or y_k (backward: stored by this
    // thread at least two steps before, or zero on a line whose forward step was skipped)
    C An[KO];
    auto fetch = [&](int it) {
      const int s = f0 + it, k = blk(s);
      const bool seen = (h ? L - 1 - k : k) >= f0;
#pragma unroll
      for (int i = 0; i < KO; ++i) {
        const int e = og + OG * i;
        An[i] = czero<C>();
        if (owner && e < kg && it < nit) {
          if (s < nf) An[i] = source(rhs(e), h ? k - 1 : k + 1, ot);
          else if (s > nf && seen) An[i] = __ldcg(yl + (size_t)k * LS + rhs(e) * b + ot);
        }
      }
    };
    if (owner && kg > 0) {
      const int k = blk(f0);
      if (f0 >= nf) {
        // the middle line comes first (see k_twist)
        for (int e = og; e < kg; e += OG) send_middle(rhs(e), czero<C>());
        mbar_wait<true>(xbar, 0, status, timed_out, a.spin);
      }
      for (int e = og; e < kg; e += OG) {
        const int c = rhs(e);
        C v = source(c, k, ot);
        if (f0 >= nf) v = v + xb[c * bs + ot];
        vb[c * 2 * VN + ot] = v;
      }
    }
    fetch(0);
    int slot = 0, nslot = 0;
    uint32_t phase = 0;
    C D[T * T], dr[T];
    auto ready = [&]() { mbar_wait<false>(&full[nslot], phase, status, timed_out, a.spin); };
    const int lrow = owner ? ot : 0;
    ready();
#pragma unroll
    for (int i = 0; i + 2 < T; i += 2) load_rows<T>(D, ring + tile_off, unit, i);
    if (timed_out) stop_at(stop, -1);
    consumer_sync(ncons);
    int halt = *(volatile int*)stop;
    for (int it = 0; it < nit; ++it) {
      const int s = f0 + it;
      const int k = blk(s);
      const bool more = it + 1 < nit;
      // the tile's last rows and the owner's operands of this block (see k_twist)
      load_rows<T>(D, ring + (size_t)slot * tg.slot_bytes + tile_off, unit, T - 2);
      const C* sl = reinterpret_cast<const C*>(ring + (size_t)slot * tg.slot_bytes);
      const C cc = sl[cpl_off + ((s < nf) == (h != 0) ? (b + 1) & ~1 : 0) + lrow];
#pragma unroll
      for (int j = 0; j < T; ++j) dr[j] = sl[doff[j]];
      C Ac[KO];
#pragma unroll
      for (int i = 0; i < KO; ++i) Ac[i] = An[i];
      fetch(it + 1);
      auto tile = [&](int e, int pb, auto refill) {
        const C* v = vb + rhs(e) * 2 * VN + (it & 1) * VN;
        C* pt = part + (pb * NG + grp) * GM * SP;
        tile_products<T, decltype(refill)::value>(
            D, v + I * T, v + J * T, worker ? pt + J * SP + I * T : dump,
            worker ? pt + I * SP + J * T : dump, [] {}, &full[nslot], phase, ready,
            ring + (size_t)nslot * tg.slot_bytes + tile_off, unit);
      };
      if (more && ++nslot == tg.nslot) {
        nslot = 0;
        phase ^= 1u;
      }
      const bool mid = s + 1 == nf;
      bool left = false;
#pragma unroll
      for (int e0 = 0; e0 < KG; e0 += ER) {
        if (e0 > 0 && e0 * NG >= K) break;              // (the same in every group)
        if (e0 > 0) consumer_sync(ncons);               // the partial sums have been read
        const int e1 = min(kg, e0 + ER);
        const bool last = more && e1 == kg && e1 > e0;  // the group's last products of the step
#pragma unroll 1
        for (int e = e0; e < (last ? e1 - 1 : e1); ++e) tile(e, e - e0, std::false_type{});
        if (last) tile(e1 - 1, e1 - 1 - e0, std::true_type{});
        if (halt < it) {                                // a wait gave up: leave together
          left = true;
          break;
        }
        consumer_sync(ncons);                           // the partial sums are there
        if (owner) {
#pragma unroll
          for (int i = 0; i < ER / OG; ++i) {
            const int at = e0 / OG + i;                   // (its place in Ac)
            const int e = e0 + og + OG * i;
            if (at >= KO || e >= e1) continue;
            const int c = rhs(e), u = e - e0;
            C vO[T], dA = czero<C>(), dB = dA;
            load_run<T>(vb + c * 2 * VN + (it & 1) * VN + OI * T, vO);
#pragma unroll
            for (int j = 0; j < T; ++j) mac(dr[j], vO[j], dA, dB);
            const C sum = row_sum<T, GM, 1>(part + (u * NG + grp) * GM * SP + ot, G, OI, 0,
                                            mk(dA.x - dA.y, dB.x + dB.y));
            C* yk = yl + (size_t)k * LS + c * b + ot;
            C nv;
            if (s < nf) {
              *yk = sum;                                // y_k (z_k)
              const C t = cmul(cc, sum);
              nv = Ac[at] - t;
              // every owner sends, timed out or not: all rows or none
              if (mid) send_middle(c, mk(-t.x, -t.y));
            } else {
              const C x = s == nf ? sum : Ac[at] - sum;
              *yk = x;
              nv = cmul(cc, x);
            }
            vb[c * 2 * VN + ((it + 1) & 1) * VN + ot] = nv;
          }
        }
      }
      if (left) break;
      if (kg == 0 && more) ready();                     // (an idle group keeps the ring's pace)
      __syncwarp();
      if (lane == 0 && !timed_out) mbar_arrive(&empty[slot]);   // see k_twist
      if (owner && mid && kg > 0) {
        // add the other half's parts of line m's right-hand side
        mbar_wait<true>(xbar, 0, status, timed_out, a.spin);
        for (int e = og; e < kg; e += OG) {
          const int c = rhs(e);
          C* nv = vb + c * 2 * VN + ((it + 1) & 1) * VN + ot;
          *nv = *nv + xb[c * bs + ot];
        }
      }
      if (timed_out) stop_at(stop, it);
      consumer_sync(ncons);                             // the next vectors are there
      halt = *(volatile int*)stop;
      slot = nslot;
    }
  }
  const bool gave_up = __syncthreads_or(timed_out) != 0;
  cluster_sync_all();                                   // both halves have left their loops
  if (gave_up && tid == 0) {
    // as k_twist: wait for the other half's parts of line m if it sent them
    if (ld_cluster_u32(mapa(smem_u32((const void*)&flags[0]), peer)) != 0)
      mbar_drain<true>(xbar, 0, status);
  }
  cluster_arrive();                                     // the other half's flag has been read
  const int o0 = h ? m + 1 : nlo, o1 = h ? nhi + 1 : m + 1;
  twist_epilogue<C, 8>(
      a, g, kind, sub, yl, LS, b, K, o0, o1, 0, b,
      [&](int c) { return reinterpret_cast<C*>(ma.lane[c]); },
      [&](int c) { return reinterpret_cast<C*>(ma.trace[c]); });
  cluster_wait();                                       // this CTA's flag has been read
}

// ---- launches ---------------------------------------------------------------------------
// Geometry of the twisted kernels for a plan, false when they do not apply: 2D lines, and (in
// 3D) planes of at most 92 nodes.  Tiles of 4 x 4 on one CTA per half up to 96 nodes: a
// 92-node line has 253 of them, two warps per scheduler, which hide one another's waits (with
// tiles of 6 x 6, one warp per scheduler, less shared-memory traffic, an application of the
// 1024^2 workload took 3.3 ms, with 4 x 4 2.9 ms).  Wider lines share tiles of 6 x 6 between
// two CTAs per half, as whole blocks no longer fit beside the line vectors.  Complex128:
// k_twist_rows, four CTAs per solve.
// columns per thread of k_twist_rows with W warps (0: too few threads for the rows)
static int rows_columns(int b, int W) {
  const int CH = std::min(kRowsMaxCH, W * 32 / ((b + 1) / 2));
  return CH < 2 ? 0 : (b + CH - 1) / CH;
}
// Warps of k_twist_rows, CTAs per SM 12 / W: 3 on lines of up to 36 nodes, 6 up to 54 (what eight
// columns per thread cover), 12 above.  Short lines are bound by the solves that run at once where
// levels are full, and where they are not by the barriers and by the sum over the column chunks,
// which fewer threads shorten.  ms per application with 12 warps -> with these (the four-CTA kernel
// on whole blocks): 16 x 16 subdomains of 20-node lines 8.8 -> 2.7 (4.8), 36 nodes 13.5 -> 4.9 (9.9),
// 52 nodes 17.8 -> 9.0 (17.9); 4 x 4 of 20 nodes 0.96 -> 0.40 (0.53), 36 nodes 1.50 -> 0.64 (1.12),
// 52 nodes 1.96 -> 1.16 (1.95).  36 nodes with 6 warps: 6.1 and 0.86.
static int rows_warps(int b) { return b <= 36 ? 3 : b <= 54 ? 6 : 12; }
// tile rows at most: lines of up to 64 nodes, up to 96, wider ones on two CTAs per half
constexpr int kGMs = 16, kGM1 = 24, kGM2 = 26;
static bool twist_geometry(const Ctx& c, Twist& t, int& GM, int& threads, size_t& smem) {
  const bool c64 = c.c64();
  const int b = c.bmax;
  const size_t es = c.welem();
  if (c.cube || (c.dim != 2 && b > 92)) return false;
  t.ts.NQ = !c64 || b <= 96 ? 1 : 2;
  t.ts.T = t.ts.NQ == 1 ? 4 : 6;
  t.Lh = c.Lmax - twist_line(c.Lmax);
  t.bs = (b + 1) & ~1;
  t.PD = c.p.prefetch_steps < 0 ? 0 : c.p.prefetch_steps;
  const int elems = std::max(part_elems(b, t.ts, 0), t.ts.NQ > 1 ? part_elems(b, t.ts, 1) : 0);
  t.slot_bytes = (unsigned)((elems * es + 127) / 128 * 128);
  size_t fixed = kTwistBars * sizeof(uint64_t);
  if (c64) {
    GM = t.ts.NQ == 2 ? kGM2 : b <= 64 ? kGMs : kGM1;
    const int G = tile_rows(b, t.ts.T);
    if (G > GM) return false;
    const int tiles = std::max(tile_count(G, t.ts.NQ, 0), t.ts.NQ > 1 ? tile_count(G, 2, 1) : 0);
    threads = (std::max(tiles, b) + 31) / 32 * 32 + 32;
    if (threads > twist_threads(t.ts.T, GM, t.ts.NQ)) return false;
    const int SP = part_stride(t.ts.T, GM);
    fixed += ((size_t)2 * t.ts.T * GM + GM * SP + 8 + (t.ts.NQ == 2 ? 3 : 1) * t.bs +
              (size_t)t.Lh * b + 1) * es;
  } else {
    GM = 0;
    if (b < 2) return false;
    const size_t vectors = fixed + (size_t)3 * t.bs * es;
    const size_t lines = (2 * (size_t)t.bs + 2 * t.Lh + (size_t)t.Lh * ((b + 1) / 2)) * es;
    t.W = rows_warps(b);
    const int nc = rows_columns(b, t.W);
    if (nc < 1 || nc > (t.W == 12 ? 16 : 8)) return false;
    const size_t limit = 228 * 1024 / (12 / t.W) - 1024;
    threads = (t.W + 1) * 32;
    // line vectors in shared memory (2D), or, where they do not fit with as many CTAs per SM, in
    // global memory: more solves at once are worth more (1024^2 in one row of 64 subdomains of
    // 36-node lines, ms per application: shared memory and 12 warps 373, global and 3 warps 177)
    for (int gl = c.dim == 2 ? 0 : 1; gl < 2; ++gl) {
      const size_t all = vectors + (gl ? 0 : lines) + t.W * 32 * es;
      if (all + 2 * (size_t)t.slot_bytes > limit) continue;
      t.gl = gl;
      t.nslot = (int)std::min<size_t>(kSoloMaxSlots, (limit - all) / t.slot_bytes);
      smem = all + (size_t)t.nslot * t.slot_bytes;
      return true;
    }
    return false;
  }
  const size_t limit = 227 * 1024;
  if (fixed + 2 * (size_t)t.slot_bytes > limit) return false;
  t.W = t.gl = 0;
  t.nslot = (int)std::min<size_t>(kSoloMaxSlots, (limit - fixed) / t.slot_bytes);
  smem = fixed + (size_t)t.nslot * t.slot_bytes;
  return true;
}
// CTAs of a solve
static int twist_ctas(const Ctx& c, const Twist& t) { return c.c64() ? 2 * t.ts.NQ : 4; }

bool twist_fits(const Ctx& c) {
  Twist t;
  int GM, th;
  size_t smem;
  return twist_geometry(c, t, GM, th, smem);
}
TileStore tile_store(const Ctx& c) {
  Twist t{};
  int GM, th;
  size_t smem;
  twist_geometry(c, t, GM, th, smem);
  return t.ts;
}

using TwistKernel = void (*)(FrontArgs, Twist, const FrontArgs*, int*);
static TwistKernel twist_kernel(const Ctx& c, const Twist& t, bool fused) {
  if (t.ts.NQ == 2) return k_twist<6, kGM2, 2, false>;
  if (fused) return c.bmax <= 64 ? k_twist<4, kGMs, 1, true> : k_twist<4, kGM1, 1, true>;
  return c.bmax <= 64 ? k_twist<4, kGMs, 1, false> : k_twist<4, kGM1, 1, false>;
}
using RowsKernel = void (*)(FrontArgs, Twist, double2*, int*);
static RowsKernel rows_kernel(const Ctx& c, const Twist& t) {
  if (t.W == 3) return t.gl ? k_twist_rows<3, 8, true> : k_twist_rows<3, 8, false>;
  if (t.W == 6) return t.gl ? k_twist_rows<6, 8, true> : k_twist_rows<6, 8, false>;
  const int nc = rows_columns(c.bmax, 12);
  if (t.gl)
    return nc <= 8 ? k_twist_rows<12, 8, true> : nc <= 12 ? k_twist_rows<12, 12, true> : k_twist_rows<12, 16, true>;
  return nc <= 8 ? k_twist_rows<12, 8, false> : nc <= 12 ? k_twist_rows<12, 12, false> : k_twist_rows<12, 16, false>;
}
static const void* twist_function(const Ctx& c, const Twist& t, bool fused) {
  return c.c64() ? (const void*)twist_kernel(c, t, fused) : (const void*)rows_kernel(c, t);
}

static void twist_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at, int ctas, int count,
                         int threads, size_t smem, cudaStream_t stream, bool pdl) {
  cfg.gridDim = dim3((unsigned)(ctas * count));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)ctas;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 2 : 1;
}

// `count` solves of one level; with `table` a level of a fused application
cudaError_t launch_twist(Ctx& c, const FrontArgs& a, int count, const FrontArgs* table,
                         cudaStream_t stream) {
  Twist t;
  int GM, th;
  size_t smem;
  if (!twist_geometry(c, t, GM, th, smem) || (table && (t.ts.NQ != 1 || !c.c64())))
    return cudaErrorInvalidConfiguration;
  cudaError_t e = cudaFuncSetAttribute(twist_function(c, t, table != nullptr),
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  twist_config(cfg, at, twist_ctas(c, t), count, th, smem, stream, c.p.pdl != 0);
  if (!c.c64()) {
    if (t.gl && !c.d_lines) return cudaErrorInvalidConfiguration;
    return cudaLaunchKernelEx(&cfg, rows_kernel(c, t), a, t, (double2*)c.d_lines, c.d_status);
  }
  return cudaLaunchKernelEx(&cfg, twist_kernel(c, t, table != nullptr), a, t, table, c.d_status);
}

// line vectors of k_twist_rows in global memory, for the largest level
size_t twist_lines_bytes(const Ctx& c) {
  Twist t;
  int GM, th;
  size_t smem;
  if (c.c64() || !factor_fits_smem(c) || !twist_geometry(c, t, GM, th, smem) || !t.gl) return 0;
  return (size_t)4 * std::max(1, c.max_tasks) * t.Lh * (t.bs / 2) * sizeof(double2);
}

// lines that a fused application takes (one CTA per half)
bool twist_fused_fits(const Ctx& c) {
  return c.c64() && c.bmax <= 92 && twist_fits(c);
}

// solves of the twisted kernel the current device runs at once
int twist_concurrency(const Ctx& c) {
  Twist t;
  int GM, th, dev = 0, sms = 0, ncl = 0;
  size_t smem;
  if (!twist_geometry(c, t, GM, th, smem)) return 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
    cudaGetLastError();
    return 152 * (c.c64() ? 1 : 12 / t.W) / twist_ctas(c, t);   // no device: a 152-SM GB300
  }
  const void* kern = twist_function(c, t, false);
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) ==
      cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    twist_config(cfg, at, twist_ctas(c, t), sms, th, smem, nullptr, false);
    if (cudaOccupancyMaxActiveClusters(&ncl, kern, &cfg) != cudaSuccess) ncl = 0;
  }
  cudaGetLastError();
  return ncl > 0 ? ncl : std::max(1, sms * (c.c64() ? 1 : 12 / t.W) / twist_ctas(c, t));
}

// Geometry of k_twist_multi: the blocks beside the vectors, partial sums and compact sources
// of the K right-hand sides (the line vectors are in global memory).  Lines of up to 64 nodes:
// two groups of workers and all partial sums of a step at once; wider ones: one group, four
// right-hand sides at a time.
constexpr int kMultiER = 4;
static bool multi_geometry(const Ctx& c, int K, Twist& t, int& threads, size_t& smem) {
  int GM;
  if (!c.c64() || c.cube || c.dim != 2 || c.bmax > 92 || K < 1 || K > kMaxRHS) return false;
  if (!twist_geometry(c, t, GM, threads, smem)) return false;
  const int SP = part_stride(t.ts.T, GM), NG = GM == kGMs ? 2 : 1;
  const int KG = (K + NG - 1) / NG, NP = NG * (KG <= 1 ? 1 : KG <= 2 ? 2 : 4);
  const size_t fixed = kTwistBars * sizeof(uint64_t) +
                       ((size_t)K * (2 * t.ts.T * GM + 3 * t.bs + 2 * t.Lh) + NP * GM * SP + 8) *
                           sizeof(float2);
  const size_t limit = 227 * 1024;
  if (fixed + 2 * (size_t)t.slot_bytes > limit) return false;
  t.nslot = (int)std::min<size_t>(kSoloMaxSlots, (limit - fixed) / t.slot_bytes);
  smem = fixed + (size_t)t.nslot * t.slot_bytes;
  threads = (threads - 32) * NG + 32;
  return threads <= 320;
}

bool multi_supported(const Ctx& c, int K) {
  Twist t;
  int th;
  size_t smem;
  return c.twisted() && multi_geometry(c, K, t, th, smem);
}

// line-vector elements of one CTA for K right-hand sides
long long multi_line_stride(const Ctx& c, int K) { return (long long)c.Lmax * K * c.bmax; }

using MultiKernel = void (*)(MultiArgs, Twist, int*);
static MultiKernel multi_kernel(const Ctx& c, int K) {
  if (c.bmax <= 64)
    return K <= 2   ? k_twist_multi<4, kGMs, 2, kMultiER, 1>
           : K <= 4 ? k_twist_multi<4, kGMs, 2, kMultiER, 2>
                    : k_twist_multi<4, kGMs, 2, kMultiER, 4>;
  return K <= 1   ? k_twist_multi<4, kGM1, 1, kMultiER, 1>
         : K <= 2 ? k_twist_multi<4, kGM1, 1, kMultiER, 2>
         : K <= 4 ? k_twist_multi<4, kGM1, 1, kMultiER, 4>
                  : k_twist_multi<4, kGM1, 1, kMultiER, 8>;
}

cudaError_t launch_front_multi(Ctx& c, int li, int K, Ctx* const* rhs, const double2* const* r) {
  Twist t;
  int threads;
  size_t smem;
  if (!multi_geometry(c, K, t, threads, smem) || !c.d_mline) return cudaErrorInvalidConfiguration;
  MultiArgs m = {};
  FrontArgs& a = m.a;
  a.subs = c.d_subs;
  a.tasks = c.d_tasks;
  a.task_off = c.launches[li].off;
  a.lcoef = c.d_lcoef;
  a.cstride = c.node_elems;
  a.fac = c.d_fac;
  a.Next = c.Next;
  a.W = c.trace_W;
  a.nsub = (int)c.subs.size();
  a.q = c.q;
  a.r = c.r;
  a.pz = c.pz;
  a.dim = c.dim;
  a.Ne = c.Ne;
  a.spin = c.spin();
  for (int i = 0; i < K; ++i) {
    m.rin[i] = r[i];
    m.lane[i] = rhs[i]->d_lane;
    m.trace[i] = rhs[i]->d_trace;
  }
  m.line = c.d_mline;
  m.line_stride = multi_line_stride(c, K);
  m.K = K;
  MultiKernel kern = multi_kernel(c, K);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  twist_config(cfg, at, 2, c.launches[li].count, threads, smem, c.stream, c.p.pdl != 0);
  return cudaLaunchKernelEx(&cfg, kern, m, t, c.d_status);
}

}  // namespace lsw
