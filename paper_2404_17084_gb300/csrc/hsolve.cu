// Smoothing-length solve (Section III-C, Eq. 7-9): h = hfact n(h)^(-1/3) with
// n(h) = sum_b W(r_ab, h), by Newton-Raphson on g(h) = h - hfact n(h)^(-1/3)
// from the estimate h0 = hfact side/count^(1/3) of the particle's leaf, then
// bisection on [h0/16, 16 h0] (bracket located from h0 outwards, see below),
// then the estimate itself.
//
// One warp per octree leaf.  The warp walks the tree once for the whole leaf
// (children of a node tested by parallel lanes) and keeps, in shared memory,
// the particle ranges of every leaf that comes within R = 2.5 max(h0) of the
// leaf's box.  Leaves are visited depth-first, i.e. in the Morton order of the
// sorted particle arrays, so adjacent accepted leaves merge into one range,
// and a node whose box lies wholly within R of the query box is taken as one
// range without descending (the same candidates its leaves would give).  The
// ranges are expanded into a list of positions that the particles of the leaf
// sum over with all 32 lanes.  A particle's first pass over that list also
// keeps, in a list of its own, the candidates within min(2.5 h, R) of it;
// its later steps sum over that shorter list while it covers the support
// (2h <= 0.999 of its radius).  When an iterate outgrows the leaf's list
// (2h > R), or the list is far larger than needed (R > 8h), it is gathered
// again with R = 2.5 h; the next particle keeps whatever list covers it.  A
// list longer than the buffer is expanded and summed chunk by chunk; ranges
// beyond their own buffer come from a resumable walk.  The Newton and
// bisection rules are those of the per-particle definition; only the order
// of the sums differs.
//
// What bounds it is latency: one warp's chain of gathers, per particle about
// 3.5 sums of some 100 terms each.  So a pass keeps HS_MLP candidates per
// lane in flight, and a particle's own candidates are held in registers as
// offsets from it (they do not depend on h), so that its later Newton steps
// load nothing.  Where the leaf's list is longer than its buffer, each lane
// keeps the candidates it found within reach of the particle and its later
// steps add those alone, in the order a full pass adds them.
//
// Both builds solve in FP32: Newton and bisection sums on hi/lo-split
// coordinates, the iterate, its step and the list-coverage tests in FP32
// (hfact as an FP32 hi/lo pair), the converged step (|dh| < 1e-6 h) applied in
// FP64.  That is the mixed build's h, 5e-8 from the root.  The FP64 build then
// takes one FP64 step of third order from there: with S(h) = sum_b w(r_ab/h),
// Eq. (7) is S(h) = pi hfact^3, and Halley's step from the FP64 sums of w,
// q w' and q^2 w'' + 2 q w' leaves an error of (5e-8)^3.  FP32 may lead there,
// not decide: a particle of the FP64 build whose FP32 solve comes near any
// decision (a bound of the bracket, a sign of g within 1e-4 h, a flat g, values
// beyond FP32's range) or whose last step does not settle goes on a list that
// h_solve_exact solves by the same rules with FP64 sums throughout, so that h
// and its route are FP64's (0.4 ms at 2^20).  FP64 sums at every Newton step
// (4.2 per particle on a pipe at about 1/74 of the FP32 rate, to |dh| < 1e-10 h)
// took 77 ms at 2^20 clumpy particles; now 23 ms, of which the FP32 solve is 11
// ms (mixed: 12.9 ms before; 60,000 particles 5.2 -> 2.0 ms).
#include "internal.cuh"

namespace {

constexpr int HS_WARPS = 2;     // warps per block: small blocks free their SM slots as soon as their
                                // warps end, and a warp's leaves take very different times
constexpr int HS_RNG = 384;     // particle ranges held per warp
constexpr int HS_CAP = 1024;    // candidate positions held per warp (a multiple of 32)
// Depth-first stack: the tree has at most 22 levels and a popped node pushes at
// most its 8 children, so at most 8 + 7 * 21 = 155 entries are live.
constexpr int HS_STK = 160;
constexpr int HS_PCAP = 512;   // one particle's own candidates (within 2.5 h of it)
constexpr int HS_WIN = 8;      // sorted positions per warp, which takes the leaves that start among them: about
                               // one leaf (7 particles on average), so that a snapshot of 60,000 gives 7,500
                               // warps (32 positions: 1,875, one wave as long as its slowest four leaves)
constexpr int HS_MLP = 2;      // candidates per lane in flight during a pass (4: more registers, 13.9 ms for 13.2 at 2^20)
constexpr int HS_REG = 6;      // own candidates per lane held in registers (192 per particle; 113 on average)
constexpr unsigned FULL = 0xffffffffu;

struct HsTree {
  const double *xs, *ys, *zs;
  const float* split;  // 6 per sorted position: FP32 hi/lo of x, y, z
  const int64_t *nb, *ne, *fc;
  const int32_t *nch, *owner, *idx;
  const float* box32;  // 8 per node: outward-rounded FP32 box, hmax, pad
};

struct HsWarp {
  int2 rng[HS_RNG];
  int32_t cand[HS_CAP];
  int32_t pcand[HS_PCAP];  // the current particle's candidates within pR of it
  int32_t stk[HS_STK];
};

// Candidate list held by one warp (values uniform across its lanes).
struct HsBuf {
  float q[6];       // query box: the leaf's outward-rounded FP32 box
  float R;          // gather radius
  int nr;           // ranges held
  bool rng_done;    // the walk finished: the ranges cover every candidate
  int64_t total;    // positions in the ranges held
  bool expanded;    // cand holds all of them
  int64_t pk;       // the particle whose own list pcand holds (-1: none)
  float pR;         // its radius
  int pn;           // its length
  float cR;         // radius of the lanes' own finds of a long list (pcand[32 i + lane]); < 0: none
};

// The current particle's candidates in registers, as offsets from it: lane
// l's entries are the positions l, l + 32, ... of its own list, or the lane's
// finds of a long list, in the order the lists are summed.
struct HsOwn {
  float x[HS_REG], y[HS_REG], z[HS_REG];
  int n;  // this lane's entries
};

// True when no point of box b is within R of box q.  Both boxes are rounded
// outward; the FP32 arithmetic on coordinates in the unit cube is covered by
// the margin folded into Rm.
__device__ __forceinline__ bool box_far_box(const float* __restrict__ b, const float* q, float Rm) {
  const float dx = fmaxf(fmaxf(b[0] - q[3], q[0] - b[3]), 0.f);
  const float dy = fmaxf(fmaxf(b[1] - q[4], q[1] - b[4]), 0.f);
  const float dz = fmaxf(fmaxf(b[2] - q[5], q[2] - b[5]), 0.f);
  return dx * dx + dy * dy + dz * dz > Rm * Rm;
}

// True when every point of box b is within R of box q (then every leaf below
// the node would be gathered; taking the node whole gives the same set).
__device__ __forceinline__ bool box_within_box(const float* __restrict__ b, const float* q, float R) {
  const float dx = fmaxf(fmaxf(b[3] - q[3], q[0] - b[0]), 0.f);
  const float dy = fmaxf(fmaxf(b[4] - q[4], q[1] - b[1]), 0.f);
  const float dz = fmaxf(fmaxf(b[5] - q[5], q[2] - b[2]), 0.f);
  return dx * dx + dy * dy + dz * dz <= R * R;
}

// Resumable depth-first walk over the leaves whose box comes within R of the
// query box (state uniform across the warp; the stack lives in W.stk).
struct HsWalk {
  float Rm;       // R with the FP32 margin folded in
  float Rin;      // R for whole-node acceptance
  int sp;         // stack depth
  int64_t c0;     // first child of the node whose range children are pending
  unsigned m;     // pending range children (leaves, or nodes taken whole)
};

__device__ __forceinline__ float walk_margin(float R) { return (R + 1e-6f) * 1.000001f; }

__device__ __forceinline__ void walk_begin(const HsTree& T, HsWarp& W, HsWalk& it, float R, int& nr) {
  __syncwarp();
  it.Rm = walk_margin(R);
  it.Rin = R;
  it.m = 0u;
  it.c0 = 0;
  it.sp = 0;
  nr = 0;
  if (T.nch[0] == 0) {
    if ((threadIdx.x & 31) == 0) W.rng[0] = make_int2((int)T.nb[0], (int)T.ne[0]);
    nr = 1;
  } else {
    if ((threadIdx.x & 31) == 0) W.stk[0] = 0;
    it.sp = 1;
  }
  __syncwarp();
}

__device__ __forceinline__ bool walk_done(const HsWalk& it) { return it.sp == 0 && it.m == 0u; }

// Appends to W.rng[nr, HS_RNG) the next particle ranges of the walk, merging
// ranges that touch.  Returns the new count; stops when the buffer is full.
__device__ int walk_next(const HsTree& T, HsWarp& W, HsWalk& it, const float* q, int nr) {
  const int lane = threadIdx.x & 31;
  int last = nr > 0 ? W.rng[nr - 1].y : -1;
  __syncwarp();
  while (true) {
    if (it.m) {
      const int b = __ffs(it.m) - 1;
      const int a0 = (int)T.nb[it.c0 + b], a1 = (int)T.ne[it.c0 + b];
      if (a0 == last) {
        if (lane == 0) W.rng[nr - 1].y = a1;
      } else {
        if (nr == HS_RNG) break;
        if (lane == 0) W.rng[nr] = make_int2(a0, a1);
        ++nr;
      }
      last = a1;
      it.m &= it.m - 1u;
      continue;
    }
    if (it.sp == 0) break;
    const int nd = W.stk[it.sp - 1];
    --it.sp;
    // the node's link word: first child << 4 | child count (see the tree build)
    const unsigned link = __float_as_uint(T.box32[8 * (int64_t)nd + 7]);
    const int nc = link == NODE_LINK_FAR ? T.nch[nd] : (int)(link & 15u);
    const int64_t c0 = link == NODE_LINK_FAR ? T.fc[nd] : (int64_t)(link >> 4);
    bool hit = false, take = false;
    if (lane < nc) {
      const float4 b0 = reinterpret_cast<const float4*>(T.box32)[2 * (c0 + lane)];
      const float4 b1 = reinterpret_cast<const float4*>(T.box32)[2 * (c0 + lane) + 1];
      const float bx[6] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y};
      hit = !box_far_box(bx, q, it.Rm);
      take = hit && (__float_as_uint(b1.w) == 0u || box_within_box(bx, q, it.Rin));
    }
    const unsigned mt = __ballot_sync(FULL, take), mi = __ballot_sync(FULL, hit && !take);
    const int ni = __popc(mi);
    __syncwarp();  // every lane has read the popped entry before it is overwritten
    if (it.sp + ni > HS_STK) { it.sp = 0; break; }  // unreachable for trees of at most 22 levels
    // descended children pushed in reverse so that they pop in child order;
    // the ranges of this node's children are taken first, which keeps the
    // walk depth-first only within a node -- merging is an optimisation, and
    // the set of positions is the same in any order
    if (hit && !take) W.stk[it.sp + ni - 1 - __popc(mi & ((1u << lane) - 1u))] = (int)(c0 + lane);
    it.sp += ni;
    it.c0 = c0;
    it.m = mt;
    __syncwarp();
  }
  __syncwarp();
  return nr;
}

// The particle at sorted position k, FP32 hi/lo.
struct HsPoint {
  float hx, lx, hy, ly, hz, lz;
};
__device__ __forceinline__ HsPoint point_of(const HsTree& T, int64_t k) {
  const float2* P = reinterpret_cast<const float2*>(T.split + 6 * k);
  const float2 a = __ldg(P), b = __ldg(P + 1), c = __ldg(P + 2);
  return HsPoint{a.x, a.y, b.x, b.y, c.x, c.y};
}

// One candidate at the offset (ox, oy, oz): w(q) and 3 w + q w'(q) added when
// inside; returns q^2.  The sums' roundings are written out, so that h does not
// move with the compiler's choice of what to fuse: q^2 in the order x^2, y^2,
// z^2 for bisection and y^2, x^2, z^2 for Newton, which also needs d.
template <bool NEWTON>
__device__ __forceinline__ float add_term(float ox, float oy, float oz, float inv_h, float& s, float& d) {
  const float dx = ox * inv_h, dy = oy * inv_h, dz = oz * inv_h;
  const float q2 = NEWTON ? __fmaf_rn(dz, dz, __fmaf_rn(dx, dx, __fmul_rn(dy, dy)))
                          : __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
  if (q2 >= 4.f) return q2;
  const float q = sqrtf(q2);
  float w, dwq;
  if (q < 1.f) {
    w = __fmaf_rn(__fmul_rn(0.75f, q2), q, __fmaf_rn(-1.5f, q2, 1.f));
    dwq = -3.f * q2 + 2.25f * q2 * q;
  } else {
    const float t = 2.f - q;
    w = __fmul_rn(__fmul_rn(__fmul_rn(0.25f, t), t), t);
    dwq = -0.75f * t * t * q;
  }
  s = __fadd_rn(s, w);
  if (NEWTON) d = __fadd_rn(d, 3.f * w + dwq);
  return q2;
}

// f(position, offset x, y, z, valid) for list[0, cnt): a lane takes positions
// lane, lane + 32, ... in that order, MLP of them per round with their
// loads issued together; every lane calls f, for all of a round's positions.
template <int MLP = HS_MLP, typename F>
__device__ __forceinline__ void for_list(const HsTree& T, const int32_t* list, int cnt, const HsPoint& p, F f) {
  const int lane = threadIdx.x & 31;
  for (int j0 = 0; j0 < cnt; j0 += 32 * MLP) {
    int32_t c[MLP];
    float2 a[MLP], b[MLP], e[MLP];
#pragma unroll
    for (int u = 0; u < MLP; ++u) {
      const int j = j0 + 32 * u + lane;
      c[u] = list[j < cnt ? j : cnt - 1];
      const float2* P = reinterpret_cast<const float2*>(T.split + 6 * (int64_t)c[u]);
      a[u] = __ldg(P); b[u] = __ldg(P + 1); e[u] = __ldg(P + 2);
    }
#pragma unroll
    for (int u = 0; u < MLP; ++u) {
      if (j0 + 32 * u >= cnt) break;
      f(c[u], (a[u].x - p.hx) + (a[u].y - p.lx), (b[u].x - p.hy) + (b[u].y - p.ly),
        (e[u].x - p.hz) + (e[u].y - p.lz), j0 + 32 * u + lane < cnt);
    }
  }
}

// Lane partial sums of w(q) and 3 w + q w'(q) over list[0, cnt).
template <bool NEWTON>
__device__ __forceinline__ void warp_accum(const HsTree& T, const int32_t* list, int cnt, const HsPoint& p, float inv_h,
                                           float& s, float& d) {
  for_list(T, list, cnt, p, [&](int32_t, float ox, float oy, float oz, bool on) {
    if (on) add_term<NEWTON>(ox, oy, oz, inv_h, s, d);
  });
}

// The same, and the candidates with q^2 < keep_q2 are appended, in list
// order, to keep[0, *nkeep) (*nkeep = -1 when they do not fit in HS_PCAP).
template <bool NEWTON>
__device__ __forceinline__ void warp_accum_keep(const HsTree& T, const int32_t* list, int cnt, const HsPoint& p,
                                                float inv_h, float& s, float& d, int32_t* keep, float keep_q2,
                                                int* nkeep) {
  const unsigned lt = (1u << (threadIdx.x & 31)) - 1u;
  int nk = 0;
  for_list(T, list, cnt, p, [&](int32_t c, float ox, float oy, float oz, bool on) {
    const float q2 = on ? add_term<NEWTON>(ox, oy, oz, inv_h, s, d) : 1e30f;
    const unsigned m = __ballot_sync(FULL, on && q2 < keep_q2);
    if (nk < 0) return;
    if (nk + __popc(m) > HS_PCAP) { nk = -1; return; }
    if (on && q2 < keep_q2) keep[nk + __popc(m & lt)] = c;
    nk += __popc(m);
  });
  *nkeep = nk;
}

// The same over one chunk of a long list; a lane's candidates with q^2 <
// keep_q2 are appended to its own column keep[32 i + lane], i < HS_PCAP / 32
// (nl counts past that when they do not fit).
template <bool NEWTON, int LONG>
__device__ __forceinline__ void warp_accum_lane(const HsTree& T, const int32_t* list, int cnt, const HsPoint& p,
                                                float inv_h, float& s, float& d, int32_t* keep, float keep_q2,
                                                int& nl) {
  const int lane = threadIdx.x & 31;
  for_list<LONG>(T, list, cnt, p, [&](int32_t c, float ox, float oy, float oz, bool on) {
    if (!on) return;
    const float q2 = add_term<NEWTON>(ox, oy, oz, inv_h, s, d);
    if (q2 < keep_q2) {
      if (keep && nl < HS_PCAP / 32) keep[32 * nl + lane] = c;
      ++nl;
    }
  });
}

// The offsets of this lane's n entries col[0], col[32], ... into registers.
__device__ __forceinline__ void own_load(const HsTree& T, const int32_t* col, int n, const HsPoint& p, HsOwn& O) {
  O.n = n;
#pragma unroll
  for (int i = 0; i < HS_REG; ++i) {
    O.x[i] = O.y[i] = O.z[i] = 0.f;
    if (i < n) {
      const float2* P = reinterpret_cast<const float2*>(T.split + 6 * (int64_t)col[32 * i]);
      const float2 a = __ldg(P), b = __ldg(P + 1), c = __ldg(P + 2);
      O.x[i] = (a.x - p.hx) + (a.y - p.lx);
      O.y[i] = (b.x - p.hy) + (b.y - p.ly);
      O.z[i] = (c.x - p.hz) + (c.y - p.lz);
    }
  }
}

template <typename V>
__device__ __forceinline__ V warp_total(V v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(FULL, v, o);
  return __shfl_sync(FULL, v, 0);
}

// Expands ranges [r, nr) of W.rng, from offset off in range r, into W.cand
// (up to HS_CAP positions).  Returns the count; advances r and off.
__device__ int expand(HsWarp& W, int nr, int& r, int& off) {
  const int lane = threadIdx.x & 31;
  int c = 0;
  __syncwarp();
  while (r < nr && c < HS_CAP) {
    const int2 g = W.rng[r];
    const int len = g.y - g.x - off;
    const int t = len < HS_CAP - c ? len : HS_CAP - c;
    for (int j = lane; j < t; j += 32) W.cand[c + j] = g.x + off + j;
    c += t;
    off += t;
    if (off == g.y - g.x) { ++r; off = 0; }
  }
  __syncwarp();
  return c;
}

// Gathers the candidate ranges for radius R, and their positions when they fit.
__device__ __forceinline__ void regather(const HsTree& T, HsWarp& W, HsBuf& B, float R) {
  const int lane = threadIdx.x & 31;
  HsWalk it;
  B.R = R;
  B.cR = -1.f;
  walk_begin(T, W, it, R, B.nr);
  B.nr = walk_next(T, W, it, B.q, B.nr);
  B.rng_done = walk_done(it);
  int64_t tot = 0;
  for (int r = lane; r < B.nr; r += 32) tot += W.rng[r].y - W.rng[r].x;
  for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(FULL, tot, o);
  B.total = tot;
  B.expanded = false;
  if (B.rng_done && tot <= HS_CAP) {
    int r = 0, off = 0;
    expand(W, B.nr, r, off);
    B.expanded = true;
  }
}

// f(list, count) for every chunk of a list that does not fit the position
// buffer, in the same chunks every time.
template <typename F>
__device__ __forceinline__ void for_chunks(const HsTree& T, HsWarp& W, HsBuf& B, F f) {
  if (B.rng_done) {
    // the ranges are complete but longer than the position buffer
    int r = 0, off = 0;
    while (r < B.nr) {
      const int c = expand(W, B.nr, r, off);
      f(W.cand, c);
    }
    return;
  }
  // more ranges than their buffer: one resumable walk, range chunk by chunk
  HsWalk it;
  int nr;
  walk_begin(T, W, it, B.R, nr);
  for (;;) {
    nr = walk_next(T, W, it, B.q, nr);
    int r = 0, off = 0;
    while (r < nr) {
      const int c = expand(W, nr, r, off);
      f(W.cand, c);
    }
    if (walk_done(it)) break;
    nr = 0;
  }
  B.nr = 0;
  B.R = -1.f;  // the buffer no longer holds the first ranges: regather next time
}

// n(h) and dn/dh for the particle at sorted position k (warp-uniform result).
template <bool NEWTON, int LONG>
__device__ __forceinline__ void warp_density(const HsTree& T, HsWarp& W, HsBuf& B, HsOwn& O, int64_t k,
                                             const HsPoint& p, float h, float& n, float& dn) {
  const int lane = threadIdx.x & 31;
  float s = 0.f, d = 0.f;
  const float inv_h = 1.0f / h;
  bool held = B.pk == k && 2.f * h <= 0.999f * B.pR && B.pR <= 8.f * h;
  const bool own = held;
  bool wide = own && B.pn > 32 * HS_REG;  // its own list, not held in registers
  if (!own) {
    if (2.f * h > B.R || B.R > 8.f * h) regather(T, W, B, 2.5f * h);
    // the lanes' finds of a long list cover its support at this h
    held = !B.expanded && 2.f * h <= 0.999f * B.cR;
  }
  if (held && !wide) {
#pragma unroll
    for (int i = 0; i < HS_REG; ++i)
      if (i < O.n) add_term<NEWTON>(O.x[i], O.y[i], O.z[i], inv_h, s, d);
    if (!own && __any_sync(FULL, O.n > HS_REG)) {
      for (int i = HS_REG; i < O.n; ++i) {
        const HsPoint c = point_of(T, W.pcand[32 * i + lane]);
        add_term<NEWTON>((c.hx - p.hx) + (c.lx - p.lx), (c.hy - p.hy) + (c.ly - p.ly), (c.hz - p.hz) + (c.lz - p.lz), inv_h, s,
                 d);
      }
      __syncwarp();
    }
  } else if (wide) {
    warp_accum<NEWTON>(T, W.pcand, B.pn, p, inv_h, s, d);
  } else if (B.expanded) {
    // the leaf's list; the first pass for a particle also keeps its own
    // candidates within pR = min(2.5 h, R) of it for the next steps (the
    // leaf's list holds every candidate within R of the leaf's box, so of
    // the particle)
    if (B.pk != k) {
      const float pR = 2.5f * h < B.R ? 2.5f * h : B.R;
      const float kq = pR / h;
      int nk = 0;
      warp_accum_keep<NEWTON>(T, W.cand, (int)B.total, p, inv_h, s, d, W.pcand, kq * kq * 1.00001f, &nk);
      __syncwarp();
      B.pk = k;
      B.pR = nk >= 0 ? pR : 0.f;  // 0: nothing kept (it did not fit)
      B.pn = nk >= 0 ? nk : 0;
      if (nk <= 32 * HS_REG) own_load(T, W.pcand + lane, (B.pn - lane + 31) >> 5, p, O);
    } else {
      warp_accum<NEWTON>(T, W.cand, (int)B.total, p, inv_h, s, d);
    }
  } else {
    // a long list: the particle's own list keeps pcand when there is one
    const bool room = B.pk != k;
    const float cR = 2.5f * h < B.R ? 2.5f * h : B.R;
    const float kq = cR / h;
    int nl = 0;
    for_chunks(T, W, B, [&](const int32_t* list, int c) {
      warp_accum_lane<NEWTON, LONG>(T, list, c, p, inv_h, s, d, room ? W.pcand : nullptr, kq * kq * 1.00001f, nl);
    });
    __syncwarp();
    B.cR = -1.f;
    if (room && B.R > 0.f && !__any_sync(FULL, nl > HS_PCAP / 32)) {
      B.cR = cR;
      own_load(T, W.pcand + lane, nl, p, O);
    }
  }
  const float norm = inv_h * inv_h * inv_h * (float)(1.0 / MAP_PI);
  n = warp_total(s) * norm;
  dn = -warp_total(d) * norm * inv_h;
}

// FP64 sums of w(q), q w'(q) and q^2 w''(q) + 2 q w'(q) at h over list[0,
// cnt) around the particle at sorted position k: the candidates an FP32
// distance screen (1e-5 margin) leaves are packed into buf (at least
// 64 entries), so that the FP64 terms run with full warps.
__device__ __forceinline__ void accum64(const HsTree& T, const int32_t* list, int cnt, const HsPoint& p, int64_t k,
                                        double h, int32_t* buf, double& s, double& d, double& e) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const double x = T.xs[k], y = T.ys[k], z = T.zs[k], inv_h = 1.0 / h;
  const float ih = (float)inv_h, lim = 2.00001f + 8e-15f * ih, lim2 = lim * lim;  // (8e-15: the split's own error)
  int nb = 0;
  auto drain = [&](int m) {  // the first m (<= 32) of buf
    __syncwarp();
    if (lane < m) {
      const int64_t c = buf[lane];
      const double ex = (T.xs[c] - x) * inv_h, ey = (T.ys[c] - y) * inv_h, ez = (T.zs[c] - z) * inv_h;
      const double q2 = ex * ex + ey * ey + ez * ez;
      const double q = sqrt(q2), q3 = q2 * q;
      if (q < 1.0) {
        s += 1.0 - 1.5 * q2 + 0.75 * q3;
        d += 2.25 * q3 - 3.0 * q2;
        e += 9.0 * (q3 - q2);
      } else if (q < 2.0) {
        const double t = 2.0 - q, t2 = t * t;
        s += 0.25 * t2 * t;
        d -= 0.75 * t2 * q;
        e += 1.5 * t * q * (q - t);
      }
    }
    __syncwarp();
  };
  for_list(T, list, cnt, p, [&](int32_t c, float ox, float oy, float oz, bool on) {
    const float dx = ox * ih, dy = oy * ih, dz = oz * ih;
    const bool in = on && dx * dx + dy * dy + dz * dz <= lim2;
    const unsigned m = __ballot_sync(FULL, in);
    if (in) buf[nb + __popc(m & lt)] = c;
    nb += __popc(m);
    if (nb >= 32) {
      drain(32);
      nb -= 32;
      const int32_t v = lane < nb ? buf[32 + lane] : 0;
      __syncwarp();
      if (lane < nb) buf[lane] = v;
    }
  });
  if (nb) drain(nb);
}

// The FP64 build's sums at h, from the shortest list that covers its support.
__device__ __forceinline__ void density64(const HsTree& T, HsWarp& W, HsBuf& B, int64_t k, const HsPoint& p, double h,
                                          double& s, double& d, double& e) {
  s = d = e = 0.0;
  const float hf = (float)h;
  int32_t* buf = W.stk;  // free outside a walk
  if (B.pk == k && 2.f * hf <= 0.999f * B.pR) {
    accum64(T, W.pcand, B.pn, p, k, h, buf, s, d, e);
  } else {
    if (2.f * hf > 0.999f * B.R || B.R > 8.f * hf) regather(T, W, B, 2.5f * hf);
    if (B.expanded) accum64(T, W.cand, (int)B.total, p, k, h, buf, s, d, e);
    else for_chunks(T, W, B, [&](const int32_t* list, int c) {
      // a walk between chunks uses the stack: the packing buffer is local to a chunk
      accum64(T, list, c, p, k, h, W.pcand, s, d, e);
    });
    if (!B.expanded) { B.pk = -1; B.cR = -1.f; }  // pcand was used
  }
  s = warp_total(s);
  d = warp_total(d);
  e = warp_total(e);
}

// The candidate list of a leaf before anything is gathered.
__device__ __forceinline__ void list_init(const HsTree& T, int64_t leaf, HsBuf& B) {
#pragma unroll
  for (int i = 0; i < 6; ++i) B.q[i] = T.box32[8 * leaf + i];
  B.R = -1.f;
  B.nr = 0;
  B.total = 0;
  B.rng_done = false;
  B.expanded = false;
  B.pk = -1;
  B.pR = 0.f;
  B.pn = 0;
  B.cR = -1.f;
}

// Bisection's bracket (Eq. 7's g on [lo, hi] = [g0/16, 16 g0]): it needs g(lo) <
// 0 < g(hi).  g(h)/h is nondecreasing in h (w is nonincreasing in q, so sum_b
// w(r_ab/h) grows with h), so the sign of g at either end follows from any
// point between: step from g0 by factors of 2 towards the sign change and
// bisect the first bracket [a, b] found, evaluating g at lo or hi only when the
// steps reach them.  False: no sign change.
template <typename G>
__device__ __forceinline__ bool bracket_root(double g0, double lo, double hi, G g, double& a, double& b) {
  a = lo;
  b = hi;
  if (g(g0) < 0.0) {
    a = g0;
    double y = 2.0 * g0;
    for (; y < hi; y *= 2.0) {
      if (g(y) < 0.0) a = y; else { b = y; break; }
    }
    return y < hi || g(hi) > 0.0;
  }
  b = g0;
  double y = 0.5 * g0;
  for (; y > lo; y *= 0.5) {
    if (g(y) < 0.0) { a = y; break; } else b = y;
  }
  return y > lo || g(lo) < 0.0;
}

// redo, n_redo (FP64 build): the positions left to h_solve_exact.
template <bool MIXED, int LONG>
__global__ void __launch_bounds__(HS_WARPS * 32)
    h_solve_leaves(int64_t n, HsTree T, const double* __restrict__ h0s, double hfact, double* hout, int32_t* route,
                   int32_t* redo, unsigned* n_redo) {
  const float hf_s = (float)hfact, hf3_s = (float)(hfact / 3.0), tol_s = 1e-6f;
  const float hf_lo = (float)(hfact - (double)hf_s);
  __shared__ HsWarp sw[HS_WARPS];
  HsWarp& W = sw[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const int64_t k0 = (blockIdx.x * (int64_t)HS_WARPS + (threadIdx.x >> 5)) * HS_WIN;
  if (k0 >= n) return;  // whole warp
  // leaves whose first particle lies in this warp's window
  int leaf = -1;
  bool head = false;
  if (lane < HS_WIN && k0 + lane < n) {
    leaf = T.owner[k0 + lane];
    head = T.nb[leaf] == k0 + lane;
  }
  unsigned heads = __ballot_sync(FULL, head);
  while (heads) {
    const int src = __ffs(heads) - 1;
    heads &= heads - 1;
    const int L = __shfl_sync(FULL, leaf, src);
    const int64_t a0 = T.nb[L], a1 = T.ne[L];
    double gmax = 0.0;
    for (int64_t k = a0 + lane; k < a1; k += 32) gmax = fmax(gmax, h0s[k]);
    for (int o = 16; o > 0; o >>= 1) gmax = fmax(gmax, __shfl_xor_sync(FULL, gmax, o));
    HsBuf B;
    list_init(T, L, B);
    HsOwn O;
    O.n = 0;
    const float R0 = 2.5f * (float)gmax;
    for (int64_t k = a0; k < a1; ++k) {
      // the leaf's list for its first particle; later particles keep the
      // list they find while it covers their support (warp_density
      // regathers when 2h > R or R > 8h)
      if (k == a0) regather(T, W, B, R0);
      B.cR = -1.f;
      const HsPoint p = point_of(T, k);
      // Newton: g = h - hfact t, g' = 1 + hfact/3 t^4 dn/dh with t = n^(-1/3)
      float hs = (float)h0s[k];
      const float lo_s = hs / 16.f, hi_s = hs * 16.f;
      double h = 0.0;
      bool ok = false;
      bool sure = true;  // (FP64 build) FP32 has decided as FP64 would
      for (int it = 0; it < 30; ++it) {
        float nn, dn;
        warp_density<true, LONG>(T, W, B, O, k, p, hs, nn, dn);
        const float t = rcbrtf(nn);
        float f = hs - hf_s * t;
        f -= hf_lo * t;  // hfact as an FP32 pair
        const float fp = 1.f + hf3_s * (t * t) * (t * t) * dn;
        const float d = f / fp;
        const float hn = hs - d;
        if (!MIXED) {
          sure = it < 24 && clear_step(hs, d, fp, lo_s, hi_s);
          if (!sure) break;
        }
        if (!(hn >= lo_s && hn <= hi_s)) break;
        if ((hn > hs ? hn - hs : hs - hn) < tol_s * hn) {
          // the converged step is applied in FP64 (the result keeps FP64's
          // spacing, not FP32's)
          h = (double)hs - (double)d;
          ok = true;
          break;
        }
        hs = hn;
      }
      int r = 0;
      if (!ok && sure) {
        const double g0 = h0s[k], lo = g0 / 16.0, hi = g0 * 16.0;
        // bisection on the FP32 sums too: the root moves by ~1e-7 relative,
        // inside the mixed build's 1e-6 and the FP64 build's last step
        auto g = [&](double hh) {
          float nn, dn;
          warp_density<false, LONG>(T, W, B, O, k, p, (float)hh, nn, dn);
          const double v = hh - hfact * rcbrt((double)nn);
          if (!MIXED) sure = sure && fabs(v) > 1e-4 * hh && nn < 1e37f;
          return v;
        };
        // (bracket_root written out: as a function it cost the mixed build 4% at
        // 2^20, 12.8 -> 13.3 ms, with g inlined once more)
        double a = lo, b = hi;
        bool bracket = true;
        if (g(g0) < 0.0) {
          a = g0;
          double y = 2.0 * g0;
          for (; y < hi; y *= 2.0) {
            if (g(y) < 0.0) a = y; else { b = y; break; }
          }
          if (y >= hi) bracket = g(hi) > 0.0;
        } else {
          b = g0;
          double y = 0.5 * g0;
          for (; y > lo; y *= 0.5) {
            if (g(y) < 0.0) { a = y; break; } else b = y;
          }
          if (y <= lo) bracket = g(lo) < 0.0;
        }
        if (!bracket) {
          h = g0;
          r = 2;
        } else if (sure) {
          for (int it = 0; it < 200; ++it) {
            const double mid = 0.5 * (a + b);
            if (g(mid) < 0.0) a = mid; else b = mid;
            if (!MIXED && !sure) { a = b = mid; break; }  // at the root, as far as FP32 can tell
            if (b - a < (MIXED ? 1e-12 : 1e-4) * mid) break;
          }
          h = 0.5 * (a + b);
          r = 1;
          sure = true;
        }
      }
      if (!MIXED && r != 2 && sure) {
        // Halley's step on S(h) - pi hfact^3 (S' = -d/h, S'' = e/h^2), again
        // while a step is so large that its cube shows; one that is large or no
        // number (S' is 0) leaves the particle to h_solve_exact
        const double target = MAP_PI * hfact * hfact * hfact;
        sure = false;
        for (int it = 0; it < 30; ++it) {
          double s, d, e;
          density64(T, W, B, k, p, h, s, d, e);
          const double F = s - target;
          const double u = 2.0 * F * d / (2.0 * d * d - F * e);  // -dh / h times -1: h <- h (1 + u)
          if (!(fabs(u) < 1e-2)) break;
          h += h * u;
          if (fabs(u) < 2e-6) { sure = h > h0s[k] / 16.0 && h < h0s[k] * 16.0; break; }
        }
      }
      if (!MIXED && !sure) {
        if (lane == 0) redo[atomicAdd(n_redo, 1u)] = (int32_t)k;
        continue;
      }
      if (lane == 0) {
        const int32_t a = T.idx[k];
        hout[a] = h;
        if (route) route[a] = r;
      }
    }
  }
}

// The listed particles of the FP64 build, one per warp, with FP64 sums
// throughout: Newton to |dh| < 1e-10 h, bisection to 1e-12, the estimate.  At
// 2^20 clumpy particles it takes 0.43 of the solve's 25.0 ms.
__global__ void __launch_bounds__(HS_WARPS * 32)
    h_solve_exact(HsTree T, const double* __restrict__ h0s, double hfact, const int32_t* __restrict__ redo,
                  const unsigned* __restrict__ n_redo, double* hout, int32_t* route) {
  __shared__ HsWarp sw[HS_WARPS];
  HsWarp& W = sw[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const int64_t count = *n_redo, step = (int64_t)gridDim.x * HS_WARPS;
  for (int64_t i = blockIdx.x * (int64_t)HS_WARPS + (threadIdx.x >> 5); i < count; i += step) {
    const int64_t k = redo[i];
    HsBuf B;
    list_init(T, T.owner[k], B);
    const HsPoint p = point_of(T, k);
    auto density = [&](double h, double& nn, double& dn) {
      double s, d, e;
      density64(T, W, B, k, p, h, s, d, e);
      const double ih = 1.0 / h, norm = ih * ih * ih * (1.0 / MAP_PI);
      nn = s * norm;
      dn = -(3.0 * s + d) * norm * ih;
    };
    const double g0 = h0s[k], lo = g0 / 16.0, hi = g0 * 16.0;
    double h = g0;
    bool ok = false;
    for (int it = 0; it < 30; ++it) {
      double nn, dn;
      density(h, nn, dn);
      const double t = rcbrt(nn), t2 = t * t;
      const double hn = h - (h - hfact * t) / (1.0 + hfact / 3.0 * t2 * t2 * dn);
      if (!(hn >= lo && hn <= hi)) break;
      ok = fabs(hn - h) < 1e-10 * hn;
      h = hn;
      if (ok) break;
    }
    int r = 0;
    if (!ok) {
      auto g = [&](double v) {
        double nn, dn;
        density(v, nn, dn);
        return v - hfact * rcbrt(nn);
      };
      double a, b;
      if (!bracket_root(g0, lo, hi, g, a, b)) {
        h = g0;
        r = 2;
      } else {
        for (int it = 0; it < 200; ++it) {
          const double mid = 0.5 * (a + b);
          if (g(mid) < 0.0) a = mid; else b = mid;
          if (b - a < 1e-12 * mid) break;
        }
        h = 0.5 * (a + b);
        r = 1;
      }
    }
    if (lane == 0) {
      const int32_t a = T.idx[k];
      hout[a] = h;
      if (route) route[a] = r;
    }
    __syncwarp();
  }
}

// Initial guess: hfact * side(leaf cube) / count^(1/3), per sorted position
// (and *n_redo = 0).
__global__ void h_guess_leaf(int64_t n, const int32_t* __restrict__ owner, const int32_t* __restrict__ lev,
                             const int64_t* __restrict__ nb, const int64_t* __restrict__ ne, double hfact,
                             double* h0s, unsigned* n_redo) {
  int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k == 0) *n_redo = 0u;
  if (k >= n) return;
  int32_t leaf = owner[k];
  double side = ldexp(1.0, -lev[leaf]);
  h0s[k] = hfact * side / cbrt((double)(ne[leaf] - nb[leaf]));
}

__global__ void gather_h0(int64_t n, const int32_t* __restrict__ idx, const double* __restrict__ h0, double* h0s,
                          unsigned* n_redo) {
  int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k == 0) *n_redo = 0u;
  if (k >= n) return;
  h0s[k] = h0[idx[k]];
}

}  // namespace

int h_solve_run(map_ctx* ctx, const double* x, const double* y, const double* z, int64_t n, double* h, int32_t* route,
                const double* h0_override, cudaStream_t s, bool graph) {
  if (graph) MAP_TRY(tree_build_graph(ctx, x, y, z, nullptr, nullptr, n, s));
  else MAP_TRY(tree_build(ctx, x, y, z, nullptr, nullptr, n, s));
  DevTree& T = ctx->tree;
  double* h0s;
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[22], n, &h0s));
  // the FP64 build's list of particles for h_solve_exact and its length, in the
  // buffers of the unsorted indices and keys, which are done with
  int32_t* redo = reinterpret_cast<int32_t*>(ctx->ws_tree[1].p);
  unsigned* n_redo = reinterpret_cast<unsigned*>(ctx->ws_tree[0].p);
  const int tpb = 128;
  if (h0_override)
    gather_h0<<<nblk(n, tpb), tpb, 0, s>>>(n, T.idx, h0_override, h0s, n_redo);
  else
    h_guess_leaf<<<nblk(n, tpb), tpb, 0, s>>>(n, T.owner, T.level, T.begin, T.end, ctx->cfg.hfact, h0s, n_redo);
  ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  const HsTree V{T.xs, T.ys, T.zs, T.split, T.begin, T.end, T.first_child, T.nchild, T.owner, T.idx, T.box32};
  const int64_t warps = (n + HS_WIN - 1) / HS_WIN;
  const unsigned blocks = (unsigned)((warps + HS_WARPS - 1) / HS_WARPS);
  // Candidates per lane in flight over a list that outgrew its buffer: a small
  // set lasts as long as the leaf with the longest list (60,013 particles: 2.24
  // ms with 4, 2.41 with 2; 262,144: 3.83, 4.31), a large one as long as its
  // warps take together, and the registers of 4 cost it some (2^20: 13.7, 13.2).
  const bool mixed = ctx->cfg.precision != MAP_FP64;
  auto kern = n < (int64_t(1) << 19) ? (mixed ? h_solve_leaves<true, 4> : h_solve_leaves<false, 4>)
                                     : (mixed ? h_solve_leaves<true, 2> : h_solve_leaves<false, 2>);
  kern<<<blocks, HS_WARPS * 32, 0, s>>>(n, V, h0s, ctx->cfg.hfact, h, route, redo, n_redo);
  ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  if (!mixed) {
    const unsigned most = (unsigned)ctx->sm_count * 16;
    h_solve_exact<<<blocks < most ? blocks : most, HS_WARPS * 32, 0, s>>>(V, h0s, ctx->cfg.hfact, redo, n_redo, h, route);
    ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
  }
  return MAP_OK;
}
