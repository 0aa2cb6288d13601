// Pair-list build: for every cell i, the particles a whose support may reach
// the cell.  The rule (the paper is silent; fixed so that lists are
// reproducible bit for bit) is
//     |r_a - s_i| < 2 h_a + R_i   and   n_f.r_a - d_f < 2 h_a for every face f,
// in FP64 with a fixed operation order and no FMA contraction
// (__dmul_rn/__dadd_rn/__dsqrt_rn).  Candidates come from a traversal of the
// particle octree pruned by node bounding box and largest h; lists are sorted
// by particle index within each cell.
#include <cub/cub.cuh>

#include "internal.cuh"
#include "wedge.cuh"

namespace {

struct PairTree {
  const double *xs, *ys, *zs, *hs;
  const float* hs32;   // h in FP32 (the screen)
  const float* split;  // 6 per sorted position: FP32 hi/lo of x, y, z
  const int32_t* idx;
  const int64_t *nb, *ne, *fc;
  const int32_t* nch;
  const float* box32;  // outward-rounded FP32 boxes and largest h (8 floats per node)
};

struct PairGrid {
  const int64_t* cfo;
  const double4_32a* plane;  // absolute planes (the exact FP64 rule)
  const float4* face32;      // site-relative planes (n, d - n.s) in FP32 (screening)
  const double* site;
  const double* rad;
  const float* rin;  // inscribed radius: smallest site-to-face-plane distance, rounded down
};

// The exact rule, FP64, fixed order, no FMA contraction.
__device__ __forceinline__ bool exact_dist(double sx, double sy, double sz, double R, double x, double y, double z,
                                           double h) {
  const double dx = __dsub_rn(x, sx), dy = __dsub_rn(y, sy), dz = __dsub_rn(z, sz);
  const double dist = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)));
  return dist < __dadd_rn(__dmul_rn(2.0, h), R);
}
__device__ __forceinline__ bool exact_face(const double4_32a P, double x, double y, double z, double h) {
  const double s = __dsub_rn(__dadd_rn(__dadd_rn(__dmul_rn(P.x, x), __dmul_rn(P.y, y)), __dmul_rn(P.z, z)), P.w);
  return s < __dmul_rn(2.0, h);
}

// The pair rule, decided in FP32 wherever the FP32 value is farther from the
// threshold than a rigorous bound on its rounding error, and by the exact
// FP64 rule otherwise -- so the outcome is always the FP64 rule's.  The FP32
// separation comes from the hi/lo split of both points,
// (hi_a - hi_s) + (lo_a - lo_s), within a few ulp of the separation itself;
// with the rounding of h, R and the squares, all FP32 roundings together stay
// below 1e-6 of the magnitudes involved, and the margin is 1e-5.  No FP64
// operation runs unless a value falls inside the margin.
struct SiteSplit {
  float hx, lx, hy, ly, hz, lz, R, rin;
};

// The screens on the distance: outside (0), listed (1), or undecided (2).
__device__ __forceinline__ int dist_screen(float d2, float reach2, float tin2) {
  if (d2 > reach2 * 1.00001f) return 0;
  // every face test passes when the particle lies within 2h + r_in of the
  // site: each face plane is at least r_in from the site, so
  // n.r - d = n.(r - s) - (d - n.s) <= |r - s| - r_in < 2h for every face (the
  // 1e-4 relative margin covers the FP32 rounding many times over)
  return d2 < fminf(reach2 * 0.99999f, tin2 * 0.9999f) ? 1 : 2;
}

// The rule for sorted position k; face(i) gives the cell's face record i of
// nf (site-relative, FP32).
template <typename F>
__device__ __forceinline__ bool pair_rule(const PairGrid& G, const PairTree& T, int64_t c, int64_t f0, int nf,
                                          const SiteSplit& S, int64_t k, F face) {
  const float2* P = reinterpret_cast<const float2*>(T.split + 6 * k);
  const float2 px = __ldg(P), py = __ldg(P + 1), pz = __ldg(P + 2);
  const float fx = (px.x - S.hx) + (px.y - S.lx);
  const float fy = (py.x - S.hy) + (py.y - S.ly);
  const float fz = (pz.x - S.hz) + (pz.y - S.lz);
  const float hf = __ldg(T.hs32 + k), thr = 2.f * hf;
  const float reach = thr + S.R, tin = thr + S.rin;
  const float reach2 = reach * reach;
  const float d2 = fx * fx + fy * fy + fz * fz;
  const int d = dist_screen(d2, reach2, tin * tin);
  if (d < 2) return d == 1;
  if (!(d2 < reach2 * 0.99999f) &&
      !exact_dist(G.site[3 * c], G.site[3 * c + 1], G.site[3 * c + 2], G.rad[c], T.xs[k], T.ys[k], T.zs[k], T.hs[k]))
    return false;
  // the largest n.r - d over the faces, four at a time with their loads issued
  // together (a chunk past the last face repeats it); |d - n.s| <= R for every
  // face, so one margin covers them all
  float smax = -INFINITY;
  for (int f = 0; f < nf; f += 4) {
    float4 Q[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) Q[i] = face(f + i < nf ? f + i : nf - 1);
#pragma unroll
    for (int i = 0; i < 4; ++i) smax = fmaxf(smax, fmaf(Q[i].x, fx, fmaf(Q[i].y, fy, fmaf(Q[i].z, fz, -Q[i].w))));
  }
  const float marg = 1e-5f * (fabsf(fx) + fabsf(fy) + fabsf(fz) + S.R + thr) + 1e-30f;
  if (smax > thr + marg) return false;
  if (smax >= thr - marg)
    for (int f = 0; f < nf; ++f)
      if (!exact_face(G.plane[f0 + f], T.xs[k], T.ys[k], T.zs[k], T.hs[k])) return false;
  return true;
}
__device__ __forceinline__ bool pair_rule(const PairGrid& G, const PairTree& T, int64_t c, const SiteSplit& S,
                                          int64_t k) {
  const int64_t f0 = G.cfo[c];
  return pair_rule(G, T, c, f0, (int)(G.cfo[c + 1] - f0), S, k, [&](int i) { return __ldg(G.face32 + f0 + i); });
}

__device__ __forceinline__ SiteSplit site_split(const PairGrid& G, int64_t c) {
  const double sx = G.site[3 * c], sy = G.site[3 * c + 1], sz = G.site[3 * c + 2];
  SiteSplit S;
  S.hx = (float)sx; S.lx = (float)(sx - (double)S.hx);
  S.hy = (float)sy; S.ly = (float)(sy - (double)S.hy);
  S.hz = (float)sz; S.lz = (float)(sz - (double)S.hz);
  S.R = (float)G.rad[c];
  S.rin = G.rin[c];
  return S;
}

// One warp walks the octree for 32 cells that are consecutive in Morton order
// of their sites (so close together), one cell per lane, depth-first, so that
// the candidates come in sorted (Morton) order and each cell's list with them.
//
// Nodes: the lanes test a popped node's children side by side against the
// box around the 32 sites; a child that survives is kept when any lane's own
// cell can reach it (FP32, outward-rounded box, 1e-6 absolute margin:
// 2 * largest h + cell radius).  Leaf children go on the stack as their
// particle range, read with the box, so that nothing is loaded at the pop.
//
// Particles: the kept leaves' particles are staged 32 at a time in shared
// memory (one load round for 32 candidates).  Every lane holds its cell in
// registers and classifies all 32 against it by the distance alone: outside,
// listed for certain (within 2h + r_in of the site), or undecided.
//
// WALK_ROWS: both kinds go to the cell's row in HBM as sorted positions, the
// undecided ones (half of them) marked; row_filter then settles those with
// one warp per cell.  A row holds PAIR_ROW entries; a longer one goes on in
// chunks of a pool (1% of the clumpy cells; the pool holds two chunks per cell
// of a small grid, 1/32 per cell beyond 2048), and a cell that finds the pool
// empty is put on the list `again`.
// WALK_COUNT / WALK_FILL: for the cells of that list, the rule is settled here
// (the undecided tests of the warp compacted over its lanes) and the pairs
// counted, or written at off[c].
//
// What bounds it: the chain of one warp, about 1000 candidates classified at
// 20 instructions for 32 cells.  At 2^20 clumpy cells the walk takes 3.4 ms
// and the filter 2.3 ms; at 60,000 the whole pair list takes 0.73 ms.  Testing
// leaf by leaf, the (cell, particle) tests of the reaching lanes spread over
// the warp, waited for the loads of every test: 12.7 ms, and 2.1 ms at 60,000,
// where a warp's chain is the whole time.  Settling the undecided tests inside
// the walk took half of its 6.2 and 0.77 ms.
constexpr int PAIR_ROW = 256;
constexpr int PT_WARPS = 4;   // warps per block of the traversal
constexpr int PT_STK = 160;   // a popped node pushes at most 8 children; 22 levels at most: 155 entries
enum { WALK_ROWS, WALK_COUNT, WALK_FILL };

// Rows of candidates: rows[c * PAIR_ROW ...], then chunks of a pool.
struct PairRows {
  int32_t* rows;
  int32_t* pool;              // npool chunks of PAIR_ROW entries
  int32_t* first;             // per cell: its first chunk (-1: none; -2: the pool was empty)
  int32_t* next;              // per chunk: the cell's next one
  int32_t npool;
  unsigned long long* used;   // chunks handed out
  int32_t* again;             // the cells that found none left
  unsigned long long* n_again;
};

using wedge::add2;
using wedge::f2;
using wedge::mul2;

struct WalkWarp {
  int2 stk[PT_STK];       // internal node: (first child, children); leaf: (first position, -particles)
  float4 ca[32], cb[32];  // staged candidates: (x hi, y hi, x lo, y lo), (z hi, 2h, z lo, -)
  int32_t k[64];          // sorted positions of the candidates gathered
  float4 ba[8], bb[8];    // the popped node's children: boxes and links
};
struct WalkExact {              // WALK_COUNT, WALK_FILL
  float4 sa[32], sb[32];        // the lanes' cells: (x hi, lo, y hi, lo), (z hi, lo, R, r_in)
  unsigned rej[32];             // undecided tests that failed
  unsigned short und[32 * 32];  // undecided tests: cell lane << 5 | candidate
};

template <int MODE>
__global__ void __launch_bounds__(PT_WARPS * 32)
    pair_traverse(int64_t ncell, const int32_t* __restrict__ order, PairTree T, PairGrid G, int64_t* count,
                  PairRows Q, const int64_t* __restrict__ off, int32_t* out, int64_t cap) {
  constexpr bool EXACT = MODE != WALK_ROWS;
  __shared__ WalkWarp s_walk[PT_WARPS];
  __shared__ WalkExact s_exact[EXACT ? PT_WARPS : 1];
  if (MODE == WALK_FILL && off[ncell] > cap) return;  // the list does not fit its buffer: nothing is written
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  WalkWarp& W = s_walk[threadIdx.x >> 5];
  WalkExact& X = s_exact[EXACT ? threadIdx.x >> 5 : 0];
  const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x);
  const bool valid = t < (EXACT ? (int64_t)*Q.n_again : ncell);
  if (!__any_sync(FULL, valid)) return;
  const int64_t c = valid ? (EXACT ? Q.again[t] : order[t]) : -1;
  SiteSplit SS{};
  if (valid) SS = site_split(G, c);
  const float hx = SS.hx, hy = SS.hy, hz = SS.hz, fR = SS.R, rin = SS.rin;
  if (EXACT) {
    X.sa[lane] = make_float4(hx, SS.lx, hy, SS.ly);
    X.sb[lane] = make_float4(hz, SS.lz, fR, rin);
  }
  // the box around the warp's sites and the largest cell radius
  float gx0 = valid ? hx : INFINITY, gx1 = valid ? hx : -INFINITY, gy0 = valid ? hy : INFINITY;
  float gy1 = valid ? hy : -INFINITY, gz0 = valid ? hz : INFINITY, gz1 = valid ? hz : -INFINITY, gR = fR;
  for (int o = 16; o > 0; o >>= 1) {
    gx0 = fminf(gx0, __shfl_xor_sync(FULL, gx0, o)); gx1 = fmaxf(gx1, __shfl_xor_sync(FULL, gx1, o));
    gy0 = fminf(gy0, __shfl_xor_sync(FULL, gy0, o)); gy1 = fmaxf(gy1, __shfl_xor_sync(FULL, gy1, o));
    gz0 = fminf(gz0, __shfl_xor_sync(FULL, gz0, o)); gz1 = fmaxf(gz1, __shfl_xor_sync(FULL, gz1, o));
    gR = fmaxf(gR, __shfl_xor_sync(FULL, gR, o));
  }
  int32_t* row = nullptr;  // where the next entry goes
  int left = INT32_MAX;    // entries that fit there
  int chunk = -1;          // the chunk it lies in (-1: the row itself; -2: no chunk was left)
  if (valid && MODE == WALK_ROWS) { row = Q.rows + c * PAIR_ROW; left = PAIR_ROW; Q.first[c] = -1; }
  if (valid && MODE == WALK_FILL) row = out + off[c];
  int cnt = 0;
  int nk = 0;  // candidates gathered (warp-uniform)

  // the first n (<= 32) candidates gathered against the 32 cells
  auto test = [&](int n) {
    __syncwarp();
    if (lane < n) {
      const int64_t k = W.k[lane];
      const float2* P = reinterpret_cast<const float2*>(T.split + 6 * k);
      const float2 px = __ldg(P), py = __ldg(P + 1), pz = __ldg(P + 2);
      W.ca[lane] = make_float4(px.x, py.x, px.y, py.y);
      W.cb[lane] = make_float4(pz.x, 2.f * __ldg(T.hs32 + k), pz.y, 0.f);
    }
    if (EXACT) X.rej[lane] = 0u;
    __syncwarp();
    unsigned acc = 0u, und = 0u;  // listed for certain, undecided
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
      const float4 A = W.ca[j], B = W.cb[j];
      // in two-lane arithmetic: (x, y) of the offset; (z hi, reach), (z lo, 2h + r_in)
      const f2 e = add2(add2(f2{A.x, A.y}, f2{-hx, -hy}), add2(f2{A.z, A.w}, f2{-SS.lx, -SS.ly}));
      const f2 u = add2(f2{B.x, B.y}, f2{-hz, fR}), v = add2(f2{B.z, B.y}, f2{-SS.lz, rin});
      const float fz = u.x + v.x;
      const float d2 = fmaf(e.x, e.x, fmaf(e.y, e.y, fz * fz));
      const f2 r2 = mul2(f2{u.y, v.y}, f2{u.y, v.y});
      const int s = dist_screen(d2, r2.x, r2.y);
      acc |= (unsigned)(s == 1) << j;
      und |= (unsigned)(s == 2) << j;
    }
    if (!valid) acc = und = 0u;
    if (!EXACT) {
      for (unsigned m = acc | und; m; m &= m - 1u) {
        const int j = __ffs(m) - 1;
        ++cnt;
        if (left == 0) {
          const unsigned long long q = chunk != -2 ? atomicAdd(Q.used, 1ULL) : ~0ULL;
          if (q >= (unsigned long long)Q.npool) { chunk = -2; continue; }
          if (chunk < 0) Q.first[c] = (int32_t)q; else Q.next[chunk] = (int32_t)q;
          chunk = (int)q;
          row = Q.pool + (int64_t)chunk * PAIR_ROW;
          left = PAIR_ROW;
        }
        *row++ = W.k[j] | (int32_t)((und >> j & 1u) << 31);
        --left;
      }
      return;
    }
    const int nu = __popc(und);
    int o = nu;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(FULL, o, d);
      if (lane >= d) o += v;
    }
    const int U = __shfl_sync(FULL, o, 31);
    o -= nu;
    for (unsigned m = und; m; m &= m - 1u) X.und[o++] = (unsigned short)(lane << 5 | (__ffs(m) - 1));
    __syncwarp();
    for (int r = 0; r < U; r += 32) {
      const bool on = r + lane < U;
      const int e = X.und[on ? r + lane : r];
      const int l = e >> 5, j = e & 31;
      const int64_t cl = __shfl_sync(FULL, c, l);
      if (on) {
        const float4 a = X.sa[l], b = X.sb[l];
        if (!pair_rule(G, T, cl, SiteSplit{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}, W.k[j])) atomicOr(&X.rej[l], 1u << j);
      }
    }
    __syncwarp();
    acc |= und & ~X.rej[lane];
    if (MODE == WALK_FILL)
      for (unsigned m = acc; m; m &= m - 1u) *row++ = T.idx[W.k[__ffs(m) - 1]];
    cnt += __popc(acc);
  };
  // particles [a, a + k) join the candidates; full rounds of 32 are tested
  auto gather = [&](int a, int k) {
    while (k > 0) {
      const int g = k < 32 ? k : 32;
      if (lane < g) W.k[nk + lane] = a + lane;
      nk += g;
      a += g;
      k -= g;
      if (nk >= 32) {
        test(32);
        nk -= 32;
        __syncwarp();
        const int32_t v = lane < nk ? W.k[32 + lane] : 0;
        __syncwarp();
        if (lane < nk) W.k[lane] = v;
      }
    }
  };

  int sp = 0;
  const int nroot = T.nch[0];
  if (nroot == 0) {
    gather((int)T.nb[0], (int)(T.ne[0] - T.nb[0]));  // the root is a leaf
  } else {
    if (lane == 0) W.stk[0] = make_int2((int)T.fc[0], nroot);
    sp = 1;
  }
  __syncwarp();
  while (sp > 0) {
    const int2 E = W.stk[--sp];
    __syncwarp();
    if (E.y < 0) {
      gather(E.x, -E.y);
      continue;
    }
    bool near = false;
    int2 mine = make_int2(0, 0);
    if (lane < E.y) {
      const int64_t nd = (int64_t)E.x + lane;
      const float4 b0 = __ldg(reinterpret_cast<const float4*>(T.box32) + 2 * nd);
      const float4 b1 = __ldg(reinterpret_cast<const float4*>(T.box32) + 2 * nd + 1);
      const float dx = fmaxf(fmaxf(b0.x - gx1, gx0 - b0.w), 0.f);
      const float dy = fmaxf(fmaxf(b0.y - gy1, gy0 - b1.x), 0.f);
      const float dz = fmaxf(fmaxf(b0.z - gz1, gz0 - b1.y), 0.f);
      const float reach = (2.f * b1.z + gR + 1e-6f) * 1.00001f;
      near = dx * dx + dy * dy + dz * dz <= reach * reach;
      if (near) {
        W.ba[lane] = b0;
        W.bb[lane] = b1;
        const unsigned link = __float_as_uint(b1.w);
        if (link == 0u) {
          const int64_t a = T.nb[nd];
          mine = make_int2((int)a, -(int)(T.ne[nd] - a));
        } else if (link == NODE_LINK_FAR) {
          mine = make_int2((int)T.fc[nd], T.nch[nd]);
        } else {
          mine = make_int2((int)(link >> 4), (int)(link & 15u));
        }
      }
    }
    unsigned m = __ballot_sync(FULL, near);
    __syncwarp();
    unsigned keep = 0u;
    for (; m; m &= m - 1u) {
      const int i = __ffs(m) - 1;
      const float4 b0 = W.ba[i], b1 = W.bb[i];
      const float dx = fmaxf(fmaxf(b0.x - hx, hx - b0.w), 0.f);
      const float dy = fmaxf(fmaxf(b0.y - hy, hy - b1.x), 0.f);
      const float dz = fmaxf(fmaxf(b0.z - hz, hz - b1.y), 0.f);
      const float reach = (2.f * b1.z + fR + 1e-6f) * 1.000001f;
      if (__any_sync(FULL, valid && dx * dx + dy * dy + dz * dz <= reach * reach)) keep |= 1u << i;
    }
    // pushed last child first, so that they pop in child order
    const int nkeep = __popc(keep);
    if (sp + nkeep > PT_STK) break;  // unreachable for trees of at most 22 levels
    if (keep >> lane & 1u) W.stk[sp + nkeep - 1 - __popc(keep & lt)] = mine;
    sp += nkeep;
    __syncwarp();
  }
  if (nk > 0) test(nk);
  if (valid && MODE != WALK_FILL) {
    count[c] = cnt;
    if (MODE == WALK_ROWS && chunk == -2) {
      Q.first[c] = -2;
      Q.again[atomicAdd(Q.n_again, 1ULL)] = (int32_t)c;
    }
  }
}

// Settles the undecided entries of a cell's row, one warp per cell: its faces
// go to shared memory in one load, its entries come 32 at a time, and the row
// is packed in place (the writes stay behind the reads) as particle indices;
// count[c] becomes the number of pairs.  Bound by the gathers of the entries'
// positions.
constexpr int RF_FACES = 64;  // faces staged; a cell with more reads them from global memory
__global__ void __launch_bounds__(128, 10) row_filter(int64_t ncell, const int32_t* __restrict__ order, PairTree T,
                                                  PairGrid G, PairRows Q, int64_t* count) {
  __shared__ float4 s_face[4][RF_FACES];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t t = blockIdx.x * 4LL + warp;
  if (t >= ncell) return;  // whole warp
  const int64_t c = order[t];
  const int link = Q.first[c];
  if (link == -2) return;  // walked again
  const int n = (int)count[c];
  const int64_t f0 = G.cfo[c];
  const int nf = (int)(G.cfo[c + 1] - f0);
  float4* sf = s_face[warp];
  const bool staged = nf <= RF_FACES;
  if (staged)
    for (int i = lane; i < nf; i += 32) sf[i] = __ldg(G.face32 + f0 + i);
  const SiteSplit SS = site_split(G, c);
  __syncwarp();
  int32_t* rp = Q.rows + c * PAIR_ROW;  // the part read, the part written
  int32_t* wp = rp;
  int rnext = link, wnext = link;       // the chunks that follow them
  int w = 0;                            // entries in the part written
  int64_t hits = 0;
  for (int b = 0; b < n; b += 32) {
    if (b > 0 && b % PAIR_ROW == 0) {
      rp = Q.pool + (int64_t)rnext * PAIR_ROW;
      rnext = Q.next[rnext];  // (of the last chunk: never followed)
    }
    bool pass = b + lane < n;
    int64_t k = 0;
    if (pass) {
      const int32_t e = rp[b % PAIR_ROW + lane];
      k = e & 0x7fffffff;
      if (e < 0)
        pass = staged ? pair_rule(G, T, c, f0, nf, SS, k, [&](int i) { return sf[i]; })
                      : pair_rule(G, T, c, f0, nf, SS, k, [&](int i) { return __ldg(G.face32 + f0 + i); });
    }
    const unsigned m = __ballot_sync(0xffffffffu, pass);
    const int at = w + __popc(m & ((1u << lane) - 1u));
    int32_t* np = w + __popc(m) > PAIR_ROW ? Q.pool + (int64_t)wnext * PAIR_ROW : nullptr;
    if (pass) {
      const int32_t a = T.idx[k];
      if (at < PAIR_ROW) wp[at] = a; else np[at - PAIR_ROW] = a;
    }
    w += __popc(m);
    hits += __popc(m);
    if (np) {
      wp = np;
      wnext = Q.next[wnext];
      w -= PAIR_ROW;
    }
    __syncwarp();
  }
  if (lane == 0) count[c] = hits;
}

// The same walk with one warp per cell, for grids with many particles per
// cell (few, large cells): lanes test a node's children in parallel, the
// particles of the leaves the cell reaches are gathered in a buffer, and all
// 32 lanes apply the pair rule to 32 candidates at a time.  FILL = false:
// count pairs per cell, keeping the first PAIR_ROW of them in the cell's row;
// FILL = true: write the pairs of the cells `again` at off[c].
constexpr int WALK_STK = 160;   // a popped node pushes at most 8 of its children; 22 levels at most
constexpr int WALK_CAND = 512;  // candidate positions gathered before they are tested

template <bool FILL>
__global__ void __launch_bounds__(128) pair_walk_warp(int64_t ncell, PairTree T, PairGrid G, int64_t* count,
                                                      PairRows Q, const int64_t* __restrict__ off, int32_t* list,
                                                      int64_t cap) {
  __shared__ int32_t s_stk[4][WALK_STK];
  if (FILL && off[ncell] > cap) return;  // the list does not fit its buffer: nothing is written
  __shared__ int32_t s_cand[4][WALK_CAND];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t t = blockIdx.x * 4 + warp;
  if (t >= (FILL ? (int64_t)*Q.n_again : ncell)) return;  // whole warp
  const int64_t c = FILL ? Q.again[t] : t;
  const SiteSplit SS = site_split(G, c);
  const float fsx = SS.hx, fsy = SS.hy, fsz = SS.hz, fR = SS.R;
  int32_t* stk = s_stk[warp];
  int32_t* cand = s_cand[warp];
  int32_t* const out = FILL ? list + off[c] : Q.rows + c * PAIR_ROW;
  int64_t cnt = 0;
  int sp = 1, nc_ = 0;  // stack depth, candidates held
  if (lane == 0) stk[0] = 0;
  __syncwarp();
  // test the candidates held, 32 at a time
  auto flush = [&]() {
    __syncwarp();  // the candidates written by every lane are visible
    for (int b = 0; b < nc_; b += 32) {
      const int j = b + lane;
      const bool hit = j < nc_ && pair_rule(G, T, c, SS, cand[j]);
      const unsigned m = __ballot_sync(0xffffffffu, hit);
      if (hit) {
        const int64_t q = cnt + __popc(m & ((1u << lane) - 1u));
        if (FILL || q < PAIR_ROW) out[q] = T.idx[cand[j]];
      }
      cnt += __popc(m);
    }
    __syncwarp();
    nc_ = 0;
  };
  while (sp > 0) {
    const int nd = stk[sp - 1];
    --sp;
    const int nch = T.nch[nd];
    if (nch == 0) {  // the root is a leaf
      const int64_t a0 = T.nb[nd], a1 = T.ne[nd];
      for (int64_t a = a0; a < a1; a += WALK_CAND) {
        const int k = (int)((a1 - a) < WALK_CAND ? (a1 - a) : WALK_CAND);
        __syncwarp();
        for (int i = lane; i < k; i += 32) cand[i] = (int32_t)(a + i);
        __syncwarp();
        nc_ = k;
        flush();
      }
      continue;
    }
    const int64_t c0 = T.fc[nd];
    bool need = false, leaf = false;
    if (lane < nch) {
      const float* b = T.box32 + 8 * (c0 + lane);
      const float dx = fsx < b[0] ? b[0] - fsx : (fsx > b[3] ? fsx - b[3] : 0.f);
      const float dy = fsy < b[1] ? b[1] - fsy : (fsy > b[4] ? fsy - b[4] : 0.f);
      const float dz = fsz < b[2] ? b[2] - fsz : (fsz > b[5] ? fsz - b[5] : 0.f);
      const float reach = (2.f * b[6] + fR + 1e-6f) * 1.000001f;
      need = dx * dx + dy * dy + dz * dz <= reach * reach;
      leaf = need && T.nch[c0 + lane] == 0;
    }
    const unsigned ml = __ballot_sync(0xffffffffu, leaf), mi = __ballot_sync(0xffffffffu, need && !leaf);
    const int ni = __popc(mi);
    __syncwarp();  // every lane has read the popped entry
    if (sp + ni > WALK_STK) break;  // unreachable for trees of at most 22 levels
    if (need && !leaf) stk[sp + ni - 1 - __popc(mi & ((1u << lane) - 1u))] = (int)(c0 + lane);
    sp += ni;
    // leaf children: gather their particles, testing whenever the buffer fills
    unsigned m = ml;
    while (m) {
      const int bl = __ffs(m) - 1;
      m &= m - 1;
      const int64_t a0 = T.nb[c0 + bl], a1 = T.ne[c0 + bl];
      for (int64_t a = a0; a < a1;) {
        if (nc_ == WALK_CAND) flush();
        const int room = WALK_CAND - nc_;
        const int k = (int)((a1 - a) < room ? (a1 - a) : room);
        for (int i = lane; i < k; i += 32) cand[nc_ + i] = (int32_t)(a + i);
        nc_ += k;
        a += k;
      }
    }
    __syncwarp();
  }
  flush();
  if (!FILL && lane == 0) count[c] = cnt;
}

// Move the rows to their place in the list (one warp per cell).
__global__ void __launch_bounds__(128) place_rows(int64_t ncell, const int64_t* __restrict__ count,
                                                  const int64_t* __restrict__ off, PairRows Q, int32_t* out,
                                                  int64_t cap) {
  const int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (c >= ncell || off[ncell] > cap) return;
  int q = Q.first[c];
  if (q == -2) return;  // written by the second walk
  const int64_t n = count[c];
  const int32_t* src = Q.rows + c * PAIR_ROW;
  int32_t* dst = out + off[c];
  for (int64_t b = 0; b < n; b += PAIR_ROW) {
    const int m = (int)(n - b < PAIR_ROW ? n - b : PAIR_ROW);
    for (int i = lane; i < m; i += 32) dst[b + i] = src[i];
    if (n - b <= PAIR_ROW) break;
    src = Q.pool + (int64_t)q * PAIR_ROW;
    q = Q.next[q];
  }
}

// The cells of pair_walk_warp whose pairs outnumber their row (no chunks
// there): first[c] and the list of cells to walk again.
__global__ void mark_again(int64_t ncell, const int64_t* __restrict__ count, PairRows Q) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= ncell) return;
  const bool over = count[c] > PAIR_ROW;
  Q.first[c] = over ? -2 : -1;
  if (over) Q.again[atomicAdd(Q.n_again, 1ULL)] = (int32_t)c;
}

// Work items: cell c's n pairs in max(1, ceil(ceil(n/32)/K)) items of at
// most K blocks of 32 pairs, K = max(1, (np/32 + ncell) / tgt) from the
// list's pair count np = off[ncell] (read on the device).
__device__ __forceinline__ int64_t item_blocks(int64_t ncell, const int64_t* __restrict__ off, int64_t tgt) {
  const int64_t blocks = off[ncell] / 32 + ncell;
  return blocks / tgt > 1 ? blocks / tgt : 1;
}
__global__ void item_count(int64_t ncell, const int64_t* __restrict__ off, int64_t tgt, int64_t* cnt) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= ncell) return;
  const int64_t K = item_blocks(ncell, off, tgt);
  const int64_t blocks = (off[c + 1] - off[c] + 31) / 32;
  cnt[c] = blocks > K ? (blocks + K - 1) / K : 1;
}
__global__ void item_fill(int64_t ncell, const int64_t* __restrict__ off, const int64_t* __restrict__ ioff,
                          int64_t tgt, PairItem* items, int64_t cap = INT64_MAX) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= ncell || ioff[ncell] > cap) return;
  const int64_t K = item_blocks(ncell, off, tgt);
  const int64_t b = off[c], n = off[c + 1] - b, span = 32 * K;
  int64_t lo = 0;
  for (int64_t i = ioff[c]; i < ioff[c + 1]; ++i) {
    const int64_t k = n - lo < span ? n - lo : span;
    items[i] = PairItem{b + lo, (int32_t)c, (int32_t)k};
    lo += k;
  }
}

// Sort each cell's pair list (<= 1024 entries) by particle index in shared
// memory, one warp per cell, bitonic, carrying f_ai: the keys are (index,
// position in the list) in 64 bits, and f_ai is gathered by position from a
// copy.  Longer lists are left to the library segmented sort.
__global__ void __launch_bounds__(128) sort_small_segments(int64_t ncell, const int64_t* __restrict__ off,
                                                           const int32_t* __restrict__ idx_in,
                                                           const double* __restrict__ frac_in, int32_t* idx,
                                                           double* frac) {
  __shared__ unsigned long long buf[4][1024];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t c = blockIdx.x * 4LL + warp;
  if (c >= ncell) return;
  const int64_t b = off[c], e = off[c + 1];
  const int L = (int)(e - b);
  if (L > 1024 || L == 0) return;
  int P = 1;
  while (P < L) P <<= 1;
  unsigned long long* v = buf[warp];
  for (int i = lane; i < P; i += 32)
    v[i] = i < L ? ((unsigned long long)(uint32_t)idx_in[b + i] << 32) | (unsigned)i : ~0ULL;
  __syncwarp();
  for (int k = 2; k <= P; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = lane; i < P; i += 32) {
        const int ixj = i ^ j;
        if (ixj > i) {
          const unsigned long long a0 = v[i], a1 = v[ixj];
          const bool up = (i & k) == 0;
          if ((a0 > a1) == up) { v[i] = a1; v[ixj] = a0; }
        }
      }
      __syncwarp();
    }
  for (int i = lane; i < L; i += 32) {
    const unsigned long long key = v[i];
    idx[b + i] = (int32_t)(key >> 32);
    if (frac) frac[b + i] = frac_in[b + (int)(key & 0xffffffffu)];
  }
}

__global__ void mark_large(int64_t ncell, const int64_t* __restrict__ off, int64_t* beg, int64_t* end,
                           unsigned long long* nlarge) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= ncell) return;
  if (off[c + 1] - off[c] > 1024) {
    const unsigned long long k = atomicAdd(nlarge, 1ULL);
    beg[k] = off[c];
    end[k] = off[c + 1];
  }
}

__global__ void site_keys(int64_t n, const double* __restrict__ site, uint32_t* keys, int32_t* idx) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  auto q = [](double v) -> uint32_t {
    double s = floor(v * 1024.0);
    s = s < 0 ? 0 : (s > 1023 ? 1023 : s);
    return (uint32_t)s;
  };
  uint32_t k = 0;
  uint32_t xi = q(site[3 * i]), yi = q(site[3 * i + 1]), zi = q(site[3 * i + 2]);
  for (int b = 9; b >= 0; --b) k = (k << 3) | (((xi >> b) & 1) << 2) | (((yi >> b) & 1) << 1) | ((zi >> b) & 1);
  keys[i] = k;
  idx[i] = (int32_t)i;
}


}  // namespace

namespace {

// A pair-list build's launches, shared by the build that reads its sizes back
// and the one that does not.
struct PairWalk {
  PairTree T;
  PairGrid G;
  PairRows Q;
  int32_t* order;
  int64_t* count;
  bool per_warp;
};

// Every cell's pairs in its row (or on the list of cells to walk again), and
// their counts.  pool = false: rows without a pool, for a budget that holds no
// more (every cell past its row is walked again).
int walk_rows(map_ctx* ctx, const PreparedGrid* g, cudaStream_t s, PairWalk& P, bool pool) {
  DevTree& T = ctx->tree;
  const int64_t nc = g->ncell;
  const int tpb = 128;
  // cells visited in Morton order of their sites for coherent traversals
  uint32_t *k_in, *k_out;
  int32_t* o_in;
  MAP_TRY(ensure_t(ctx, ctx->ws_pairs[4], nc, &k_in));
  MAP_TRY(ensure_t(ctx, ctx->ws_pairs[5], nc, &k_out));
  MAP_TRY(ensure_t(ctx, ctx->ws_pairs[6], nc, &o_in));
  MAP_TRY(ensure_t(ctx, ctx->ws_pairs[14], nc, &P.order));  // kept for the inverse mapping's gather order
  site_keys<<<nblk(nc, 256), 256, 0, s>>>(nc, g->site, k_in, o_in); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  size_t tb = 0;
  CUDA_TRY(cub::DeviceRadixSort::SortPairs(nullptr, tb, k_in, k_out, o_in, P.order, nc, 0, 30, s));
  MAP_TRY(ctx_ensure(ctx, ctx->cub_tmp, tb));
  CUDA_TRY(cub::DeviceRadixSort::SortPairs(ctx->cub_tmp.p, tb, k_in, k_out, o_in, P.order, nc, 0, 30, s));

  P.T = PairTree{T.xs, T.ys, T.zs, T.hs, T.hs32, T.split, T.idx, T.begin, T.end, T.first_child, T.nchild, T.box32};
  P.G = PairGrid{g->cell_face_off, g->face_plane, g->face32, g->site, g->rad, g->rin};
  MAP_TRY(ensure_t(ctx, ctx->ws_pairs[0], nc + 1, &P.count));
  const int64_t npool = pool ? nc / 32 + (2 * nc < 4096 ? 2 * nc : 4096) : 0;
  int32_t* buf;
  ctx->rows_done = false;
  MAP_TRY(ensure_t(ctx, ctx->ws_pairs[9], nc, &P.Q.again));
  MAP_TRY(ensure_t(ctx, ctx->ws_pairs[8], (size_t)(nc + npool) * (PAIR_ROW + 1), &buf));
  P.Q.rows = buf;
  P.Q.pool = buf + nc * PAIR_ROW;
  P.Q.first = P.Q.pool + npool * PAIR_ROW;
  P.Q.next = P.Q.first + nc;
  P.Q.npool = (int32_t)npool;
  P.Q.used = ctx->d_counters + 5;
  P.Q.n_again = ctx->d_counters + 6;
  CUDA_TRY(cudaMemsetAsync(P.Q.used, 0, 2 * sizeof(unsigned long long), s));
  CUDA_TRY(cudaMemsetAsync(P.count + nc, 0, sizeof(int64_t), s));
  // many particles per cell (few, large cells): one warp per cell
  P.per_warp = T.n > 16 * nc;
  if (P.per_warp) {
    pair_walk_warp<false><<<nblk(nc, 4), tpb, 0, s>>>(nc, P.T, P.G, P.count, P.Q, nullptr, nullptr, 0); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
    mark_again<<<nblk(nc, 256), 256, 0, s>>>(nc, P.count, P.Q); ++ctx->launches;
  } else {
    const unsigned blocks = nblk(nc, PT_WARPS * 32);
    pair_traverse<WALK_ROWS><<<blocks, PT_WARPS * 32, 0, s>>>(nc, P.order, P.T, P.G, P.count, P.Q, nullptr, nullptr, 0);
    ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
    row_filter<<<nblk(nc, 4), 128, 0, s>>>(nc, P.order, P.T, P.G, P.Q, P.count); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
    pair_traverse<WALK_COUNT><<<blocks, PT_WARPS * 32, 0, s>>>(nc, P.order, P.T, P.G, P.count, P.Q, nullptr, nullptr, 0);
    ++ctx->launches;
  }
  CUDA_TRY(cudaGetLastError());
  return MAP_OK;
}

// The rows and the cells walked again into the list (nothing is written when
// off[nc] exceeds cap).
int walk_list(map_ctx* ctx, const PairWalk& P, int64_t nc, const int64_t* off, int32_t* list, int64_t cap,
              cudaStream_t s) {
  place_rows<<<nblk(nc * 32, 128), 128, 0, s>>>(nc, P.count, off, P.Q, list, cap); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  if (P.per_warp)
    pair_walk_warp<true><<<nblk(nc, 4), 128, 0, s>>>(nc, P.T, P.G, nullptr, P.Q, off, list, cap);
  else
    pair_traverse<WALK_FILL><<<nblk(nc, PT_WARPS * 32), PT_WARPS * 32, 0, s>>>(nc, P.order, P.T, P.G, nullptr, P.Q, off,
                                                                               list, cap);
  ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  ctx->rows_done = true;
  return MAP_OK;
}

// The walk, the list's offsets and the list (np < 0: its length is read back,
// else np is its room).
int walk_to_list(map_ctx* ctx, const PreparedGrid* g, cudaStream_t s, const PairBufs& out, bool pool, int64_t& np,
                 int64_t** off, int32_t** list) {
  const int64_t nc = g->ncell;
  PairWalk P;
  MAP_TRY(walk_rows(ctx, g, s, P, pool));
  MAP_TRY(ensure_t(ctx, out.off ? *out.off : ctx->ws_pairs[1], nc + 1, off));
  size_t tb = 0;
  CUDA_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tb, P.count, *off, nc + 1, s));
  MAP_TRY(ctx_ensure(ctx, ctx->cub_tmp, tb));
  CUDA_TRY(cub::DeviceScan::ExclusiveSum(ctx->cub_tmp.p, tb, P.count, *off, nc + 1, s));
  const bool read = np < 0;
  if (read) {
    CUDA_TRY(cudaMemcpyAsync(ctx->h_scratch, *off + nc, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaStreamSynchronize(s));
    np = ctx->h_scratch[0];
  }
  MAP_TRY(ensure_t(ctx, out.idx ? *out.idx : ctx->ws_pairs[3], np + 1, list));
  return walk_list(ctx, P, nc, *off, *list, read ? INT64_MAX : np, s);
}

// The same, without the pool when the budget does not hold it: later calls on
// as many cells do not try it again, which would walk twice on each.
int build_list(map_ctx* ctx, const PreparedGrid* g, cudaStream_t s, const PairBufs& out, int64_t& np, int64_t** off,
               int32_t** list) {
  const int64_t np0 = np;
  const bool pool = g->ncell < ctx->no_pool_from;
  const int r = walk_to_list(ctx, g, s, out, pool, np, off, list);
  if (r != MAP_ENOMEM || !pool) return r;
  DevBuf& rows = ctx->ws_pairs[8];
  dev_free(ctx, rows.p);
  ctx->bytes_in_use -= rows.cap;
  rows = DevBuf();
  np = np0;
  MAP_TRY(walk_to_list(ctx, g, s, out, false, np, off, list));
  ctx->no_pool_from = g->ncell;
  return MAP_OK;
}

}  // namespace

int pairs_build(map_ctx* ctx, const PreparedGrid* g, cudaStream_t s, const PairBufs& out) {
  const int64_t nc = g->ncell;
  // the list in the walk's order (deterministic); map_get_pairs and
  // map_copy_pairs sort each cell's entries by particle index when read
  int64_t np = -1, *off;
  int32_t* list;
  MAP_TRY(build_list(ctx, g, s, out, np, &off, &list));
  ctx->n_pairs = np;
  ctx->pair_off = off;
  ctx->pair_idx = list;
  ctx->pairs_sorted = false;
  ctx->inv_ready = false;
  ctx->last_ncell = nc;
  return items_build(ctx, off, nc, np, ctx->item_target, s, out);
}

// Work items of a pair list: K blocks of 32 pairs at most, K chosen so that
// the launch has at least `target` items per resident warp (4 warps x 6 CTAs
// per SM); the autotuner may raise the target (smaller items).
int items_build(map_ctx* ctx, const int64_t* off, int64_t nc, int64_t np, int target, cudaStream_t s,
                const PairBufs& out) {
  (void)np;
  const int64_t tgt = (int64_t)target * ctx->sm_count * 24;
  int64_t *icnt, *ioff;
  MAP_TRY(ensure_t(ctx, ctx->ws_pairs[0], nc + 1, &icnt));  // the pair counts are no longer needed
  MAP_TRY(ensure_t(ctx, out.ioff ? *out.ioff : ctx->ws_pairs[11], nc + 1, &ioff));
  item_count<<<nblk(nc, 256), 256, 0, s>>>(nc, off, tgt, icnt); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  CUDA_TRY(cudaMemsetAsync(icnt + nc, 0, sizeof(int64_t), s));
  size_t tb = 0;
  CUDA_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tb, icnt, ioff, nc + 1, s));
  MAP_TRY(ctx_ensure(ctx, ctx->cub_tmp, tb));
  CUDA_TRY(cub::DeviceScan::ExclusiveSum(ctx->cub_tmp.p, tb, icnt, ioff, nc + 1, s));
  CUDA_TRY(cudaMemcpyAsync(ctx->h_scratch, ioff + nc, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  const int64_t nitems = ctx->h_scratch[0];
  PairItem* items;
  double* part;
  MAP_TRY(ensure_t(ctx, out.items ? *out.items : ctx->ws_pairs[10], nitems, &items));
  MAP_TRY(ensure_t(ctx, out.part ? *out.part : ctx->ws_pairs[12], nitems, &part));
  item_fill<<<nblk(nc, 256), 256, 0, s>>>(nc, off, ioff, tgt, items); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  ctx->items = items;
  ctx->item_off = ioff;
  ctx->partial = part;
  ctx->n_items = nitems;
  return MAP_OK;
}

// pairs_build with no host reads: the list's and the items' sizes stay on
// the device; the buffers hold cap_pairs and cap_items, and a build that
// needs more writes nothing beyond them (its off[nc] or ioff[nc] says so).
int pairs_build_graph(map_ctx* ctx, const PreparedGrid* g, cudaStream_t s, const PairBufs& out, int64_t cap_pairs,
                      int64_t cap_items) {
  if (!out.off || !out.idx || !out.items || !out.ioff || !out.part) return MAP_EINVAL;
  const int64_t nc = g->ncell;
  int64_t np = cap_pairs, *off;
  int32_t* list;
  MAP_TRY(build_list(ctx, g, s, out, np, &off, &list));
  // the work items (the item size from the device-side pair count)
  const int64_t tgt = (int64_t)ctx->item_target * ctx->sm_count * 24;
  int64_t *icnt, *ioff;
  MAP_TRY(ensure_t(ctx, ctx->ws_pairs[0], nc + 1, &icnt));
  MAP_TRY(ensure_t(ctx, *out.ioff, nc + 1, &ioff));
  item_count<<<nblk(nc, 256), 256, 0, s>>>(nc, off, tgt, icnt); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  CUDA_TRY(cudaMemsetAsync(icnt + nc, 0, sizeof(int64_t), s));
  size_t tb = 0;
  CUDA_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tb, icnt, ioff, nc + 1, s));
  MAP_TRY(ctx_ensure(ctx, ctx->cub_tmp, tb));
  CUDA_TRY(cub::DeviceScan::ExclusiveSum(ctx->cub_tmp.p, tb, icnt, ioff, nc + 1, s));
  PairItem* items;
  double* part;
  MAP_TRY(ensure_t(ctx, *out.items, cap_items, &items));
  MAP_TRY(ensure_t(ctx, *out.part, cap_items, &part));
  item_fill<<<nblk(nc, 256), 256, 0, s>>>(nc, off, ioff, tgt, items, cap_items); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  ctx->n_pairs = -1;
  ctx->pair_off = off;
  ctx->pair_idx = list;
  ctx->pairs_sorted = false;
  ctx->inv_ready = false;
  ctx->last_ncell = nc;
  ctx->items = items;
  ctx->item_off = ioff;
  ctx->partial = part;
  ctx->n_items = -1;
  return MAP_OK;
}

// Sorts the last mapping call's lists by particle index within each cell,
// f_ai alongside, in place (through copies), on stream s.
int pairs_sort_lists(map_ctx* ctx, cudaStream_t s) {
  if (ctx->pairs_sorted || !ctx->pair_off || !ctx->pair_idx) return MAP_OK;
  const int64_t nc = ctx->last_ncell, np = ctx->n_pairs;
  if (np > 0) {
    int32_t* idx = const_cast<int32_t*>(ctx->pair_idx);
    double* frac = ctx->pair_frac;
    int32_t* idx_in;
    double* frac_in = nullptr;
    MAP_TRY(ensure_t(ctx, ctx->ws_pairs[2], np, &idx_in));
    CUDA_TRY(cudaMemcpyAsync(idx_in, idx, np * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    if (frac) {
      MAP_TRY(ensure_t(ctx, ctx->ws_pairs[13], np, &frac_in));
      CUDA_TRY(cudaMemcpyAsync(frac_in, frac, np * sizeof(double), cudaMemcpyDeviceToDevice, s));
    }
    sort_small_segments<<<nblk(nc, 4), 128, 0, s>>>(nc, ctx->pair_off, idx_in, frac_in, idx, frac); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
    int64_t *lb, *le;
    MAP_TRY(ensure_t(ctx, ctx->ws_misc[1], nc + 1, &lb));
    MAP_TRY(ensure_t(ctx, ctx->ws_misc[2], nc + 1, &le));
    unsigned long long* d_nl = ctx->d_counters + 5;
    CUDA_TRY(cudaMemsetAsync(d_nl, 0, sizeof(unsigned long long), s));
    mark_large<<<nblk(nc, 256), 256, 0, s>>>(nc, ctx->pair_off, lb, le, d_nl); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
    CUDA_TRY(cudaMemcpyAsync(ctx->h_scratch, d_nl, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaStreamSynchronize(s));
    const int64_t nlarge = ctx->h_scratch[0];
    if (nlarge > 0) {
      size_t tb = 0;
      if (frac) {
        CUDA_TRY(cub::DeviceSegmentedSort::SortPairs(nullptr, tb, idx_in, idx, frac_in, frac, np, nlarge, lb, le, s));
        MAP_TRY(ctx_ensure(ctx, ctx->cub_tmp, tb));
        CUDA_TRY(cub::DeviceSegmentedSort::SortPairs(ctx->cub_tmp.p, tb, idx_in, idx, frac_in, frac, np, nlarge, lb,
                                                     le, s));
      } else {
        CUDA_TRY(cub::DeviceSegmentedSort::SortKeys(nullptr, tb, idx_in, idx, np, nlarge, lb, le, s));
        MAP_TRY(ctx_ensure(ctx, ctx->cub_tmp, tb));
        CUDA_TRY(cub::DeviceSegmentedSort::SortKeys(ctx->cub_tmp.p, tb, idx_in, idx, np, nlarge, lb, le, s));
      }
      CUDA_TRY(cudaStreamSynchronize(s));  // the lists are complete for any stream
    }
  }
  ctx->pairs_sorted = true;
  return MAP_OK;
}
