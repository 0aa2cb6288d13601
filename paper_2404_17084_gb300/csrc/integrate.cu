// Pair integrals and cell sums (Section II-B, Eq. 1-3).
//
// Persistent kernel, one warp per work item (a cell's pairs, or a slice of
// them) at a time: a warp pulls an item from a device work queue and takes its
// pairs 32 at a time, one pair per lane.  Warps share nothing and never wait
// for one another.
//
// For each face (r0 from the plane; the inside flag) a lane whose face can
// reach its support queues the face's edges as (pair, edge) records.  The
// warp splits 32 records at a time, each edge integral K'_e into pieces -- at
// most one inner piece, two middle pieces and two pieces beyond the support --
// as (r0, R0, lo, hi) and the sign s_f s_e.  The pieces beyond the support
// (-r0 E(r0) dPhi, one atan2 for both) are added by the lane itself.  Inner
// and middle pieces are pushed onto two per-warp stacks, one per kind;
// whenever a stack holds 32 pieces the whole warp evaluates them together
// (every lane the same code), so the costly evaluations run with all lanes
// busy; the stacks are flushed after the last face.
// A face whose plane passes within 1e-4 h of the particle has its side and
// distance taken from the FP64 plane and position; its edges then run through
// the FP32 pipeline like any other.
//
// Per pair: f_ai = [inside] + sum_f sum_e s_f s_e K'_e (see wedge.cuh).
// M_i = sum_a m_a f_ai is accumulated in FP64 and reduced across the warp;
// rho_i = M_i / V_i.
//
// This file holds the mixed build's kernel and what every build shares;
// integrate64.cu holds the FP64 build's, table.cu the table variant's.
#include <cub/cub.cuh>
#include <type_traits>

#include "internal.cuh"
#include "wedge.cuh"

namespace {

// Mixed build: a face whose plane passes within TAU (in units of h) of the
// particle has its side and distance decided in FP64: FP32 rounding (~1e-7 h)
// could otherwise put the particle on the wrong side of the plane; with the
// FP64 distance, the face's integrals are as accurate in FP32 as any other
// (they are smooth in r0, and continuous as the particle crosses the plane).
// A separate FP64 evaluation of such faces was measured: every cell of a
// 2^18 clumpy snapshot agreed with it and with the FP64 build to the same
// 3.1e-6, and the FP64 path's registers cost the kernel 15%.
constexpr float TAU = 1e-4f;
constexpr unsigned FULL = 0xffffffffu;
constexpr int LCAP = 96;  // stack depth: < 32 left after a drain + up to 2 pieces per lane

// One edge record (EDGE_STRIDE words, 16-byte aligned) in vector loads:
// e0..e2 the in-plane edge normal m, e3 its offset delta, e4..e6 the edge
// direction t, e7, e8 the vertices' positions along t.  The FP32 record is
// interleaved, (m.x, t.x, m.y, t.y), (m.z, t.z, a_A, a_B), (delta), so that
// the pairs the two-lane arithmetic takes sit in adjacent registers.
__device__ __forceinline__ void load_edge(const float* E, float& e0, float& e1, float& e2, float& e3, float& e4,
                                          float& e5, float& e6, float& e7, float& e8) {
  const float4 a = __ldg(reinterpret_cast<const float4*>(E)), b = __ldg(reinterpret_cast<const float4*>(E) + 1);
  const float4 c = __ldg(reinterpret_cast<const float4*>(E) + 2);
  e0 = a.x; e4 = a.y; e1 = a.z; e5 = a.w; e2 = b.x; e6 = b.y; e7 = b.z; e8 = b.w; e3 = c.x;
}

// Per-warp piece stacks (inner, middle) and the results' accumulators:
// col[o][l] sums the pieces of owner lane o that lane l evaluated, so that in
// a drain every lane adds into its own column (bank l, no conflicts and no
// ordering between lanes); after the last drain of a block each owner adds up
// its row (compensated) and clears it.  Every cell sees its own lane's pieces
// in program order, so the result is bit-reproducible.
struct WarpStacks {
  float4 e[2][LCAP];           // (r0, R0, lo, hi): inner, middle
  unsigned char own[2][LCAP];  // owner lane, the sign s_f s_e in bit 7
  float col[32][32];           // [owner][evaluating lane]
  SnapDesc d;                  // the snapshot of the warp's current cell
};

// Evaluates the queued pieces: every stack holding 32 or more (all that is
// left when flush), 32 at a time from the top, and adds each result to its
// owner lane's accumulator.
__device__ __forceinline__ void drain(WarpStacks& S, int& cnt0, int& cnt1, bool flush, unsigned& t0, unsigned& t1) {
  const int lane = threadIdx.x & 31;
  for (;;) {
    int K, n;
    if (cnt1 >= 32 || (flush && cnt1 > 0)) { K = 1; n = cnt1 < 32 ? cnt1 : 32; cnt1 -= n; t1 += n; }
    else if (cnt0 >= 32 || (flush && cnt0 > 0)) { K = 0; n = cnt0 < 32 ? cnt0 : 32; cnt0 -= n; t0 += n; }
    else break;
    const int base = K == 0 ? cnt0 : cnt1;
    const bool on = lane < n;
    float v = 0.f;
    // every lane evaluates (an idle lane a copy of the first piece) and
    // adds its value or 0: no divergent region
    const int idx = base + (on ? lane : 0);
    const float4 P = S.e[K][idx];
    const int o = S.own[K][idx];
    if (K == 1) v = wedge::piece_mid<float, true>(P.x, P.y, P.z, P.w);
    else v = wedge::piece_inner<float>(P.x, P.y, P.z, P.w);
    v = __int_as_float(__float_as_int(v) ^ ((o & 0x80) << 24));
    S.col[o & 31][lane] += on ? v : 0.f;  // this lane's column: no other lane touches it
    __syncwarp();
  }
}

// This lane's row of the column accumulators, summed with compensation
// (Kahan) in a fixed order and cleared for the next block.  Lane o starts at
// column o, so the 32 lanes read 32 different banks at every step.
__device__ __forceinline__ float take_row(float (*col)[32], int o, float& comp) {
  float s = 0.f, c = 0.f;
#pragma unroll 8
  for (int j = 0; j < 32; ++j) {
    const int k = (j + o) & 31;
    const float y = col[o][k] - c;
    col[o][k] = 0.f;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
  }
  comp = c;
  return s;
}

// Mixed build: the particle in the cell's site-relative frame, in units of
// h, and its signed distance to a face plane (> 0 on the inner side), every
// rounding explicit (no contraction left to the compiler).
__device__ __forceinline__ void pair_frame(const SnapDesc& A, int32_t a, double sx, double sy, double sz, float& yx,
                                           float& yy, float& yz, float& hinv) {
  hinv = __frcp_rn((float)__ldg(A.h + a));
  yx = __fmul_rn((float)(__ldg(A.x + a) - sx), hinv);
  yy = __fmul_rn((float)(__ldg(A.y + a) - sy), hinv);
  yz = __fmul_rn((float)(__ldg(A.z + a) - sz), hinv);
}
__device__ __forceinline__ float face_r0s(const float4& F, float yx, float yy, float yz, float hinv) {
  return __fsub_rn(__fmul_rn(F.w, hinv), __fmaf_rn(F.x, yx, __fmaf_rn(F.y, yy, __fmul_rn(F.z, yz))));
}

// ---------------------------------------------------------------- mixed build
// The mixed build compacts the work twice.  The face loop runs with one pair
// per lane; a lane whose face is within its support -- plane within 2h and
// face bounding sphere not wholly beyond 2h (such a face contributes nothing:
// every point of it lies beyond the support, so the particle's projection is
// outside the polygon and the angles of its edges cancel) -- pushes one
// (pair, edge) record per edge of the face on a per-warp stack.  Every 32
// records the warp splits those 32 edges, one per lane, and pushes their
// inner and middle pieces on the piece stacks as before; the beyond-support
// part is evaluated in the lane.  All results go to the owner pair's row of
// the column accumulators.
constexpr int CCAP = 64;  // (pair, edge) records: < 32 left + up to 32 pushed per edge

// A work item's face records (plane, bounding sphere, loop end) are staged in
// the warp's shared memory when the cell has at most FSTAGE faces (read from
// global memory otherwise): the face loop then reads them as broadcasts,
// once per block of 32 pairs, without the global-memory latency.
constexpr int FSTAGE = 48;
struct MixWarp {
  float4 fpl[FSTAGE];    // the item's face planes (site-relative, FP32)
  float4 fsp[FSTAGE];    // their bounding spheres
  int fend[FSTAGE];      // loop end of each face, relative to the cell's first loop entry
  WarpStacks st;  // piece stacks, column accumulators, snapshot
  uint4 cmb[CCAP];       // (r0 bits, c0 bits, edge record offset in floats, fin << 5 | owner)
  float4 py[2][32];      // per pair: (y.x, y.x, y.y, y.y), (y.z, y.z, 1/h, 1/h), y site-relative in units of h
};

// Splits the n (<= 32) records on top of the record stack, one per lane.
template <bool COUNT>
__device__ __forceinline__ void edge_round(MixWarp& M, const float* __restrict__ ecell, int base, int n, int& cnt0,
                                           int& cnt1, unsigned& n_in, unsigned& n_mid, wedge::WorkCount& wc,
                                           unsigned& n_split, unsigned& n_out) {
  WarpStacks& S = M.st;
  const int lane = threadIdx.x & 31;
  __syncwarp();
  const bool on = lane < n;
  const uint4 C = M.cmb[base + (on ? lane : 0)];  // an idle lane takes a copy of the first record
  __syncwarp();  // the records are taken: new ones may overwrite them
  const int o = (int)(C.w & 31u);
  const bool fin = C.w & 32u;
  const float r0 = __uint_as_float(C.x), c0f = __uint_as_float(C.y);
  const float4 Y0 = M.py[0][o], Y1 = M.py[1][o];
  float e0, e1, e2, e3, e4, e5, e6, e7, e8;
  load_edge(ecell + C.z, e0, e1, e2, e3, e4, e5, e6, e7, e8);
  // R0 = m.y - delta/h and the foot's along-edge position e.y, side by side
  // in two-lane arithmetic, then the vertices' positions from the foot
  using wedge::f2;
  const f2 g = wedge::fma2(f2{e2, e6}, f2{Y1.x, Y1.y},
                           wedge::fma2(f2{e1, e5}, f2{Y0.z, Y0.w}, wedge::mul2(f2{e0, e4}, f2{Y0.x, Y0.y})));
  const float R0s = fmaf(-e3, Y1.z, g.x);
  const bool ein = R0s >= 0.f;
  const float R0 = fabsf(R0s);
  const f2 ab = wedge::fma2(f2{e7, e8}, f2{Y1.z, Y1.w}, wedge::sp(-g.y));
  // the edge's pieces as wedge::split_edge_flat cuts them, written with
  // min/max instructions for the clamps and one predicate per piece (the
  // same bounds: no value is NaN, and a +-0 bound gives the same integrals)
  const float aa = ab.x, bb = ab.y;
  const float c2 = fmaf(r0, r0, R0 * R0);
  const bool far = c2 >= 4.f, lt1 = c2 < 1.f;
  float s1, s2;
  {
    // the breakpoints sqrt(4 - c^2), sqrt(1 - c^2): reciprocal square root
    // and one Newton step y (3/2 - r y/2), both in two-lane arithmetic
    const f2 xs = f2{4.f - c2, 1.f - c2};
    const f2 r = f2{rsqrtf(xs.x), rsqrtf(xs.y)};
    const f2 y = wedge::mul2(xs, r);
    const f2 q = wedge::mul2(y, wedge::fma2(wedge::mul2(wedge::sp(-0.5f), r), y, wedge::sp(1.5f)));
    s2 = far ? 0.f : q.x;
    s1 = lt1 ? q.y : 0.f;
  }
  const float x0 = fmaxf(aa, -s2), x1 = fminf(bb, s2);
  const float len = x1 - x0;
  const bool whole = !lt1 && len * len <= c2;
  const float l0 = fmaxf(x0, -s1), h0 = fminf(x1, s1);
  const float h1 = whole ? x1 : fminf(x1, -s1);
  const float l2 = fmaxf(x0, s1);
  const float h3 = far ? bb : fminf(bb, -s2);
  const float l4 = fmaxf(aa, s2);
  const bool v0 = on && h0 > l0, v1 = on && h1 > x0, v2 = on && !whole && x1 > l2;
  const bool v3 = h3 > aa, v4 = !far && bb > l4;
  const bool pos = fin == ein;
  if (COUNT && on) {
    wc.edges++;
    if (v0 || v1 || v2 || v3 || v4) wc.terms++;
    n_split += v1 && v2 && !lt1;
    n_out += (unsigned)v3 + (unsigned)v4;
  }
  // inner pieces (0 or 1 per record): one ballot; middle pieces: two
  const unsigned lt = (1u << lane) - 1u;
  const unsigned bin = __ballot_sync(FULL, v0), bm1 = __ballot_sync(FULL, v1), bm2 = __ballot_sync(FULL, v2);
  const int t0 = __popc(bin), t1 = __popc(bm1) + __popc(bm2);
  const int o0 = cnt0 + __popc(bin & lt);
  const int o1 = cnt1 + __popc(bm1 & lt) + __popc(bm2 & lt);
  // pieces go unfolded; their sign s_f s_e rides in the owner's bit 7
  const unsigned char ow = (unsigned char)(o | (pos ? 0 : 0x80));
  if (v0) { S.e[0][o0] = float4{r0, R0, l0, h0}; S.own[0][o0] = ow; }
  if (v1) { S.e[1][o1] = float4{r0, R0, x0, h1}; S.own[1][o1] = ow; }
  if (v2) { const int q = o1 + (int)v1; S.e[1][q] = float4{r0, R0, l2, x1}; S.own[1][q] = ow; }
  // beyond the support: -c0 (dPhi_left + dPhi_right) as the argument of the
  // product of the two intervals' numbers (R0^2 + lo hi) + i (hi - lo) R0
  {
    const float R02 = R0 * R0;
    const float ar = v3 ? fmaf(aa, h3, R02) : 1.f, ai = v3 ? (h3 - aa) * R0 : 0.f;
    const float br = v4 ? fmaf(l4, bb, R02) : 1.f, bi = v4 ? (bb - l4) * R0 : 0.f;
    const f2 z = wedge::fma2(f2{-ai, ai}, f2{bi, br}, wedge::mul2(wedge::sp(ar), f2{br, bi}));
    S.col[o][lane] += on ? (pos ? -c0f : c0f) * wedge::xatan2(z.y, z.x) : 0.f;
  }
  cnt0 += t0;
  cnt1 += t1;
  __syncwarp();
  if (cnt0 >= 32 || cnt1 >= 32) {
    drain(S, cnt0, cnt1, false, n_in, n_mid);
  }
}

template <int NW, int MINB, bool COUNT>
__global__ void __launch_bounds__(NW * 32, MINB) pair_integrals_mixed(BatchArgs B) {
  __shared__ MixWarp mw[NW];
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  MixWarp& M = mw[threadIdx.x >> 5];
  WarpStacks& S = M.st;
  const SnapDesc& A = S.d;
  wedge::WorkCount wc;
  unsigned n_in = 0, n_mid = 0, n_split = 0, n_out = 0;
  int n64 = 0;
  int cur = -1;
  for (int r = 0; r < 32; ++r) S.col[r][lane] = 0.f;
  __syncwarp();

  const int64_t total = queue_total(B);
  for (;;) {
    int64_t g = 0;
    if (lane == 0) g = (int64_t)atomicAdd(&B.counters[3], 1ULL);
    g = __shfl_sync(FULL, g, 0);
    if (g >= total) break;
    int jl = 0, jh = B.nsnap - 1;
    while (jl < jh) {
      const int jm = (jl + jh + 1) >> 1;
      if (B.item_base[jm] <= g) jl = jm; else jh = jm - 1;
    }
    if (jl != cur) {
      __syncwarp();
      const unsigned long long* src = reinterpret_cast<const unsigned long long*>(B.snaps + jl);
      unsigned long long* dst = reinterpret_cast<unsigned long long*>(&S.d);
      for (int i = lane; i < (int)(sizeof(SnapDesc) / 8); i += 32) dst[i] = src[i];
      __syncwarp();
      cur = jl;
    }
    const int64_t it = g - B.item_base[jl];
    const PairItem item = A.items[it];
    const int64_t c = item.cell;
    const float4* __restrict__ face = A.face;
    const float4* __restrict__ fsph = A.fsph;
    const int64_t f0 = A.cfo[c];
    const int nf = (int)(A.cfo[c + 1] - f0);
    const int64_t l0 = A.fvo[f0];
    const float* __restrict__ ecell = A.edge + l0 * EDGE_STRIDE;
    const double sx = A.site[3 * c], sy = A.site[3 * c + 1], sz = A.site[3 * c + 2];
    const bool staged = nf <= FSTAGE;
    if (staged) {
      __syncwarp();
      for (int i = lane; i < nf; i += 32) {
        M.fpl[i] = face[f0 + i];
        M.fsp[i] = fsph[f0 + i];
        M.fend[i] = (int)(A.fvo[f0 + i + 1] - l0);
      }
      __syncwarp();
    }
    double macc = 0.0;
    // the block loop compiled twice: shared-memory face records (STAGED)
    // or global ones, so that each reads its own memory space
    auto blocks = [&](auto stag) {
      constexpr bool STAGED = decltype(stag)::value;
      const int64_t pb = item.lo, pe = item.lo + item.cnt;
      for (int64_t p0 = pb; p0 < pe; p0 += 32) {
        const int64_t p = p0 + lane;
        const bool active = p < pe;
        float yx = 0.f, yy = 0.f, yz = 0.f, hinv = 0.f;
        int32_t a = 0;
        if (active) {
          a = __ldg(A.pair_idx + p);
          pair_frame(A, a, sx, sy, sz, yx, yy, yz, hinv);
        }
        M.py[0][lane] = make_float4(yx, yx, yy, yy);
        M.py[1][lane] = make_float4(yz, yz, hinv, hinv);
        bool inside = true;
        int cntc = 0, cnt0 = 0, cnt1 = 0;  // stack heights (warp-uniform)
        __syncwarp();
        int kb = 0;
        for (int fi = 0; fi < nf; ++fi) {
          const float4 F = STAGED ? M.fpl[fi] : face[f0 + fi];
          const int ke = STAGED ? M.fend[fi] : (int)(A.fvo[f0 + fi + 1] - l0);
          const float r0s = face_r0s(F, yx, yy, yz, hinv);
          bool fin = r0s >= 0.f;
          float r0 = fabsf(r0s);
          bool inrange = active && r0 < 2.f;
          if (COUNT && active) wc.faces++;
          if (inrange && r0 < TAU) {
            // the plane passes within TAU h: its side and distance from the
            // FP64 plane and position, so that FP32 rounding cannot put the
            // particle on the wrong side; its edges then run as any other
            const double hh = 1.0 / A.h[a];
            const double* st = A.site + 3 * c;
            const double4_32a G = A.face64[f0 + fi];
            const double rs = G.w * hh - (G.x * ((A.x[a] - st[0]) * hh) + G.y * ((A.y[a] - st[1]) * hh) +
                                          G.z * ((A.z[a] - st[2]) * hh));
            fin = rs >= 0.0;
            r0 = (float)fabs(rs);
            if (COUNT) ++n64;
          }
          inside = inside && fin;
          if (inrange) {
            // the face's bounding sphere wholly beyond the support: nothing to add
            const float4 Q = STAGED ? M.fsp[fi] : fsph[f0 + fi];
            const float dx = yx - Q.x * hinv, dy = yy - Q.y * hinv, dz = yz - Q.z * hinv;
            const float rr = 2.f + Q.w * hinv;
            if (dx * dx + dy * dy + dz * dz >= rr * rr * 1.00001f) inrange = false;
          }
          const unsigned mn = __ballot_sync(FULL, inrange);
          if (mn) {
            const int nn = __popc(mn), rank = __popc(mn & lt);
            const float c0f = wedge::c0_of(r0);
            const unsigned tag = (unsigned)lane | (fin ? 32u : 0u);
            for (int k = kb; k < ke; ++k) {
              if (inrange)
                M.cmb[cntc + rank] = make_uint4(__float_as_uint(r0), __float_as_uint(c0f), (unsigned)k * EDGE_STRIDE, tag);
              cntc += nn;
              if (cntc >= 32) {
                cntc -= 32;
                edge_round<COUNT>(M, ecell, cntc, 32, cnt0, cnt1, n_in, n_mid, wc, n_split, n_out);
              }
            }
          }
          kb = ke;
        }
        // what is left: fewer than 32 records, then fewer than 32 pieces of each kind
        if (cntc) edge_round<COUNT>(M, ecell, 0, cntc, cnt0, cnt1, n_in, n_mid, wc, n_split, n_out);
        if (cnt0 || cnt1) drain(S, cnt0, cnt1, true, n_in, n_mid);
        __syncwarp();
        float comp;
        const float rs = take_row(S.col, lane, comp);
        if (active) {
          const double f = (inside ? 1.0 : 0.0) + ((double)rs - (double)comp);
          if (A.frac) A.frac[p] = f;
          macc += A.m[a] * f;
        }
        __syncwarp();
      }
    };
    if (staged) blocks(std::true_type{}); else blocks(std::false_type{});
    for (int o = 16; o > 0; o >>= 1) macc += __shfl_down_sync(FULL, macc, o);
    if (lane == 0) A.partial[it] = macc;
    __syncwarp();
  }
  if (!COUNT) return;
  auto wsum = [](unsigned long long v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(FULL, v, o);
    return v;
  };
  const unsigned long long terms = wsum((unsigned long long)wc.terms), faces = wsum((unsigned long long)wc.faces);
  const unsigned long long edges = wsum((unsigned long long)wc.edges), fp64 = wsum((unsigned long long)n64);
  const unsigned long long split = wsum((unsigned long long)n_split);
  const unsigned long long outs = wsum((unsigned long long)n_out);
  if (lane == 0) {
    atomicAdd(&B.counters[1], terms);
    atomicAdd(&B.counters[2], fp64);
    atomicAdd(&B.counters[8], faces);
    atomicAdd(&B.counters[9], edges);
    atomicAdd(&B.counters[10], 2ull * n_in);
    atomicAdd(&B.counters[11], (unsigned long long)n_mid - split);
    atomicAdd(&B.counters[12], outs);
    atomicAdd(&B.counters[13], split);
  }
}

// CTAs per SM of a launch of shape (NW, MINB): as many as are resident at
// once, at most MINB (a persistent launch beyond residency would only queue).
template <int NW, int MINB, bool COUNT = false>
int mixed_per_sm(int* per_sm, int* regs) {
  auto kern = pair_integrals_mixed<NW, MINB, COUNT>;
  CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kern, NW * 32, 0));
  if (*per_sm > MINB) *per_sm = MINB;
  if (*per_sm < 1) *per_sm = 1;
  if (regs) {
    cudaFuncAttributes a;
    CUDA_TRY(cudaFuncGetAttributes(&a, kern));
    *regs = a.numRegs;
  }
  return MAP_OK;
}

template <int NW, int MINB, bool COUNT = false>
int launch_mixed(map_ctx* ctx, const BatchArgs& B, cudaStream_t s) {
  auto kern = pair_integrals_mixed<NW, MINB, COUNT>;
  int per_sm = 0;
  MAP_TRY((mixed_per_sm<NW, MINB, COUNT>(&per_sm, nullptr)));
  int64_t blocks = (int64_t)per_sm * ctx->sm_count;
  const int64_t need = (B.total + NW - 1) / NW;
  if (blocks > need) blocks = need > 0 ? need : 1;
  kern<<<(unsigned)blocks, NW * 32, 0, s>>>(B); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  return MAP_OK;
}

// Descriptor upload through kernel parameters: the values are captured at
// launch, so the host copy may be reused at once and the launch can sit in a
// CUDA graph.
constexpr int DESC_CHUNK = 16;  // 16 x 192 bytes of parameters per launch
struct DescChunk {
  SnapDesc d[DESC_CHUNK];
  int n;
};
__global__ void put_descs(DescChunk c, SnapDesc* dst) {
  if ((int)threadIdx.x < c.n) dst[threadIdx.x] = c.d[threadIdx.x];
}
constexpr int I64_CHUNK = 480;
struct I64Chunk {
  int64_t v[I64_CHUNK];
  int n;
};
__global__ void put_i64(I64Chunk c, int64_t* dst) {
  for (int i = threadIdx.x; i < c.n; i += blockDim.x) dst[i] = c.v[i];
}

// M_i = sum of cell i's item partials, in item order; rho_i = M_i / V_i.
// One thread per cell over the cells of all snapshots.
__global__ void cell_sums(const SnapDesc* __restrict__ d, const int64_t* __restrict__ cell_base, int nsnap,
                          int64_t total_cells, const int64_t* bad) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= total_cells || (bad && *bad)) return;
  int jl = 0, jh = nsnap - 1;
  while (jl < jh) {
    const int jm = (jl + jh + 1) >> 1;
    if (cell_base[jm] <= g) jl = jm; else jh = jm - 1;
  }
  const SnapDesc& D = d[jl];
  const int64_t c = g - cell_base[jl];
  double M = 0.0;
  for (int64_t i = D.item_off[c]; i < D.item_off[c + 1]; ++i) M += D.partial[i];
  D.cell_mass[c] = M;
  if (D.cell_rho) D.cell_rho[c] = M / D.vol[c];
}

// sum_i M_i of each snapshot, in a fixed order: one block per SUM_CELLS cells,
// its part left in the place of the snapshot's item partials (summed by then;
// at least one per cell), and the parts added by a second launch when there
// are more than one.  (One block took 0.33 ms for 2^20 cells, waiting on its
// own loads.)
constexpr int64_t SUM_CELLS = 16384;
__global__ void __launch_bounds__(256) sum_parts(const SnapDesc* __restrict__ d, double* totals, bool last) {
  typedef cub::BlockReduce<double, 256> BR;
  __shared__ typename BR::TempStorage tmp;
  const SnapDesc& D = d[blockIdx.y];
  const int64_t lo = blockIdx.x * SUM_CELLS, hi = lo + SUM_CELLS < D.ncell ? lo + SUM_CELLS : D.ncell;
  if (lo >= D.ncell) return;  // whole block
  double acc = 0.0;
  for (int64_t i = lo + threadIdx.x; i < hi; i += 256) acc += D.cell_mass[i];
  const double t = BR(tmp).Sum(acc);
  if (threadIdx.x == 0) {
    if (last) totals[D.orig] = t; else D.partial[blockIdx.x] = t;
  }
}
__global__ void sum_snapshots(const SnapDesc* __restrict__ d, double* totals) {
  const SnapDesc& D = d[blockIdx.x];
  const int64_t parts = (D.ncell + SUM_CELLS - 1) / SUM_CELLS;
  double acc = 0.0;
  for (int64_t i = threadIdx.x; i < parts; i += 32) acc += D.partial[i];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if (threadIdx.x == 0) totals[D.orig] = acc;
}

}  // namespace

int integrals_upload(map_ctx* ctx, const SnapDesc* h_desc, const int64_t* h_ibase, const int64_t* h_cbase,
                     int nsnap, SnapDesc* d_desc, int64_t* d_ibase, int64_t* d_cbase, cudaStream_t s) {
  for (int j0 = 0; j0 < nsnap; j0 += DESC_CHUNK) {
    DescChunk c;
    c.n = nsnap - j0 < DESC_CHUNK ? nsnap - j0 : DESC_CHUNK;
    for (int i = 0; i < c.n; ++i) c.d[i] = h_desc[j0 + i];
    put_descs<<<1, DESC_CHUNK, 0, s>>>(c, d_desc + j0); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
  }
  for (int k = 0; k < 2; ++k) {
    const int64_t* h = k == 0 ? h_ibase : h_cbase;
    int64_t* dd = k == 0 ? d_ibase : d_cbase;
    for (int j0 = 0; j0 <= nsnap; j0 += I64_CHUNK) {
      I64Chunk c;
      c.n = nsnap + 1 - j0 < I64_CHUNK ? nsnap + 1 - j0 : I64_CHUNK;
      for (int i = 0; i < c.n; ++i) c.v[i] = h[j0 + i];
      put_i64<<<1, 128, 0, s>>>(c, dd + j0); ++ctx->launches;
      CUDA_TRY(cudaGetLastError());
    }
  }
  return MAP_OK;
}

int integrals_enqueue(map_ctx* ctx, const BatchArgs& B, int variant, cudaStream_t s) {
  CUDA_TRY(cudaMemsetAsync(ctx->d_counters, 0, 4 * sizeof(unsigned long long), s));
  CUDA_TRY(cudaMemsetAsync(ctx->d_counters + 8, 0, 8 * sizeof(unsigned long long), s));
  const bool count = ctx->cfg.count_work != 0;
  if (ctx->cfg.precision == MAP_TABLE) {
    MAP_TRY(launch_table(ctx, B, s));
  } else if (ctx->cfg.precision == MAP_MIXED && count) {
    MAP_TRY((launch_mixed<4, 5, true>(ctx, B, s)));
  } else if (ctx->cfg.precision == MAP_MIXED) {
    switch (variant) {
      case 1: MAP_TRY((launch_mixed<4, 4>(ctx, B, s))); break;
      case 2: MAP_TRY((launch_mixed<2, 9>(ctx, B, s))); break;
      case 3: MAP_TRY((launch_mixed<8, 2>(ctx, B, s))); break;
      default: MAP_TRY((launch_mixed<4, 5>(ctx, B, s))); break;
    }
  } else {
    MAP_TRY(launch_fp64(ctx, B, s));
  }
  if (B.total_cells > 0) {
    cell_sums<<<nblk(B.total_cells, 256), 256, 0, s>>>(B.snaps, B.cell_base, B.nsnap, B.total_cells, B.bad);
    ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
  }
  return MAP_OK;
}

int integrals_shape(map_ctx* ctx, int v, int* warps, int* ctas, int* regs) {
  CUDA_TRY(cudaSetDevice(ctx->device));
  switch (v) {
    case 0: *warps = 4; return mixed_per_sm<4, 5>(ctas, regs);
    case 1: *warps = 4; return mixed_per_sm<4, 4>(ctas, regs);
    case 2: *warps = 2; return mixed_per_sm<2, 9>(ctas, regs);
    case 3: *warps = 8; return mixed_per_sm<8, 2>(ctas, regs);
    default: return MAP_EINVAL;
  }
}

int integrals_sum(map_ctx* ctx, const SnapDesc* d_desc, int nsnap, int64_t max_cells, double* totals, cudaStream_t s) {
  const int64_t parts = (max_cells + SUM_CELLS - 1) / SUM_CELLS;
  for (int j0 = 0; j0 < nsnap; j0 += 65535) {  // (the grid's second dimension)
    const dim3 grid((unsigned)parts, (unsigned)(nsnap - j0 < 65535 ? nsnap - j0 : 65535));
    sum_parts<<<grid, 256, 0, s>>>(d_desc + j0, totals, parts <= 1); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
  }
  if (parts > 1) {
    sum_snapshots<<<nsnap, 32, 0, s>>>(d_desc, totals); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
  }
  return MAP_OK;
}

SnapDesc make_desc(map_ctx* ctx, const PreparedGrid* g, const map_particles* p, const map_outputs* out,
                   const int64_t* pair_off, const int32_t* pair_idx, double* frac, int orig) {
  SnapDesc d;
  d.ncell = g->ncell;
  d.cfo = g->cell_face_off;
  d.fvo = g->face_vert_off;
  d.site = g->site;
  d.vol = g->vol;
  d.pair_off = pair_off;
  d.pair_idx = pair_idx;
  d.x = p->x; d.y = p->y; d.z = p->z; d.m = p->m; d.h = p->h;
  d.frac = frac;
  d.cell_mass = out->cell_mass;
  d.cell_rho = out->cell_rho;
  d.face = g->face32;
  d.edge = g->edge32;
  d.face64 = g->face64;
  d.edge64 = g->edge64;
  d.fsph = g->fsph32;
  d.face_vert = g->face_vert;
  d.vx = g->vx;
  d.vy = g->vy;
  d.vz = g->vz;
  d.items = ctx->items;
  d.item_off = ctx->item_off;
  d.partial = ctx->partial;
  d.nitems = ctx->n_items;
  d.orig = orig;
  return d;
}

int integrals_run(map_ctx* ctx, const PreparedGrid* g, const map_particles* p, map_outputs* out, cudaStream_t s) {
  double* frac;
  MAP_TRY(ensure_t(ctx, ctx->ws_misc[0], ctx->n_pairs + 1, &frac));
  ctx->pair_frac = frac;
  ctx->inv_ready = false;
  SnapDesc* d_desc;
  int64_t* d_base;
  MAP_TRY(ensure_t(ctx, ctx->ws_misc[3], 1, &d_desc));
  MAP_TRY(ensure_t(ctx, ctx->ws_misc[4], 4, &d_base));
  auto upload = [&](BatchArgs& Bo) -> int {
    const SnapDesc h = make_desc(ctx, g, p, out, ctx->pair_off, ctx->pair_idx, frac, 0);
    const int64_t ibase[2] = {0, ctx->n_items}, cbase[2] = {0, g->ncell};
    MAP_TRY(integrals_upload(ctx, &h, ibase, cbase, 1, d_desc, d_base, d_base + 2, s));
    Bo = BatchArgs{d_desc, d_base, d_base + 2, 1, ctx->n_items, g->ncell, ctx->d_counters};
    return MAP_OK;
  };
  BatchArgs B;
  MAP_TRY(upload(B));
  if (ctx->cfg.autotune && ctx->cfg.precision == MAP_MIXED && !ctx->tune_done[MAP_MIXED]) {
    auto rebuild = [&](int target, BatchArgs& Bo) -> int {
      MAP_TRY(items_build(ctx, ctx->pair_off, g->ncell, ctx->n_pairs, target, s));
      return upload(Bo);
    };
    MAP_TRY(integrals_autotune(ctx, rebuild, B, s));
  }
  phase_begin(ctx, 2, s);
  MAP_TRY(integrals_enqueue(ctx, B, ctx->tuned[ctx->cfg.precision == MAP_MIXED ? MAP_MIXED : MAP_FP64], s));
  phase_end(ctx, 2, s);
  if (out->cell_vol) CUDA_TRY(cudaMemcpyAsync(out->cell_vol, g->vol, g->ncell * sizeof(double), cudaMemcpyDeviceToDevice, s));
  MAP_TRY(integrals_sum(ctx, d_desc, 1, g->ncell, ctx->d_total, s));
  return MAP_OK;
}
