// Pair integrals of the FP64 build.
//
// The mixed build's persistent kernel (see integrate.cu) with every value in
// FP64: a warp takes a work item's pairs 32 at a time, one per lane; a lane
// whose face can reach its support queues the face's edges as (pair, edge)
// records; the warp splits 32 records at a time and stacks their pieces, and a
// stack that holds 32 pieces is evaluated by the whole warp.
//
// What bounds it is the FP64 pipe (about 1.8 lanes per clock and SM): a
// warp's FP64 instruction takes 70 issue slots of its scheduler, so
// everything else is next to free, and the design spends it.  Stacks keep
// every FP64 instruction at 32 busy lanes (the kernel this replaces walked
// every edge with all lanes in lockstep); comparisons, clamps, conversions and
// signs are integer operations; square roots, arctangents and logarithms are
// dmath.cuh's; and the pieces are arranged for few of them.  In units of
// 1 / (120 pi), with p(u) = (2 - u)^5 (1 + u):
//   middle  the part [x0, x1] of the edge within the support, as one piece
//           whatever lies inside u = 1:
//             -(32 - 30 r0^4 - r0^6) dOmega + k dPhi + r0 R0 [P], with
//             k = p(r0) - C = 2 (1 - r0)^5 (1 + 2 r0) below r0 = 1 and 0 above,
//             C = 120 pi r0 E(r0);
//   inner   where u < 1, the difference of the two branches,
//             30 (1/u - 7/5 + ...) - (32/u - 48 + ...)
//               = -2/u + 6 - 20 u^2 + 30 u^3 - 18 u^4 + 4 u^5
//               = -2 (1 - u)^5 (1 + 2u) / u,
//           integrated over [max(x0, -s1), min(x1, s1)];
//   beyond  -C dPhi over the rest.
// Each difference of an angle between a piece's ends is one arctangent, of
// the product of the ends' complex numbers, each difference of
// L = asinh(s/c) one logarithm; P collects the terms in s, sU and L with
// coefficients in c^2 and r0^2 (from wedge.cuh's int U^k).
//
// Per piece about 85 FP64 instructions (middle), 90 (inner), 13 (beyond), per
// record 17; the lockstep kernel took two square roots, two arctangents and
// two asinh for each end of each piece.  2^20 clumpy cells (1.3e8 pairs):
// 5.34 -> 1.34 s; 60,013: 297 -> 75.4 ms; 4096 uniform: 19.0 -> 5.0 ms.
#include "dmath.cuh"
#include "internal.cuh"
#include "wedge.cuh"

namespace {

constexpr unsigned FULL = 0xffffffffu;
// An exact zero (particle on a face plane or an edge line) is moved to +EPS on
// the inner side: the integral is continuous in the particle position, and
// treating every exact zero as 'inside' is one consistent displacement of the
// particle into the cell.
constexpr double EPS = 1e-12;
constexpr int DW = 2;       // warps per CTA (21.9 KB of shared memory each)
constexpr int DCTA = 5;     // CTAs per SM
constexpr int DFACES = 48;  // faces staged per work item (more: read from global memory)
constexpr int DREC = 64;    // records: < 32 left + up to 32 pushed per edge
constexpr int DPIECE = 64;  // middle and inner pieces: < 32 left + up to 32 per round
constexpr int DOUT = 96;    // beyond: up to 2 per record

struct DWarp {
  double4_32a fpl[DFACES];  // the item's face planes (site-relative)
  float4 fsp[DFACES];       // their bounding spheres
  int fend[DFACES];         // loop end of each face, relative to the cell's first loop entry
  double py[4][32];         // per pair: y site-relative in units of h, 1/h
  double rec[3][DREC];      // (pair, edge) records: r0, C, k
  uint2 rtag[DREC];         // edge, fin << 5 | owner
  double mid[5][DPIECE];    // r0, R0, lo, hi, k
  double inn[4][DPIECE];    // r0, R0, x0, x1
  double out[4][DOUT];      // C, R0, lo, hi
  unsigned char omid[DPIECE], oinn[DPIECE], oout[DOUT];  // owner lane, bit 7 the sign
  double col[32][32];       // [owner][evaluating lane]
  SnapDesc d;
};

using dm::arg;
using dm::log_ratio;
using dm::root;

// The ends' part of L(hi) - L(lo): |s| + U per end, joined by the signs
// (E(s) = s + U for s >= 0 and c^2 / (|s| + U) below).
__device__ __forceinline__ double dasinh(double lo, double U0, double hi, double U1, double c2, const double2* lg) {
  const double a = dm::abs2(hi) + U1, b = dm::abs2(lo) + U0;
  const bool sh = dm::sign(hi), sl = dm::sign(lo);
  // both >= 0: a / b; both < 0: b / a; lo < 0 <= hi: a b / c^2
  const bool mixed = sl && !sh;
  const double N = mixed ? a * b : (sh ? b : a), D = mixed ? c2 : (sh ? a : b);
  return log_ratio(N, D, lg);
}

// Omega(hi) - Omega(lo), Omega = atan(s R0 (U - r0) / (R0^2 U + r0 s^2)).
__device__ __forceinline__ double domega(double r0, double R0, double R02, double lo, double s20, double U0, double hi,
                                         double s21, double U1, const double* at) {
  const double n1 = hi * R0 * (U1 - r0), d1 = fma(R02, U1, r0 * s21);
  const double n0 = lo * R0 * (U0 - r0), d0 = fma(R02, U0, r0 * s20);
  return arg(fma(n1, d0, -(n0 * d1)), fma(d1, d0, n1 * n0), at);
}

__device__ __forceinline__ double eval_mid(double r0, double R0, double lo, double hi, double k, const dm::Tables* T) {
  const double r02 = r0 * r0, R02 = R0 * R0, c2 = r02 + R02;
  const double s20 = lo * lo, s21 = hi * hi;
  const double U20 = c2 + s20, U21 = c2 + s21;
  const double U0 = root(U20), U1 = root(U21);
  const double dO = domega(r0, R0, R02, lo, s20, U0, hi, s21, U1, T->at);
  const double dP = arg((hi - lo) * R0, fma(lo, hi, R02), T->at);
  const double dL = dasinh(lo, U0, hi, U1, c2, T->lg);
  // 40 P2 - 30 P3 + 9 P4 - P5 = R0 (s (al + 3 s^2) + s U (be - U^2 / 4) + ga L)
  const double al = fma(9.0, c2, fma(9.0, r02, 40.0));
  const double be = fma(-0.375, c2, fma(-0.5, r02, -15.0));
  const double ga = fma(fma(0.5, c2, r02), -30.0 - r02, (c2 * -0.375) * c2);
  const double p1 = hi * fma(U1, fma(-0.25, U21, be), fma(3.0, s21, al));
  const double p0 = lo * fma(U0, fma(-0.25, U20, be), fma(3.0, s20, al));
  const double P = fma(ga, dL, p1 - p0);
  const double r04 = r02 * r02;
  const double K = fma(r04, 30.0 + r02, -32.0);
  return fma(r0 * R0, P, fma(K, dO, k * dP));
}

// (x0, x1: the part within the support; nothing when it misses u < 1)
__device__ __forceinline__ double eval_inner(double r0, double R0, double x0, double x1, const dm::Tables* T) {
  const double r02 = r0 * r0, R02 = R0 * R0, c2 = r02 + R02;
  const double m = 1.0 - c2;
  const double s1 = root(dm::max2(m, 1e-24));
  const double lo = dm::max2(x0, dm::neg(s1)), hi = dm::min2(x1, s1);
  const bool any = dm::gt(hi, lo) && dm::gt(m, 1e-24);
  const double s20 = lo * lo, s21 = hi * hi;
  const double U20 = c2 + s20, U21 = c2 + s21;
  const double U0 = root(U20), U1 = root(U21);
  const double dO = domega(r0, R0, R02, lo, s20, U0, hi, s21, U1, T->at);
  const double dP = arg((hi - lo) * R0, fma(lo, hi, R02), T->at);
  const double dL = dasinh(lo, U0, hi, U1, c2, T->lg);
  // -20 P2 + 30 P3 - 18 P4 + 4 P5
  const double al = fma(-18.0, c2, fma(-18.0, r02, -20.0));
  const double be = fma(1.5, c2, fma(2.0, r02, 15.0));
  const double ga = fma(fma(0.5, c2, r02), fma(4.0, r02, 30.0), (c2 * 1.5) * c2);
  const double p1 = hi * fma(U1, U21 + be, fma(-6.0, s21, al));
  const double p0 = lo * fma(U0, U20 + be, fma(-6.0, s20, al));
  const double P = fma(ga, dL, p1 - p0);
  // r0 [D(U) - D(r0)]'s angle, then D(r0) r0 dPhi = -k dPhi
  const double r04 = r02 * r02;
  const double K = fma(r04, fma(-4.0, r02, -30.0), 2.0);
  const double v = 1.0 - r0, v2 = v * v;
  const double k = (v2 * v2) * (v * fma(4.0, r0, 2.0));
  const double w = fma(r0 * R0, P, fma(K, dO, -(k * dP)));
  return any ? w : 0.0;
}

// Evaluates every stack that holds 32 pieces (all that is left when flush),
// 32 at a time from the top; each lane adds into its own column.
__device__ __forceinline__ void drain(DWarp& W, const dm::Tables* T, int& cm, int& ci, int& co, bool flush,
                                      unsigned& n_mid, unsigned& n_in, unsigned& n_out) {
  const int lane = threadIdx.x & 31;
  for (;;) {
    int n, b, o;
    double v;
    if (cm >= 32 || (flush && cm > 0)) {
      n = cm < 32 ? cm : 32; cm -= n; n_mid += n;
      b = cm + (lane < n ? lane : 0);  // an idle lane takes a copy of the first piece
      o = W.omid[b];
      v = eval_mid(W.mid[0][b], W.mid[1][b], W.mid[2][b], W.mid[3][b], W.mid[4][b], T);
    } else if (co >= 32 || (flush && co > 0)) {
      n = co < 32 ? co : 32; co -= n; n_out += n;
      b = co + (lane < n ? lane : 0);
      o = W.oout[b];
      const double R0 = W.out[1][b], lo = W.out[2][b], hi = W.out[3][b];
      v = dm::neg(W.out[0][b]) * arg((hi - lo) * R0, fma(lo, hi, R0 * R0), T->at);
    } else if (ci >= 32 || (flush && ci > 0)) {
      n = ci < 32 ? ci : 32; ci -= n; n_in += n;
      b = ci + (lane < n ? lane : 0);
      o = W.oinn[b];
      v = eval_inner(W.inn[0][b], W.inn[1][b], W.inn[2][b], W.inn[3][b], T);
    } else {
      break;
    }
    if (lane < n) W.col[o & 31][lane] += dm::neg_if(v, (o & 0x80) != 0);
    __syncwarp();  // the pieces are taken: new ones may overwrite them
  }
}

// Splits the n (<= 32) records on top of the record stack, one per lane.
template <bool COUNT>
__device__ __forceinline__ void edge_round(DWarp& W, const dm::Tables* T, const double* __restrict__ ecell, int base,
                                           int n, int& cm, int& ci, int& co, unsigned& n_mid, unsigned& n_in,
                                           unsigned& n_out, wedge::WorkCount& wc) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  const bool on = lane < n;
  const int b = base + (on ? lane : 0);
  const double r0 = W.rec[0][b], C = W.rec[1][b], k = W.rec[2][b];
  const uint2 tag = W.rtag[b];
  const int o = (int)(tag.y & 31u);
  const double2* E = reinterpret_cast<const double2*>(ecell + (size_t)tag.x * EDGE64_STRIDE);
  const double2 e01 = __ldg(E), e23 = __ldg(E + 1), e45 = __ldg(E + 2), e67 = __ldg(E + 3), e8_ = __ldg(E + 4);
  const double yx = W.py[0][o], yy = W.py[1][o], yz = W.py[2][o], hi_ = W.py[3][o];
  __syncwarp();  // the records are taken: new ones may overwrite them
  // R0 = m.y - delta / h (> 0 inside) and the vertices' positions along the edge.
  // Offsets over h stay unrounded here as in the planes' distances: the rounding
  // of y is then one displacement of the particle for all of them, and one that
  // lies on several planes to the last bit has the same side of each everywhere.
  const double R0s = fma(-e23.y, hi_, fma(e01.x, yx, fma(e01.y, yy, e23.x * yz)));
  const double foot = fma(e45.x, yx, fma(e45.y, yy, e67.x * yz));
  const double aa = fma(e67.y, hi_, -foot), bb = fma(e8_.x, hi_, -foot);
  const bool ein = !dm::sign(R0s) || R0s == 0.0;
  const double R0 = dm::max2(dm::abs2(R0s), EPS);
  const double c2 = fma(R0, R0, r0 * r0);
  const bool far = !dm::gt(4.0, c2);
  const double s2 = far ? 0.0 : root(dm::max2(4.0 - c2, 1e-24));
  const double x0 = dm::max2(aa, dm::neg(s2)), x1 = dm::min2(bb, s2);
  const bool vm = on && dm::gt(x1, x0);
  // u < 1 somewhere on it: an FP32 screen, eval_inner decides
  bool vi = false;
  const float c2f = dm::f32(c2);
  if (vm && c2f < 1.0f) {
    const float s1 = sqrtf(1.0f - c2f) + 1e-3f;
    vi = dm::f32(x1) > -s1 && dm::f32(x0) < s1;
  }
  const double h3 = far ? bb : dm::min2(bb, dm::neg(s2)), l4 = dm::max2(aa, s2);
  const bool v3 = on && dm::gt(h3, aa), v4 = on && !far && dm::gt(bb, l4);
  if (COUNT && on) {
    wc.edges++;
    if (vm || v3 || v4) wc.terms++;
  }
  const unsigned lt = (1u << lane) - 1u;
  const unsigned bm = __ballot_sync(FULL, vm), bi = __ballot_sync(FULL, vi);
  const unsigned b3 = __ballot_sync(FULL, v3), b4 = __ballot_sync(FULL, v4);
  const unsigned char ow = (unsigned char)(o | (((tag.y & 32u) != 0) == ein ? 0 : 0x80));
  if (vm) {
    const int q = cm + __popc(bm & lt);
    W.mid[0][q] = r0; W.mid[1][q] = R0; W.mid[2][q] = x0; W.mid[3][q] = x1; W.mid[4][q] = k;
    W.omid[q] = ow;
  }
  if (vi) {
    const int q = ci + __popc(bi & lt);
    W.inn[0][q] = r0; W.inn[1][q] = R0; W.inn[2][q] = x0; W.inn[3][q] = x1;
    W.oinn[q] = ow;
  }
  if (v3) {
    const int q = co + __popc(b3 & lt);
    W.out[0][q] = C; W.out[1][q] = R0; W.out[2][q] = aa; W.out[3][q] = h3;
    W.oout[q] = ow;
  }
  co += __popc(b3);
  if (v4) {
    const int q = co + __popc(b4 & lt);
    W.out[0][q] = C; W.out[1][q] = R0; W.out[2][q] = l4; W.out[3][q] = bb;
    W.oout[q] = ow;
  }
  co += __popc(b4);
  cm += __popc(bm);
  ci += __popc(bi);
  __syncwarp();
  if (cm >= 32 || ci >= 32 || co >= 32) drain(W, T, cm, ci, co, false, n_mid, n_in, n_out);
}

template <bool COUNT>
__global__ void __launch_bounds__(DW * 32, DCTA) pair_integrals_fp64(BatchArgs B, const dm::Tables* __restrict__ T) {
  __shared__ DWarp dw[DW];
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  DWarp& W = dw[threadIdx.x >> 5];
  const SnapDesc& A = W.d;
  wedge::WorkCount wc;
  unsigned n_mid = 0, n_in = 0, n_out = 0;  // pieces evaluated by this warp
  int cur = -1;                             // snapshot held in W.d
  for (int r = 0; r < 32; ++r) W.col[r][lane] = 0.0;
  __syncwarp();

  const int64_t total = queue_total(B);
  for (;;) {
    int64_t g = 0;
    if (lane == 0) g = (int64_t)atomicAdd(&B.counters[3], 1ULL);
    g = __shfl_sync(FULL, g, 0);
    if (g >= total) break;
    // the snapshot owning queue position g: last j with item_base[j] <= g
    int jl = 0, jh = B.nsnap - 1;
    while (jl < jh) {
      const int jm = (jl + jh + 1) >> 1;
      if (B.item_base[jm] <= g) jl = jm; else jh = jm - 1;
    }
    if (jl != cur) {
      __syncwarp();
      const unsigned long long* src = reinterpret_cast<const unsigned long long*>(B.snaps + jl);
      unsigned long long* dst = reinterpret_cast<unsigned long long*>(&W.d);
      for (int i = lane; i < (int)(sizeof(SnapDesc) / 8); i += 32) dst[i] = src[i];
      __syncwarp();
      cur = jl;
    }
    const int64_t it = g - B.item_base[jl];
    const PairItem item = A.items[it];
    const int64_t c = item.cell;
    const int64_t f0 = A.cfo[c];
    const int nf = (int)(A.cfo[c + 1] - f0);
    const int64_t l0 = A.fvo[f0];
    const double* __restrict__ ecell = A.edge64 + l0 * EDGE64_STRIDE;
    const double sx = A.site[3 * c], sy = A.site[3 * c + 1], sz = A.site[3 * c + 2];
    const bool staged = nf <= DFACES;
    __syncwarp();
    if (staged)
      for (int i = lane; i < nf; i += 32) {
        W.fpl[i] = A.face64[f0 + i];
        W.fsp[i] = A.fsph[f0 + i];
        W.fend[i] = (int)(A.fvo[f0 + i + 1] - l0);
      }
    __syncwarp();
    double macc = 0.0;
    const int64_t pe = item.lo + item.cnt;
    for (int64_t p0 = item.lo; p0 < pe; p0 += 32) {
      const int64_t p = p0 + lane;
      const bool active = p < pe;
      double yx = 0.0, yy = 0.0, yz = 0.0, hinv = 0.0;
      int32_t a = 0;
      if (active) {
        a = __ldg(A.pair_idx + p);
        hinv = 1.0 / __ldg(A.h + a);
        yx = (__ldg(A.x + a) - sx) * hinv;
        yy = (__ldg(A.y + a) - sy) * hinv;
        yz = (__ldg(A.z + a) - sz) * hinv;
      }
      W.py[0][lane] = yx; W.py[1][lane] = yy; W.py[2][lane] = yz; W.py[3][lane] = hinv;
      // (reach: the support and FP32's error of an offset from y, in units of h)
      const float fx = (float)yx, fy = (float)yy, fz = (float)yz, fh = (float)hinv;
      const float reach = 2.f + 1e-6f * (fabsf(fx) + fabsf(fy) + fabsf(fz));
      bool inside = true;
      int cr = 0, cm = 0, ci = 0, co = 0;  // stack heights (warp-uniform)
      __syncwarp();
      int kb = 0;
      for (int fi = 0; fi < nf; ++fi) {
        const double4_32a F = staged ? W.fpl[fi] : A.face64[f0 + fi];
        const float4 Q = staged ? W.fsp[fi] : A.fsph[f0 + fi];
        const int ke = staged ? W.fend[fi] : (int)(A.fvo[f0 + fi + 1] - l0);
        const double r0s = fma(F.w, hinv, -fma(F.x, yx, fma(F.y, yy, F.z * yz)));
        const bool fin = !dm::sign(r0s) || r0s == 0.0;
        const double r0 = dm::max2(dm::abs2(r0s), EPS);
        if (COUNT && active) wc.faces++;
        inside = inside && fin;
        // within the support: the plane, and not the face's bounding sphere
        // wholly beyond it (an FP32 test that keeps every face it is not sure
        // of: its errors are 3e-7 of |y| and of the sphere's distance in units of
        // h, of which one is at most the other, 2 and the radius)
        bool near = active && dm::gt(2.0, r0);
        if (near) {
          const float dx = fx - Q.x * fh, dy = fy - Q.y * fh, dz = fz - Q.z * fh;
          const float rr = reach + Q.w * fh;
          near = !(dx * dx + dy * dy + dz * dz > rr * rr * 1.00001f);
        }
        const unsigned mn = __ballot_sync(FULL, near);
        if (mn) {
          const int nn = __popc(mn), rank = __popc(mn & lt);
          // C = 120 pi r0 E(r0) = (2 - r0)^5 (1 + r0) - k
          const double t = 2.0 - r0, t2 = t * t, v = dm::max2(1.0 - r0, 0.0), v2 = v * v;
          const double k = (v2 * v2) * (v * fma(4.0, r0, 2.0));
          const double C = fma((t2 * t2) * t, 1.0 + r0, dm::neg(k));
          const unsigned tag = (unsigned)lane | (fin ? 32u : 0u);
          for (int e = kb; e < ke; ++e) {
            if (near) {
              const int q = cr + rank;
              W.rec[0][q] = r0; W.rec[1][q] = C; W.rec[2][q] = k;
              W.rtag[q] = make_uint2((unsigned)e, tag);
            }
            cr += nn;
            if (cr >= 32) {
              cr -= 32;
              edge_round<COUNT>(W, T, ecell, cr, 32, cm, ci, co, n_mid, n_in, n_out, wc);
            }
          }
        }
        kb = ke;
      }
      // what is left: fewer than 32 records, then fewer than 32 pieces of each kind
      if (cr) edge_round<COUNT>(W, T, ecell, 0, cr, cm, ci, co, n_mid, n_in, n_out, wc);
      if (cm || ci || co) drain(W, T, cm, ci, co, true, n_mid, n_in, n_out);
      __syncwarp();
      // this lane's row, in a fixed order, cleared for the next block (lane o
      // starts at column o: 32 different banks)
      double s = 0.0;
#pragma unroll 4
      for (int j = 0; j < 32; ++j) {
        const int q = (j + lane) & 31;
        s += W.col[lane][q];
        W.col[lane][q] = 0.0;
      }
      if (active) {
        const double f = fma(s, 1.0 / (120.0 * MAP_PI), inside ? 1.0 : 0.0);
        if (A.frac) A.frac[p] = f;
        macc += A.m[a] * f;
      }
      __syncwarp();
    }
    for (int o = 16; o > 0; o >>= 1) macc += __shfl_down_sync(FULL, macc, o);
    if (lane == 0) A.partial[it] = macc;  // summed per cell by cell_sums
    __syncwarp();
  }
  if (!COUNT) return;
  auto wsum = [](unsigned long long v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(FULL, v, o);
    return v;
  };
  const unsigned long long terms = wsum((unsigned long long)wc.terms), faces = wsum((unsigned long long)wc.faces);
  const unsigned long long edges = wsum((unsigned long long)wc.edges);
  if (lane == 0) {
    atomicAdd(&B.counters[1], terms);
    atomicAdd(&B.counters[8], faces);
    atomicAdd(&B.counters[9], edges);
    atomicAdd(&B.counters[10], 2ull * n_in);
    atomicAdd(&B.counters[11], (unsigned long long)n_mid);
    atomicAdd(&B.counters[12], (unsigned long long)n_out);
  }
}

template <bool COUNT>
int launch(map_ctx* ctx, const BatchArgs& B, cudaStream_t s) {
  auto kern = pair_integrals_fp64<COUNT>;
  int per_sm = 0;
  CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, DW * 32, 0));
  if (per_sm < 1) per_sm = 1;
  int64_t blocks = (int64_t)per_sm * ctx->sm_count;
  const int64_t need = (B.total + DW - 1) / DW;
  if (blocks > need) blocks = need > 0 ? need : 1;
  kern<<<(unsigned)blocks, DW * 32, 0, s>>>(B, static_cast<const dm::Tables*>(ctx->d_tables)); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  return MAP_OK;
}

}  // namespace

int fp64_tables(map_ctx* ctx) {
  dm::Tables T;
  dm::fill_tables(&T);
  CUDA_TRY(cudaMalloc(&ctx->d_tables, sizeof(T)));
  CUDA_TRY(cudaMemcpy(ctx->d_tables, &T, sizeof(T), cudaMemcpyHostToDevice));
  return MAP_OK;
}

int launch_fp64(map_ctx* ctx, const BatchArgs& B, cudaStream_t s) {
  return ctx->cfg.count_work ? launch<true>(ctx, B, s) : launch<false>(ctx, B, s);
}
