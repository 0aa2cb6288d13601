// FP64 functions of the FP64 build with as few FP64 instructions as their
// accuracy allows.  GB300 issues about 1.8 FP64 lanes per clock and SM, 1/74
// of its FP32 rate: every FP64 instruction of a warp costs as much as some 70
// FP32 or integer ones of a scheduler.  So seeds, table indices, comparisons,
// conversions and the last, small terms run on the FP32 and integer pipes, and
// only what carries the result's 53 bits is FP64: 4 instructions for a square
// root, 6 for an arctangent, 10 for the logarithm of a quotient.
//
// Host and device (the host takes its seeds from sqrtf and a divide), so that
// the arithmetic can be checked without a GPU.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

namespace dm {

#define DM_FN __host__ __device__ __forceinline__

DM_FN int64_t bits(double v) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(v);
#else
  int64_t b; memcpy(&b, &v, 8); return b;
#endif
}
DM_FN double from_bits(int64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double v; memcpy(&v, &b, 8); return v;
#endif
}
DM_FN uint32_t fbits(float v) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(v);
#else
  uint32_t b; memcpy(&b, &v, 4); return b;
#endif
}
DM_FN float from_fbits(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float v; memcpy(&v, &b, 4); return v;
#endif
}
DM_FN int hi32(double v) { return (int)(bits(v) >> 32); }
DM_FN double mk(uint32_t hi, uint32_t lo) { return from_bits((int64_t)(((uint64_t)hi << 32) | lo)); }

// FP32 of v, truncated; 0 below FP32's normal range (v below its largest)
DM_FN float f32(double v) {
  const uint64_t b = (uint64_t)bits(v);
  const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b, e = hi & 0x7fffffffu;
  const uint32_t m = ((e - 0x38000000u) << 3) | (lo >> 29);
  return from_fbits((hi & 0x80000000u) | (e < 0x38100000u ? 0u : m));
}
// FP64 of a normal FP32 value (a zero becomes 2^-127)
DM_FN double f64(float v) {
  const uint32_t b = fbits(v);
  return mk((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u), b << 29);
}
// a > b as integers (no NaN; -0 equals +0)
DM_FN int64_t key(double v) {
  const int64_t b = bits(v);
  return b < 0 ? (int64_t)(0x8000000000000000ull - (uint64_t)b) : b;
}
DM_FN bool gt(double a, double b) { return key(a) > key(b); }
DM_FN double max2(double a, double b) { return gt(a, b) ? a : b; }
DM_FN double min2(double a, double b) { return gt(a, b) ? b : a; }
DM_FN double abs2(double v) { return from_bits(bits(v) & 0x7fffffffffffffffll); }
DM_FN double neg(double v) { return from_bits(bits(v) ^ (int64_t)0x8000000000000000ull); }
DM_FN double neg_if(double v, bool c) { return from_bits(bits(v) ^ ((int64_t)c << 63)); }
DM_FN bool sign(double v) { return bits(v) < 0; }

DM_FN float rsqrt_seed(float x) {
#ifdef __CUDA_ARCH__
  return rsqrtf(x);
#else
  return 1.0f / sqrtf(x);
#endif
}
DM_FN float rcp_seed(float x) {
#ifdef __CUDA_ARCH__
  return __fdividef(1.0f, x);
#else
  return 1.0f / x;
#endif
}

// sqrt(x), 1e-24 <= x < 1e30: the FP32 root, then two corrections
// (x - g^2) / 2g, each residual exact in one FMA and its quotient FP32
// (errors 2^-22, 2^-45, then the last addition's rounding; below 1e-22 the
// last residual leaves FP32's range, 6e-15 relative).
DM_FN double root(double x) {
  const float r = rsqrt_seed(f32(x)), hr = 0.5f * r;
  double g = f64(f32(x) * r);
  g += f64(f32(fma(-g, g, x)) * hr);
  g += f64(f32(fma(-g, g, x)) * hr);
  return g;
}

// a / b, |a| < |b|, normal: both scaled by b's exponent (integer operations),
// then an FP32 quotient and two corrections by exact residuals (2^-54 of 1).
DM_FN double quot(double a, double b) {
  const int64_t sh = (int64_t)(0x3ff00000 - (hi32(b) & 0x7ff00000)) << 32;
  const double A = from_bits(bits(a) + sh), B = from_bits(bits(b) + sh);
  const float r = rcp_seed(f32(B));
  double v = f64(f32(A) * r);
  v += f64(f32(fma(-B, v, A)) * r);
  v += f64(f32(fma(-B, v, A)) * r);
  return v;
}
// the length of a squared length d2 < 1e30, and 1 / len, len < 1e15
DM_FN double length(double d2) { return d2 > 1e-20 ? root(d2) : sqrt(d2); }
DM_FN double inverse(double len) {
  const float r = rcp_seed(f32(len));
  double v = f64(r);
  v += f64(f32(fma(-len, v, 1.0)) * r);
  v += f64(f32(fma(-len, v, 1.0)) * r);
  return len > 1e-18 ? v : 1.0 / len;
}

// Tables of atan(i / 512), i = 0..512, and of c and -ln c for the 512
// intervals of [1, 2): c = the reciprocal of an interval's middle.
constexpr int TAB = 512;
struct Tables {
  double at[TAB + 1];
  double pad;
  double2 lg[TAB];
};

// atan2(y, x).  The larger of |x|, |y| is scaled to [1, 2) by its exponent
// (exact); t = smaller / larger to FP32 picks the node i / 512, an exact
// rotation by it leaves x' and y' with |y'/x'| <= 2^-9.9, whose quotient is an
// FP32 one corrected once by its exact residual, and
// atan t = t - t^3/3 + t^5/5 takes its small terms in FP32 (2^-55).
DM_FN double arg(double y, double x, const double* __restrict__ at) {
  double ax = abs2(x), ay = abs2(y);
  const bool swap = bits(ay) > bits(ax);
  const double mx = swap ? ay : ax, mn = swap ? ax : ay;
  const int32_t e = hi32(mx) & 0x7ff00000;  // scale by 2^(1023 - e)
  const int32_t d = 0x3ff00000 - e;
  const int64_t sh = (int64_t)d << 32;
  const double X = from_bits(bits(mx) + sh);
  // (below 2^-64 of the larger, or both zero: no angle)
  const double Y = e && (hi32(mn) & 0x7ff00000) + d > 0x3ff00000 - (64 << 20) ? from_bits(bits(mn) + sh) : 0.0;
  const float Xf = f32(X), Yf = f32(Y);
  const float q = Yf * rcp_seed(Xf);
#ifdef __CUDA_ARCH__
  const int i = __float2int_rn(q * (float)TAB);
#else
  const int i = (int)lrintf(q * (float)TAB);
#endif
  const float tf = (float)i * (1.0f / TAB);
  const double ti = i ? f64(tf) : 0.0;
  const double xr = fma(Y, ti, X), yr = fma(-X, ti, Y);
  const float rf = rcp_seed(f32(xr));
  const float t0f = f32(yr) * rf;
  const double t0 = t0f != 0.0f ? f64(t0f) : 0.0;
  const float z = t0f * t0f;
  const float s = f32(fma(-xr, t0, yr)) * rf + t0f * z * (z * 0.2f - 0.333333333f);
  const bool nx = sign(x);
  // pi/2 - a (swap), pi - a, pi/2 + a (both): base + a or base - a
  const bool minus = swap != nx;
  const double base = swap ? 1.57079632679489661923 : (nx ? 3.14159265358979323846 : 0.0);
  const double u = t0 + (s != 0.0f ? f64(s) : 0.0);
  return neg_if((base + neg_if(at[i], minus)) + neg_if(u, minus), sign(y));
}

// ln(N / D), N and D positive and normal: each is 2^e m, m c = 1 + r with
// |r| <= 2^-10, and ln(1 + rN) - ln(1 + rD) = d - d s / 2 + cubic, d = rN - rD,
// s = rN + rD, the cubic and higher terms in FP32 (2^-54).
DM_FN double log_ratio(double N, double D, const double2* __restrict__ lg) {
  const uint64_t bn = (uint64_t)bits(N), bd = (uint64_t)bits(D);
  const int hn = (int)(bn >> 32), hd = (int)(bd >> 32);
  const double mn = mk((hn & 0xfffff) | 0x3ff00000, (uint32_t)bn), md = mk((hd & 0xfffff) | 0x3ff00000, (uint32_t)bd);
#ifdef __CUDA_ARCH__
  const double2 cn = __ldg(lg + ((hn >> 11) & (TAB - 1))), cd = __ldg(lg + ((hd >> 11) & (TAB - 1)));
#else
  const double2 cn = lg[(hn >> 11) & (TAB - 1)], cd = lg[(hd >> 11) & (TAB - 1)];
#endif
  const int k = (hn >> 20) - (hd >> 20);
  const double rn = fma(mn, cn.x, -1.0), rd = fma(md, cd.x, -1.0);
  const double d = rn - rd, s = rn + rd;
  const double v = fma(d * -0.5, s, d);
  const float a = f32(rn), b = f32(rd), a3 = a * a * a, b3 = b * b * b;
  const float c = (a3 * (0.333333333f - a * (0.25f - 0.2f * a))) - (b3 * (0.333333333f - b * (0.25f - 0.2f * b)));
  double l = cn.y - cd.y;
  l = fma(k ? f64((float)k) : 0.0, 0.693147180559945309417, l);
  return l + (v + (c != 0.0f ? f64(c) : 0.0));
}

inline void fill_tables(Tables* T) {
  for (int i = 0; i <= TAB; ++i) T->at[i] = (double)atanl((long double)i / TAB);
  T->pad = 0.0;
  for (int i = 0; i < TAB; ++i) {
    const double c = 1.0 / (1.0 + (i + 0.5) / TAB);
    T->lg[i].x = c;
    T->lg[i].y = (double)(-logl((long double)c));
  }
}

}  // namespace dm
