// Pseudo-particles (Section III-A/B) and their smoothing lengths (Section III-C/D).
//
// Walk (Eq. 5): a node is opened when r_node = 0 or s_node^2 > theta^2 r_node^2,
// r_node being the distance from its centre of mass to the nearest source, or
// when one of the walk controls of Section III-B asks for it (r_part, r_leaf,
// regions of an earlier step; see the opening rule below).  A
// node is reached when all its ancestors are opened; reached nodes that are
// not opened become pseudo-particles (centre of mass, node mass); reached
// leaves that are opened yield their particles, which keep their h.  Because
// every node is a contiguous range of the Morton-sorted particles, the
// accepted nodes and extracted particles partition that order, and listing
// them by first sorted position is the depth-first order of the walk.
//
// h of the accepted nodes: h = hfact n^(-1/3), n = sum_b W(r_ab, h) over the
// node set (accepted nodes plus opened leaves standing in for their
// particles), initial guess hfact * 2 s_node (Eq. 9; a node of size 0 starts
// from its first particle's h).  Candidates are all members when there are at
// most ngb_bruteforce_max of them (Section III-D), otherwise the members whose
// ancestor on level k_mid (one level above the highest member) lies within
// r_cut of the target, r_cut = sqrt(3) s_mid, replaced by 4 hfact s_above
// (s_above: the target's ancestor two levels up) when that is larger (Eq. 10).
#include <cub/cub.cuh>

#include "internal.cuh"

namespace {


constexpr int64_t KIND_PARTICLE = (int64_t)1 << 62;

// Opening rule of the walk (Eq. 5 and the controls of Section III-B), every
// distance compared squared with each product and sum rounded once.
struct WalkRule {
  const double* src;  // 3 per source
  int nsrc;
  double theta, r_part, r_leaf;
  const double* reg;  // 5 per region: centre, radius, smallest size
  int nreg;
};

__device__ __forceinline__ double sq3(double dx, double dy, double dz) {
  return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

__global__ void open_flags(int64_t nn, const double* __restrict__ com, const unsigned long long* __restrict__ size_bits,
                           const int32_t* __restrict__ nchild, WalkRule R, int8_t* open) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nn) return;
  const double s = bitsd(size_bits[i]);
  const bool leaf = nchild[i] == 0;
  const double s2 = __dmul_rn(s, s), th2 = __dmul_rn(R.theta, R.theta);
  const double tp = __dadd_rn(R.r_part, s), tl = __dadd_rn(R.r_leaf, s);
  const double tp2 = __dmul_rn(tp, tp), tl2 = __dmul_rn(tl, tl);
  const double cx = com[3 * i], cy = com[3 * i + 1], cz = com[3 * i + 2];
  bool op = false;
  for (int k = 0; k < R.nsrc; ++k) {
    const double r2 = sq3(__dsub_rn(cx, R.src[3 * k]), __dsub_rn(cy, R.src[3 * k + 1]), __dsub_rn(cz, R.src[3 * k + 2]));
    if (r2 == 0.0 || s2 > __dmul_rn(th2, r2)) op = true;
    else if (R.r_part > 0.0 && r2 < tp2) op = true;
    else if (!leaf && R.r_leaf > 0.0 && r2 < tl2) op = true;
  }
  for (int k = 0; k < R.nreg; ++k) {
    const double* g = R.reg + 5 * k;
    const double d2 = sq3(__dsub_rn(cx, g[0]), __dsub_rn(cy, g[1]), __dsub_rn(cz, g[2]));
    if (d2 < __dmul_rn(g[3], g[3]) && s > g[4]) op = true;
  }
  open[i] = op ? 1 : 0;
}

// Status per node: 0 not reached / opened internal, 1 accepted, 2 opened leaf.
__global__ void walk_status(int64_t nn, const int32_t* __restrict__ parent, const int8_t* __restrict__ open,
                            const int32_t* __restrict__ nchild, int8_t* status) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nn) return;
  bool reached = true;
  for (int32_t a = parent[i]; a >= 0; a = parent[a])
    if (!open[a]) { reached = false; break; }
  int8_t st = 0;
  if (reached) {
    if (!open[i]) st = 1;
    else if (nchild[i] == 0) st = 2;
  }
  status[i] = st;
}

__global__ void mark_heads(int64_t nn, const int8_t* __restrict__ status, const int64_t* __restrict__ nb,
                           const int64_t* __restrict__ ne, int64_t* head, int32_t* is_head) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nn) return;
  if (status[i] == 1) {
    head[nb[i]] = i;
    is_head[nb[i]] = 1;
  } else if (status[i] == 2) {
    for (int64_t p = nb[i]; p < ne[i]; ++p) {
      head[p] = KIND_PARTICLE | p;
      is_head[p] = 1;
    }
  }
}

__global__ void write_pseudo(int64_t n, const int64_t* __restrict__ head, const int32_t* __restrict__ is_head,
                             const int64_t* __restrict__ slot, const double* __restrict__ com,
                             const double* __restrict__ mass, const int64_t* __restrict__ label,
                             const double* __restrict__ xs, const double* __restrict__ ys, const double* __restrict__ zs,
                             const double* __restrict__ ms, const double* __restrict__ hs,
                             const int32_t* __restrict__ idx, double* ox, double* oy, double* oz, double* om, double* oh,
                             int32_t* kind, int64_t* ident, int32_t* node_of_slot) {
  int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= n || !is_head[p]) return;
  const int64_t j = slot[p];
  const int64_t hd = head[p];
  if (hd & KIND_PARTICLE) {
    const int64_t q = hd & (KIND_PARTICLE - 1);
    ox[j] = xs[q]; oy[j] = ys[q]; oz[j] = zs[q]; om[j] = ms[q]; oh[j] = hs[q];
    if (kind) kind[j] = 1;
    if (ident) ident[j] = idx[q];
    node_of_slot[j] = -1;
  } else {
    ox[j] = com[3 * hd]; oy[j] = com[3 * hd + 1]; oz[j] = com[3 * hd + 2]; om[j] = mass[hd]; oh[j] = 0.0;
    if (kind) kind[j] = 0;
    if (ident) ident[j] = label[hd];
    node_of_slot[j] = (int32_t)hd;
  }
}

// The node set for the h solve: accepted nodes and opened leaves, in node order.
__global__ void member_flags(int64_t nn, const int8_t* __restrict__ status, int32_t* flag) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nn) return;
  flag[i] = status[i] != 0 ? 1 : 0;
}

__global__ void member_write(int64_t nn, const int32_t* __restrict__ flag, const int64_t* __restrict__ pos,
                             int32_t* members) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nn || !flag[i]) return;
  members[pos[i]] = (int32_t)i;
}

// The members' centres of mass in the order they are scanned, as FP32 hi/lo
// pairs: x, y, z rounded to FP32 and the node, then what the rounding left.
__global__ void member_points(int64_t nm, const int32_t* __restrict__ members, const double* __restrict__ com, float4* hi,
                              float4* lo) {
  const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j >= nm) return;
  const int32_t b = members[j];
  const double x = com[3 * (int64_t)b], y = com[3 * (int64_t)b + 1], z = com[3 * (int64_t)b + 2];
  const float hx = (float)x, hy = (float)y, hz = (float)z;
  hi[j] = make_float4(hx, hy, hz, __int_as_float(b));
  lo[j] = make_float4((float)(x - (double)hx), (float)(y - (double)hy), (float)(z - (double)hz), 0.f);
}

struct NodeSet {
  int64_t nm;        // members
  const float4* hi;  // their points (member_points); with use_kmid grouped by their k_mid ancestor
  const float4* lo;
  const double* com;  // node centre of mass (3 per node)
  // k_mid candidates (used when use_kmid)
  int use_kmid;
  int64_t mid_begin, mid_end;  // node id range of level k_mid
  const int64_t* mid_off;      // per mid node: its range of members (size nmid+1)
};

// What bounds the solve is latency, each sum a chain of gathers over up to
// 10^4 members or the members of each flagged level-k_mid node: so a warp
// gathers the candidates within 2.5 h once, as FP32 offsets in shared memory,
// and iterates on those; FP64 comes in for one last step of third order (as in
// the full-resolution solve).  FP32 leads there and decides only what is clear
// in FP32: a node that comes near a bound of the bracket, a sign of g within
// 1e-4 h, a flat g, or neighbours at a distance that the hi/lo split does not
// resolve (h < 1e-8), or whose last step does not settle, is solved with FP64
// sums throughout.  A node's size may be 1e-17 (one particle's rounded centre of
// mass), where n(h) leaves FP32's range: there only a node by itself is clear,
// and its g is known.
// Scanning every candidate in FP64 at every
// Newton step took 2.1 ms for 927 nodes and 17 ms for 16,000; this takes 0.25
// and 2.6 ms (with lists of 512 and bisection to 1e-12 before the FP64 step:
// 0.67 and 3.6 ms, the far nodes' bisections scanning at every step).
constexpr int PS_CAP = 1024;  // candidates held per warp
constexpr int PS_WARPS = 2;
struct PseudoWarp {
  float x[PS_CAP], y[PS_CAP], z[PS_CAP];
  int32_t node[PS_CAP];
};
constexpr unsigned PFULL = 0xffffffffu;
constexpr float SPLIT_ERR = 8e-15f;  // error of a hi/lo offset beyond FP32's relative one
constexpr float H_SPLIT = 1e-8f;     // from here up a relative margin of 1e-5 covers it

template <typename V>
__device__ __forceinline__ V lanes_sum(V v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(PFULL, v, o);
  return v;
}

struct PseudoSolve {
  const NodeSet& S;
  PseudoWarp& W;
  int lane;
  double px, py, pz;                // the node's centre of mass
  float hx, lx, hy, ly, hz, lz;     // its FP32 hi/lo
  double rcut;
  float R = -1.f;  // radius the list covers (-1: none)
  int n = 0;       // its length; -1: it does not fit, every pass scans
  bool sure = true;  // every density so far was within FP32's accuracy
  bool alone = false;  // the last one was a tiny node's without neighbours: n = 1 / (pi h^3)

  // f(offset x, y, z, node, valid) over the candidates, 32 at a time, every lane calling
  template <typename F>
  __device__ __forceinline__ void scan(F f) const {
    auto range = [&](int64_t a, int64_t b) {
      for (int64_t j0 = a; j0 < b; j0 += 32) {
        const int64_t j = j0 + lane < b ? j0 + lane : b - 1;
        const float4 H = __ldg(S.hi + j), L = __ldg(S.lo + j);
        f((H.x - hx) + (L.x - lx), (H.y - hy) + (L.y - ly), (H.z - hz) + (L.z - lz), __float_as_int(H.w), j0 + lane < b);
      }
    };
    if (!S.use_kmid) { range(0, S.nm); return; }
    // the lanes test 32 level-k_mid nodes at a time, then share out the
    // members of each flagged one
    const double rc2 = rcut * rcut;
    for (int64_t m0 = S.mid_begin; m0 < S.mid_end; m0 += 32) {
      const int64_t m = m0 + lane;
      bool flag = false;
      if (m < S.mid_end) {
        const double dx = S.com[3 * m] - px, dy = S.com[3 * m + 1] - py, dz = S.com[3 * m + 2] - pz;
        flag = dx * dx + dy * dy + dz * dz < rc2;
      }
      for (unsigned bal = __ballot_sync(PFULL, flag); bal; bal &= bal - 1) {
        const int64_t k = m0 + (__ffs(bal) - 1) - S.mid_begin;
        range(S.mid_off[k], S.mid_off[k + 1]);
      }
    }
  }

  __device__ __forceinline__ void gather(float r) {
    const unsigned lt = (1u << lane) - 1u;
    const float wide = (r + SPLIT_ERR) * 1.00001f, r2 = r >= 2.f * H_SPLIT ? r * r * 1.00001f : wide * wide;
    int c = 0;
    __syncwarp();
    scan([&](float x, float y, float z, int node, bool on) {
      const bool in = on && x * x + y * y + z * z < r2;
      const unsigned m = __ballot_sync(PFULL, in);
      const int k = c + __popc(m & lt);
      if (in && k < PS_CAP) { W.x[k] = x; W.y[k] = y; W.z[k] = z; W.node[k] = node; }
      c += __popc(m);
    });
    __syncwarp();
    R = r;
    n = c <= PS_CAP ? c : -1;
  }

  // a list that covers the support 2h and is not far larger than it
  __device__ __forceinline__ void cover(float h) {
    if (2.f * h > 0.999f * R || (n < 0 ? R > 2.6f * h : R > 8.f * h)) gather(2.5f * h);
  }

  // n(h) and dn/dh, FP32
  __device__ __forceinline__ void density(float h, float& nn, float& dn) {
    cover(h);
    // (the node itself lies at the offset 0 exactly)
    alone = h < H_SPLIT && n == 1;
    sure = sure && (h >= H_SPLIT || alone);
    const float ih = 1.0f / h;
    float s = 0.f, d = 0.f;
    auto add = [&](float x, float y, float z) {
      const float dx = x * ih, dy = y * ih, dz = z * ih;
      const float q2 = dx * dx + dy * dy + dz * dz;
      if (q2 >= 4.f) return;
      const float q = sqrtf(q2);
      float w, dwq;
      if (q < 1.f) { w = 1.f - 1.5f * q2 + 0.75f * q2 * q; dwq = -3.f * q2 + 2.25f * q2 * q; }
      else { const float t = 2.f - q; w = 0.25f * t * t * t; dwq = -0.75f * t * t * q; }
      s += w;
      d += 3.f * w + dwq;
    };
    if (n >= 0)
      for (int j = lane; j < n; j += 32) add(W.x[j], W.y[j], W.z[j]);
    else
      scan([&](float x, float y, float z, int, bool on) { if (on) add(x, y, z); });
    const float norm = ih * ih * ih * (float)(1.0 / MAP_PI);
    nn = lanes_sum(s) * norm;
    dn = -lanes_sum(d) * norm * ih;
  }

  // sums of w(q), q w'(q) and q^2 w''(q) + 2 q w'(q) at h, FP64 behind an FP32 screen
  __device__ __forceinline__ void sums64(double h, double& s, double& d, double& e) {
    const float hf = (float)h, wide = 2.00001f * hf + SPLIT_ERR, r2 = hf >= H_SPLIT ? 4.00004f * hf * hf : wide * wide;
    cover(hf);
    s = d = e = 0.0;
    const double ih = 1.0 / h;
    auto add = [&](int node) {
      const double* c = S.com + 3 * (int64_t)node;
      const double ex = (c[0] - px) * ih, ey = (c[1] - py) * ih, ez = (c[2] - pz) * ih;
      const double q2 = ex * ex + ey * ey + ez * ez, q = sqrt(q2), q3 = q2 * q;
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
    };
    if (n >= 0) {
      for (int j = lane; j < n; j += 32)
        if (W.x[j] * W.x[j] + W.y[j] * W.y[j] + W.z[j] * W.z[j] <= r2) add(W.node[j]);
    } else {
      scan([&](float x, float y, float z, int node, bool on) { if (on && x * x + y * y + z * z <= r2) add(node); });
    }
    s = lanes_sum(s);
    d = lanes_sum(d);
    e = lanes_sum(e);
  }

  // n(h) and dn/dh by FP64 sums
  __device__ __forceinline__ void density64(double h, double& nn, double& dn) {
    cover((float)h);
    const double R2 = 4.0 * h * h, ih = 1.0 / h, norm = 1.0 / (MAP_PI * h * h * h);
    double s = 0.0, d = 0.0;
    auto add = [&](int node) {
      const double* c = S.com + 3 * (int64_t)node;
      const double dx = c[0] - px, dy = c[1] - py, dz = c[2] - pz;
      const double r2 = dx * dx + dy * dy + dz * dz;
      if (r2 >= R2) return;
      const double q = sqrt(r2) * ih;
      if (q < 1.0) {
        const double w = 1.0 - 1.5 * q * q + 0.75 * q * q * q;
        s += w;
        d += 3.0 * w + q * (2.25 * q * q - 3.0 * q);
      } else if (q < 2.0) {
        const double t = 2.0 - q, w = 0.25 * t * t * t;
        s += w;
        d += 3.0 * w - 0.75 * t * t * q;
      }
    };
    if (n >= 0)
      for (int j = lane; j < n; j += 32) add(W.node[j]);
    else
      scan([&](float, float, float, int node, bool on) { if (on) add(node); });
    nn = lanes_sum(s) * norm;
    dn = -lanes_sum(d) * norm * ih;
  }
};

// One warp per output slot holding an accepted node: Newton-Raphson on
// h = hfact n(h)^(-1/3) from Eq. (9)'s guess, bisection on [h0/16, 16 h0]
// when it fails, the guess itself when that has no sign change (Section
// III-C); then Halley's step on sum_b w = pi hfact^3 in FP64.  What FP32 cannot
// decide is solved once more in FP64.  The lanes hold identical sums, so the
// iteration is warp-uniform.
__global__ void __launch_bounds__(PS_WARPS * 32) pseudo_h(int64_t nout, const int32_t* __restrict__ node_of_slot, NodeSet S,
                         const unsigned long long* __restrict__ size_bits, const int32_t* __restrict__ parent,
                         const int32_t* __restrict__ level, const int64_t* __restrict__ nb, const double* __restrict__ hs,
                         int kmid, double hfact, double* oh) {
  __shared__ PseudoWarp sw[PS_WARPS];
  const int lane = threadIdx.x & 31;
  const int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (j >= nout) return;
  const int32_t nd = node_of_slot[j];
  if (nd < 0) return;  // extracted particle keeps its h
  const double x = S.com[3 * (int64_t)nd], y = S.com[3 * (int64_t)nd + 1], z = S.com[3 * (int64_t)nd + 2];
  const float hx = (float)x, hy = (float)y, hz = (float)z;
  PseudoSolve P{S, sw[threadIdx.x >> 5], lane, x, y, z, hx, (float)(x - (double)hx), hy, (float)(y - (double)hy),
                hz, (float)(z - (double)hz), 0.0};
  const double s_node = bitsd(size_bits[nd]);
  const double g0 = s_node > 0.0 ? hfact * 2.0 * s_node : hs[nb[nd]];
  if (S.use_kmid) {
    int32_t a = nd;
    while (level[a] > kmid) a = parent[a];
    P.rcut = 1.7320508075688772 * bitsd(size_bits[a]);
    const double r2h = 4.0 * hfact * s_node;
    if (P.rcut < r2h) {
      int32_t up = nd;
      for (int k = 0; k < 2 && parent[up] >= 0; ++k) up = parent[up];
      P.rcut = 4.0 * hfact * bitsd(size_bits[up]);
    }
  }
  const float hf_s = (float)hfact, hf_lo = (float)(hfact - (double)hf_s), hf3_s = (float)(hfact / 3.0);
  const double lo = g0 / 16.0, hi = g0 * 16.0;
  const float lo_s = (float)lo, hi_s = (float)hi;
  // (of a node by itself: g = h (1 - hfact pi^(1/3)), and Newton's step is h)
  const double g_alone = 1.0 - hfact * 1.4645918875615233;
  double h = g0;
  bool ok = false, root = true, sure = true;
  float h32 = (float)g0;
  for (int it = 0; it < 30; ++it) {
    float nn, dn;
    P.density(h32, nn, dn);
    if (P.alone && fabs(g_alone) > 1e-3) break;
    const float t = rcbrtf(nn);
    const float f = (h32 - hf_s * t) - hf_lo * t;
    const float fp = 1.f + hf3_s * (t * t) * (t * t) * dn;
    const float d = f / fp, hn = h32 - d;
    sure = P.sure && it < 24 && clear_step(h32, d, fp, lo_s, hi_s);
    if (!sure || !(hn >= lo_s && hn <= hi_s)) break;
    if (fabsf(hn - h32) < 1e-6f * hn) { h = (double)h32 - (double)d; ok = true; break; }
    h32 = hn;
  }
  if (!ok && sure) {
    auto g = [&](double v) {
      float nn, dn;
      P.density((float)v, nn, dn);
      const double w = P.alone ? v * g_alone : v - hfact * rcbrt((double)nn);
      sure = sure && P.sure && fabs(w) > 1e-4 * v;
      return w;
    };
    if (!(g(lo) < 0.0 && g(hi) > 0.0)) {
      h = g0;
      root = false;
    } else if (sure) {
      double a0 = lo, b0 = hi;
      for (int it = 0; it < 200; ++it) {
        const double mid = 0.5 * (a0 + b0);
        if (g(mid) < 0.0) a0 = mid; else b0 = mid;
        if (b0 - a0 < 1e-5 * mid) break;  // the FP64 steps below finish
      }
      h = 0.5 * (a0 + b0);
      sure = P.sure;  // (a sign taken wrongly is one at the root)
    }
  }
  if (root && sure) {
    // h <- h (1 + u), S' = -d/h, S'' = e/h^2; again while a step is so large that its cube shows
    const double target = MAP_PI * hfact * hfact * hfact;
    sure = false;
    for (int it = 0; it < 30; ++it) {
      double s, d, e;
      P.sums64(h, s, d, e);
      const double F = s - target;
      const double u = 2.0 * F * d / (2.0 * d * d - F * e);
      if (!(fabs(u) < 1e-2)) break;  // (no number where S' is 0)
      h += h * u;
      if (fabs(u) < 2e-6) { sure = h > lo && h < hi; break; }
    }
  }
  if (!sure) {
    h = g0;
    ok = false;
    for (int it = 0; it < 30; ++it) {
      double nn, dn;
      P.density64(h, nn, dn);
      const double t = rcbrt(nn), t2 = t * t;
      const double hn = h - (h - hfact * t) / (1.0 + hfact / 3.0 * (t2 * t2 * dn));
      if (!(hn >= lo && hn <= hi)) break;
      ok = fabs(hn - h) < 1e-10 * hn;
      h = hn;
      if (ok) break;
    }
    if (!ok) {
      auto g = [&](double v) {
        double nn, dn;
        P.density64(v, nn, dn);
        return v - hfact * rcbrt(nn);
      };
      h = g0;
      if (g(lo) < 0.0 && g(hi) > 0.0) {
        double a0 = lo, b0 = hi;
        for (int it = 0; it < 200; ++it) {
          const double mid = 0.5 * (a0 + b0);
          if (g(mid) < 0.0) a0 = mid; else b0 = mid;
          if (b0 - a0 < 1e-12 * mid) break;
        }
        h = 0.5 * (a0 + b0);
      }
    }
  }
  if (lane == 0) oh[j] = h;
}

__global__ void member_anc(int64_t nm, const int32_t* __restrict__ members, const int32_t* __restrict__ parent,
                           const int32_t* __restrict__ level, int kmid, int64_t mid_begin, uint64_t* key, int32_t* val) {
  int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j >= nm) return;
  int32_t a = members[j];
  while (level[a] > kmid) a = parent[a];
  key[j] = (uint64_t)(a - mid_begin);
  val[j] = members[j];
}

__global__ void mid_ranges(int64_t nm, int64_t nmid, const uint64_t* __restrict__ key_sorted, int64_t* off) {
  // off[k] = first j with key >= k (lower bound), for k in [0, nmid]
  int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k > nmid) return;
  int64_t lo = 0, hi = nm;
  while (lo < hi) {
    int64_t m = (lo + hi) >> 1;
    if (key_sorted[m] < (uint64_t)k) lo = m + 1; else hi = m;
  }
  off[k] = lo;
}

__global__ void min_member_level(int64_t nm, const int32_t* __restrict__ members, const int32_t* __restrict__ level,
                                 unsigned long long* out) {
  int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j >= nm) return;
  atomicMin(out, (unsigned long long)level[members[j]]);
}

}  // namespace

int pseudo_run(map_ctx* ctx, const map_particles* full, const map_walk* walk, map_particles* out, int32_t* kind,
               int64_t* ident, int64_t* n_pseudo, cudaStream_t s) {
  const int nsrc = walk->nsrc, nreg = walk->nregion;
  const int64_t n = full->n;
  MAP_TRY(tree_build(ctx, full->x, full->y, full->z, full->m, full->h, n, s, true));
  DevTree& T = ctx->tree;
  const int64_t nn = T.nnodes;
  const int tpb = 256;
  double* d_src;
  int8_t *open, *status;
  int64_t *head, *slot, *mpos;
  int32_t *is_head, *node_of_slot, *mflag, *members;
  MAP_TRY(ensure_t(ctx, ctx->ws_misc[1], 3 * nsrc + 5 * nreg, &d_src));
  MAP_TRY(ensure_t(ctx, ctx->ws_misc[2], 2 * nn, &open));
  status = open + nn;
  MAP_TRY(ensure_t(ctx, ctx->ws_misc[3], 2 * (n + 1), &head));
  slot = head + (n + 1);
  MAP_TRY(ensure_t(ctx, ctx->ws_misc[4], 2 * (n + 1), &is_head));
  node_of_slot = is_head + (n + 1);
  MAP_TRY(ensure_t(ctx, ctx->ws_misc[5], 2 * (nn + 1), &mflag));
  members = mflag + (nn + 1);
  MAP_TRY(ensure_t(ctx, ctx->ws_misc[6], nn + 1, &mpos));
  CUDA_TRY(cudaMemcpyAsync(d_src, walk->src, 3 * nsrc * sizeof(double), cudaMemcpyHostToDevice, s));
  if (nreg > 0)
    CUDA_TRY(cudaMemcpyAsync(d_src + 3 * nsrc, walk->regions, 5 * nreg * sizeof(double), cudaMemcpyHostToDevice, s));
  const WalkRule rule{d_src, nsrc, ctx->cfg.theta, walk->r_part, walk->r_leaf, d_src + 3 * nsrc, nreg};
  open_flags<<<nblk(nn, tpb), tpb, 0, s>>>(nn, T.com, T.size_bits, T.nchild, rule, open); ++ctx->launches;
  walk_status<<<nblk(nn, tpb), tpb, 0, s>>>(nn, T.parent, open, T.nchild, status); ++ctx->launches;
  CUDA_TRY(cudaMemsetAsync(is_head, 0, (n + 1) * sizeof(int32_t), s));
  mark_heads<<<nblk(nn, tpb), tpb, 0, s>>>(nn, status, T.begin, T.end, head, is_head); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  size_t tb = 0;
  CUDA_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tb, is_head, slot, n + 1, s));
  MAP_TRY(ctx_ensure(ctx, ctx->cub_tmp, tb));
  CUDA_TRY(cub::DeviceScan::ExclusiveSum(ctx->cub_tmp.p, tb, is_head, slot, n + 1, s));
  CUDA_TRY(cudaMemcpyAsync(ctx->h_scratch, slot + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  const int64_t nout = ctx->h_scratch[0];
  *n_pseudo = nout;
  if (nout > out->n) return MAP_ECAPACITY;
  if (!out->x || !out->y || !out->z || !out->h) return MAP_EINVAL;
  double* om = const_cast<double*>(out->m);
  if (!om) return MAP_EINVAL;
  write_pseudo<<<nblk(n, tpb), tpb, 0, s>>>(n, head, is_head, slot, T.com, T.mass, T.label, T.xs, T.ys, T.zs, T.ms,
                                           T.hs, T.idx, const_cast<double*>(out->x), const_cast<double*>(out->y),
                                           const_cast<double*>(out->z), om, out->h, kind, ident, node_of_slot); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  // node set for the h solve
  member_flags<<<nblk(nn, tpb), tpb, 0, s>>>(nn, status, mflag); ++ctx->launches;
  CUDA_TRY(cudaMemsetAsync(mflag + nn, 0, sizeof(int32_t), s));
  tb = 0;
  CUDA_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tb, mflag, mpos, nn + 1, s));
  MAP_TRY(ctx_ensure(ctx, ctx->cub_tmp, tb));
  CUDA_TRY(cub::DeviceScan::ExclusiveSum(ctx->cub_tmp.p, tb, mflag, mpos, nn + 1, s));
  member_write<<<nblk(nn, tpb), tpb, 0, s>>>(nn, mflag, mpos, members); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  CUDA_TRY(cudaMemcpyAsync(ctx->h_scratch, mpos + nn, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  const int64_t nm = ctx->h_scratch[0];
  NodeSet S{};
  S.nm = nm;
  S.com = T.com;
  const int32_t* scanned = members;
  S.use_kmid = nm > ctx->cfg.ngb_bruteforce_max ? 1 : 0;
  int kmid = 0;
  if (S.use_kmid) {
    unsigned long long* d_min = ctx->d_counters + 5;
    unsigned long long big = 1ULL << 40;
    CUDA_TRY(cudaMemcpyAsync(d_min, &big, sizeof(big), cudaMemcpyHostToDevice, s));
    min_member_level<<<nblk(nm, tpb), tpb, 0, s>>>(nm, members, T.level, d_min); ++ctx->launches;
    CUDA_TRY(cudaMemcpyAsync(ctx->h_scratch, d_min, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaStreamSynchronize(s));
    kmid = (int)ctx->h_scratch[0] - 1;
    if (kmid < 0) kmid = 0;
    S.mid_begin = T.level_begin[kmid];
    S.mid_end = T.level_begin[kmid + 1];
    const int64_t nmid = S.mid_end - S.mid_begin;
    uint64_t *kin, *kout;
    int32_t *vin, *vout;
    int64_t* moff;
    MAP_TRY(ensure_t(ctx, ctx->ws_pairs[4], nm, &kin));
    MAP_TRY(ensure_t(ctx, ctx->ws_pairs[5], nm, &kout));
    MAP_TRY(ensure_t(ctx, ctx->ws_pairs[6], nm, &vin));
    MAP_TRY(ensure_t(ctx, ctx->ws_pairs[7], nm, &vout));
    MAP_TRY(ensure_t(ctx, ctx->ws_misc[7], nmid + 1, &moff));
    member_anc<<<nblk(nm, tpb), tpb, 0, s>>>(nm, members, T.parent, T.level, kmid, S.mid_begin, kin, vin); ++ctx->launches;
    tb = 0;
    CUDA_TRY(cub::DeviceRadixSort::SortPairs(nullptr, tb, kin, kout, vin, vout, nm, 0, 40, s));
    MAP_TRY(ctx_ensure(ctx, ctx->cub_tmp, tb));
    CUDA_TRY(cub::DeviceRadixSort::SortPairs(ctx->cub_tmp.p, tb, kin, kout, vin, vout, nm, 0, 40, s));
    mid_ranges<<<nblk(nmid + 1, tpb), tpb, 0, s>>>(nm, nmid, kout, moff); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
    S.mid_off = moff;
    scanned = vout;
  }
  float4* points;
  MAP_TRY(ensure_t(ctx, ctx->ws_pairs[2], 2 * nm, &points));
  S.hi = points;
  S.lo = points + nm;
  if (nm > 0) {
    member_points<<<nblk(nm, tpb), tpb, 0, s>>>(nm, scanned, T.com, points, points + nm); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
  }
  pseudo_h<<<nblk(nout * 32, PS_WARPS * 32), PS_WARPS * 32, 0, s>>>(nout, node_of_slot, S, T.size_bits, T.parent, T.level, T.begin, T.hs,
                                           kmid, ctx->cfg.hfact, out->h); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  return MAP_OK;
}
