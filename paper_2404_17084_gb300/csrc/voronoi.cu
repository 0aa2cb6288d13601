// Grid construction on the device (Section II-A): the Voronoi grid generated
// by point sites, clipped to the unit cube, after merging tightly packed
// sites and a number of Lloyd iterations.
//
// Each cell is built by one warp in shared memory: the cube, relative to the
// site, cut by the bisector planes of the neighbouring sites.  Neighbours come
// from a uniform bucket grid: first the 32 nearest of the 27 buckets around the
// site, nearest first, then every other site ring by ring; a site at distance D
// cuts along a plane at D/2, so once every unvisited site is at least twice
// the cell's largest vertex radius away the cell is final.  A cut keeps the
// part n.x <= d: each face loop is clipped in turn (a vertex within a relative
// 1e-13 of the plane counts as on it), and the vertices on the plane, ordered
// by angle around their mean, form the new face.  At the end vertices within a
// relative 1e-11 are welded and faces left with fewer than three vertices
// dropped.  Walls have exact planes; a bisector's plane passes through the
// midpoint of its two sites.
//
// What bounds it is the FP64 pipe (1.8 lanes per clock and SM: an FP64
// instruction of a warp costs as much as 70 others of its scheduler) and, behind
// it, the chain of a cell's cuts.  So all that only selects runs in FP32 with
// margins that keep it exact -- FP32's rounding, and the split's own 8e-15, which
// counts once sites are closer than 1e-9 or so: distances on hi/lo-split
// coordinates (buckets and sites beyond reach), and each remaining site's plane
// against all vertices of the current cell, 32 sites at a time, one per lane -- a
// plane that clears every vertex clears every later, smaller cell too.  About 70 sites come
// within reach of a cell and 17 cut it; those 17 take FP64, with lanes over the
// vertices, the crossing edges and the faces, about 25 FP64 instructions each.
// One thread per cell with its polyhedra in local memory (3.9 of 32 lanes busy)
// took 49 ms per tessellation of 130,003 clumpy sites and 14 ms for 1000; this
// takes 10 and 0.5 ms (2^20 sites 520 -> 106 ms, the whole call).
//
// Lloyd iteration: every site moves to its cell's centroid (the
// volume-weighted mean of the tetrahedra site / fan triangle of a face).
// Merging: a site within merge_tol of any site of lower index is dropped.
//
// The cells are written to fixed slots (VOR_MAXV vertices, VOR_MAXF faces,
// VOR_MAXL loop entries); a cell that outgrows them makes the call fail with
// MAP_ECAPACITY.  A scan then packs the slots into the CSR layout of map_grid,
// which the resident-grid preparation takes as it is.
#include <cub/cub.cuh>

#include "dmath.cuh"
#include "internal.cuh"

namespace {

constexpr int VOR_MAXV = 96;
constexpr int VOR_MAXF = 48;
constexpr int VOR_MAXL = 320;
constexpr int VOR_NEAR = 32;  // nearest sites of the surrounding 27 buckets, cut first and in order

// a cell as written to its slot (site-relative vertices)
struct Slot {
  int nv, nf, nl, ok;
};

struct Buckets {
  int G;
  const int64_t* off;    // [G^3 + 1]
  const int32_t* sites;  // site indices grouped by bucket, ascending within one
  const float4* hi;      // in that order: x, y, z rounded to FP32, site index
  const float4* lo;      // what the rounding left
};

__host__ __device__ __forceinline__ int bucket_coord(double v, int G) {
  int b = (int)floor(v * G);
  return b < 0 ? 0 : (b >= G ? G - 1 : b);
}

__global__ void vor_bucket_keys(int64_t n, const double* __restrict__ x, const double* __restrict__ y,
                                const double* __restrict__ z, int G, int32_t* key, int32_t* idx) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  key[i] = (bucket_coord(z[i], G) * G + bucket_coord(y[i], G)) * G + bucket_coord(x[i], G);
  idx[i] = (int32_t)i;
}

// off[b] = first position whose bucket is >= b
__global__ void vor_bucket_bounds(int64_t n, int64_t nb, const int32_t* __restrict__ key, int64_t* off) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k > n) return;
  const int64_t prev = k == 0 ? -1 : key[k - 1];
  const int64_t cur = k == n ? nb : key[k];
  for (int64_t b = prev + 1; b <= cur; ++b) off[b] = k;
}

// the sites' coordinates in bucket order, as FP32 hi/lo pairs: the difference
// of two of them, (hi - hi) + (lo - lo), is good to FP32's relative accuracy and
// SPLIT_ERR, whichever is larger (lo is rounded at 2^-50, a difference of two
// lo at 2^-49, on each axis)
constexpr float SPLIT_ERR = 8e-15f;

__global__ void vor_split(int64_t n, const double* __restrict__ x, const double* __restrict__ y,
                          const double* __restrict__ z, const int32_t* __restrict__ sites, float4* hi, float4* lo) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= n) return;
  const int32_t i = sites[k];
  const double px = x[i], py = y[i], pz = z[i];
  const float hx = (float)px, hy = (float)py, hz = (float)pz;
  hi[k] = make_float4(hx, hy, hz, __int_as_float(i));
  lo[k] = make_float4((float)(px - (double)hx), (float)(py - (double)hy), (float)(pz - (double)hz), 0.f);
}

// squared distance of p to the box of buckets [bx0, bx1] x {by} x {bz}, less a
// margin: every site of those buckets is at least that far away
__device__ __forceinline__ float box_dist2(float px, float py, float pz, int bx0, int bx1, int by, int bz, float bw) {
  const float dx = fmaxf(fmaxf(bx0 * bw - px, px - (bx1 + 1) * bw), 0.f);
  const float dy = fmaxf(fmaxf(by * bw - py, py - (by + 1) * bw), 0.f);
  const float dz = fmaxf(fmaxf(bz * bw - pz, pz - (bz + 1) * bw), 0.f);
  const float d = sqrtf(dx * dx + dy * dy + dz * dz) - 1e-6f;
  return d > 0.f ? d * d * 0.99999f : 0.f;
}

// merging: drop site i when a site of lower index lies within tol (the buckets
// that reach within tol of it; FP32 distances rule out the sites beyond it by
// more than their own error, FP64 decides the rest)
__global__ void vor_merge_flags(int64_t n, const double* __restrict__ x, const double* __restrict__ y,
                                const double* __restrict__ z, Buckets B, double tol, int64_t* keep) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i > n) return;
  if (i == n) { keep[n] = 0; return; }
  const int G = B.G;
  const double px = x[i], py = y[i], pz = z[i];
  const int bx = bucket_coord(px, G), by = bucket_coord(py, G), bz = bucket_coord(pz, G);
  const float hx = (float)px, hy = (float)py, hz = (float)pz;
  const float lx = (float)(px - (double)hx), ly = (float)(py - (double)hy), lz = (float)(pz - (double)hz);
  const float bw = 1.0f / G, reach = ((float)tol + SPLIT_ERR) * 1.00001f, far2 = reach * reach;
  bool k = true;
  for (int dz = -1; dz <= 1 && k; ++dz)
    for (int dy = -1; dy <= 1 && k; ++dy)
      for (int dx = -1; dx <= 1 && k; ++dx) {
        const int cx = bx + dx, cy = by + dy, cz = bz + dz;
        if (cx < 0 || cy < 0 || cz < 0 || cx >= G || cy >= G || cz >= G) continue;
        if (box_dist2(hx, hy, hz, cx, cx, cy, cz, bw) > far2) continue;
        const int64_t b = ((int64_t)cz * G + cy) * G + cx;
        for (int64_t q = B.off[b]; q < B.off[b + 1]; ++q) {
          const float4 H = __ldg(B.hi + q);
          const int32_t j = __float_as_int(H.w);
          if (j >= i) continue;
          const float4 D = __ldg(B.lo + q);
          const float fx = (H.x - hx) + (D.x - lx), fy = (H.y - hy) + (D.y - ly), fz = (H.z - hz) + (D.z - lz);
          if (fx * fx + fy * fy + fz * fz > far2) continue;
          const double ex = x[j] - px, ey = y[j] - py, ez = z[j] - pz;
          if (ex * ex + ey * ey + ez * ez < tol * tol) { k = false; break; }
        }
      }
  keep[i] = k ? 1 : 0;
}

__global__ void vor_merge_pack(int64_t n, const int64_t* __restrict__ keep, const int64_t* __restrict__ pos,
                               const double* __restrict__ x, const double* __restrict__ y, const double* __restrict__ z,
                               double* sx, double* sy, double* sz, int64_t* kept) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n || !keep[i]) return;
  const int64_t j = pos[i];
  sx[j] = x[i]; sy[j] = y[i]; sz[j] = z[i];
  if (kept) kept[j] = i;
}

struct SlotArrays {
  Slot* info;
  double* v;            // 3 * VOR_MAXV per cell (site-relative)
  unsigned char* loop;  // VOR_MAXL per cell
  short* fs;            // VOR_MAXF per cell
  unsigned char* fl;    // VOR_MAXF per cell
  int* nb;              // VOR_MAXF per cell
};

constexpr int VW = 4;  // warps (cells) per block

// One warp's cell: the polyhedron before and after a cut.
struct CellWarp {
  double x[2][VOR_MAXV], y[2][VOR_MAXV], z[2][VOR_MAXV], r2[2][VOR_MAXV];  // vertices, squared radii
  double s[VOR_MAXV];                 // signed distances to the cut's plane
  float4 v32[VOR_MAXV];               // the vertices in FP32 (the screens)
  int nb[2][VOR_MAXF];                // neighbour site, or -1-w for wall w
  short fs[2][VOR_MAXF];              // first loop entry of each face
  unsigned char fl[2][VOR_MAXF];      // loop length
  unsigned char loop[2][VOR_MAXL];
  unsigned char face[2][VOR_MAXL];    // the face of each loop entry
  unsigned char cut[VOR_MAXL];        // the vertex a cut makes on the edge that starts here (255: none)
  unsigned char remap[VOR_MAXV];
  signed char cls[VOR_MAXV];          // side of the plane: -1 kept, 0 on it, 1 cut off
  unsigned char on[VOR_MAXV];         // the new face's vertices
  short key[2 * VOR_MAXV];            // crossing edges in loop order
  int b, nv, nf, nl;                  // the copy in use and its counts
  double rmax2;                       // the largest squared radius
};

constexpr unsigned VFULL = 0xffffffffu;

__device__ __forceinline__ int64_t warp_max(int64_t v) {
  for (int o = 16; o > 0; o >>= 1) {
    const int64_t w = __shfl_xor_sync(VFULL, v, o);
    v = w > v ? w : v;
  }
  return v;
}

// The lanes' counts laid end to end: end = the end of this lane's stretch;
// returns the total.
__device__ __forceinline__ int warp_ends(int count, int& end) {
  end = count;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(VFULL, end, o);
    if ((int)(threadIdx.x & 31) >= o) end += v;
  }
  return __shfl_sync(VFULL, end, 31);
}
// The lane whose stretch holds place f (31 past the end), and f's place in it.
__device__ __forceinline__ int warp_owner(int f, int end, int count, int& rest) {
  int l = 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    if (__shfl_sync(VFULL, end, l + o - 1) <= f) l += o;
  rest = f - (__shfl_sync(VFULL, end, l) - __shfl_sync(VFULL, count, l));
  return l;
}

__device__ __forceinline__ double dist2(double ex, double ey, double ez) {
  return __fma_rn(ez, ez, __fma_rn(ey, ey, __dmul_rn(ex, ex)));
}

__device__ __forceinline__ float rmax_of(double rmax2) { return sqrtf(dm::f32(rmax2)); }
__device__ __forceinline__ float4 f32_of(double x, double y, double z) {
  return make_float4(dm::f32(x), dm::f32(y), dm::f32(z), 0.f);
}

__device__ __forceinline__ void cell_box(CellWarp& W, double sx, double sy, double sz) {
  const int lane = threadIdx.x & 31;
  int64_t r = 0;
  if (lane < 8) {
    const double x = (lane & 1) ? 1.0 - sx : -sx, y = (lane & 2) ? 1.0 - sy : -sy, z = (lane & 4) ? 1.0 - sz : -sz;
    const double r2 = dist2(x, y, z);
    W.x[0][lane] = x; W.y[0][lane] = y; W.z[0][lane] = z; W.r2[0][lane] = r2;
    W.v32[lane] = f32_of(x, y, z);
    r = dm::bits(r2);
  }
  // loops counter-clockwise seen from outside: x<=1, x>=0, y<=1, y>=0, z<=1, z>=0
  // (a hexadecimal digit per entry, from the last to the first)
  if (lane < 24) {
    const uint64_t L = lane < 12 ? 0x376226405731ull : 0x132067544510ull;
    W.loop[0][lane] = (unsigned char)(L >> (4 * (lane % 12)) & 15u);
    W.face[0][lane] = (unsigned char)(lane >> 2);
  }
  if (lane < 6) { W.fs[0][lane] = (short)(4 * lane); W.fl[0][lane] = 4; W.nb[0][lane] = -1 - lane; }
  r = warp_max(r);
  if (lane == 0) { W.b = 0; W.nv = 8; W.nf = 6; W.nl = 24; W.rmax2 = dm::from_bits(r); }
  __syncwarp();
}

// Whether the plane (n, d) (unit n, FP32) may cut the cell: false only when it
// clears every vertex by more than FP32's rounding and err, what the plane's
// own error may move it by within rmax of the site.
__device__ __forceinline__ bool may_cut(const CellWarp& W, int nv, float nx, float ny, float nz, float d, float rmax,
                                        float err = 0.f) {
  float s = -INFINITY;
#pragma unroll 4
  for (int i = 0; i < nv; ++i) {
    const float4 v = W.v32[i];
    s = fmaxf(s, fmaf(nx, v.x, fmaf(ny, v.y, nz * v.z)));
  }
  return s > d - (1e-5f * (rmax + d) + err);
}

// Cut the cell by n.x <= d.  Returns 0 when nothing changed, 1 when the cell
// was cut, -1 on overflow.  Lanes over vertices, then over loop entries (edges
// of a face), then over faces.
__device__ __noinline__ int cell_clip(CellWarp& W, double nx, double ny, double nz, double d, int nbid) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int b = W.b, q = b ^ 1, pv = W.nv, pf = W.nf, pl = W.nl;
  const double tol = dm::f64(1e-13f * rmax_of(W.rmax2));
  // the vertices' sides
  bool any = false;
  for (int i0 = 0; i0 < pv; i0 += 32) {
    const int i = i0 + lane;
    int c = -1;
    if (i < pv) {
      const double s = fma(nx, W.x[b][i], fma(ny, W.y[b][i], fma(nz, W.z[b][i], -d)));
      c = dm::gt(dm::neg(tol), s) ? -1 : (dm::gt(s, tol) ? 1 : 0);
      W.s[i] = s;
      W.cls[i] = (signed char)c;
    }
    any = any || __any_sync(VFULL, c > 0);
  }
  if (!any) return 0;
  // the kept ones, in order; those on the plane start the new face
  int nv = 0, non = 0;
  int64_t r2 = 0;
  __syncwarp();
  for (int i0 = 0; i0 < pv; i0 += 32) {
    const int i = i0 + lane;
    const int c = i < pv ? (int)W.cls[i] : 1;
    const unsigned mk = __ballot_sync(VFULL, c <= 0), mo = __ballot_sync(VFULL, c == 0);
    if (c <= 0) {
      const int k = nv + __popc(mk & lt);
      const double x = W.x[b][i], y = W.y[b][i], z = W.z[b][i], r = W.r2[b][i];
      W.remap[i] = (unsigned char)k;
      W.x[q][k] = x; W.y[q][k] = y; W.z[q][k] = z; W.r2[q][k] = r;
      if (c == 0) W.on[non + __popc(mo & lt)] = (unsigned char)k;
      r2 = dm::bits(r) > r2 ? dm::bits(r) : r2;
    }
    nv += __popc(mk);
    non += __popc(mo);
  }
  __syncwarp();
  // crossing edges: every edge is in two faces; the first in loop order makes
  // the vertex.  Their list (loop entry) goes through W.key when it exceeds a
  // warp.
  int nx_ = 0;
  for (int e0 = 0; e0 < pl; e0 += 32) {
    const int e = e0 + lane;
    bool cross = false;
    if (e < pl) {
      const int f = W.face[b][e], l = W.fs[b][f] + W.fl[b][f] - 1;
      const int a = W.loop[b][e], c = W.loop[b][e == l ? W.fs[b][f] : e + 1];
      cross = W.cls[a] * W.cls[c] < 0;
      W.cut[e] = 255;
    }
    const unsigned m = __ballot_sync(VFULL, cross);
    if (cross) {
      const int k = nx_ + __popc(m & lt);
      if (k < 2 * VOR_MAXV) W.key[k] = (short)e;
    }
    nx_ += __popc(m);
  }
  if (nx_ > 2 * VOR_MAXV) return -1;
  __syncwarp();
  const int nkept = nv;
  for (int k0 = 0; k0 < nx_; k0 += 32) {
    const int k = k0 + lane;
    const bool on = k < nx_;
    int a = 0, c = 0, e = 0, first = k;
    if (on) {
      e = W.key[k];
      const int f = W.face[b][e], l = W.fs[b][f] + W.fl[b][f] - 1;
      a = W.loop[b][e];
      c = W.loop[b][e == l ? W.fs[b][f] : e + 1];
    }
    // the same edge earlier in the list (from the face on its other side)
    const int ends = (a < c ? a << 8 | c : c << 8 | a);
    first = k0 + __ffs(__match_any_sync(VFULL, on ? ends : 1 << 16 | lane)) - 1;
    for (int j = 0; on && j < k0; ++j) {
      const int ej = W.key[j], fj = W.face[b][ej], lj = W.fs[b][fj] + W.fl[b][fj] - 1;
      const int aj = W.loop[b][ej], cj = W.loop[b][ej == lj ? W.fs[b][fj] : ej + 1];
      if ((aj == c && cj == a) || (aj == a && cj == c)) { first = j; break; }
    }
    const unsigned mf = __ballot_sync(VFULL, on && first == k);
    const int id = nv + __popc(mf & lt);
    if (nv + __popc(mf) > VOR_MAXV) return -1;
    if (on && first == k) {
      const double sa = W.s[a], t = dm::quot(sa, sa - W.s[c]);
      const double xa = W.x[b][a], ya = W.y[b][a], za = W.z[b][a];
      const double x = fma(W.x[b][c] - xa, t, xa), y = fma(W.y[b][c] - ya, t, ya), z = fma(W.z[b][c] - za, t, za);
      const double r = dist2(x, y, z);
      W.x[q][id] = x; W.y[q][id] = y; W.z[q][id] = z; W.r2[q][id] = r;
      W.cut[e] = (unsigned char)id;
      r2 = dm::bits(r) > r2 ? dm::bits(r) : r2;
    }
    nv += __popc(mf);
    __syncwarp();
    if (on && first != k) W.cut[e] = W.cut[W.key[first]];
    __syncwarp();
  }
  for (int i = nkept + lane; i < nv; i += 32) W.on[non + i - nkept] = (unsigned char)i;
  non += nv - nkept;
  // the faces' loops, one face per lane: entries counted, then written;
  // consecutive duplicates and loops of fewer than three are dropped
  int nf = 0, nl = 0;
  bool stray = false;
  for (int f0 = 0; f0 < pf; f0 += 32) {
    const int f = f0 + lane;
    int len = 0, head = -1, last = -1, fb = 0, L = 0;
    if (f < pf) {
      fb = W.fs[b][f]; L = W.fl[b][f];
      for (int k = 0; k < L; ++k) {
        const int a = W.loop[b][fb + k], x = W.cut[fb + k];
        if (W.cls[a] <= 0) {
          const int v = W.remap[a];
          if (v != last) { last = v; if (!len++) head = v; }
        }
        if (x != 255 && x != last) { last = x; if (!len++) head = x; }
      }
      // (a loop's end that repeats its head; more of them would be dropped one by one)
      if (len > 1 && last == head) --len;
    }
    const bool keep = len >= 3;
    stray = stray || __any_sync(VFULL, len > 0 && !keep);
    const unsigned mk = __ballot_sync(VFULL, keep);
    int at = keep ? len : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(VFULL, at, o);
      if (lane >= o) at += v;
    }
    const int tot = __shfl_sync(VFULL, at, 31);
    if (nf + __popc(mk) > VOR_MAXF || nl + tot > VOR_MAXL) return -1;
    if (keep) {
      const int g = nf + __popc(mk & lt);
      int w = nl + at - len;
      const int end = w + len;
      W.fs[q][g] = (short)w;
      W.fl[q][g] = (unsigned char)len;
      W.nb[q][g] = W.nb[b][f];
      last = -1;
      auto put = [&](int v) {
        if (v == last || w >= end) return;
        last = v;
        W.loop[q][w] = (unsigned char)v;
        W.face[q][w] = (unsigned char)g;
        ++w;
      };
      for (int k = 0; k < L; ++k) {
        const int a = W.loop[b][fb + k], x = W.cut[fb + k];
        if (W.cls[a] <= 0) put(W.remap[a]);
        if (x != 255) put(x);
      }
    }
    nf += __popc(mk);
    nl += tot;
  }
  __syncwarp();
  // the new face: the vertices on the plane ordered by angle around their
  // mean, from -pi.  FP32 on offsets from the first of them (FP64 differences)
  // decides unless two angles, or an angle and -pi, are close; FP64 then.
  if (non >= 3) {
    if (nf >= VOR_MAXF || nl + non > VOR_MAXL) return -1;
    const int v0 = W.on[0];
    const double X0 = W.x[q][v0], Y0 = W.y[q][v0], Z0 = W.z[q][v0];
    const bool flat = dm::gt(0.6, dm::abs2(nx));  // the axis the in-plane frame starts from: x, or y
    bool done = false;
    if (non <= 32) {
      const int v = W.on[lane < non ? lane : 0];
      const float px = dm::f32(W.x[q][v] - X0), py = dm::f32(W.y[q][v] - Y0), pz = dm::f32(W.z[q][v] - Z0);
      float cx = lane < non ? px : 0.f, cy = lane < non ? py : 0.f, cz = lane < non ? pz : 0.f;
      for (int o = 16; o > 0; o >>= 1) {
        cx += __shfl_xor_sync(VFULL, cx, o); cy += __shfl_xor_sync(VFULL, cy, o); cz += __shfl_xor_sync(VFULL, cz, o);
      }
      const float in = 1.0f / non;
      const float rx = px - cx * in, ry = py - cy * in, rz = pz - cz * in;
      const float fx = dm::f32(nx), fy = dm::f32(ny), fz = dm::f32(nz), bx = flat ? 1.f : 0.f, by = 1.f - bx;
      float ux = -fz * by, uy = fz * bx, uz = fx * by - fy * bx;  // n x a
      const float un = rsqrtf(ux * ux + uy * uy + uz * uz);
      ux *= un; uy *= un; uz *= un;
      const float wx = fy * uz - fz * uy, wy = fz * ux - fx * uz, wz = fx * uy - fy * ux;
      const float pu = rx * ux + ry * uy + rz * uz, pw = rx * wx + ry * wy + rz * wz;
      float sc = lane < non ? fabsf(pu) + fabsf(pw) : 0.f;
      float big = sc;
      for (int o = 16; o > 0; o >>= 1) big = fmaxf(big, __shfl_xor_sync(VFULL, big, o));
      // a monotone stand-in for the angle: -2 .. 2 from -pi to pi
      const float tq = pu / sc;
      const float an = pw < 0.f ? tq - 1.f : 1.f - tq;
      // FP32's error of an is some 1e-6 big / sc
      const float err = 2e-5f * big;
      bool close = lane < non && (!(sc > 100.f * err) || (pu < 0.f && fabsf(pw) < err));
      int rank = 0;
      for (int j = 0; j < non; ++j) {
        const float aj = __shfl_sync(VFULL, an, j), sj = __shfl_sync(VFULL, sc, j);
        rank += aj < an;
        close = close || (lane < non && j != lane && fabsf(aj - an) * fminf(sj, sc) < err);
      }
      if (!__any_sync(VFULL, close)) {
        if (lane < non) { W.loop[q][nl + rank] = (unsigned char)v; W.face[q][nl + rank] = (unsigned char)nf; }
        done = true;
      }
    }
    if (!done) {
      // FP64: angles in W.s (no longer needed), ranks with ties by vertex number
      double cx = 0.0, cy = 0.0, cz = 0.0;
      for (int i = 0; i < non; ++i) { cx += W.x[q][W.on[i]]; cy += W.y[q][W.on[i]]; cz += W.z[q][W.on[i]]; }
      cx /= non; cy /= non; cz /= non;
      const double ax = flat ? 1.0 : 0.0, ay = 1.0 - ax;
      double ux = -nz * ay, uy = nz * ax, uz = nx * ay - ny * ax;
      const double un = sqrt(ux * ux + uy * uy + uz * uz);
      ux /= un; uy /= un; uz /= un;
      const double wx = ny * uz - nz * uy, wy = nz * ux - nx * uz, wz = nx * uy - ny * ux;
      __syncwarp();
      for (int i = lane; i < non; i += 32) {
        const int v = W.on[i];
        const double rx = W.x[q][v] - cx, ry = W.y[q][v] - cy, rz = W.z[q][v] - cz;
        W.s[i] = atan2(rx * wx + ry * wy + rz * wz, rx * ux + ry * uy + rz * uz);
      }
      __syncwarp();
      for (int i = lane; i < non; i += 32) {
        int rank = 0;
        for (int j = 0; j < non; ++j) rank += W.s[j] < W.s[i] || (W.s[j] == W.s[i] && j < i);
        W.loop[q][nl + rank] = W.on[i];
        W.face[q][nl + rank] = (unsigned char)nf;
      }
    }
    if (lane == 0) { W.fs[q][nf] = (short)nl; W.fl[q][nf] = (unsigned char)non; W.nb[q][nf] = nbid; }
    ++nf;
    nl += non;
  } else {
    stray = stray || non > 0;
  }
  __syncwarp();
  if (stray) {
    // a face lost its last one or two vertices: drop those no face refers to
    for (int i = lane; i < nv; i += 32) W.remap[i] = 255;
    __syncwarp();
    for (int e = lane; e < nl; e += 32) W.remap[W.loop[q][e]] = 0;
    __syncwarp();
    int k = 0;
    r2 = 0;
    for (int i0 = 0; i0 < nv; i0 += 32) {
      const int i = i0 + lane;
      const bool used = i < nv && W.remap[i] == 0;
      const unsigned m = __ballot_sync(VFULL, used);
      double x = 0, y = 0, z = 0, r = 0;
      if (used) { x = W.x[q][i]; y = W.y[q][i]; z = W.z[q][i]; r = W.r2[q][i]; }
      __syncwarp();
      if (used) {
        const int t = k + __popc(m & lt);  // t <= i: entries below i0 + 32 have been read
        W.remap[i] = (unsigned char)t;
        W.x[q][t] = x; W.y[q][t] = y; W.z[q][t] = z; W.r2[q][t] = r;
        r2 = dm::bits(r) > r2 ? dm::bits(r) : r2;
      }
      k += __popc(m);
      __syncwarp();
    }
    nv = k;
    for (int e = lane; e < nl; e += 32) W.loop[q][e] = W.remap[W.loop[q][e]];
    __syncwarp();
  }
  for (int i = lane; i < nv; i += 32)
    W.v32[i] = f32_of(W.x[q][i], W.y[q][i], W.z[q][i]);
  r2 = warp_max(r2);
  if (lane == 0) { W.b = q; W.nv = nv; W.nf = nf; W.nl = nl; W.rmax2 = dm::from_bits(r2); }
  __syncwarp();
  return 1;
}

// Welds vertices within a relative 1e-11 and drops faces left with fewer than
// three (lane 0 alone, only when two vertices are that close).
__device__ __forceinline__ void cell_weld(CellWarp& W) {
  const int lane = threadIdx.x & 31;
  const int b = W.b;
  const double scale = sqrt(fmax(W.rmax2, 1e-300));
  const double tol2 = (1e-11 * scale) * (1e-11 * scale);
  bool weld = false;
  const float t32 = 1e-5f * (float)scale;
  for (int i = lane; i < W.nv; i += 32) {
    const float4 v = W.v32[i];
    for (int j = 0; j < i; ++j) {
      const float4 u = W.v32[j];
      if (fabsf(u.x - v.x) < t32 && fabsf(u.y - v.y) < t32 && fabsf(u.z - v.z) < t32)
        weld = weld || dist2(W.x[b][i] - W.x[b][j], W.y[b][i] - W.y[b][j], W.z[b][i] - W.z[b][j]) < tol2;
    }
  }
  if (__any_sync(VFULL, weld)) {
    if (lane == 0) {
      for (int i = 0; i < W.nv; ++i) {
        W.remap[i] = (unsigned char)i;
        for (int j = 0; j < i; ++j)
          if (W.remap[j] == j &&
              dist2(W.x[b][i] - W.x[b][j], W.y[b][i] - W.y[b][j], W.z[b][i] - W.z[b][j]) < tol2) {
            W.remap[i] = (unsigned char)j;
            break;
          }
      }
      int nf = 0, nl = 0;
      for (int f = 0; f < W.nf; ++f) {
        const int start = nl, fb = W.fs[b][f];
        for (int k = 0; k < W.fl[b][f]; ++k) {
          const unsigned char r = W.remap[W.loop[b][fb + k]];
          if (nl > start && W.loop[b][nl - 1] == r) continue;
          W.loop[b][nl++] = r;  // (never past fb + k)
        }
        while (nl - start > 1 && W.loop[b][start] == W.loop[b][nl - 1]) --nl;
        if (nl - start >= 3) {
          W.nb[b][nf] = W.nb[b][f];
          W.fs[b][nf] = (short)start;
          W.fl[b][nf] = (unsigned char)(nl - start);
          ++nf;
        } else {
          nl = start;
        }
      }
      W.nf = nf;
      W.nl = nl;
    }
    __syncwarp();
  }
}

// Numbers the vertices in the order the loops first use them: W.remap[old] =
// new (255: unused); returns how many are used.
__device__ __forceinline__ int cell_number(CellWarp& W) {
  const int lane = threadIdx.x & 31;
  const int b = W.b;
  // the loop entry at which a vertex appears first (in W.key)
  int used = 0;
  for (int i0 = 0; i0 < W.nv; i0 += 32) {
    const int i = i0 + lane;
    int first = VOR_MAXL;
    if (i < W.nv)
      for (int e = 0; e < W.nl; ++e)
        if (W.loop[b][e] == i) { first = e; break; }
    if (i < W.nv) W.key[i] = (short)first;
    used += __popc(__ballot_sync(VFULL, first < VOR_MAXL));
  }
  __syncwarp();
  for (int i = lane; i < W.nv; i += 32) {
    int rank = 0;
    for (int j = 0; j < W.nv; ++j) rank += W.key[j] < W.key[i];
    W.remap[i] = W.key[i] < VOR_MAXL ? (unsigned char)rank : 255;
  }
  __syncwarp();
  return used;
}

// One warp per site, the sites taken in bucket order so that neighbouring
// warps read the same buckets: its cell to its slot, or (ox not null) its
// centroid -- site + volume-weighted mean of the fan tetrahedra -- alone.
__global__ void __launch_bounds__(VW * 32) vor_cells(int64_t n, const double* __restrict__ x,
                                                     const double* __restrict__ y, const double* __restrict__ z,
                                                     Buckets B, SlotArrays S, double* ox, double* oy, double* oz,
                                                     unsigned long long* overflow) {
  __shared__ CellWarp cw[VW];
  const int lane = threadIdx.x & 31;
  CellWarp& W = cw[threadIdx.x >> 5];
  const int64_t t = blockIdx.x * (int64_t)VW + (threadIdx.x >> 5);
  if (t >= n) return;  // whole warp
  const int32_t i = B.sites[t];
  const float4 H0 = __ldg(B.hi + t), L0 = __ldg(B.lo + t);
  const double sx = x[i], sy = y[i], sz = z[i];
  const int G = B.G;
  const double bw = 1.0 / G;
  const float bwf = (float)bw;
  const int bx = bucket_coord(sx, G), by = bucket_coord(sy, G), bz = bucket_coord(sz, G);
  cell_box(W, sx, sy, sz);

  // The VOR_NEAR nearest sites of the surrounding 27 buckets, one per lane in
  // order of (distance, index).  The site's own bucket comes first and sets a
  // bound for the others; sites within the bound (FP32, with a margin for its
  // own error) gather in W.s's place 32 at a time and are merged by their FP64
  // distance.
  double kd = INFINITY;  // this lane's entry
  int kj = INT32_MAX;
  double kth = INFINITY;     // the last lane's
  float kthf = INFINITY;     // no site within kth has a larger FP32 distance
  int* const queue = reinterpret_cast<int*>(W.s);  // 64 positions
  int nq = 0;
  auto before = [](double da, int ja, double db, int jb) {
    const int64_t a = dm::bits(da), b = dm::bits(db);  // distances are positive
    return a < b || (a == b && ja < jb);
  };
  // the first m (<= 32) of the queue: sorted descending, then the entrywise
  // minimum with the list, which is bitonic
  auto merge = [&](int m) {
    __syncwarp();
    double d2 = INFINITY;
    int j = INT32_MAX;
    if (lane < m) {
      j = __float_as_int(__ldg(B.hi + queue[lane]).w);
      d2 = dist2(x[j] - sx, y[j] - sy, z[j] - sz);
      if (!(d2 > 0.0)) { d2 = INFINITY; j = INT32_MAX; }
    }
#pragma unroll 1
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll 1
      for (int h = k >> 1; h > 0; h >>= 1) {
        const double od = __shfl_xor_sync(VFULL, d2, h);
        const int oj = __shfl_xor_sync(VFULL, j, h);
        const bool least = ((lane & h) == 0) == ((lane & k) != 0);
        if (before(od, oj, d2, j) == least && !(oj == j)) { d2 = od; j = oj; }
      }
    if (before(d2, j, kd, kj)) { kd = d2; kj = j; }
#pragma unroll 1
    for (int h = 16; h > 0; h >>= 1) {
      const double od = __shfl_xor_sync(VFULL, kd, h);
      const int oj = __shfl_xor_sync(VFULL, kj, h);
      if (before(od, oj, kd, kj) == ((lane & h) == 0) && !(oj == kj)) { kd = od; kj = oj; }
    }
    kth = __shfl_sync(VFULL, kd, 31);
    const float kr = (sqrtf((float)kth) + SPLIT_ERR) * 1.00001f;
    kthf = kr * kr;
    const int v = lane + 32 < nq ? queue[lane + 32] : 0;
    __syncwarp();
    if (lane + 32 < nq) queue[lane] = v;
    nq -= m;
  };
  {
    // lanes 0..26: the buckets, the site's own as lane 0
    int p0 = 0, p1 = 0;
    float dist = INFINITY;
    if (lane < 27) {
      const int o = lane == 0 ? 13 : (lane <= 13 ? lane - 1 : lane);
      const int cx = bx + o % 3 - 1, cy = by + o / 3 % 3 - 1, cz = bz + o / 9 - 1;
      if (cx >= 0 && cy >= 0 && cz >= 0 && cx < G && cy < G && cz < G) {
        const int64_t cell = ((int64_t)cz * G + cy) * G + cx;
        p0 = (int)B.off[cell];
        p1 = (int)B.off[cell + 1];
        dist = box_dist2(H0.x, H0.y, H0.z, cx, cx, cy, cz, bwf);
      }
    }
    for (int pass = 0; pass < 2; ++pass) {
      // own bucket, then the others within the bound, end to end
      const int mine = (lane == 0) == (pass == 0) && dist <= kthf ? p1 - p0 : 0;
      int end;
      const int tot = warp_ends(mine, end);
      for (int f0 = 0; f0 < tot; f0 += 32) {
        const int f = f0 + lane;
        int rest;
        const int l = warp_owner(f, end, mine, rest);
        const int64_t q = __shfl_sync(VFULL, p0, l) + rest;
        bool in = false;
        if (f < tot && q != t) {
          const float4 H = __ldg(B.hi + q), D = __ldg(B.lo + q);
          const float fx = (H.x - H0.x) + (D.x - L0.x), fy = (H.y - H0.y) + (D.y - L0.y), fz = (H.z - H0.z) + (D.z - L0.z);
          in = fx * fx + fy * fy + fz * fz <= kthf;
        }
        const unsigned m = __ballot_sync(VFULL, in);
        if (in) queue[nq + __popc(m & ((1u << lane) - 1u))] = (int)q;
        nq += __popc(m);
        if (nq >= 32) merge(32);
      }
    }
    if (nq) merge(nq);
  }
  const int kn = __popc(__ballot_sync(VFULL, kj != INT32_MAX));
  bool bad = false;
  // their planes, one per lane; cut in order, the clear ones skipped together
  {
    double nx = 0, ny = 0, nz = 0, len = 0;
    if (lane < kn) {
      len = dm::length(kd);
      const double il = dm::inverse(len);
      nx = (x[kj] - sx) * il; ny = (y[kj] - sy) * il; nz = (z[kj] - sz) * il;
    }
    const float fx = dm::f32(nx), fy = dm::f32(ny), fz = dm::f32(nz), fd = 0.5f * dm::f32(len);
    unsigned todo = kn == 32 ? VFULL : (1u << kn) - 1u;
    while (todo) {
      const bool may = (todo >> lane & 1u) && may_cut(W, W.nv, fx, fy, fz, fd, rmax_of(W.rmax2));
      todo = __ballot_sync(VFULL, may);
      int rc = 0;
      while (todo && rc == 0) {
        const int k = __ffs(todo) - 1;
        todo &= todo - 1u;
        const double dk = __shfl_sync(VFULL, kd, k);
        if (!dm::gt(4.0 * W.rmax2, dk)) { todo = 0u; break; }
        rc = cell_clip(W, __shfl_sync(VFULL, nx, k), __shfl_sync(VFULL, ny, k), __shfl_sync(VFULL, nz, k),
                       0.5 * __shfl_sync(VFULL, len, k), __shfl_sync(VFULL, kj, k));
      }
      if (rc < 0) { bad = true; break; }
    }
  }
  // then every other site, ring by ring (the 27 buckets again only when the
  // nearest list was full: sites closer than its last entry are done).  A row
  // of buckets along x is one range of sites; lanes find 32 rows' ranges at a
  // time.
  const float kin = fmaxf(sqrtf((float)kth) * 0.99999f - SPLIT_ERR, 0.f), done2 = kin * kin;  // closer: in the list
  for (int r = kn == VOR_NEAR ? 0 : 2; r <= G && !bad; ++r) {
    // every site outside rings 0..r-1 is at least (r-1) bucket widths away
    const double reach = (r - 1) * bw;
    if (r >= 2 && reach * reach >= 4.0 * W.rmax2) break;
    const int side = 2 * r + 1, rows = side * side;
    for (int r0 = 0; r0 < rows && !bad; r0 += 32) {
      // this lane's row: one range, or two single buckets (x - r and x + r)
      int a0 = 0, a1 = 0, c0 = 0, c1 = 0;
      const int row = r0 + lane;
      if (row < rows) {
        const int dz = row / side - r, dy = row % side - r;
        const int cy = by + dy, cz = bz + dz;
        if (cy >= 0 && cz >= 0 && cy < G && cz < G) {
          const float far2 = 4.0f * dm::f32(W.rmax2) * 1.00001f;
          const int64_t at = ((int64_t)cz * G + cy) * G;
          auto range = [&](int u, int v, int& p0, int& p1) {
            u = u < 0 ? 0 : u;
            v = v >= G ? G - 1 : v;
            if (u > v || box_dist2(H0.x, H0.y, H0.z, u, v, cy, cz, bwf) > far2) return;
            p0 = (int)B.off[at + u];
            p1 = (int)B.off[at + v + 1];
          };
          if (dz == -r || dz == r || dy == -r || dy == r) {
            range(bx - r, bx + r, a0, a1);
          } else {
            if (bx - r >= 0) range(bx - r, bx - r, a0, a1);
            if (bx + r < G) range(bx + r, bx + r, c0, c1);
          }
        }
      }
      // the rows' sites end to end, 32 at a time
      const int na = a1 - a0, mine = na + (c1 - c0);
      int end;
      const int tot = warp_ends(mine, end);
      for (int f0 = 0; f0 < tot && !bad; f0 += 32) {
        const int f = f0 + lane;
        int rest;
        const int l = warp_owner(f, end, mine, rest);
        const int la = __shfl_sync(VFULL, na, l), pa = __shfl_sync(VFULL, a0, l), pc = __shfl_sync(VFULL, c0, l);
        const int64_t q = rest < la ? pa + rest : pc + (rest - la);
        float fx = 0, fy = 0, fz = 0, d2 = 0;
        int j = 0;
        bool may = false;
        if (f < tot && q != t) {
          const float4 H = __ldg(B.hi + q), D = __ldg(B.lo + q);
          fx = (H.x - H0.x) + (D.x - L0.x); fy = (H.y - H0.y) + (D.y - L0.y); fz = (H.z - H0.z) + (D.z - L0.z);
          d2 = fx * fx + fy * fy + fz * fz;
          j = __float_as_int(H.w);
          const float far = (2.0f * rmax_of(W.rmax2) + SPLIT_ERR) * 1.00001f;
          may = d2 < far * far && !(r <= 1 && d2 < done2);
        }
        if (!__any_sync(VFULL, may)) continue;
        // (an offset off by SPLIT_ERR turns the normal by twice that over its length)
        const float il = d2 > 0.f ? rsqrtf(d2) : 0.f, rmax = rmax_of(W.rmax2);
        may = may && may_cut(W, W.nv, fx * il, fy * il, fz * il, 0.5f * d2 * il, rmax, SPLIT_ERR * (2.f * rmax * il + 1.f));
        for (unsigned todo = __ballot_sync(VFULL, may); todo; todo &= todo - 1u) {
          const int jk = __shfl_sync(VFULL, j, __ffs(todo) - 1);
          const double ex = x[jk] - sx, ey = y[jk] - sy, ez = z[jk] - sz;
          const double e2 = dist2(ex, ey, ez);
          if (e2 <= 0.0 || e2 >= 4.0 * W.rmax2) continue;
          if (r <= 1 && (e2 < kth || (e2 == kth && jk <= __shfl_sync(VFULL, kj, 31)))) continue;  // in the list
          const double len = dm::length(e2), inv = dm::inverse(len);
          if (cell_clip(W, ex * inv, ey * inv, ez * inv, 0.5 * len, jk) < 0) { bad = true; break; }
        }
      }
    }
  }
  if (bad) {
    if (lane == 0) {
      atomicAdd(overflow, 1ULL);
      if (!ox) S.info[i] = Slot{0, 0, 0, 0};
    }
    return;
  }
  cell_weld(W);
  const int b = W.b;
  if (ox) {
    double tv = 0.0, gx = 0.0, gy = 0.0, gz = 0.0;
    for (int f = lane; f < W.nf; f += 32) {
      const int fb = W.fs[b][f], L = W.fl[b][f];
      const int a = W.loop[b][fb];
      const double ax = W.x[b][a], ay = W.y[b][a], az = W.z[b][a];
      int p = W.loop[b][fb + 1];
      double px = W.x[b][p], py = W.y[b][p], pz = W.z[b][p];
      for (int k = 2; k < L; ++k) {
        p = W.loop[b][fb + k];
        const double qx = W.x[b][p], qy = W.y[b][p], qz = W.z[b][p];
        // 6 x the volume of (site, a, p, q), 4 x its centroid
        const double v = ax * (py * qz - pz * qy) - ay * (px * qz - pz * qx) + az * (px * qy - py * qx);
        tv += v;
        gx = fma(v, ax + px + qx, gx);
        gy = fma(v, ay + py + qy, gy);
        gz = fma(v, az + pz + qz, gz);
        px = qx; py = qy; pz = qz;
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      tv += __shfl_xor_sync(VFULL, tv, o);
      gx += __shfl_xor_sync(VFULL, gx, o);
      gy += __shfl_xor_sync(VFULL, gy, o);
      gz += __shfl_xor_sync(VFULL, gz, o);
    }
    if (lane == 0) {
      ox[i] = sx + gx * 0.25 / tv;
      oy[i] = sy + gy * 0.25 / tv;
      oz[i] = sz + gz * 0.25 / tv;
    }
    return;
  }
  const int nv = cell_number(W);
  double* v = S.v + (size_t)i * 3 * VOR_MAXV;
  for (int k = lane; k < W.nv; k += 32) {
    const int m = W.remap[k];
    if (m != 255) { v[3 * m] = W.x[b][k]; v[3 * m + 1] = W.y[b][k]; v[3 * m + 2] = W.z[b][k]; }
  }
  unsigned char* lp = S.loop + (size_t)i * VOR_MAXL;
  for (int k = lane; k < W.nl; k += 32) lp[k] = W.remap[W.loop[b][k]];
  for (int f = lane; f < W.nf; f += 32) {
    S.fs[(size_t)i * VOR_MAXF + f] = W.fs[b][f];
    S.fl[(size_t)i * VOR_MAXF + f] = W.fl[b][f];
    S.nb[(size_t)i * VOR_MAXF + f] = W.nb[b][f];
  }
  if (lane == 0) S.info[i] = Slot{nv, W.nf, W.nl, 1};
}

__global__ void vor_counts(int64_t n, const Slot* __restrict__ info, int64_t* nf, int64_t* nl, int64_t* nv) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i > n) return;
  if (i == n) { nf[i] = 0; nl[i] = 0; nv[i] = 0; return; }
  nf[i] = info[i].nf; nl[i] = info[i].nl; nv[i] = info[i].nv;
}

// pack the slots into the CSR arrays of map_grid (absolute coordinates)
__global__ void vor_pack(int64_t n, const double* __restrict__ x, const double* __restrict__ y,
                         const double* __restrict__ z, SlotArrays S, const int64_t* __restrict__ fo,
                         const int64_t* __restrict__ lo, const int64_t* __restrict__ vo, int64_t* cell_face_off,
                         int64_t* face_vert_off, int32_t* face_vert, double* face_plane, double* vx, double* vy,
                         double* vz, double* site) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i > n) return;
  if (i == n) {
    cell_face_off[n] = fo[n];
    face_vert_off[fo[n]] = lo[n];
    return;
  }
  const Slot info = S.info[i];
  const double sx = x[i], sy = y[i], sz = z[i];
  site[3 * i] = sx; site[3 * i + 1] = sy; site[3 * i + 2] = sz;
  cell_face_off[i] = fo[i];
  const double* v = S.v + (size_t)i * 3 * VOR_MAXV;
  for (int k = 0; k < info.nv; ++k) {
    vx[vo[i] + k] = sx + v[3 * k];
    vy[vo[i] + k] = sy + v[3 * k + 1];
    vz[vo[i] + k] = sz + v[3 * k + 2];
  }
  const unsigned char* lp = S.loop + (size_t)i * VOR_MAXL;
  int64_t l = lo[i];
  for (int f = 0; f < info.nf; ++f) {
    const int64_t F = fo[i] + f;
    face_vert_off[F] = l;
    const int b = S.fs[(size_t)i * VOR_MAXF + f], L = S.fl[(size_t)i * VOR_MAXF + f];
    for (int k = 0; k < L; ++k) face_vert[l++] = (int32_t)(vo[i] + lp[b + k]);
    const int w = S.nb[(size_t)i * VOR_MAXF + f];
    double nx, ny, nz, d;
    if (w < 0) {
      const int ax = (-1 - w) / 2, sg = ((-1 - w) % 2 == 0) ? 1 : -1;
      nx = ax == 0 ? sg : 0.0; ny = ax == 1 ? sg : 0.0; nz = ax == 2 ? sg : 0.0;
      d = sg > 0 ? 1.0 : 0.0;
    } else {
      const double ex = x[w] - sx, ey = y[w] - sy, ez = z[w] - sz;
      const double len = sqrt(ex * ex + ey * ey + ez * ez);
      nx = ex / len; ny = ey / len; nz = ez / len;
      d = nx * (0.5 * (sx + x[w])) + ny * (0.5 * (sy + y[w])) + nz * (0.5 * (sz + z[w]));
    }
    face_plane[4 * F] = nx; face_plane[4 * F + 1] = ny; face_plane[4 * F + 2] = nz; face_plane[4 * F + 3] = d;
  }
}

template <typename T>
int scan_excl(map_ctx* ctx, const T* in, T* out, int64_t n, cudaStream_t s) {
  size_t tb = 0;
  CUDA_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tb, in, out, n, s));
  MAP_TRY(ctx_ensure(ctx, ctx->cub_tmp, tb));
  CUDA_TRY(cub::DeviceScan::ExclusiveSum(ctx->cub_tmp.p, tb, in, out, n, s));
  return MAP_OK;
}

// bucket grid over the sites x, y, z (n of them)
int vor_buckets(map_ctx* ctx, const double* x, const double* y, const double* z, int64_t n, Buckets& B,
                cudaStream_t s) {
  int G = (int)floor(cbrt((double)n / 2.0));
  G = G < 1 ? 1 : (G > 1024 ? 1024 : G);
  const int64_t nb = (int64_t)G * G * G;
  int32_t *key, *idx, *key_s, *idx_s;
  int64_t* off;
  MAP_TRY(ensure_t(ctx, ctx->ws_vor[0], n, &key));
  MAP_TRY(ensure_t(ctx, ctx->ws_vor[1], n, &idx));
  MAP_TRY(ensure_t(ctx, ctx->ws_vor[2], n, &key_s));
  MAP_TRY(ensure_t(ctx, ctx->ws_vor[3], n, &idx_s));
  MAP_TRY(ensure_t(ctx, ctx->ws_vor[4], nb + 1, &off));
  vor_bucket_keys<<<nblk(n, 256), 256, 0, s>>>(n, x, y, z, G, key, idx); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  int bits = 1;
  while (bits < 31 && (int64_t(1) << bits) < nb) ++bits;
  size_t tb = 0;
  CUDA_TRY(cub::DeviceRadixSort::SortPairs(nullptr, tb, key, key_s, idx, idx_s, n, 0, bits, s));
  MAP_TRY(ctx_ensure(ctx, ctx->cub_tmp, tb));
  CUDA_TRY(cub::DeviceRadixSort::SortPairs(ctx->cub_tmp.p, tb, key, key_s, idx, idx_s, n, 0, bits, s));
  vor_bucket_bounds<<<nblk(n + 1, 256), 256, 0, s>>>(n, nb, key_s, off); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  float4 *hi, *lo;  // (in the place of the grid's face planes, written last)
  MAP_TRY(ensure_t(ctx, ctx->ws_vor[19], 2 * n, &hi));
  lo = hi + n;
  vor_split<<<nblk(n, 256), 256, 0, s>>>(n, x, y, z, idx_s, hi, lo); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  B = Buckets{G, off, idx_s, hi, lo};
  return MAP_OK;
}

// The cells of the sites x, y, z: into the slots (ox null), or their centroids
// into ox, oy, oz.  MAP_ECAPACITY on overflow.
int vor_tessellate(map_ctx* ctx, const double* x, const double* y, const double* z, int64_t n, SlotArrays& S,
                   double* ox, double* oy, double* oz, cudaStream_t s) {
  Buckets B;
  MAP_TRY(vor_buckets(ctx, x, y, z, n, B, s));
  if (!ox) {
    MAP_TRY(ensure_t(ctx, ctx->ws_vor[5], n, &S.info));
    MAP_TRY(ensure_t(ctx, ctx->ws_vor[6], (size_t)n * 3 * VOR_MAXV, &S.v));
    MAP_TRY(ensure_t(ctx, ctx->ws_vor[7], (size_t)n * VOR_MAXL, &S.loop));
    MAP_TRY(ensure_t(ctx, ctx->ws_vor[8], (size_t)n * VOR_MAXF, &S.fs));
    MAP_TRY(ensure_t(ctx, ctx->ws_vor[9], (size_t)n * VOR_MAXF, &S.fl));
    MAP_TRY(ensure_t(ctx, ctx->ws_vor[10], (size_t)n * VOR_MAXF, &S.nb));
  }
  unsigned long long* d_over = ctx->d_counters + 7;
  CUDA_TRY(cudaMemsetAsync(d_over, 0, sizeof(unsigned long long), s));
  vor_cells<<<nblk(n, VW), VW * 32, 0, s>>>(n, x, y, z, B, S, ox, oy, oz, d_over); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  CUDA_TRY(cudaMemcpyAsync(ctx->h_scratch, d_over, sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  return ctx->h_scratch[0] == 0 ? MAP_OK : MAP_ECAPACITY;
}

__global__ void vor_iota_k(int64_t n, int64_t* out) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) out[i] = i;
}

int vor_iota(map_ctx* ctx, int64_t* out, int64_t n, cudaStream_t s) {
  vor_iota_k<<<nblk(n, 256), 256, 0, s>>>(n, out); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  return MAP_OK;
}

}  // namespace

extern "C" int map_grid_build(map_ctx* ctx, const double* x, const double* y, const double* z, int64_t n, int lloyd,
                              double merge_tol, int* handle, int64_t* kept, int64_t* n_kept, void* stream) {
  if (!ctx || !x || !y || !z || n < 1 || n >= (int64_t(1) << 31) || lloyd < 0 || !handle) return MAP_EINVAL;
  if (!(merge_tol >= 0.0) || !std::isfinite(merge_tol)) return MAP_EINVAL;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  MAP_ENTER(ctx, s);
  map_particles chk{n, x, y, z, nullptr, nullptr};
  MAP_TRY(check_particles(ctx, &chk, false, false, s));  // finite, inside the cube
  // the sites, merged, in one of two ping-pong buffers (x block, y block, z block)
  double *sa, *sb;
  MAP_TRY(ensure_t(ctx, ctx->ws_vor[11], 3 * n, &sa));
  MAP_TRY(ensure_t(ctx, ctx->ws_vor[12], 3 * n, &sb));
  int64_t m = n;
  if (merge_tol > 0.0) {
    Buckets B;
    MAP_TRY(vor_buckets(ctx, x, y, z, n, B, s));
    int64_t *keep, *pos;
    MAP_TRY(ensure_t(ctx, ctx->ws_vor[13], n + 1, &keep));
    MAP_TRY(ensure_t(ctx, ctx->ws_vor[14], n + 1, &pos));
    vor_merge_flags<<<nblk(n + 1, 256), 256, 0, s>>>(n, x, y, z, B, merge_tol, keep); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
    MAP_TRY(scan_excl<int64_t>(ctx, keep, pos, n + 1, s));
    CUDA_TRY(cudaMemcpyAsync(ctx->h_scratch, pos + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaStreamSynchronize(s));
    m = ctx->h_scratch[0];
    vor_merge_pack<<<nblk(n, 256), 256, 0, s>>>(n, keep, pos, x, y, z, sa, sa + m, sa + 2 * m, kept); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
  } else {
    CUDA_TRY(cudaMemcpyAsync(sa, x, n * sizeof(double), cudaMemcpyDeviceToDevice, s));
    CUDA_TRY(cudaMemcpyAsync(sa + n, y, n * sizeof(double), cudaMemcpyDeviceToDevice, s));
    CUDA_TRY(cudaMemcpyAsync(sa + 2 * n, z, n * sizeof(double), cudaMemcpyDeviceToDevice, s));
    if (kept) MAP_TRY(vor_iota(ctx, kept, n, s));
  }
  if (n_kept) *n_kept = m;
  // Lloyd iterations, then the final cells
  SlotArrays S{};
  for (int it = 0; it < lloyd; ++it) {
    MAP_TRY(vor_tessellate(ctx, sa, sa + m, sa + 2 * m, m, S, sb, sb + m, sb + 2 * m, s));
    double* t = sa; sa = sb; sb = t;
  }
  MAP_TRY(vor_tessellate(ctx, sa, sa + m, sa + 2 * m, m, S, nullptr, nullptr, nullptr, s));
  // CSR offsets and the packed arrays
  int64_t *cf, *cl, *cv, *fo, *lo, *vo;
  MAP_TRY(ensure_t(ctx, ctx->ws_vor[15], 6 * (m + 1), &cf));
  cl = cf + (m + 1); cv = cl + (m + 1); fo = cv + (m + 1); lo = fo + (m + 1); vo = lo + (m + 1);
  vor_counts<<<nblk(m + 1, 256), 256, 0, s>>>(m, S.info, cf, cl, cv); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  MAP_TRY(scan_excl<int64_t>(ctx, cf, fo, m + 1, s));
  MAP_TRY(scan_excl<int64_t>(ctx, cl, lo, m + 1, s));
  MAP_TRY(scan_excl<int64_t>(ctx, cv, vo, m + 1, s));
  CUDA_TRY(cudaMemcpyAsync(ctx->h_scratch, fo + m, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaMemcpyAsync(ctx->h_scratch + 1, lo + m, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaMemcpyAsync(ctx->h_scratch + 2, vo + m, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  const int64_t nf = ctx->h_scratch[0], nl = ctx->h_scratch[1], nv = ctx->h_scratch[2];
  int64_t *cfo, *fvo;
  int32_t* fv;
  double *fpl, *vx, *vy, *vz, *site;
  MAP_TRY(ensure_t(ctx, ctx->ws_vor[16], m + 1, &cfo));
  MAP_TRY(ensure_t(ctx, ctx->ws_vor[17], nf + 1, &fvo));
  MAP_TRY(ensure_t(ctx, ctx->ws_vor[18], nl, &fv));
  MAP_TRY(ensure_t(ctx, ctx->ws_vor[19], 4 * nf, &fpl));
  MAP_TRY(ensure_t(ctx, ctx->ws_vor[20], 3 * nv, &vx));
  vy = vx + nv; vz = vy + nv;
  MAP_TRY(ensure_t(ctx, ctx->ws_vor[21], 3 * m, &site));
  vor_pack<<<nblk(m + 1, 128), 128, 0, s>>>(m, sa, sa + m, sa + 2 * m, S, fo, lo, vo, cfo, fvo, fv, fpl, vx, vy, vz,
                                            site); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  const map_grid grid{m, nf, nl, nv, cfo, fvo, fv, fpl, vx, vy, vz, site};
  return map_grid_upload(ctx, &grid, handle, stream);
}
