// Device octree over a particle set.
//
// Octree (Section III-A, built as an octree with a leaf capacity instead of
// the paper's RCB tree): 63-bit Morton keys (21 bits per axis) are radix
// sorted; a node at level L is the cube of side 2^-L holding a contiguous key
// range, split while it holds more than leaf_size particles (up to level 21).
// Labels carry a leading 1 bit, so parent = label >> 3 (the paper's heap-style
// label arithmetic with eight children).  Node mass and centre of mass are
// summed bottom-up; node size (distance from the centre of mass to the
// furthest particle, Section III-A), largest h and bounding box are reduced
// over each node's particles.
//
// The nodes follow from the sorted keys alone, in three launches of a fixed
// shape: the levels at which each position starts a node as bit maps, their
// ranks by one scan, and the node records.  One more launch sums them bottom
// up, a node by the thread that finishes its last child.  What bounds it is the
// sort and, for small sets, the chain of about 20 launches.  Level by level,
// with the node counts read back after each of 10 to 22 levels and two
// launches per level for the sums, the same tree took 0.38 ms for 4,096
// particles and 0.70 ms for 60,000; it takes 0.14 and 0.26 ms.
#include <cub/cub.cuh>

#include "internal.cuh"

namespace {

constexpr int MORTON_BITS = 21;
constexpr int64_t BIG_NODE = 4096;

struct MaxOp {
  __device__ __forceinline__ double operator()(double a, double b) const { return a > b ? a : b; }
};

__device__ __forceinline__ uint64_t spread3(uint64_t v) {
  v &= 0x1fffff;
  v = (v | v << 32) & 0x1f00000000ffffULL;
  v = (v | v << 16) & 0x1f0000ff0000ffULL;
  v = (v | v << 8) & 0x100f00f00f00f00fULL;
  v = (v | v << 4) & 0x10c30c30c30c30c3ULL;
  v = (v | v << 2) & 0x1249249249249249ULL;
  return v;
}

__device__ __forceinline__ uint64_t coord21(double v) {
  double s = floor(v * 2097152.0);
  if (!(s >= 0.0)) s = 0.0;
  if (s > 2097151.0) s = 2097151.0;
  return (uint64_t)s;
}

__global__ void morton_keys(int64_t n, const double* __restrict__ x, const double* __restrict__ y,
                            const double* __restrict__ z, uint64_t* keys, int32_t* idx) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  keys[i] = (spread3(coord21(x[i])) << 2) | (spread3(coord21(y[i])) << 1) | spread3(coord21(z[i]));
  idx[i] = (int32_t)i;
}

// The keys of a small set sorted in one block: a bitonic network over (key,
// index) in shared memory, P places (a power of two, P >= n), the index as the
// second key, so that the order is the stable sort's.  Exchanges of up to 32
// places stay within the warp that owns their 64 places and need no block
// barrier.  Above 2000 or so the library's radix sort takes 8 passes over the
// 63 bits, each mostly launch and look-back latency at these sizes: octree of
// 4096 particles 193 -> 140 us with this; 2000: the same (the library sorts
// them in one block too); 8192: 206 and 203 us, 16384: 223 and 324 us, so the
// line lies at 4096.
constexpr int SORT_THREADS = 1024;
constexpr int SORT_SMALL = 4096;

__global__ void __launch_bounds__(SORT_THREADS) sort_small(int n, int P, const uint64_t* __restrict__ keys,
                                                           uint64_t* __restrict__ out, int32_t* __restrict__ idx) {
  __shared__ uint64_t sk[SORT_SMALL];
  __shared__ unsigned short si[SORT_SMALL];
  for (int i = threadIdx.x; i < P; i += SORT_THREADS) {
    sk[i] = i < n ? keys[i] : ~0ull;  // (padding goes last: a key has 63 bits)
    si[i] = (unsigned short)i;
  }
  __syncthreads();
  for (int k = 2; k <= P; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < P / 2; t += SORT_THREADS) {
        const int a = 2 * t - (t & (j - 1)), b = a + j;
        const uint64_t ka = sk[a], kb = sk[b];
        const unsigned short ia = si[a], ib = si[b];
        const bool greater = ka > kb || (ka == kb && ia > ib);
        if (greater == ((a & k) == 0)) {
          sk[a] = kb; sk[b] = ka;
          si[a] = ib; si[b] = ia;
        }
      }
      if (j > 32 || (j == 1 && k >= 64)) __syncthreads(); else __syncwarp();
    }
  for (int i = threadIdx.x; i < n; i += SORT_THREADS) {
    out[i] = sk[i];
    idx[i] = si[i];
  }
}

__global__ void gather_sorted(int64_t n, const int32_t* __restrict__ idx, const double* __restrict__ x,
                              const double* __restrict__ y, const double* __restrict__ z,
                              const double* __restrict__ m, const double* __restrict__ h, double* xs, double* ys,
                              double* zs, double* ms, double* hs, float* split, float* hs32) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  int32_t a = idx[i];
  const double px = x[a] + 0.0, py = y[a] + 0.0, pz = z[a] + 0.0;  // + 0.0: -0.0 -> +0.0 (bit-ordered min/max)
  xs[i] = px;
  ys[i] = py;
  zs[i] = pz;
  ms[i] = m ? m[a] : 1.0;
  hs[i] = h ? h[a] : 0.0;
  if (hs32) hs32[i] = (float)h[a];  // set only for trees built with h
  // FP32 hi/lo split of the coordinates: x = hi + lo to ~2^-48, so that the
  // difference of two nearby points, (hi_j - hi_i) + (lo_j - lo_i), keeps
  // ~24 bits relative to the separation
  const float hx = (float)px, hy = (float)py, hz = (float)pz;
  split[6 * i + 0] = hx; split[6 * i + 1] = (float)(px - (double)hx);
  split[6 * i + 2] = hy; split[6 * i + 3] = (float)(py - (double)hy);
  split[6 * i + 4] = hz; split[6 * i + 5] = (float)(pz - (double)hz);
}

// One node's sums: leaves sum their particles in sorted order, internal nodes
// sum their children in octant order (mass, mass-weighted position); bounding
// box and largest h are the union / maximum over the particles (leaves) or the
// children (internal nodes), exact in any order.  The children's values come
// from L2 (other threads of this launch wrote them).
struct NodeArrays {
  const int64_t *nb, *ne, *fc;
  const int32_t *nch, *parent;
  const double *xs, *ys, *zs, *ms, *hs;
  double *mass, *msum, *com;  // msum: 3 per node, sum m x
  unsigned long long *size_bits, *hmax_bits, *bbox;
  float* box32;
  int32_t* owner;
  int32_t* arrived;  // children finished
};

__device__ __forceinline__ double ldcg_bits(const unsigned long long* p) { return bitsd(__ldcg(p)); }

__device__ __forceinline__ void node_sum_one(int64_t i, const NodeArrays& A) {
  double M = 0, Sx = 0, Sy = 0, Sz = 0, hm = 0;
  double lo0 = 1e300, lo1 = 1e300, lo2 = 1e300, hi0 = 0, hi1 = 0, hi2 = 0;
  const int nc = A.nch[i];
  const int64_t f = A.fc[i];
  if (nc == 0) {
    const int64_t b = A.nb[i], e = A.ne[i];
    for (int64_t k = b; k < e; ++k) {
      const double mk = A.ms[k], x = A.xs[k], y = A.ys[k], z = A.zs[k];
      M += mk;
      Sx += mk * x;
      Sy += mk * y;
      Sz += mk * z;
      hm = fmax(hm, A.hs[k]);
      lo0 = fmin(lo0, x); lo1 = fmin(lo1, y); lo2 = fmin(lo2, z);
      hi0 = fmax(hi0, x); hi1 = fmax(hi1, y); hi2 = fmax(hi2, z);
      A.owner[k] = (int32_t)i;
    }
  } else {
    for (int64_t c = f; c < f + nc; ++c) {
      M += __ldcg(A.mass + c);
      Sx += __ldcg(A.msum + 3 * c);
      Sy += __ldcg(A.msum + 3 * c + 1);
      Sz += __ldcg(A.msum + 3 * c + 2);
      hm = fmax(hm, ldcg_bits(A.hmax_bits + c));
      const unsigned long long* q = A.bbox + 6 * c;
      lo0 = fmin(lo0, ldcg_bits(q)); lo1 = fmin(lo1, ldcg_bits(q + 1)); lo2 = fmin(lo2, ldcg_bits(q + 2));
      hi0 = fmax(hi0, ldcg_bits(q + 3)); hi1 = fmax(hi1, ldcg_bits(q + 4)); hi2 = fmax(hi2, ldcg_bits(q + 5));
    }
  }
  A.mass[i] = M;
  A.msum[3 * i] = Sx;
  A.msum[3 * i + 1] = Sy;
  A.msum[3 * i + 2] = Sz;
  A.hmax_bits[i] = dbits(hm);
  unsigned long long* q = A.bbox + 6 * i;
  q[0] = dbits(lo0); q[1] = dbits(lo1); q[2] = dbits(lo2);
  q[3] = dbits(hi0); q[4] = dbits(hi1); q[5] = dbits(hi2);
  A.com[3 * i] = Sx / M;
  A.com[3 * i + 1] = Sy / M;
  A.com[3 * i + 2] = Sz / M;
  A.size_bits[i] = 0ULL;
  // The walks' node record, two 16-byte loads: the FP32 box rounded outward,
  // the largest h rounded up, and (bits of the last float) first child << 4 |
  // child count for an internal node with a first child below 2^28, 0 for a
  // leaf, and NODE_LINK_FAR when the index does not fit (read the arrays then).
  const unsigned link = nc == 0 ? 0u : (f < (1LL << 28) ? ((unsigned)f << 4) | (unsigned)nc : NODE_LINK_FAR);
  float4* R = reinterpret_cast<float4*>(A.box32) + 2 * i;
  R[0] = make_float4(__double2float_rd(lo0), __double2float_rd(lo1), __double2float_rd(lo2), __double2float_ru(hi0));
  R[1] = make_float4(__double2float_ru(hi1), __double2float_ru(hi2), __double2float_ru(hm), __uint_as_float(link));
}

// Every node's sums in one launch: a thread takes a leaf and then its
// ancestors, each as the thread that finishes its last child (no thread waits
// for another).  total: the node count.
__global__ void node_sums(const int32_t* __restrict__ total, NodeArrays A) {
  const int64_t nn = *total, stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nn; t += stride) {
    if (A.nch[t] != 0) continue;
    for (int64_t i = t;;) {
      node_sum_one(i, A);
      const int32_t p = A.parent[i];
      if (p < 0) break;
      __threadfence();
      if (atomicAdd(A.arrived + p, 1) != A.nch[p] - 1) break;
      __threadfence();
      i = p;
    }
  }
}

// Node size (distance from the centre of mass to the furthest particle,
// Section III-A), needed by the pseudo-particle walk only: the largest squared
// distance first (node_extent_*), its root at the end (node_size; a correctly
// rounded root is monotone, so this is the largest distance).  A particle whose
// FP32 distance is short of the largest so far by more than FP32's rounding of
// the unit cube's coordinates takes no FP64.
struct Extent {
  double cx, cy, cz;
  float fx, fy, fz;
};
__device__ __forceinline__ Extent extent_of(const double* com, int64_t i) {
  const double x = com[3 * i], y = com[3 * i + 1], z = com[3 * i + 2];
  return Extent{x, y, z, (float)x, (float)y, (float)z};
}
__device__ __forceinline__ float reach32(double r2) {
  const float r = sqrtf((float)r2) - 1e-6f;
  return r > 0.f ? r * r : 0.f;
}
__device__ __forceinline__ bool farther(const Extent& E, float x, float y, float z, float reach2) {
  const float dx = x - E.fx, dy = y - E.fy, dz = z - E.fz;
  return dx * dx + dy * dy + dz * dz >= reach2;
}
__device__ __forceinline__ double extent2(const Extent& E, double x, double y, double z) {
  const double dx = x - E.cx, dy = y - E.cy, dz = z - E.cz;
  return dx * dx + dy * dy + dz * dz;
}

// Small nodes: every particle walks up from its leaf while the node holds at
// most BIG_NODE particles.
__global__ void node_extent_small(int64_t n, const int32_t* __restrict__ owner, const int32_t* __restrict__ parent,
                                  const int64_t* __restrict__ nb, const int64_t* __restrict__ ne,
                                  const double* __restrict__ xs, const double* __restrict__ ys,
                                  const double* __restrict__ zs, const double* __restrict__ com,
                                  unsigned long long* size_bits) {
  int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= n) return;
  const double x = xs[k], y = ys[k], z = zs[k];
  const float fx = (float)x, fy = (float)y, fz = (float)z;
  int32_t node = owner[k];
  while (node >= 0 && ne[node] - nb[node] <= BIG_NODE) {
    const Extent E = extent_of(com, node);
    if (farther(E, fx, fy, fz, reach32(bitsd(__ldcg(size_bits + node)))))
      atomicMax(&size_bits[node], dbits(extent2(E, x, y, z)));
    node = parent[node];
  }
}

// Big nodes in slices of BIG_NODE particles: the list of (node << 32 | slice).
__global__ void collect_big(int64_t nn, const int64_t* __restrict__ nb, const int64_t* __restrict__ ne, int64_t* big,
                            unsigned long long* nbig) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nn) return;
  const int64_t m = ne[i] - nb[i];
  if (m <= BIG_NODE) return;
  const int64_t slices = (m + BIG_NODE - 1) / BIG_NODE;
  int64_t* out = big + atomicAdd(nbig, (unsigned long long)slices);
  for (int64_t k = 0; k < slices; ++k) out[k] = i << 32 | k;
}

__global__ void __launch_bounds__(256) node_extent_big(const int64_t* __restrict__ big,
                                                       const unsigned long long* __restrict__ nbig,
                                                       const int64_t* __restrict__ nb, const int64_t* __restrict__ ne,
                                                       const float* __restrict__ split, const double* __restrict__ xs,
                                                       const double* __restrict__ ys, const double* __restrict__ zs,
                                                       const double* __restrict__ com, unsigned long long* size_bits) {
  typedef cub::BlockReduce<double, 256> BR;
  __shared__ typename BR::TempStorage tmp;
  const int64_t count = (int64_t)*nbig;
  for (int64_t t = blockIdx.x; t < count; t += gridDim.x) {
    const int64_t node = big[t] >> 32, lo = nb[node] + (big[t] & 0xffffffff) * BIG_NODE;
    const int64_t hi = lo + BIG_NODE < ne[node] ? lo + BIG_NODE : ne[node];
    const Extent E = extent_of(com, node);
    double r2 = bitsd(__ldcg(size_bits + node));
    float reach = reach32(r2);
    for (int64_t k = lo + threadIdx.x; k < hi; k += 256) {
      if (!farther(E, split[6 * k], split[6 * k + 2], split[6 * k + 4], reach)) continue;
      const double d = extent2(E, xs[k], ys[k], zs[k]);
      if (d > r2) { r2 = d; reach = reach32(d); }
    }
    r2 = BR(tmp).Reduce(r2, MaxOp());
    if (threadIdx.x == 0) atomicMax(&size_bits[node], dbits(r2));
    __syncthreads();
  }
}

__global__ void node_size(int64_t nn, unsigned long long* size_bits) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < nn) size_bits[i] = dbits(sqrt(bitsd(size_bits[i])));
}

// ---------------------------------------------------------------- nodes from the sorted keys
// The nodes are numbered level by level, each level in key order.  With
// pfx_L(k) = k >> 3 (21 - L) the level-L prefix, the node (L, P) exists iff
// L = 0 or its parent prefix at level L - 1 holds more than leaf_size
// particles (then every ancestor holds more too, so all of them split), and
// it starts at the sorted position of its first particle.  Bit i of level L's
// map says whether position i starts a node there; the words' bit counts, laid
// out level-major (22 maps of nw = ceil(n / 32) words), are scanned, so that a
// node's number is its word's entry plus the bits below it: rank(L, i).
// rank(L, 0) is the first node of level L, entry 22 nw the node count.
constexpr int LEVELS = MORTON_BITS + 1;

__device__ __forceinline__ uint64_t pfx(uint64_t key, int L) { return key >> (3 * (MORTON_BITS - L)); }

// Whether the node of level L that holds position i has more than leaf
// particles: its first position, or one leaf places before i, decides.
__device__ __forceinline__ bool splits(const uint64_t* __restrict__ keys, int64_t n, int64_t i, int L, int leaf) {
  const uint64_t P = pfx(keys[i], L);
  int64_t lo = i > leaf ? i - leaf : 0, hi = i;
  if (i >= leaf && pfx(keys[lo], L) == P) return true;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (pfx(keys[mid], L) < P) lo = mid + 1; else hi = mid;
  }
  return lo + leaf < n && pfx(keys[lo + leaf], L) == P;
}

// one past the last position from i on whose level-L prefix equals i's
__device__ __forceinline__ int64_t prefix_end(const uint64_t* __restrict__ keys, int64_t i, int64_t n, int L) {
  const uint64_t P = pfx(keys[i], L);
  int64_t step = 8, lo = i + 1;
  while (lo - 1 + step < n && pfx(keys[lo - 1 + step], L) == P) { lo += step; step *= 2; }
  int64_t hi = lo - 1 + step < n ? lo - 1 + step : n;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (pfx(keys[mid], L) <= P) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// The levels at which each position starts a node: from d, the shallowest
// where its prefix differs from the position before, down while the enclosing
// node splits.
__global__ void __launch_bounds__(256) tree_bits(int64_t n, int64_t nw, const uint64_t* __restrict__ keys, int leaf,
                                                 uint32_t* __restrict__ map, int32_t* __restrict__ count) {
  const int lane = threadIdx.x & 31;
  const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (w >= nw) return;  // whole warp
  const int64_t i = w * 32 + lane;
  unsigned mine = 0u;
  if (i < n) {
    const uint64_t k = keys[i];
    int d = 0;
    if (i > 0) {
      const uint64_t x = keys[i - 1] ^ k;
      d = x == 0 ? LEVELS : MORTON_BITS - (63 - __clzll((long long)x)) / 3;
    }
    for (int L = d; L < LEVELS; ++L) {
      // below d the enclosing node starts here: its first leaf + 1 places decide
      if (L > 0 && !(L > d ? i + leaf < n && pfx(keys[i + leaf], L - 1) == pfx(k, L - 1)
                           : splits(keys, n, i, L - 1, leaf)))
        break;
      mine |= 1u << L;
    }
  }
  for (int L = 0; L < LEVELS; ++L) {
    const unsigned m = __ballot_sync(0xffffffffu, mine >> L & 1u);
    if (lane == 0) { map[L * nw + w] = m; count[L * nw + w] = __popc(m); }
  }
  if (w == 0 && lane == 0) count[LEVELS * nw] = 0;
}

__device__ __forceinline__ int32_t node_rank(const uint32_t* __restrict__ map, const int32_t* __restrict__ base, int64_t nw,
                                             int L, int64_t i) {
  const int64_t w = L * nw + (i >> 5);
  const unsigned below = (1u << (i & 31)) - 1u;
  return base[w] + (below ? __popc(map[w] & below) : 0);  // (i = n may lie past the level's last word)
}

// the node records
__global__ void __launch_bounds__(256) tree_fill(int64_t n, int64_t nw, const uint64_t* __restrict__ keys, int leaf,
                                                 const uint32_t* __restrict__ map, const int32_t* __restrict__ base,
                                                 int64_t* nb, int64_t* ne, int32_t* lev, int64_t* label,
                                                 int64_t* first_child, int32_t* nchild, int32_t* parent) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint64_t k = keys[i];
  for (int L = 0; L < LEVELS; ++L) {
    if (!(map[L * nw + (i >> 5)] >> (i & 31) & 1u)) continue;
    const int64_t id = node_rank(map, base, nw, L, i);
    const int64_t e = prefix_end(keys, i, n, L);
    nb[id] = i;
    ne[id] = e;
    lev[id] = L;
    label[id] = (int64_t)((1ULL << (3 * L)) | pfx(k, L));
    // the parent is the last node of the level above to start at or before i
    parent[id] = L == 0 ? -1 : node_rank(map, base, nw, L - 1, i) - 1 + (int)(map[(L - 1) * nw + (i >> 5)] >> (i & 31) & 1u);
    if (e - i > leaf && L < MORTON_BITS) {
      const int64_t f = node_rank(map, base, nw, L + 1, i);
      first_child[id] = f;
      nchild[id] = (int32_t)(node_rank(map, base, nw, L + 1, e) - f);
    } else {
      first_child[id] = -1;
      nchild[id] = 0;
    }
  }
}

__global__ void level_starts(int64_t nw, const int32_t* __restrict__ base, int64_t* out) {
  if (threadIdx.x <= LEVELS) out[threadIdx.x] = base[threadIdx.x * nw];
}

}  // namespace

// ---------------------------------------------------------------- tree build

// The node arrays, for at least need nodes (nothing in them outlives a build).
static int ensure_nodes(map_ctx* ctx, int64_t need) {
  DevTree& T = ctx->tree;
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[8], need, &T.label));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[9], need, &T.level));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[10], need, &T.begin));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[11], need, &T.end));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[12], need, &T.first_child));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[13], need, &T.nchild));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[14], need, &T.parent));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[15], need, &T.mass));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[16], 3 * need, &T.com));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[17], need, &T.size_bits));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[18], need, &T.hmax_bits));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[19], 6 * need, &T.bbox_bits));
  return MAP_OK;
}

// The sorted particles, and the node maps and their scan in the buffers of the
// unsorted keys (maps and counts, 5.5 of 8 bytes per particle) and indices (the
// scan, 2.75 of 4), which are done with then.
static int tree_nodes(map_ctx* ctx, const double* x, const double* y, const double* z, const double* m, const double* h,
                      int64_t n, cudaStream_t s, uint32_t** map, int32_t** base) {
  DevTree& T = ctx->tree;
  T.n = n;
  const int tpb = 256;
  uint64_t* keys_in;
  int32_t* idx_in;
  const int64_t nw = (n + 31) / 32, entries = LEVELS * nw, room = n > entries + 1 ? n : entries + 1;
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[0], room, &keys_in));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[1], room, &idx_in));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[2], n, &T.keys));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[3], n, &T.idx));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[4], 5 * n, &T.xs));
  T.ys = T.xs + n; T.zs = T.xs + 2 * n; T.ms = T.xs + 3 * n; T.hs = T.xs + 4 * n;
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[5], n, &T.owner));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[23], 6 * n, &T.split));
  T.hs32 = nullptr;
  if (h) MAP_TRY(ensure_t(ctx, ctx->ws_tree[27], n, &T.hs32));
  morton_keys<<<nblk(n, tpb), tpb, 0, s>>>(n, x, y, z, keys_in, idx_in); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  if (n <= SORT_SMALL) {
    int P = 64;
    while (P < n) P *= 2;
    sort_small<<<1, SORT_THREADS, 0, s>>>((int)n, P, keys_in, T.keys, T.idx); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
  } else {
    size_t tmp_bytes = 0;
    CUDA_TRY(cub::DeviceRadixSort::SortPairs(nullptr, tmp_bytes, keys_in, T.keys, idx_in, T.idx, n, 0, 63, s));
    MAP_TRY(ctx_ensure(ctx, ctx->cub_tmp, tmp_bytes));
    CUDA_TRY(cub::DeviceRadixSort::SortPairs(ctx->cub_tmp.p, tmp_bytes, keys_in, T.keys, idx_in, T.idx, n, 0, 63, s));
  }
  gather_sorted<<<nblk(n, tpb), tpb, 0, s>>>(n, T.idx, x, y, z, m, h, T.xs, T.ys, T.zs, T.ms, T.hs, T.split,
                                             T.hs32); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  *map = reinterpret_cast<uint32_t*>(keys_in);
  int32_t* count = reinterpret_cast<int32_t*>(*map + entries);
  *base = idx_in;
  tree_bits<<<nblk(nw * 32, tpb), tpb, 0, s>>>(n, nw, T.keys, ctx->cfg.leaf_size, *map, count); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  size_t sb = 0;
  CUDA_TRY(cub::DeviceScan::ExclusiveSum(nullptr, sb, count, *base, entries + 1, s));
  MAP_TRY(ctx_ensure(ctx, ctx->cub_tmp, sb));
  CUDA_TRY(cub::DeviceScan::ExclusiveSum(ctx->cub_tmp.p, sb, count, *base, entries + 1, s));
  return MAP_OK;
}

// The node records and sums; the node arrays hold cap nodes.
static int tree_records(map_ctx* ctx, int64_t n, int64_t cap, const uint32_t* map, const int32_t* base, cudaStream_t s) {
  DevTree& T = ctx->tree;
  const int tpb = 256;
  const int64_t nw = (n + 31) / 32;
  double* msum;
  int32_t* arrived;
  float* box32;
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[20], 3 * cap + LEVELS + 1, &msum));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[21], cap, &arrived));
  MAP_TRY(ensure_t(ctx, ctx->ws_tree[24], 8 * cap, &box32));
  T.box32 = box32;
  CUDA_TRY(cudaMemsetAsync(arrived, 0, cap * sizeof(int32_t), s));
  tree_fill<<<nblk(n, tpb), tpb, 0, s>>>(n, nw, T.keys, ctx->cfg.leaf_size, map, base, T.begin, T.end, T.level, T.label,
                                         T.first_child, T.nchild, T.parent); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  const NodeArrays A{T.begin, T.end, T.first_child, T.nchild, T.parent, T.xs, T.ys, T.zs, T.ms, T.hs, T.mass, msum,
                     T.com, T.size_bits, T.hmax_bits, T.bbox_bits, box32, T.owner, arrived};
  // (at most n leaves and as many threads; a small grid strides over the rest)
  const int64_t blocks = cap / 128 + 1 < ctx->sm_count * 16 ? cap / 128 + 1 : ctx->sm_count * 16;
  node_sums<<<(unsigned)blocks, 128, 0, s>>>(base + LEVELS * nw, A); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  return MAP_OK;
}

int tree_build(map_ctx* ctx, const double* x, const double* y, const double* z, const double* m, const double* h,
               int64_t n, cudaStream_t s, bool want_size) {
  DevTree& T = ctx->tree;
  const int tpb = 256;
  uint32_t* map;
  int32_t* base;
  MAP_TRY(tree_nodes(ctx, x, y, z, m, h, n, s, &map, &base));
  const int64_t nw = (n + 31) / 32;
  // the node arrays take the count (one read), n / 4 nodes at least, or what a
  // fixed-workspace context has from the start
  int64_t cap = n / 4 + 64;
  if (ctx->node_cap0 > cap) cap = ctx->node_cap0;
  MAP_TRY(ensure_nodes(ctx, cap));
  int32_t* total = reinterpret_cast<int32_t*>(ctx->h_scratch);
  CUDA_TRY(cudaMemcpyAsync(total, base + LEVELS * nw, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  T.nnodes = *total;
  if (T.nnodes > cap) MAP_TRY(ensure_nodes(ctx, T.nnodes));
  T.level_begin.clear();
  MAP_TRY(tree_records(ctx, n, T.nnodes, map, base, s));
  if (want_size) {
    // the walk also needs the levels' first nodes (in the place of the sums of m
    // x) and the node sizes (the slices' list in the maps' place): both done with
    int64_t* starts = reinterpret_cast<int64_t*>(ctx->ws_tree[20].p);
    int64_t* big = reinterpret_cast<int64_t*>(ctx->ws_tree[0].p);
    level_starts<<<1, 32, 0, s>>>(nw, base, starts); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
    T.level_begin.resize(LEVELS + 1);
    CUDA_TRY(cudaMemcpyAsync(T.level_begin.data(), starts, (LEVELS + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    unsigned long long* d_nbig = ctx->d_counters + 4;
    CUDA_TRY(cudaMemsetAsync(d_nbig, 0, sizeof(unsigned long long), s));
    collect_big<<<nblk(T.nnodes, tpb), tpb, 0, s>>>(T.nnodes, T.begin, T.end, big, d_nbig); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
    node_extent_big<<<(unsigned)(ctx->sm_count * 4), 256, 0, s>>>(big, d_nbig, T.begin, T.end, T.split, T.xs, T.ys,
                                                                  T.zs, T.com, T.size_bits); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
    node_extent_small<<<nblk(n, tpb), tpb, 0, s>>>(n, T.owner, T.parent, T.begin, T.end, T.xs, T.ys, T.zs, T.com,
                                                   T.size_bits); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
    node_size<<<nblk(T.nnodes, tpb), tpb, 0, s>>>(T.nnodes, T.size_bits); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
    CUDA_TRY(cudaStreamSynchronize(s));  // level_begin is read
  }
  return MAP_OK;
}

int64_t tree_scan_entries(int64_t n) { return LEVELS * ((n + 31) / 32) + 1; }

// ---------------------------------------------------------------- tree build with no host reads

int64_t tree_nodes_max(int64_t n, int leaf_size) {
  // internal nodes of one level hold disjoint sets of more than leaf_size
  // particles, so each level has at most n / (leaf_size + 1) of them (21
  // levels split); every leaf holds at least one particle; plus the root
  const int64_t per_level = n / ((int64_t)(leaf_size > 0 ? leaf_size : 0) + 1);
  return n + (int64_t)MORTON_BITS * per_level + 64;
}

int tree_build_graph(map_ctx* ctx, const double* x, const double* y, const double* z, const double* m,
                     const double* h, int64_t n, cudaStream_t s) {
  DevTree& T = ctx->tree;
  uint32_t* map;
  int32_t* base;
  MAP_TRY(tree_nodes(ctx, x, y, z, m, h, n, s, &map, &base));
  const int64_t cap = tree_nodes_max(n, ctx->cfg.leaf_size);
  MAP_TRY(ensure_nodes(ctx, cap));
  MAP_TRY(tree_records(ctx, n, cap, map, base, s));
  // host-side sizes are unknown without a read: an upper bound, no levels
  T.nnodes = cap;
  T.level_begin.clear();
  return MAP_OK;
}
