// Inverse mapping (Section II-B, Eq. 4): a per-cell quantity (the ionic
// fraction f_ion,i the radiative transfer step leaves in every cell) back onto
// the particles,
//     f_ion,a = sum_i f_ion,i f_ai,   f_ai = int_{V_i} W(|r'-r_a|, h_a) dV',
// with the pair integrals f_ai of the last mapping call.  The same weights
// carry the particle masses forward (M_i = sum_a m_a f_ai), so the ionised
// mass is the same on both sides: sum_a m_a f_ion,a = sum_i f_ion,i M_i.
//
// The pair list is cell-major; the sum runs over particles.  The first call
// after a mapping builds a particle-major copy of the list (a stable radix
// sort, so each particle's entries stay in ascending cell order) holding the
// cell and f_ai of every entry; later calls with other cell values reuse it.
// Each particle's terms are fused into its running sum one at a time in
// ascending cell order (acc <- RN(acc + v_i f_ai), one rounding per term), so
// the result equals that sequential FP64 sum bit for bit.
//
// Layout: the particles are taken along the octree's Morton curve (the
// permutation the context's tree holds; any permutation gives the same sums),
// 32 of nearly the same entry count from each 1024 neighbours, and the entries
// of such a group are interleaved: entry q of its particle l at 32 q + l.  A
// lane then sums its own particle straight from coalesced loads, several rounds
// in flight, with nothing staged.  An entry holds the Morton rank of its
// cell's site (the order the pair walk visits cells in) instead of the cell
// index, and every call first permutes the caller's cell values into that
// order: a group's cells are neighbours, and the value gathers hit L1.
// Groups taken from all particles by count, their rows staged 8 entries at a
// time through shared memory, waited for each round's loads in turn: 133 us
// for 200,003 clumpy particles (2.5e7 pairs), 0.58 ms for 2^20; this takes 98 us
// and 0.39 ms.
#include <cub/cub.cuh>

#include "internal.cuh"

namespace {

constexpr int INV_THREADS = 128;

// the place of every particle on the curve (the tree's order; the particles' own
// when there is none of this size), and rank[morton[k]] = k, the Morton rank of
// every cell
__global__ void inv_places(int64_t n, const int32_t* __restrict__ idx, int32_t* __restrict__ place,
                           int32_t* __restrict__ pid, int64_t nc, const int32_t* __restrict__ morton,
                           int32_t* __restrict__ rank) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += stride) {
    const int32_t a = idx ? idx[k] : (int32_t)k;
    place[a] = (int32_t)k;
    pid[k] = a;
  }
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nc; k += stride) rank[morton[k]] = (int32_t)k;
}

// entry p of the cell-major list: its particle's place (the sort key), and its
// cell's rank (high word) and position (the value)
__global__ void inv_pack(int64_t nc, const int64_t* __restrict__ off, const int32_t* __restrict__ idx,
                         const int32_t* __restrict__ place, const int32_t* __restrict__ rank, int32_t* __restrict__ key,
                         unsigned long long* __restrict__ val) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t c = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < nc; c += nw) {
    const int64_t b = off[c], e = off[c + 1];
    const unsigned long long r = (unsigned long long)rank[c] << 32;
    for (int64_t p = b + lane; p < e; p += 32) {
      key[p] = __ldg(place + idx[p]);
      val[p] = r | (unsigned long long)p;
    }
  }
}

// the caller's cell values in Morton order: out[k] = v[morton[k]]
__global__ void inv_permute(int64_t nc, const int32_t* __restrict__ morton, const double* __restrict__ v,
                            double* __restrict__ out) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nc; k += stride) out[k] = __ldg(v + morton[k]);
}

// ioff[a] = number of entries whose particle's place is below a (a = 0..n)
__global__ void inv_bounds(int64_t np, int64_t n, const int32_t* __restrict__ key, int64_t* __restrict__ ioff) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k <= np; k += stride) {
    const int64_t prev = k == 0 ? -1 : (int64_t)key[k - 1];
    const int64_t cur = k == np ? n : (int64_t)key[k];
    for (int64_t a = prev + 1; a <= cur; ++a) ioff[a] = k;
  }
}

// The order of the work: first the particles of more than INV_LONG entries,
// then windows of 2^INV_WINDOW places, by decreasing count within one, to two
// entries (8 bits of the sort's key: up to 2^17 particles sort in two passes).
constexpr unsigned INV_LONG = 256;
constexpr int INV_WINDOW = 10;

// (long_above: INV_LONG, or 0 when every particle with entries is long; nlong,
// zeroed: the number of long particles)
__global__ void inv_keys(int64_t n, int64_t long_above, const int64_t* __restrict__ ioff, uint32_t* __restrict__ key,
                         int32_t* __restrict__ ids, unsigned long long* nlong) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; a < n; a += stride) {
    const int64_t c = ioff[a + 1] - ioff[a];
    key[a] = c > long_above ? 0u : (uint32_t)(((a >> INV_WINDOW) + 1) << 8 | (int64_t)((INV_LONG - c) >> 1));
    ids[a] = (int32_t)a;
    const unsigned here = __activemask(), m = __ballot_sync(here, c > long_above);
    if (m && (int)(threadIdx.x & 31) == __ffs(here) - 1) atomicAdd(nlong, (unsigned long long)__popc(m));
  }
}

// Work items: one per long particle, its entries contiguous, then one per 32
// others in that order, interleaved up to the longest's count.  Items beyond
// the last (up to room, for the most long particles there can be) are empty.
__device__ __forceinline__ int64_t item_count(int64_t n, int64_t nlong) { return nlong + (n - nlong + 31) / 32; }

// an item's entries, padding included (one warp per item)
__global__ void inv_sizes(int64_t n, int64_t room, const int64_t* __restrict__ nlong_p, const int32_t* __restrict__ order,
                          const int64_t* __restrict__ ioff, int64_t* __restrict__ size) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5, nlong = *nlong_p, items = item_count(n, nlong);
  for (int64_t it = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < room; it += nw) {
    if (it >= items) {  // nothing from here on: 32 places at a time
      for (int64_t k = it + (int64_t)lane * nw; k < room; k += 32 * nw) size[k] = 0;
      return;
    }
    const int64_t k = it < nlong ? it : nlong + 32 * (it - nlong) + lane;
    const int64_t r = k < n ? order[k] : -1;
    // (a group's counts are at most INV_LONG; a long particle's, all lanes alike, may not fit 32 bits)
    const int64_t c = r >= 0 ? ioff[r + 1] - ioff[r] : 0;
    const int64_t most = it < nlong ? c : 32 * (int64_t)__reduce_max_sync(0xffffffffu, (unsigned)c);
    if (lane == 0) size[it] = most;
  }
}

// the items' entries: the cell's rank and f_ai of the sorted values
// (FILL_PARTS warps per item)
constexpr int FILL_PARTS = 4;
__global__ void inv_fill(int64_t n, const int64_t* __restrict__ nlong_p, const int32_t* __restrict__ order,
                         const int64_t* __restrict__ ioff, const int64_t* __restrict__ base,
                         const unsigned long long* __restrict__ val, const double* __restrict__ frac,
                         int32_t* __restrict__ cell, double* __restrict__ f) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5, nlong = *nlong_p, items = item_count(n, nlong);
  for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < FILL_PARTS * items; t += nw) {
    const int64_t it = t / FILL_PARTS;
    const int64_t b = base[it], size = base[it + 1] - b;
    const bool whole = it < nlong;
    const int64_t k = whole ? it : nlong + 32 * (it - nlong) + lane;
    const int64_t r = k < n ? order[k] : -1;
    const int64_t lo = r >= 0 ? ioff[r] : 0, cnt = r >= 0 ? ioff[r + 1] - lo : 0;
#pragma unroll 4
    for (int64_t j = 32 * (t % FILL_PARTS) + lane; j < size; j += 32 * FILL_PARTS) {
      const int64_t q = whole ? j : j >> 5;
      const bool on = q < cnt;
      const unsigned long long v = on ? __ldg(val + lo + q) : 0ull;
      cell[b + j] = (int32_t)(v >> 32);
      f[b + j] = on ? __ldg(frac + (v & 0xffffffffull)) : 0.0;
    }
  }
}

// A long particle: chunks of INV_CHUNK entries loaded coalesced, staged in
// shared memory as (cell value, f_ai) and fused into the running sum by lane 0
// in order, the next chunk's loads in flight.  A group: lane l sums particle l,
// INV_U rounds of entries in flight.
constexpr int INV_CHUNK = 256;
constexpr int INV_U = 8;

__global__ void __launch_bounds__(INV_THREADS) inv_apply(int64_t n, const int64_t* __restrict__ nlong_p,
                                                         const int32_t* __restrict__ order,
                                                         const int32_t* __restrict__ pid,
                                                         const int64_t* __restrict__ ioff,
                                                         const int64_t* __restrict__ base,
                                                         const int32_t* __restrict__ cell,
                                                         const double* __restrict__ f,
                                                         const double* __restrict__ cv, double* __restrict__ out) {
  __shared__ double2 sp[INV_THREADS / 32][INV_CHUNK];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t nlong = *nlong_p, items = item_count(n, nlong);
  const int64_t it = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (it >= items) return;  // whole warp
  const int64_t b = base[it];
  const int64_t size = base[it + 1] - b;
  int c[INV_U];
  double g[INV_U], v[INV_U];
  // the entries of places q, q + 32, ... of the item (its last one repeated past the end)
  auto load = [&](int64_t q) {
#pragma unroll
    for (int u = 0; u < INV_U; ++u) {
      const int64_t k = q + 32 * u < size ? q + 32 * u : size - 1;
      c[u] = __ldg(cell + b + k);
      g[u] = __ldg(f + b + k);
    }
  };
  auto values = [&]() {
#pragma unroll
    for (int u = 0; u < INV_U; ++u) v[u] = __ldg(cv + c[u]);
  };
  double acc = 0.0;
  if (it < nlong) {
    load(lane);
    for (int64_t q0 = 0; q0 < size; q0 += INV_CHUNK) {
      values();
#pragma unroll
      for (int u = 0; u < INV_U; ++u) sp[w][32 * u + lane] = make_double2(v[u], g[u]);
      __syncwarp();
      if (q0 + INV_CHUNK < size) load(q0 + INV_CHUNK + lane);
      if (lane == 0) {
        const int m = size - q0 < INV_CHUNK ? (int)(size - q0) : INV_CHUNK;
        for (int q = 0; q < m; ++q) acc = __fma_rn(sp[w][q].x, sp[w][q].y, acc);
      }
      __syncwarp();
    }
    if (lane == 0) out[pid[order[it]]] = acc;
    return;
  }
  const int64_t k = nlong + 32 * (it - nlong) + lane;
  const int64_t r = k < n ? order[k] : -1;
  const int cnt = r >= 0 ? (int)(ioff[r + 1] - ioff[r]) : 0;
  if (size > 0) {
    load(lane);
    for (int q = 0; 32 * (int64_t)q < size; q += INV_U) {
      values();
      double h[INV_U];
#pragma unroll
      for (int u = 0; u < INV_U; ++u) h[u] = g[u];
      if (32 * (int64_t)(q + INV_U) < size) load(32 * (int64_t)(q + INV_U) + lane);
#pragma unroll
      for (int u = 0; u < INV_U; ++u)
        if (q + u < cnt) acc = __fma_rn(v[u], h[u], acc);
    }
  }
  if (r >= 0) out[pid[r]] = acc;
}

// bits that hold every value below n (at most 32)
int bits_for(int64_t n) {
  int b = 1;
  while (b < 32 && (int64_t(1) << b) < n) ++b;
  return b;
}

// groups = false: every particle's entries contiguous, summed by a warp of its
// own, for a budget that does not hold the groups' padding.
int build_index(map_ctx* ctx, cudaStream_t s, bool groups) {
  const int64_t np = ctx->n_pairs, nc = ctx->last_ncell, n = ctx->last_npart;
  int64_t* ioff;
  MAP_TRY(ensure_t(ctx, ctx->ws_inv[0], n + 1, &ioff));
  ctx->inv_off = ioff;
  const unsigned g = (unsigned)ctx->sm_count * 8;
  int32_t *place, *pid;
  MAP_TRY(ensure_t(ctx, ctx->ws_inv[6], n, &place));
  MAP_TRY(ensure_t(ctx, ctx->ws_inv[13], n, &pid));
  // the pair walk's Morton order of the cells, sorted by pairs_build with the
  // list this copy is made from (a buffer no other step writes)
  int32_t* rank = nullptr;
  if (np > 0) {
    if (ctx->ws_pairs[14].cap < (size_t)nc * sizeof(int32_t)) return MAP_EINVAL;
    ctx->inv_morton = static_cast<const int32_t*>(ctx->ws_pairs[14].p);
    MAP_TRY(ensure_t(ctx, ctx->ws_inv[11], nc, &rank));
  }
  inv_places<<<g, 256, 0, s>>>(n, ctx->tree.n == n ? ctx->tree.idx : nullptr, place, pid, np > 0 ? nc : 0,
                               ctx->inv_morton, rank);
  ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  ctx->inv_pid = pid;
  // A window's groups, by decreasing count to two entries, are padded by at most
  // 32 x (its largest - its smallest count + a 1 for each of 33 groups), the group
  // that crosses into the next window by 32 x 256, the last one by its missing
  // lanes: 18 entries per particle and 4 x 8192 hold them all.
  const int64_t room = groups ? np + 18 * n + 4 * 8192 : np;
  // (the particles of more than INV_LONG entries: at most np / (INV_LONG + 1))
  const int64_t longest = groups && np / (INV_LONG + 1) < n ? np / (INV_LONG + 1) : n;
  unsigned long long* val_s = nullptr;
  if (np > 0) {
    unsigned long long* val;  // (in the place of f_ai, and key in the cells' place, which are written after the sort)
    int32_t *key, *key_s;
    MAP_TRY(ensure_t(ctx, ctx->ws_inv[1], room, &key));
    MAP_TRY(ensure_t(ctx, ctx->ws_inv[2], room, &val));
    MAP_TRY(ensure_t(ctx, ctx->ws_inv[3], np, &val_s));
    MAP_TRY(ensure_t(ctx, ctx->ws_inv[4], np, &key_s));
    inv_pack<<<g, 256, 0, s>>>(nc, ctx->pair_off, ctx->pair_idx, place, rank, key, val); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
    size_t tb = 0;
    const int nb = bits_for(n);
    CUDA_TRY(cub::DeviceRadixSort::SortPairs(nullptr, tb, key, key_s, val, val_s, np, 0, nb, s));
    MAP_TRY(ctx_ensure(ctx, ctx->cub_tmp, tb));
    CUDA_TRY(cub::DeviceRadixSort::SortPairs(ctx->cub_tmp.p, tb, key, key_s, val, val_s, np, 0, nb, s));
    inv_bounds<<<g, 256, 0, s>>>(np, n, key_s, ioff); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
  } else {
    CUDA_TRY(cudaMemsetAsync(ioff, 0, (n + 1) * sizeof(int64_t), s));
    ctx->inv_cell = nullptr;
    ctx->inv_frac = nullptr;
  }
  uint32_t *okey, *okey_s;
  int32_t *ids, *order;
  MAP_TRY(ensure_t(ctx, ctx->ws_inv[7], 2 * n, &okey));
  ids = place;  // (done with)
  MAP_TRY(ensure_t(ctx, ctx->ws_inv[9], n, &order));
  okey_s = okey + n;
  int64_t* nlong;
  MAP_TRY(ensure_t(ctx, ctx->ws_inv[10], 1, &nlong));
  CUDA_TRY(cudaMemsetAsync(nlong, 0, sizeof(int64_t), s));
  inv_keys<<<g, 256, 0, s>>>(n, groups ? INV_LONG : 0, ioff, okey, ids, reinterpret_cast<unsigned long long*>(nlong));
  ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  size_t tb2 = 0;
  const int cb = bits_for(((n >> INV_WINDOW) + 2) << 8);
  CUDA_TRY(cub::DeviceRadixSort::SortPairs(nullptr, tb2, okey, okey_s, ids, order, n, 0, cb, s));
  MAP_TRY(ctx_ensure(ctx, ctx->cub_tmp, tb2));
  CUDA_TRY(cub::DeviceRadixSort::SortPairs(ctx->cub_tmp.p, tb2, okey, okey_s, ids, order, n, 0, cb, s));
  if (np > 0) {
    int32_t* cell = static_cast<int32_t*>(ctx->ws_inv[1].p);
    double* f = static_cast<double*>(ctx->ws_inv[2].p);
    const int64_t items = longest + (n - longest + 31) / 32 + 1;
    int64_t *size, *base;
    MAP_TRY(ensure_t(ctx, ctx->ws_inv[14], 2 * items, &size));
    base = size + items;
    inv_sizes<<<g, 256, 0, s>>>(n, items, nlong, order, ioff, size); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
    size_t tb = 0;
    CUDA_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tb, size, base, items, s));
    MAP_TRY(ctx_ensure(ctx, ctx->cub_tmp, tb));
    CUDA_TRY(cub::DeviceScan::ExclusiveSum(ctx->cub_tmp.p, tb, size, base, items, s));
    inv_fill<<<g, 256, 0, s>>>(n, nlong, order, ioff, base, val_s, ctx->pair_frac, cell, f); ++ctx->launches;
    CUDA_TRY(cudaGetLastError());
    ctx->inv_cell = cell;
    ctx->inv_frac = f;
    ctx->inv_base = base;
  }
  ctx->inv_order = order;
  ctx->inv_nlong = nlong;
  ctx->inv_longest = longest;
  double* cv;  // (the call's cell values, so that a call after this one finds its room)
  MAP_TRY(ensure_t(ctx, ctx->ws_inv[12], nc, &cv));
  ctx->inv_ready = true;
  // the copy reads the pair list, which a later map_get_pairs sorts in place:
  // that sort runs on this call's stream or one ordered after it (ctx_enter)
  return MAP_OK;
}

}  // namespace

extern "C" int map_cells_to_particles(map_ctx* ctx, const double* cell_value, double* particle_value, int64_t n,
                                      void* stream) {
  if (!ctx || !particle_value || (!cell_value && ctx->last_ncell > 0)) return MAP_EINVAL;
  if (!ctx->pair_off || !ctx->pair_frac || n != ctx->last_npart) return MAP_EINVAL;
  if (ctx->n_pairs >= (int64_t(1) << 32) || ctx->last_ncell >= (int64_t(1) << 31)) return MAP_EINVAL;
  if (n == 0) return MAP_OK;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  MAP_ENTER(ctx, s);
  if (!ctx->inv_ready) {
    int r = build_index(ctx, s, true);
    if (r == MAP_ENOMEM) {
      for (int k : {1, 2, 14}) {
        DevBuf& b = ctx->ws_inv[k];
        dev_free(ctx, b.p);
        ctx->bytes_in_use -= b.cap;
        b = DevBuf();
      }
      r = build_index(ctx, s, false);
    }
    if (r != MAP_OK) return r;
  }
  if (!ctx->inv_cell) {  // no pairs: every sum is empty
    CUDA_TRY(cudaMemsetAsync(particle_value, 0, n * sizeof(double), s));
    return MAP_OK;
  }
  const int64_t nc = ctx->last_ncell;
  double* cv;
  MAP_TRY(ensure_t(ctx, ctx->ws_inv[12], nc, &cv));
  inv_permute<<<(unsigned)ctx->sm_count * 8, 256, 0, s>>>(nc, ctx->inv_morton, cell_value, cv); ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  // a warp per item; their number, one for each long particle and one for 32 of
  // the rest, stays on the device
  const int64_t longest = ctx->inv_longest, items = longest + (n - longest + 31) / 32 + 1;
  inv_apply<<<nblk(items * 32, INV_THREADS), INV_THREADS, 0, s>>>(n, ctx->inv_nlong, ctx->inv_order, ctx->inv_pid,
                                                                  ctx->inv_off, ctx->inv_base, ctx->inv_cell,
                                                                  ctx->inv_frac, cv, particle_value);
  ++ctx->launches;
  CUDA_TRY(cudaGetLastError());
  return MAP_OK;
}
