// Epoch order of the blocked SGD (Algorithms 1-2), laid out on the device.
//
// Algorithm 1 visits the blocks in the steps of Figure 2 and Algorithm 2
// walks a block row by row, then column by column. What fixes the result is
// only, for every user and every item, the order in which its ratings are
// processed: a rating reads and writes one user's and one item's parameters
// and nothing else. The training kernels (kernels_sgd.cu) keep exactly those
// two orders and run everything else in parallel. This file makes what they
// need:
//   * tasks: one side owns its parameters while it works. The side with the
//     fewer ids owns (items when n <= m; its ids have the longer lists of
//     ratings, and the longest list is the longest chain). A task is one
//     owner's ratings in one block, ordered by the other side's local index;
//   * the ratings in task order, the tasks ordered by (step, owner's local
//     index, block within the step). A task then only ever waits for ratings
//     of earlier tasks;
//   * for every rating, how many ratings of its other-side id come before it
//     in the epoch, and for every task the same for its owner: the versions
//     of the parameters that it has to find.
//
// The order is a stable radix sort (radix_sort.cuh) of the key (step, owner's
// local index, block in the step, other side's local index). Stability keeps repeated cells in input order. The
// versions are ranks within equal ids, from two more stable sorts (by the
// other side's id, by the owner's id) of the positions in task order, which
// list every id's ratings in its own epoch order.
//
// Counting, bucket scatter with atomics and a sort of every
// bucket, which this replaces, took 350 us (8 x 8 blocks) to 610 us (64 x 64)
// for 900,189 ratings, most of it in the one-CTA scan of q m buckets and in
// the buckets' insertion sorts.
#include <type_traits>

#include "kernels.h"
#include "radix_sort.cuh"

namespace bsvd {

namespace {

// What a key is made of: the owner's side, and the ranges of its parts.
struct KeyDesc {
  int own_items;
  int64_t lown;       // largest block extent on the owner's side
  int64_t slots;      // blocks per step, at most
  int minor_bits;     // bits of the other side's local index
};

__device__ __forceinline__ u64 task_key(const GridDesc &g, const KeyDesc &d,
                                        int32_t blk, int32_t r, int32_t c,
                                        int32_t *minor) {
  int64_t step, slot;
  if (g.diag) {
    step = 0;
    slot = blk;
  } else {
    // Figure 2: step s holds the blocks ((j + s) mod p, j), or
    // (i, (i + s) mod q) when there are fewer block rows than columns
    const int32_t bi = blk / g.q, bj = blk % g.q;
    if (g.p >= g.q) {
      step = bi >= bj ? bi - bj : bi - bj + g.p;
      slot = bj;
    } else {
      step = bj >= bi ? bj - bi : bj - bi + g.q;
      slot = bi;
    }
  }
  *minor = d.own_items ? r : c;
  const int64_t lo = d.own_items ? c : r;
  return (u64)((step * d.lown + lo) * d.slots + slot);
}

// Sort keys. part 0: task key above the minor index; part 1: the minor index
// alone, part 2: the task key alone of the ratings listed in `list` (two
// sorts, for grids whose whole key does not fit 64 bits). A rating with an id
// out of range is reported; its key is that of cell (0, 0) of block 0, whether
// or not the block has one (sgd_max_tasks counts it).
template <typename V>
__global__ void __launch_bounds__(256)
k_sgd_keys(GridDesc g, KeyDesc d, int64_t nnz, const int32_t *__restrict__ u,
           const int32_t *__restrict__ it, int part,
           const V *__restrict__ list, u64 *__restrict__ key, int32_t *err) {
  pdl_wait();
  pdl_trigger();
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nnz;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = list ? (int64_t)list[t] : t;
    int32_t blk = 0, r = 0, c = 0, minor;
    if (!locate(g, u[e], it[e], &blk, &r, &c)) {
      atomicOr(err, kErrIndex);
      blk = r = c = 0;
    }
    const u64 tk = task_key(g, d, blk, r, c, &minor);
    key[t] = part == 0 ? (tk << d.minor_bits) | (u64)minor
             : part == 1 ? (u64)minor
                         : tk;
  }
}

// The ratings in task order, and how many tasks start in every 4,096 of
// them. `key` is the sorted key, the task key above `shift`.
template <typename V>
__global__ void __launch_bounds__(256)
k_sgd_gather(GridDesc g, int64_t nnz, const V *__restrict__ src,
             const u64 *__restrict__ key, int shift,
             const int32_t *__restrict__ u, const int32_t *__restrict__ it,
             const float *__restrict__ x, int32_t *__restrict__ su,
             int32_t *__restrict__ si, float *__restrict__ sx,
             V *__restrict__ tile_tasks) {
  pdl_wait();
  pdl_trigger();
  __shared__ int starts;
  if (threadIdx.x == 0) starts = 0;
  __syncthreads();
  int mine = 0;
  const int64_t base = (int64_t)blockIdx.x * kRsTile;
#pragma unroll 4
  for (int j = 0; j < kRsTile / 256; ++j) {
    const int64_t t = base + j * 256 + threadIdx.x;
    if (t >= nnz) break;
    const int64_t s = (int64_t)src[t];
    int32_t uu = u[s], ii = it[s];
    // out of range: reported by k_sgd_keys; kept inside the arrays here
    if (uu < 0 || (int64_t)uu >= g.m) uu = 0;
    if (ii < 0 || (int64_t)ii >= g.n) ii = 0;
    su[t] = uu;
    si[t] = ii;
    sx[t] = x[s];
    mine += t == 0 || (key[t] >> shift) != (key[t - 1] >> shift);
  }
  if (mine) atomicAdd(&starts, mine);
  __syncthreads();
  if (threadIdx.x == 0) tile_tasks[blockIdx.x] = (V)starts;
}

// One CTA: exclusive scan of the tiles' task counts; the total to *ntasks.
template <typename V>
__global__ void __launch_bounds__(1024)
k_sgd_task_scan(V *__restrict__ tile_tasks, int64_t ntiles,
                int64_t *__restrict__ ntasks) {
  pdl_wait();
  pdl_trigger();
  __shared__ V part[1024];
  V run = 0;
  for (int64_t b = 0; b < ntiles; b += 1024) {
    const int64_t e = b + threadIdx.x;
    const V v = e < ntiles ? tile_tasks[e] : 0;
    part[threadIdx.x] = v;
    __syncthreads();
    for (int w = 1; w < 1024; w <<= 1) {
      const V o = threadIdx.x >= w ? part[threadIdx.x - w] : 0;
      __syncthreads();
      part[threadIdx.x] += o;
      __syncthreads();
    }
    if (e < ntiles) tile_tasks[e] = run + part[threadIdx.x] - v;
    run += part[1023];
    __syncthreads();
  }
  if (threadIdx.x == 0) *ntasks = (int64_t)run;
}

// First rating of every task, in order; task_first[ntasks] = nnz.
template <typename V>
__global__ void __launch_bounds__(256)
k_sgd_task_first(int64_t nnz, const u64 *__restrict__ key, int shift,
                 const V *__restrict__ tile_tasks,
                 const int64_t *__restrict__ ntasks,
                 V *__restrict__ task_first) {
  pdl_wait();
  pdl_trigger();
  __shared__ int wcount[8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t base = (int64_t)blockIdx.x * kRsTile;
  V run = tile_tasks[blockIdx.x];
  for (int j = 0; j < kRsTile / 256; ++j) {
    const int64_t t = base + j * 256 + threadIdx.x;
    const bool start =
        t < nnz && (t == 0 || (key[t] >> shift) != (key[t - 1] >> shift));
    const unsigned b = __ballot_sync(0xffffffffu, start);
    if (lane == 0) wcount[warp] = __popc(b);
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      before += w < warp ? wcount[w] : 0;
      all += wcount[w];
    }
    if (start)
      task_first[run + before + __popc(b & ((1u << lane) - 1u))] = (V)t;
    run += all;
    __syncthreads();
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) task_first[*ntasks] = (V)nnz;
}

__global__ void __launch_bounds__(256)
k_sgd_id_keys(int64_t nnz, const int32_t *__restrict__ id,
              u64 *__restrict__ key) {
  pdl_wait();
  pdl_trigger();
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nnz;
       t += (int64_t)gridDim.x * blockDim.x)
    key[t] = (u64)id[t];
}

// Start of every id's run in the list sorted by id.
template <typename V>
__global__ void __launch_bounds__(256)
k_sgd_run_start(int64_t nnz, const u64 *__restrict__ key,
                V *__restrict__ start) {
  pdl_wait();
  pdl_trigger();
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nnz;
       t += (int64_t)gridDim.x * blockDim.x)
    if (t == 0 || key[t] != key[t - 1]) start[key[t]] = (V)t;
}

// ver[position] = ratings of the same id before it (modulo 2^32).
template <typename V>
__global__ void __launch_bounds__(256)
k_sgd_versions(int64_t nnz, const u64 *__restrict__ key,
               const V *__restrict__ pos, const V *__restrict__ start,
               unsigned *__restrict__ ver) {
  pdl_wait();
  pdl_trigger();
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nnz;
       t += (int64_t)gridDim.x * blockDim.x)
    ver[pos[t]] = (unsigned)((V)t - start[key[t]]);
}

int bits_of(int64_t largest) {
  int b = 0;
  while (largest > 0) {
    ++b;
    largest >>= 1;
  }
  return b;
}

int grid_of(int64_t n) {
  int64_t want = (n + 255) / 256;
  if (want < 1) want = 1;
  if (want > 152 * 8) want = 152 * 8;
  return (int)want;
}

template <typename V>
cudaError_t order_impl(const GridDesc &g, const SgdOrder &o, int64_t nnz,
                       const int32_t *u, const int32_t *i, const float *x,
                       int64_t *launches, int32_t *err, cudaStream_t st) {
  u64 *const key[2] = {static_cast<u64 *>(o.key[0]),
                       static_cast<u64 *>(o.key[1])};
  V *const val[2] = {static_cast<V *>(o.val[0]), static_cast<V *>(o.val[1])};
  const int64_t ntiles = (nnz + kRsTile - 1) / kRsTile;
  V *hist = static_cast<V *>(o.hist);
  V *total = hist + 256 * ntiles;
  V *tile_tasks = total + 256;
  V *first = static_cast<V *>(o.task_first);
  V *start = static_cast<V *>(o.start);
  KeyDesc d;
  d.own_items = o.own_items;
  d.lown = o.own_items ? o.max_cols : o.max_rows;
  d.slots = g.diag ? g.p : (g.p >= g.q ? g.q : g.p);
  const int64_t other = o.own_items ? o.max_rows : o.max_cols;
  d.minor_bits = bits_of(other - 1);
  const int64_t steps = g.diag ? 1 : (g.p >= g.q ? g.p : g.q);
  const int tbits = bits_of(steps * d.lown * d.slots - 1);
  int cur = 0, shift = d.minor_bits;
  cudaError_t e;
  const dim3 each(grid_of(nnz)), tiles((unsigned)ntiles), cta(256);
  auto keys = [&](int part, const V *list, u64 *out) -> cudaError_t {
    ++*launches;
    return launch_pdl(k_sgd_keys<V>, each, cta, 0, st, g, d, nnz, u, i, part,
                      list, out, err);
  };
  if (tbits + d.minor_bits <= 64) {
    if ((e = keys(0, nullptr, key[0])) != cudaSuccess) return e;
    e = radix_sort<V>(key, val, &cur, true, nnz, tbits + d.minor_bits, hist,
                      total, launches, st);
  } else {
    if ((e = keys(1, nullptr, key[0])) != cudaSuccess) return e;
    e = radix_sort<V>(key, val, &cur, true, nnz, d.minor_bits, hist, total,
                      launches, st);
    if (e != cudaSuccess) return e;
    if ((e = keys(2, val[cur], key[cur])) != cudaSuccess) return e;
    e = radix_sort<V>(key, val, &cur, false, nnz, tbits, hist, total, launches,
                      st);
    shift = 0;
  }
  if (e != cudaSuccess) return e;
  if ((e = launch_pdl(k_sgd_gather<V>, tiles, cta, 0, st, g, nnz,
                      (const V *)val[cur], (const u64 *)key[cur], shift, u, i,
                      x, o.su, o.si, o.sx, tile_tasks)) != cudaSuccess)
    return e;
  if ((e = launch_pdl(k_sgd_task_scan<V>, dim3(1), dim3(1024), 0, st,
                      tile_tasks, ntiles, o.ntasks)) != cudaSuccess)
    return e;
  if ((e = launch_pdl(k_sgd_task_first<V>, tiles, cta, 0, st, nnz,
                      (const u64 *)key[cur], shift, (const V *)tile_tasks,
                      (const int64_t *)o.ntasks, first)) != cudaSuccess)
    return e;
  *launches += 3;
  // the versions: other side, then owner
  for (int side = 0; side < 2; ++side) {
    const bool items = (side == 0) != (o.own_items != 0);
    const int32_t *id = items ? o.si : o.su;
    cur = 0;
    if ((e = launch_pdl(k_sgd_id_keys, each, cta, 0, st, nnz, id, key[0])) !=
        cudaSuccess)
      return e;
    e = radix_sort<V>(key, val, &cur, true, nnz,
                      bits_of((items ? g.n : g.m) - 1), hist, total, launches,
                      st);
    if (e != cudaSuccess) return e;
    if ((e = launch_pdl(k_sgd_run_start<V>, each, cta, 0, st, nnz,
                        (const u64 *)key[cur], start)) != cudaSuccess)
      return e;
    if ((e = launch_pdl(k_sgd_versions<V>, each, cta, 0, st, nnz,
                        (const u64 *)key[cur], (const V *)val[cur],
                        (const V *)start,
                        side == 0 ? o.other_ver : o.own_ver)) != cudaSuccess)
      return e;
    *launches += 3;
  }
  return cudaGetLastError();
}

}  // namespace

size_t sgd_index_bytes(int64_t nnz) {
  return nnz <= (int64_t)UINT32_MAX ? sizeof(unsigned) : sizeof(u64);
}

size_t sgd_hist_bytes(int64_t nnz) {
  const int64_t ntiles = (nnz + kRsTile - 1) / kRsTile;
  return sgd_index_bytes(nnz) * (size_t)(257 * ntiles + 256);
}

cudaError_t launch_sgd_order(const GridDesc &g, const SgdOrder &o, int64_t nnz,
                             const int32_t *u, const int32_t *i, const float *x,
                             int64_t *launches, int32_t *err,
                             cudaStream_t st) {
  if (nnz <= 0) return cudaMemsetAsync(o.ntasks, 0, sizeof(int64_t), st);
  return nnz <= (int64_t)UINT32_MAX
             ? order_impl<unsigned>(g, o, nnz, u, i, x, launches, err, st)
             : order_impl<u64>(g, o, nnz, u, i, x, launches, err, st);
}

}  // namespace bsvd
