// Partition, block means and dense scatter (Section 3, Eq. "datax").
//
// Pass 1 (k_count) maps every training rating to its block and adds its
// count and its value to per-block totals. Values are summed as 64-bit
// fixed point with 32 fraction bits (x * 2^32), so the totals are exact
// integers and do not depend on the order of the atomic adds.
// Pass 2 (k_means) turns the totals into mu_b = fl32(fl64(sum) / count).
// Pass 3 (k_scatter, or k_scatter_planes for the exact tensor-core Gram)
// writes fl32(x - mu_b), or its bf16 rounding, or the bf16 offset and the
// observation mask, into the zeroed dense blocks.
//
// Every pass looks up a block per rating. A CTA keeps the grid's bounds and
// what it needs of each block in shared memory (BoundsTable, Dest); from
// global memory a rating's six or more lookups touch up to 32 lines per warp
// each. A thread takes kRatings ratings at a time, so that their loads
// overlap: counting 90 million ratings into 256 blocks takes 0.87 ms (1.43
// before both). The scatter of that many into 17 GB of bf16 cells stays at 3.2
// to 3.8 ms: each 2-byte write is a 32-byte sector of its own that DRAM reads
// and writes, about 28 billion a second at any number of ratings in flight.
#include <type_traits>

#include "kernels.h"

namespace bsvd {

namespace {

constexpr int kSmemBlocks = 2048;   // per-CTA histogram size limit
constexpr int kRatings = 4;            // ratings a thread has in flight

// A batch's ids to the stacked coordinates, in place: 16 bytes of traffic a
// rating; the piece is found by bisection (the table stays in the L1).
__global__ void k_stack_ids(int64_t nnz, int nb,
                            const int64_t *__restrict__ starts,
                            const int64_t *__restrict__ add,
                            int32_t *__restrict__ ids) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nnz;
       t += (int64_t)gridDim.x * blockDim.x) {
    int lo = 0, hi = nb;                 // starts[lo] <= t < starts[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (starts[mid] <= t) lo = mid;
      else hi = mid;
    }
    ids[t] = (int32_t)((uint32_t)ids[t] + (uint32_t)add[lo]);
  }
}

__global__ void k_perm_mark(const int32_t *perm, int64_t n, int32_t *seen,
                            int32_t *err) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    int32_t v = perm[t];
    if (v < 0 || (int64_t)v >= n) { atomicOr(err, kErrBadPerm); continue; }
    atomicAdd(&seen[v], 1);
  }
}

__global__ void k_perm_verify(const int32_t *seen, int64_t n, int32_t *err) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x)
    if (seen[t] != 1) atomicOr(err, kErrBadPerm);
}

__device__ __forceinline__ bool rating_ok(float x) {
  return isfinite(x) && fabsf(x) < 2147483648.0f;
}

__device__ __forceinline__ long long fixed32(float x) {
  // x * 2^32 is exact in float64; round to the nearest integer. (An
  // integer-only version with a branch per exponent range measured about
  // 1 ms slower per pass over the large workload's 90 million ratings.)
  return __double2ll_rn(__dmul_rn((double)x, 4294967296.0));
}

// Counts and fixed-point sums per block. In shared memory a sum is two 32-bit
// words, added separately: the low one is zero for whole ratings and is then
// left alone, and a carry out of it goes to the high one (64-bit shared
// atomics are loops of compare and swap). When a warp's ratings are all in one
// block, as in a batch of matrices one after another, they are summed in
// registers first (16 matrices of the served form: 341 -> 56 us).
struct CountTable {
  unsigned cnt[kSmemBlocks], lo[kSmemBlocks], hi[kSmemBlocks];
  BoundsTable bounds;
};

template <bool TABLE>
__global__ void __launch_bounds__(256)
k_count(GridDesc g, int64_t nnz, const int32_t *__restrict__ u,
        const int32_t *__restrict__ it, const float *__restrict__ x,
        int32_t nblocks, unsigned long long *counts, long long *sums,
        unsigned int *maxabs_bits, int32_t *err) {
  extern __shared__ unsigned char smem[];
  CountTable &t = *reinterpret_cast<CountTable *>(smem);
  __shared__ unsigned int s_max;
  const bool use_smem = nblocks <= kSmemBlocks;
  if (use_smem) {
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x)
      t.cnt[b] = t.lo[b] = t.hi[b] = 0;
  }
  if (TABLE) t.bounds.fill(g);
  if (threadIdx.x == 0) s_max = 0;
  __syncthreads();
  unsigned int local_max = 0;
  int32_t local_err = 0;
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  // whole warps, so that every lane takes part in the votes
  for (int64_t t0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31);
       t0 < nnz; t0 += kRatings * stride) {
    int32_t uu[kRatings], ii[kRatings];
    float xx[kRatings];
#pragma unroll
    for (int k = 0; k < kRatings; ++k) {
      const int64_t e = t0 + k * stride + lane;
      const bool in = e < nnz;
      uu[k] = in ? u[e] : 0;
      ii[k] = in ? it[e] : 0;
      xx[k] = in ? x[e] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < kRatings; ++k) {
      bool ok = t0 + k * stride + lane < nnz;
      int32_t blk = -1, ru, ci;
      if (ok) {
        if (!find_block<TABLE>(g, t.bounds, uu[k], ii[k], &blk, &ru, &ci)) {
          local_err |= kErrIndex;
          ok = false;
        } else if (!rating_ok(xx[k])) {
          local_err |= kErrValue;
          ok = false;
        }
      }
      const unsigned on = __ballot_sync(0xffffffffu, ok);
      if (on == 0) continue;
      if (ok) local_max = max(local_max, __float_as_uint(fabsf(xx[k])));
      const long long fx = ok ? fixed32(xx[k]) : 0;
      if (!use_smem) {
        if (ok) {
          atomicAdd(&counts[blk], 1ull);
          atomicAdd((unsigned long long *)&sums[blk], (unsigned long long)fx);
        }
        continue;
      }
      const unsigned lo = (unsigned)fx, hi = (unsigned)(fx >> 32);
      const int first = __ffs(on) - 1;
      const int32_t b0 = __shfl_sync(0xffffffffu, blk, first);
      const bool same = __all_sync(0xffffffffu, !ok || (blk == b0 && lo == 0));
      if (same) {
        const unsigned sum = __reduce_add_sync(0xffffffffu, hi);
        if (lane == first) {
          atomicAdd(&t.cnt[b0], (unsigned)__popc(on));
          atomicAdd(&t.hi[b0], sum);
        }
      } else if (ok) {
        atomicAdd(&t.cnt[blk], 1u);
        unsigned up = hi;
        if (lo) {
          const unsigned old = atomicAdd(&t.lo[blk], lo);
          up += old + lo < old ? 1u : 0u;
        }
        atomicAdd(&t.hi[blk], up);
      }
    }
  }
  // warp-reduce the max and the error bits, one shared atomic per warp
  for (int o = 16; o > 0; o >>= 1) {
    local_max = max(local_max, __shfl_xor_sync(0xffffffffu, local_max, o));
    local_err |= __shfl_xor_sync(0xffffffffu, local_err, o);
  }
  if (lane == 0) {
    atomicMax(&s_max, local_max);
    if (local_err) atomicOr(err, local_err);
  }
  __syncthreads();
  if (use_smem) {
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
      if (t.cnt[b]) {
        atomicAdd(&counts[b], (unsigned long long)t.cnt[b]);
        atomicAdd((unsigned long long *)&sums[b],
                  ((unsigned long long)t.hi[b] << 32) + t.lo[b]);
      }
    }
  }
  if (threadIdx.x == 0 && s_max) atomicMax(maxabs_bits, s_max);
}

__global__ void __launch_bounds__(1024)
k_means(int32_t nblocks, const unsigned long long *counts,
        const long long *sums, const unsigned int *maxabs_bits, float *mu,
        int32_t *err) {
  __shared__ unsigned long long s_c[1024];
  __shared__ long long s_s[1024];
  unsigned long long c = 0;
  long long s = 0;
  for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
    c += counts[b];
    s += sums[b];
  }
  s_c[threadIdx.x] = c;
  s_s[threadIdx.x] = s;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      s_c[threadIdx.x] += s_c[threadIdx.x + w];
      s_s[threadIdx.x] += s_s[threadIdx.x + w];
    }
    __syncthreads();
  }
  const unsigned long long total_c = s_c[0];
  const long long total_s = s_s[0];
  const double xmax = (double)__uint_as_float(*maxabs_bits);
  // |sum| <= count * max|x| * 2^32 must stay inside int64
  if ((double)total_c * xmax >= 2147483648.0) {
    if (threadIdx.x == 0) atomicOr(err, kErrSumRange);
  }
  float gmean = 0.0f;
  if (total_c)
    gmean = __double2float_rn(__ddiv_rn(__dmul_rn((double)total_s, 0x1p-32),
                                        (double)total_c));
  for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
    unsigned long long cb = counts[b];
    mu[b] = cb ? __double2float_rn(__ddiv_rn(
                     __dmul_rn((double)sums[b], 0x1p-32), (double)cb))
               : gmean;
  }
}

__global__ void __launch_bounds__(256)
k_plane_shift(int32_t nblocks, const unsigned long long *counts,
              const long long *sums, float *shift, float *delta) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nblocks;
       b += gridDim.x * blockDim.x) {
    const unsigned long long cb = counts[b];
    double mu = 0.0;
    if (cb) mu = __ddiv_rn(__dmul_rn((double)sums[b], 0x1p-32), (double)cb);
    const double c = rint(mu);
    shift[b] = (float)c;
    delta[b] = __double2float_rn(mu - c);
  }
}

// What a scatter needs of a block: where its cells are, what is subtracted,
// and for the planes the mask's offset from the offsets' plane and the largest
// exact |offset|.
struct __align__(16) Dest {
  int64_t off, mask;
  int32_t row0, col0, L_pad, flags;   // flags 1: W = B^T, 2: held here
  float sub, lim;
};
enum { kToFloat, kToBf16, kToPlanes };

struct DestTable {
  Dest dest[kTableBlocks];
  BoundsTable bounds;
};

template <int TO>
__device__ __forceinline__ Dest dest_of(const BlockMeta *meta,
                                        const float *sub, int32_t b) {
  const BlockMeta &bm = meta[b];
  Dest d;
  d.off = TO == kToFloat ? bm.w_off : bm.vx_off;
  d.mask = (int64_t)bm.s128 * bm.L_pad;
  d.row0 = (int32_t)bm.row0;
  d.col0 = (int32_t)bm.col0;
  d.L_pad = bm.L_pad;
  d.flags = (bm.trans ? 1 : 0) | (bm.owned ? 2 : 0);
  d.sub = sub[b];
  // exact in bf16, and every Gram partial sum below 2^24 in f32:
  // |y|^2 L_pad < 2^24
  d.lim = TO == kToPlanes ? fminf(sqrtf(16777216.f / (float)bm.L_pad), 256.f)
                          : 0.f;
  return d;
}

// out (zeroed): cell = x - sub, where sub is the block's mean (kToFloat,
// kToBf16) or its rounded mean (kToPlanes: the offset y in bf16, and 1 in the
// mask's plane). *flag (kToPlanes): kErrNotExact when some y is not a whole
// number of at most lim, kErrNotHalf when some is not a multiple of one half
// of at most lim / 2 (four times the sums, in quarters), kErrNotRebuilt when
// some x is not fl32(y + sub).
template <int TO, bool TABLE>
__global__ void __launch_bounds__(256)
k_scatter(GridDesc g, const BlockMeta *__restrict__ meta, int64_t nnz,
          const int32_t *__restrict__ u, const int32_t *__restrict__ it,
          const float *__restrict__ x, const float *__restrict__ sub,
          void *__restrict__ out, int32_t *flag) {
  extern __shared__ __align__(16) unsigned char smem[];
  DestTable &t = *reinterpret_cast<DestTable *>(smem);
  if (TABLE) {
    const int nb = g.diag ? g.p : g.p * g.q;
    for (int b = threadIdx.x; b < nb; b += blockDim.x)
      t.dest[b] = dest_of<TO>(meta, sub, b);
    t.bounds.fill(g);
    __syncthreads();
  }
  int32_t bad = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t0 < nnz;
       t0 += kRatings * stride) {
    int32_t uu[kRatings], ii[kRatings];
    float xx[kRatings];
#pragma unroll
    for (int k = 0; k < kRatings; ++k) {
      const int64_t e = t0 + k * stride;
      const bool in = e < nnz;
      uu[k] = in ? u[e] : -1;
      ii[k] = in ? it[e] : -1;
      xx[k] = in ? x[e] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < kRatings; ++k) {
      int32_t blk, ru, ci;
      // ids out of range were flagged when the ratings were counted
      if (!find_block<TABLE>(g, t.bounds, uu[k], ii[k], &blk, &ru, &ci))
        continue;
      const Dest d = TABLE ? t.dest[blk] : dest_of<TO>(meta, sub, blk);
      if (!(d.flags & 2)) continue;            // another shard's block
      const int32_t r = ru - d.row0, c = ci - d.col0;
      const int64_t cell =
          d.off + ((d.flags & 1) ? (int64_t)c * d.L_pad + r
                                 : (int64_t)r * d.L_pad + c);
      const float y = __fsub_rn(xx[k], d.sub);
      if (TO == kToFloat) {
        static_cast<float *>(out)[cell] = y;
      } else {
        __nv_bfloat16 *o = static_cast<__nv_bfloat16 *>(out);
        o[cell] = __float2bfloat16_rn(y);
        if (TO == kToPlanes) {
          o[cell + d.mask] = __float2bfloat16_rn(1.f);
          const float ay = fabsf(y);
          if (!(y == rintf(y) && ay <= d.lim)) bad |= kErrNotExact;
          if (!(2.f * y == rintf(2.f * y) && 2.f * ay <= d.lim))
            bad |= kErrNotHalf;
          if (!(__fadd_rn(y, d.sub) == xx[k])) bad |= kErrNotRebuilt;
        }
      }
    }
  }
  if (TO == kToPlanes) {
    const int32_t all = __reduce_or_sync(0xffffffffu, bad);
    if (all && (threadIdx.x & 31) == 0) atomicOr(flag, all);
  }
}

int grid_for(int64_t n, int per_thread) {
  int64_t want = (n + 256LL * per_thread - 1) / (256LL * per_thread);
  if (want < 1) want = 1;
  if (want > 152 * 8) want = 152 * 8;
  return (int)want;
}

}  // namespace

cudaError_t launch_plane_shift(int32_t nblocks, const unsigned long long *counts,
                               const long long *sums, float *shift,
                               float *delta, cudaStream_t st) {
  if (nblocks <= 0) return cudaSuccess;
  k_plane_shift<<<(nblocks + 255) / 256, 256, 0, st>>>(nblocks, counts, sums,
                                                       shift, delta);
  return cudaGetLastError();
}

cudaError_t launch_perm_check(const int32_t *perm, int64_t n, int32_t *seen,
                              int32_t *err, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(seen, 0, sizeof(int32_t) * n, st);
  if (e != cudaSuccess) return e;
  k_perm_mark<<<grid_for(n, 4), 256, 0, st>>>(perm, n, seen, err);
  k_perm_verify<<<grid_for(n, 4), 256, 0, st>>>(seen, n, err);
  return cudaGetLastError();
}

cudaError_t launch_count(const GridDesc &g, int64_t nnz, const int32_t *u,
                         const int32_t *i, const float *x, int32_t nblocks,
                         unsigned long long *counts, long long *sums,
                         unsigned int *maxabs_bits, int32_t *err,
                         cudaStream_t st) {
  if (nnz <= 0) return cudaSuccess;
  // big grids flush many per-CTA histograms: use fewer, longer CTAs
  int grid = grid_for(nnz, nblocks > 256 ? 16 : 4);
  const size_t sm = nblocks <= kSmemBlocks ? sizeof(CountTable) : 0;
  if (fits_table(g))
    k_count<true><<<grid, 256, sm, st>>>(g, nnz, u, i, x, nblocks, counts,
                                         sums, maxabs_bits, err);
  else
    k_count<false><<<grid, 256, sm, st>>>(g, nnz, u, i, x, nblocks, counts,
                                          sums, maxabs_bits, err);
  return cudaGetLastError();
}

cudaError_t launch_stack_ids(int64_t nnz, int32_t nb, const int64_t *starts,
                             const int64_t *add, int32_t *ids,
                             cudaStream_t st) {
  if (nnz <= 0) return cudaSuccess;
  k_stack_ids<<<grid_for(nnz, 4), 256, 0, st>>>(nnz, nb, starts, add, ids);
  return cudaGetLastError();
}

cudaError_t launch_means(int32_t nblocks, const unsigned long long *counts,
                         const long long *sums,
                         const unsigned int *maxabs_bits, float *mu,
                         int32_t *err, cudaStream_t st) {
  k_means<<<1, 1024, 0, st>>>(nblocks, counts, sums, maxabs_bits, mu, err);
  return cudaGetLastError();
}

template <int TO>
static cudaError_t scatter_to(const GridDesc &g, const BlockMeta *meta,
                              int64_t nnz, const int32_t *u, const int32_t *i,
                              const float *x, const float *sub, void *out,
                              int32_t *flag, cudaStream_t st) {
  if (nnz <= 0) return cudaSuccess;
  const int grid = grid_for(nnz, 4);
  if (fits_table(g))
    k_scatter<TO, true><<<grid, 256, sizeof(DestTable), st>>>(
        g, meta, nnz, u, i, x, sub, out, flag);
  else
    k_scatter<TO, false><<<grid, 256, 0, st>>>(g, meta, nnz, u, i, x, sub, out,
                                               flag);
  return cudaGetLastError();
}

cudaError_t launch_scatter(const GridDesc &g, const BlockMeta *meta,
                           int64_t nnz, const int32_t *u, const int32_t *i,
                           const float *x, const float *mu, float *W,
                           cudaStream_t st) {
  return scatter_to<kToFloat>(g, meta, nnz, u, i, x, mu, W, nullptr, st);
}

cudaError_t launch_scatter_bf16(const GridDesc &g, const BlockMeta *meta,
                                int64_t nnz, const int32_t *u,
                                const int32_t *i, const float *x,
                                const float *mu, __nv_bfloat16 *Wh,
                                cudaStream_t st) {
  return scatter_to<kToBf16>(g, meta, nnz, u, i, x, mu, Wh, nullptr, st);
}

cudaError_t launch_scatter_planes(const GridDesc &g, const BlockMeta *meta,
                                  int64_t nnz, const int32_t *u,
                                  const int32_t *i, const float *x,
                                  const float *shift, __nv_bfloat16 *VX,
                                  int32_t *flag, cudaStream_t st) {
  return scatter_to<kToPlanes>(g, meta, nnz, u, i, x, shift, VX, flag, st);
}

}  // namespace bsvd
