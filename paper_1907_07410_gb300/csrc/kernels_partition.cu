// Partition, block means and dense scatter (Section 3, Eq. "datax").
//
// Pass 1 (k_count) maps every training rating to its block and adds its
// count and its value to per-block totals. Values are summed as 64-bit
// fixed point with 32 fraction bits (x * 2^32), so the totals are exact
// integers and do not depend on the order of the atomic adds.
// Pass 2 (k_means) turns the totals into mu_b = fl32(fl64(sum) / count).
// Pass 3 writes fl32(x - mu_b), or its bf16 rounding, or the bf16 offset and
// the observation mask: k_scatter into zeroed dense blocks, or for large
// planes k_bucket and k_fill, which write every cell once.
//
// Every pass looks up a block per rating. A CTA keeps the grid's bounds and
// what it needs of each block in shared memory (BoundsTable, Dest); from
// global memory a rating's six or more lookups touch up to 32 lines per warp
// each. A thread takes kRatings ratings at a time, so that their loads
// overlap: counting 90 million ratings into 256 blocks took 0.90 ms with both
// (1.43 before). A random access of the L2 a rating (the position of an id, a
// counter, a list's place) takes about 75 us per ten million, which is what
// the counting and listing of a large matrix are bound by.
#include <type_traits>

#include "kernels.h"

namespace bsvd {

namespace {

constexpr int kSmemBlocks = 2048;   // per-CTA histogram size limit
constexpr int kManyBlocks = 8192;   // eight a thread of k_means
constexpr int kRatings = 4;            // ratings a thread has in flight
// planes from this size on are filled chunk by chunk (k_fill): smaller ones
// stay in the L2 from the memset to the scatter
constexpr int64_t kChunkedBytes = 256 << 20;

// A batch's ids to the stacked coordinates, in place: 16 bytes of traffic a
// rating; the piece is found by bisection (the tables stay in the L1). bounds:
// where each matrix begins. An id that its matrix does not have becomes -1,
// which the counting reports: moved along it could be a cell of the next
// matrix.
__global__ void k_stack_ids(int64_t nnz, int nb,
                            const int64_t *__restrict__ starts,
                            const int64_t *__restrict__ bounds,
                            int32_t *__restrict__ ids) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nnz;
       t += (int64_t)gridDim.x * blockDim.x) {
    int lo = 0, hi = nb;                 // starts[lo] <= t < starts[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (starts[mid] <= t) lo = mid;
      else hi = mid;
    }
    const int32_t id = ids[t];
    const int64_t first = bounds[lo];
    ids[t] = id >= 0 && id < bounds[lo + 1] - first ? (int32_t)(first + id) : -1;
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

// x * 2^32, rounded to the nearest integer, for |x| < 2^31. From 2^-9 on it is
// the mantissa shifted left, in integers: the product in float64 (below 2^-9)
// is three instructions of a pipe that takes 19 cycles an SM for each, which
// was most of k_count (10.8 million ratings: 113 -> 72 us). An integer form with a branch per exponent
// range had been slower still.
__device__ __forceinline__ long long fixed32(float x) {
  const uint32_t bits = __float_as_uint(x);
  const int sh = (int)(bits >> 23 & 0xff) - 118;    // 2^-9 has exponent 118
  if (sh >= 0) {
    const long long v = (long long)(bits & 0x7fffffu | 0x800000u) << (sh & 63);
    return (int32_t)bits < 0 ? -v : v;
  }
  if (x == 0.f) return 0;
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
};

// Where a cell of a block's bf16 plane is: its chunk and its place in it.
struct Place {
  int32_t row0, col0, L_pad, flags, ck0;   // flags as Dest
};
__device__ __forceinline__ Place place_of(const BlockMeta &bm) {
  return {(int32_t)bm.row0, (int32_t)bm.col0, bm.L_pad,
          (bm.trans ? 1 : 0) | (bm.owned ? 2 : 0), bm.ck0};
}
__device__ __forceinline__ int64_t plane_cell(const Place &p, int32_t ru,
                                              int32_t ci) {
  const int32_t r = ru - p.row0, c = ci - p.col0;
  return (p.flags & 1) ? (int64_t)c * p.L_pad + r : (int64_t)r * p.L_pad + c;
}

// Chunk ck's counter. Neighbouring chunks are busy together (the head of a
// long-tailed matrix is dense), and the L2 adds to one line at about one a
// nanosecond: consecutive chunks are spread over the table, a power of two
// long (mask + 1), which also is the order of the chunks' lists. With
// neighbours side by side the 10.8 million additions below took 600 us.
__device__ __forceinline__ int32_t chunk_slot(int32_t ck, uint32_t mask) {
  return (int32_t)((uint32_t)ck * 0x9E3779B1u & mask);     // odd: one to one
}

// A rating's place in the planes: its chunk's slot, and its block and cell in
// the chunk (16 bits each; at most kTableBlocks blocks). It is written by
// k_count and read by k_bucket, which saves looking up the ids' positions, a
// random access each, again.
constexpr uint32_t kNowhere = 0xffffffffu;

// One more entry in chunk ck for every lane with `on`; returns the lane's
// place among the chunk's entries. A whole warp: when its ratings are all in
// one chunk (a matrix sorted by rows), one lane adds for all.
__device__ __forceinline__ unsigned chunk_add(unsigned *cnt, bool on,
                                              int32_t ck) {
  const unsigned m = __ballot_sync(0xffffffffu, on);
  if (m == 0) return 0;
  const int lane = threadIdx.x & 31, first = __ffs(m) - 1;
  const int32_t c0 = __shfl_sync(0xffffffffu, ck, first);
  if (__all_sync(0xffffffffu, !on || ck == c0)) {
    unsigned base = 0;
    if (lane == first) base = atomicAdd(&cnt[c0], (unsigned)__popc(m));
    base = __shfl_sync(0xffffffffu, base, first);
    return base + __popc(m & ((1u << lane) - 1));
  }
  return on ? atomicAdd(&cnt[ck], 1u) : 0;
}

// CHUNKS: also the ratings per plane chunk (see k_fill); then TABLE.
template <bool TABLE, bool CHUNKS>
__global__ void __launch_bounds__(256)
k_count(GridDesc g, int64_t nnz, const int32_t *__restrict__ u,
        const int32_t *__restrict__ it, const float *__restrict__ x,
        int32_t nblocks, unsigned long long *counts, long long *sums,
        unsigned int *maxabs_bits, int32_t *err,
        const BlockMeta *__restrict__ meta, unsigned *chunks, uint32_t mask,
        uint2 *__restrict__ where) {
  extern __shared__ unsigned char smem[];
  // the counts when they fit, CHUNKS: the places (at most kTableBlocks blocks,
  // so the counts fit), then the bounds
  CountTable &t = *reinterpret_cast<CountTable *>(smem);
  Place *place = reinterpret_cast<Place *>(smem + sizeof(CountTable));
  if (CHUNKS) {
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x)
      place[b] = place_of(meta[b]);
  }
  __shared__ unsigned int s_max;
  const bool use_smem = nblocks <= kSmemBlocks;
  if (use_smem) {
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x)
      t.cnt[b] = t.lo[b] = t.hi[b] = 0;
  }
  BoundsTable bounds;
  if (TABLE)
    bounds.fill(g, CHUNKS ? sizeof(CountTable) + sizeof(Place) * kTableBlocks
                   : use_smem ? sizeof(CountTable) : 0);
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
      int32_t blk = -1, ru = 0, ci = 0;
      if (ok) {
        if (!find_block<TABLE>(g, bounds, uu[k], ii[k], &blk, &ru, &ci)) {
          local_err |= kErrIndex;
          ok = false;
        }
      }
      if (CHUNKS) {
        Place pl = {};
        if (ok) pl = place[blk];
        const bool held = ok && (pl.flags & 2);
        const int64_t cell = plane_cell(pl, ru, ci);
        const int32_t slot =
            chunk_slot(pl.ck0 + (int32_t)(cell >> kPlaneChunkLog), mask);
        chunk_add(chunks, held, slot);
        const int64_t e = t0 + k * stride + lane;
        if (e < nnz)
          where[e] = make_uint2(
              held ? (uint32_t)slot : kNowhere,
              (uint32_t)blk << 16 | (uint32_t)(cell & (kPlaneChunk - 1)));
      }
      if (ok && !rating_ok(xx[k])) {
        local_err |= kErrValue;
        ok = false;
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

__global__ void __launch_bounds__(256)
k_clear(int32_t nblocks, unsigned long long *counts, long long *sums,
        unsigned int *maxabs_bits) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < nblocks) {
    counts[b] = 0;
    sums[b] = 0;
  }
  if (b == 0) *maxabs_bits = 0;
}

// The block means, and for the planes (shift != null) the rounded mean and
// what it leaves. One CTA of as many warps as the blocks need; the totals by
// shuffles (ten barriers of 1,024 threads took longer than the rest: 7.5 us,
// now 3.3, the rounded means included).
__global__ void __launch_bounds__(1024)
k_means(int32_t nblocks, const unsigned long long *counts,
        const long long *sums, const unsigned int *maxabs_bits, float *mu,
        float *shift, float *delta, int32_t *err) {
  __shared__ unsigned long long s_c[32];
  __shared__ long long s_s[32];
  unsigned long long c = 0;
  long long s = 0;
  for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
    c += counts[b];
    s += sums[b];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    c += __shfl_xor_sync(0xffffffffu, c, o);
    s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  if ((threadIdx.x & 31) == 0) {
    s_c[threadIdx.x >> 5] = c;
    s_s[threadIdx.x >> 5] = s;
  }
  __syncthreads();
  unsigned long long total_c = 0;
  long long total_s = 0;
  for (int w = 0; w < (int)blockDim.x / 32; ++w) {
    total_c += s_c[w];
    total_s += s_s[w];
  }
  const double xmax = (double)__uint_as_float(*maxabs_bits);
  // |sum| <= count * max|x| * 2^32 must stay inside int64
  if ((double)total_c * xmax >= 2147483648.0) {
    if (threadIdx.x == 0) atomicOr(err, kErrSumRange);
  }
  // An empty block's mean is the mean of all ratings (0 without any). A float64
  // division is some twenty operations of 63 cycles: where a thread has many
  // blocks it is taken once (1,350,000 blocks, most of them empty: 4.8 ms with
  // one for each, 3.7 so; 2,400 blocks: 12.7 us with one for each, 15.2 so).
  auto mean_of = [](long long sum, unsigned long long count) {
    return count ? __ddiv_rn(__dmul_rn((double)sum, 0x1p-32), (double)count)
                 : 0.0;
  };
  const bool many = nblocks > kManyBlocks;
  const double every = many ? mean_of(total_s, total_c) : 0.0;
  for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
    const unsigned long long cb = counts[b];
    double m = every;
    if (cb || !many) m = mean_of(cb ? sums[b] : total_s, cb ? cb : total_c);
    mu[b] = __double2float_rn(m);
    if (shift) {
      if (!cb) m = 0.0;
      const double r = rint(m);
      shift[b] = (float)r;
      delta[b] = __double2float_rn(m - r);
    }
  }
}

// k_means' shift and delta where a thread of it would have many blocks (50,000
// blocks: 53 us there, 3.6 here).
__global__ void __launch_bounds__(256)
k_shifts(int32_t nblocks, const unsigned long long *__restrict__ counts,
         const long long *__restrict__ sums, float *__restrict__ shift,
         float *__restrict__ delta) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nblocks) return;
  const unsigned long long cb = counts[b];
  const double m = cb ? __ddiv_rn(__dmul_rn((double)sums[b], 0x1p-32), (double)cb)
                      : 0.0;
  const double r = rint(m);
  shift[b] = (float)r;
  delta[b] = __double2float_rn(m - r);
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

// What a CTA keeps in shared memory: nothing, the bounds, or a Dest per block
// and the bounds. A bisection through bounds in global memory is a chain of
// loads, which the warp's votes and the rounds of kRatings make longer (900,189
// ratings on a 30 x 30 quantile grid, counting / float32 scatter: 43 / 22 us
// with bounds in global memory, 22 / 20 with them here; 36 / 19 a rating at a
// time).
enum { kNoTable, kBoundsTable, kFullTable };

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

// Why y, the offset of x from sub, does not do in the planes.
__device__ __forceinline__ int32_t plane_flags(float y, float sub, float lim,
                                               float x) {
  const float ay = fabsf(y);
  int32_t bad = 0;
  if (!(y == rintf(y) && ay <= lim)) bad |= kErrNotExact;
  if (!(2.f * y == rintf(2.f * y) && 2.f * ay <= lim)) bad |= kErrNotHalf;
  if (!(__fadd_rn(y, sub) == x)) bad |= kErrNotRebuilt;
  return bad;
}

// out (zeroed): cell = x - sub, where sub is the block's mean (kToFloat,
// kToBf16) or its rounded mean (kToPlanes: the offset y in bf16, and 1 in the
// mask's plane). *flag (kToPlanes): kErrNotExact when some y is not a whole
// number of at most lim, kErrNotHalf when some is not a multiple of one half
// of at most lim / 2 (four times the sums, in quarters), kErrNotRebuilt when
// some x is not fl32(y + sub).
template <int TO, int TABLE>
__global__ void __launch_bounds__(256)
k_scatter(GridDesc g, const BlockMeta *__restrict__ meta, int64_t nnz,
          const int32_t *__restrict__ u, const int32_t *__restrict__ it,
          const float *__restrict__ x, const float *__restrict__ sub,
          void *__restrict__ out, int32_t *flag) {
  extern __shared__ __align__(16) unsigned char smem[];
  Dest *dest = reinterpret_cast<Dest *>(smem);
  BoundsTable bounds;
  if (TABLE != kNoTable) {
    if (TABLE == kFullTable) {
      const int nb = g.diag ? g.p : g.p * g.q;
      for (int b = threadIdx.x; b < nb; b += blockDim.x)
        dest[b] = dest_of<TO>(meta, sub, b);
    }
    bounds.fill(g, TABLE == kFullTable ? sizeof(Dest) * kTableBlocks : 0);
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
      if (!find_block<TABLE != kNoTable>(g, bounds, uu[k], ii[k], &blk, &ru,
                                         &ci))
        continue;
      const Dest d =
          TABLE == kFullTable ? dest[blk] : dest_of<TO>(meta, sub, blk);
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
          bad |= plane_flags(y, d.sub, d.lim, xx[k]);
        }
      }
    }
  }
  if (TO == kToPlanes) {
    const int32_t all = __reduce_or_sync(0xffffffffu, bad);
    if (all && (threadIdx.x & 31) == 0) atomicOr(flag, all);
  }
}

// The planes of a large matrix, chunk by chunk. Ratings scattered into zeroed
// planes cost a 32-byte DRAM sector each, written part by part at 25 to 30
// billion a second whatever the order of issue: 10.8 million ratings in
// 3.8 GB of planes took 635 us after a memset of 590. Instead the ratings are
// counted by chunk of 2^13 cells (in k_count), put into their chunk's list
// (k_bucket, 4 bytes each: 13 bits of place, the bf16 offset), and a CTA lays
// out one chunk at a time in shared memory and stores it as it is (k_fill),
// zeros included: 158 + 673 us and 52 more in k_count; 17 GB of one plane and
// 90 million ratings 1.56 + 3.10 ms, from 2.7 + 3.8; 0.35 GB and 6.2 million in
// a batch 118 + 71 us, from 348 + 60. Chunks of 2^12 or 2^14
// cells are within 5 % on the large ones; 2^14 costs the batch 60 us (fewer
// counters, more waiting at each).
//
// Exclusive scan of the chunks' counts in two levels: within kScanTile
// counts here, the tiles' totals in k_chunk_tops.
constexpr int kScanTile = 4096;

__device__ __forceinline__ unsigned scan_1024(unsigned v, unsigned *warp_sum,
                                              unsigned *total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  unsigned inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned up = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += up;
  }
  if (lane == 31) warp_sum[w] = inc;
  __syncthreads();
  if (w == 0) {
    const unsigned ws = warp_sum[lane];
    unsigned wi = ws;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned up = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += up;
    }
    warp_sum[lane] = wi - ws;
    if (lane == 31) *total = wi;
  }
  __syncthreads();
  return warp_sum[w] + inc - v;
}

__global__ void __launch_bounds__(1024)
k_chunk_scan(int32_t nslots, unsigned *cnt, unsigned *tops) {
  __shared__ unsigned ws[32], total;
  const int64_t e0 = (int64_t)blockIdx.x * kScanTile + 4 * threadIdx.x;
  unsigned v[4], sum = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = e0 + k < nslots ? cnt[e0 + k] : 0;
    sum += v[k];
  }
  unsigned at = scan_1024(sum, ws, &total);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (e0 + k < nslots) cnt[e0 + k] = at;
    at += v[k];
  }
  if (threadIdx.x == 0) tops[blockIdx.x] = total;
}

__global__ void __launch_bounds__(1024)
k_chunk_tops(int32_t ntiles, unsigned *tops) {
  __shared__ unsigned ws[32], total;
  unsigned carry = 0;
  for (int t0 = 0; t0 < ntiles; t0 += 1024) {
    const int t = t0 + threadIdx.x;
    const unsigned v = t < ntiles ? tops[t] : 0;
    const unsigned at = scan_1024(v, ws, &total);
    if (t < ntiles) tops[t] = carry + at;
    carry += total;
    __syncthreads();                     // ws and total are written again
  }
}

// Every rating into its chunk's list. cursor: the chunks' starts (within
// their scan tile), moved to their ends.
template <int TO>
__global__ void __launch_bounds__(256)
k_bucket(int nb, const BlockMeta *__restrict__ meta, int64_t nnz,
         const uint2 *__restrict__ where, const float *__restrict__ x,
         const float *__restrict__ sub, const unsigned *__restrict__ tops,
         unsigned *cursor, uint32_t *__restrict__ list, int32_t *flag) {
  __shared__ float2 sub_lim[kTableBlocks];
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    const Dest d = dest_of<TO>(meta, sub, b);
    sub_lim[b] = make_float2(d.sub, d.lim);
  }
  __syncthreads();
  int32_t bad = 0;
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t t0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31);
       t0 < nnz; t0 += kRatings * stride) {
    uint2 wh[kRatings];
    float xx[kRatings];
#pragma unroll
    for (int k = 0; k < kRatings; ++k) {
      const int64_t e = t0 + k * stride + lane;
      wh[k] = e < nnz ? where[e] : make_uint2(kNowhere, 0);
      xx[k] = e < nnz ? x[e] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < kRatings; ++k) {
      const bool on = wh[k].x != kNowhere;
      const int32_t slot = (int32_t)wh[k].x;
      const unsigned at = chunk_add(cursor, on, slot);
      if (!on) continue;
      const float2 sl = sub_lim[wh[k].y >> 16];
      const float y = __fsub_rn(xx[k], sl.x);
      const uint32_t entry =
          (wh[k].y & 0xffffu) |
          (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(y)) << 16;
      const int64_t pos = (int64_t)tops[slot / kScanTile] + at;
      if (pos < nnz) list[pos] = entry;
      if (TO == kToPlanes) bad |= plane_flags(y, sl.x, sl.y, xx[k]);
    }
  }
  if (TO == kToPlanes) {
    const int32_t all = __reduce_or_sync(0xffffffffu, bad);
    if (all && lane == 0) atomicOr(flag, all);
  }
}

// out: every cell of the planes (PLANES = 2: the offsets, then the mask).
// The chunk in shared memory is zero between chunks: the cells that were set
// are set back. Six CTAs an SM with two planes, eleven with one (as many chunks
// fit its shared memory), so that the others work while one's store drains.
constexpr int kFillThreads = kPlaneChunk / 64;
constexpr int kHold = 4;
template <int PLANES>
__global__ void __launch_bounds__(kFillThreads)
k_fill(const BlockMeta *__restrict__ meta, int32_t nb, int32_t nchunks,
       const unsigned *__restrict__ tops, const unsigned *__restrict__ ends,
       uint32_t mask,
       const uint32_t *__restrict__ list, __nv_bfloat16 *__restrict__ out) {
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned short *y = reinterpret_cast<unsigned short *>(smem);
  unsigned short *mk = y + kPlaneChunk;
  __shared__ int32_t ck0[kTableBlocks];
  for (int b = threadIdx.x; b < nb; b += blockDim.x) ck0[b] = meta[b].ck0;
  for (int e = threadIdx.x; e < PLANES * kPlaneChunk / 8; e += blockDim.x)
    reinterpret_cast<uint4 *>(smem)[e] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  auto edge = [&](int32_t slot) -> int64_t {    // where the list there ends
    return (int64_t)tops[slot / kScanTile] + ends[slot];
  };
  struct Job {
    int64_t from, to;
    uint32_t v[kHold];                 // the first entries of this thread
    __nv_bfloat16 *dst;                // thread 0: where the chunk goes
    int64_t plane;
    uint32_t bytes;
  };
  auto fetch = [&](int32_t ck) {
    Job j;
    j.from = j.to = 0;
    if (ck >= nchunks) return j;
    const int32_t slot = chunk_slot(ck, mask);
    j.from = slot % kScanTile ? edge(slot - 1) : tops[slot / kScanTile];
    j.to = edge(slot);
    if (threadIdx.x == 0) {
      const BlockMeta &bm = meta[upper_index(ck0, nb, ck)];
      const int64_t c0 = (int64_t)(ck - bm.ck0) << kPlaneChunkLog;
      j.plane = (int64_t)bm.s128 * bm.L_pad;
      j.dst = out + bm.vx_off + c0;
      // a plane is a multiple of 128 x 32 cells: whole 16-byte units
      j.bytes = 2 * (uint32_t)min(j.plane - c0, (int64_t)kPlaneChunk);
    }
#pragma unroll
    for (int h = 0; h < kHold; ++h) {
      const int64_t e = j.from + h * kFillThreads + threadIdx.x;
      if (e < j.to) j.v[h] = list[e];
    }
    return j;
  };
  auto put = [&](const Job &j, bool set) {
    auto one = [&](uint32_t v) {
      y[v & 0xffff] = set ? (unsigned short)(v >> 16) : 0;
      if (PLANES == 2) mk[v & 0xffff] = set ? 0x3f80 : 0;        // 1
    };
#pragma unroll
    for (int h = 0; h < kHold; ++h)
      if (j.from + h * kFillThreads + threadIdx.x < j.to) one(j.v[h]);
    for (int64_t e = j.from + kHold * kFillThreads + threadIdx.x; e < j.to;
         e += kFillThreads)
      one(list[e]);
  };
  Job job = fetch(blockIdx.x);
  for (int32_t ck = blockIdx.x; ck < nchunks; ck += gridDim.x) {
    put(job, true);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
      for (int p = 0; p < PLANES; ++p)
        asm volatile(
            "cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(
                job.dst + p * job.plane),
            "r"((uint32_t)__cvta_generic_to_shared(y + p * kPlaneChunk)),
            "r"(job.bytes)
            : "memory");
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    }
    const Job next = fetch(ck + gridDim.x);
    if (threadIdx.x == 0)
      asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    __syncthreads();
    put(job, false);
    job = next;
    __syncthreads();
  }
  if (threadIdx.x == 0)
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// One block's cells, row-major, from its planes, as the scatter to the float32
// arena would have written them.
__global__ void __launch_bounds__(256)
k_rebuild_block(BlockMeta bm, int32_t b, const __nv_bfloat16 *__restrict__ VX,
                const float *__restrict__ shift, const float *__restrict__ mu,
                float *__restrict__ out) {
  const float sh = shift[b], mean = mu[b];
  const __nv_bfloat16 *y = VX + bm.vx_off;
  const __nv_bfloat16 *mask = y + (int64_t)bm.s128 * bm.L_pad;
  const int64_t n = (int64_t)bm.mb * bm.nb;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / bm.nb, c = e - r * bm.nb;
    const int64_t cell = bm.trans ? c * bm.L_pad + r : r * bm.L_pad + c;
    const float x = __fadd_rn(__bfloat162float(y[cell]), sh);
    out[e] = __bfloat162float(mask[cell]) != 0.f ? __fsub_rn(x, mean) : 0.f;
  }
}

// How much of an SM's 256 KB is shared memory for a kernel, in percent of 228
// KB; the rest is the L1, which holds what the ratings look up (positions of
// ids, metadata). Left to itself the runtime makes room for all CTAs that fit.
// Ten / 90 million ratings on a quantile grid counted with their chunks at 45,
// 58, 72, 100 %: 152, 146, 168, 209 us / 1.31, 1.16, 1.21, 1.78 ms; the float32
// scatter with a full table at 45, 58, 100 %: 331, 355, 356 us. The planes'
// (matrices of a million ratings) 21.1, 20.4, 20.8 us. Without a full table
// there is little to make room for, and the metadata wants the L1 (900 blocks,
// five million ratings: 133 us, 253 at 45 %).
constexpr int kCountCarveout = 58, kScatterCarveout = 45, kPlanesCarveout = 58;
template <typename K>
cudaError_t carve_out(K *kernel, int percent) {
  return cudaFuncSetAttribute(
      kernel, cudaFuncAttributePreferredSharedMemoryCarveout, percent);
}

int grid_for(int64_t n, int per_thread) {
  int64_t want = (n + 256LL * per_thread - 1) / (256LL * per_thread);
  if (want < 1) want = 1;
  if (want > 152 * 8) want = 152 * 8;
  return (int)want;
}

}  // namespace

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
                         cudaStream_t st, const BlockMeta *meta,
                         unsigned *chunks, int64_t nchunks, uint2 *where) {
  if (nnz <= 0) return cudaSuccess;
  const uint32_t mask = (uint32_t)(chunk_slots(nchunks) - 1);
  // big grids flush many per-CTA histograms: use fewer, longer CTAs
  const bool hist = nblocks <= kSmemBlocks;
  const int grid = grid_for(nnz, hist && nblocks > 256 ? 16 : 4);
  const size_t sm = hist ? sizeof(CountTable) : 0, bounds = bounds_bytes(g);
  auto kernel = chunks           ? k_count<true, true>
                : fits_bounds(g) ? k_count<true, false>
                                 : k_count<false, false>;
  const size_t bytes = sm + (chunks ? sizeof(Place) * kTableBlocks : 0) +
                       (chunks || fits_bounds(g) ? bounds : 0);
  const cudaError_t e = carve_out(kernel, kCountCarveout);
  if (e != cudaSuccess) return e;
  kernel<<<grid, 256, bytes, st>>>(g, nnz, u, i, x, nblocks, counts, sums,
                                   maxabs_bits, err, meta, chunks, mask, where);
  return cudaGetLastError();
}

cudaError_t launch_stack_ids(int64_t nnz, int32_t nb, const int64_t *starts,
                             const int64_t *bounds, int32_t *ids,
                             cudaStream_t st) {
  if (nnz <= 0) return cudaSuccess;
  k_stack_ids<<<grid_for(nnz, 4), 256, 0, st>>>(nnz, nb, starts, bounds, ids);
  return cudaGetLastError();
}

cudaError_t launch_clear(int32_t nblocks, unsigned long long *counts,
                         long long *sums, unsigned int *maxabs_bits,
                         cudaStream_t st) {
  k_clear<<<nblocks / 256 + 1, 256, 0, st>>>(nblocks, counts, sums,
                                             maxabs_bits);
  return cudaGetLastError();
}

cudaError_t launch_means(int32_t nblocks, const unsigned long long *counts,
                         const long long *sums,
                         const unsigned int *maxabs_bits, float *mu,
                         float *shift, float *delta, int32_t *err,
                         cudaStream_t st, int64_t *launches) {
  int threads = (nblocks + 31) / 32 * 32;
  threads = threads < 32 ? 32 : threads > 1024 ? 1024 : threads;
  const bool apart = shift && nblocks > kManyBlocks;
  k_means<<<1, threads, 0, st>>>(nblocks, counts, sums, maxabs_bits, mu,
                                 apart ? nullptr : shift, delta, err);
  if (apart)
    k_shifts<<<(nblocks + 255) / 256, 256, 0, st>>>(nblocks, counts, sums, shift,
                                                    delta);
  if (launches) *launches += apart ? 2 : 1;
  return cudaGetLastError();
}

template <int TO>
static cudaError_t scatter_to(const GridDesc &g, const BlockMeta *meta,
                              int64_t nnz, const int32_t *u, const int32_t *i,
                              const float *x, const float *sub, void *out,
                              int32_t *flag, cudaStream_t st) {
  if (nnz <= 0) return cudaSuccess;
  const int grid = grid_for(nnz, 4);
  auto kernel = fits_table(g)    ? k_scatter<TO, kFullTable>
                : fits_bounds(g) ? k_scatter<TO, kBoundsTable>
                                 : k_scatter<TO, kNoTable>;
  const size_t bytes = (fits_table(g) ? sizeof(Dest) * kTableBlocks : 0) +
                       (fits_bounds(g) ? bounds_bytes(g) : 0);
  if (fits_table(g)) {
    const cudaError_t e = carve_out(
        kernel, TO == kToPlanes ? kPlanesCarveout : kScatterCarveout);
    if (e != cudaSuccess) return e;
  }
  kernel<<<grid, 256, bytes, st>>>(g, meta, nnz, u, i, x, sub, out, flag);
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

cudaError_t launch_rebuild_block(const BlockMeta &bm, int32_t b,
                                 const __nv_bfloat16 *VX, const float *shift,
                                 const float *mu, float *out,
                                 cudaStream_t st) {
  const int64_t n = (int64_t)bm.mb * bm.nb;
  if (n <= 0) return cudaSuccess;
  k_rebuild_block<<<grid_for(n, 4), 256, 0, st>>>(bm, b, VX, shift, mu, out);
  return cudaGetLastError();
}

bool chunked_planes(const GridDesc &g, int64_t nnz, int64_t nchunks,
                    int64_t plane_bytes, int64_t list_cap) {
  return fits_table(g) && nnz > 0 && nnz <= list_cap && nnz < INT32_MAX &&
         nchunks > 0 && nchunks <= (1 << 30) && plane_bytes >= kChunkedBytes;
}

int64_t chunk_slots(int64_t nchunks) {
  int64_t n = 1;
  while (n < nchunks) n *= 2;
  return n;
}

int64_t chunk_words(int64_t nchunks) {
  const int64_t n = chunk_slots(nchunks);
  return n + (n + kScanTile - 1) / kScanTile;
}

template <int TO>
static cudaError_t planes_to(const GridDesc &g, const BlockMeta *meta,
                             int64_t nnz, const uint2 *where, const float *x,
                             const float *sub, int32_t nchunks,
                             unsigned *chunks, uint32_t *list,
                             __nv_bfloat16 *out, int32_t *flag,
                             cudaStream_t st) {
  constexpr int PLANES = TO == kToPlanes ? 2 : 1;
  constexpr int kBytes = PLANES * kPlaneChunk * 2;
  const int32_t nslots = (int32_t)chunk_slots(nchunks);
  const uint32_t mask = (uint32_t)nslots - 1;
  const int ntiles = (nslots + kScanTile - 1) / kScanTile;
  unsigned *tops = chunks + nslots;
  k_chunk_scan<<<ntiles, 1024, 0, st>>>(nslots, chunks, tops);
  k_chunk_tops<<<1, 1024, 0, st>>>(ntiles, tops);
  k_bucket<TO><<<grid_for(nnz, 4), 256, 0, st>>>(
      grid_blocks(g), meta, nnz, where, x, sub, tops, chunks, list, flag);
  cudaError_t e = cudaFuncSetAttribute(
      k_fill<PLANES>, cudaFuncAttributeMaxDynamicSharedMemorySize, kBytes);
  if (e != cudaSuccess) return e;
  const int per_sm = (215 << 10) / (kBytes + 2048 + 1024);
  k_fill<PLANES><<<nchunks < 152 * per_sm ? nchunks : 152 * per_sm, kFillThreads,
                   kBytes, st>>>(meta, grid_blocks(g), nchunks, tops, chunks,
                                 mask, list, out);
  return cudaGetLastError();
}

cudaError_t launch_chunked_bf16(const GridDesc &g, const BlockMeta *meta,
                                int64_t nnz, const uint2 *where, const float *x,
                                const float *mu, int32_t nchunks,
                                unsigned *chunks, uint32_t *list,
                                __nv_bfloat16 *Wh, cudaStream_t st) {
  return planes_to<kToBf16>(g, meta, nnz, where, x, mu, nchunks, chunks, list,
                       Wh, nullptr, st);
}

cudaError_t launch_chunked_planes(const GridDesc &g, const BlockMeta *meta,
                                  int64_t nnz, const uint2 *where, const float *x,
                                  const float *shift, int32_t nchunks,
                                  unsigned *chunks, uint32_t *list,
                                  __nv_bfloat16 *VX, int32_t *flag,
                                  cudaStream_t st) {
  return planes_to<kToPlanes>(g, meta, nnz, where, x, shift, nchunks, chunks, list,
                       VX, flag, st);
}

}  // namespace bsvd
