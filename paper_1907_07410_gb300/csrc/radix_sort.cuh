// Stable radix sort of 64-bit keys, least significant digit first, 8 bits a
// pass. A pass is three launches: digit counts per tile of 4,096 keys, one CTA
// per digit that scans its tiles' counts, and the scatter, whose eight warps
// each rank 512 consecutive keys with a match over equal digits per 32. Up to
// kRsFewTiles tiles every CTA of the scatter adds up the counts itself, and the
// scan is left out. The launches overlap (pdl_wait), as the chains that call the
// sort do: laying out 1,000 / 20,000 / 900,189 ratings for the blocked SGD, 4
// to 8 passes among 22 to 34 launches, took 139 / 247 / 348 us and takes 82 /
// 161 / 286.
#pragma once
#include "common.cuh"

namespace bsvd {

namespace {

typedef unsigned long long u64;

constexpr int kRsThreads = 256;
constexpr int kRsItems = 16;                   // keys per thread
constexpr int kRsTile = kRsThreads * kRsItems; // keys per CTA
constexpr int kRsWarps = kRsThreads / 32;
constexpr int kRsFewTiles = 16;

template <typename V>
__global__ void __launch_bounds__(kRsThreads)
k_rs_count(const u64 *__restrict__ key, int64_t n, int shift, unsigned mask,
           int64_t ntiles, V *__restrict__ hist) {
  __shared__ unsigned cnt[256];
  cnt[threadIdx.x] = 0;
  pdl_wait();
  pdl_trigger();
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * kRsTile;
#pragma unroll
  for (int j = 0; j < kRsItems; ++j) {
    const int64_t e = base + j * kRsThreads + threadIdx.x;
    if (e < n) atomicAdd(&cnt[(unsigned)(key[e] >> shift) & mask], 1u);
  }
  __syncthreads();
  hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = cnt[threadIdx.x];
}

// CTA d: exclusive scan of digit d's tile counts, and their total.
template <typename V>
__global__ void __launch_bounds__(kRsThreads)
k_rs_scan(V *__restrict__ hist, int64_t ntiles, V *__restrict__ total) {
  __shared__ V part[kRsThreads];
  V *h = hist + (int64_t)blockIdx.x * ntiles;
  V run = 0;
  pdl_wait();
  pdl_trigger();
  for (int64_t b = 0; b < ntiles; b += kRsThreads) {
    const int64_t e = b + threadIdx.x;
    const V v = e < ntiles ? h[e] : 0;
    part[threadIdx.x] = v;
    __syncthreads();
    for (int w = 1; w < kRsThreads; w <<= 1) {
      const V o = threadIdx.x >= w ? part[threadIdx.x - w] : 0;
      __syncthreads();
      part[threadIdx.x] += o;
      __syncthreads();
    }
    if (e < ntiles) h[e] = run + part[threadIdx.x] - v;
    run += part[kRsThreads - 1];
    __syncthreads();
  }
  if (threadIdx.x == 0) total[blockIdx.x] = run;
}

// Stable scatter of one tile. vin == nullptr: the values are the positions;
// vout == nullptr: keys alone. FEW: hist holds the tiles' counts as they are,
// not their scan, and total nothing.
template <typename V, bool FEW>
__global__ void __launch_bounds__(kRsThreads)
k_rs_scatter(const u64 *__restrict__ kin, const V *__restrict__ vin, int64_t n,
             int shift, unsigned mask, int64_t ntiles,
             const V *__restrict__ hist, const V *__restrict__ total,
             u64 *__restrict__ kout, V *__restrict__ vout) {
  __shared__ unsigned wc[kRsWarps][256];
  __shared__ V base[256];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
#pragma unroll
  for (int w = 0; w < kRsWarps; ++w) wc[w][tid] = 0;
  pdl_wait();
  pdl_trigger();
  // this digit's keys in the tiles before this one, and in all
  V before = 0, all = 0;
  if (FEW) {
    for (int64_t b = 0; b < ntiles; ++b) {
      const V c = hist[(int64_t)tid * ntiles + b];
      before += b < blockIdx.x ? c : 0;
      all += c;
    }
  } else {
    before = hist[(int64_t)tid * ntiles + blockIdx.x];
    all = total[tid];
  }
  // global start of every digit: a scan over the 256 totals
  base[tid] = all;
  __syncthreads();
  for (int w = 1; w < 256; w <<= 1) {
    const V o = tid >= w ? base[tid - w] : 0;
    __syncthreads();
    base[tid] += o;
    __syncthreads();
  }
  const V digit0 = base[tid] - all;
  const int64_t w0 =
      (int64_t)blockIdx.x * kRsTile + warp * (32 * kRsItems) + lane;
  u64 k[kRsItems];
  unsigned rank[kRsItems];
#pragma unroll
  for (int j = 0; j < kRsItems; ++j) {
    const int64_t e = w0 + 32 * j;
    k[j] = e < n ? kin[e] : 0;
  }
#pragma unroll
  for (int j = 0; j < kRsItems; ++j) {
    const bool has = w0 + 32 * j < n;
    const unsigned d = (unsigned)(k[j] >> shift) & mask;
    const unsigned same = __match_any_sync(0xffffffffu, has ? d : 256u);
    const unsigned ahead = __popc(same & ((1u << lane) - 1u));
    const unsigned seen = has ? wc[warp][d] : 0u;
    __syncwarp();
    if (has && ahead == 0) wc[warp][d] = seen + __popc(same);
    __syncwarp();
    rank[j] = seen + ahead;
  }
  __syncthreads();
  {
    unsigned run = 0;
#pragma unroll
    for (int w = 0; w < kRsWarps; ++w) {
      const unsigned c = wc[w][tid];
      wc[w][tid] = run;
      run += c;
    }
    base[tid] = digit0 + before;
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kRsItems; ++j) {
    const int64_t e = w0 + 32 * j;
    if (e >= n) continue;
    const unsigned d = (unsigned)(k[j] >> shift) & mask;
    const V pos = base[d] + wc[warp][d] + rank[j];
    kout[pos] = k[j];
    if (vout) vout[pos] = vin ? vin[e] : (V)e;
  }
}

// Stable sort by the key's bits from `low` on, `bits` of them, from the buffers
// `cur` of the pairs (key[], val[]) into whichever holds the result (returned
// in *cur). identity: the values start as the positions; val[] null: keys
// alone. hist: 256 words per tile of 4,096 keys, total: 256.
template <typename V>
cudaError_t radix_sort(u64 *const key[2], V *const val[2], int *cur,
                       bool identity, int64_t n, int bits, V *hist, V *total,
                       int64_t *launches, cudaStream_t st, int low = 0) {
  const int64_t ntiles = (n + kRsTile - 1) / kRsTile;
  if (bits < 1) bits = 1;         // one pass still writes the values
  for (int shift = 0; shift < bits; shift += 8) {
    const int w = bits - shift < 8 ? bits - shift : 8;
    const unsigned mask = (1u << w) - 1u;
    const int c = *cur;
    const dim3 grid((unsigned)ntiles), block(kRsThreads);
    const bool few = ntiles <= kRsFewTiles;
    cudaError_t e = launch_pdl(k_rs_count<V>, grid, block, 0, st,
                               (const u64 *)key[c], n, low + shift, mask,
                               ntiles, hist);
    if (e == cudaSuccess && !few)
      e = launch_pdl(k_rs_scan<V>, dim3(256), block, 0, st, hist, ntiles, total);
    if (e == cudaSuccess)
      e = launch_pdl(few ? k_rs_scatter<V, true> : k_rs_scatter<V, false>, grid,
                     block, 0, st, (const u64 *)key[c],
                     (const V *)(identity && shift == 0 ? nullptr : val[c]), n,
                     low + shift, mask, ntiles, (const V *)hist,
                     (const V *)total, key[c ^ 1], val[c ^ 1]);
    if (e != cudaSuccess) return e;
    *cur = c ^ 1;
    *launches += few ? 2 : 3;
  }
  return cudaGetLastError();
}

}  // namespace

}  // namespace bsvd
