// Held-out prediction and scoring.
//
// A rating is predicted from its block's factors (Section 2.1, Eq. 2, with
// the singular values merged into one side): yhat = mu_b + P[r,:] . V[c,:].
// In W orientation that is mu_b + F_s[a,:] . F_L[l,:]. The score is the RMSE
// of Section 5 (Table 1, "Test RMSE").
//
// The squared errors are summed in float64 with a fixed grid, a fixed
// per-thread stride and a fixed reduction tree. The sum therefore does not
// depend on scheduling, and reruns are bit-identical.
#include <type_traits>

#include "kernels.h"

namespace bsvd {

namespace {

constexpr int kPredictThreads = 256;
constexpr int64_t kFewQueries = 40000;   // about eight lanes each in one wave
constexpr int kSqerrThreads = 512;   // 304 CTAs of them fill the SMs

// Where a query's block keeps what a prediction reads. A CTA copies the
// grid's bounds and a Place per block into shared memory once (see
// BoundsTable): six lookups per query in global memory, each touching up to 32
// lines per warp, cost about as much as its factor rows.
struct __align__(16) Place {
  int64_t fs, fl;            // first row of F_s and F_L, in floats
  int32_t row0, col0;        // first position
  float mu;
  int32_t flags;             // 1: has factors, 2: W = B^T, 4: held here
};

struct Table {
  Place *place = nullptr;        // kTableBlocks of them, then the bounds
  BoundsTable bounds;
};
inline size_t table_bytes(const GridDesc &g) {
  return sizeof(Place) * kTableBlocks + bounds_bytes(g);
}

__device__ __forceinline__ Place place_of(const PredictArgs &a, int32_t blk) {
  const BlockMeta &bm = a.meta[blk];
  Place p;
  p.fs = bm.fs_off;
  p.fl = bm.fl_off;
  p.row0 = (int32_t)bm.row0;
  p.col0 = (int32_t)bm.col0;
  p.mu = a.mu[blk];
  p.flags = (bm.keff > 0 ? 1 : 0) | (bm.trans ? 2 : 0) | (bm.owned ? 4 : 0);
  return p;
}

// Every thread of the CTA; ends with a barrier.
__device__ __forceinline__ void fill_table(const PredictArgs &a, Table &t,
                                           void *smem) {
  t.place = static_cast<Place *>(smem);
  const int nb = a.g.diag ? a.g.p : a.g.p * a.g.q;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) t.place[b] = place_of(a, b);
  t.bounds.fill(a.g, t.place + kTableBlocks);
  __syncthreads();
}

// The two factor rows of a query (null: the prediction is the mean alone).
struct Rows {
  const float4 *fs, *fl;
};

// One query per lane (skip: none); every lane of the warp calls. Where the
// query is valid, *out is its prediction and the result true; *held says
// whether this context holds its block.
//
// A row of kp floats is read by LPQ neighbouring lanes, 16 bytes each, so a
// warp's load touches 32 / LPQ rows. With a lane per query every load touched
// 32 rows, and the lines a load can look up per cycle bound the kernel: ten
// million queries at kp = 40 took 0.58 ms, and take 0.38 ms with both changes,
// 78% of the L1's rate. The lanes' sums of a row are added in a fixed tree.
// The rows of UN steps are loaded together (kp = 56, ten million queries, UN =
// 2 / 4 at eight lanes: 0.65 / 0.55 ms, but 0.64 / 0.91 with the squared
// errors, which run at half the warps).
template <int LPQ, int UN, bool TABLE>
__device__ __forceinline__ bool predict_warp(const PredictArgs &a,
                                             const Table &tb, bool skip,
                                             int32_t u, int32_t i, Rows *wq,
                                             float *wdot, float *out,
                                             bool *held) {
  constexpr int QPI = 32 / LPQ;              // queries per step
  const int lane = threadIdx.x & 31;
  bool ok = false;
  float mu = 0.f;
  Rows mine = {nullptr, nullptr};
  *held = true;
  if (!skip) {
    int32_t blk, ru, ci;
    ok = find_block<TABLE>(a.g, tb.bounds, u, i, &blk, &ru, &ci);
    if (ok) {
      const Place p = TABLE ? tb.place[blk] : place_of(a, blk);
      mu = p.mu;
      *held = (p.flags & 4) != 0;
      if ((p.flags & 1) && (*held || !a.owned_only)) {
        const int32_t r = ru - p.row0, c = ci - p.col0;
        const bool trans = (p.flags & 2) != 0;
        mine.fs = reinterpret_cast<const float4 *>(
            a.Fs + p.fs + (int64_t)(trans ? c : r) * a.kp);
        mine.fl = reinterpret_cast<const float4 *>(
            a.FL + p.fl + (int64_t)(trans ? r : c) * a.kp);
      }
    }
  }
  wq[lane] = mine;
  __syncwarp();
  const int n4 = a.kp / 4, sub = lane % LPQ;
#pragma unroll 1
  for (int s = 0; s < 32; s += QPI * UN) {
    Rows q[UN];
    float dot[UN];
#pragma unroll
    for (int x = 0; x < UN; ++x) {
      q[x] = wq[s + x * QPI + lane / LPQ];
      dot[x] = 0.f;
    }
    for (int j = sub; j < n4; j += LPQ) {
      float4 p[UN], v[UN];
#pragma unroll
      for (int x = 0; x < UN; ++x) {
        p[x] = v[x] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (q[x].fs) {
          p[x] = __ldg(q[x].fs + j);
          v[x] = __ldg(q[x].fl + j);
        }
      }
#pragma unroll
      for (int x = 0; x < UN; ++x) {
        dot[x] = fmaf(p[x].x, v[x].x, dot[x]);
        dot[x] = fmaf(p[x].y, v[x].y, dot[x]);
        dot[x] = fmaf(p[x].z, v[x].z, dot[x]);
        dot[x] = fmaf(p[x].w, v[x].w, dot[x]);
      }
    }
#pragma unroll
    for (int x = 0; x < UN; ++x) {
#pragma unroll
      for (int o = LPQ / 2; o > 0; o >>= 1)
        dot[x] += __shfl_xor_sync(0xffffffffu, dot[x], o);
      if (sub == 0) wdot[s + x * QPI + lane / LPQ] = dot[x];
    }
  }
  __syncwarp();
  float y = mu + wdot[lane];
  __syncwarp();                    // wq and wdot are the next call's
  if (a.clamp) y = fminf(fmaxf(y, a.lo), a.hi);
  *out = y;
  return ok;
}

template <int LPQ, bool TABLE>
__global__ void __launch_bounds__(kPredictThreads)
k_predict(PredictArgs a, int64_t nq, const int32_t *__restrict__ u,
          const int32_t *__restrict__ it, float *__restrict__ yhat,
          int32_t *err) {
  __shared__ Rows wq[kPredictThreads];
  __shared__ float wdot[kPredictThreads];
  extern __shared__ __align__(16) unsigned char table[];
  Table tb;
  if (TABLE) fill_table(a, tb, table);
  const int w0 = threadIdx.x & ~31, lane = threadIdx.x & 31;
  int32_t bad = 0;
  for (int64_t t0 = blockIdx.x * (int64_t)blockDim.x + w0; t0 < nq;
       t0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = t0 + lane;
    const bool in = t < nq;
    float y = 0.f;
    bool held;
    const bool ok =
        predict_warp<LPQ, LPQ / 2, TABLE>(a, tb, !in, in ? u[t] : 0, in ? it[t] : 0,
                                 wq + w0, wdot + w0, &y, &held);
    if (in) {
      if (!ok) bad = kErrIndex;
      yhat[t] = ok ? y : 0.f;
    }
  }
  if (bad) atomicOr(err, bad);
}

// Few queries: LPQ lanes take one query from its ids to its sum, so every load
// of the call is under way at once and no CTA fills a table first. The chunks
// of a row and the tree of its sum are those of predict_warp: the same bits.
// A call of 2,000 / 20,000 queries, kp = 40 on an 8 x 4 quantile grid: 24 / 26
// us, 31 / 31 by k_predict; kp = 56, 13 x 9 equal blocks 22 / 24, 31 / 31. From
// 40,000 on both take the same, and from 400,000 on the table wins.
template <int LPQ>
__global__ void __launch_bounds__(kPredictThreads)
k_predict_few(PredictArgs a, int64_t nq, const int32_t *__restrict__ u,
              const int32_t *__restrict__ it, float *__restrict__ yhat,
              int32_t *err) {
  const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / LPQ;
  const int sub = threadIdx.x % LPQ, n4 = a.kp / 4;
  const bool in = t < nq;
  int32_t blk = 0, r = 0, c = 0;
  const bool ok = in && locate(a.g, u[t], it[t], &blk, &r, &c);
  float mu = 0.f, dot = 0.f;
  if (ok) {
    const BlockMeta &bm = a.meta[blk];
    mu = a.mu[blk];
    if (bm.keff > 0 && (bm.owned || !a.owned_only)) {
      const float4 *fs = reinterpret_cast<const float4 *>(
          a.Fs + bm.fs_off + (int64_t)(bm.trans ? c : r) * a.kp);
      const float4 *fl = reinterpret_cast<const float4 *>(
          a.FL + bm.fl_off + (int64_t)(bm.trans ? r : c) * a.kp);
#pragma unroll 4
      for (int j = sub; j < n4; j += LPQ) {
        const float4 p = __ldg(fs + j), v = __ldg(fl + j);
        dot = fmaf(p.x, v.x, dot);
        dot = fmaf(p.y, v.y, dot);
        dot = fmaf(p.z, v.z, dot);
        dot = fmaf(p.w, v.w, dot);
      }
    }
  }
#pragma unroll
  for (int o = LPQ / 2; o > 0; o >>= 1)
    dot += __shfl_xor_sync(0xffffffffu, dot, o);
  if (!in || sub != 0) return;
  float y = mu + dot;
  if (a.clamp) y = fminf(fmaxf(y, a.lo), a.hi);
  yhat[t] = ok ? y : 0.f;
  if (!ok) atomicOr(err, kErrIndex);
}

// With a.owned_only, queries in blocks this context does not hold are
// skipped; the CTA's count of summed queries goes to counts.
template <int LPQ, bool TABLE>
__global__ void __launch_bounds__(kSqerrThreads)
k_sqerr(PredictArgs a, int64_t nq, const int32_t *__restrict__ u,
        const int32_t *__restrict__ it, const float *__restrict__ y,
        double *__restrict__ partials, long long *__restrict__ counts,
        int32_t *err) {
  __shared__ double red[kSqerrThreads];
  __shared__ long long cnt[kSqerrThreads];
  __shared__ Rows wq[kSqerrThreads];
  __shared__ float wdot[kSqerrThreads];
  extern __shared__ __align__(16) unsigned char table[];
  Table tb;
  if (TABLE) fill_table(a, tb, table);
  const int w0 = threadIdx.x & ~31, lane = threadIdx.x & 31;
  double acc = 0.0;
  long long n = 0;
  int32_t bad = 0;
  for (int64_t t0 = blockIdx.x * (int64_t)blockDim.x + w0; t0 < nq;
       t0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = t0 + lane;
    const bool in = t < nq;
    float yh;
    bool held;
    const bool ok =
        predict_warp<LPQ, 2, TABLE>(a, tb, !in, in ? u[t] : 0, in ? it[t] : 0,
                                 wq + w0, wdot + w0, &yh, &held);
    if (!in || (ok && a.owned_only && !held)) continue;
    if (!ok) {
      bad = kErrIndex;
      continue;
    }
    const double d = (double)yh - (double)y[t];
    acc = fma(d, d, acc);
    ++n;
  }
  if (bad) atomicOr(err, bad);
  red[threadIdx.x] = acc;
  cnt[threadIdx.x] = n;
  __syncthreads();
  for (int w = kSqerrThreads / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      red[threadIdx.x] += red[threadIdx.x + w];
      cnt[threadIdx.x] += cnt[threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = red[0];
    counts[blockIdx.x] = cnt[0];
  }
}

// out[0] = sum of the partial sums (fixed tree); out[1] = their count, as
// a float64 holding an exact integer below 2^53.
__global__ void __launch_bounds__(512)
k_sum_partials(const double *__restrict__ partials,
               const long long *__restrict__ counts, int n, double *out) {
  __shared__ double red[512];
  __shared__ long long cnt[512];
  red[threadIdx.x] = threadIdx.x < n ? partials[threadIdx.x] : 0.0;
  cnt[threadIdx.x] = threadIdx.x < n ? counts[threadIdx.x] : 0;
  __syncthreads();
  for (int w = 256; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      red[threadIdx.x] += red[threadIdx.x + w];
      cnt[threadIdx.x] += cnt[threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[0] = red[0];
    out[1] = (double)cnt[0];
  }
}

int grid_for(int64_t n) {
  int64_t g = (n + kPredictThreads - 1) / kPredictThreads;
  if (g < 1) g = 1;
  if (g > 152 * 8) g = 152 * 8;
  return (int)g;
}

// Four lanes a query or eight: whichever leaves fewer lanes without a chunk
// over the passes that a row of kp / 4 chunks takes, eight (fewer loads) when
// both leave the same. Ten million queries, four / eight lanes: kp = 12 206 /
// 259 us, 20 339 / 274, 40 404 / 443, 56 623 / 540.
template <typename F>
cudaError_t by_shape(const PredictArgs &a, F &&f) {
  const int n4 = a.kp / 4;
  auto lanes = [&](auto tb) {
    if ((n4 + 3) / 4 * 4 < (n4 + 7) / 8 * 8)
      return f(std::integral_constant<int, 4>(), tb);
    return f(std::integral_constant<int, 8>(), tb);
  };
  return fits_table(a.g) ? lanes(std::true_type()) : lanes(std::false_type());
}

}  // namespace

cudaError_t launch_predict(const PredictArgs &a, int64_t nq, const int32_t *u,
                           const int32_t *i, float *yhat, int32_t *err,
                           cudaStream_t st) {
  if (nq <= 0) return cudaSuccess;
  return by_shape(a, [&](auto l, auto tb) {
    constexpr int LPQ = decltype(l)::value;
    constexpr bool TB = decltype(tb)::value;
    if (nq <= kFewQueries) {
      const int64_t ctas = (nq * LPQ + kPredictThreads - 1) / kPredictThreads;
      k_predict_few<LPQ><<<(unsigned)ctas, kPredictThreads, 0, st>>>(
          a, nq, u, i, yhat, err);
      return cudaGetLastError();
    }
    k_predict<LPQ, TB><<<grid_for(nq), kPredictThreads, TB ? table_bytes(a.g) : 0,
                         st>>>(a, nq, u, i, yhat, err);
    return cudaGetLastError();
  });
}

cudaError_t launch_sqerr(const PredictArgs &a, int64_t nq, const int32_t *u,
                         const int32_t *i, const float *y, double *partials,
                         double *out, int32_t *err, cudaStream_t st) {
  static_assert(kSqerrBlocks <= 512, "final sum is one CTA of 512");
  long long *counts = reinterpret_cast<long long *>(partials + kSqerrBlocks);
  const cudaError_t e = by_shape(a, [&](auto l, auto tb) {
    constexpr int LPQ = decltype(l)::value;
    constexpr bool TB = decltype(tb)::value;
    k_sqerr<LPQ, TB><<<kSqerrBlocks, kSqerrThreads, TB ? table_bytes(a.g) : 0,
                       st>>>(a, nq, u, i, y, partials, counts, err);
    return cudaGetLastError();
  });
  if (e != cudaSuccess) return e;
  k_sum_partials<<<1, 512, 0, st>>>(partials, counts, kSqerrBlocks, out);
  return cudaGetLastError();
}

}  // namespace bsvd
