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
constexpr int64_t kFewQueries = 250000;  // see launch_predict
constexpr int64_t kFewLanes = 200000;
constexpr int kLanes = 4;                // lanes a query's squared error takes
// 304 CTAs of them fill the SMs
constexpr int kSqerrThreads = 512, kSqerrFewThreads = 256;
// One to one and a half queries a lane of the fewer, which need no table: one
// query at kp = 40 3.9 us (5.2 with a table and 512 threads), 20,000 4.9 (7.5).
template <int LPQ>
constexpr int64_t kSqerrFew = LPQ == 8 ? 77824 : LPQ == 4 ? 100000 : 130000;

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
  t.bounds.fill(a.g, sizeof(Place) * kTableBlocks);
  __syncthreads();
}

// The two factor rows of a query (null: the prediction is the mean alone).
struct Rows {
  const float4 *fs, *fl;
};

// 16-byte chunks of a row, which has LPQ sums: as many, where there are one or
// two (by_shape), and then no loop.
template <int LPQ>
__device__ __forceinline__ int chunks(const PredictArgs &a) {
  return LPQ <= 2 ? LPQ : a.kp / 4;
}

// The sum of LPQ partial sums, of which lane `sub` of L neighbours holds numbers
// sub, sub + L, ...: added in halves, the order of LPQ lanes' xor shuffles.
template <int LPQ, int L>
__device__ __forceinline__ float tree_sum(float (&dot)[LPQ / L]) {
#pragma unroll
  for (int o = LPQ / L / 2; o > 0; o >>= 1)
#pragma unroll
    for (int w = 0; w < o; ++w) dot[w] += dot[w + o];
#pragma unroll
  for (int o = L / 2; o > 0; o >>= 1)
    dot[0] += __shfl_xor_sync(0xffffffffu, dot[0], o);
  return dot[0];
}

// One query per lane (skip: none); every lane of the warp calls. Where the
// query is valid, *out is its prediction and the result true; *held says
// whether this context holds its block.
//
// A row of kp floats is read by L neighbouring lanes, 16 bytes each, so a
// warp's load touches 32 / L rows. With a lane per query every load touched
// 32 rows, and the lines a load can look up per cycle bound the kernel: ten
// million queries at kp = 40 took 0.58 ms, and take 0.38 ms with both changes,
// 78% of the L1's rate. The chunks of a row are dealt to LPQ sums, LPQ / L of
// them in each lane, which are added in a fixed tree: the same bits whatever L.
// The rows of UN steps are loaded together (kp = 56, ten million queries, UN =
// 2 / 4 at eight lanes: 0.65 / 0.55 ms). The squared errors, at half the warps,
// take four lanes and UN = 2: 0.37 ms at kp = 56 and 0.23 at 20 on 4 x 4 blocks
// (eight lanes 0.44, 0.26), 0.45 and 0.29 on 900 blocks (0.84, 0.47).
template <int LPQ, int LANES, int STEPS, bool TABLE>
__device__ __forceinline__ bool predict_warp(const PredictArgs &a,
                                             const Table &tb, bool skip,
                                             int32_t u, int32_t i, Rows *wq,
                                             float *wdot, float *out,
                                             bool *held) {
  constexpr int L = LANES < LPQ ? LANES : LPQ;
  constexpr int UN = STEPS < L ? STEPS : L;
  constexpr int QPI = 32 / L;                // queries per step
  constexpr int W = LPQ / L;                 // sums per lane
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
  if (L > 1) {
    wq[lane] = mine;
    __syncwarp();
  }
  const int n4 = chunks<LPQ>(a), sub = lane % L;
  float own = 0.f;                           // L = 1: this lane's own sum
#pragma unroll 1
  for (int s = 0; s < 32; s += QPI * UN) {
    Rows q[UN];
    float dot[UN][W];
#pragma unroll
    for (int x = 0; x < UN; ++x) {
      q[x] = L > 1 ? wq[s + x * QPI + lane / L] : mine;
#pragma unroll
      for (int w = 0; w < W; ++w) dot[x][w] = 0.f;
    }
    // (with several sums a lane, as many rounds in every lane)
    for (int j = W == 1 ? sub : 0; j < n4; j += LPQ) {
      float4 p[UN][W], v[UN][W];
#pragma unroll
      for (int x = 0; x < UN; ++x)
#pragma unroll
        for (int w = 0; w < W; ++w) {
          const int jw = W == 1 ? j : j + w * L + sub;
          p[x][w] = v[x][w] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (q[x].fs && (W == 1 || jw < n4)) {
            p[x][w] = __ldg(q[x].fs + jw);
            v[x][w] = __ldg(q[x].fl + jw);
          }
        }
#pragma unroll
      for (int x = 0; x < UN; ++x)
#pragma unroll
        for (int w = 0; w < W; ++w) {
          dot[x][w] = fmaf(p[x][w].x, v[x][w].x, dot[x][w]);
          dot[x][w] = fmaf(p[x][w].y, v[x][w].y, dot[x][w]);
          dot[x][w] = fmaf(p[x][w].z, v[x][w].z, dot[x][w]);
          dot[x][w] = fmaf(p[x][w].w, v[x][w].w, dot[x][w]);
        }
    }
#pragma unroll
    for (int x = 0; x < UN; ++x) {
      const float d = tree_sum<LPQ, L>(dot[x]);
      if (L == 1) own = d;
      else if (sub == 0) wdot[s + x * QPI + lane / L] = d;
    }
  }
  if (L > 1) {
    __syncwarp();
    own = wdot[lane];
    __syncwarp();                  // wq and wdot are the next call's
  }
  float y = mu + own;
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
        predict_warp<LPQ, LPQ, (LPQ > 2 ? LPQ / 2 : LPQ), TABLE>(
            a, tb, !in, in ? u[t] : 0, in ? it[t] : 0, wq + w0, wdot + w0, &y,
            &held);
    if (in) {
      if (!ok) bad = kErrIndex;
      yhat[t] = ok ? y : 0.f;
    }
  }
  if (bad) atomicOr(err, bad);
}

// L lanes take one query from its ids to its sum, so every load of a short call
// is under way at once and no CTA fills a table first. The chunks of a row are
// dealt to LPQ sums, LPQ / L of them in each lane, and these are added in the
// tree of predict_warp: the same bits whatever L.
template <int LPQ, int L>
__global__ void __launch_bounds__(kPredictThreads)
k_predict_few(PredictArgs a, int64_t nq, const int32_t *__restrict__ u,
              const int32_t *__restrict__ it, float *__restrict__ yhat,
              int32_t *err) {
  constexpr int W = LPQ / L;                 // sums per lane
  const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / L;
  const int sub = threadIdx.x % L, n4 = chunks<LPQ>(a);
  const bool in = t < nq;
  int32_t blk = 0, r = 0, c = 0;
  const bool ok = in && locate(a.g, u[t], it[t], &blk, &r, &c);
  float mu = 0.f, dot[W];
#pragma unroll
  for (int w = 0; w < W; ++w) dot[w] = 0.f;
  if (ok) {
    const BlockMeta &bm = a.meta[blk];
    mu = a.mu[blk];
    if (bm.keff > 0 && (bm.owned || !a.owned_only)) {
      const float4 *fs = reinterpret_cast<const float4 *>(
          a.Fs + bm.fs_off + (int64_t)(bm.trans ? c : r) * a.kp);
      const float4 *fl = reinterpret_cast<const float4 *>(
          a.FL + bm.fl_off + (int64_t)(bm.trans ? r : c) * a.kp);
#pragma unroll(4 / W)
      for (int j = W == 1 ? sub : 0; j < n4; j += LPQ) {
#pragma unroll
        for (int w = 0; w < W; ++w) {
          const int jw = W == 1 ? j : j + w * L + sub;
          if (W > 1 && jw >= n4) continue;
          const float4 p = __ldg(fs + jw), v = __ldg(fl + jw);
          dot[w] = fmaf(p.x, v.x, dot[w]);
          dot[w] = fmaf(p.y, v.y, dot[w]);
          dot[w] = fmaf(p.z, v.z, dot[w]);
          dot[w] = fmaf(p.w, v.w, dot[w]);
        }
      }
    }
  }
  const float sum = tree_sum<LPQ, L>(dot);
  if (!in || sub != 0) return;
  float y = mu + sum;
  if (a.clamp) y = fminf(fmaxf(y, a.lo), a.hi);
  yhat[t] = ok ? y : 0.f;
  if (!ok) atomicOr(err, kErrIndex);
}

// Sum over the CTA's THREADS threads in a fixed tree; thread 0's is the result.
// Across the warps first: a float64 addition takes the SM 19 cycles a warp, so
// the shuffles are left to one of them.
template <int THREADS>
__device__ __forceinline__ void cta_sum(double *acc, long long *n) {
  __shared__ double red[THREADS];
  __shared__ long long cnt[THREADS];
  const int t = threadIdx.x;
#pragma unroll
  for (int w = THREADS / 2; w >= 32; w >>= 1) {
    if (t >= w && t < 2 * w) {
      red[t] = *acc;
      cnt[t] = *n;
    }
    __syncthreads();
    if (t < w) {
      *acc += red[t + w];
      *n += cnt[t + w];
    }
  }
  if (t >= 32) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    *acc += __shfl_xor_sync(0xffffffffu, *acc, o);
    *n += __shfl_xor_sync(0xffffffffu, *n, o);
  }
}

// With a.owned_only, queries in blocks this context does not hold are
// skipped; the CTA's count of summed queries goes to counts.
template <int LPQ, int UN, bool TABLE, int THREADS>
__global__ void __launch_bounds__(THREADS)
k_sqerr(PredictArgs a, int64_t nq, const int32_t *__restrict__ u,
        const int32_t *__restrict__ it, const float *__restrict__ y,
        double *__restrict__ partials, long long *__restrict__ counts,
        int32_t *err) {
  __shared__ Rows wq[THREADS];
  __shared__ float wdot[THREADS];
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
    const bool ok = predict_warp<LPQ, kLanes, UN, TABLE>(
        a, tb, !in, in ? u[t] : 0, in ? it[t] : 0, wq + w0, wdot + w0, &yh,
        &held);
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
  cta_sum<THREADS>(&acc, &n);
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = acc;
    counts[blockIdx.x] = n;
  }
}

// out[0] = sum of the partial sums (fixed tree); out[1] = their count, as
// a float64 holding an exact integer below 2^53.
__global__ void __launch_bounds__(512)
k_sum_partials(const double *__restrict__ partials,
               const long long *__restrict__ counts, int n, double *out) {
  double acc = threadIdx.x < n ? partials[threadIdx.x] : 0.0;
  long long cnt = threadIdx.x < n ? counts[threadIdx.x] : 0;
  cta_sum<512>(&acc, &cnt);
  if (threadIdx.x == 0) {
    out[0] = acc;
    out[1] = (double)cnt;
  }
}

int grid_for(int64_t n) {
  int64_t g = (n + kPredictThreads - 1) / kPredictThreads;
  if (g < 1) g = 1;
  if (g > 152 * 8) g = 152 * 8;
  return (int)g;
}

// A row of one or two chunks (of 16 bytes) has as many sums. Longer ones have
// four or eight: whichever leaves fewer of them without a chunk over the passes
// that the kp / 4 chunks take, eight when both leave the same.
template <typename F>
cudaError_t by_shape(const PredictArgs &a, F &&f) {
  const int n4 = a.kp / 4;
  auto lanes = [&](auto tb) {
    if (n4 <= 1) return f(std::integral_constant<int, 1>(), tb);
    if (n4 == 2) return f(std::integral_constant<int, 2>(), tb);
    if ((n4 + 3) / 4 * 4 < (n4 + 7) / 8 * 8)
      return f(std::integral_constant<int, 4>(), tb);
    return f(std::integral_constant<int, 8>(), tb);
  };
  return fits_table(a.g) ? lanes(std::true_type()) : lanes(std::false_type());
}

}  // namespace

template <int LPQ, int L>
static cudaError_t few(const PredictArgs &a, int64_t nq, const int32_t *u,
                       const int32_t *i, float *yhat, int32_t *err,
                       cudaStream_t st) {
  const int64_t ctas = (nq * L + kPredictThreads - 1) / kPredictThreads;
  k_predict_few<LPQ, L><<<(unsigned)ctas, kPredictThreads, 0, st>>>(
      a, nq, u, i, yhat, err);
  return cudaGetLastError();
}

// Which form, and how many lanes a query. While all queries' lanes are no more
// than two thirds of a wave (kFewLanes of 152 x 2,048), one lane a sum. Beyond
// that two lanes for rows of up to five chunks, one for rows of one or two, up
// to kFewQueries, and then, or for longer rows at once, the form with a table
// (for grids without one the same, with the blocks read in place; with explicit
// bounds, rows of three chunks stay with two lanes there). Short rows leave that
// form's lanes idle: without the rule ten million queries at kp = 4 took 143 us.
// The kernel alone, us, a lane per query / now: 4 x 4 equal blocks, 40,000
// queries kp = 8 3.4 / 3.1, 20 4.4 / 3.6, 40 6.0 / 3.9; 120,000 queries 4.4 /
// 4.5, 6.4 / 5.9, 9.7 / 7.1; ten million kp = 4 107 / 91, 8 137 / 123, 12 175 /
// 150, 20 260 / 205, 40 491 / 281, 56 685 / 307; 900 blocks, ten million kp = 8
// 184 / 180, 12 224 / 202, 20 310 / 254, 56 751 / 423.
cudaError_t launch_predict(const PredictArgs &a, int64_t nq, const int32_t *u,
                           const int32_t *i, float *yhat, int32_t *err,
                           cudaStream_t st) {
  if (nq <= 0) return cudaSuccess;
  const int n4 = a.kp / 4;
  const bool equal = a.g.equal_rows && a.g.equal_cols;
  return by_shape(a, [&](auto l, auto tb) {
    constexpr int LPQ = decltype(l)::value;
    constexpr bool TB = decltype(tb)::value;
    // (a lane beyond the row's chunks adds zeros)
    if (nq * 4 <= kFewLanes)
      return nq * 8 <= kFewLanes && LPQ == 8
                 ? few<8, 8>(a, nq, u, i, yhat, err, st)
                 : few<(LPQ > 4 ? LPQ : 4), 4>(a, nq, u, i, yhat, err, st);
    if constexpr (LPQ == 1) {
      return few<1, 1>(a, nq, u, i, yhat, err, st);
    } else {
      if (LPQ == 2 && nq * 2 > kFewLanes && (nq <= 2 * kFewQueries || !TB))
        return few<LPQ, 1>(a, nq, u, i, yhat, err, st);
      if (n4 <= 5 && (nq <= kFewQueries || (n4 == 3 && !TB && !equal)))
        return few<LPQ, 2>(a, nq, u, i, yhat, err, st);
      k_predict<LPQ, TB><<<grid_for(nq), kPredictThreads,
                           TB ? table_bytes(a.g) : 0, st>>>(a, nq, u, i, yhat,
                                                            err);
      return cudaGetLastError();
    }
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
    if (nq <= kSqerrFew<LPQ>)
      k_sqerr<LPQ, 4, false, kSqerrFewThreads>
          <<<kSqerrBlocks, kSqerrFewThreads, 0, st>>>(a, nq, u, i, y, partials,
                                                      counts, err);
    else
      k_sqerr<LPQ, 2, TB, kSqerrThreads>
          <<<kSqerrBlocks, kSqerrThreads, TB ? table_bytes(a.g) : 0, st>>>(
              a, nq, u, i, y, partials, counts, err);
    return cudaGetLastError();
  });
  if (e != cudaSuccess) return e;
  k_sum_partials<<<1, 512, 0, st>>>(partials, counts, kSqerrBlocks, out);
  return cudaGetLastError();
}

}  // namespace bsvd
