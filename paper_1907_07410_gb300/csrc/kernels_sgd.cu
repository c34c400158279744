// The paper's own method: blocked stochastic gradient descent on the biased
// latent-factor model (Section 2.2, Eq. 3 and 10-13; Algorithms 1-2).
//
// One launch runs one epoch. The ratings come in tasks (kernels_sgd_order.cu):
// a task is the ratings of one owner (an item when n <= m, else a user) in
// one block, and a warp runs it with the owner's parameters in registers.
// A rating needs its owner's and its other id's parameters as the previous
// rating of that id left them; everything else may run at the same time. So
// instead of walking the blocks of a step one rating after another, warps
// take tasks in epoch order and wait, rating by rating, until the other id's
// parameters have reached the version that the epoch's order gives. Every
// rating reads exactly the values it would read in the sequential walk, so
// the results equal it bit for bit, whatever the timing.
//
// What bounds it is the longest chain of dependent ratings. On a long-tailed
// 6040 x 3952 matrix of 900,189 ratings that is 5,754 ratings on an 8 x 8 grid
// (the most popular item alone has 5,444), where a warp per block of a step walked
// the 129,645 ratings of the eight steps' heaviest blocks of an 8 x 8 grid
// one after another. A float64 operation on GB300 takes 63 cycles to the
// next one of the same warp, dependent or not (measured; an SM issues one
// each 19 cycles), so a float64 rating costs a warp its number of float64
// instructions: 21 at k = 13, with both sides' parameters in one register.
// Measured with nothing to wait for: 1.04 us a rating in float64, 0.37 us in
// float32 (0.8 and 0.15 us of it arithmetic). Epochs of that matrix, one
// warp per block of a step -> now: 8 x 8 grid 187 -> 6.9 ms (float64),
// 48 -> 3.2 ms (float32); 64 x 64: 48 -> 6.3 ms, 10 -> 2.8 ms.
//
// Hand-over. A parameter's words carry their version: a float is stored as
// one 64-bit word (value, version), a double as two (half, version). Reading
// a parameter and checking that it is the awaited one is then a single
// relaxed load per lane, with no flag beside the data and no fence: the
// store and the polling load are one trip to L2 each.
//
// Waiting ends: tasks are claimed in an order in which every task depends
// only on earlier ones, and a warp works on one task at a time, so the
// earliest unfinished task never waits for a task that has not been claimed.
// A wait that sees nothing happen anywhere for idle_polls polls (no task
// claimed, no 32 ratings done) gives up: kErrTimeout, and every warp leaves.
#include <type_traits>

#include "kernels.h"

namespace bsvd {

namespace {

typedef unsigned long long u64;
constexpr unsigned kAll = 0xffffffffu;
constexpr unsigned kLookPolls = 1u << 12;   // polls between looks at ctl
constexpr int kSgdThreads = 256;
// Resident CTAs per SM: 16 warps. Every warp that waits holds a task, so too
// few of them keep tasks on the longest chain from starting (8 x 8 epochs,
// float64: 9.1 ms with one CTA, 6.9 with two, 7.6 with three; float32: 3.7,
// 3.2, 3.7).
constexpr int kSgdCtas = 2;

// ---- parameters with versions ---------------------------------------------

// One parameter: its value, and the version in each of its words.
template <typename T>
struct Cell;

template <>
struct Cell<double> {
  static constexpr int kWords = 2;
  u64 a, b;
  __device__ __forceinline__ void load(const u64 *p) {
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];"
                 : "=l"(a)
                 : "l"(p)
                 : "memory");
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];"
                 : "=l"(b)
                 : "l"(p + 1)
                 : "memory");
  }
  __device__ __forceinline__ bool is(unsigned ver) const {
    return (unsigned)(a >> 32) == ver && (unsigned)(b >> 32) == ver;
  }
  __device__ __forceinline__ double value() const {
    return __hiloint2double((int)(unsigned)b, (int)(unsigned)a);
  }
  static __device__ __forceinline__ void store(u64 *p, double v, unsigned ver,
                                               bool on) {
    const u64 t = (u64)ver << 32;
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %3, 0;\n\t"
        "@q st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};\n\t}" ::"l"(p),
        "l"(t | (unsigned)__double2loint(v)),
        "l"(t | (unsigned)__double2hiint(v)), "r"((int)on)
        : "memory");
  }
};

template <>
struct Cell<float> {
  static constexpr int kWords = 1;
  u64 a;
  __device__ __forceinline__ void load(const u64 *p) {
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];"
                 : "=l"(a)
                 : "l"(p)
                 : "memory");
  }
  __device__ __forceinline__ bool is(unsigned ver) const {
    return (unsigned)(a >> 32) == ver;
  }
  __device__ __forceinline__ float value() const {
    return __uint_as_float((unsigned)a);
  }
  static __device__ __forceinline__ void store(u64 *p, float v, unsigned ver,
                                               bool on) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %2, 0;\n\t"
        "@q st.relaxed.gpu.global.u64 [%0], %1;\n\t}" ::"l"(p),
        "l"(((u64)ver << 32) | __float_as_uint(v)), "r"((int)on)
        : "memory");
  }
};

// Every operation rounds once, in the parameters' type.
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// The epoch's control words: [0] tasks claimed, [1] progress (32 ratings of a
// task done), [2] nonzero when a wait gave up.
struct Wait {
  unsigned polls = 0, idle = 0;
  u64 seen = 0;
  // Called after a poll that failed, by the whole warp; false: give up. The
  // words are what lane 0 sees of them, so that the whole warp goes on or the
  // whole warp leaves.
  __device__ __forceinline__ bool again(const SgdEpoch &a) {
    if (++polls % kLookPolls != 0) return true;
    volatile u64 *ctl = a.ctl;
    if (__shfl_sync(kAll, ctl[2], 0) != 0) return false;
    // both only grow
    const u64 now = __shfl_sync(kAll, ctl[0] + ctl[1], 0);
    idle = now == seen ? idle + kLookPolls : 0;
    seen = now;
    if (idle < a.idle_polls) return true;
    if ((threadIdx.x & 31) == 0) {
      atomicOr(a.err, kErrTimeout);
      ctl[2] = 1;
    }
    return false;
  }
};

// A task's ratings, 32 at a time: lane l holds rating base + l.
struct Chunk {
  int32_t id;
  unsigned ver;
  float x;
  __device__ __forceinline__ void load(const SgdEpoch &a, int64_t t,
                                       int64_t end) {
    id = 0;
    ver = 0;
    x = 0.f;
    if (t < end) {
      id = a.other[t];
      ver = a.other_ver[t];
      x = a.x[t];
    }
  }
};

// Takes the next task. A warp claims when its last task's last rating has its
// inputs, and the number arrives while that rating is worked on: a task
// claimed any earlier would wait for whatever the warp still waits for (with
// one claimed at the start of the one before, an 8 x 8 epoch took 22 ms).
__device__ __forceinline__ u64 claim(const SgdEpoch &a) {
  return (threadIdx.x & 31) == 0 ? atomicAdd(&a.ctl[0], 1ull) : 0ull;
}
__device__ __forceinline__ int64_t claimed(u64 t) {
  return (int64_t)__shfl_sync(kAll, t, 0);
}

// How many ratings ahead the other rows are loaded. A trip to L2 is shorter
// than a float64 rating and longer than a float32 one (8 x 8 epochs in
// float32: 3.8 ms one ahead, 3.2 two, 3.3 three; float64: 6.9 ms, 7.1 two).
template <typename T>
constexpr int kAhead = sizeof(T) == 8 ? 1 : 2;

// A rating of the task whose other row is on its way.
template <typename T, int N>
struct Coming {
  u64 *row;
  unsigned ver;
  T x;
  Cell<T> cell[N];
};

__device__ __forceinline__ int64_t first_of(const SgdEpoch &a, int64_t task) {
  return a.index32 ? (int64_t)static_cast<const unsigned *>(a.task_first)[task]
                   : (int64_t)static_cast<const u64 *>(a.task_first)[task];
}

// Dot product in factor order, from products held by lanes 0 .. K - 1: every
// lane fetches them all, then adds. The first product came from a fused
// multiply-add onto +0, which equals rounding the product and adding it to
// +0, and +0 in the place of a later product of -0 changes no sum (the
// running sum is never -0).
template <typename T, int K>
__device__ __forceinline__ T ordered_sum(T prod) {
  T s[K];
#pragma unroll
  for (int j = 0; j < K; ++j) s[j] = __shfl_sync(kAll, prod, j);
  T dot = s[0];
#pragma unroll
  for (int j = 1; j < K; ++j) dot = add_rn(dot, s[j]);
  return dot;
}

// One epoch with k = K factors.
//
// K <= 15: lanes 0 .. K hold the owner's factors and bias, lanes 16 .. 16 + K
// the other id's, so that one instruction updates both sides. K > 15: lane f
// holds factor f of both sides, lane K both biases (K = 32: every lane holds
// and updates the biases alike). A bias is a factor whose partner is 1 (e * 1
// is exact) with rates of its own.
template <typename T, int K>
__global__ void __launch_bounds__(kSgdThreads)
k_sgd_epoch(SgdEpoch a) {
  constexpr int W = Cell<T>::kWords, ROW = (K + 1) * W, D = kAhead<T>;
  constexpr bool PACK = K <= 15, ALL = K == 32;
  constexpr int N = ALL ? 2 : 1;               // cells per lane
  const int lane = threadIdx.x & 31, f = PACK ? lane & 15 : lane;
  const bool on = f <= K, bias = f == K;
  const bool oi = a.own_items != 0;
  // this lane's part of the owner's and of the other id's row
  const bool has_own = on && (!PACK || lane < 16);
  const bool has_other = on && (!PACK || lane >= 16);
  const int fo = on ? f * W : 0;
  auto rate = [&](bool user, bool b, double fu, double fi, double bu_,
                  double bi_) {
    return (T)(b ? (user ? bu_ : bi_) : (user ? fu : fi));
  };
  const bool s0_user = PACK ? (lane >= 16) == oi : !oi;   // v's side
  const T al0 = rate(s0_user, bias, a.r.a_user, a.r.a_item, a.r.a_ubias, a.r.a_ibias);
  const T be0 = rate(s0_user, bias, a.r.b_user, a.r.b_item, a.r.b_ubias, a.r.b_ibias);
  const T al1 = rate(oi, bias, a.r.a_user, a.r.a_item, a.r.a_ubias, a.r.a_ibias);
  const T be1 = rate(oi, bias, a.r.b_user, a.r.b_item, a.r.b_ubias, a.r.b_ibias);
  const int64_t ntasks = *a.ntasks;
  for (u64 ticket = claim(a);;) {
    const int64_t task = claimed(ticket);
    if (task >= ntasks) return;
    const int64_t t0 = first_of(a, task);
    const int64_t n = first_of(a, task + 1) - t0;
    Chunk c, cn;
    c.load(a, t0 + lane, t0 + n);
    cn.load(a, t0 + 32 + lane, t0 + n);
    u64 *own = a.own_rows + (int64_t)a.own[t0] * ROW;
    const unsigned own_ver = a.own_ver[t0];
    Coming<T, N> q[D];
    // rating r of the task (in order): its ids, and its row on its way
    auto fetch = [&](int64_t r, Coming<T, N> &w) {
      const int j = (int)r & 31;
      if (j == 0 && r > 0) {
        c = cn;
        cn.load(a, t0 + r + 32 + lane, t0 + n);
        if (lane == 0) atomicAdd(&a.ctl[1], 1ull);
      }
      w.ver = __shfl_sync(kAll, c.ver, j);
      w.row = a.other_rows + (int64_t)__shfl_sync(kAll, c.id, j) * ROW;
      w.x = (T)__shfl_sync(kAll, c.x, j);
      w.cell[0].load(w.row + fo);
      if (ALL) w.cell[N - 1].load(w.row + K * W);
    };
    auto here = [&](const Coming<T, N> &w) {
      bool ok = w.cell[0].is(w.ver);
      if (ALL) ok = ok && w.cell[N - 1].is(w.ver);
      return __all_sync(kAll, ok);
    };
    Cell<T> co[N];
#pragma unroll
    for (int d = 0; d < D; ++d) {
      q[d] = Coming<T, N>();
      if (d < n) fetch(d, q[d]);
    }
    {
      Wait w;
      for (;;) {
        co[0].load(own + fo);
        if (ALL) co[N - 1].load(own + K * W);
        bool ok = co[0].is(own_ver);
        if (ALL) ok = ok && co[N - 1].is(own_ver);
        if (__all_sync(kAll, ok)) break;
        if (!w.again(a)) return;
      }
    }
    // PACK: v holds the owner's parameter or the other id's, by lane; else v
    // holds the owner's and y the other id's. ALL: the biases bo, bx.
    T v = has_own ? co[0].value() : (T)0, y = (T)0, bo = (T)0, bx = (T)0;
    if (ALL) bo = co[N - 1].value();
    // rating r, waiting in s (which then takes rating r + D); false: give up.
    // The slots are used in turn rather than shifted: copying a register
    // whose load is in flight would wait for the load.
    auto rating = [&](int64_t r, Coming<T, N> &s) -> bool {
      if (!here(s)) {
        Wait w;
        do {
          if (!w.again(a)) return false;
          s.cell[0].load(s.row + fo);
          if (ALL) s.cell[N - 1].load(s.row + K * W);
        } while (!here(s));
      }
      if (has_other) (PACK ? v : y) = s.cell[0].value();
      if (ALL) bx = s.cell[N - 1].value();
      u64 *row = s.row;
      const unsigned ver = s.ver;
      const T x = s.x;
      const bool more = r + 1 < n;
      T w, bu, bi;                     // the partner, and the two biases
      if constexpr (PACK) {
        w = __shfl_xor_sync(kAll, v, 16);
        bu = __shfl_sync(kAll, v, (oi ? 16 : 0) + K);
        bi = __shfl_sync(kAll, v, (oi ? 0 : 16) + K);
      } else {
        w = y;
        const T b0 = ALL ? bo : __shfl_sync(kAll, v, K & 31);
        const T b1 = ALL ? bx : __shfl_sync(kAll, y, K & 31);
        bu = oi ? b1 : b0;
        bi = oi ? b0 : b1;
      }
      if (!more) ticket = claim(a);
      if (r + D < n) fetch(r + D, s);
      const T prod = fma_rn(v, w, (T)0);
      const T dot = ordered_sum<T, K>(prod);
      const T e = sub_rn(sub_rn(sub_rn(x, bu), bi), dot);
      const T w1 = bias ? (T)1 : w;
      T y1 = (T)0;
      if constexpr (!PACK)
        y1 = add_rn(y, mul_rn(al1, sub_rn(mul_rn(e, bias ? (T)1 : v),
                                          mul_rn(be1, y))));
      v = add_rn(v, mul_rn(al0, sub_rn(mul_rn(e, w1), mul_rn(be0, v))));
      Cell<T>::store(row + fo, PACK ? v : y1, ver + 1, has_other);
      if constexpr (ALL) {
        const T ao = (T)(oi ? a.r.a_ibias : a.r.a_ubias);
        const T bo_ = (T)(oi ? a.r.b_ibias : a.r.b_ubias);
        const T ax = (T)(oi ? a.r.a_ubias : a.r.a_ibias);
        const T bx_ = (T)(oi ? a.r.b_ubias : a.r.b_ibias);
        const T bx1 = add_rn(bx, mul_rn(ax, sub_rn(e, mul_rn(bx_, bx))));
        bo = add_rn(bo, mul_rn(ao, sub_rn(e, mul_rn(bo_, bo))));
        Cell<T>::store(row + K * W, bx1, ver + 1, lane == 0);
      }
      return true;
    };
    for (int64_t r = 0; r < n;) {
#pragma unroll
      for (int d = 0; d < D; ++d) {
        if (r >= n) break;
        if (!rating(r, q[d])) return;
        ++r;
      }
    }
    Cell<T>::store(own + fo, v, own_ver + (unsigned)n, has_own);
    if (ALL) Cell<T>::store(own + K * W, bo, own_ver + (unsigned)n, lane == 0);
  }
}

// P, Q (rows of k), bu, bi in float64 <-> the versioned rows of k + 1
// parameters (factors, then the bias). PACK: float64 -> rows, rounded to T;
// else rows -> float64 (exact). Either way every version becomes 0, and the
// epoch's control words too, for the epoch that follows.
template <typename T, bool PACK>
__global__ void __launch_bounds__(256)
k_sgd_rows(int64_t m, int64_t n, int32_t k, double *__restrict__ P,
           double *__restrict__ Q, double *__restrict__ bu,
           double *__restrict__ bi, u64 *__restrict__ prow,
           u64 *__restrict__ qrow, u64 *__restrict__ ctl) {
  constexpr int W = Cell<T>::kWords;
  const int64_t kk = k + 1, np = m * kk, total = np + n * kk;
  if (blockIdx.x == 0 && threadIdx.x < 3) ctl[threadIdx.x] = 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const bool user = e < np;
    const int64_t q = user ? e : e - np;
    const int64_t row = q / kk;
    const int f = (int)(q - row * kk);
    double *d = user ? (f < k ? P + row * k + f : bu + row)
                     : (f < k ? Q + row * k + f : bi + row);
    u64 *c = (user ? prow : qrow) + q * W;
    T v;
    if (PACK) {
      v = (T)*d;
    } else {
      Cell<T> cell;
      cell.load(c);
      v = cell.value();
      *d = (double)v;
    }
    Cell<T>::store(c, v, 0, true);
  }
}

// Eq. 3 in the oracle's order: (sum_f p_f q_f, in f order) + bu + bi
__device__ __forceinline__ double sgd_eval(int32_t k, const double *P,
                                           const double *Q, const double *bu,
                                           const double *bi, int32_t uu,
                                           int32_t ii) {
  const double *p = P + (int64_t)uu * k;
  const double *q = Q + (int64_t)ii * k;
  double dot = 0.0;
  for (int f = 0; f < k; ++f) dot = __dadd_rn(dot, __dmul_rn(p[f], q[f]));
  return __dadd_rn(__dadd_rn(dot, bu[uu]), bi[ii]);
}

__global__ void __launch_bounds__(256)
k_sgd_predict(int64_t nq, const int32_t *__restrict__ u,
              const int32_t *__restrict__ it, int32_t k, int64_t m, int64_t n,
              const double *__restrict__ P, const double *__restrict__ Q,
              const double *__restrict__ bu, const double *__restrict__ bi,
              double *__restrict__ yhat, int32_t *err) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nq;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t uu = u[t], ii = it[t];
    if (uu < 0 || uu >= m || ii < 0 || ii >= n) {
      atomicOr(err, kErrIndex);
      yhat[t] = 0.0;
      continue;
    }
    yhat[t] = sgd_eval(k, P, Q, bu, bi, uu, ii);
  }
}

// Squared training errors: per-CTA partial sums in a fixed tree, then one
// CTA adds the partials in index order.
__global__ void __launch_bounds__(256)
k_sgd_sqerr(int64_t nnz, const int32_t *__restrict__ u,
            const int32_t *__restrict__ it, const float *__restrict__ x,
            int32_t k, const double *__restrict__ P,
            const double *__restrict__ Q, const double *__restrict__ bu,
            const double *__restrict__ bi, double *__restrict__ partials) {
  __shared__ double red[256];
  double acc = 0.0;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nnz;
       t += (int64_t)gridDim.x * blockDim.x) {
    const double d = __dsub_rn((double)x[t], sgd_eval(k, P, Q, bu, bi, u[t],
                                                      it[t]));
    acc = __dadd_rn(acc, __dmul_rn(d, d));
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) partials[blockIdx.x] = red[0];
}

__global__ void __launch_bounds__(512)
k_sgd_sum(const double *__restrict__ partials, int n, double *out) {
  __shared__ double red[512];
  red[threadIdx.x] = threadIdx.x < n ? partials[threadIdx.x] : 0.0;
  __syncthreads();
  for (int w = 256; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0];
}

int sgd_grid(int64_t n) {
  int64_t want = (n + 255) / 256;
  if (want < 1) want = 1;
  if (want > 152 * 8) want = 152 * 8;
  return (int)want;
}

}  // namespace

size_t sgd_row_bytes(int32_t k, int32_t f32) {
  return sizeof(u64) * (size_t)(k + 1) * (f32 ? 1 : 2);
}

template <typename T>
static cudaError_t rows_impl(int pack, int64_t m, int64_t n, int32_t k,
                             double *P, double *Q, double *bu, double *bi,
                             void *prow, void *qrow, unsigned long long *ctl,
                             cudaStream_t st) {
  const int g = sgd_grid((m + n) * (k + 1));
  u64 *pr = static_cast<u64 *>(prow), *qr = static_cast<u64 *>(qrow);
  if (pack)
    k_sgd_rows<T, true><<<g, 256, 0, st>>>(m, n, k, P, Q, bu, bi, pr, qr, ctl);
  else
    k_sgd_rows<T, false><<<g, 256, 0, st>>>(m, n, k, P, Q, bu, bi, pr, qr, ctl);
  return cudaGetLastError();
}

cudaError_t launch_sgd_rows(int32_t pack, int32_t f32, int64_t m, int64_t n,
                            int32_t k, double *P, double *Q, double *bu,
                            double *bi, void *prow, void *qrow, unsigned long long *ctl,
                            cudaStream_t st) {
  return f32 ? rows_impl<float>(pack, m, n, k, P, Q, bu, bi, prow, qrow, ctl, st)
             : rows_impl<double>(pack, m, n, k, P, Q, bu, bi, prow, qrow, ctl,
                                 st);
}

template <typename T, int K>
static cudaError_t epoch_k(const SgdEpoch &a, int ctas, cudaStream_t st) {
  if (a.k == K) {
    k_sgd_epoch<T, K><<<ctas, kSgdThreads, 0, st>>>(a);
    return cudaGetLastError();
  }
  if constexpr (K < 32) return epoch_k<T, K + 1>(a, ctas, st);
  return cudaErrorInvalidValue;
}

cudaError_t launch_sgd_epoch(const SgdEpoch &a, int64_t nnz, int32_t f32,
                             int32_t nsm, cudaStream_t st) {
  if (nnz <= 0) return cudaSuccess;
  const int64_t want = (nnz + 7) / 8;          // at most a warp per rating
  const int ctas = (int)(want < kSgdCtas * nsm ? want : kSgdCtas * nsm);
  SgdEpoch e = a;
  e.index32 = sgd_index_bytes(nnz) == sizeof(unsigned) ? 1 : 0;
  return f32 ? epoch_k<float, 1>(e, ctas, st) : epoch_k<double, 1>(e, ctas, st);
}

cudaError_t launch_sgd_sqerr(int64_t nnz, const int32_t *u, const int32_t *i,
                             const float *x, int32_t k, const double *P,
                             const double *Q, const double *bu,
                             const double *bi, double *partials, double *out,
                             cudaStream_t st) {
  static_assert(kSqerrBlocks <= 512, "final sum is one CTA of 512");
  k_sgd_sqerr<<<kSqerrBlocks, 256, 0, st>>>(nnz, u, i, x, k, P, Q, bu, bi,
                                            partials);
  k_sgd_sum<<<1, 512, 0, st>>>(partials, kSqerrBlocks, out);
  return cudaGetLastError();
}

cudaError_t launch_sgd_predict(int64_t nq, const int32_t *u, const int32_t *i,
                               int32_t k, int64_t m, int64_t n,
                               const double *P, const double *Q,
                               const double *bu, const double *bi,
                               double *yhat, int32_t *err, cudaStream_t st) {
  if (nq <= 0) return cudaSuccess;
  k_sgd_predict<<<sgd_grid(nq), 256, 0, st>>>(nq, u, i, k, m, n, P, Q, bu, bi,
                                              yhat, err);
  return cudaGetLastError();
}

}  // namespace bsvd
