// Rank-k reconstruction of one block on the tcgen05 tensor cores.
//
// Section 2 approximates a block by its rank-k truncation U_k S_k V_k^T; the
// library holds it as two factors, the user side P = U_k S_k (mb x k) and
// the item side V (nb x k), so the dense reconstruction is one product with
// a short contraction:
//   out[r, c] = mu + sum_{j < k} P[r, j] V[c, j]     (mb x nb, row-major).
// In the library's storage the Gram side's factor is F_s (s x kp) and the
// other side's F_L (L x kp), both row-major with the k values of a row
// contiguous (K-major, as the MMA wants both operands); P is F_s when the
// Gram side is the users, else F_L.
//
// The contraction is at most 56 long, so the kernel is bound by writing out
// (4 bytes per cell against 2k flops), and what decides its speed is how the
// accumulators reach memory:
//   * A thread of tcgen05.ld holds one lane of tensor memory, so the tile is
//     computed transposed: V's rows are the MMA's M side (128 lanes: columns
//     of out) and P's rows its N side. A warp's 32 lanes then hold 32
//     consecutive columns of one row in every register, and each register
//     goes out as one 128-byte store, with no pass through shared memory.
//   * A row of an odd number of floats starts anywhere in a 128-byte line, and
//     stores that straddle lines cost about twice (60,013 x 4,001 against
//     4,000 columns, the loads left out: 0.33 against 0.18 ms). Row r starts
//     (r nb) mod 32 floats into a line, the same for all rows of one residue
//     modulo G = 32 / gcd(nb, 32). So a strip is up to 128 rows r, r + G,
//     r + 2 G, ... of one residue, and its tiles start that many columns
//     early: every store of the strip covers one whole line. A block of
//     fewer than kClassRows rows per residue takes G = 1 instead: its strips
//     would be mostly empty.
// 60,013 x 4,001 at k = 40: 0.20 ms (0.48 ms with the tile as rows of
// tensor memory, one shared-memory buffer and twelve writing warps; 0.14 ms
// at the measured copy bandwidth). Tried and slower: the lanes' values rotated
// to whole lines by shuffles (0.29 ms, 13 instructions a row), and the tile
// staged in shared memory and written by one bulk copy a row (0.29 ms).
//
// Persistent: one CTA per SM walks a contiguous run of 128 x 128 output tiles
// (strip by strip, so consecutive tiles share their rows of P):
//   * warps 0-7 load: the strip's rows of P when the strip changes and the
//     tile's 128 rows of V (kp floats each, two threads a row, the next tile's
//     in flight while this one's buffer is waited for), split every value x
//     into hi = x rounded to 10 mantissa bits and lo = x - hi, and write both
//     into shared memory in the 128-byte-swizzled K-major layout (two
//     32-float atoms along K, zeros past kp and past the block's edge);
//   * warp 8 issues, per K = 8 slice, the products P_hi V_hi, P_hi V_lo and
//     P_lo V_hi (kind::tf32, M = N = 128) into one of two tensor-memory
//     accumulators: the dropped lo x lo term is below 2^-21 relative, as in
//     the panel products;
//   * warps 9-24 write: warp w takes tensor-memory lanes 32 (w mod 4) .. + 31
//     and 32 of the tile's rows, frees the accumulator once it has it in
//     registers, adds mu and stores.
// V rows and accumulators are double-buffered, so the next tile's loads and
// MMAs run while the last one is written. Every wait is an mbarrier wait with
// a bound; a timeout sets kErrTimeout and every group stops.
#include "kernels.h"
#include "tc_ptx.cuh"

namespace bsvd {

namespace {

constexpr int RT = 128;                       // tile rows (MMA N)
constexpr int CT = 128;                       // tile columns (MMA M)
constexpr int RK = 64;                        // K padded to two swizzle atoms
constexpr int kRLoaders = 8;                  // warps 0-7
constexpr int kRMma = kRLoaders;              // warp 8
constexpr int kRWriters = 16;                 // warps 9-24
constexpr int kRThreads = 32 * (kRLoaders + 1 + kRWriters);
constexpr uint32_t kRSpin = 1u << 22;         // mbarrier polls before giving up
constexpr int ATOM = 128 * 128;               // 16 KiB: 128 rows x 32 floats
constexpr int PART = 2 * ATOM;                // one part of P or V, K = 64
constexpr int WR = 32;                        // rows per writing warp
static_assert(kRWriters * WR * 32 == RT * CT, "a tile");
constexpr int V_OFF = 2 * PART;               // V buffers (hi, lo) x 2
constexpr int C_OFF = V_OFF + 4 * PART;       // the control block
// 3,000 x 4,001 (93 rows a residue): 41 us by residue, 39 with G = 1; 9,000 x
// 4,001 (281): 66 and 65; 20,000 x 2,002 (1,250): 54 and 66; 60,013 x 1,777
// (1,875): 130 and 152.
constexpr int kClassRows = 512;

struct RCtrl {
  uint64_t mma[2];      // the tile's MMAs completed (buffer b)
  uint64_t tfree[2];    // the writers read accumulator b (16 warps)
  uint64_t loaded[2];   // V (and P) rows of buffer b written (8 warps)
  uint32_t tmem;
  int abort;
};
constexpr int kRSmem = C_OFF + (int)sizeof(RCtrl) + 1024;

__device__ __forceinline__ uint32_t swz(int r, int c) {
  return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4));
}

__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Every other 16-byte chunk (from chunk `odd` on) of one row of a kp-column
// factor: zeros past kp, and all of it when !valid. All loads are issued
// before any is used.
struct HalfRow {
  float4 v[RK / 8];
  __device__ __forceinline__ void load(const float *src, bool valid, int kp,
                                       int odd) {
#pragma unroll
    for (int i = 0; i < RK / 8; ++i) {
      const int q = 2 * i + odd;
      v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (valid && 4 * q < kp)
        v[i] = __ldg(reinterpret_cast<const float4 *>(src + 4 * q));
    }
  }
  // Its hi and lo parts into row r of an operand: 16-byte chunk q (4 floats
  // of K) goes to atom q / 8, chunk q mod 8 of the swizzled row. Only the
  // K = 8 slices in use are written.
  __device__ __forceinline__ void put(unsigned char *part, int r, int kp,
                                      int odd) const {
#pragma unroll
    for (int i = 0; i < RK / 8; ++i) {
      if (8 * i >= kp) continue;
      const int q = 2 * i + odd;
      const float4 x = v[i];
      const float4 h = make_float4(tf32_hi(x.x), tf32_hi(x.y), tf32_hi(x.z),
                                   tf32_hi(x.w));
      const float4 l = make_float4(__fsub_rn(x.x, h.x), __fsub_rn(x.y, h.y),
                                   __fsub_rn(x.z, h.z), __fsub_rn(x.w, h.w));
      const uint32_t off = (uint32_t)((q >> 3) * ATOM) + swz(r, q & 7);
      *reinterpret_cast<float4 *>(part + off) = h;
      *reinterpret_cast<float4 *>(part + PART + off) = l;
    }
  }
};

// The tiles of a block. Strip number t: rows first + G k of the residue
// first, from k0 on; its tiles are 128 columns from -shift on.
struct Tiling {
  int64_t mb, nb, strips, nct;
  int G, per_class, odd;     // odd: out's own offset in a line, in floats
  __host__ __device__ Tiling(int64_t mb_, int64_t nb_, const float *out)
      : mb(mb_), nb(nb_) {
    G = 32;
    while (G > 1 && (nb * (G / 2)) % 32 == 0) G /= 2;
    if (mb < (int64_t)kClassRows * G) G = 1;
    odd = (int)((reinterpret_cast<uintptr_t>(out) >> 2) & 31);
    const int64_t rows = (mb + G - 1) / G;       // of the largest residue
    per_class = (int)((rows + RT - 1) / RT);
    strips = (int64_t)G * per_class;
    nct = (nb + (G > 1 || nb % 32 == 0 ? 31 : 0) + CT - 1) / CT;
  }
  __device__ __forceinline__ int64_t row(int64_t strip, int k) const {
    return strip / per_class + (int64_t)G * (strip % per_class * RT + k);
  }
  __device__ __forceinline__ int shift(int64_t strip) const {
    if (G == 1 && nb % 32 != 0) return 0;
    return (int)((odd + strip / per_class * nb) & 31);
  }
};

__global__ void __launch_bounds__(kRThreads, 1)
k_reconstruct_tc(const BlockMeta *__restrict__ meta, int32_t b,
                 const float *__restrict__ Fs, const float *__restrict__ FL,
                 int32_t kp, const float *__restrict__ mean,
                 float *__restrict__ out, int32_t *err) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char *base = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char *p_op = base;                   // P: hi, then lo
  auto v_op = [&](int buf) { return base + V_OFF + buf * 2 * PART; };
  RCtrl &ct = *reinterpret_cast<RCtrl *>(base + C_OFF);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const BlockMeta bm = meta[b];
  // P (rows r of out) and V (columns c) in the library's storage
  const float *P = bm.trans ? FL + bm.fl_off : Fs + bm.fs_off;
  const float *V = bm.trans ? Fs + bm.fs_off : FL + bm.fl_off;
  const Tiling tl(bm.mb, bm.nb, out);
  const int64_t nct = tl.nct, units = tl.strips * nct;
  const int64_t per = (units + gridDim.x - 1) / gridDim.x;
  const int64_t u0 = (int64_t)blockIdx.x * per;
  const int64_t u1 = u0 + per < units ? u0 + per : units;
  const int ntile = u1 > u0 ? (int)(u1 - u0) : 0;

  if (warp == 0) tc::tmem_alloc(&ct.tmem, 2 * RT);
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&ct.mma[i], 1);
      tc::mbar_init(&ct.tfree[i], kRWriters);
      tc::mbar_init(&ct.loaded[i], kRLoaders);
    }
    ct.abort = 0;
    tc::mbar_init_fence();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t taddr = ct.tmem;
  volatile int *abort_flag = &ct.abort;
  auto give_up = [&]() {
    if (lane == 0) atomicOr(err, kErrTimeout);
    ct.abort = 1;
  };

  if (warp < kRLoaders) {
    // loading warps: thread t takes half of row t mod 128 of P and of V's
    // tile; the next tile's loads are in flight while this one's buffer is
    // waited for
    const int t = threadIdx.x & 127, odd = threadIdx.x >> 7;
    HalfRow row;
    auto load_v = [&](int j) {
      const int64_t su = (u0 + j) / nct;
      const int64_t c = (u0 + j) % nct * CT - tl.shift(su) + t;
      row.load(V + c * kp, c >= 0 && c < bm.nb, kp, odd);
    };
    int64_t strip = -1;
    if (ntile > 0) load_v(0);
    for (int j = 0; j < ntile; ++j) {
      const int64_t su = (u0 + j) / nct;
      const int buf = j & 1;
      const uint32_t par = (j >> 1) & 1;
      // buffer j mod 2 is free once the MMAs of tile j - 2 completed
      bool ok = tc::mbar_wait(&ct.mma[buf], par ^ 1, kRSpin);
      // P is rewritten for a new strip once the last MMAs that read it
      // (tile j - 1's) completed
      if (ok && su != strip && j > 0)
        ok = tc::mbar_wait(&ct.mma[(j - 1) & 1], ((j - 1) >> 1) & 1, kRSpin);
      ok = __all_sync(0xffffffffu, ok && !*abort_flag);
      if (!ok) {
        give_up();
        break;
      }
      row.put(v_op(buf), t, kp, odd);
      if (su != strip) {
        const int64_t r = tl.row(su, t);
        row.load(P + r * kp, r < bm.mb, kp, odd);
        row.put(p_op, t, kp, odd);
        strip = su;
      }
      fence_async_smem();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&ct.loaded[buf]);
      if (j + 1 < ntile) load_v(j + 1);
    }
  } else if (warp == kRMma) {
    const int nks = (kp + 7) / 8;                 // K = 8 slices in use
    constexpr uint32_t idesc = tc::idesc_tf32_f32(CT, RT);
    for (int j = 0; j < ntile; ++j) {
      const int buf = j & 1;
      const uint32_t par = (j >> 1) & 1;
      // the operands are there, and the writers have read tile j - 2's
      // accumulator
      const bool ok = __all_sync(
          0xffffffffu, tc::mbar_wait(&ct.loaded[buf], par, kRSpin) &&
                           tc::mbar_wait(&ct.tfree[buf], par ^ 1, kRSpin) &&
                           !*abort_flag);
      if (!ok) {
        give_up();
        break;
      }
      tc::fence_after_sync();
      if (tc::elect_one()) {
        const uint32_t d = taddr + (uint32_t)(buf * RT);
        for (int kk = 0; kk < nks; ++kk) {
          const uint32_t o = (uint32_t)((kk >> 2) * ATOM);
          const uint32_t k2 = 2 * (kk & 3);
          const uint32_t pa = tc::smem_u32(p_op + o);
          const uint32_t va = tc::smem_u32(v_op(buf) + o);
          const uint64_t ph = tc::sdesc_kmajor_sw128(pa) + k2;
          const uint64_t pl = tc::sdesc_kmajor_sw128(pa + PART) + k2;
          const uint64_t vh = tc::sdesc_kmajor_sw128(va) + k2;
          const uint64_t vl = tc::sdesc_kmajor_sw128(va + PART) + k2;
          tc::mma_tf32(d, vh, ph, idesc, kk > 0 ? 1u : 0u);
          tc::mma_tf32(d, vl, ph, idesc, 1u);
          tc::mma_tf32(d, vh, pl, idesc, 1u);
        }
        tc::mma_commit(&ct.mma[buf]);
      }
      __syncwarp();
    }
  } else {
    const float mu = mean ? mean[b] : 0.f;
    const int q = warp & 3;                       // lane quarter
    const int h = (warp - kRMma - 1) >> 2;        // which WR rows
    const uint32_t ta0 = taddr + ((uint32_t)(q * 32) << 16) + (uint32_t)(h * WR);
    const int64_t nb = bm.nb, stride = nb * tl.G;
    for (int j = 0; j < ntile; ++j) {
      const int64_t su = (u0 + j) / nct;
      const int64_t c = (u0 + j) % nct * CT - tl.shift(su) + q * 32 + lane;
      const int64_t r0 = tl.row(su, h * WR);
      const int buf = j & 1;
      const bool ok = __all_sync(
          0xffffffffu,
          tc::mbar_wait(&ct.mma[buf], (j >> 1) & 1, kRSpin) && !*abort_flag);
      if (!ok) {
        give_up();
        break;
      }
      tc::fence_after_sync();
      float v[WR];
      tc::tmem_ld32(ta0 + (uint32_t)(buf * RT), v);
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&ct.tfree[buf]);
      if (c < 0 || c >= nb) continue;
      float *dst = out + r0 * nb + c;
      // the strip's rows from r0 on that the block has
      const int64_t left = (bm.mb - r0 + tl.G - 1) / tl.G;
      if (left >= WR) {
#pragma unroll
        for (int r = 0; r < WR; ++r, dst += stride)
          *dst = mu + v[r];
      } else {
#pragma unroll
        for (int r = 0; r < WR; ++r, dst += stride)
          if (r < left) *dst = mu + v[r];
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (threadIdx.x == 0 && ct.abort) {
    // MMAs issued but never seen to finish: wait (bounded) before freeing
    for (int i = 0; i < 2; ++i) {
      tc::mbar_wait(&ct.mma[i], 0, kRSpin);
      tc::mbar_wait(&ct.mma[i], 1, kRSpin);
    }
  }
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(taddr, 2 * RT);
}

}  // namespace

cudaError_t launch_reconstruct(const BlockMeta *meta, const BlockMeta &host,
                               int32_t b, const float *Fs, const float *FL,
                               int32_t kp, const float *mean, float *out,
                               int32_t *err, cudaStream_t st) {
  if (host.mb <= 0 || host.nb <= 0) return cudaSuccess;
  if (kp <= 0 || kp > RK || kp % 4 != 0) return cudaErrorInvalidValue;
  int dev = 0, nsm = 152;
  if (cudaGetDevice(&dev) == cudaSuccess)
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const Tiling tl(host.mb, host.nb, out);
  const int64_t units = tl.strips * tl.nct;
  const int grid = (int)(units < nsm ? units : nsm);
  static_assert(kRSmem <= 227 * 1024, "shared memory");
  cudaError_t e = cudaFuncSetAttribute(
      k_reconstruct_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kRSmem);
  if (e != cudaSuccess) return e;
  k_reconstruct_tc<<<grid, kRThreads, kRSmem, st>>>(meta, b, Fs, FL, kp, mean,
                                                   out, err);
  return cudaGetLastError();
}

}  // namespace bsvd
