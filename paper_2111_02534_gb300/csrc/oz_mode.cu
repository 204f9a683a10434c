// One mode product of the 2D H-apply (Eq. tensor_op2D) in one kernel: FP64 wave functions in,
// FP64 result out, the digit products of the Ozaki scheme (see ozaki_tc.cu for the scheme and
// its error) on tcgen05 in between, for modes of up to 64 points.
//
//   out[m][j] (+)= sum_i psi[m][i] K[j][i],   m a fiber of the mode, i, j its points
//
// What bounds it: instruction issue.  An element costs about 30 integer and packed FP16
// instructions to cut into digits and an output about 60 to put together from its eight
// levels, 0.38 ms per 8-vector apply at 48^4 if every scheduler issued every cycle, against
// 0.3 ms of tensor time and 0.6 ms for the 24 bytes per element and mode that have to move
// (psi read, out read and written).  A split kernel that writes the digits to memory and a
// product kernel that reads them back move 54 bytes.  Measured, 8 vectors at 48^4: 3.62 ms with
// the two kernels, 1.98 ms with this one.
//
// One CTA per SM works through tiles of 128 fibers, every stage of several tiles in flight:
//   warps 0-7   load psi (two threads per fiber, half of its points each, in registers), take
//               the fiber's exponent and write the seven digit slices straight into the
//               operand layout in shared memory (two stages; one for more than 48 points);
//   warps 8-15  drain the accumulators, recombine the levels and store;
//   warp 16     issues the MMAs.
// The output columns are taken 16 at a time, eight levels x 16 columns = 128 TMEM columns, so
// that four of these sub-tiles fit in tensor memory and the epilogue of one runs under the MMAs
// of the next.  A narrow MMA costs ~45 cycles whatever its width (measured), and a product of
// one digit pair is only 16 wide; but the levels of one sub-tile lie side by side, so A's slice
// i times B's slices 0 .. 7 - i (stacked as rows) is ONE product of width 16 (8 - i) whose
// columns land on the levels i .. 7: 7 MMAs per 16 points of K instead of 35.
//
// Operand layout: no swizzle, core matrices of 8 rows x 16 bytes, rows in order (128 bytes
// apart per 8 rows), the 16-byte columns of K 2048 bytes apart (128 rows).  A warp writing the
// same 16-byte column of consecutive rows writes consecutive addresses: no bank conflicts, no
// padding of K beyond a multiple of 16.
//
// Digits: base 256, seven of a 55-bit integer for psi, eight of a 62-bit one for K, in FP16
// (integers up to 2048 are exact).  q + 128 (1 + 256 + .. ) has the digits plus 128 as its
// bytes, so a digit of two neighbours is one byte permute, one OR with FP16 1024 (whose unit is
// 1) and one packed subtraction of 1152.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>

#include "oz_mode.cuh"
#include "ozaki_tc.cuh"
#include "pdl.cuh"
#include "split_digits.cuh"
#include "tps_internal.h"

namespace tps {
namespace ozm {
namespace {

constexpr int kSA = 7, kSB = 8, kL = 8;  // digits of psi, of K, levels kept (i + j <= 7)
constexpr int kRows = 128;               // fibers per tile
constexpr int kCols = 16;                // output columns per sub-tile
constexpr int kAcc = 4;                  // sub-tiles in tensor memory
constexpr int kProdWarps = 8, kEpiWarps = 8, kMmaWarp = kProdWarps + kEpiWarps;
constexpr int kThreads = 32 * (kMmaWarp + 1);
constexpr int kExpRing = 8;              // tiles whose fiber exponents are kept
constexpr uint32_t kChunk = kRows * 16;  // bytes of one 16-byte column of K
constexpr uint32_t kTmemCols = 512;
static_assert(kAcc * kL * kCols <= (int)kTmemCols, "sub-tiles must fit in tensor memory");
static_assert(kSB * kCols == kRows, "A and B images share one layout");

template <int KC>  // K in units of 16 points; also the sub-tiles of 16 output columns
struct Cfg {
  static constexpr uint32_t kSlice = 2 * KC * kChunk;          // one digit slice, 128 rows
  static constexpr uint32_t kAStage = kSA * kSlice;
  static constexpr uint32_t kB = KC * kSlice;                  // 8 slices x 16 rows per sub-tile
  static constexpr int kStages = KC <= 3 ? 2 : 1;
  static constexpr uint32_t kSmem =
      1024 + kStages * kAStage + kB + kExpRing * kRows * 4 + KC * kCols * 4 + 256;
};

struct Args {
  const double *psi, *V, *theta_dev;
  double *out;
  long long N;
  unsigned M, n, sigma;
  const uint4 *image;
  const unsigned *eK;
  double theta0;
  int *err;
  long long tiles;
  unsigned tm;   // tiles per vector
  int store, vec;  // vec: sigma == 1 and 32-byte accesses are aligned
};

// Shared-memory matrix descriptor, K-major, no swizzle: bits 0-13 start address >> 4, bits
// 16-29 offset between core matrices along K >> 4, bits 32-45 offset between groups of 8 rows
// >> 4, bits 46-48 fixed 0b001, bits 61-63 layout 0.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(kChunk >> 4) << 16) |
         ((uint64_t)(128 >> 4) << 32) | ((uint64_t)1 << 46);
}

// Instruction descriptor of kind::f16 with FP16 A and B (formats 0), FP32 accumulator.
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void ld4(const double *p, double (&v)[4]) {
  asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
               : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3])
               : "l"(p));
}
__device__ __forceinline__ void st4(double *p, const double (&v)[4]) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(v[0]), "d"(v[1]),
               "d"(v[2]), "d"(v[3])
               : "memory");
}

// round(x 2^(55 - E)) + 128 (1 + 2^8 + .. + 2^48), E = raw_max - 1022 (|x| < 2^E): bytes 0 .. 5
// are the lower six digits plus 128, the bits from 48 on the top digit plus 128 (0 .. 256).
// Subnormals count as zero.
__device__ __forceinline__ uint64_t biased55(double x, unsigned raw_max) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned ex = (hi >> 20) & 0x7FFu;
  const unsigned sh = ex ? min(raw_max - ex, 63u) : 63u;
  // the mantissa times 8 (56 bits), shifted right, rounded to nearest (half away from zero)
  const uint64_t m =
      ((uint64_t)((((hi & 0xFFFFFu) | 0x100000u) << 3) | (lo >> 29)) << 32) | (lo << 3);
  const uint64_t a = ((m >> sh) + 1) >> 1;
  const uint64_t bias = 0x0080808080808080ULL;
  return (hi >> 31) ? bias - a : bias + a;
}

// The seven digits of two neighbouring elements as FP16 pairs, most significant first.
__device__ __forceinline__ void digit_pairs(uint64_t u0, uint64_t u1, uint32_t (&d)[kSA]) {
  const uint32_t l0 = (uint32_t)u0, h0 = (uint32_t)(u0 >> 32);
  const uint32_t l1 = (uint32_t)u1, h1 = (uint32_t)(u1 >> 32);
  const __half2 off = __half2half2(__ushort_as_half(0x6480));  // 1152
  uint32_t w[kSA];
  w[0] = __byte_perm(h0, h1, 0x7632) | 0x64006400u;
  w[1] = (__byte_perm(h0, h1, 0x5511) & 0x00FF00FFu) | 0x64006400u;
  w[2] = (__byte_perm(h0, h1, 0x5410) & 0x00FF00FFu) | 0x64006400u;
  w[3] = (__byte_perm(l0, l1, 0x7733) & 0x00FF00FFu) | 0x64006400u;
  w[4] = (__byte_perm(l0, l1, 0x7632) & 0x00FF00FFu) | 0x64006400u;
  w[5] = (__byte_perm(l0, l1, 0x5511) & 0x00FF00FFu) | 0x64006400u;
  w[6] = (__byte_perm(l0, l1, 0x5410) & 0x00FF00FFu) | 0x64006400u;
#pragma unroll
  for (int i = 0; i < kSA; ++i) {
    const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&w[i]), off);
    d[i] = *reinterpret_cast<const uint32_t *>(&h);
  }
}

// The digit image of K (n x n, row-major): for every sub-tile of 16 rows of K, 128 rows (digit
// j of row c at 16 j + c) x 16 KC points in the operand layout; zeros beyond n.
__global__ void k_build_image(const double *__restrict__ K, int n, int kc,
                              uint4 *__restrict__ image, unsigned *__restrict__ eK) {
  extern __shared__ unsigned ex[];  // exponents of the n rows
  for (int r = threadIdx.x; r < n; r += blockDim.x) {
    unsigned e = 0;
    for (int i = 0; i < n; ++i) {
      const unsigned t = b256::raw_exp(K[(long long)r * n + i]);
      e = t > e ? t : e;
    }
    ex[r] = e;
    if (blockIdx.x == 0) eK[r] = e;
  }
  __syncthreads();
  const int total = kc * 2 * kc * kRows;  // 16-byte pieces: sub-tile, 16-byte column, row
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < total; p += gridDim.x * blockDim.x) {
    const int row = p % kRows, col = (p / kRows) % (2 * kc), s = p / (kRows * 2 * kc);
    const int j = row / kCols, r = s * kCols + row % kCols;
    __half h[8];
    for (int e = 0; e < 8; ++e) {
      const int i = col * 8 + e;
      int d = 0;
      if (r < n && i < n && ex[r]) {
        // digit j of the 62-bit integer of K[r][i]
        const unsigned long long x =
            (unsigned long long)__double_as_longlong(K[(long long)r * n + i]);
        const int raw = (int)((x >> 52) & 0x7FF);
        long long q = 0;
        if (raw) {
          const long long mant = (long long)((x & ((1ULL << 52) - 1)) | (1ULL << 52));
          const int sh = raw - (int)ex[r] + 9;
          if (sh >= 0)
            q = mant << sh;
          else if (sh > -63)
            q = (mant + (1LL << (-sh - 1))) >> (-sh);
          if (x >> 63) q = -q;
        }
        const unsigned long long u = (unsigned long long)q + 0x0080808080808080ULL;
        d = j == 0 ? (int)((long long)u >> 56) : (int)((u >> (8 * (7 - j))) & 0xFF) - 128;
      }
      h[e] = __int2half_rn(d);
    }
    image[p] = *reinterpret_cast<const uint4 *>(h);
  }
}

template <int KC>
__global__ void __launch_bounds__(kThreads, 1) k_mode_product(const __grid_constant__ Args g) {
  using C = Cfg<KC>;
  extern __shared__ uint8_t raw_smem[];
  __shared__ int abort_flag;
  uint8_t *base = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(raw_smem) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t *sA = base, *sB = base + C::kStages * C::kAStage;
  unsigned *sExp = reinterpret_cast<unsigned *>(sB + C::kB);  // [kExpRing][kRows]
  int *sEn = reinterpret_cast<int *>(sExp + kExpRing * kRows);
  uint64_t *bars = reinterpret_cast<uint64_t *>(sEn + KC * kCols);
  uint64_t *fullA = bars, *emptyA = bars + 2, *accum = bars + 4, *accfree = accum + kAcc;
  uint64_t *drained = accfree + kAcc;
  uint32_t *holder = reinterpret_cast<uint32_t *>(drained + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    pdl_trigger();
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&fullA[i], kProdWarps);
      tc::mbar_init(&emptyA[i], 1);
    }
    for (int i = 0; i < kAcc; ++i) {
      tc::mbar_init(&accum[i], 1);
      tc::mbar_init(&accfree[i], kEpiWarps);
    }
    tc::mbar_init(drained, 1);
    abort_flag = 0;
    tc::fence_barrier_init();
  }
  if (warp == kMmaWarp) tc::tmem_alloc(holder, kTmemCols);
  {
    uint4 *dst = reinterpret_cast<uint4 *>(sB);
    for (unsigned i = threadIdx.x; i < C::kB / 16; i += kThreads) dst[i] = g.image[i];
    for (unsigned i = threadIdx.x; i < KC * kCols; i += kThreads)
      sEn[i] = i < g.n ? (int)g.eK[i] - 1022 : 0;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = *holder;
  // the operator's image above is older than the previous kernel; everything below is not
  pdl_wait();

  if (warp < kProdWarps) {
    // ---- producers: thread (fiber, half of the points)
    constexpr int PT = KC * 8;
    const unsigned fib = warp * 16 + (lane & 15), half = lane >> 4;
    const unsigned i0 = half * PT;
    int it = 0;
    for (long long t = blockIdx.x; t < g.tiles; t += gridDim.x, ++it) {
      const unsigned v = (unsigned)(t / g.tm), r = (unsigned)(t - (long long)v * g.tm);
      const unsigned m = r * kRows + fib;
      const bool valid = m < g.M;
      const double *p = g.psi + (long long)v * g.N +
                        (valid ? (long long)(m / g.sigma) * ((long long)g.n * g.sigma) +
                                     m % g.sigma
                               : 0);
      double x[PT];
      if (g.vec) {  // contiguous fibers of a multiple of four points
#pragma unroll
        for (int e = 0; e < PT; e += 4) {
          double w[4] = {0.0, 0.0, 0.0, 0.0};
          if (valid && i0 + e < g.n) ld4(p + i0 + e, w);
#pragma unroll
          for (int k = 0; k < 4; ++k) x[e + k] = w[k];
        }
      } else {
#pragma unroll
        for (int e = 0; e < PT; ++e)
          x[e] = valid && i0 + e < g.n ? p[(long long)(i0 + e) * g.sigma] : 0.0;
      }
      unsigned mx = 0;
#pragma unroll
      for (int e = 0; e < PT; ++e) mx = max(mx, (unsigned)__double2hiint(x[e]) & 0x7FF00000u);
      mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 16)) >> 20;
      const int st = it % C::kStages;
      bool ok = tc::mbar_wait(&emptyA[st], ((it / C::kStages) & 1) ^ 1, g.err, 2);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok || *((volatile int *)&abort_flag)) {
        atomicExch(&abort_flag, 1);
        break;
      }
      if (half == 0) sExp[(it % kExpRing) * kRows + fib] = mx;
      uint8_t *dst = sA + st * C::kAStage + (half * KC) * kChunk + fib * 16;
#pragma unroll
      for (int c = 0; c < KC; ++c) {
        uint32_t d[4][kSA];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          digit_pairs(biased55(x[c * 8 + 2 * k], mx), biased55(x[c * 8 + 2 * k + 1], mx), d[k]);
#pragma unroll
        for (int i = 0; i < kSA; ++i)
          *reinterpret_cast<uint4 *>(dst + i * C::kSlice + c * kChunk) =
              make_uint4(d[0][i], d[1][i], d[2][i], d[3][i]);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&fullA[st]);
    }
  } else if (warp < kMmaWarp) {
    // ---- epilogue: TMEM lanes 32 (warp % 4) .. + 31 (fibers), 8 of a sub-tile's 16 columns
    const int quarter = warp & 3, half = (warp - kProdWarps) >> 2;
    const unsigned row = 32 * quarter + lane;
    const uint32_t trow = tmem + ((uint32_t)(32 * quarter) << 16) + half * 8;
    int it = 0;
    unsigned u = 0;  // sub-tile counter
    bool alive = true;
    for (long long t = blockIdx.x; t < g.tiles && alive; t += gridDim.x, ++it) {
      const unsigned v = (unsigned)(t / g.tm), r = (unsigned)(t - (long long)v * g.tm);
      const unsigned m = r * kRows + row;
      const bool valid = m < g.M;
      const long long mb = valid ? (long long)(m / g.sigma) * ((long long)g.n * g.sigma) +
                                       m % g.sigma
                                 : 0;
      double *o = g.out + (long long)v * g.N + mb;
      for (int s = 0; s < KC; ++s, ++u) {
        const unsigned st = u % kAcc;
        bool ok = tc::mbar_wait(&accum[st], (u / kAcc) & 1, g.err, 5);
        ok = __all_sync(0xffffffffu, ok);
        const int aborted = __shfl_sync(0xffffffffu, *((volatile int *)&abort_flag), 0);
        if (!ok || aborted) {
          alive = false;
          break;
        }
        tc::tc_fence_after();
        const int Em = (int)sExp[(it % kExpRing) * kRows + row] - 1022;
        double val[8];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t rr[kL][4];
#pragma unroll
          for (int l = 0; l < kL; ++l)
            tc::tmem_ld_x4(trow + st * (kL * kCols) + l * kCols + h * 4, rr[l]);
          tc::tmem_ld_wait();
          if (h == 1) {  // the accumulators are read: the MMAs may overwrite them
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&accfree[st]);
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            int d[kL];
#pragma unroll
            for (int l = 0; l < kL; ++l) d[l] = __float2int_rn(__uint_as_float(rr[l][q]));
            const long long hi = (((long long)d[0] * 256 + d[1]) * 256 + d[2]) * 256 + d[3];
            const long long lo = (((long long)d[4] * 256 + d[5]) * 256 + d[6]) * 256 + d[7];
            val[h * 4 + q] =
                b256::combine(hi, lo, Em + sEn[s * kCols + half * 8 + h * 4 + q] + 1);
          }
        }
        const unsigned c0 = s * kCols + half * 8;
        if (!valid) continue;
        if (g.store) {
          const double th = g.theta_dev ? g.theta_dev[v] : g.theta0;
          const double *pp = g.psi + (long long)v * g.N + mb, *vp = g.V + mb;
          if (g.vec) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const unsigned c = c0 + 4 * h;
              if (c < g.n) {
                double a[4], b[4], w[4];
                ld4(vp + c, a);
                ld4(pp + c, b);
#pragma unroll
                for (int q = 0; q < 4; ++q) w[q] = fma(a[q] - th, b[q], val[h * 4 + q]);
                st4(o + c, w);
              }
            }
          } else {
#pragma unroll
            for (int q = 0; q < 8; ++q)
              if (c0 + q < g.n) {
                const long long i = (long long)(c0 + q) * g.sigma;
                o[i] = fma(vp[i] - th, pp[i], val[q]);
              }
          }
        } else {
          // each element belongs to one thread of one CTA per launch: the sum of the modes
          // is taken in launch order
#pragma unroll
          for (int q = 0; q < 8; ++q)
            if (c0 + q < g.n) atomicAdd(o + (long long)(c0 + q) * g.sigma, val[q]);
        }
      }
    }
  } else if (lane == 0) {
    // ---- MMA issuer
    bool ok = true;
    int it = 0;
    unsigned u = 0;
    const uint32_t a0 = tc::smem_addr(sA), b0 = tc::smem_addr(sB);
    for (long long t = blockIdx.x; t < g.tiles && ok; t += gridDim.x, ++it) {
      const int st = it % C::kStages;
      if (!tc::mbar_wait(&fullA[st], (it / C::kStages) & 1, g.err, 4)) {
        ok = false;
        break;
      }
      const uint64_t adesc = smem_desc(a0 + st * C::kAStage);
      for (int s = 0; s < KC; ++s, ++u) {
        const unsigned ac = u % kAcc;
        if (!tc::mbar_wait(&accfree[ac], ((u / kAcc) & 1) ^ 1, g.err, 6)) {
          ok = false;
          break;
        }
        tc::tc_fence_after();
        const uint64_t bdesc = smem_desc(b0 + s * C::kSlice);
        const uint32_t d = tmem + ac * (kL * kCols);
#pragma unroll
        for (int kk = 0; kk < KC; ++kk)
#pragma unroll
          for (int i = 0; i < kSA; ++i)  // levels i .. 7 at once
            tc::mma_bf16(d + i * kCols, adesc + (uint64_t)((i * C::kSlice + 2 * kk * kChunk) >> 4),
                         bdesc + (uint64_t)((2 * kk * kChunk) >> 4),
                         idesc_f16(kRows, kCols * (kL - i)), (kk > 0 || i > 0) ? 1u : 0u);
        tc::mma_commit(&accum[ac]);
      }
      if (ok) tc::mma_commit(&emptyA[st]);
    }
    if (!ok) atomicExch(&abort_flag, 1);
    // nothing of this thread's is in flight when the tensor memory is freed
    tc::mma_commit(drained);
    tc::mbar_wait(drained, 0, g.err, 7);
  }
  __syncwarp();
  tc::tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) tc::tmem_dealloc(tmem, kTmemCols);
}

template <int KC>
cudaError_t launch_kc(const Args &g, cudaStream_t s) {
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  std::call_once(once, [] {
    attr = cudaFuncSetAttribute(k_mode_product<KC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)Cfg<KC>::kSmem);
  });
  if (attr != cudaSuccess) return attr;
  const unsigned grid = (unsigned)(g.tiles < 152 ? g.tiles : 152);
  count_launch();
  const cudaError_t e = launch_pdl(k_mode_product<KC>, dim3(grid), dim3(kThreads),
                                   Cfg<KC>::kSmem, s, g);
  return e != cudaSuccess ? e : cudaGetLastError();
}

int units(int n) { return (n + 15) / 16; }

}  // namespace

size_t image_bytes(int n) {
  const size_t kc = units(n);
  return kc * 2 * kc * kChunk;
}

void launch_build_image(const double *K, int n, uint4 *image, unsigned *eK, cudaStream_t s) {
  count_launch();
  k_build_image<<<16, 256, n * sizeof(unsigned), s>>>(K, n, units(n), image, eK);
}

cudaError_t launch_mode_product(const ModeArgs &a, cudaStream_t s) {
  if (a.n < 1 || a.n > kMaxModePoints || a.nvec < 1) return cudaErrorInvalidValue;
  const long long M = a.N / a.n;
  if (M > 0x7FFFFFFFLL) return cudaErrorInvalidValue;
  Args g = {};
  g.psi = a.psi;
  g.V = a.V;
  g.theta_dev = a.theta_dev;
  g.out = a.out;
  g.N = a.N;
  g.M = (unsigned)M;
  g.n = (unsigned)a.n;
  g.sigma = (unsigned)a.sigma;
  g.image = a.image;
  g.eK = a.eK;
  g.theta0 = a.theta0;
  g.err = a.err;
  g.tm = (unsigned)((M + kRows - 1) / kRows);
  g.tiles = (long long)g.tm * a.nvec;
  g.store = a.store ? 1 : 0;
  const uintptr_t al = reinterpret_cast<uintptr_t>(a.psi) | reinterpret_cast<uintptr_t>(a.out) |
                       reinterpret_cast<uintptr_t>(a.V);
  g.vec = a.sigma == 1 && a.n % 4 == 0 && (al & 31) == 0;
  switch (units(a.n)) {
    case 1: return launch_kc<1>(g, s);
    case 2: return launch_kc<2>(g, s);
    case 3: return launch_kc<3>(g, s);
    default: return launch_kc<4>(g, s);
  }
}

}  // namespace ozm
}  // namespace tps
