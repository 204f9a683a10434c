// One mode product of the 2D H-apply (Eq. tensor_op2D) in one kernel: FP64 wave functions in,
// FP64 result out, the digit products of the Ozaki scheme (see ozaki_tc.cu for the scheme and
// its error) on tcgen05 in between, for modes of up to 64 points.
//
//   out[m][j] (+)= sum_i psi[m][i] K[j][i],   m a fiber of the mode, i, j its points
//
// What bounds it: the integer pipe.  An output costs about 124 instructions of a lane in all (118
// where it is stored), most of them to cut an element into digits and to put an output together
// from its eight levels; the ALU (16 lanes per cycle and scheduler) is 56 % busy, issue 61 %, and
// the 24 bytes per element and mode that have to move (psi read, out read and written) take 0.6 of
// the time at the copy rate.  (A split kernel that writes the digits to memory and a product kernel
// that reads them back move 54 bytes.)  Measured at 48^4 for 3 vectors: 94 us for each of y1, x2 and
// x1, 107 for y2, 64 for the potential term; a whole apply of 8 vectors 1.13 ms, 3.63 with the split
// and product kernels.
//
// One CTA per SM works through tiles of 128 fibers, every stage of several tiles in flight
// (warps for a mode of 33 to 48 points):
//   warps 0-11   load psi (a warp takes 16 points of 32 fibers, in registers), agree on the
//                fibers' exponents and write the seven digit slices straight into the operand
//                layout in shared memory (two stages; one for more than 48 points);
//   warps 12-27  copy the operator's image, then drain the accumulators, recombine the levels
//                and store;
//   warp 28      issues the MMAs.
// (Eight producer and eight epilogue warps, with twice the registers, took 15 % more.)
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
// Digits (split_digits.cuh): base 256 in FP16, seven of a 55-bit integer for psi, eight of a
// 62-bit one for K.
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
  static constexpr int kProdWarps = 4 * KC;           // a unit of 16 points of 32 fibers each
  static constexpr int kEpiWarps = KC <= 3 ? 16 : 8;  // as many as 1024 threads leave
  static constexpr int kEpiCols = 4 * kCols / kEpiWarps;  // columns of a sub-tile per warp
  static constexpr int kMmaWarp = kProdWarps + kEpiWarps;
  static constexpr int kThreads = 32 * (kMmaWarp + 1);
  static constexpr uint32_t kSmem = 1024 + kStages * kAStage + kB +
                                    (kExpRing + 2 * KC) * kRows * 4 + KC * kCols * 4 + 256;
};

struct Args {
  const double *psi;
  double *out;
  long long N;
  unsigned M, n, sigma;
  const uint4 *image;
  const unsigned *eK;
  int *err;
  long long tiles;
  unsigned tm;   // tiles per vector
  b256::LevelWeights weights;
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

// The digit image of K (n x n, row-major): for every sub-tile of 16 rows of K, 128 rows (digit
// j of row c at 16 j + c) x 16 KC points in the operand layout; zeros beyond n.  A row's
// exponent is its absolute sum's (see level_sum).
__global__ void k_build_image(const double *__restrict__ K, int n, int kc,
                              uint4 *__restrict__ image, unsigned *__restrict__ eK) {
  extern __shared__ unsigned ex[];  // exponents of the n rows
  for (int r = threadIdx.x; r < n; r += blockDim.x) {
    double sum = 0.0;
    for (int i = 0; i < n; ++i) sum += fabs(K[(long long)r * n + i]);
    const unsigned e = b256::raw_exp(sum);
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
      const int d = r < n && i < n && ex[r] ? b256::digit62(K[(long long)r * n + i], ex[r], j) : 0;
      h[e] = __int2half_rn(d);
    }
    image[p] = *reinterpret_cast<const uint4 *>(h);
  }
}

// What the epilogue does with a product: adds it to memory, by an atomic that returns nothing
// (one term per element and launch, so the sum of the modes is taken in launch order); stores
// it; stores it, the fibers' points being contiguous and 32-byte accesses aligned.
enum Epi { kAdd = 0, kStore = 1, kStoreVec = 2 };

template <int KC, Epi EPI>
__global__ void __launch_bounds__(Cfg<KC>::kThreads, 1)
k_mode_product(const __grid_constant__ Args g) {
  using C = Cfg<KC>;
  extern __shared__ uint8_t raw_smem[];
  __shared__ int abort_flag;
  uint8_t *base = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(raw_smem) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t *sA = base, *sB = base + C::kStages * C::kAStage;
  unsigned *sExp = reinterpret_cast<unsigned *>(sB + C::kB);  // [kExpRing][kRows]
  unsigned *sMax = sExp + kExpRing * kRows;                   // [2][KC][kRows]
  int *sEn = reinterpret_cast<int *>(sMax + 2 * KC * kRows);  // [KC * kCols]
  uint64_t *bars = reinterpret_cast<uint64_t *>(sEn + KC * kCols);
  uint64_t *fullA = bars, *emptyA = bars + 2, *accum = bars + 4, *accfree = accum + kAcc;
  uint64_t *drained = accfree + kAcc, *image = drained + 1;
  uint32_t *holder = reinterpret_cast<uint32_t *>(image + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&fullA[i], C::kProdWarps);
      tc::mbar_init(&emptyA[i], 1);
    }
    for (int i = 0; i < kAcc; ++i) {
      tc::mbar_init(&accum[i], 1);
      tc::mbar_init(&accfree[i], C::kEpiWarps);
    }
    tc::mbar_init(drained, 1);
    tc::mbar_init(image, C::kEpiWarps);
    abort_flag = 0;
    tc::fence_barrier_init();
  }
  if (warp == C::kMmaWarp) tc::tmem_alloc(holder, kTmemCols);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  // only now: a dependent kernel's CTA must not take tensor memory that this one waits for
  if (threadIdx.x == 0) pdl_trigger();
  const uint32_t tmem = *holder;
  // every global access follows: the previous kernel may be the one that built the image
  pdl_wait();

  if (warp < C::kProdWarps) {
    // ---- producers: a warp takes one unit of 16 points of 32 fibers, lane = fiber
    const unsigned group = warp & 3, unit = warp >> 2;
    const unsigned i0 = unit * 16;
    // kAdd: lane = fiber, its 16 points, loads across fibers.  kStoreVec: the unit is 128
    // contiguous bytes of a fiber; a lane takes a quarter of it of four fibers (lane % 8 + 8 k),
    // so that a warp's load covers whole lines of 8 fibers
    constexpr int FL = EPI == kStoreVec ? 4 : 1;  // fibers per lane
    const unsigned f0 = group * 32 + (EPI == kStoreVec ? lane & 7 : lane);
    const unsigned piece = EPI == kStoreVec ? lane >> 3 : 0;
    int it = 0;
    for (long long t = blockIdx.x; t < g.tiles; t += gridDim.x, ++it) {
      const unsigned v = (unsigned)(t / g.tm), r = (unsigned)(t - (long long)v * g.tm);
      double x[16];
      unsigned mx[FL];
      if constexpr (EPI == kStoreVec) {  // a multiple of four points
        const unsigned i = i0 + piece * 4;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const unsigned m = r * kRows + f0 + 8 * k;
          double w[4] = {0.0, 0.0, 0.0, 0.0};
          if (m < g.M && i < g.n) ld4(g.psi + (long long)v * g.N + (long long)m * g.n + i, w);
#pragma unroll
          for (int e = 0; e < 4; ++e) x[4 * k + e] = w[e];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          unsigned e = 0;
#pragma unroll
          for (int j = 0; j < 4; ++j)
            e = max(e, (unsigned)__double2hiint(x[4 * k + j]) & 0x7FF00000u);
          e = max(e, __shfl_xor_sync(0xffffffffu, e, 8));
          mx[k] = max(e, __shfl_xor_sync(0xffffffffu, e, 16));
        }
      } else {
        const unsigned m = r * kRows + f0;
        const bool valid = m < g.M;
        const double *p = g.psi + (long long)v * g.N + (long long)i0 * g.sigma;
        if (valid) p += (long long)(m / g.sigma) * ((long long)g.n * g.sigma) + m % g.sigma;
        const int points = valid ? (int)g.n - (int)i0 : 0;  // of this thread
        unsigned e0 = 0;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          x[e] = e < points ? *p : 0.0;
          p += g.sigma;
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) e0 = max(e0, (unsigned)__double2hiint(x[e]) & 0x7FF00000u);
        mx[0] = e0;
      }
      if constexpr (KC > 1) {  // the fibers' exponents over their units
        unsigned *s = sMax + (it & 1) * (KC * kRows) + f0;
        if (piece == 0)
#pragma unroll
          for (int k = 0; k < FL; ++k) s[unit * kRows + 8 * k] = mx[k];
        asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "r"(32 * KC) : "memory");
#pragma unroll
        for (int k = 0; k < FL; ++k)
#pragma unroll
          for (int j = 0; j < KC; ++j) mx[k] = max(mx[k], s[j * kRows + 8 * k]);
      }
      const int st = it % C::kStages;
      // after a failure the units of a group still meet at their barrier: all of them go on
      // to the last tile without waiting or writing
      bool ok = !__shfl_sync(0xffffffffu, *((volatile int *)&abort_flag), 0);
      if (ok) ok = tc::mbar_wait(&emptyA[st], ((it / C::kStages) & 1) ^ 1, g.err, 2);
      if (!__all_sync(0xffffffffu, ok)) {
        atomicExch(&abort_flag, 1);
        continue;
      }
      if (unit == 0 && piece == 0)
#pragma unroll
        for (int k = 0; k < FL; ++k) sExp[(it % kExpRing) * kRows + f0 + 8 * k] = mx[k] >> 20;
      uint8_t *dst = sA + st * C::kAStage + (unit * 2) * kChunk + f0 * 16;
      if constexpr (EPI == kStoreVec) {
        dst += (piece >> 1) * kChunk + (piece & 1) * 8;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          uint32_t d[2][kSA];
#pragma unroll
          for (int j = 0; j < 2; ++j)
            b256::digit_pairs(b256::biased55(x[4 * k + 2 * j], mx[k]),
                              b256::biased55(x[4 * k + 2 * j + 1], mx[k]), d[j]);
#pragma unroll
          for (int i = 0; i < kSA; ++i)
            *reinterpret_cast<uint2 *>(dst + i * C::kSlice + 8 * k * 16) =
                make_uint2(d[0][i], d[1][i]);
        }
      } else {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t d[4][kSA];
#pragma unroll
          for (int k = 0; k < 4; ++k)
            b256::digit_pairs(b256::biased55(x[c * 8 + 2 * k], mx[0]), b256::biased55(x[c * 8 + 2 * k + 1], mx[0]),
                        d[k]);
#pragma unroll
          for (int i = 0; i < kSA; ++i)
            *reinterpret_cast<uint4 *>(dst + i * C::kSlice + c * kChunk) =
                make_uint4(d[0][i], d[1][i], d[2][i], d[3][i]);
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&fullA[st]);
    }
  } else if (warp < C::kMmaWarp) {
    // ---- epilogue: TMEM lanes 32 (warp % 4) .. + 31 (fibers), kEpiCols columns of a sub-tile
    constexpr int EC = C::kEpiCols;
    static_assert(C::kProdWarps % 4 == 0 && EC % 4 == 0, "");
    const int quarter = warp & 3, part = (warp - C::kProdWarps) >> 2;
    const unsigned row = 32 * quarter + lane;
    const uint32_t trow = tmem + ((uint32_t)(32 * quarter) << 16) + part * EC;
    {  // the operator's image, while the producers load and cut the first tile
      const unsigned first = threadIdx.x - 32 * C::kProdWarps, step = 32 * C::kEpiWarps;
      uint4 *dst = reinterpret_cast<uint4 *>(sB);
#pragma unroll 4
      for (unsigned i = first; i < C::kB / 16; i += step) dst[i] = g.image[i];
      for (unsigned i = first; i < KC * kCols; i += step)
        sEn[i] = i < g.n ? (int)g.eK[i] - 1022 : 0;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(image);
      asm volatile("bar.sync 5, %0;" ::"r"(step) : "memory");  // sEn, for these warps
    }
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
        const unsigned c0 = s * kCols + part * EC;
        bool ok = tc::mbar_wait(&accum[st], (u / kAcc) & 1, g.err, 5);
        ok = __all_sync(0xffffffffu, ok);
        const int aborted = __shfl_sync(0xffffffffu, *((volatile int *)&abort_flag), 0);
        if (!ok || aborted) {
          alive = false;
          break;
        }
        tc::tc_fence_after();
        const int Em = (int)sExp[(it % kExpRing) * kRows + row] - 1022;
#pragma unroll
        for (int h = 0; h < EC; h += 4) {
          uint32_t rr[kL][4];
#pragma unroll
          for (int l = 0; l < kL; ++l)
            tc::tmem_ld_x4(trow + st * (kL * kCols) + l * kCols + h, rr[l]);
          tc::tmem_ld_wait();
          if (h + 4 == EC) {  // the accumulators are read: the MMAs may overwrite them
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&accfree[st]);
          }
          double val[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            int d[kL];
#pragma unroll
            for (int l = 0; l < kL; ++l) d[l] = __float2int_rn(__uint_as_float(rr[l][q]));
            val[q] = b256::level_sum(d, Em + sEn[c0 + h + q], g.weights);
          }
          const unsigned c = c0 + h;
          if (valid) {
            if constexpr (EPI == kStoreVec) {
              if (c < g.n) st4(o + c, val);
            } else {
              double *oc = o + (long long)c * g.sigma;
#pragma unroll
              for (int q = 0; q < 4; ++q, oc += g.sigma)
                if (c + q < g.n) {
                  if constexpr (EPI == kStore)
                    *oc = val[q];
                  else
                    atomicAdd(oc, val[q]);
                }
            }
          }
        }
      }
    }
  } else if (lane == 0) {
    // ---- MMA issuer
    bool ok = tc::mbar_wait(image, 0, g.err, 8);
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
  if (warp == C::kMmaWarp) tc::tmem_dealloc(tmem, kTmemCols);
}

// out += (V - theta) psi.  Bound by memory: V is read once for all vectors, psi and out read,
// out written, two unknowns per thread where 16-byte accesses are aligned.  (In a mode
// product's epilogue, whose loads of V and psi wait for memory in line with the products, the
// term cost 83 us for 3 vectors at 48^4, here 63.)
template <int W>
__global__ void __launch_bounds__(256)
k_potential_term(const double *__restrict__ psi, const double *__restrict__ V,
                 double *out, long long N, int nvec,
                 const double *__restrict__ theta_dev, double theta0) {
  if (threadIdx.x == 0) pdl_trigger();
  pdl_wait();
  const long long i = ((long long)blockIdx.x * 256 + threadIdx.x) * W;
  if (i >= N) return;
  double w[W], x[4][W], y[4][W];
#pragma unroll
  for (int k = 0; k < W; ++k) w[k] = V[i + k];
  if (!theta_dev)
#pragma unroll
    for (int k = 0; k < W; ++k) w[k] -= theta0;
  for (int v0 = 0; v0 < nvec; v0 += 4) {
#pragma unroll
    for (int v = 0; v < 4; ++v)
      if (v0 + v < nvec) {
        const long long j = (long long)(v0 + v) * N + i;
        if constexpr (W == 2) {
          const double2 a = *reinterpret_cast<const double2 *>(psi + j);
          const double2 b = *reinterpret_cast<const double2 *>(out + j);
          x[v][0] = a.x;
          x[v][1] = a.y;
          y[v][0] = b.x;
          y[v][1] = b.y;
        } else {
          x[v][0] = psi[j];
          y[v][0] = out[j];
        }
      }
#pragma unroll
    for (int v = 0; v < 4; ++v)
      if (v0 + v < nvec) {
        double *o = out + (long long)(v0 + v) * N + i;
        const double th = theta_dev ? theta_dev[v0 + v] : 0.0;
#pragma unroll
        for (int k = 0; k < W; ++k) y[v][k] = fma(theta_dev ? w[k] - th : w[k], x[v][k], y[v][k]);
        if constexpr (W == 2)
          *reinterpret_cast<double2 *>(o) = make_double2(y[v][0], y[v][1]);
        else
          *o = y[v][0];
      }
  }
}

template <int KC, Epi EPI>
cudaError_t launch_kc(const Args &g, cudaStream_t s) {
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  std::call_once(once, [] {
    attr = cudaFuncSetAttribute(k_mode_product<KC, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)Cfg<KC>::kSmem);
  });
  if (attr != cudaSuccess) return attr;
  const unsigned grid = (unsigned)(g.tiles < 152 ? g.tiles : 152);
  count_launch();
  const cudaError_t e = launch_pdl(k_mode_product<KC, EPI>, dim3(grid), dim3(Cfg<KC>::kThreads),
                                   Cfg<KC>::kSmem, s, g);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <int KC>
cudaError_t launch_epi(const Args &g, Epi epi, cudaStream_t s) {
  switch (epi) {
    case kStore: return launch_kc<KC, kStore>(g, s);
    case kStoreVec: return launch_kc<KC, kStoreVec>(g, s);
    default: return launch_kc<KC, kAdd>(g, s);
  }
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

cudaError_t launch_potential_term(const double *psi, const double *V, double *out, long long N,
                                  int nvec, const double *theta_dev, double theta0,
                                  cudaStream_t s) {
  const uintptr_t al = reinterpret_cast<uintptr_t>(psi) | reinterpret_cast<uintptr_t>(out) |
                       reinterpret_cast<uintptr_t>(V);
  const bool two = N % 2 == 0 && (al & 15) == 0;
  const long long blocks = (N / (two ? 2 : 1) + 255) / 256;
  if (blocks > 0x7FFFFFFFLL) return cudaErrorInvalidValue;
  count_launch();
  const cudaError_t e =
      launch_pdl(two ? k_potential_term<2> : k_potential_term<1>, dim3((unsigned)blocks),
                 dim3(256), 0, s, psi, V, out, N, nvec, theta_dev, theta0);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_mode_product(const ModeArgs &a, cudaStream_t s) {
  if (a.n < 1 || a.n > kMaxModePoints || a.nvec < 1) return cudaErrorInvalidValue;
  const long long M = a.N / a.n;
  if (M > 0x7FFFFFFFLL) return cudaErrorInvalidValue;
  Args g = {};
  g.psi = a.psi;
  g.out = a.out;
  g.N = a.N;
  g.M = (unsigned)M;
  g.n = (unsigned)a.n;
  g.sigma = (unsigned)a.sigma;
  g.image = a.image;
  g.eK = a.eK;
  g.err = a.err;
  g.tm = (unsigned)((M + kRows - 1) / kRows);
  g.tiles = (long long)g.tm * a.nvec;
  g.weights = b256::level_weights();
  const uintptr_t al = reinterpret_cast<uintptr_t>(a.psi) | reinterpret_cast<uintptr_t>(a.out);
  const bool vec = a.sigma == 1 && a.n % 4 == 0 && (al & 31) == 0;
  const Epi epi = !a.store ? kAdd : vec ? kStoreVec : kStore;
  switch (units(a.n)) {
    case 1: return launch_epi<1>(g, epi, s);
    case 2: return launch_epi<2>(g, epi, s);
    case 3: return launch_epi<3>(g, epi, s);
    default: return launch_epi<4>(g, epi, s);
  }
}

}  // namespace ozm
}  // namespace tps
