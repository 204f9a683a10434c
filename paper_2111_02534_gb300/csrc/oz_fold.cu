// The 1D H-apply on the tensor cores, folded by the symmetry of its mode matrices.
//
// The second derivative on a periodic grid of n points is a symmetric circulant matrix: it
// commutes with the reflection j -> -j and, for even n, with the shift by n/2.  In the
// coordinates
//   F_b[r] = sum_g chi_b(g) psi[g r],    g in the symmetry group G, chi_b its characters
// (|G| = 4 where 4 divides n, else the reflection alone) K falls into |G| blocks of n / |G|
// points,
//   (K psi)[g r] = sum_b chi_b(g) Z_b[r],  Z_b[r] = sum_s B_b[r][s] F_b[s],
//   |G| B_b[r][s] = sum over the distinct images s' of s of chi_b(s') K[r][s'],
// a quarter of the multiplications of the dense product.  The mode of a heavy-exchange sector is
// symmetric under the reversal of its points (|G| = 2).  The blocks are short enough (at most
// 146 points) for base-256 digits, 36 digit products instead of the 54 that base 64 needs for
// 512 points, so that of the tensor work of the dense product a sixth is left.
//
// The arithmetic between the rounding of the operands and that of the result is on integers: a
// line of psi is scaled by a power of two and rounded to 62 - log2|G| bits, the sums F_b are taken
// in 64-bit integers and cut into eight base-256 digits, the entries of |G| B_b likewise (62 bits
// of the row's absolute sum).  The eight levels of digit products (ozaki_tc.cu) are exact; they are
// added to one 64-bit integer per Z_b[r], with a common unit u for all blocks (2^-62 of the line's
// scale times the row's), level 7 rounded to u, and the sums over b are again exact.  Left out are
// the digit pairs with i + j >= 8: of a block of 146 points at most 7 2^14 146 2^-14 = 1022 u, about
// 11 u as a root mean square, twice and four times that for a result of four blocks (2^-57 and, at
// most, 2^-50 of the scales; an FP64 product of 512 terms is bounded by 2^-44 of them).  A product
// is rounded once, as in the dense scheme, whose psi keeps 54 bits.
//
// Three kernels:
//   k_fold_split    reads 16 lines (rows for y, columns for x) into shared memory, takes their
//                   exponents, and writes the digits of the folded lines in the operand layout
//                   of the tensor cores;
//   k_fold_gemm     persistent, one CTA per SM, over tiles of 128 lines x up to 64 points of a
//                   block, both modes and all blocks in one list; stages of 16 points of K come
//                   by one bulk copy per operand; levels lie side by side in tensor memory, so
//                   a digit slice of F times all the digit slices of B it meets is one or two
//                   MMAs (as in oz_mode.cu); writes the 64-bit sums;
//   k_fold_combine  a thread per pair of representatives (r_x, r_y) and image of r_x: unfolds
//                   both modes, adds the potential term and writes the |G_y| outputs.
//
// Measured, 8 vectors at 512 x 512: 102 us, 476 by the dense base-64 products.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>
#include <new>
#include <type_traits>

#include "oz_fold.cuh"
#include "ozaki_tc.cuh"
#include "pdl.cuh"
#include "split_digits.cuh"

namespace tps {
namespace ozf {
namespace {

constexpr int kS = 8;         // digits of either operand; levels kept: i + j <= 7
constexpr int kRows = 128;    // lines per tile
constexpr int kMaxBlock = 146;  // points of a block: 7 2^14 146 < 2^24 (the top digits are
                                // at most 64, so level 7 counts as seven pairs)
constexpr int kMaxCols = 64;  // output points per tile: 8 levels x 64 = 512 TMEM columns
constexpr int kLines = 16;    // lines per block of the split
constexpr uint32_t kAStage = kS * kRows * 32;     // 16 points of K: bytes of A
constexpr uint32_t kBStage = kS * kMaxCols * 32;  // and, at most, of B
constexpr int kStages = 4;
constexpr uint32_t kTmemCols = 512;
constexpr int kEpiWarps = 8;
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr size_t kGemmSmem = 1024 + kStages * (kAStage + kBStage) + 256;

enum Kind { kNone = 0, kCirculant = 1, kMirror = 2 };

// A mode of n points folded by a group of G elements; block b has size[b] positions.
struct Mode {
  int n, kind, G, reps;
  int size[4];
  int kc[4];  // 16-point units of its contraction
  int w[4], tn[4];  // tiles of its output positions: tn of w (a multiple of 16)
};

Mode make_mode(int n, int kind) {
  Mode m = {};
  m.n = n;
  m.kind = kind;
  if (kind == kCirculant && n % 4 == 0) {
    m.G = 4;
    m.reps = n / 4 + 1;
    m.size[0] = n / 4 + 1;
    m.size[1] = m.size[2] = m.size[3] = n / 4;
  } else if (kind == kCirculant) {  // n even
    m.G = 2;
    m.reps = n / 2 + 1;
    m.size[0] = n / 2 + 1;
    m.size[1] = n / 2;
  } else if (kind == kMirror && n >= 2) {
    m.G = 2;
    m.reps = (n + 1) / 2;
    m.size[0] = (n + 1) / 2;
    m.size[1] = n / 2;
  } else {
    m.G = 1;
    m.reps = m.size[0] = n;
  }
  for (int b = 0; b < m.G; ++b) {
    m.kc[b] = (m.size[b] + 15) / 16;
    m.tn[b] = (m.size[b] + kMaxCols - 1) / kMaxCols;
    m.w[b] = 16 * ((m.size[b] + 16 * m.tn[b] - 1) / (16 * m.tn[b]));
  }
  return m;
}

// Image t of representative r.
__host__ __device__ __forceinline__ int image_of(const Mode &m, int r, int t) {
  if (t == 0) return r;
  if (m.kind == kMirror) return m.n - 1 - r;
  if (t == 1) return r ? m.n - r : 0;
  return t == 2 ? m.n / 2 - r : m.n / 2 + r;
}
// Whether block b's character is -1 on image t (bit 0 of b: the reflection, bit 1: the
// reflection about n / 4).
__host__ __device__ __forceinline__ bool negative(int b, int t) {
  return t == 1 ? b & 1 : t == 2 ? b >> 1 : t == 3 ? (b & 1) ^ (b >> 1) : false;
}
// The representative at position p of block b, or -1 if that place is empty.  A point that the
// group leaves in place has no part in the blocks whose character changes its sign; the
// representative n / 4 takes the place that 0 leaves in the block odd under the reflection only.
__host__ __device__ __forceinline__ int rep_at(const Mode &m, int b, int p) {
  if (m.kind == kCirculant && m.G == 4) {
    const int q = m.n / 4;
    if (b == 0) return p <= q ? p : -1;
    if (b == 1) return p == 0 ? q : (p < q ? p : -1);
    if (b == 2) return p < q ? p : -1;
    return p > 0 && p < q ? p : -1;
  }
  if (m.kind == kCirculant) {
    if (b == 0) return p <= m.n / 2 ? p : -1;
    return p > 0 && p < m.n / 2 ? p : -1;
  }
  return p < m.size[b] ? p : -1;
}
// The position of representative r in block b, or -1.
__device__ __forceinline__ int pos_of(const Mode &m, int b, int r) {
  if (m.kind == kCirculant && m.G == 4 && b == 1 && r == m.n / 4) return 0;
  return rep_at(m, b, r) == r ? r : -1;
}

// round(x 2^(bits - E)), E = raw_max - 1022 (|x| < 2^E), bits = 62 - log2 G; subnormals count
// as zero.
__device__ __forceinline__ long long scaled(double x, unsigned raw_max, int bits) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned ex = (hi >> 20) & 0x7FFu;
  const unsigned sh = ex ? min(raw_max - ex, 63u) : 63u;
  const unsigned long long m =
      ((unsigned long long)((hi & 0xFFFFFu) | 0x100000u) << 32 | lo) << (bits - 52);
  const long long a = (long long)(((m >> sh) + 1) >> 1);
  return (int)hi < 0 ? -a : a;
}

// The digits of two neighbouring integers |q| <= 2^62 as FP16 pairs, most significant first:
// q + 128 (1 + 2^8 + .. + 2^56) has the digits plus 128 as its bytes; byte b as the FP16 number
// 1024 + b, minus 1152.
__device__ __forceinline__ void digit_pairs(long long q0, long long q1, uint32_t (&d)[kS]) {
  const unsigned long long bias = 0x8080808080808080ULL;
  const unsigned long long u0 = (unsigned long long)q0 + bias, u1 = (unsigned long long)q1 + bias;
  const uint32_t l0 = (uint32_t)u0, h0 = (uint32_t)(u0 >> 32);
  const uint32_t l1 = (uint32_t)u1, h1 = (uint32_t)(u1 >> 32);
  const __half2 off = __half2half2(__ushort_as_half(0x6480));  // 1152
  const uint32_t w[kS] = {__byte_perm(h0, h1, 0x7733), __byte_perm(h0, h1, 0x7632),
                          __byte_perm(h0, h1, 0x5511), __byte_perm(h0, h1, 0x5410),
                          __byte_perm(l0, l1, 0x7733), __byte_perm(l0, l1, 0x7632),
                          __byte_perm(l0, l1, 0x5511), __byte_perm(l0, l1, 0x5410)};
#pragma unroll
  for (int i = 0; i < kS; ++i) {
    const uint32_t v = (w[i] & 0x00FF00FFu) | 0x64006400u;
    const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&v), off);
    d[i] = *reinterpret_cast<const uint32_t *>(&h);
  }
}

// ------------------------------- the operator's image -------------------------------
// Digits of |G| B_b: per tile of w output positions and unit of 16 positions of K, 8 w rows
// (digit j of column c at j w + c) in the operand layout: the first 8 positions of all rows, 16
// bytes a row, then the other 8.  eB[r]: exponent of the absolute sum of row r of K.
__global__ void k_row_sums(const double *__restrict__ K, Mode m, int *__restrict__ eB) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= m.reps) return;
  double sum = 0.0;
  for (int i = 0; i < m.n; ++i) sum += fabs(K[(long long)r * m.n + i]);
  eB[r] = (int)b256::raw_exp(sum) - 1022;
}

__global__ void k_fold_image(const double *__restrict__ K, Mode m, int b,
                             const int *__restrict__ eB, uint4 *__restrict__ image) {
  const int w = m.w[b], rows = kS * w;
  const long long total = (long long)m.tn[b] * m.kc[b] * 2 * rows;
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < total;
       p += (long long)gridDim.x * blockDim.x) {
    const int row = (int)(p % rows), sub = (int)(p / rows % 2);
    const int k = (int)(p / (2 * rows) % m.kc[b]), tile = (int)(p / (2 * rows) / m.kc[b]);
    const int j = row / w, ro = rep_at(m, b, tile * w + row % w);
    __half h[8];
    for (int e = 0; e < 8; ++e) {
      const int rk = rep_at(m, b, k * 16 + sub * 8 + e);
      long long q = 0;
      if (ro >= 0 && rk >= 0) {
        const unsigned raw = (unsigned)(eB[ro] + 1022);
        for (int t = 0; t < m.G; ++t) {
          const int s = image_of(m, rk, t);
          bool seen = false;
          for (int u = 0; u < t; ++u) seen |= image_of(m, rk, u) == s;
          if (seen) continue;
          const long long a = raw ? scaled(K[(long long)ro * m.n + s], raw, 62) : 0;
          q += negative(b, t) ? -a : a;
        }
      }
      const unsigned long long u = (unsigned long long)q + 0x8080808080808080ULL;
      h[e] = __int2half_rn((int)((u >> (8 * (7 - j))) & 0xFF) - 128);
    }
    image[p] = *reinterpret_cast<const uint4 *>(h);
  }
}

// ------------------------------------- split -------------------------------------
struct SplitArgs {
  const double *psi;
  long long N;
  int ny, nlines[2];      // lines of the y mode (rows) and of the x mode (columns)
  Mode m[2];              // y, x
  uint16_t *A[2][4];      // folded digits of a mode's block
  int *eL[2];             // exponents of the lines
  int first_x;            // first block of the x lines
};

// 16 lines per block: loaded once (y: along the lines; x: 128-byte pieces across them), the
// exponents taken, then a warp takes 8 positions of the 16 lines at a time (a lane 4 positions
// of one line), so that its stores are 256 contiguous bytes.  Exponents and digits in one pass:
// the separate exponent kernel and the second read of psi cost 9 us of 40 at 512 x 512, 8
// vectors.
__global__ void __launch_bounds__(256) k_fold_split(const __grid_constant__ SplitArgs g) {
  extern __shared__ double tile[];  // [kLines][n | 1]
  __shared__ unsigned ex[kLines];
  if (threadIdx.x == 0) pdl_trigger();
  const int d = (int)blockIdx.x >= g.first_x;
  const Mode &m = g.m[d];
  const int n = m.n, ld = n | 1, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int line0 = ((int)blockIdx.x - (d ? g.first_x : 0)) * kLines;
  if (tid < kLines) ex[tid] = 0;
  __syncthreads();
  pdl_wait();
  if (d == 0) {
    for (int l = warp; l < kLines; l += 8) {
      unsigned mx = 0;
      const bool in = line0 + l < g.nlines[0];
      const double *p = g.psi + (long long)(line0 + l) * n;
      for (int i = lane; i < n; i += 32) {
        const double x = in ? p[i] : 0.0;
        tile[l * ld + i] = x;
        mx = max(mx, b256::raw_exp(x));
      }
      mx = __reduce_max_sync(0xffffffffu, mx);
      if (lane == 0) ex[l] = mx;
    }
  } else {
    const int l = tid & (kLines - 1), line = line0 + l;
    const bool in = line < g.nlines[1];
    const int v = line / g.ny, iy = line - v * g.ny;
    const double *p = g.psi + (long long)v * g.N + iy;
    unsigned mx = 0;
#pragma unroll 4
    for (int i = tid / kLines; i < n; i += 256 / kLines) {
      const double x = in ? p[(long long)i * g.ny] : 0.0;
      tile[l * ld + i] = x;
      mx = max(mx, b256::raw_exp(x));
    }
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
    if (lane < kLines) atomicMax(&ex[l], mx);
  }
  __syncthreads();
  if (tid < kLines && line0 + tid < g.nlines[d]) g.eL[d][line0 + tid] = (int)ex[tid] - 1022;
  // the scaled integers in place of the values (each is used by every block of its images)
  const int bits = m.G == 4 ? 60 : m.G == 2 ? 61 : 62;
  for (int k = warp; k < kLines; k += 8) {
    const unsigned raw = ex[k];
#pragma unroll 4
    for (int i = lane; i < n; i += 32)
      tile[k * ld + i] = __longlong_as_double(scaled(tile[k * ld + i], raw, bits));
  }
  __syncthreads();
  const int l = lane >> 1;
  const long long *x = reinterpret_cast<const long long *>(tile) + l * ld;
  const int chunks = 2 * m.kc[0];  // the largest block's
  // the line's place in the operand layout
  const long long rt = (line0 + l) / kRows;
  const int row = (line0 + l) % kRows;
  for (int c = warp; c < chunks; c += 8) {
    const int p0 = c * 8 + (lane & 1) * 4;
    long long a[4][4];  // [position][image]
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int t = 0; t < 4; ++t)
        a[k][t] = t < m.G && p0 + k < m.reps ? x[image_of(m, p0 + k, t)] : 0;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      if (b >= m.G || c >= 2 * m.kc[b]) continue;
      long long f[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int r = rep_at(m, b, p0 + k);
        long long s = 0;
        if (r == p0 + k) {
#pragma unroll
          for (int t = 0; t < 4; ++t) s += negative(b, t) ? -a[k][t] : a[k][t];
        } else if (r >= 0) {  // the representative n / 4 at position 0
          for (int t = 0; t < m.G; ++t) {
            const long long y = x[image_of(m, r, t)];
            s += negative(b, t) ? -y : y;
          }
        }
        f[k] = s;
      }
      uint32_t d0[kS], d1[kS];
      digit_pairs(f[0], f[1], d0);
      digit_pairs(f[2], f[3], d1);
      // [row tile][unit of 16][slice][half of the unit][row][8 positions]
      uint16_t *dst = g.A[d][b] + (rt * m.kc[b] + (c >> 1)) * (kAStage / 2) + (c & 1) * kRows * 8 +
                      row * 8 + (lane & 1) * 4;
#pragma unroll
      for (int i = 0; i < kS; ++i)
        *reinterpret_cast<uint2 *>(dst + i * (kRows * 16)) = make_uint2(d0[i], d1[i]);
    }
  }
}

// ------------------------------------- product -------------------------------------
struct Entry {  // one block of one mode
  const uint16_t *A;
  const uint4 *B;
  long long *T;      // y: [line][ld] of positions; x: [position][ld] of lines
  int units, tn, w, kc, ld, x;
};
struct GemmArgs {
  Entry e[8];
  int n, total;
  int w2, w10, w18, w26;  // powers of two (see below)
  int *err;
};

__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lead) {
  // K-major, no swizzle: start >> 4, offset between the two 8-point columns, between groups of
  // 8 rows (128 bytes), fixed 0b001
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lead >> 4) << 16) |
         ((uint64_t)(128 >> 4) << 32) | ((uint64_t)1 << 46);
}
__device__ __forceinline__ uint32_t idesc_f16(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes,
                                          uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(tc::smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(tc::smem_addr(bar))
      : "memory");
}
__device__ __forceinline__ const Entry &find_unit(const GemmArgs &g, int u, int &at) {
  int k = 0;
  while (k + 1 < g.n && u >= g.e[k].units) u -= g.e[k++].units;
  at = u;
  return g.e[k];
}

// Warp 0 copies, warp 1 issues the MMAs, warps 2-9 drain (TMEM lanes 32 (warp % 4) .. + 31, half
// of the columns each).  A stage is one unit of 16 points of K (32 KB of A, up to 16 KB of B):
// 1152 cycles of MMA for 64 columns, 41 bytes per cycle and SM from L2.
__global__ void __launch_bounds__(kThreads, 1)
k_fold_gemm(const __grid_constant__ GemmArgs g) {
  extern __shared__ uint8_t raw_smem[];
  __shared__ int abort_flag;
  uint8_t *base = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(raw_smem) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t *bars = reinterpret_cast<uint64_t *>(base + kStages * (kAStage + kBStage));
  uint64_t *full = bars, *empty = bars + kStages, *accum = empty + kStages, *accfree = accum + 1;
  uint64_t *drained = accfree + 1;
  uint32_t *holder = reinterpret_cast<uint32_t *>(drained + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) {
      tc::mbar_init(&full[i], 1);
      tc::mbar_init(&empty[i], 1);
    }
    tc::mbar_init(accum, 1);
    tc::mbar_init(accfree, kEpiWarps);
    tc::mbar_init(drained, 1);
    abort_flag = 0;
    tc::fence_barrier_init();
  }
  if (warp == 1) tc::tmem_alloc(holder, kTmemCols);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  // only now: a dependent kernel's CTA must not take tensor memory that this one waits for
  if (threadIdx.x == 0) pdl_trigger();
  const uint32_t tmem = *holder;
  pdl_wait();

  if (warp == 0) {
    if (lane == 0) {
      bool ok = true;
      int it = 0;
      for (int u = blockIdx.x; u < g.total && ok; u += gridDim.x) {
        int at;
        const Entry &e = find_unit(g, u, at);
        const int rt = at / e.tn, tile = at % e.tn;
        const uint32_t bbytes = kS * e.w * 32;
        const uint8_t *A = reinterpret_cast<const uint8_t *>(e.A) + (long long)rt * e.kc * kAStage;
        const uint8_t *B = reinterpret_cast<const uint8_t *>(e.B) + (long long)tile * e.kc * bbytes;
        for (int k = 0; k < e.kc; ++k, ++it) {
          const int st = it % kStages;
          if (!tc::mbar_wait(&empty[st], ((it / kStages) & 1) ^ 1, g.err, 1)) {
            ok = false;
            break;
          }
          uint8_t *s = base + st * (kAStage + kBStage);
          tc::mbar_arrive_expect_tx(&full[st], kAStage + bbytes);
          bulk_load(s, A + (long long)k * kAStage, kAStage, &full[st]);
          bulk_load(s + kAStage, B + (long long)k * bbytes, bbytes, &full[st]);
        }
      }
      if (!ok) {
        // wind down: let the copies in flight land before the CTA exits
        atomicExch(&abort_flag, 1);
        for (int k = it < kStages ? 0 : it - kStages; k < it; ++k)
          tc::mbar_wait(&full[k % kStages], (k / kStages) & 1, nullptr, 0);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      bool ok = true;
      int it = 0, done = 0;
      for (int u = blockIdx.x; u < g.total && ok; u += gridDim.x, ++done) {
        int at;
        const Entry &e = find_unit(g, u, at);
        const int w = e.w;
        if (!tc::mbar_wait(accfree, (done & 1) ^ 1, g.err, 6)) {
          ok = false;
          break;
        }
        tc::tc_fence_after();
        for (int k = 0; k < e.kc; ++k, ++it) {
          const int st = it % kStages;
          if (!tc::mbar_wait(&full[st], (it / kStages) & 1, g.err, 3)) {
            ok = false;
            break;
          }
          tc::tc_fence_after();
          const uint32_t s = tc::smem_addr(base) + st * (kAStage + kBStage);
          const uint64_t ad = smem_desc(s, kRows * 16), bd = smem_desc(s + kAStage, kS * w * 16);
#pragma unroll
          for (int i = 0; i < kS; ++i) {  // levels i .. 7, at most 256 columns at a time
            const int cols = w * (kS - i), c1 = cols < 256 ? cols : 256;
            tc::mma_bf16(tmem + i * w, ad + (uint64_t)(i * (kRows * 32 >> 4)), bd,
                         idesc_f16(kRows, c1), (k > 0 || i > 0) ? 1u : 0u);
            if (cols > c1)
              tc::mma_bf16(tmem + i * w + c1, ad + (uint64_t)(i * (kRows * 32 >> 4)),
                           bd + (uint64_t)c1, idesc_f16(kRows, cols - c1),
                           (k > 0 || i > 0) ? 1u : 0u);
          }
          tc::mma_commit(&empty[st]);
        }
        if (ok) tc::mma_commit(accum);
      }
      if (!ok) atomicExch(&abort_flag, 1);
      tc::mma_commit(drained);
      tc::mbar_wait(drained, 0, g.err, 7);
    }
  } else {
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    const uint32_t trow = tmem + ((uint32_t)(32 * quarter) << 16);
    int done = 0;
    for (int u = blockIdx.x; u < g.total; u += gridDim.x, ++done) {
      int at;
      const Entry &e = find_unit(g, u, at);
      const int rt = at / e.tn, tile = at % e.tn, w = e.w;
      bool ok = tc::mbar_wait(accum, done & 1, g.err, 5);
      ok = __all_sync(0xffffffffu, ok);
      const int aborted = __shfl_sync(0xffffffffu, *((volatile int *)&abort_flag), 0);
      if (!ok || aborted) break;
      tc::tc_fence_after();
      const long long line = (long long)rt * kRows + 32 * quarter + lane;
      for (int c = half * (w / 2); c < (half + 1) * (w / 2); c += 4) {
        uint32_t r[kS][4];
#pragma unroll
        for (int l = 0; l < kS; ++l) tc::tmem_ld_x4(trow + l * w + c, r[l]);
        tc::tmem_ld_wait();
        // sum_l d_l 2^(50 - 8 l) modulo 2^64 (the sum is below 2^62; of level 7 the part below
        // the unit is rounded away); the powers of two come from the arguments so that the
        // products run as multiply-adds on the FMA pipe
        long long t[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          int d[kS];
#pragma unroll
          for (int l = 0; l < kS; ++l) d[l] = __float2int_rn(__uint_as_float(r[l][q]));
          const int t7 = (d[7] + 32) >> 6;
          asm("{\n\t.reg .b64 t;\n\t"
              "cvt.s64.s32 t, %5;\n\t"
              "mad.wide.s32 t, %4, %6, t;\n\t"
              "mad.wide.s32 t, %3, %7, t;\n\t"
              "mad.wide.s32 t, %2, %8, t;\n\t"
              "mad.wide.s32 %0, %1, %9, t;\n\t}"
              : "=l"(t[q])
              : "r"(d[3]), "r"(d[4]), "r"(d[5]), "r"(d[6]), "r"(t7), "r"(g.w2), "r"(g.w10),
                "r"(g.w18), "r"(g.w26));
          const unsigned top = (unsigned)(d[0] * g.w18) + (unsigned)(d[1] * g.w10) +
                               (unsigned)(d[2] * g.w2);
          t[q] = (long long)((unsigned long long)t[q] + ((unsigned long long)top << 32));
        }
        const int p = tile * w + c;
        if (e.x) {
#pragma unroll
          for (int q = 0; q < 4; ++q) e.T[(long long)(p + q) * e.ld + line] = t[q];
        } else {
          asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(
                           e.T + line * e.ld + p),
                       "l"(t[0]), "l"(t[1]), "l"(t[2]), "l"(t[3])
                       : "memory");
        }
      }
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(accfree);
    }
  }
  __syncwarp();
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 1) tc::tmem_dealloc(tmem, kTmemCols);
}

// ------------------------------------- combine -------------------------------------
// t 2^e rounded to FP64 by integer arithmetic (ties away from zero): the FP64 pipe, on which a
// conversion takes ~64 cycles of a scheduler, has the sums and the potential term to do.
__device__ __forceinline__ double round_int(long long t, int e) {
  const unsigned sg = (unsigned)(t >> 63);
  const unsigned long long u =
      ((unsigned long long)t ^ (unsigned long long)(long long)(int)sg) + (sg & 1u);
  unsigned a = (unsigned)(u >> 32), b = (unsigned)u;
  int be = e + 1086;  // exponent field of a leading bit at 63
  if (a == 0) {
    a = b;
    b = 0;
    be -= 32;
  }
  if (a == 0) return 0.0;
  const int s = __clz((int)a);
  be -= s;
  if (be <= 0 || be >= 2046) {  // near the ends of the range: two factors
    const int h = e / 2;
    return (double)t * b256::pow2d(h) * b256::pow2d(e - h);
  }
  const unsigned wh = __funnelshift_l(b, a, s), wl = b << s;
  // 53 bits (the leading one adds 1 to the exponent field) and the rounding bit
  const unsigned long long m =
      (((unsigned long long)(wh >> 11) << 32) | __funnelshift_r(wl, wh, 11)) +
      ((wl >> 10) & 1u) + ((unsigned long long)(unsigned)(be - 1) << 52);
  return __longlong_as_double(
      (long long)(m | ((unsigned long long)(sg & 0x80000000u) << 32)));
}

struct CombineArgs {
  Mode my, mx;
  const long long *Ty[4], *Tx[4];
  int ldy[4], ldx;
  const int *eLy, *eLx, *eBy, *eBx;  // exponents of the lines and of the operators' rows
  const double *psi, *V, *theta_dev;
  double *out;
  long long N;
  double theta0;
};

// A thread per pair of representatives and image of the one of x (threadIdx.y), adjacent lanes
// on adjacent representatives of y, so that accesses are contiguous (or contiguous backwards).
// The images of r_x read the same sums of the x mode, from L1.  (All images in one thread, 105
// registers and a warp per row of representatives: 43 us at 512 x 512, 8 vectors.)
template <int GX, int GY>
__global__ void __launch_bounds__(64 * GX) k_fold_combine(const __grid_constant__ CombineArgs g) {
  if (threadIdx.x == 0 && threadIdx.y == 0) pdl_trigger();
  pdl_wait();
  const int e = blockIdx.x * 64 + threadIdx.x, a = threadIdx.y, v = blockIdx.y;
  const int rx = e / g.my.reps, ry = e - rx * g.my.reps;
  if (rx >= g.mx.reps) return;
  const int nx = g.mx.n, ny = g.my.n;
  const int ix = image_of(g.mx, rx, a);
  for (int c = 0; c < a; ++c)
    if (image_of(g.mx, rx, c) == ix) return;  // a point that the group leaves in place
  const double th = g.theta_dev ? g.theta_dev[v] : g.theta0;
  const int ey = g.eLy[v * nx + ix] + g.eBy[ry] - 62, ebx = g.eBx[rx] - 62;
  long long ty[GY], px[GX];
#pragma unroll
  for (int b = 0; b < GY; ++b) {
    const int p = pos_of(g.my, b, ry);
    ty[b] = p >= 0 ? g.Ty[b][((long long)v * nx + ix) * g.ldy[b] + p] : 0;
  }
#pragma unroll
  for (int b = 0; b < GX; ++b) px[b] = pos_of(g.mx, b, rx);
  int iy[GY];
#pragma unroll
  for (int t = 0; t < GY; ++t) {
    iy[t] = image_of(g.my, ry, t);
    bool dup = false;
#pragma unroll
    for (int c = 0; c < t; ++c) dup |= iy[c] == iy[t];
    if (dup) continue;
    const long long at = (long long)ix * ny + iy[t], col = (long long)v * ny + iy[t];
    long long sy = 0, sx = 0;
#pragma unroll
    for (int b = 0; b < GX; ++b) {
      const long long z = px[b] >= 0 ? g.Tx[b][px[b] * g.ldx + col] : 0;
      sx += negative(b, a) ? -z : z;
    }
#pragma unroll
    for (int b = 0; b < GY; ++b) sy += negative(b, t) ? -ty[b] : ty[b];
    const double y = round_int(sy, ey), x = round_int(sx, g.eLx[col] + ebx);
    g.out[(long long)v * g.N + at] = fma(g.V[at] - th, g.psi[(long long)v * g.N + at], y) + x;
  }
}

template <int GX>
cudaError_t launch_combine(const CombineArgs &c, dim3 grid, cudaStream_t s) {
  const dim3 block(64, GX);
  count_launch();
  switch (c.my.G) {
    case 1: return launch_pdl(k_fold_combine<GX, 1>, grid, block, 0, s, c);
    case 2: return launch_pdl(k_fold_combine<GX, 2>, grid, block, 0, s, c);
    default: return launch_pdl(k_fold_combine<GX, 4>, grid, block, 0, s, c);
  }
}

int kind_of(const DevOperator &op, int k) {
  return op.symmetry[k] == kModeCirculant ? kCirculant
                                          : op.symmetry[k] == kModeMirror ? kMirror : kNone;
}

}  // namespace

struct Operator {
  Mode m[2];       // y, x
  int chunk = 0;   // vectors per launch
  int rows[2] = {0, 0};  // lines of a chunk, padded to tiles
  uint4 *B[2][4] = {};
  int *eB[2] = {nullptr, nullptr};
  uint16_t *A[2][4] = {};
  int *eL[2] = {nullptr, nullptr};
  long long *T[2][4] = {};
  uint8_t *arena = nullptr;
  int *err = nullptr;
};

bool supported(const DevOperator &op) {
  if (op.nmodes != 2) return false;
  for (int k = 0; k < 2; ++k) {
    const Mode m = make_mode(op.n[k], kind_of(op, k));
    if (m.size[0] > kMaxBlock) return false;
  }
  return true;
}

void destroy(Operator *o) {
  if (!o) return;
  cudaFree(o->arena);
  delete o;
}

Operator *create(const DevOperator &op, int *err, cudaStream_t s, cudaError_t *e) {
  *e = cudaErrorMemoryAllocation;
  Operator *o = new (std::nothrow) Operator();
  if (!o) return nullptr;
  o->err = err;
  const int lines[2] = {op.n[0], op.n[1]};  // per vector: rows for y, columns for x
  long long per_vec = 0;  // bytes
  for (int d = 0; d < 2; ++d) {
    o->m[d] = make_mode(op.n[1 - d], kind_of(op, 1 - d));
    for (int b = 0; b < o->m[d].G; ++b)
      per_vec += (long long)lines[d] * (o->m[d].kc[b] * (kAStage / kRows) +
                                        8 * o->m[d].w[b] * o->m[d].tn[b]);
  }
  // vectors per launch: as many as keep the workspace near 256 MB
  const long long ch = (256LL << 20) / per_vec;
  o->chunk = (int)(ch < 1 ? 1 : (ch > 64 ? 64 : ch));
  // everything in one allocation: sizes first, then the addresses
  for (int pass = 0; pass < 2; ++pass) {
    size_t at = 0;
    auto take = [&](auto *&p, size_t bytes) {
      if (pass) p = reinterpret_cast<std::remove_reference_t<decltype(p)>>(o->arena + at);
      at += (bytes + 255) / 256 * 256;
    };
    for (int d = 0; d < 2; ++d) {
      const Mode &m = o->m[d];
      o->rows[d] = (lines[d] * o->chunk + kRows - 1) / kRows * kRows;
      take(o->eB[d], sizeof(int) * m.reps);
      take(o->eL[d], sizeof(int) * o->rows[d]);
      for (int b = 0; b < m.G; ++b) {
        take(o->B[d][b], (size_t)m.tn[b] * m.kc[b] * kS * m.w[b] * 32);
        take(o->A[d][b], (size_t)(o->rows[d] / kRows) * m.kc[b] * kAStage);
        take(o->T[d][b], sizeof(long long) * (size_t)o->rows[d] * m.w[b] * m.tn[b]);
      }
    }
    if (!pass) *e = cudaMalloc(&o->arena, at);
    if (*e != cudaSuccess) {
      destroy(o);
      return nullptr;
    }
  }
  for (int d = 0; d < 2; ++d) {
    const Mode &m = o->m[d];
    count_launch();
    k_row_sums<<<(m.reps + 63) / 64, 64, 0, s>>>(op.K[1 - d], m, o->eB[d]);
    for (int b = 0; b < m.G; ++b) {
      count_launch();
      k_fold_image<<<152, 256, 0, s>>>(op.K[1 - d], m, b, o->eB[d], o->B[d][b]);
    }
  }
  *e = cudaGetLastError();
  if (*e != cudaSuccess) {
    destroy(o);
    return nullptr;
  }
  return o;
}

cudaError_t apply(const Operator &o, const DevOperator &op, const double *psi, double *out,
                  int nvec, const double *theta_dev, double theta, cudaStream_t s) {
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  const size_t most = sizeof(double) * kLines * (4 * kMaxBlock + 1);  // the longest line
  std::call_once(once, [&] {
    attr = cudaFuncSetAttribute(k_fold_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kGemmSmem);
    if (attr == cudaSuccess)
      attr = cudaFuncSetAttribute(k_fold_split, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)most);
  });
  if (attr != cudaSuccess) return attr;
  const int nx = op.n[0], ny = op.n[1];
  for (int v0 = 0; v0 < nvec; v0 += o.chunk) {
    const int nv = nvec - v0 < o.chunk ? nvec - v0 : o.chunk;
    const double *P = psi + (long long)v0 * op.N;
    double *O = out + (long long)v0 * op.N;
    SplitArgs a = {};
    a.psi = P;
    a.N = op.N;
    a.ny = ny;
    a.nlines[0] = nv * nx;
    a.nlines[1] = nv * ny;
    GemmArgs g = {};
    for (int d = 0; d < 2; ++d) {
      a.m[d] = o.m[d];
      a.eL[d] = o.eL[d];
      for (int b = 0; b < 4; ++b) a.A[d][b] = o.A[d][b];
    }
    a.first_x = (a.nlines[0] + kLines - 1) / kLines;
    const int blocks = a.first_x + (a.nlines[1] + kLines - 1) / kLines;
    const int longest = nx > ny ? nx : ny;
    count_launch();
    cudaError_t e = launch_pdl(k_fold_split, dim3((unsigned)blocks), dim3(256),
                               sizeof(double) * kLines * (longest | 1), s, a);
    if (e != cudaSuccess) return e;
    // the tiles with the most work first
    for (int b = 0; b < 4; ++b)
      for (int d = 0; d < 2; ++d) {
        const Mode &m = o.m[d];
        if (b >= m.G) continue;
        Entry &n = g.e[g.n];
        n.A = o.A[d][b];
        n.B = o.B[d][b];
        n.T = o.T[d][b];
        n.tn = m.tn[b];
        n.w = m.w[b];
        n.kc = m.kc[b];
        n.ld = d ? o.rows[1] : m.w[b] * m.tn[b];
        n.x = d;
        n.units = (a.nlines[d] + kRows - 1) / kRows * m.tn[b];
        g.total += n.units;
        ++g.n;
      }
    g.w2 = 1 << 2;
    g.w10 = 1 << 10;
    g.w18 = 1 << 18;
    g.w26 = 1 << 26;
    g.err = o.err;
    count_launch();
    e = launch_pdl(k_fold_gemm, dim3((unsigned)(g.total < 152 ? g.total : 152)), dim3(kThreads),
                   kGemmSmem, s, g);
    if (e != cudaSuccess) return e;
    CombineArgs c = {};
    c.my = o.m[0];
    c.mx = o.m[1];
    for (int b = 0; b < 4; ++b) {
      c.Ty[b] = o.T[0][b];
      c.Tx[b] = o.T[1][b];
      c.ldy[b] = o.m[0].w[b] * o.m[0].tn[b];
    }
    c.ldx = o.rows[1];
    c.eLy = o.eL[0];
    c.eLx = o.eL[1];
    c.eBy = o.eB[0];
    c.eBx = o.eB[1];
    c.psi = P;
    c.V = op.V;
    c.theta_dev = theta_dev ? theta_dev + v0 : nullptr;
    c.theta0 = theta;
    c.out = O;
    c.N = op.N;
    const dim3 grid((c.my.reps * c.mx.reps + 63) / 64, nv);
    e = c.mx.G == 4 ? launch_combine<4>(c, grid, s)
                    : c.mx.G == 2 ? launch_combine<2>(c, grid, s) : launch_combine<1>(c, grid, s);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace ozf
}  // namespace tps
