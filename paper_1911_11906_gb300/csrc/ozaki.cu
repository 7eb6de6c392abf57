// FP64-accurate GEMM from BF16 tensor-core products (Ozaki's error-free
// splitting: K. Ozaki, T. Ogita, S. Oishi, S. M. Rump, Numer. Algorithms 59,
// 2012), written from the method's mathematics.
//
// Every row i of op(A) is scaled by 2^-e_i (e_i: the exponent of its largest
// entry) and cut into balanced digits of radix 2^r, r = w + 1:
// a = 2^(e_i - t) sum_p d_p 2^(r (D - 1 - p)) with t = r D - 1 fraction bits
// and every digit an integer in [-2^w, 2^w] (exact in BF16 for w <= 8);
// likewise every column j of op(B) with 2^f_j.  A product of two digits is at
// most 2^2w, so a sum of 2^(24-2w) of them is exact in an FP32 accumulator: the
// tensor cores compute P_pq = A_p B_q exactly in K-chunks of that length (1024
// for w = 7, 256 for w = 8), and the exact chunk sums are added, scaled by
// 2^-r(p+q), into an FP64 accumulator per output element.  Balanced digits
// carry one bit more than the magnitude w that bounds the chunk (the sign),
// so 7 digits (28 pairs) hold the 56 bits that sign-magnitude digits of w
// bits need 8 (36 pairs) for, at the same chunk length.  Pairs with p + q < D
// are kept; the D - 1 dropped pairs of the next diagonal and the rounding of the
// last digit are below about (D + 1) 2^-rD (r D = 64: 2 (D + 1) 2^-rD) relative to
// |row max| |column max| per term, with either sign.
// The result C = alpha 2^(e_i + f_j) sum + beta C is formed in FP64.
//
// Two tensor-core kernels compute the slice products: the sm_103a one uses
// tcgen05.mma with operands brought into shared memory by TMA
// (cp.async.bulk.tensor, 128-byte swizzle) and the FP32 chunk accumulators in
// tensor memory (four buffers at 128 columns, two at 256), so that the
// draining of finished chunks overlaps the products of the next ones; a plain mma.sync m16n8k16 kernel is kept as the reference route
// for checking it.
#include <cuda.h>
#include <cuda_bf16.h>

#include <mutex>

#include "internal.cuh"
#include "tc_common.cuh"

namespace fraclap {
namespace {

using namespace tc;

constexpr int OZ_BM = 64, OZ_BN = 64, OZ_BK = 32, OZ_NT = 128;
constexpr int OZ_KPAD = 64;  // slice rows padded to a multiple of 64 (one TMA box)
constexpr int OZ_LDS = OZ_BK / 2 + 4;  // shared row stride in 32-bit words (padded)

// e with every |entry| < 2^e, from the largest |entry| t given as the bits
// of its IEEE pattern with the sign cleared.
__device__ __forceinline__ int exponent_above(unsigned long long t) {
  int e = 0;
  const int E = (int)(t >> 52);
  if (E > 0) e = E - 1022;  // t = f 2^e, f in [0.5, 1): every |entry| < 2^e
  else if (t != 0) frexp(__longlong_as_double((long long)t), &e);  // subnormal maximum
  return e;
}

// Exponent of the largest |entry| of each row of op(A), rows contiguous (length K);
// an infinity or NaN, which has no digits, sets *nonfinite.
// One block per row.  The magnitudes are compared as the integers of their
// IEEE bit patterns with the sign cleared (the same order as the values), so
// the FP64 pipe is not used.
__global__ void row_exponents(const double* A, int64_t lda, int64_t K, int* ex, int* nonfinite) {
  const int64_t i = blockIdx.x;
  unsigned long long m = 0;
  for (int64_t k = threadIdx.x; k < K; k += blockDim.x) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(A[k + i * lda]) & 0x7FFFFFFFFFFFFFFFull;
    m = u > m ? u : m;
  }
  __shared__ unsigned long long red[32];
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, m, o);
    m = v > m ? v : m;
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    for (unsigned w = 0; w < blockDim.x / 32; ++w) t = red[w] > t ? red[w] : t;
    ex[i] = exponent_above(t);
    if (nonfinite && (t >> 52) == 2047) *nonfinite = 1;
  }
}

// The same for the rows of an untransposed column-major M x K operand, whose
// rows are strided: a thread per row over a chunk of kch columns (the reads
// of a warp are contiguous), the chunks' maxima merged by an integer
// atomicMax on the bit patterns (order-free, so the same maximum), then
// exponents_of_max.
constexpr int OZ_MAX_KCH = 64;
__global__ void row_absmax_strided(const double* A, int64_t lda, int64_t M, int64_t K, unsigned long long* mx) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M) return;
  const int64_t k0 = (int64_t)blockIdx.y * OZ_MAX_KCH;
  const int64_t k1 = (k0 + OZ_MAX_KCH < K) ? k0 + OZ_MAX_KCH : K;
  unsigned long long m = 0;
  for (int64_t k = k0; k < k1; ++k) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(A[i + k * lda]) & 0x7FFFFFFFFFFFFFFFull;
    m = u > m ? u : m;
  }
  if (m != 0) atomicMax(&mx[i], m);
}
__global__ void exponents_of_max(const unsigned long long* mx, int64_t M, int* ex, int* nonfinite) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M) return;
  ex[i] = exponent_above(mx[i]);
  if (nonfinite && (mx[i] >> 52) == 2047) *nonfinite = 1;
}

// Fraction bits of D digits of radix 2^r: r D - 1 (the leading digit reaches
// 2^w = 2^(r-1) itself), one less for r D = 64 so that the biased integer below
// fits 64 bits.
__host__ __device__ inline int digit_frac_bits(int w, int D) {
  const int rb = w + 1;
  return (rb * D == 64) ? 62 : rb * D - 1;
}

// Slices of op(A) (M x K): S[p][i][k] (k contiguous, Kp >= K, zero padded).
// An entry a of a row of exponent e becomes the integer
// U = round(a 2^(t - e)), |U| <= 2^t, read off as balanced digits: adding
// 2^w in every digit place makes all digits nonnegative, so digit p is a bit
// field of V = U + sum_i 2^(r i + w), less 2^w (the leading field takes the
// bits above it: it may reach 2^r).
__device__ __forceinline__ unsigned long long biased_digits(double a, int e, int tb, unsigned long long bias) {
  // |a| = m 2^(E - 1075) (m with its hidden bit; subnormals take E = 1)
  const unsigned long long bitsA = (unsigned long long)__double_as_longlong(a);
  const int E = (int)((bitsA >> 52) & 0x7FF);
  const unsigned long long mant = (bitsA & 0xFFFFFFFFFFFFFull) | (E ? (1ull << 52) : 0ull);
  const int sh = (E ? E : 1) - 1075 + tb - e;
  unsigned long long u;
  if (sh >= 0) u = (sh >= 64) ? 0ull : (mant << sh);
  else u = (sh < -53) ? 0ull : ((mant + (1ull << (-sh - 1))) >> -sh);
  return ((long long)bitsA < 0) ? bias - u : bias + u;
}
__host__ __device__ inline unsigned long long digit_bias(int w, int D) {
  unsigned long long b = 0;
  for (int i = 0; i < D; ++i) b |= 1ull << ((w + 1) * i + w);
  return b;
}
// A field f of 0..2^9 less 2^w as a float: f is put into the low bits of
// 2^23's pattern, which one exact subtraction turns into the integer (no
// conversion instruction).
__device__ __forceinline__ float field_value(uint32_t f, float off) { return __uint_as_float(0x4B000000u | f) - off; }

// The bits of |a| 2^-e (a of a row of exponent e, so below 1) as BF16, rounded
// towards zero; a nonzero entry below 2^-60 (or subnormal) counts as 2^-60.
__device__ __forceinline__ uint32_t magnitude_bits(double a, int e) {
  const unsigned long long t = (unsigned long long)__double_as_longlong(a) & 0x7FFFFFFFFFFFFFFFull;
  if (t == 0) return 0u;
  const int E = (int)(t >> 52), f = E - 1023 - e + 127;
  return (E == 0 || f < 67) ? 67u << 7 : ((uint32_t)f << 7) | (uint32_t)((t >> 45) & 127u);
}

// The D digits of one entry a of row i (exponent e = ex[i]) into S[p * pstride].
__device__ __forceinline__ void write_digits(double a, int e, int D, int w, __nv_bfloat16* S, int64_t pstride) {
  const int rb = w + 1;
  if (rb * D <= 64) {
    const unsigned long long v = biased_digits(a, e, digit_frac_bits(w, D), digit_bias(w, D));
    const float off = 8388608.0f + (float)(1 << w);
    for (int p = 0; p < D; ++p) {
      uint32_t f = (uint32_t)(v >> (rb * (D - 1 - p)));
      if (p > 0) f &= (1u << rb) - 1u;
      S[p * pstride] = __float2bfloat16_rn(field_value(f, off));
    }
  } else {  // more than 64 bits: the digits peeled one by one in FP64 (every step exact)
    double x = ldexp(a, -e);
    for (int p = 0; p < D; ++p) {
      const double y = ldexp(x, p == 0 ? w : rb);
      const double q = rint(y);
      S[p * pstride] = __float2bfloat16_rn((float)q);
      x = y - q;
    }
  }
}

__global__ void make_slices(const double* A, int64_t lda, bool trans, int64_t M, int64_t K,
                            int64_t Kp, const int* ex, int D, int w, int mag, __nv_bfloat16* S) {
  const int64_t total = M * Kp;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    int64_t i, k;
    if (trans) { k = t % Kp; i = t / Kp; } else { i = t % M; k = t / M; }
    const double a = (k < K) ? (trans ? A[k + i * lda] : A[i + k * lda]) : 0.0;
    write_digits(a, ex[i], D, w, S + i * Kp + k, M * Kp);
    if (mag) S[D * M * Kp + i * Kp + k] = __ushort_as_bfloat16((unsigned short)magnitude_bits(a, ex[i]));
  }
}

// One digit (shift rs, field mask) of eight entries as a 16-byte store.
__device__ __forceinline__ void put_eight(const unsigned long long (&v)[8], int rs, uint32_t mask, float off,
                                          __nv_bfloat16* out) {
  uint32_t o[4];
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    const __nv_bfloat162 two = __floats2bfloat162_rn(field_value((uint32_t)(v[2 * h] >> rs) & mask, off),
                                                     field_value((uint32_t)(v[2 * h + 1] >> rs) & mask, off));
    o[h] = *reinterpret_cast<const uint32_t*>(&two);
  }
  *reinterpret_cast<uint4*>(out) = make_uint4(o[0], o[1], o[2], o[3]);
}

// Eight magnitudes as a 16-byte store.
__device__ __forceinline__ void put_eight(const uint32_t (&m)[8], __nv_bfloat16* out) {
  *reinterpret_cast<uint4*>(out) =
      make_uint4(m[0] | m[1] << 16, m[2] | m[3] << 16, m[4] | m[5] << 16, m[6] | m[7] << 16);
}

// The slices of an operand whose rows are contiguous (trans), for r D <= 64:
// a thread takes eight consecutive entries of a row and writes each digit's
// eight BF16 values as one 16-byte store (Kp is a multiple of 64, so every
// store is aligned); the digits are those of write_digits.  MAG: the magnitudes
// are one plane more.
template <bool MAG>
__global__ void make_slices_rows(const double* A, int64_t lda, int64_t M, int64_t K, int64_t Kp,
                                 const int* ex, int D, int w, __nv_bfloat16* S) {
  const int64_t per_row = Kp / 8, total = M * per_row;
  const int rb = w + 1, tb = digit_frac_bits(w, D);
  const unsigned long long bias = digit_bias(w, D);
  const float off = 8388608.0f + (float)(1 << w);
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = t / per_row, k0 = (t % per_row) * 8;
    const int e = ex[i];
    unsigned long long v[8];
    uint32_t m[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const double a = (k0 + q < K) ? A[k0 + q + i * lda] : 0.0;
      v[q] = biased_digits(a, e, tb, bias);
      if (MAG) m[q] = magnitude_bits(a, e);
    }
    if (MAG) put_eight(m, S + ((int64_t)D * M + i) * Kp + k0);
    for (int p = 0; p < D; ++p) put_eight(v, rb * (D - 1 - p), p > 0 ? (1u << rb) - 1u : 0xFFFFFFFFu, off,
                                          S + ((int64_t)p * M + i) * Kp + k0);
  }
}

// The same slices of an untransposed column-major operand (rows strided), for
// r D <= 64: 64 x 64 tiles of (i, k) staged in shared memory, read along i and
// written along k, a digit's eight consecutive values of a row as one 16-byte
// store, so that eight lanes fill a 128-byte line (a 2-byte store per lane and
// digit before: exponents and slices of an 8835 x 8835 operand at 7 digits 0.77
// -> 0.58 ms).  256 threads; grid (ceil(M / 64), Kp / 64).
template <bool MAG>
__global__ void __launch_bounds__(256) make_slices_strided(const double* A, int64_t lda, int64_t M, int64_t K,
                                                           int64_t Kp, const int* ex, int D, int w, __nv_bfloat16* S) {
  __shared__ double tile[64][65];
  const int64_t i0 = (int64_t)blockIdx.x * 64, k0 = (int64_t)blockIdx.y * 64;
  for (int t = threadIdx.x; t < 64 * 64; t += 256) {
    const int64_t i = i0 + t % 64, k = k0 + t / 64;
    tile[t / 64][t % 64] = (i < M && k < K) ? A[i + k * lda] : 0.0;
  }
  __syncthreads();
  const int rb = w + 1, tb = digit_frac_bits(w, D);
  const unsigned long long bias = digit_bias(w, D);
  const float off = 8388608.0f + (float)(1 << w);
  const int kk = (threadIdx.x & 7) * 8;
  for (int r = threadIdx.x >> 3; r < 64; r += 32) {
    const int64_t i = i0 + r;
    if (i >= M) break;
    const int e = ex[i];
    unsigned long long v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = biased_digits(tile[kk + q][r], e, tb, bias);
    if (MAG) {
      uint32_t m[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) m[q] = magnitude_bits(tile[kk + q][r], e);
      put_eight(m, S + D * M * Kp + i * Kp + k0 + kk);
    }
    for (int p = 0; p < D; ++p) put_eight(v, rb * (D - 1 - p), p > 0 ? (1u << rb) - 1u : 0xFFFFFFFFu, off,
                                          S + ((int64_t)p * M + i) * Kp + k0 + kk);
  }
}

__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// C tile 64 x 64 per CTA, 4 warps of 32 x 32 (2 x 4 mma tiles each).
__global__ void __launch_bounds__(OZ_NT)
ozaki_kernel(const __nv_bfloat16* __restrict__ SA, const __nv_bfloat16* __restrict__ SB,
             const int* __restrict__ ea, const int* __restrict__ eb, int64_t M, int64_t N,
             int64_t arows, int64_t Kp, int s, int bits, int64_t chunk, double alpha, double beta, double* C,
             int64_t ldc, bool lower) {  // arows: rows of A's slices, of which M are multiplied
  __shared__ uint32_t As[OZ_BM][OZ_LDS];
  __shared__ uint32_t Bs[OZ_BN][OZ_LDS];
  const int64_t m0 = (int64_t)blockIdx.x * OZ_BM, n0 = (int64_t)blockIdx.y * OZ_BN;
  if (lower && m0 + OZ_BM - 1 < n0) return;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, tg = lane & 3;
  const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
  double sum[2][4][4];
  float acc[2][4][4];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int c = 0; c < 4; ++c) sum[a][b][c] = 0.0;

  for (int p = 0; p < s; ++p) {
    for (int q = 0; p + q < s; ++q) {  // slices p, q (0-based): p + q <= s - 1
      const __nv_bfloat16* Ap = SA + (int64_t)p * arows * Kp;
      const __nv_bfloat16* Bq = SB + (int64_t)q * N * Kp;
      const double scale = ldexp(1.0, (bits + 1) * (2 * s - 2 - p - q) - 2 * digit_frac_bits(bits, s));
      for (int64_t c0 = 0; c0 < Kp; c0 += chunk) {
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[a][b][c] = 0.f;
        const int64_t cend = (c0 + chunk < Kp) ? c0 + chunk : Kp;
        for (int64_t k0 = c0; k0 < cend; k0 += OZ_BK) {
          // 64 rows x 32 bf16 = 64 x 16 words per operand; 128 threads x 8 words each
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            const int idx = tid + r * OZ_NT;  // 0 .. 1023
            const int row = idx >> 4, w = idx & 15;
            const int64_t gm = m0 + row, gn = n0 + row;
            As[row][w] = (gm < M) ? reinterpret_cast<const uint32_t*>(Ap + gm * Kp + k0)[w] : 0u;
            Bs[row][w] = (gn < N) ? reinterpret_cast<const uint32_t*>(Bq + gn * Kp + k0)[w] : 0u;
          }
          __syncthreads();
#pragma unroll
          for (int kk = 0; kk < OZ_BK / 2; kk += 8) {  // two k16 steps (8 words each)
            uint32_t af[2][4], bf[4][2];
#pragma unroll
            for (int a = 0; a < 2; ++a) {
              const int r0 = wm + a * 16 + g;
              af[a][0] = As[r0][kk + tg];
              af[a][1] = As[r0 + 8][kk + tg];
              af[a][2] = As[r0][kk + tg + 4];
              af[a][3] = As[r0 + 8][kk + tg + 4];
            }
#pragma unroll
            for (int b = 0; b < 4; ++b) {
              const int c = wn + b * 8 + g;
              bf[b][0] = Bs[c][kk + tg];
              bf[b][1] = Bs[c][kk + tg + 4];
            }
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
              for (int b = 0; b < 4; ++b) mma_bf16(acc[a][b], af[a], bf[b]);
          }
          __syncthreads();
        }
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int c = 0; c < 4; ++c) sum[a][b][c] = fma((double)acc[a][b][c], scale, sum[a][b][c]);
      }
    }
  }
  // epilogue: c0,c1 at (g, 2tg..), c2,c3 at (g + 8, 2tg..)
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int64_t gm = m0 + wm + a * 16 + g + ((c >> 1) << 3);
        const int64_t gn = n0 + wn + b * 8 + 2 * tg + (c & 1);
        if (gm >= M || gn >= N || (lower && gm < gn)) continue;
        const double v = ldexp(sum[a][b][c], ea[gm] + eb[gn]);
        double* cp = C + gm + gn * ldc;
        *cp = (beta == 0.0) ? alpha * v : alpha * v + beta * *cp;
      }
}


// ----------------------------------------------------------------------------
// tcgen05 route.  A work item is one output tile (128 rows of op(A) x TCN
// columns of op(B)) and one group of digit pairs of a diagonal p + q = dg (all
// of them, or a few when the tiles alone do not fill the SMs): its CTA adds the
// pairs' exact chunk sums in int32 and stores them to the item's plane of an
// int32 array; combine_planes then forms C.  Warp 0: TMA producer; warp 1: TMEM
// owner and MMA issuer; TCN / 16 epilogue warps, each one quarter of the TMEM
// lanes and 64 columns: a thread keeps 64 sums, which fit its registers at
// every tile width (folding each diagonal into C in FP64 here kept the
// epilogue to 8 warps, whose 96 or 128 sums spilled, and held the MMAs up).
//
// Tiles: 128 x 256 moves 48 KB of slices per 4.2 MFLOP k-block against 32 KB
// per 2.1 MFLOP at 128 x 128, with four stages instead of six and two
// accumulators in the 512 TMEM columns instead of four.  Bound: the MMAs and
// their shared-memory feed.  GB300, 8810 x 8810 x 8810 at 7 slices (28 pairs,
// 3.83e13 flop): 256 columns 27.6 ms (1.39 PFLOP/s), 192 31.3 ms, against 38.9
// at 192 with the folds; outputs of few columns, whose tiles now share the SMs
// by diagonals: 2867 x 7 x 2867 0.44 -> 0.10 ms.
// ----------------------------------------------------------------------------
constexpr int TC_M = 128, TC_KB = 64;
constexpr int TC_EPI_COLS = 64;  // columns per epilogue thread
constexpr int TC_A_BYTES = TC_M * TC_KB * 2;
template <int TCN>
struct OzTile {
  static_assert(TCN == 128 || TCN == 192 || TCN == 256, "tile width 128, 192 or 256");
  static constexpr int STAGES = (TCN == 256) ? 4 : (TCN == 192) ? 5 : 6;
  static constexpr int B_BYTES = TCN * TC_KB * 2;
  static constexpr int STAGE_BYTES = TC_A_BYTES + B_BYTES;
  static constexpr int EPI_WARPS = TCN / TC_EPI_COLS * 4;
  static constexpr int THREADS = 64 + 32 * EPI_WARPS;
  // FP32 chunk accumulators in the 512 TMEM columns: four at 128 columns,
  // two at 192 or 256; the allocation is the whole (power-of-two) 512 columns
  static constexpr int NBUF = 512 / TCN;
  static constexpr uint32_t TMEM_COLS = 512;
  // kind::f16 instruction descriptor: D F32, A and B BF16, both K-major, M 128, N TCN.
  static constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TCN >> 3) << 17) |
                                    ((uint32_t)(TC_M >> 4) << 24);
};

// 2^e for e in [-1022, 1023], from its bit pattern.
__device__ __forceinline__ double pow2i(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }

// The digit pairs (p, q = dg - p) of one item, for D digits, nchunk K-chunks and
// at most U pairs per item: diagonals from the longest (dg = D - 1) down, so that
// the longest items start first.  An item adds at most kMaxChunks chunk sums,
// which fit 31 bits (127 2^24 < 2^31); K beyond that many chunks is multiplied
// in ranges (see ozaki_gemm).
// Guarded products (see ozaki_gemm) keep one diagonal more, dg = D, and have a
// last item that multiplies the magnitudes (plane D of both operands).
constexpr int kMaxChunks = 127;
struct OzParts {
  int D, U, nchunk, guard;
  __host__ __device__ int top() const { return D - 1 + guard; }
  __host__ __device__ int pairs(int dg) const { return dg < D ? dg + 1 : 2 * D - 1 - dg; }
  __host__ __device__ int of_diag(int dg) const { return (pairs(dg) + U - 1) / U; }
  __host__ __device__ int count() const {  // items of digits
    int t = 0;
    for (int dg = 0; dg <= top(); ++dg) t += of_diag(dg);
    return t;
  }
  __host__ __device__ int items() const { return count() + guard; }
  __device__ void get(int part, int* dg, int* p0, int* p1) const {
    int d = top();
    while (d >= 0 && part >= of_diag(d)) part -= of_diag(d--);
    if (d < 0) {  // the magnitudes
      *dg = 2 * D;
      *p0 = D;
      *p1 = D + 1;
      return;
    }
    const int first = d < D ? 0 : d - D + 1, end = first + pairs(d);
    *dg = d;
    *p0 = first + part * U;
    *p1 = (*p0 + U < end) ? *p0 + U : end;
  }
};
// A plane: M x N column-major, or (lower, M >= N) its columns from the diagonal
// down, packed.  plane_column(j) + i is entry (i, j).
__host__ __device__ inline int64_t plane_size(int64_t M, int64_t N, bool lower) {
  return lower ? M * N - N * (N - 1) / 2 : M * N;
}
__host__ __device__ inline int64_t plane_column(int64_t j, int64_t M, bool lower) {
  return lower ? j * M - j * (j + 1) / 2 : j * M;
}
// U: all pairs of a diagonal, fewer when the longest item would then exceed an
// even share of all pairs over the SMs (a function of the sizes alone, so that
// the workspace and the sums do not depend on the context).
inline OzParts oz_parts(int64_t M, int64_t N, int64_t Kp, int D, int w, bool lower, bool guard) {
  OzParts o;
  const int64_t chunk = (int64_t)1 << (24 - 2 * w);
  o.D = D;
  o.guard = (guard && D > 1) ? 1 : 0;
  o.nchunk = (int)cdiv(Kp, chunk);
  const int64_t tiles = cdiv(M, TC_M) * cdiv(N, TC_M) / (lower ? 2 : 1);
  const int64_t even = cdiv(std::max<int64_t>(tiles, 1) * (D * (D + 1) / 2 + o.guard * D), 152);
  o.U = (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(D, even), kMaxChunks / o.nchunk));
  return o;
}

// Order of the output tiles over the CTAs: groups of G consecutive tile rows;
// inside a group, the G rows of one tile column are consecutive CTAs, then
// the next column.  The CTAs resident at one time then cover a G x (152 / G)
// block of tiles, whose A rows and B columns L2 holds while every CTA of the
// block streams them (in the plain order a wave spans every tile row, so each
// slice pair re-streams all of A).  With `lower`, a group only has the columns
// up to its last row: tiles entirely above the diagonal are not enumerated.
// The host sizes the grid with the same count (ozaki_tile_count).  Tiles
// are TCM rows by TCN columns; with `lower`, a group of tile rows ending at
// tile row r needs the tile columns that start at or below row r TCM + TCM - 1.
__host__ __device__ inline int ozaki_group_cols(int g0, int Gg, int TN, int TCM, int TCN, bool lower) {
  if (!lower) return TN;
  const int64_t last_row = (int64_t)(g0 + Gg - 1) * TCM + TCM - 1;
  const int64_t c = last_row / TCN + 1;
  return (int)(c < TN ? c : TN);
}
__host__ __device__ inline int64_t ozaki_tile_count(int TM, int TN, int G, bool lower, int TCM, int TCN) {
  int64_t tot = 0;
  for (int g0 = 0; g0 < TM; g0 += G) {
    const int Gg = (TM - g0 < G) ? TM - g0 : G;
    tot += (int64_t)Gg * ozaki_group_cols(g0, Gg, TN, TCM, TCN, lower);
  }
  return tot;
}
__device__ __forceinline__ void ozaki_tile_of(int64_t idx, int TM, int TN, int G, bool lower, int TCM, int TCN,
                                              int* tm, int* tn) {
  int64_t base = 0;
  for (int g0 = 0; g0 < TM; g0 += G) {
    const int Gg = (TM - g0 < G) ? TM - g0 : G;
    const int ncol = ozaki_group_cols(g0, Gg, TN, TCM, TCN, lower);
    const int64_t cnt = (int64_t)Gg * ncol;
    if (idx < base + cnt) {
      const int r = (int)(idx - base);
      *tn = r / Gg;
      *tm = g0 + r % Gg;
      return;
    }
    base += cnt;
  }
  *tm = TM;  // past the end: no tile
  *tn = 0;
}

// CS = 2: a cluster of CS CTAs takes CS consecutive tile rows of one tile
// column.  They need the same B tile, so each CTA loads 1/CS of it (TCN / CS
// rows of op(B)) with one TMA multicast into the same stage of every CTA of
// the cluster: the L2-to-SM bytes per k-block drop from A + B to A + B / CS.
// A stage may then be refilled only once all CS CTAs have consumed it, so
// every MMA warp's stage-release commit is multicast to the empty barriers of
// the whole cluster, which count CS arrivals.  Every CTA of a cluster runs
// the whole pipeline (its peers need its share of B), also when its tile
// lies past the last row or above the diagonal; its epilogue then writes
// nothing.
template <int TCN, int CS, bool GUARD>
__global__ void __launch_bounds__(OzTile<TCN>::THREADS, 1)
ozaki_tc_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, int64_t M, int64_t N,
                int64_t Kp, OzParts parts, int64_t chunk, int tiles, int32_t* P, int lower, int group, long long limit,
                int32_t* status) {
  constexpr int TC_N = TCN, TC_STAGES = OzTile<TCN>::STAGES;
  constexpr int TC_STAGE_BYTES = OzTile<TCN>::STAGE_BYTES, TC_EPI_WARPS = OzTile<TCN>::EPI_WARPS;
  constexpr uint32_t TC_TMEM_COLS = OzTile<TCN>::TMEM_COLS, TC_IDESC = OzTile<TCN>::IDESC;
  constexpr int NBUF = OzTile<TCN>::NBUF;
  constexpr int B_ROWS = TCN / CS;  // rows of the B tile this CTA loads (and multicasts)
  static_assert(CS == 1 || CS == 2 || CS == 4, "cluster of 1, 2 or 4 CTAs");
  static_assert((B_ROWS * 128) % 1024 == 0, "a B share starts on a 128-byte-swizzle atom");
  extern __shared__ __align__(1024) unsigned char tc_smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)tc_smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full_bar[TC_STAGES], empty_bar[TC_STAGES];
  __shared__ __align__(8) uint64_t acc_full[OzTile<TCN>::NBUF], acc_empty[OzTile<TCN>::NBUF], done_bar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int TM = (int)((M + TC_M - 1) / TC_M), TN = (int)((N + TC_N - 1) / TC_N);
  const int rank = (CS > 1) ? (int)cluster_ctarank() : 0;
  // items: all tiles (or clusters of tiles) of the first group of pairs, then of the next
  const int unit = (int)(blockIdx.x / CS), part = unit / tiles, tile = unit - part * tiles;
  int dg, pbeg, pend;
  parts.get(part, &dg, &pbeg, &pend);
  const int nchunk = parts.nchunk;
  int tm, tn;
  if (CS == 1) {
    ozaki_tile_of(tile, TM, TN, group, lower != 0, TC_M, TC_N, &tm, &tn);
    if (tm >= TM || tn >= TN) return;
    if (lower && (int64_t)tm * TC_M + TC_M - 1 < (int64_t)tn * TC_N) return;  // tile above the diagonal
  } else {
    // the grid holds whole clusters of CS tile rows: no CTA leaves early
    int tc;
    ozaki_tile_of(tile, (TM + CS - 1) / CS, TN, group, lower != 0, CS * TC_M, TC_N, &tc, &tn);
    tm = tc * CS + rank;
  }
  const int64_t m0 = (int64_t)tm * TC_M, n0 = (int64_t)tn * TC_N;

  if (threadIdx.x == 0) {
    for (int i = 0; i < TC_STAGES; ++i) {
      mbar_init(&full_bar[i], 1);
      mbar_init(&empty_bar[i], CS);
    }
    for (int i = 0; i < NBUF; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], TC_EPI_WARPS);
    }
    mbar_init(&done_bar, 1);
    abort_sh = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_base_sh)),
                 "r"(TC_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  if (CS > 1) cluster_sync_all();  // every CTA's barriers exist before any multicast reaches them
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      int it = 0;
      bool ok = true;
      for (int p = pbeg; p < pend && ok; ++p)
          for (int c = 0; c < nchunk && ok; ++c) {
            const int q = dg - p;
            const int64_t c0 = (int64_t)c * chunk;
            const int nkb = (int)(((Kp - c0) < chunk ? (Kp - c0) : chunk) / TC_KB);
            for (int kb = 0; kb < nkb; ++kb, ++it) {
              const int st = it % TC_STAGES;
              if (!mbar_wait(&empty_bar[st], ((it / TC_STAGES) & 1) ^ 1, limit) || *(volatile int*)&abort_sh) {
                ok = false;
                break;
              }
              unsigned char* a = smem + st * TC_STAGE_BYTES;
              unsigned char* b = a + TC_A_BYTES;
              mbar_expect_tx(&full_bar[st], TC_STAGE_BYTES);  // A and the whole B tile (all CS shares)
              const int kc = (int)(c0 + kb * TC_KB);
              tma_load_3d(a, &mapA, &full_bar[st], kc, (int)m0, p);
              if (CS == 1)
                tma_load_3d(b, &mapB, &full_bar[st], kc, (int)n0, q);
              else
                tma_load_3d_multicast(b + rank * (B_ROWS * 128), &mapB, &full_bar[st], kc,
                                      (int)(n0 + rank * B_ROWS), q, (uint16_t)((1u << CS) - 1u));
            }
          }
      if (CS > 1 && ok) {
        // every peer's last releases of this CTA's stages have arrived: no
        // remote arrive can reach this CTA's barriers after it exits
        for (int j = (it > TC_STAGES ? it - TC_STAGES : 0); j < it && ok; ++j)
          ok = mbar_wait(&empty_bar[j % TC_STAGES], ((j / TC_STAGES) & 1), limit);
      }
      if (!ok) {
        atomicCAS(status, 0, FRACLAP_ERR_TIMEOUT);
        abort_sh = 1;
        // let the copies already issued land before the CTA can exit
        for (int j = (it > TC_STAGES ? it - TC_STAGES : 0); j < it; ++j)
          mbar_wait(&full_bar[j % TC_STAGES], (j / TC_STAGES) & 1, limit);
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      int it = 0, chunk_i = 0;
      bool ok = true;
      for (int p = pbeg; p < pend && ok; ++p)
          for (int c = 0; c < nchunk && ok; ++c, ++chunk_i) {
            const int buf = chunk_i % NBUF;
            if (!mbar_wait(&acc_empty[buf], ((chunk_i / NBUF) & 1) ^ 1, limit) || *(volatile int*)&abort_sh) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t d = tmem + (uint32_t)(buf * TC_N);
            const int64_t c0 = (int64_t)c * chunk;
            const int nkb = (int)(((Kp - c0) < chunk ? (Kp - c0) : chunk) / TC_KB);
            for (int kb = 0; kb < nkb; ++kb, ++it) {
              const int st = it % TC_STAGES;
              if (!mbar_wait(&full_bar[st], (it / TC_STAGES) & 1, limit) || *(volatile int*)&abort_sh) {
                ok = false;
                break;
              }
              tc_fence_after();
              const uint32_t a = smem_u32(smem + st * TC_STAGE_BYTES);
              const uint32_t b = a + TC_A_BYTES;
#pragma unroll
              for (int kk = 0; kk < TC_KB / 16; ++kk)  // K = 16 per instruction: 32 bytes
                umma<false>(d, sdesc_k128(a + kk * 32), sdesc_k128(b + kk * 32), TC_IDESC, (kb > 0 || kk > 0) ? 1u : 0u);
              if (CS == 1)
                umma_commit(&empty_bar[st]);  // frees the stage once these MMAs have read it
              else
                umma_commit_multicast(&empty_bar[st], (uint16_t)((1u << CS) - 1u));  // in every CTA of the cluster
            }
            if (!ok) break;
            umma_commit(&acc_full[buf]);  // the chunk's accumulator is complete
          }
      if (!ok) {
        atomicCAS(status, 0, FRACLAP_ERR_TIMEOUT);
        abort_sh = 1;
      }
      umma_commit(&done_bar);  // every MMA issued so far has finished when this fires
      mbar_wait(&done_bar, 0, limit);
    }
  } else {
    // ---------------- epilogue: exact integer sums ----------------
    // A chunk sum is an integer of at most 2^24 (exact in FP32), so it converts
    // exactly to int32, and an item's at most kMaxChunks of them add exactly.
    const int lg = warp & 3;                          // TMEM lane quarter of this warp
    const int cbase = ((warp - 2) >> 2) * TC_EPI_COLS;  // this warp's columns of the tile
    const int64_t row = m0 + lg * 32 + lane;          // output row of this thread
    int acc[TC_EPI_COLS];
#pragma unroll
    for (int j = 0; j < TC_EPI_COLS; ++j) acc[j] = 0;
    const int nacc = (pend - pbeg) * nchunk;
    const bool magnitudes = GUARD && pbeg == parts.D;
    bool ok = true;
    for (int chunk_i = 0; chunk_i < nacc; ++chunk_i) {
      const int buf = chunk_i % NBUF;
      if (!mbar_wait(&acc_full[buf], (chunk_i / NBUF) & 1, limit) || *(volatile int*)&abort_sh) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t taddr = tmem + ((uint32_t)(lg * 32) << 16) + (uint32_t)(buf * TC_N + cbase);
#pragma unroll
      for (int j0 = 0; j0 < TC_EPI_COLS; j0 += 16) {
        uint32_t r[16];
        tmem_ld16(taddr + j0, r);
        tmem_wait_ld();
        if (!magnitudes) {
#pragma unroll
          for (int j = 0; j < 16; ++j) acc[j0 + j] += __float2int_rz(__uint_as_float(r[j]));
        } else {  // a sum of FP32, in the same registers
#pragma unroll
          for (int j = 0; j < 16; ++j) acc[j0 + j] = __float_as_int(__int_as_float(acc[j0 + j]) + __uint_as_float(r[j]));
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[buf]);
    }
    if (ok && row < M) {
      int32_t* out = P + part * plane_size(M, N, lower != 0) + row;
#pragma unroll
      for (int j = 0; j < TC_EPI_COLS; ++j) {
        const int64_t col = n0 + cbase + j;
        if (col < N && !(lower && row < col)) out[plane_column(col, M, lower != 0)] = acc[j];
      }
    }
    if (!ok) {
      if (lane == 0) atomicCAS(status, 0, FRACLAP_ERR_TIMEOUT);
      abort_sh = 1;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_TMEM_COLS)
                 : "memory");
  }
  if (CS > 1) cluster_sync_all();  // no CTA leaves while a peer may still signal it
}

// C = alpha 2^(e_i + f_j - 2t + r (2D - 2)) sum_dg 2^(-r dg) P_dg + beta C from the
// items' planes.  Up to four diagonals at a time are one exact 64-bit integer: a
// diagonal is at most D kMaxChunks chunk sums of 2^24, below 2^34.2, and three
// shifts of at most 9 bits follow, so that a group stays below 2^61.3.  An
// element costs a conversion and an FMA per four diagonals; the lowest diagonals
// are added first.  Guarded (never lower): a column of 32 rows with an entry whose
// sum of magnitudes is neither 0 nor at least kGuardSum is marked (i0, j0: the
// block's place in C, rows32: tiles along the rows).
__global__ void combine_planes(const int32_t* __restrict__ P, const int* __restrict__ ea, const int* __restrict__ eb,
                               int64_t M, int64_t N, OzParts parts, int w, double alpha, double beta, double* C,
                               int64_t ldc, int lower, unsigned* marks, int64_t i0, int64_t j0, int64_t rows32) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = plane_size(M, N, lower != 0);
  const unsigned lanes = __ballot_sync(0xffffffffu, i < M);
  if (i >= M) return;
  const int rb = w + 1, D = parts.D;
  const int e0 = ea[i] - 2 * digit_frac_bits(w, D) + rb * (2 * D - 2);
  for (int64_t j = blockIdx.y; j < N; j += gridDim.y) {
    if (lower && i < j) break;
    const int32_t* q = P + i + plane_column(j, M, lower != 0);
    double v = 0.0;
    int plane = 0;
    for (int d = parts.top(); d >= 0;) {  // planes from the highest dg (lowest weight) up
      const int lo = (d >= 4) ? d - 3 : 0, g = d - lo + 1;
      long long acc = 0;  // in units of 2^(-rb d), d the group's highest diagonal
      for (int sh = 0; d >= lo; --d, sh += rb) {
        long long t = 0;
        for (int u = parts.of_diag(d); u > 0; --u, ++plane) t += __ldcs(q + plane * stride);
        acc += t * (1ll << sh);
      }
      v = v * pow2i(-4 * rb) + (double)acc;  // every group but the last holds four diagonals
      if (d >= 0) continue;
      int e = e0 + eb[j] - rb * (g - 1);
      // two exact power-of-two steps (each factor normal); beyond |e| = 2044 the
      // result is 0 or infinite either way
      e = (e < -2044) ? -2044 : (e > 2044 ? 2044 : e);
      const int e1 = e / 2;
      v = alpha * ((v * pow2i(e1)) * pow2i(e - e1));
    }
    double* c = C + i + j * ldc;
    *c = (beta == 0.0) ? v : v + beta * *c;
    if (parts.guard) {
      const float sum = __int_as_float(__ldcs(q + plane * stride));
      const bool mark = __any_sync(lanes, sum != 0.0f && !(sum >= kGuardSum));
      if (mark && threadIdx.x % 32 == 0)
        atomicOr(marks + ((j0 + j) / kGuardCols * rows32 + (i0 + i) / kGuardRows), 1u << ((j0 + j) % kGuardCols));
    }
  }
}

// 3-D map over `rows` rows of the slices S[s][of][Kp] (bf16), box 64 (K) x box_rows x 1.
bool slice_map(CUtensorMap* map, const __nv_bfloat16* S, int64_t rows, int64_t of, int64_t Kp, int s, int box_rows) {
  EncodeTiledFn fn = encode_tiled();
  if (!fn) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)Kp, (cuuint64_t)rows, (cuuint64_t)s};
  const cuuint64_t strides[2] = {(cuuint64_t)Kp * 2, (cuuint64_t)of * Kp * 2};
  const cuuint32_t box[3] = {TC_KB, (cuuint32_t)box_rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, (void*)S, dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
template <int TCN, int CS, bool GUARD>
int launch_tc(fraclap_ctx* ctx, const __nv_bfloat16* SA, const __nv_bfloat16* SB, int64_t M, int64_t N, int64_t arows,
              int64_t Kp, const OzParts& parts, int64_t chunk, int32_t* P, bool lower, cudaStream_t st) {
  CUtensorMap ma, mb;
  const int planes = parts.D + parts.guard;
  FL_CHECK(ctx, slice_map(&ma, SA, M, arows, Kp, planes, TC_M) && slice_map(&mb, SB, N, N, Kp, planes, TCN / CS),
           FRACLAP_ERR_CUDA, "ozaki_gemm: tensor map encoding failed");
  const size_t smem = (size_t)OzTile<TCN>::STAGES * OzTile<TCN>::STAGE_BYTES + 1024;
  auto kern = ozaki_tc_kernel<TCN, CS, GUARD>;
  FL_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  // the raster counts clusters of CS tile rows (a tile of CS * 128 rows)
  const int TM = (int)cdiv(cdiv(M, TC_M), CS), TN = (int)cdiv(N, TCN);
  const int G = std::max(1, std::min(ctx->oz_group > 0 ? ctx->oz_group : TM, TM));
  const int64_t tiles = ozaki_tile_count(TM, TN, G, lower, CS * TC_M, TCN);
  FL_CHECK(ctx, tiles * parts.items() * CS <= INT32_MAX, FRACLAP_ERR_UNSUPPORTED, "ozaki_gemm: too many tiles");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(tiles * parts.items() * CS));
  cfg.blockDim = dim3(OzTile<TCN>::THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)CS;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = (CS > 1) ? 1 : 0;
  FL_CUDA(ctx, cudaLaunchKernelEx(&cfg, kern, ma, mb, M, N, Kp, parts, chunk, (int)tiles, P, lower ? 1 : 0, G,
                                  ctx->wait_cycles, ctx->d_status));
  return 0;
}

}  // namespace

// The longest K of one pass: kMaxChunks chunks of digits of magnitude w.
static int64_t oz_range(int w) { return (int64_t)kMaxChunks << (24 - 2 * w); }
// The most digits that s slices are cut into (see ozaki_gemm), and the most
// planes of the tensor-core route for up to that many, at either digit width.
static int max_digits(int s) { return (s <= 5 || s == 8) ? s + 1 : s; }
static int max_planes(int64_t M, int64_t N, int64_t Kp, int D, bool lower, bool guard) {
  int t = 0;
  for (int d = 1; d <= D; ++d)
    for (int w = 7; w <= 8; ++w) t = std::max(t, oz_parts(M, N, std::min(Kp, oz_range(w)), d, w, lower, guard).items());
  return t;
}
static int64_t padded(int64_t K) { return cdiv(std::max<int64_t>(K, 1), OZ_KPAD) * OZ_KPAD; }

// The scratch of one range: A's digits, and for a block of C (mb rows of nb
// columns) B's digits and the planes.  The planes are four bytes an entry of C
// and item of the diagonals (7 to 28 of them for 7 slices), so C is formed block
// by block where they do not fit beside the digits: strips of columns, each with
// its own digits of B, and rows of a strip where even one tile column of all
// rows does not fit.
struct OzBlocks {
  int64_t mb, nb;
};
struct OzScratch {
  __nv_bfloat16 *SA, *SB;
  int *ea, *eb;
  unsigned long long* mx;
  int32_t* P;
};
static OzScratch oz_take(Arena* ar, int64_t M, OzBlocks c, int64_t Kp, int D, int planes, bool lower) {
  OzScratch w;
  w.SA = ar->take<__nv_bfloat16>((int64_t)D * M * Kp);
  w.SB = ar->take<__nv_bfloat16>((int64_t)D * c.nb * Kp);
  w.ea = ar->take<int>(M);
  w.eb = ar->take<int>(c.nb);
  w.mx = ar->take<unsigned long long>(std::max(M, c.nb));
  w.P = ar->take<int32_t>(planes * plane_size(c.mb, c.nb, lower));
  return w;
}
static size_t oz_bytes(int64_t M, OzBlocks c, int64_t Kp, int D, int planes, bool lower) {
  Arena ar;
  oz_take(&ar, M, c, Kp, D, planes, lower);
  return ar.off;
}
// The largest blocks that fit `room` bytes (mb = 0: none does): all of C, else
// even strips of a multiple of 256 columns, else even blocks of a multiple of 128
// rows of one such strip.
static OzBlocks oz_blocks(int64_t M, int64_t N, int64_t Kp, int D, int planes, bool lower, size_t room) {
  const auto fits = [&](int64_t mb, int64_t nb) { return oz_bytes(M, {mb, nb}, Kp, D, planes, lower) <= room; };
  const auto part = [](int64_t total, int64_t unit, int64_t count) { return std::min(total, cdiv(cdiv(total, count), unit) * unit); };
  if (fits(M, N)) return {M, N};
  const auto most = [&](int64_t total, int64_t unit, auto ok) {  // fewest even parts that fit, 0: none
    int64_t lo = 1, hi = cdiv(total, unit) + 1;
    while (lo < hi) {
      const int64_t c = (lo + hi) / 2;
      if (ok(part(total, unit, c))) hi = c;
      else lo = c + 1;
    }
    return lo > cdiv(total, unit) ? (int64_t)0 : part(total, unit, lo);
  };
  if (const int64_t nb = most(N, 256, [&](int64_t v) { return fits(M, v); })) return {M, nb};
  if (lower) return {0, 0};
  const int64_t nb = std::min<int64_t>(N, 256);
  return {most(M, 128, [&](int64_t v) { return fits(v, nb); }), nb};
}

// All of C in one block up to 4 GiB, or up to what the digits of s slices took
// without planes where that is more (16 (M + N) K bytes for 7 slices; `tight`:
// only that): no product needs more than it did when every diagonal was folded
// into C on the fly, but for small ones.
size_t ozaki_ws(int64_t M, int64_t N, int64_t K, int s, bool lower, int digits, bool tight, bool guard) {
  const int64_t Kp = padded(std::min(K, oz_range(7)));
  const int digs = (digits > 0) ? digits : max_digits(s), planes = max_planes(M, N, Kp, digs, lower, guard);
  const int D = digs + (guard ? 1 : 0);  // and the magnitudes
  const size_t whole = oz_bytes(M, {M, N}, Kp, D, planes, lower);
  const size_t least = oz_bytes(M, {lower ? M : std::min<int64_t>(M, 1024), std::min<int64_t>(N, 256)}, Kp, D, planes, lower);
  const size_t fold = align256((size_t)((8 * s + 6) / 7) * 2 * (size_t)(M + N) * (size_t)padded(K));
  return std::min(whole, std::max({least, fold, tight ? (size_t)0 : (size_t)4 << 30}));
}

// Exponents and digit slices of the rows of op(X) (R rows of length K):
// contiguous rows (trans) one block per row; strided rows through the
// column-parallel maximum and the tiled slicing.  More than 64 bits of digits
// take the general kernel.
int slice_operand(fraclap_ctx* ctx, const double* X, int64_t ldx, bool trans, int64_t R, int64_t K, int64_t Kp,
                  int sl, int bits, bool mag, int* ex, __nv_bfloat16* S, unsigned long long* mx, int* nonfinite,
                  cudaStream_t st) {
  const bool fits = sl * (bits + 1) <= 64;
  if (trans) {
    row_exponents<<<(unsigned)R, 256, 0, st>>>(X, ldx, K, ex, nonfinite);
  } else {
    FL_CUDA(ctx, cudaMemsetAsync(mx, 0, sizeof(unsigned long long) * (size_t)R, st));
    row_absmax_strided<<<dim3((unsigned)cdiv(R, 256), (unsigned)std::max<int64_t>(cdiv(K, OZ_MAX_KCH), 1)), 256, 0,
                         st>>>(X, ldx, R, K, mx);
    count_launch(ctx);
    exponents_of_max<<<(unsigned)cdiv(R, 256), 256, 0, st>>>(mx, R, ex, nonfinite);
  }
  count_launch(ctx);
  if (trans && fits) {
    const unsigned gs = (unsigned)std::min<int64_t>(cdiv(R * (Kp / 8), 256), 152 * 16);
    (mag ? make_slices_rows<true> : make_slices_rows<false>)<<<gs, 256, 0, st>>>(X, ldx, R, K, Kp, ex, sl, bits, S);
  } else if (fits) {  // (K of a range: both grids' second dimension is below 2100)
    (mag ? make_slices_strided<true> : make_slices_strided<false>)<<<dim3((unsigned)cdiv(R, 64), (unsigned)(Kp / 64)),
                                                                     256, 0, st>>>(X, ldx, R, K, Kp, ex, sl, bits, S);
  } else {
    const unsigned gs = (unsigned)std::min<int64_t>(cdiv(R * Kp, 256), 152 * 32);
    make_slices<<<gs, 256, 0, st>>>(X, ldx, trans, R, K, Kp, ex, sl, bits, mag ? 1 : 0, S);
  }
  count_launch(ctx);
  FL_CUDA(ctx, cudaGetLastError());
  return 0;
}

// One block of C from (i0, j0): M rows of A's slices (of `arows`), N columns of B's.
static int ozaki_block(fraclap_ctx* ctx, const OzScratch& z, const __nv_bfloat16* SA, const int* ea, int64_t M, int64_t N,
                       int64_t arows, int64_t Kp, const OzParts& parts, int bits, double alpha, double beta, double* C,
                       int64_t ldc, bool lower, const OzGuard* guard, int64_t i0, int64_t j0, cudaStream_t st) {
  const int64_t chunk = (int64_t)1 << (24 - 2 * bits);
  if (ctx->tensor_route == 1) {
    const int tw = (N <= 128) ? 128 : ctx->oz_tile_n;  // a narrow output takes the 128-column tile
    const int cs = ctx->oz_cluster;
#define FL_OZ_LAUNCH(W, K)                                                                          \
  (parts.guard ? launch_tc<W, K, true>(ctx, SA, z.SB, M, N, arows, Kp, parts, chunk, z.P, lower, st) \
               : launch_tc<W, K, false>(ctx, SA, z.SB, M, N, arows, Kp, parts, chunk, z.P, lower, st))
    if (cs == 2) {
      FL_TRY(tw == 256 ? FL_OZ_LAUNCH(256, 2) : tw == 192 ? FL_OZ_LAUNCH(192, 2) : FL_OZ_LAUNCH(128, 2));
    } else {
      FL_TRY(tw == 256 ? FL_OZ_LAUNCH(256, 1) : tw == 192 ? FL_OZ_LAUNCH(192, 1) : FL_OZ_LAUNCH(128, 1));
    }
#undef FL_OZ_LAUNCH
    count_launch(ctx);
    combine_planes<<<dim3((unsigned)cdiv(M, 256), (unsigned)std::min<int64_t>(N, 16384)), 256, 0, st>>>(
        z.P, ea, z.eb, M, N, parts, bits, alpha, beta, C, ldc, lower ? 1 : 0, guard ? guard->marks : nullptr, i0, j0,
        cdiv(arows, kGuardRows));
  } else {
    dim3 grid((unsigned)cdiv(M, OZ_BM), (unsigned)cdiv(N, OZ_BN));
    ozaki_kernel<<<grid, OZ_NT, 0, st>>>(SA, z.SB, ea, z.eb, M, N, arows, Kp, parts.D, bits, chunk, alpha, beta, C, ldc,
                                         lower);
  }
  count_launch(ctx);
  FL_CUDA(ctx, cudaGetLastError());
  return 0;
}

// One range of K (see ozaki_gemm): D digits of magnitude `bits` per operand.
static int ozaki_range(fraclap_ctx* ctx, bool ta, bool tb, int64_t M, int64_t N, int64_t K, double alpha, const double* A,
                       int64_t lda, const double* B, int64_t ldb, double beta, double* C, int64_t ldc, int D, int bits,
                       bool lower, Arena ar, cudaStream_t st, const OzGuard* guard) {
  const int64_t Kp = padded(K);
  const OzParts parts = oz_parts(M, N, Kp, D, bits, lower, guard != nullptr);
  const bool mag = parts.guard != 0;
  int* nonfinite = guard ? guard->nonfinite : nullptr;
  const OzBlocks c = oz_blocks(M, N, Kp, D + mag, parts.items(), lower, ar.cap - ar.off);
  FL_CHECK(ctx, c.mb > 0, FRACLAP_ERR_ALLOC, "ozaki_gemm: workspace too small");
  const OzScratch z = oz_take(&ar, M, c, Kp, D + mag, parts.items(), lower);
  // rows of op(A) and columns of op(B): contiguous when trans, else strided
  FL_TRY(slice_operand(ctx, A, lda, ta, M, K, Kp, D, bits, mag, z.ea, z.SA, z.mx, nonfinite, st));
  for (int64_t j = 0; j < N; j += c.nb) {
    const int64_t nb = std::min(c.nb, N - j);
    FL_TRY(slice_operand(ctx, B + (tb ? j : j * ldb), ldb, !tb, nb, K, Kp, D, bits, mag, z.eb, z.SB, z.mx, nonfinite, st));
    StageTimer tm(ctx, kStageSliceProducts, st);
    for (int64_t i = lower ? j : 0; i < M; i += lower ? M : c.mb) {
      const int64_t mb = lower ? M - j : std::min(c.mb, M - i);
      FL_TRY(ozaki_block(ctx, z, z.SA + i * Kp, z.ea + i, mb, nb, M, Kp, parts, bits, alpha, beta, C + i + j * ldc, ldc, lower,
                         guard, i, j, st));
    }
  }
  return 0;
}

// C = alpha op(A) op(B) + beta C, FP64-accurate through s BF16 slices
// (s = 7 for full FP64 accuracy of the products).  lower: only C(i,j), i >= j.
// digits > 0 sets the digits per operand itself (8 bits each at w = 7), width > 0
// their magnitude bits w.
// guard (may be null) keeps the diagonal p + q = D too and tells which entries
// the digits hold to the accuracy of an FP64 sum.  The digits are relative to
// the largest entry of the row of op(A) and the column of op(B); in units of
// 2^(e_i + f_j), an entry of C is off by at most K (2 2^-63 + 6 2^-70) < K 2^-61.9
// for 8 digits, an FP64 sum by K 2^-53 times the sum of its terms' magnitudes.  A
// product of the magnitudes (8 bits each, rounded down) gives that sum: where it
// is at least kGuardSum = 2^-8 the digits' bound is K 2^-53.9 of it, and where it
// is 0 every term is; columns of 32 rows with any other entry are marked for the
// caller's FP64 product (2^-6 marked 2 % of the tiles of the n = 8835 apply, the
// nodes beside the corners, for 0.4 ms more).  An infinity or NaN, which has no digits, sets *nonfinite: C is
// then meaningless.
int ozaki_gemm(fraclap_ctx* ctx, bool ta, bool tb, int64_t M, int64_t N, int64_t K, double alpha,
               const double* A, int64_t lda, const double* B, int64_t ldb, double beta, double* C,
               int64_t ldc, int s, bool lower, Arena* ar, cudaStream_t st, int digits, const OzGuard* guard, int width) {
  if (M <= 0 || N <= 0) return 0;
  FL_CHECK(ctx, s >= 1 && s <= 8, FRACLAP_ERR_INVALID_ARG, "ozaki_gemm: slices must be 1..8");
  FL_CHECK(ctx, cdiv(N, OZ_BN) <= 65535, FRACLAP_ERR_UNSUPPORTED, "ozaki_gemm: N too large");
  FL_CHECK(ctx, !lower || M >= N, FRACLAP_ERR_INVALID_ARG, "ozaki_gemm: a lower product needs M >= N");
  // Digit magnitude w and count D for s slices of 8 bits: with w = 8 (short K,
  // one chunk; or the knob) s digits of 9 bits (7 for s = 8: 63 bits, within
  // the FP64 rounding of the result); with w = 7 digits of 8 bits, one more
  // than s up to s = 5 and at s = 8, so that no s is less accurate than
  // ceil(8 s / 7) sign-magnitude digits of 7 bits (s = 6 and 7 reach that with
  // s).  Measured at 8810 x 8810 x 8810 on 128 x 192 tiles, those against
  // these: s = 7 52.3 ms and 3.3e-15 from FP64, now 39.6 ms and 3.2e-15; s = 6
  // 41.0 ms and 1.0e-13, now 30.2 ms and 9.3e-14.  (On 128 x 256 tiles without
  // the folds 28.8 and 21.4 ms; w = 8 at s = 7 32.0 ms: the same pairs and four
  // times more chunk sums to drain and convert.)
  int bits = 8, sl = std::min(s, 7);
  if (width == 7 || (width == 0 && K > 256 && ctx->oz_bits != 8)) {
    bits = 7;
    sl = (s <= 5 || s == 8) ? s + 1 : s;  // s = 8: 72 bits
  }
  if (digits > 0) sl = digits;
  // K in ranges, each added into C in FP64: 130048 (w = 7) or 32512 (w = 8), so
  // that the integer sums of a range cannot overflow whatever the operands
  int64_t k0 = 0;
  do {
    const int64_t kr = std::min(K - k0, oz_range(bits));
    FL_TRY(ozaki_range(ctx, ta, tb, M, N, kr, alpha, A + (ta ? k0 : k0 * lda), lda, B + (tb ? k0 * ldb : k0), ldb,
                       k0 == 0 ? beta : 1.0, C, ldc, sl, bits, lower, *ar, st, guard));
    k0 += kr;
  } while (k0 < K);
  return 0;
}

}  // namespace fraclap

using namespace fraclap;

extern "C" size_t fraclap_dgemm_ozaki_workspace_bytes(int64_t m, int64_t n, int64_t k, int slices) {
  if (m < 0 || n < 0 || k < 0 || slices < 1 || slices > 8) return 0;
  return ozaki_ws(m, n, k, slices) + 1024;
}

extern "C" int fraclap_dgemm_ozaki(fraclap_ctx* ctx, int trans_a, int trans_b, int64_t m, int64_t n,
                                   int64_t k, double alpha, const double* A_dev, int64_t lda,
                                   const double* B_dev, int64_t ldb, double beta, double* C_dev,
                                   int64_t ldc, int slices, void* work_dev, size_t work_bytes,
                                   fraclap_stream_t stream) {
  if (!ctx) return FRACLAP_ERR_INVALID_ARG;
  FL_CHECK(ctx, m >= 0 && n >= 0 && k >= 0, FRACLAP_ERR_INVALID_ARG, "dgemm_ozaki: negative size");
  if (m == 0 || n == 0) return 0;
  FL_CHECK(ctx, C_dev && A_dev && B_dev, FRACLAP_ERR_INVALID_ARG, "dgemm_ozaki: null pointer");
  FL_CHECK(ctx, ldc >= m && lda >= (trans_a ? k : m) && ldb >= (trans_b ? n : k),
           FRACLAP_ERR_INVALID_ARG, "dgemm_ozaki: leading dimension too small");
  Arena ar;
  int rc = get_workspace(ctx, work_dev, work_bytes, ozaki_ws(m, n, k, slices) + 1024, &ar);
  if (rc == FRACLAP_ERR_ALLOC) rc = get_workspace(ctx, work_dev, work_bytes, ozaki_ws(m, n, k, slices, false, 0, true) + 1024, &ar);
  if (rc != 0) return rc;
  return ozaki_gemm(ctx, trans_a != 0, trans_b != 0, m, n, k, alpha, A_dev, lda, B_dev, ldb, beta,
                    C_dev, ldc, slices, false, &ar, (cudaStream_t)stream);
}

extern "C" int fraclap_set_schedule(fraclap_ctx* ctx, int knob, int value) {
  if (!ctx) return FRACLAP_ERR_INVALID_ARG;
  switch (knob) {
    case FRACLAP_SCHED_OZAKI_GROUP:
      FL_CHECK(ctx, value >= 0 && value <= 4096, FRACLAP_ERR_INVALID_ARG, "set_schedule: group must be 0..4096");
      ctx->oz_group = value;
      return 0;
    case FRACLAP_SCHED_OZAKI_BITS:
      FL_CHECK(ctx, value == 7 || value == 8, FRACLAP_ERR_INVALID_ARG, "set_schedule: digit width must be 7 or 8");
      ctx->oz_bits = value;
      return 0;
    case FRACLAP_SCHED_FP32_STAGES:
      FL_CHECK(ctx, value == 0 || value == 1, FRACLAP_ERR_INVALID_ARG, "set_schedule: FP32 stage route must be 0 or 1");
      ctx->fp32_stages_tc = value;
      return 0;
    case FRACLAP_SCHED_OZAKI_TILE_N:
      FL_CHECK(ctx, value == 128 || value == 192 || value == 256, FRACLAP_ERR_INVALID_ARG,
               "set_schedule: tile width must be 128, 192 or 256");
      ctx->oz_tile_n = value;
      return 0;
    case FRACLAP_SCHED_Q2_PARTS:
      FL_CHECK(ctx, value == 0 || value == 4 || value == 8 || value == 16, FRACLAP_ERR_INVALID_ARG,
               "set_schedule: Q2 parts must be 0, 4, 8 or 16");
      ctx->q2_parts = value;
      return 0;
    case FRACLAP_SCHED_OZAKI_CLUSTER:
      FL_CHECK(ctx, value == 1 || value == 2, FRACLAP_ERR_INVALID_ARG,
               "set_schedule: slice-product cluster must be 1 or 2 CTAs");
      ctx->oz_cluster = value;
      return 0;
    default:
      return set_error(ctx, FRACLAP_ERR_INVALID_ARG, "set_schedule: unknown knob %d", knob);
  }
}

extern "C" int fraclap_get_schedule(const fraclap_ctx* ctx, int knob) {
  if (!ctx) return FRACLAP_ERR_INVALID_ARG;
  switch (knob) {
    case FRACLAP_SCHED_OZAKI_GROUP: return ctx->oz_group;
    case FRACLAP_SCHED_OZAKI_BITS: return ctx->oz_bits;
    case FRACLAP_SCHED_FP32_STAGES: return ctx->fp32_stages_tc;
    case FRACLAP_SCHED_OZAKI_TILE_N: return ctx->oz_tile_n;
    case FRACLAP_SCHED_Q2_PARTS: return ctx->q2_parts;
    case FRACLAP_SCHED_OZAKI_CLUSTER: return ctx->oz_cluster;
    default: return FRACLAP_ERR_INVALID_ARG;
  }
}
