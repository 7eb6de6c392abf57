// FP64 GEMM engine.
//
// On GB300 the FP64 pipe delivers ~1.2 TFLOP/s for both DFMA and DMMA
// (measured: DFMA 1.20, mma.sync f64 1.05, cuBLAS DGEMM 1.10 TFLOP/s), i.e.
// about 2 FMA per clock per SM.  A 64x64 output tile with a 16-deep k step
// needs 1 KB of operands per 4096 FMAs, so a plain shared-memory tiled SIMT
// kernel is bound by the FP64 pipe, not by memory; the design goal is to keep
// that pipe busy (enough resident warps, 16 independent accumulators per
// thread) while supporting the operand forms the eigensolver needs: both
// transposes, a symmetric A read from its lower triangle, a lower-triangular
// C, a fused second product (symmetric rank-2k update), split-K with atomics
// and device-side batched descriptors.
#include <cooperative_groups.h>

#include <type_traits>

#include "internal.cuh"

namespace fraclap {
namespace {

namespace cg = cooperative_groups;

constexpr int BM = 64, BN = 64, BK = 16, NT = 256;

template <class T, bool TA, int MODE>
__device__ __forceinline__ void load_a(T (*As)[BM + 1], const T* A, int64_t lda,
                                       int64_t M, int64_t K, int64_t m0, int64_t k0) {
  const int tid = threadIdx.x;
  if (MODE == kGemmSymA) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = tid % BM, k = tid / BM + 4 * i;
      const int64_t gm = m0 + m, gk = k0 + k;
      T v = T(0);
      if (gm < M && gk < K) v = (gm >= gk) ? A[gm + gk * lda] : A[gk + gm * lda];
      As[k][m] = v;
    }
  } else if (!TA) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = tid % BM, k = tid / BM + 4 * i;
      const int64_t gm = m0 + m, gk = k0 + k;
      As[k][m] = (gm < M && gk < K) ? A[gm + gk * lda] : T(0);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = tid % BK, m = tid / BK + 16 * i;
      const int64_t gm = m0 + m, gk = k0 + k;
      As[k][m] = (gm < M && gk < K) ? A[gk + gm * lda] : T(0);
    }
  }
}

template <class T, bool TB>
__device__ __forceinline__ void load_b(T (*Bs)[BN + 1], const T* B, int64_t ldb,
                                       int64_t N, int64_t K, int64_t n0, int64_t k0) {
  const int tid = threadIdx.x;
  if (!TB) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = tid % BK, n = tid / BK + 16 * i;
      const int64_t gn = n0 + n, gk = k0 + k;
      Bs[k][n] = (gn < N && gk < K) ? B[gk + gn * ldb] : T(0);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int n = tid % BN, k = tid / BN + 4 * i;
      const int64_t gn = n0 + n, gk = k0 + k;
      Bs[k][n] = (gn < N && gk < K) ? B[gn + gk * ldb] : T(0);
    }
  }
}

template <class T, bool TA, bool TB, int MODE>
__device__ __forceinline__ void accumulate(T (&acc)[4][4], T (*As)[BM + 1],
                                           T (*Bs)[BN + 1], const T* A, int64_t lda,
                                           const T* B, int64_t ldb, int64_t M, int64_t N,
                                           int64_t K, int64_t m0, int64_t n0, int64_t kbeg,
                                           int64_t kend) {
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  for (int64_t k0 = kbeg; k0 < kend; k0 += BK) {
    load_a<T, TA, MODE>(As, A, lda, M, kend, m0, k0);
    load_b<T, TB>(Bs, B, ldb, N, kend, n0, k0);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      T a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[k][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[k][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
}

template <class T, bool TA, bool TB, int MODE, bool ATOMIC>
__device__ __forceinline__ void gemm_tile(const GemmDescT<T>& d, int64_t m0, int64_t n0, int64_t kbeg,
                                          int64_t kend) {
  __shared__ T As[BK][BM + 1];
  __shared__ T Bs[BK][BN + 1];
  if (MODE == kGemmLowerC && m0 + BM - 1 < n0) return;  // tile entirely above the diagonal
  T acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = T(0);
  accumulate<T, TA, TB, MODE>(acc, As, Bs, d.A, d.lda, d.B, d.ldb, d.M, d.N, d.K, m0, n0, kbeg, kend);
  if (d.K2 > 0 && kbeg == 0)
    accumulate<T, TA, TB, MODE>(acc, As, Bs, d.A2, d.lda2, d.B2, d.ldb2, d.M, d.N, d.K2, m0, n0, 0,
                                d.K2);
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t gm = m0 + ty + 16 * i;
    if (gm >= d.M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int64_t gn = n0 + tx + 16 * j;
      if (gn >= d.N) continue;
      if (MODE == kGemmLowerC && gm < gn) continue;
      T* c = d.C + gm + gn * d.ldc;
      const T v = T(d.alpha) * acc[i][j];
      if (ATOMIC) {
        atomicAdd(c, v);
      } else {
        *c = (d.beta == 0.0) ? v : v + T(d.beta) * *c;
      }
    }
  }
}

template <class T, bool TA, bool TB, int MODE, bool ATOMIC>
__global__ void __launch_bounds__(NT) gemm_kernel(GemmDescT<T> d, int64_t kchunk) {
  if (d.only_if && *d.only_if == 0) return;
  const int64_t m0 = (int64_t)blockIdx.x * BM, n0 = (int64_t)blockIdx.y * BN;
  const int64_t kbeg = (int64_t)blockIdx.z * kchunk;
  const int64_t kend = (kbeg + kchunk < d.K) ? kbeg + kchunk : d.K;
  if (kbeg > 0 && kbeg >= d.K) return;  // z-slice 0 always runs (K = 0: C = beta C)
  gemm_tile<T, TA, TB, MODE, ATOMIC>(d, m0, n0, kbeg, kend);
}

template <class T, bool TA, bool TB>
__global__ void __launch_bounds__(NT) gemm_batched_kernel(const GemmDescT<T>* descs) {
  const GemmDescT<T> d = descs[blockIdx.z];
  const int64_t m0 = (int64_t)blockIdx.x * BM, n0 = (int64_t)blockIdx.y * BN;
  if (d.M <= 0 || d.N <= 0 || m0 >= d.M || n0 >= d.N) return;
  if (d.K <= 0) {  // C = beta C
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    for (int i = 0; i < 4; ++i)
      for (int j = 0; j < 4; ++j) {
        const int64_t gm = m0 + ty + 16 * i, gn = n0 + tx + 16 * j;
        if (gm < d.M && gn < d.N) {
          T* c = d.C + gm + gn * d.ldc;
          *c = (d.beta == 0.0) ? T(0) : T(d.beta) * *c;
        }
      }
    return;
  }
  gemm_tile<T, TA, TB, kGemmPlain, false>(d, m0, n0, 0, d.K);
}

// ---------------------------------------------------------------------------
// FP32 products: 128 threads per output tile, each TM x TN outputs in registers,
// k steps of 16 (8 on the large tile) double-buffered in shared memory (the next step is fetched
// into registers while the current one is multiplied).  The multiplications are
// packed pairs (fma.rn.f32x2) along the rows: half the issue slots, so that the
// shared-memory reads -- (TM + TN) / (TM TN) words an FMA, what bounds a SIMT
// product on this chip -- fit beside them.  128 x 128 tiles at 16 x 8 outputs a
// thread for outputs of at least 256 x 256; 128 x 64 and 64 x 128 at 8 x 8 for
// narrow outputs, whose long sums a cluster of CTAs along K shares (partial
// tiles added over distributed shared memory in rank order: no atomics, no
// zeroing).  Forms: plain, lower-C, symmetric A (its lower triangle read:
// blocks above the diagonal from their mirror, in either case coalesced), a
// second product into the same C, batched.  GB300, before and now: 8192^3 45.1
// -> 53.0 TFLOP/s; symmetric 4405 x 64 some 230 -> 93 us, 1114 x 32 98 -> 15 us;
// the merges' products at n = 7735 21.5 -> 15.0 ms, the first back-transformation
// there 39.7 -> 35.4 ms, the band reduction 90 -> 79 ms.
constexpr int SG_NT = 128, SG_K = 16, SG_K_BIG = 8;

__device__ __forceinline__ unsigned long long sg_pair(float a, float b) {
  unsigned long long v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
  return v;
}
__device__ __forceinline__ void sg_fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

// One operand's k step in registers: BX entries along x (rows of op(A) or
// columns of op(B)) by SG_K along k.  XC: x is the contiguous direction of the
// storage; entry (x, k) at p[x + k ld], else at p[k + x ld].
template <int BX, bool XC, int SG_K>
struct SgStep {
  static constexpr int PER = BX * SG_K / SG_NT;
  static __device__ __forceinline__ int x_of(int q) {
    return XC ? ((BX == 128) ? (int)threadIdx.x : (int)(threadIdx.x % BX)) : (int)(threadIdx.x / SG_K) + (SG_NT / SG_K) * q;
  }
  static __device__ __forceinline__ int k_of(int q) {
    return XC ? ((BX == 128) ? q : (int)(threadIdx.x / BX) + (SG_NT / BX) * q) : (int)(threadIdx.x % SG_K);
  }
  static __device__ __forceinline__ void fetch(float (&r)[PER], const float* p, int64_t ld, int64_t X, int64_t kend,
                                               int64_t x0, int64_t k0) {
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int64_t x = x0 + x_of(q), k = k0 + k_of(q);
      r[q] = (x < X && k < kend) ? (XC ? p[x + k * ld] : p[k + x * ld]) : 0.0f;
    }
  }
  // symmetric storage, lower triangle: entry (x, k) at p[x + k ld] if x >= k, else its mirror
  static __device__ __forceinline__ void fetch_sym(float (&r)[PER], const float* p, int64_t ld, int64_t X, int64_t kend,
                                                   int64_t x0, int64_t k0) {
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int64_t x = x0 + x_of(q), k = k0 + k_of(q);
      r[q] = (x < X && k < kend) ? (x >= k ? p[x + k * ld] : p[k + x * ld]) : 0.0f;
    }
  }
  static __device__ __forceinline__ void stash(float* s, const float (&r)[PER]) {  // s: SG_K x (BX + 4)
#pragma unroll
    for (int q = 0; q < PER; ++q) s[k_of(q) * (BX + 4) + x_of(q)] = r[q];
  }
};

template <int BM, int BN, int TM, int TN, int SG_K>
struct SgTile {
  static_assert((BM / TM) * (BN / TN) == SG_NT, "128 threads");
  static constexpr int GX = BM / TM, GY = BN / TN;  // threads along the rows and columns
  static constexpr int STEP = SG_K * (BM + 4 + BN + 4);  // words of one buffered k step
  // thread (tx, ty): rows 4 (tx + GX i) + e, columns 4 (ty + GY j) + e
  static __device__ __forceinline__ int row(int i) { return 4 * ((int)threadIdx.x % GX + GX * (i / 4)) + i % 4; }
  static __device__ __forceinline__ int col(int j) { return 4 * ((int)threadIdx.x / GX + GY * (j / 4)) + j % 4; }
};

template <int BM, int BN, int TM, int TN, int SG_K, bool TA, bool TB, int MODE>
__device__ __forceinline__ void sg_accumulate(unsigned long long (&acc)[TM / 2][TN], float* smem, const float* A,
                                              int64_t lda, const float* B, int64_t ldb, int64_t M, int64_t N,
                                              int64_t m0, int64_t n0, int64_t kbeg, int64_t kend) {
  using Tile = SgTile<BM, BN, TM, TN, SG_K>;
  using SA = SgStep<BM, !TA, SG_K>;
  using SM = SgStep<BM, false, SG_K>;  // the mirrored half of a symmetric A
  using SB = SgStep<BN, TB, SG_K>;
  float ra[SA::PER], rb[SB::PER];
  // symmetric A: 0 below the diagonal, 1 above it, 2 across it
  auto side = [&](int64_t k0) { return k0 + SG_K - 1 <= m0 ? 0 : (k0 >= m0 + BM - 1 ? 1 : 2); };
  auto fetch = [&](int64_t k0) {
    if (MODE == kGemmSymA) {
      const int sd = side(k0);
      if (sd == 0) SA::fetch(ra, A, lda, M, kend, m0, k0);
      else if (sd == 1) SM::fetch(ra, A, lda, M, kend, m0, k0);
      else SA::fetch_sym(ra, A, lda, M, kend, m0, k0);
    } else {
      SA::fetch(ra, A, lda, M, kend, m0, k0);
    }
    SB::fetch(rb, B, ldb, N, kend, n0, k0);
  };
  auto stash = [&](float* buf, int64_t k0) {
    if (MODE == kGemmSymA && side(k0) == 1) SM::stash(buf, ra);
    else SA::stash(buf, ra);
    SB::stash(buf + SG_K * (BM + 4), rb);
  };
  fetch(kbeg);
  __syncthreads();  // the buffers may still be read by a previous product
  stash(smem, kbeg);
  __syncthreads();
  int buf = 0;
  for (int64_t k0 = kbeg; k0 < kend; k0 += SG_K) {
    const bool more = k0 + SG_K < kend;
    if (more) fetch(k0 + SG_K);
    const float* as = smem + buf * Tile::STEP;
    const float* bs = as + SG_K * (BM + 4);
#pragma unroll
    for (int k = 0; k < SG_K; ++k) {
      unsigned long long a[TM / 2];
#pragma unroll
      for (int i = 0; i < TM; i += 4) {
        const float4 v = *reinterpret_cast<const float4*>(as + k * (BM + 4) + Tile::row(i));
        a[i / 2] = sg_pair(v.x, v.y);
        a[i / 2 + 1] = sg_pair(v.z, v.w);
      }
#pragma unroll
      for (int j = 0; j < TN; j += 4) {
        const float4 v = *reinterpret_cast<const float4*>(bs + k * (BN + 4) + Tile::col(j));
        const float b[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const unsigned long long bb = sg_pair(b[e], b[e]);
#pragma unroll
          for (int i = 0; i < TM / 2; ++i) sg_fma2(acc[i][j + e], a[i], bb);
        }
      }
    }
    if (more) stash(smem + (buf ^ 1) * Tile::STEP, k0 + SG_K);
    __syncthreads();
    buf ^= 1;
  }
}

template <int MODE>
__device__ __forceinline__ void sg_write(const GemmDescT<float>& d, int64_t gm, int64_t gn, float v) {
  if (gm >= d.M || gn >= d.N || (MODE == kGemmLowerC && gm < gn)) return;
  float* c = d.C + gm + gn * d.ldc;
  v *= (float)d.alpha;
  *c = (d.beta == 0.0) ? v : v + (float)d.beta * *c;
}

// One tile over k in [kbeg, kend) (and the whole second product), shared by the
// CTAs of a cluster along K when CLUSTER.
template <int BM, int BN, int TM, int TN, int SG_K, bool TA, bool TB, int MODE, bool CLUSTER>
__device__ __forceinline__ void sg_tile(const GemmDescT<float>& d, int64_t m0, int64_t n0, int64_t kbeg, int64_t kend) {
  using Tile = SgTile<BM, BN, TM, TN, SG_K>;
  constexpr int WORDS = CLUSTER ? (2 * Tile::STEP > BM * BN ? 2 * Tile::STEP : BM * BN) : 2 * Tile::STEP;
  __shared__ __align__(16) float smem[WORDS];
  unsigned long long acc[TM / 2][TN];
#pragma unroll
  for (int i = 0; i < TM / 2; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0ull;
  if (kend > kbeg)
    sg_accumulate<BM, BN, TM, TN, SG_K, TA, TB, MODE>(acc, smem, d.A, d.lda, d.B, d.ldb, d.M, d.N, m0, n0, kbeg, kend);
  if (d.K2 > 0)  // (a product with a second one is not shared along K)
    sg_accumulate<BM, BN, TM, TN, SG_K, TA, TB, MODE>(acc, smem, d.A2, d.lda2, d.B2, d.ldb2, d.M, d.N, m0, n0, 0, d.K2);
  if (CLUSTER) {
    cg::cluster_group cluster = cg::this_cluster();
    const int S = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    if (S > 1) {
      // (the last k step ended with a barrier; a CTA without steps has read nothing)
#pragma unroll
      for (int j = 0; j < TN; ++j)
#pragma unroll
        for (int i = 0; i < TM; i += 4) {
          float4 v;
          asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(acc[i / 2][j]));
          asm("mov.b64 {%0, %1}, %2;" : "=f"(v.z), "=f"(v.w) : "l"(acc[i / 2 + 1][j]));
          *reinterpret_cast<float4*>(&smem[Tile::col(j) * BM + Tile::row(i)]) = v;
        }
      cluster.sync();
      for (int e = rank * SG_NT + (int)threadIdx.x; e < BM * BN; e += S * SG_NT) {
        float v = 0.0f;
        for (int q = 0; q < S; ++q) v += cluster.map_shared_rank(smem, q)[e];
        sg_write<MODE>(d, m0 + e % BM, n0 + e / BM, v);
      }
      cluster.sync();  // a peer's tile stays until it is read
      return;
    }
  }
#pragma unroll
  for (int j = 0; j < TN; ++j)
#pragma unroll
    for (int i = 0; i < TM; i += 2) {
      float x, y;
      asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(acc[i / 2][j]));
      sg_write<MODE>(d, m0 + Tile::row(i), n0 + Tile::col(j), x);
      sg_write<MODE>(d, m0 + Tile::row(i) + 1, n0 + Tile::col(j), y);
    }
}

template <bool TA, bool TB, int MODE>
__global__ void __launch_bounds__(SG_NT, 2) sgemm_big_kernel(GemmDescT<float> d) {
  const int64_t m0 = (int64_t)blockIdx.x * 128, n0 = (int64_t)blockIdx.y * 128;
  if (MODE == kGemmLowerC && m0 + 127 < n0) return;  // tile entirely above the diagonal
  sg_tile<128, 128, 16, 8, SG_K_BIG, TA, TB, MODE, false>(d, m0, n0, 0, d.K);
}

template <bool TA, bool TB>
__global__ void __launch_bounds__(SG_NT, 2) sgemm_big_batched_kernel(const GemmDescT<float>* descs) {
  const GemmDescT<float> d = descs[blockIdx.z];
  const int64_t m0 = (int64_t)blockIdx.x * 128, n0 = (int64_t)blockIdx.y * 128;
  if (d.M <= 0 || d.N <= 0 || m0 >= d.M || n0 >= d.N) return;
  sg_tile<128, 128, 16, 8, SG_K_BIG, TA, TB, kGemmPlain, false>(d, m0, n0, 0, d.K > 0 ? d.K : 0);
}

template <int BM, int BN, bool TA, bool TB, int MODE>
__global__ void __launch_bounds__(SG_NT, 4) sgemm_narrow_kernel(GemmDescT<float> d, int64_t kper) {
  const int S = (int)cg::this_cluster().num_blocks();
  const int64_t m0 = (int64_t)(blockIdx.x / S) * BM, n0 = (int64_t)blockIdx.y * BN;
  const int64_t kbeg = (int64_t)cg::this_cluster().block_rank() * kper;
  if (MODE == kGemmLowerC && m0 + BM - 1 < n0) return;  // tile entirely above the diagonal (S = 1)
  sg_tile<BM, BN, 8, 8, SG_K, TA, TB, MODE, true>(d, m0, n0, kbeg, (kbeg + kper < d.K) ? kbeg + kper : d.K);
}

// The 128 x 128 tiles pay off once both output dimensions fill them.
inline bool sg_big(int64_t M, int64_t N) { return M >= 256 && N >= 256; }
// Narrow outputs: one dimension of at most 128, the other of at least as much.
inline bool sg_narrow(int64_t M, int64_t N) { return std::min(M, N) <= 128 && std::max(M, N) >= 128; }

template <int BM, int BN, bool TA, bool TB, int MODE>
int launch_sg_narrow(fraclap_ctx* ctx, const GemmDescT<float>& d, cudaStream_t st) {
  const int64_t sms = ctx->sm_count > 0 ? ctx->sm_count : 152;
  const int64_t gx = cdiv(d.M, BM), gy = cdiv(d.N, BN);
  FL_CHECK(ctx, gy <= 65535, FRACLAP_ERR_UNSUPPORTED, "gemm: N = %lld too large", (long long)d.N);
  int S = 1;  // CTAs per tile along K: until three CTAs an SM, at least 64 of K each
  while (MODE != kGemmLowerC && S < 8 && gx * gy * S < 3 * sms && d.K2 == 0 && d.K >= 128 * (int64_t)S) S *= 2;
  const int64_t kper = std::max<int64_t>(cdiv(cdiv(d.K, S), SG_K) * SG_K, SG_K);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(gx * S), (unsigned)gy, 1);
  cfg.blockDim = dim3(SG_NT);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)S;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  FL_CUDA(ctx, cudaLaunchKernelEx(&cfg, sgemm_narrow_kernel<BM, BN, TA, TB, MODE>, d, kper));
  count_launch(ctx);
  return 0;
}

// ---------------------------------------------------------------------------
// FP64 products without padding.  The FP64 pipe retires about 1.7 FMAs per
// clock and SM, so a warp's FMA occupies it for some 19 cycles and every
// operand can come straight from L1 at no cost; what a narrow or small product
// pays for on the 64 x 64 tile is the padding (5 columns cost 64) and the SMs
// its few tiles leave idle.  These kernels skip the columns past N one by one,
// and a cluster of CTAs along K splits the sum of a tile until the tiles cover
// the SMs; the CTAs' partial sums meet in distributed shared memory and are
// added in rank order, so the result does not depend on the schedule.
// Bound: the FP64 pipe.  GB300, column counts as given, against the 64 x 64
// tile: 2304 x 5 x 2304 (A^T B) 2409 -> 143 us and 2304 x 20 x 2304 2411 ->
// 294 us (both with the caller's wait of some 50 us), 8835 x 128 x 8835 17.9
// -> 16.6 ms (1.20 TFLOP/s); the apply at n = 2304 with 5 columns and 20 pairs
// 4.80 -> 0.36 ms, at n = 144 0.31 -> 0.04 ms.
constexpr int DG_NT = 256, DG_NC = 8, DG_ROWS = 32;

// Adds the partial sums of the cluster's CTAs (one value per thread) and
// writes C from rank 0.  Every thread of every CTA of the cluster calls it.
template <int MODE>
__device__ __forceinline__ void dg_finish(const GemmDescT<double>& d, double v, int64_t gm, int64_t gn) {
  __shared__ double part[DG_NT];
  cg::cluster_group cluster = cg::this_cluster();
  const unsigned S = cluster.num_blocks();
  if (S > 1) {
    part[threadIdx.x] = v;
    cluster.sync();
    if (cluster.block_rank() == 0)
      for (unsigned q = 1; q < S; ++q) v += *cluster.map_shared_rank(&part[threadIdx.x], q);
    cluster.sync();  // a peer's partial sums stay until they are read
    if (cluster.block_rank() != 0) return;
  }
  if (gm >= d.M || gn >= d.N) return;
  double* c = d.C + gm + gn * d.ldc;
  v *= d.alpha;
  *c = (d.beta == 0.0) ? v : v + d.beta * *c;
}

// The columns of its tile, one bit each, that this cluster forms: all nc of them,
// the marked ones, or none.  (The same in every CTA of the cluster.)
__device__ __forceinline__ unsigned dg_columns(const GemmDescT<double>& d, int nc) {
  const unsigned all = (1u << nc) - 1u;
  if (d.only_if && *d.only_if == 0) return 0u;
  if (!d.only_marked) return all;
  const int64_t S = cg::this_cluster().num_blocks();
  return d.only_marked[(int64_t)blockIdx.y * (gridDim.x / S) + blockIdx.x / S] & all;
}

// op(A) = A (or symmetric, lower triangle read): a lane per row, eight warps
// interleaved over K, up to eight columns in registers; the reads of A are
// coalesced along the rows (in the mirrored half of a symmetric A a lane walks
// along its own column, whose lines L1 keeps), B is one address per warp.
template <bool TB, int MODE>
__global__ void __launch_bounds__(DG_NT) dgemm_rows_kernel(GemmDescT<double> d, int64_t kper, int ncol) {
  __shared__ double red[DG_NC][DG_NC][DG_ROWS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t m0 = (int64_t)(blockIdx.x / cg::this_cluster().num_blocks()) * DG_ROWS, n0 = (int64_t)blockIdx.y * ncol;
  const unsigned cols = dg_columns(d, (int)((d.N - n0 < ncol) ? d.N - n0 : ncol));
  if (cols == 0) return;
  const int64_t kbeg = (int64_t)cg::this_cluster().block_rank() * kper;
  const int64_t kend = (kbeg + kper < d.K) ? kbeg + kper : d.K;
  const int64_t row = m0 + lane;
  const int64_t i = (row < d.M) ? row : d.M - 1;
  const int64_t bk = TB ? d.ldb : 1, bj = TB ? 1 : d.ldb;
  const double* Bp = d.B + n0 * bj;
  auto a_at = [&](int64_t k) -> double {
    if (MODE == kGemmSymA) return (i >= k) ? d.A[i + k * d.lda] : d.A[k + i * d.lda];
    return d.A[i + k * d.lda];
  };
  double acc[DG_NC];
#pragma unroll
  for (int j = 0; j < DG_NC; ++j) acc[j] = 0.0;
  constexpr int KU = 4;
  for (int64_t k0 = kbeg + KU * warp; k0 < kend; k0 += KU * (DG_NT / 32)) {
    if (k0 + KU <= kend) {
      double a[KU];
#pragma unroll
      for (int u = 0; u < KU; ++u) a[u] = a_at(k0 + u);
#pragma unroll
      for (int j = 0; j < DG_NC; ++j)
        if (cols >> j & 1) {
          const double* b = Bp + j * bj + k0 * bk;
#pragma unroll
          for (int u = 0; u < KU; ++u) acc[j] = fma(a[u], b[u * bk], acc[j]);
        }
    } else {
      for (int64_t k = k0; k < kend; ++k) {
        const double a = a_at(k);
#pragma unroll
        for (int j = 0; j < DG_NC; ++j)
          if (cols >> j & 1) acc[j] = fma(a, Bp[j * bj + k * bk], acc[j]);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < DG_NC; ++j) red[warp][j][lane] = acc[j];
  __syncthreads();
  double v = 0.0;  // thread (warp, lane): column warp, row lane, the warps' sums in order
#pragma unroll
  for (int w = 0; w < DG_NT / 32; ++w) v += red[w][warp][lane];
  dg_finish<MODE>(d, v, row, (cols >> warp & 1) ? n0 + warp : d.N);
}

// op(A) = A^T, op(B) = B (both contiguous along K): the lanes of a warp share
// K, each warp holds four rows x eight columns, and a butterfly that halves
// the 32 sums at every step leaves one output per lane.
__global__ void __launch_bounds__(DG_NT) dgemm_dots_kernel(GemmDescT<double> d, int64_t kper, int ncol) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t m0 = (int64_t)(blockIdx.x / cg::this_cluster().num_blocks()) * DG_ROWS + 4 * warp;
  const int64_t n0 = (int64_t)blockIdx.y * ncol;
  const unsigned cols = dg_columns(d, (int)((d.N - n0 < ncol) ? d.N - n0 : ncol));
  if (cols == 0) return;
  const int64_t kbeg = (int64_t)cg::this_cluster().block_rank() * kper;
  const int64_t kend = (kbeg + kper < d.K) ? kbeg + kper : d.K;
  const double* Ap[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) Ap[r] = d.A + ((m0 + r < d.M) ? m0 + r : d.M - 1) * d.lda;
  const double* Bp = d.B + n0 * d.ldb;
  double acc[4 * DG_NC];
#pragma unroll
  for (int q = 0; q < 4 * DG_NC; ++q) acc[q] = 0.0;
  for (int64_t k = kbeg + lane; k < kend; k += 32) {
    double a[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) a[r] = Ap[r][k];
#pragma unroll
    for (int j = 0; j < DG_NC; ++j)
      if (cols >> j & 1) {
        const double b = Bp[j * d.ldb + k];
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[r * DG_NC + j] = fma(a[r], b, acc[r * DG_NC + j]);
      }
  }
  int idx = 0;  // output this lane ends with: row idx / 8, column idx % 8
#pragma unroll
  for (int half = 16; half >= 1; half >>= 1) {
    const bool up = (lane & half) != 0;
#pragma unroll
    for (int q = 0; q < half; ++q) {
      const double send = up ? acc[q] : acc[q + half];
      const double keep = up ? acc[q + half] : acc[q];
      acc[q] = keep + __shfl_xor_sync(0xffffffffu, send, half);
    }
    if (up) idx += half;
  }
  const int j = idx % DG_NC;
  dg_finish<kGemmPlain>(d, acc[0], m0 + idx / DG_NC, (cols >> j & 1) ? n0 + j : d.N);
}

// Lower C = alpha (A B^T + A2 B2^T) + beta C of short sums (the reduction's
// rank-2b updates), and the batched C = alpha A B + beta C (the merges of divide
// and conquer): 32 x 32 tiles, a lane per row, eight warps of four columns, the
// operands straight from L1, every entry's sum in the order of the 64 x 64 tile.
// Four times the tiles even out the SMs' shares of the FP64 pipe, which bounds
// both: GB300, b = 32, the band reduction at n = 779 5.8 -> 5.0 ms, 2351 36.6 ->
// 32.7, 4016 116.6 -> 110.7; the merges: divide and conquer at n = 779 4.1 -> 3.8,
// 2351 29.2 -> 26.5, 4016 115 -> 111, 7735 725 -> 709.
template <bool TB>
__device__ __forceinline__ void dgemm_small_sum(double (&acc)[4], const double* A, int64_t lda, const double* B, int64_t ldb, int64_t K,
                                                int64_t row, const int64_t (&col)[4]) {
#pragma unroll 4
  for (int64_t k = 0; k < K; ++k) {
    const double a = A[row + k * lda];
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[j] = fma(a, TB ? B[col[j] + k * ldb] : B[k + col[j] * ldb], acc[j]);
  }
}
template <bool TB, bool LOWER>
__device__ __forceinline__ void dgemm_small_tile(const GemmDescT<double>& d) {
  const int64_t m0 = (int64_t)blockIdx.x * 32, n0 = (int64_t)blockIdx.y * 32;
  if (m0 >= d.M || n0 >= d.N || (LOWER && m0 + 31 < n0)) return;  // past C, or entirely above its diagonal
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t gm = m0 + lane, gn = n0 + 4 * warp;
  int64_t col[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) col[j] = gn + j < d.N ? gn + j : d.N - 1;
  const int64_t row = gm < d.M ? gm : d.M - 1;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  dgemm_small_sum<TB>(acc, d.A, d.lda, d.B, d.ldb, d.K, row, col);
  if (LOWER && d.K2 > 0) dgemm_small_sum<TB>(acc, d.A2, d.lda2, d.B2, d.ldb2, d.K2, row, col);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (gm >= d.M || gn + j >= d.N || (LOWER && gm < gn + j)) continue;
    double* c = d.C + gm + (gn + j) * d.ldc;
    const double v = d.alpha * acc[j];
    *c = (d.beta == 0.0) ? v : v + d.beta * *c;
  }
}
__global__ void __launch_bounds__(DG_NT) dgemm_lower_kernel(GemmDescT<double> d) { dgemm_small_tile<true, true>(d); }
__global__ void __launch_bounds__(DG_NT) dgemm_small_batched_kernel(const GemmDescT<double>* descs) {
  const GemmDescT<double> d = descs[blockIdx.z];
  dgemm_small_tile<false, false>(d);
}

// True when the FP64 product takes the kernels above.  A B: fewer than four 64 x
// 64 tiles per SM (a last wave of idle SMs costs more than a tile's reuse of its
// operands saves; at 9 tiles per SM, 2304 x 2304 x 32, both take 357 us), or
// more than a tenth of the tiles is padding.  A^T B, whose dot products reach
// 0.78 of the tile's rate (64 x 8810 x 4405 6.1 against 4.7 ms): when the tiles'
// waves cost more than that (64 x 4000 x 2000 1.1 against 2.1 ms).
inline bool dg_narrow(const fraclap_ctx* ctx, bool ta, int64_t M, int64_t N) {
  const int64_t sms = ctx->sm_count > 0 ? ctx->sm_count : 152;
  const int64_t tiles = cdiv(M, BM) * cdiv(N, BN);
  if (ta) return (double)(cdiv(tiles, sms) * sms * BM * BN) > 1.28 * (double)M * (double)N;
  return tiles < 4 * sms || (double)(tiles * BM * BN) > 1.1 * (double)M * (double)N;
}

template <bool TA, bool TB, int MODE>
int launch_narrow(fraclap_ctx* ctx, const GemmDescT<double>& d, cudaStream_t st) {
  const int64_t sms = ctx->sm_count > 0 ? ctx->sm_count : 152;
  constexpr int64_t kMostCols = 65535 * (int64_t)DG_NC;  // a grid's second dimension; more columns in turn
  if (d.N > kMostCols) {
    for (int64_t j = 0; j < d.N; j += kMostCols) {
      GemmDescT<double> part = d;
      part.N = (d.N - j < kMostCols) ? d.N - j : kMostCols;
      part.B += TB ? j : j * d.ldb;
      part.C += j * d.ldc;
      if (d.only_marked) part.only_marked += j / DG_NC * cdiv(d.M, DG_ROWS);
      FL_TRY((launch_narrow<TA, TB, MODE>(ctx, part, st)));
    }
    return 0;
  }
  const int64_t gx = cdiv(d.M, DG_ROWS), gy = cdiv(d.N, DG_NC);
  static_assert(DG_ROWS == kGuardRows && DG_NC == kGuardCols, "the marks' tiles");
  const int ncol = d.only_marked ? DG_NC : (int)cdiv(d.N, gy);  // the columns dealt evenly
  int S = 1;
  // (few tiles of a grid are marked: four CTAs a tile whatever the grid)
  while (S < 8 && (gx * gy * S < 4 * sms || (d.only_marked && S < 4)) && d.K >= 256 * (int64_t)S) S *= 2;
  const int64_t kper = cdiv(cdiv(d.K > 0 ? d.K : 1, S), 32) * 32;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(gx * S), (unsigned)gy, 1);
  cfg.blockDim = dim3(DG_NT);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)S;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if constexpr (TA)
    FL_CUDA(ctx, cudaLaunchKernelEx(&cfg, dgemm_dots_kernel, d, kper, ncol));
  else
    FL_CUDA(ctx, cudaLaunchKernelEx(&cfg, dgemm_rows_kernel<TB, MODE>, d, kper, ncol));
  count_launch(ctx);
  return 0;
}

template <class T, bool TA, bool TB, int MODE>
int launch(fraclap_ctx* ctx, const GemmDescT<T>& d, int split_k, cudaStream_t st) {
  if constexpr (std::is_same<T, float>::value) {
    // short sums into large outputs are bound by C's traffic and latency: the
    // smaller tile has four CTAs an SM to overlap them
    const bool shallow = d.K + d.K2 <= 160 && cdiv(d.N, 64) <= 65535;
    if (MODE != kGemmSymA && sg_big(d.M, d.N) && shallow) return launch_sg_narrow<128, 64, TA, TB, MODE>(ctx, d, st);
    if (MODE != kGemmSymA && sg_big(d.M, d.N)) {
      const int64_t gx = cdiv(d.M, 128), gy = cdiv(d.N, 128);
      FL_CHECK(ctx, gy <= 65535, FRACLAP_ERR_UNSUPPORTED, "gemm: N = %lld too large", (long long)d.N);
      sgemm_big_kernel<TA, TB, MODE><<<dim3((unsigned)gx, (unsigned)gy, 1), SG_NT, 0, st>>>(d);
      count_launch(ctx);
      FL_CUDA(ctx, cudaGetLastError());
      return 0;
    }
    // (and small ones with a long sum, unless the caller splits it)
    const bool deep = split_k <= 1 && d.K >= 512 && std::max(d.M, d.N) <= 128;
    if (MODE != kGemmLowerC && d.K2 == 0 && (sg_narrow(d.M, d.N) || deep))
      return d.M >= d.N ? launch_sg_narrow<128, 64, TA, TB, MODE>(ctx, d, st)
                        : launch_sg_narrow<64, 128, TA, TB, MODE>(ctx, d, st);
  }
  if constexpr (std::is_same<T, double>::value && MODE != kGemmLowerC && !(TA && TB)) {
    // (a caller that splits the sums of 64 tiles or more fills the SMs by itself)
    const bool own = TA && split_k > 1 && cdiv(d.M, BM) * cdiv(d.N, BN) >= 64;
    if (d.only_marked || (d.K2 == 0 && !own && dg_narrow(ctx, TA, d.M, d.N))) return launch_narrow<TA, TB, MODE>(ctx, d, st);
  }
  if constexpr (std::is_same<T, double>::value && MODE == kGemmLowerC && !TA && TB) {
    // short sums; long ones take the 64 x 64 tile's shared memory
    if ((split_k <= 1 || d.K2 > 0) && d.K + d.K2 <= 160 && cdiv(d.N, 32) <= 65535 && d.M > 0 && d.N > 0) {
      dgemm_lower_kernel<<<dim3((unsigned)cdiv(d.M, 32), (unsigned)cdiv(d.N, 32)), DG_NT, 0, st>>>(d);
      count_launch(ctx);
      FL_CUDA(ctx, cudaGetLastError());
      return 0;
    }
  }
  const int64_t gx = cdiv(d.M, BM), gy = cdiv(d.N, BN);
  FL_CHECK(ctx, gy <= 65535, FRACLAP_ERR_UNSUPPORTED, "gemm: N = %lld too large", (long long)d.N);
  if (split_k <= 1 || d.K2 > 0) {
    gemm_kernel<T, TA, TB, MODE, false><<<dim3((unsigned)gx, (unsigned)gy, 1), NT, 0, st>>>(
        d, d.K > 0 ? d.K : 1);
    count_launch(ctx);
  } else {
    int64_t kchunk = cdiv(cdiv(d.K, split_k), BK) * BK;
    const int64_t gz = cdiv(d.K, kchunk);
    gemm_kernel<T, TA, TB, MODE, true><<<dim3((unsigned)gx, (unsigned)gy, (unsigned)gz), NT, 0, st>>>(
        d, kchunk);
    count_launch(ctx);
  }
  FL_CUDA(ctx, cudaGetLastError());
  return 0;
}

}  // namespace

template <class T>
int gemm(fraclap_ctx* ctx, bool ta, bool tb, GemmMode mode, const GemmDescT<T>& d, int split_k,
         cudaStream_t st) {
  if (d.M <= 0 || d.N <= 0) return 0;
  FL_CHECK(ctx, mode != kGemmSymA || (!ta && d.M == d.K), FRACLAP_ERR_INVALID_ARG,
           "gemm: symmetric A must be square and untransposed");
  FL_CHECK(ctx, split_k <= 1 || d.beta == 1.0, FRACLAP_ERR_INVALID_ARG,
           "gemm: split-K accumulates into C (beta must be 1)");
  if constexpr (std::is_same<T, float>::value) {
    if ((d.K > 0 || d.K2 > 0) && tf32_route_fits(ctx, mode, d, split_k))
      return gemm_tf32x3(ctx, ta, tb, mode, d, split_k, st);
  }
  if (d.K <= 0 && d.K2 <= 0) {  // C = beta C
    GemmDescT<T> z = d;
    z.K = 0;
    z.K2 = 0;
    return launch<T, false, false, kGemmPlain>(ctx, z, 1, st);
  }
#define FL_GEMM_CASE(TA, TB)                                                           \
  if (ta == TA && tb == TB) {                                                          \
    if (mode == kGemmPlain) return launch<T, TA, TB, kGemmPlain>(ctx, d, split_k, st);  \
    if (mode == kGemmLowerC) return launch<T, TA, TB, kGemmLowerC>(ctx, d, split_k, st); \
  }
  FL_GEMM_CASE(false, false)
  FL_GEMM_CASE(false, true)
  FL_GEMM_CASE(true, false)
  FL_GEMM_CASE(true, true)
#undef FL_GEMM_CASE
  if (mode == kGemmSymA) {
    if (tb) return launch<T, false, true, kGemmSymA>(ctx, d, split_k, st);
    return launch<T, false, false, kGemmSymA>(ctx, d, split_k, st);
  }
  return set_error(ctx, FRACLAP_ERR_INVALID_ARG, "gemm: bad mode");
}

template <class T>
int gemm_batched(fraclap_ctx* ctx, bool ta, bool tb, const GemmDescT<T>* d_descs, int count,
                 int64_t max_m, int64_t max_n, cudaStream_t st) {
  if (count <= 0 || max_m <= 0 || max_n <= 0) return 0;
  if constexpr (std::is_same<T, float>::value) {
    if (sg_big(max_m, max_n)) {
      const int64_t gx = cdiv(max_m, 128), gy = cdiv(max_n, 128);
      FL_CHECK(ctx, gy <= 65535 && count <= 65535, FRACLAP_ERR_UNSUPPORTED, "gemm_batched: too large");
      dim3 grid((unsigned)gx, (unsigned)gy, (unsigned)count);
      if (!ta && !tb) sgemm_big_batched_kernel<false, false><<<grid, SG_NT, 0, st>>>(d_descs);
      else if (!ta && tb) sgemm_big_batched_kernel<false, true><<<grid, SG_NT, 0, st>>>(d_descs);
      else if (ta && !tb) sgemm_big_batched_kernel<true, false><<<grid, SG_NT, 0, st>>>(d_descs);
      else sgemm_big_batched_kernel<true, true><<<grid, SG_NT, 0, st>>>(d_descs);
      count_launch(ctx);
      FL_CUDA(ctx, cudaGetLastError());
      return 0;
    }
  }
  const int64_t gx = cdiv(max_m, BM), gy = cdiv(max_n, BN);
  FL_CHECK(ctx, 2 * gy <= 65535 && count <= 65535, FRACLAP_ERR_UNSUPPORTED, "gemm_batched: too large");
  dim3 grid((unsigned)gx, (unsigned)gy, (unsigned)count);
  if (!ta && !tb) {
    if constexpr (std::is_same<T, double>::value)
      dgemm_small_batched_kernel<<<dim3((unsigned)cdiv(max_m, 32), (unsigned)cdiv(max_n, 32), (unsigned)count), DG_NT, 0, st>>>(d_descs);
    else
      gemm_batched_kernel<T, false, false><<<grid, NT, 0, st>>>(d_descs);
  }
  else if (!ta && tb) gemm_batched_kernel<T, false, true><<<grid, NT, 0, st>>>(d_descs);
  else if (ta && !tb) gemm_batched_kernel<T, true, false><<<grid, NT, 0, st>>>(d_descs);
  else gemm_batched_kernel<T, true, true><<<grid, NT, 0, st>>>(d_descs);
  count_launch(ctx);
  FL_CUDA(ctx, cudaGetLastError());
  return 0;
}

template int gemm<double>(fraclap_ctx*, bool, bool, GemmMode, const GemmDescT<double>&, int, cudaStream_t);
template int gemm<float>(fraclap_ctx*, bool, bool, GemmMode, const GemmDescT<float>&, int, cudaStream_t);
template int gemm_batched<double>(fraclap_ctx*, bool, bool, const GemmDescT<double>*, int, int64_t, int64_t, cudaStream_t);
template int gemm_batched<float>(fraclap_ctx*, bool, bool, const GemmDescT<float>*, int, int64_t, int64_t, cudaStream_t);

}  // namespace fraclap
