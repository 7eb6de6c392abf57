// Stage 1 of the two-stage reduction: dense symmetric -> band of half-width b.
//
// Panel j (columns j0..j0+b-1) is factorised P = Q_j R with Q_j = I - V T V^T
// (compact WY) on one thread-block cluster, its rows split over the CTAs'
// registers or, for taller panels, shared memory; each Householder column costs
// one cluster barrier (the dot products of the pivot column with every other
// column, from which the reflector and its effect on the panel follow).  Panels
// past a cluster's room take a cooperative kernel over all SMs, with FP64 atomics
// and a grid barrier per column.  The trailing matrix is then updated as
// A22 <- Q^T A22 Q = A22 - W V^T - V W^T with X = A22 (V T), W = X - 1/2 V ((V T)^T X),
// through the GEMM engine (symmetric A22 read from its lower triangle;
// lower-triangular rank-2b update).  In FP64 or FP32; the Householder scalars are
// FP64 in both, and FP32 norms are added over the CTAs to 2^-59 of the largest.
#include <cooperative_groups.h>

#include "internal.cuh"

namespace fraclap {
namespace {

namespace cg = cooperative_groups;

constexpr int PQR_NT = 256;
constexpr int kClusterMax = 16;                  // CTAs of the cluster panel kernel (non-portable above 8)
constexpr int kPanelClusterSmemMax = 217 * 1024;  // panel rows one CTA of the cluster holds
constexpr int64_t kPanelFp64Rows = 4096;          // FP64 panels of the cluster kernels
constexpr int kPanelSmemMax = 180 * 1024;  // largest panel slice one CTA holds

// Cooperative panel QR.  P: m x bw panel (ld ldp) in the working matrix.
// On exit P holds R on and above its diagonal (the band block) and the
// reflectors below it; Vout gets the explicit unit lower-trapezoidal V
// (m x bw, ld ldv); tau[bw]; T: bw x bw upper triangular (ld bw).
template <class T>
__global__ void __launch_bounds__(PQR_NT)
panel_qr_kernel(T* P, int64_t ldp, int64_t m, int bw, T* Vout, int64_t ldv,
                double* tau, T* Tf, double* partials, double* gram, unsigned* bar,
                long long limit, int32_t* status, int64_t rows_per_cta) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* S = reinterpret_cast<T*>(smem_raw);  // rows_per_cta x bw, column-major (ld rows_per_cta)
  __shared__ double red[2 * 64 + 4];
  __shared__ double sw[64];
  __shared__ double s_coef[4];  // beta, v0, tau
  const unsigned G = gridDim.x;
  const int64_t rb = (int64_t)blockIdx.x * rows_per_cta;
  const int64_t re = (rb + rows_per_cta < m) ? rb + rows_per_cta : m;
  const int64_t nr = (re > rb) ? re - rb : 0;
  const int64_t ld = rows_per_cta;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = PQR_NT / 32;

  for (int c = 0; c < bw; ++c)
    for (int64_t r = tid; r < nr; r += PQR_NT) S[r + c * ld] = P[(rb + r) + c * ldp];
  __syncthreads();

  const int nref = (m < bw) ? (int)m : bw;
  const int stride = 2 * bw;
  for (int c = 0; c < nref; ++c) {
    // column sums over all CTAs: FP64 atomics into one of three buffers
    // (zeroed two columns ahead, after the barrier that ends its last use)
    double* acc = partials + (size_t)(c % 3) * stride;
    // partial dot products over this CTA's rows r >= c
    const int64_t r0 = (c > rb) ? c - rb : 0;  // first local row with global row >= c
    for (int j = c + warp; j < bw; j += nwarp) {
      double s = 0.0;
      for (int64_t r = r0 + lane; r < nr; r += 32) {
        const int64_t gr = rb + r;
        if (j == c && gr == c) continue;  // g_c is the tail sum of squares (rows > c)
        s += (double)S[r + c * ld] * (double)S[r + j * ld];
      }
      s = warp_sum(s);
      if (lane == 0 && s != 0.0) atomicAdd(acc + j, s);
    }
    if (c >= rb && c < re)
      for (int j = c + tid; j < bw; j += PQR_NT) acc[bw + j] = (double)S[(c - rb) + j * ld];
    if (!grid_barrier(bar, G, limit, status)) return;
    if (blockIdx.x == 0)
      for (int t = tid; t < stride; t += PQR_NT) partials[(size_t)((c + 2) % 3) * stride + t] = 0.0;
    for (int t = tid; t < 2 * (bw - c); t += PQR_NT) {
      const int slot = (t < bw - c) ? c + t : bw + c + (t - (bw - c));
      red[(t < bw - c) ? t : 64 + (t - (bw - c))] = __ldcg(acc + slot);
    }
    __syncthreads();
    if (tid == 0) {
      const double tail = red[0], x0 = red[64];
      double beta = x0, v0 = 1.0, tu = 0.0;
      if (tail > 0.0 && m - c > 1) {
        const double alpha = sqrt(x0 * x0 + tail);
        beta = (x0 >= 0.0) ? -alpha : alpha;
        v0 = x0 - beta;
        tu = (beta - x0) / beta;
      }
      s_coef[0] = beta;
      s_coef[1] = v0;
      s_coef[2] = tu;
      if (blockIdx.x == 0) tau[c] = tu;
    }
    __syncthreads();
    const double beta = s_coef[0], v0 = s_coef[1], tu = s_coef[2];
    // w_j = tau v^T p_j, v^T p_j = (g_j - beta p_j(c)) / v0
    for (int j = c + 1 + tid; j < bw; j += PQR_NT) {
      const double g = red[j - c], pc = red[64 + (j - c)];
      sw[j] = (tu == 0.0) ? 0.0 : tu * (g - beta * pc) / v0;
    }
    __syncthreads();
    // update own rows (global row >= c)
    const double inv_v0 = 1.0 / v0;
    for (int64_t r = r0 + tid; r < nr; r += PQR_NT) {
      const int64_t gr = rb + r;
      double vr;
      if (gr == c) {
        vr = 1.0;
        S[r + c * ld] = (T)beta;
      } else {
        vr = (tu == 0.0) ? 0.0 : (double)S[r + c * ld] * inv_v0;
        S[r + c * ld] = (T)vr;
      }
      if (tu != 0.0) {
        const T vt = (T)vr;
        for (int j = c + 1; j < bw; ++j) S[r + j * ld] -= vt * (T)sw[j];
      }
    }
    __syncthreads();
  }
  for (int c = nref; c < bw && blockIdx.x == 0 && tid == 0; ++c) tau[c] = 0.0;

  // write back the panel (R and the reflectors) and the explicit V
  for (int c = 0; c < bw; ++c)
    for (int64_t r = tid; r < nr; r += PQR_NT) {
      const int64_t gr = rb + r;
      const T s = S[r + c * ld];
      P[gr + c * ldp] = s;
      T v = T(0);
      if (c < nref) v = (gr < c) ? T(0) : (gr == c ? T(1) : s);
      Vout[gr + c * ldv] = v;
    }
  // Gram matrix V^T V (upper part) accumulated over CTAs
  for (int p = tid; p < bw * bw; p += PQR_NT) {
    const int i = p % bw, j = p / bw;
    if (i > j || j >= nref) continue;
    double s = 0.0;
    for (int64_t r = 0; r < nr; ++r) {
      const int64_t gr = rb + r;
      if (gr < j) continue;
      const double vi = (gr == i) ? 1.0 : (gr < i ? 0.0 : (double)S[r + i * ld]);
      const double vj = (gr == j) ? 1.0 : (double)S[r + j * ld];
      s += vi * vj;
    }
    if (s != 0.0) atomicAdd(&gram[i + j * bw], s);
  }
  if (!grid_barrier(bar, G, limit, status)) return;
  if (blockIdx.x != 0) return;
  // T: T(i,i) = tau_i, T(0:i, i) = -tau_i T(0:i,0:i) (V^T v_i)(0:i)
  __shared__ double Ts[64 * 64];
  __shared__ double y[64];
  for (int p = tid; p < bw * bw; p += PQR_NT) Ts[p] = 0.0;
  __syncthreads();
  for (int i = 0; i < bw; ++i) {
    const double ti = __ldcg(tau + i);
    if (tid < i) y[tid] = __ldcg(gram + tid + i * bw);
    __syncthreads();
    if (tid < i) {
      double s = 0.0;
      for (int q = tid; q < i; ++q) s += Ts[tid + q * bw] * y[q];
      Ts[tid + i * bw] = -ti * s;
    }
    if (tid == 0) Ts[i + i * bw] = ti;
    __syncthreads();
  }
  for (int p = tid; p < bw * bw; p += PQR_NT) Tf[p] = (T)Ts[p];
}

// Columns j, j + step, ... of T (a warp): the inverse of diag(1/tau) +
// strictly-upper(G), T(k, j) = -tau_k sum_{k < q <= j} G(k, q) T(q, j) from k = j
// down, in FP64; G(i, k) at 65 k + i.
template <class TG, class T>
__device__ __forceinline__ void panel_t_columns(const TG* G, const double* s_tau, int bw, int j, int step, int lane, T* Tf) {
  for (; j < bw; j += step) {
    double a0 = 0.0, a1 = 0.0, t0 = 0.0, t1 = 0.0;  // rows lane and lane + 32: sum so far, T(., j)
    for (int k = j; k >= 0; --k) {
      const double sum = __shfl_sync(0xffffffffu, (k < 32) ? a0 : a1, k & 31);
      const double x = (k == j) ? s_tau[j] : -s_tau[k] * sum;
      if (lane == (k & 31)) {
        if (k < 32) t0 = x;
        else t1 = x;
      }
      if (lane < k) a0 = fma((double)G[k * 65 + lane], x, a0);
      if (lane + 32 < k) a1 = fma((double)G[k * 65 + lane + 32], x, a1);
    }
    if (lane < bw) Tf[lane + j * bw] = (T)t0;
    if (lane + 32 < bw) Tf[lane + 32 + j * bw] = (T)t1;
  }
}

// The same panel factorisation on one thread-block cluster (up to 16 CTAs)
// when the panel fits in their shared memory, with T of the compact WY form.
// Per column, every CTA's partial dot products and the pivot row are written
// into all CTAs' shared memory (distributed shared memory) before one hardware
// cluster barrier and added there in rank order; the buffers alternate by
// column parity, so one barrier a column suffices.  One warp forms the
// reflector's scalars while the others add the columns' sums.  Then G = V^T V
// (each CTA's rows in 4 x 4 register tiles, the partial sums added over the
// cluster), and T, the inverse of diag(1/tau) + strictly-upper(G) (Schreiber
// and Van Loan's form of H_1 ... H_bw = I - V T V^T), column by column, dealt to
// the CTAs, a warp each: T(k, j) = -tau_k sum_{k < q <= j} G(k, q) T(q, j) from
// k = j down, in FP64, which holds for tau_k = 0 as well.
// Bound: the chain of a column (dots, barrier, FP64 scalars, update), some 6 us
// at 480 rows a CTA.  It takes the panels past the register kernel's rows: in FP32
// those of more than some 9000 rows, in FP64 those of a batch's workers with fewer
// than 16 SMs.
// G, a CTA's part and the FP64 sum, in the place of V
template <class T>
constexpr size_t panel_gram_smem() {
  return 64 * 64 * sizeof(T) + 64 * 65 * sizeof(double);
}
template <class T>
__global__ void __launch_bounds__(PQR_NT)
panel_qr_cluster_kernel(T* P, int64_t ldp, int64_t m, int bw, T* Vout, int64_t ldv, double* tau, T* Tf,
                        int rows_per_cta, int ld) {
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* S = reinterpret_cast<T*>(smem_raw);  // rows_per_cta x bw, column-major (ld)
  __shared__ T recv[2][kClusterMax][64];  // every CTA's partial dot products
  __shared__ T piv[2][64];                // the pivot row
  __shared__ double g[64];                // their sums
  __shared__ T swt[64];
  __shared__ double s_tau[64];
  __shared__ double s_coef[3];            // beta, tau, 1 / (x0 - beta)
  const int rank = (int)cluster.block_rank(), CS = (int)cluster.num_blocks();
  const int64_t rb = (int64_t)rank * rows_per_cta;
  const int nr = (int)((rb + rows_per_cta < m) ? rows_per_cta : (m > rb ? m - rb : 0));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = PQR_NT / 32;

  for (int c = 0; c < bw; ++c)
    for (int r = tid; r < nr; r += PQR_NT) S[r + c * ld] = P[(rb + r) + c * ldp];
  cluster.sync();  // every CTA of the cluster runs before its shared memory is written

  const int nref = (m < bw) ? (int)m : bw;
  for (int c = 0; c < nref; ++c) {
    const int buf = c & 1;
    const int r0 = (c > rb) ? (int)((c - rb < nr) ? c - rb : nr) : 0;  // first local row with global row >= c
    {
      // partial dots in the working precision (the cluster sum is FP64); a warp
      // takes columns j = c + warp + 8 q in one pass over its rows
      constexpr int QMAX = 64 / 8;
      T sum[QMAX];
#pragma unroll
      for (int q = 0; q < QMAX; ++q) sum[q] = T(0);
      for (int r = r0 + lane; r < nr; r += 32) {
        const T pc = S[r + c * ld];
        const bool pivot = rb + r == c;  // g_c: rows > c only
#pragma unroll
        for (int q = 0; q < QMAX; ++q) {
          const int j = c + warp + nwarp * q;
          if (j < bw && !(j == c && pivot)) sum[q] += pc * S[r + j * ld];
        }
      }
      // eight sums over 32 lanes: three halving exchanges leave one per lane,
      // two butterflies finish it; four lanes then hold column idx
      int idx = 0;
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        const int half = QMAX >> (s + 1), o = 16 >> s;
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int q = 0; q < QMAX / 2; ++q)
          if (q < half) {
            const T send = up ? sum[q] : sum[q + half];
            const T keep = up ? sum[q + half] : sum[q];
            sum[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
          }
        if (up) idx += half;
      }
      T v = sum[0];
      v += __shfl_xor_sync(0xffffffffu, v, 2);
      v += __shfl_xor_sync(0xffffffffu, v, 1);
      const int j = c + warp + nwarp * idx;
      if (j < bw)
        for (int q = lane & 3; q < CS; q += 4) *cluster.map_shared_rank(&recv[buf][rank][j], q) = v;
    }
    if (c >= rb && c < rb + nr) {
      const int j = tid & 63;
      if (j >= c && j < bw) {
        const T v = S[(int)(c - rb) + j * ld];
        for (int q = tid >> 6; q < CS; q += PQR_NT / 64) *cluster.map_shared_rank(&piv[buf][j], q) = v;
      }
    }
    cluster.sync();
    if (warp == 0) {
      double tail = (lane < CS) ? (double)recv[buf][lane][c] : 0.0;
#pragma unroll
      for (int o = 8; o >= 1; o >>= 1) tail += __shfl_xor_sync(0xffffffffu, tail, o);
      tail = __shfl_sync(0xffffffffu, tail, 0);
      const double x0 = (double)piv[buf][c];
      double beta = x0, tu = 0.0, inv = 0.0;
      if (tail > 0.0 && m - c > 1) {
        if (sizeof(T) == 4) householder_scalars_f32(x0, tail, lane, &beta, &tu, &inv);
        else householder_scalars(x0, tail, lane, &beta, &tu, &inv);
      }
      if (lane == 0) {
        s_coef[0] = beta;
        s_coef[1] = tu;
        s_coef[2] = inv;
        s_tau[c] = tu;
        if (rank == 0) tau[c] = tu;
      }
    } else {
      // the other columns' sums: two lanes a column, rank order halves
      const int t = tid - 32, j = c + 1 + (t >> 1), q0 = (t & 1) * (kClusterMax / 2);
      double s = 0.0;
      if (j < bw)
        for (int q = q0; q < q0 + kClusterMax / 2 && q < CS; ++q) s += (double)recv[buf][q][j];
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      if (j < bw && (t & 1) == 0) g[j] = s;
    }
    __syncthreads();
    const double beta = s_coef[0], tu = s_coef[1], inv = s_coef[2];
    // w_j = tau v^T p_j, v^T p_j = (g_j - beta p_j(c)) / v0
    if (tid < 64 && tid > c && tid < bw) swt[tid] = (T)(tu * (g[tid] - beta * (double)piv[buf][tid]) * inv);
    __syncthreads();
    const T ih = (T)inv, il = (T)(inv - (double)ih);  // the product with inv rounded once
    for (int r = r0 + tid; r < nr; r += PQR_NT) {
      T vt;
      if (rb + r == c) {
        vt = T(1);
        S[r + c * ld] = (T)beta;
      } else {
        const T x = S[r + c * ld];
        vt = (sizeof(T) == 8) ? x * ih : fma(x, ih, x * il);  // 0 when tau = 0 (inv = 0)
        S[r + c * ld] = vt;
      }
      if (tu != 0.0)
        for (int j = c + 1; j < bw; ++j) S[r + j * ld] -= vt * swt[j];
    }
    __syncthreads();
  }
  for (int c = nref + tid; c < bw; c += PQR_NT) {
    s_tau[c] = 0.0;
    if (rank == 0) tau[c] = 0.0;
  }
  // R and the reflectors to P, V to Vout; S becomes V (rows past nr are zero)
  for (int c = 0; c < bw; ++c)
    for (int r = tid; r < rows_per_cta; r += PQR_NT) {
      T v = T(0);
      if (r < nr) {
        const int64_t gr = rb + r;
        const T sv = S[r + c * ld];
        P[gr + c * ldp] = sv;
        if (c < nref) v = (gr < c) ? T(0) : (gr == c ? T(1) : sv);
        Vout[gr + c * ldv] = v;
      }
      S[r + c * ld] = v;
    }
  __syncthreads();
  // this CTA's part of G: entries (ti + 16 a, tj + 16 b) of the upper triangle
  const int ti = tid & 15, tj = tid >> 4;
  T acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
  const int nb = (bw + 15) / 16;
  for (int r = 0; r < nr; ++r) {
    T x[4], y[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      x[a] = (a < nb && ti + 16 * a < bw) ? S[r + (ti + 16 * a) * ld] : T(0);
      y[a] = (a < nb && tj + 16 * a < bw) ? S[r + (tj + 16 * a) * ld] : T(0);
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = a; b < 4; ++b) acc[a][b] += x[a] * y[b];
  }
  __syncthreads();
  T* Gp = S;                                       // 64 x 64: this CTA's part
  double* Gd = reinterpret_cast<double*>(smem_raw + 64 * 64 * sizeof(T));  // [column][row], 64 x 65: the sum
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = a; b < 4; ++b) Gp[(ti + 16 * a) + (tj + 16 * b) * 64] = acc[a][b];
  cluster.sync();
  for (int e = rank * PQR_NT + tid; e < 64 * 64; e += CS * PQR_NT) {
    const int i = e & 63, k = e >> 6;
    if (i >= k || k >= bw) continue;
    T s = T(0);
    for (int q = 0; q < CS; ++q) s += cluster.map_shared_rank(Gp, q)[e];
    for (int q = 0; q < CS; ++q) cluster.map_shared_rank(Gd, q)[k * 65 + i] = (double)s;
  }
  cluster.sync();
  panel_t_columns<double>(Gd, s_tau, bw, rank + CS * warp, CS * nwarp, lane, Tf);
}

// The same factorisation with the panel in registers, for panels of at most 32 R
// rows a CTA: warp w of a CTA holds its rows of columns w, w + NW, ..., lane l
// rows l + 32 i, so that a column's step reads only the reflector from shared
// memory.  A step: every column's dot product with the rows of p_c below the
// pivot goes to all CTAs with the pivot row (gathered first: one row of 16-byte
// stores for each CTA; single values cost some 2 clocks each), one cluster
// barrier, then
//   j = c: sum of squares, the reflector's scalars (FP64, one warp);
//   j > c: w_j = tau (p_j(c) + (p_c^T p_j) / (x0 - beta)), p_j -= w_j v;
//   j < c: G(j, c) = V_j(c) + (p_c^T V_j) / (x0 - beta), the Gram matrix of T.
// Bound: the chain of that step.  GB300, FP32, b = 64, clocks a column at m = 2551
// (5111): dots 680 (820), exchange and barrier 1340 (1350), scalars 2230 (2280), w
// 430 (760), update 1050 (1000), in all some 190 (209) us a panel with T and the
// loads; the kernel on shared memory took 257 and 418.  The band reduction at n =
// 1114 7.0 -> 5.1 ms, 2753 15.6 -> 11.1, 7735 78.2 -> 53.9, FP64 779 7.2 -> 5.8.
// A warp's FP64 operation holds the SM's FP64 pipe for some 16 clocks, so only
// the scalars and w are FP64 there; FP32 panels' sums over the CTAs are carried in
// pairs of FP32 values, some 48 bits.  (The FP32 kernels of 16 and 18 rows a lane
// spill some 50 and 320 bytes a thread.)
template <class T>
constexpr int kPanelRegsWarps = sizeof(T) == 8 ? 8 : 16;
// s + v = s' + e exactly (Knuth)
__device__ __forceinline__ void two_sum(float& s, float v, float& e) {
  const float t = __fadd_rn(s, v), z = __fadd_rn(t, -s);
  e = __fadd_rn(e, __fadd_rn(__fadd_rn(s, -__fadd_rn(t, -z)), __fadd_rn(v, -z)));
  s = t;
}
__device__ __forceinline__ void two_sum(double& s, double v, double&) { s += v; }

// The sum of the first 16 lanes' values >= 0 (the others hold 0), in every lane.  FP32 values are
// added as integers in units of 2^-59 of the largest one's exponent and rounded
// once: no FP64 operation, each of which costs a lone warp some 100 clocks.
__device__ __forceinline__ double warp_sum_nonneg(double v) {
#pragma unroll
  for (int o = 8; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return __shfl_sync(0xffffffffu, v, 0);
}
__device__ __forceinline__ double warp_sum_nonneg(float v) {
  const unsigned bits = __float_as_uint(v) & 0x7fffffffu;
  const unsigned top = __reduce_max_sync(0xffffffffu, bits);
  if (top >= 0x7f800000u) return warp_sum_nonneg((double)v);  // an infinity or a NaN
  const int ex = (int)(bits >> 23), em = (int)(top >> 23);
  const unsigned man = (bits & 0x7fffffu) | (ex > 0 ? 0x800000u : 0u);
  const int drop = max(em, 1) - max(ex, 1);  // man 2^(max(ex, 1) - 150)
  const unsigned long long u = drop < 59 ? ((unsigned long long)man << 35) >> drop : 0ull;
  // values below 2^59, in pieces whose sums fit 32 bits
  const unsigned long long a = __reduce_add_sync(0xffffffffu, (unsigned)(u & 0x7ffffffu));
  const unsigned long long b = __reduce_add_sync(0xffffffffu, (unsigned)((u >> 27) & 0x7ffffffu));
  const unsigned long long c = __reduce_add_sync(0xffffffffu, (unsigned)(u >> 54));
  const unsigned long long total = a + (b << 27) + (c << 54);  // < 2^64
  if (total == 0) return 0.0;
  // total 2^(max(em, 1) - 185) to 53 bits, nearest even, without the FP64 pipe
  const int z = __clzll((long long)total);
  const unsigned long long norm = total << z, rem = norm & 0x7ff;
  unsigned long long d = (norm >> 11) + ((unsigned long long)(1022 + 63 - z + max(em, 1) - 185) << 52);
  if (rem > 0x400 || (rem == 0x400 && (d & 1))) ++d;  // a carry moves to the next exponent
  return __longlong_as_double((long long)d);
}

template <class T, int Q, int R>
__global__ void __launch_bounds__(32 * kPanelRegsWarps<T>, 1)
panel_qr_regs_kernel(T* P, int64_t ldp, int64_t m, int bw, T* Vout, int64_t ldv, double* tau, T* Tf,
                     int rows_per_cta) {
  constexpr int NW = kPanelRegsWarps<T>, NT = 32 * NW;
  constexpr int GL = NW / 4;              // lanes that share a later column's sum, on warps 1 .. 2 GL
  constexpr int EW = 2 * GL + 1;          // the earlier columns' sums, on warps EW and EW + 1
  static_assert(NW * Q <= 64 && (Q & (Q - 1)) == 0 && EW + 2 <= NW, "columns and warps");
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* G = reinterpret_cast<T*>(smem_raw);  // 64 x 65: G(j, c) at 65 c + j
  __shared__ T col[2][32 * R];            // this CTA's rows of the column in work
  __shared__ __align__(16) T part[2][64];               // this CTA's dot products, the pivot row
  __shared__ __align__(16) T recv[2][kClusterMax][64];  // every CTA's
  __shared__ __align__(16) T piv[2][64];
  __shared__ T g[2][64];                  // their sums
  __shared__ T sw[64];
  __shared__ double s_tau[64];
  __shared__ double s_coef[3];            // beta, tau, 1 / (x0 - beta)
  __shared__ T s_work[3];                 // the last in two parts, beta
  __shared__ int s_any;                   // tau != 0
  const int rank = (int)cluster.block_rank(), CS = (int)cluster.num_blocks();
  const int64_t rb = (int64_t)rank * rows_per_cta;
  const int nr = (int)((rb + rows_per_cta < m) ? rows_per_cta : (m > rb ? m - rb : 0));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  T x[Q][R];
#pragma unroll
  for (int q = 0; q < Q; ++q)
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int r = lane + 32 * i, j = warp + NW * q;
      x[q][i] = (r < nr && j < bw) ? P[(rb + r) + j * ldp] : T(0);
    }
  for (int e = tid; e < 64 * 65; e += NT) G[e] = T(0);
  if (tid < 64) {
    s_tau[tid] = 0.0;
    part[0][tid] = part[1][tid] = T(0);
  }
  if (warp == 0) {
#pragma unroll
    for (int i = 0; i < R; ++i) col[0][lane + 32 * i] = x[0][i];
  }
  cluster.sync();  // every CTA of the cluster runs before its shared memory is written

  const int nref = (m < bw) ? (int)m : bw;
  for (int c = 0; c < nref; ++c) {
    const int buf = c & 1;
    const int top = (int)((c > rb) ? c - rb : (c == rb ? 0 : -1));  // rows past `top` lie below the pivot
    const int pr = (c >= rb && c < rb + nr) ? (int)(c - rb) : -1;   // the pivot's row, if it is here
    T pc[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const T v = col[buf][lane + 32 * i];
      pc[i] = (lane + 32 * i > top) ? v : T(0);
    }
    {
      T sum[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        sum[q] = T(0);
#pragma unroll
        for (int i = 0; i < R; ++i) sum[q] += pc[i] * x[q][i];
      }
      // Q sums over 32 lanes: halving exchanges leave one per lane, butterflies
      // finish it; 32 / Q lanes then hold column warp + NW idx
      int idx = 0, o = 16;
#pragma unroll
      for (int half = Q / 2; half >= 1; half >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int q = 0; q < half; ++q) {
          const T send = up ? sum[q] : sum[q + half];
          const T keep = up ? sum[q + half] : sum[q];
          sum[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
        if (up) idx += half;
      }
      T v = sum[0];
#pragma unroll
      for (int d = 16 / Q; d >= 1; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
      if ((lane & (32 / Q - 1)) == 0) part[0][warp + NW * idx] = v;
      if (pr >= 0 && lane == (pr & 31)) {  // one of the first 64 rows: registers 0 and 1
#pragma unroll
        for (int q = 0; q < Q; ++q) part[1][warp + NW * q] = (pr >= 32) ? x[q][R > 1 ? 1 : 0] : x[q][0];
      }
    }
    __syncthreads();
    for (int q = warp; q < CS; q += NW) {
      constexpr int V16 = 64 * (int)sizeof(T) / 16;  // 16-byte pieces of a row
      if (lane < V16)
        reinterpret_cast<int4*>(cluster.map_shared_rank(&recv[buf][rank][0], q))[lane] = reinterpret_cast<const int4*>(part[0])[lane];
      if (pr >= 0 && (lane & (V16 - 1)) == lane)
        reinterpret_cast<int4*>(cluster.map_shared_rank(&piv[buf][0], q))[lane] = reinterpret_cast<const int4*>(part[1])[lane];
    }
    cluster.sync();
    T gs = T(0);
    if (warp == 0) {
      const double tail = warp_sum_nonneg((lane < CS) ? recv[buf][lane][c] : T(0));
      const double x0 = (double)piv[buf][c];
      double beta = x0, tu = 0.0, inv = 0.0;
      // (a float's sum: by its bits, a NaN like the compare)
      const bool some = sizeof(T) == 4 ? __double2hiint(tail) > 0 && __double2hiint(tail) <= 0x7ff00000 : tail > 0.0;
      if (some && m - c > 1) {
        if (sizeof(T) == 4) householder_scalars_f32(x0, tail, lane, &beta, &tu, &inv);
        else householder_scalars(x0, tail, lane, &beta, &tu, &inv);
      }
      if (lane == 0) {
        s_coef[0] = beta;
        s_coef[1] = tu;
        s_coef[2] = inv;
        s_tau[c] = tu;
        if (rank == 0) tau[c] = tu;
      }
    } else if (warp < EW) {
      // the later columns' sums: GL lanes a column
      const int t = tid - 32, j = c + 1 + t / GL, q0 = (t & (GL - 1)) * (kClusterMax / GL);
      T s = T(0), e = T(0);
      if (j < bw)
        for (int q = q0; q < q0 + kClusterMax / GL && q < CS; ++q) two_sum(s, recv[buf][q][j], e);
#pragma unroll
      for (int o = 1; o < GL; o *= 2) {
        const T s2 = __shfl_xor_sync(0xffffffffu, s, o);
        if (sizeof(T) == 4) e += __shfl_xor_sync(0xffffffffu, e, o);
        two_sum(s, s2, e);
      }
      if (j < bw && (t & (GL - 1)) == 0) {
        g[0][j] = s;
        g[1][j] = e;
      }
    } else if (tid - EW * 32 < c) {
      for (int q = 0; q < CS; ++q) gs += recv[buf][q][tid - EW * 32];
    }
    __syncthreads();
    if (tid < 64) {
      if (tid > c && tid < bw) {
        const double sum = (sizeof(T) == 8) ? (double)g[0][tid] : (double)g[0][tid] + (double)g[1][tid];
        sw[tid] = (T)(s_coef[1] * fma(sum, s_coef[2], (double)piv[buf][tid]));
      }
    } else if (tid == 64) {
      const T ih = (T)s_coef[2];
      s_work[0] = ih;  // the products with 1 / (x0 - beta) are rounded once
      s_work[1] = (sizeof(T) == 8) ? T(0) : (T)(s_coef[2] - (double)ih);
      s_work[2] = (T)s_coef[0];
      s_any = s_coef[1] != 0.0;
    }
    __syncthreads();
    const T ih = s_work[0], il = s_work[1], beta = s_work[2];
    const bool any = s_any != 0;
    T w[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) w[q] = sw[warp + NW * q];
    // pc becomes v: 0 above the pivot, 1 in it
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const T v = (sizeof(T) == 8) ? pc[i] * ih : fma(pc[i], ih, pc[i] * il);  // 0 when tau = 0
      pc[i] = (lane + 32 * i == pr) ? T(1) : v;
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int j = warp + NW * q;
      if (j > c && j < bw) {
        if (any) {
#pragma unroll
          for (int i = 0; i < R; ++i) x[q][i] -= pc[i] * w[q];
        }
        if (j == c + 1) {
#pragma unroll
          for (int i = 0; i < R; ++i) col[buf ^ 1][lane + 32 * i] = x[q][i];
        }
      } else if (j == c) {
#pragma unroll
        for (int i = 0; i < R; ++i) {
          if (lane + 32 * i == pr) x[q][i] = beta;
          else if (lane + 32 * i > top) x[q][i] = pc[i];
        }
      }
    }
    if (tid >= EW * 32 && tid - EW * 32 < c) {
      const int j = tid - EW * 32;
      G[c * 65 + j] = piv[buf][j] + ((sizeof(T) == 8) ? gs * ih : fma(gs, ih, gs * il));
    }
    __syncthreads();
  }
  if (rank == 0)
    for (int c = nref + tid; c < bw; c += NT) tau[c] = 0.0;
  // R and the reflectors to P, V to Vout
#pragma unroll
  for (int q = 0; q < Q; ++q)
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int r = lane + 32 * i, j = warp + NW * q;
      if (r < nr && j < bw) {
        const int64_t gr = rb + r;
        P[gr + j * ldp] = x[q][i];
        Vout[gr + j * ldv] = (j >= nref || gr < j) ? T(0) : (gr == j ? T(1) : x[q][i]);
      }
    }
  __syncthreads();
  panel_t_columns<T>(G, s_tau, bw, rank + CS * warp, CS * NW, lane, Tf);
}

// Band extraction: band(off, j) = A(j + off, j) for off <= b, 0 for b < off < ldb.
template <class T>
__global__ void extract_band(const T* A, int64_t lda, int64_t n, int b, T* band, int ldb) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n * ldb) return;
  const int off = (int)(p % ldb);
  const int64_t j = p / ldb;
  const int64_t i = j + off;
  band[p] = (off <= b && i < n) ? A[i + j * lda] : T(0);
}

}  // namespace

int64_t stage1_panels(int64_t n, int b) { return (n > b) ? cdiv(n - b, b) : 0; }

template <class T>
int stage1_take(Arena* ar, int64_t n, int b, int G, Stage1T<T>* s) {
  s->npanel = stage1_panels(n, b);
  s->vtotal = 0;
  for (int64_t j = 0; j < s->npanel; ++j) s->vtotal += (n - j * b - b) * b;
  s->Vstore = ar->take<T>(s->vtotal);
  s->Tstore = ar->take<T>(s->npanel * b * b);
  s->tau = ar->take<double>(s->npanel * b);
  // X and XT are one buffer: the back-transformation's block factors of one step fit it
  const int64_t x = cdiv(n * b, 64) * 64;
  s->xx_len = x + n * b + 2 * (int64_t)b * b;
  s->XX = ar->take<T>(s->xx_len);
  s->X = s->XX;
  s->XT = s->XX ? s->XX + x : nullptr;
  // (up to 64 MiB, n = 4096 in FP64, V T of every panel costs no problem its memory)
  s->XTstore = (sizeof(T) * (size_t)s->vtotal <= ((size_t)64 << 20)) ? ar->take<T>(s->vtotal) : nullptr;
  s->Mm = ar->take<T>((int64_t)b * b);
  s->gram = ar->take<double>((int64_t)b * b);
  s->partials = ar->take<double>(3 * 2 * (int64_t)b);
  return 0;
}

static int panel_grid(fraclap_ctx* ctx, int64_t m, int bw, size_t elem, int64_t* rows_per_cta,
                      size_t* smem) {
  int G = ctx->sm_count;
  if (m < (int64_t)G * 8) G = (int)cdiv(m, 8);
  if (G < 1) G = 1;
  *rows_per_cta = cdiv(m, G);
  G = (int)cdiv(m, *rows_per_cta);
  *smem = (size_t)(*rows_per_cta) * bw * elem;
  return G;
}

template <class T>
using PanelRegsKernel = void (*)(T*, int64_t, int64_t, int, T*, int64_t, double*, T*, int);

// The register kernel for `rows` rows a CTA, or null past its sizes.
template <class T>
PanelRegsKernel<T> panel_regs_kernel(int rows, int b) {
  const int r = (rows + 31) / 32;
  if constexpr (sizeof(T) == 8) {
    if (b <= 32) return r <= 2 ? panel_qr_regs_kernel<T, 4, 2> : r <= 3 ? panel_qr_regs_kernel<T, 4, 3> : r <= 4 ? panel_qr_regs_kernel<T, 4, 4>
                      : r <= 6 ? panel_qr_regs_kernel<T, 4, 6> : r <= 8 ? panel_qr_regs_kernel<T, 4, 8> : nullptr;
    return r <= 2 ? panel_qr_regs_kernel<T, 8, 2> : r <= 3 ? panel_qr_regs_kernel<T, 8, 3> : r <= 4 ? panel_qr_regs_kernel<T, 8, 4>
         : r <= 6 ? panel_qr_regs_kernel<T, 8, 6> : r <= 8 ? panel_qr_regs_kernel<T, 8, 8> : nullptr;
  } else {
    if (b <= 32) return r <= 4 ? panel_qr_regs_kernel<T, 2, 4> : r <= 8 ? panel_qr_regs_kernel<T, 2, 8> : r <= 12 ? panel_qr_regs_kernel<T, 2, 12>
                      : r <= 20 ? panel_qr_regs_kernel<T, 2, 20> : nullptr;
    return r <= 4 ? panel_qr_regs_kernel<T, 4, 4> : r <= 8 ? panel_qr_regs_kernel<T, 4, 8> : r <= 12 ? panel_qr_regs_kernel<T, 4, 12>
         : r <= 16 ? panel_qr_regs_kernel<T, 4, 16> : r <= 18 ? panel_qr_regs_kernel<T, 4, 18> : nullptr;
  }
}

// Panel on one cluster.  Returns 1 (nothing launched) when the panel does not
// fit in a cluster or no cluster of that size can be resident; < 0 on a CUDA
// error.
template <class T>
int panel_cluster(fraclap_ctx* ctx, T* P, int64_t ldp, int64_t m, int b, T* V, double* tau, T* Tf, cudaStream_t st) {
  // FP64: up to the register kernel's 4096 rows the cluster wins over the grid
  // kernel (b = 32, n = 4016: the band reduction 132 -> 117 ms with its panels on
  // the cluster, n = 2351 45 -> 37); past them sixteen SMs' FP64 pipes would lose
  if (sizeof(T) == 8 && m > kPanelFp64Rows) return 1;
  const int64_t most = sizeof(T) == 8 ? kPanelClusterSmemMax - 10 * 1024 : kPanelClusterSmemMax;
  const int64_t cap = most / ((int64_t)b * (int64_t)sizeof(T)) - 1;
  const int limit = std::max(1, std::min(kClusterMax, ctx->sm_count));
  int CS = (int)std::max<int64_t>(cdiv(m, cap), std::min<int64_t>(limit, cdiv(m, sizeof(T) == 8 ? 48 : 128)));
  if (CS > limit) return 1;
  const int rows = (int)cdiv(m, CS);
  CS = (int)cdiv(m, rows);
  const int ld = rows | 1;  // odd: the Gram tiles read 16 columns of a row at once
  auto kern = panel_qr_cluster_kernel<T>;
  PanelRegsKernel<T> regs = panel_regs_kernel<T>(rows, b);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)CS);
  cfg.blockDim = dim3(regs ? 32 * kPanelRegsWarps<T> : PQR_NT);
  cfg.dynamicSmemBytes = regs ? 64 * 65 * sizeof(T) : std::max<size_t>((size_t)ld * b * sizeof(T), panel_gram_smem<T>());
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)CS;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // asked once per context, for kClusterMax CTAs (a batch's workers have fewer SMs,
  // and other numbers of them in another batch): every kernel of the panels is
  // resident at its largest size
  int& fits = ctx->panel_cluster_fits[sizeof(T) == 8 ? 1 : 0];
  if (fits < 0) {
    bool all = true;
    const auto resident = [&](const void* k, int threads, size_t smem) -> int {
      FL_CUDA(ctx, cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
      FL_CUDA(ctx, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
      cudaLaunchAttribute big = attr[0];
      big.val.clusterDim.x = kClusterMax;
      cudaLaunchConfig_t full = cfg;
      full.gridDim = dim3(kClusterMax);
      full.blockDim = dim3((unsigned)threads);
      full.dynamicSmemBytes = smem;
      full.attrs = &big;
      full.numAttrs = 1;
      int clusters = 0;
      if (cudaOccupancyMaxActiveClusters(&clusters, k, &full) != cudaSuccess) cudaGetLastError();
      all = all && clusters >= 1;
      return 0;
    };
    FL_TRY(resident((const void*)kern, PQR_NT, (size_t)most));
    for (int bb : {32, 64})
      for (int r = 1; panel_regs_kernel<T>(r, bb); r += 32)
        FL_TRY(resident((const void*)panel_regs_kernel<T>(r, bb), 32 * kPanelRegsWarps<T>, 64 * 65 * sizeof(T)));
    fits = all ? 1 : 0;
  }
  if (!fits) return 1;
  count_launch(ctx);
  if (regs) FL_CUDA(ctx, cudaLaunchKernelEx(&cfg, regs, P, ldp, m, b, V, m, tau, Tf, rows));
  else FL_CUDA(ctx, cudaLaunchKernelEx(&cfg, kern, P, ldp, m, b, V, m, tau, Tf, rows, ld));
  return 0;
}

// Reduces Aw (n x n, lower triangle valid, overwritten) to band form and
// writes the band (ld 2b, offsets 0..2b-1, zero beyond b) to `band`.
template <class T>
int sy2sb_run(fraclap_ctx* ctx, T* Aw, int64_t n, int64_t lda, int b, T* band, Stage1T<T>* s,
              cudaStream_t st) {
  const int ldb = 2 * b;
  int64_t voff = 0;
  for (int64_t p = 0; p < s->npanel; ++p) {
    const int64_t j0 = p * b, m = n - j0 - b;
    T* P = Aw + (j0 + b) + j0 * lda;
    T* V = s->Vstore + voff;
    T* Tf = s->Tstore + p * b * b;
    const int crc = panel_cluster(ctx, P, lda, m, b, V, s->tau + p * b, Tf, st);
    if (crc < 0) return crc;
    if (crc == 0) {
      // done on one cluster
    } else {
    int64_t rows_per_cta;
    size_t smem;
    const int G = panel_grid(ctx, m, b, sizeof(T), &rows_per_cta, &smem);
    FL_CHECK(ctx, smem <= (size_t)kPanelSmemMax, FRACLAP_ERR_UNSUPPORTED, "sy2sb: panel too tall (%lld)", (long long)m);
    FL_CUDA(ctx, cudaMemsetAsync(s->gram, 0, sizeof(double) * b * b, st));
    FL_CUDA(ctx, cudaMemsetAsync(s->partials, 0, sizeof(double) * 3 * 2 * b, st));
    FL_CUDA(ctx, cudaMemsetAsync(ctx->d_barrier, 0, 2 * sizeof(unsigned), st));
    {
      double* tau = s->tau + p * b;
      int64_t ldp = lda, ldv = m, mm = m;
      int bw = b;
      double* partials = s->partials;
      double* gram = s->gram;
      unsigned* bar = ctx->d_barrier;
      long long limit = ctx->wait_cycles;
      int32_t* status = ctx->d_status;
      void* args[] = {&P, &ldp, &mm, &bw, &V, &ldv, &tau, &Tf, &partials, &gram, &bar, &limit, &status, &rows_per_cta};
      // the permitted maximum, not this panel's size: the attribute belongs to
      // the function, and concurrent callers on other streams share it
      FL_CUDA(ctx, cudaFuncSetAttribute(panel_qr_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPanelSmemMax));
      count_launch(ctx);
      FL_CUDA(ctx, cudaLaunchCooperativeKernel((void*)panel_qr_kernel<T>, dim3(G), dim3(PQR_NT), args, smem, st));
    }
    }
    T* A22 = Aw + (j0 + b) + (j0 + b) * lda;
    using D = GemmDescT<T>;
    // XT = V T  (m x b)
    T* XT = s->XTstore ? s->XTstore + voff : s->XT;
    FL_TRY(gemm<T>(ctx, false, false, kGemmPlain, D{m, b, b, V, m, Tf, b, XT, m, nullptr, 0, nullptr, 0, 0, 1.0, 0.0}, 1, st));
    // X = A22 XT (A22 symmetric, lower triangle); narrow products share their
    // long sums by themselves, the TF32 route splits them into a zeroed X
    const bool tf32 = sizeof(T) == 4 && ctx->tc_scratch;
    if (tf32) FL_CUDA(ctx, cudaMemsetAsync(s->X, 0, sizeof(T) * m * b, st));
    FL_TRY(gemm<T>(ctx, false, false, kGemmSymA, D{m, b, m, A22, lda, XT, m, s->X, m, nullptr, 0, nullptr, 0, 0, 1.0, tf32 ? 1.0 : 0.0}, tf32 ? (int)std::min<int64_t>(cdiv(m, 1024), 16) : 1, st));
    // Mm = XT^T X  (b x b): narrow products share the long sum over a cluster's
    // eight CTAs; past 4096 rows more CTAs with atomics are faster in FP32
    const bool split = sizeof(T) == 4 && m > 4096;
    if (split) FL_CUDA(ctx, cudaMemsetAsync(s->Mm, 0, sizeof(T) * b * b, st));
    FL_TRY(gemm<T>(ctx, true, false, kGemmPlain, D{b, b, m, XT, m, s->X, m, s->Mm, b, nullptr, 0, nullptr, 0, 0, 1.0, split ? 1.0 : 0.0}, split ? (int)cdiv(m, 256) : 1, st));
    // W = X - 1/2 V Mm  (in X)
    FL_TRY(gemm<T>(ctx, false, false, kGemmPlain, D{m, b, b, V, m, s->Mm, b, s->X, m, nullptr, 0, nullptr, 0, 0, -0.5, 1.0}, 1, st));
    // A22 -= W V^T + V W^T  (lower triangle)
    FL_TRY(gemm<T>(ctx, false, true, kGemmLowerC, D{m, m, b, s->X, m, V, m, A22, lda, V, m, s->X, m, b, -1.0, 1.0}, 1, st));
    voff += m * b;
  }
  extract_band<T><<<(unsigned)cdiv(n * ldb, 256), 256, 0, st>>>(Aw, lda, n, b, band, ldb);
  count_launch(ctx);
  FL_CUDA(ctx, cudaGetLastError());
  return 0;
}

// Back-transformation by Q1 = Q_0 Q_1 ... Q_{p-1}: Z <- Q1 Z (n x ncols).
// Applied from the last panel to the first: Z(rows_j, :) -= (V_j T_j) (V_j^T Z(rows_j, :)),
// V_j T_j as the reduction formed it where the caller had room for its n^2 / 2
// entries, else formed again (some 6 us a panel).
template <class T>
int q1_apply_run(fraclap_ctx* ctx, const Stage1T<T>* s, int64_t n, int b, T* Z, int64_t ldz,
                 int64_t ncols, T* W1, cudaStream_t st) {
  int64_t voff = s->vtotal;
  using D = GemmDescT<T>;
  const auto vt = [&](int64_t p, int64_t m, const T* V, const T** XT) -> int {
    *XT = s->XTstore ? s->XTstore + voff : s->XT;
    if (s->XTstore) return 0;
    return gemm<T>(ctx, false, false, kGemmPlain, D{m, b, b, V, m, s->Tstore + p * b * b, b, s->XT, m, nullptr, 0, nullptr, 0, 0, 1.0, 0.0}, 1, st);
  };
  const T* XT;
  if (sizeof(T) == 4 && ctx->tc_scratch) {
    // tensor-core shapes (tall and wide products): W1^T = Z_r^T V (n x b), Z_r -=
    // (V T) W1 -- the same products, transposed
    for (int64_t p = s->npanel - 1; p >= 0; --p) {
      const int64_t j0 = p * b, m = n - j0 - b;
      voff -= m * b;
      const T* V = s->Vstore + voff;
      T* Zr = Z + (j0 + b);
      FL_CUDA(ctx, cudaMemsetAsync(W1, 0, sizeof(T) * b * ncols, st));
      FL_TRY(gemm<T>(ctx, true, false, kGemmPlain, D{ncols, b, m, Zr, ldz, V, m, W1, ncols, nullptr, 0, nullptr, 0, 0, 1.0, 1.0}, (int)std::min<int64_t>(cdiv(m, 1024), 16), st));
      FL_TRY(vt(p, m, V, &XT));
      FL_TRY(gemm<T>(ctx, false, true, kGemmPlain, D{m, ncols, b, XT, m, W1, ncols, Zr, ldz, nullptr, 0, nullptr, 0, 0, -1.0, 1.0}, 1, st));
    }
    return 0;
  }
  for (int64_t p = s->npanel - 1; p >= 0; --p) {
    const int64_t j0 = p * b, m = n - j0 - b;
    voff -= m * b;
    const T* V = s->Vstore + voff;
    T* Zr = Z + (j0 + b);
    // W1 = V^T Zr  (b x ncols); FP64 with 64 tiles of columns or more: the tiles'
    // sums split by the caller (n = 7735, the whole stage 884 -> 810 ms)
    const bool split = sizeof(T) == 8 && ncols >= 64 * 64;
    if (split) FL_CUDA(ctx, cudaMemsetAsync(W1, 0, sizeof(T) * b * ncols, st));
    FL_TRY(gemm<T>(ctx, true, false, kGemmPlain, D{b, ncols, m, V, m, Zr, ldz, W1, b, nullptr, 0, nullptr, 0, 0, 1.0, split ? 1.0 : 0.0}, split ? (int)std::min<int64_t>(cdiv(m, 1024), 16) : 1, st));
    // Zr -= (V T) W1
    FL_TRY(vt(p, m, V, &XT));
    FL_TRY(gemm<T>(ctx, false, false, kGemmPlain, D{m, ncols, b, XT, m, W1, b, Zr, ldz, nullptr, 0, nullptr, 0, 0, -1.0, 1.0}, 1, st));
  }
  return 0;
}

template int stage1_take<double>(Arena*, int64_t, int, int, Stage1T<double>*);
template int stage1_take<float>(Arena*, int64_t, int, int, Stage1T<float>*);
template int sy2sb_run<double>(fraclap_ctx*, double*, int64_t, int64_t, int, double*, Stage1T<double>*, cudaStream_t);
template int sy2sb_run<float>(fraclap_ctx*, float*, int64_t, int64_t, int, float*, Stage1T<float>*, cudaStream_t);
template int q1_apply_run<double>(fraclap_ctx*, const Stage1T<double>*, int64_t, int, double*, int64_t, int64_t, double*, cudaStream_t);
template int q1_apply_run<float>(fraclap_ctx*, const Stage1T<float>*, int64_t, int, float*, int64_t, int64_t, float*, cudaStream_t);

}  // namespace fraclap
