// Stage 2 of the two-stage reduction: band (half-width b) -> tridiagonal,
// by bulge chasing with Householder reflectors of length <= b, and the
// back-transformation by the stage-2 orthogonal factor.
//
// Sweep s annihilates column s below the subdiagonal (reflector on rows
// s+1..s+b), applies it to the diagonal block and, from the right, to the
// block below, which creates a bulge; step k then annihilates the first
// column of the previous window in rows s+1+kb..s+(k+1)b and pushes the
// bulge one window further.  Only that first column is annihilated; the rest
// of the fill stays within 2b-1 diagonals of storage and is absorbed by the
// later sweeps.  Step k of sweep s touches only entries in rows
// [s+1+kb, s+(k+2)b]; step k' of sweep s-1 touches rows from s+k'b on, so
// the two are disjoint once k' >= k+3; at k' = k+2 they share only the
// entry (s+(k+2)b, s+(k+1)b), which step k+2 of sweep s-1 sets to the new
// subdiagonal value beta of its reflector before anything else.  Sweep s may
// therefore start step k as soon as sweep s-1 has finished its step k+1, and
// takes that one entry from the word in which sweep s-1 publishes the beta of
// its step k+2 as soon as it is computed: sweeps run in a pipeline, one CTA per
// sweep in flight, each CTA waiting (bounded in time) for its predecessor.
//
// The reflectors H(s,k) of one sweep act on disjoint rows; H(s,k) and
// H(s',k') with k > k', s > s' or k < k', s < s' act on disjoint rows as
// well, so Q2 = prod_s prod_k H(s,k) = prod_{k descending} prod_{s ascending}
// H(s,k).  For fixed k the reflectors form a staircase shifted by one row per
// sweep; Z <- Q2 Z applies k = 0, 1, ... in turn with s descending, keeping a
// sliding window of b rows of Z in shared memory (one lane per column).
#include "internal.cuh"

namespace fraclap {
namespace {


__device__ __forceinline__ int64_t sb_nsteps(int64_t s, int64_t n, int b) {
  return (n - 2 - s) / b + 1;  // valid for s <= n - 2
}

template <class T>
struct SbArgs {
  T* band;        // ld = 2b, band(i - j, j) = A(i, j)
  int64_t n;
  int b;
  int64_t kmax;   // steps of sweep 0
  T* refl;        // (n-1) * kmax * b
  double* rtau;   // (n-1) * kmax
  int* progress;  // n, completed steps per sweep
  T* beta;        // (n-1) * kmax, subdiagonal values as they are computed (all bits set until then)
  int32_t* status;
  long long limit;
};

// Step of one sweep: thread (t, g) = (tid % B, tid / B) owns row t of the
// step's blocks and the columns u = g + NG i (i < B / NG) of each: the column
// block [x | F] (u = 0 is x, u >= 1 the block F to its right), the diagonal
// block D (symmetric, both triangles) and the block E below it, all in
// registers.  Sums over t (F^T v) are butterfly reduce-scatters inside a warp,
// plus one shared-memory add when a row range spans two warps; sums over u
// (D v, E v) are per-thread partials added across the NG column groups in
// shared memory.  The block E of step k is [x | F] of step k + 1 (same rows,
// columns shifted by b), so it stays in the same registers and step k + 1
// writes it back.
template <class T, int C, int W>
__device__ __forceinline__ T sb_reduce_scatter(T (&v)[C], int lane, int* idx) {
  constexpr int LOGC = (C >= 16) ? 4 : (C >= 8) ? 3 : (C >= 4) ? 2 : (C >= 2) ? 1 : 0;
  static_assert((1 << LOGC) == C && 2 * C <= W, "column count per thread");
  int base = 0;
#pragma unroll
  for (int j = 0; j < LOGC; ++j) {
    const int half = C >> (j + 1);
    const int o = W >> (j + 1);
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int q = 0; q < C / 2; ++q) {
      if (q < half) {
        const T send = up ? v[q] : v[q + half];
        const T keep = up ? v[q + half] : v[q];
        v[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    }
    if (up) base += half;
  }
  T r = v[0];
#pragma unroll
  for (int o = W / (2 * C); o >= 1; o /= 2) r += __shfl_xor_sync(0xffffffffu, r, o);
  *idx = base;
  return r;
}

template <int B, int NG>
struct SbShape {
  static constexpr int C = B / NG;                       // columns per thread
  static constexpr int NT = (B * NG < 32) ? 32 : B * NG;  // threads
  static constexpr int W = (B < 32) ? B : 32;            // lanes of one row range in a warp
  static constexpr int H = B / W;                        // warps one row range spans
  static constexpr int NW = NT / 32;
};

// Named barrier `id` over `count` threads (a multiple of 32).
__device__ __forceinline__ void bar_sync(int id, int count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int count) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// One published word: a NaN is made the canonical one, so that no value is the
// "not yet" pattern of all bits set.
__device__ __forceinline__ void sb_publish(float* p, float v) {
  const unsigned b = (v != v) ? 0x7FC00000u : __float_as_uint(v);
  asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(b) : "memory");
}
__device__ __forceinline__ void sb_publish(double* p, double v) {
  const long long b = (v != v) ? 0x7FF8000000000000ll : __double_as_longlong(v);
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(b) : "memory");
}
__device__ __forceinline__ bool sb_published(const float* p, float* v) {
  unsigned b;
  asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(b) : "l"(p) : "memory");
  *v = __uint_as_float(b);
  return b != 0xFFFFFFFFu;
}
__device__ __forceinline__ bool sb_published(const double* p, double* v) {
  long long b;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(b) : "l"(p) : "memory");
  *v = __longlong_as_double(b);
  return b != -1ll;
}

// The step is a chain, so what it need not wait for is taken off it by two
// extra warps.  The Householder warp forms the next reflector's scalars from
// the column x, the first that a step's update finishes, and publishes beta,
// while the NT working threads finish and store the step, wait for the
// predecessor and load the next D and E; the
// release warp orders the step's stores and advances the progress counter
// while the working threads are already in the next step.  Barriers of a step:
// X (x is in shared memory: the working threads arrive, the Householder warp
// waits), ready (everybody), work (twice, the working threads), done (the
// working threads arrive, the release warp waits); an arrival cannot overtake
// the wait of the step before, which the ready barrier follows.  The abort flag
// alternates with the step, so that a warp that is late to read it at one ready
// barrier does not see what is raised on the way to the next.
//
// Bound: the lag between sweeps, two steps and a hand-over.  GB300, FP32 b = 64,
// n = 8810: 117 ms with the scalars (a chain of some 4000 cycles of FP64
// latency), the release fences and the beta counter on the step's chain, 83 with
// the two warps, 77 with x published before the rest of the update and the
// shorter scalars, 62 with beta as a self-validating word (7.0 us a sweep);
// n = 3001 38 -> 18.5 ms; FP64 b = 32, n = 2304 43.7 -> 29.1 ms, there bound by
// the FP64 pipe (some 8000 of a step's 11000 cycles).
// In a waiting loop that began at t0: true when another CTA has failed or the
// wait has reached its limit (which is then reported).
template <class T>
__device__ __forceinline__ bool sb_give_up(const SbArgs<T>& a, long long t0) {
  if (*(volatile int32_t*)a.status != 0) return true;
  if (clock64() - t0 <= a.limit) return false;
  raise_status(a.status, FRACLAP_ERR_TIMEOUT);
  return true;
}

template <class T, int B, int NG>
__global__ void __launch_bounds__(SbShape<B, NG>::NT + 64) sb2st_kernel(SbArgs<T> a) {
  using Sh = SbShape<B, NG>;
  constexpr int C = Sh::C, W = Sh::W, H = Sh::H, NW = Sh::NW, LDS = B + 1, NT = Sh::NT;
  constexpr int kBarX = 1, kBarReady = 2, kBarWork = 3, kBarDone = 4;
  __shared__ T Ds[B * LDS];     // transpose of D's lower triangle
  __shared__ T xs[B];           // the column x
  __shared__ T red_p[NG][B], red_e[NG][B];
  __shared__ T wpart[H][B];
  __shared__ T kpart[NW];
  __shared__ T wfull[B], eyfull[B], wqfull[B];  // w = p - K v, tau E v, tau F^T v
  __shared__ double s_hh[3];    // beta, tau, 1 / v0
  __shared__ int s_abort[2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t n = a.n;
  constexpr int ldb = 2 * B;
  T* band = a.band;
#define BAND(i, j) band[((i) - (j)) + (int64_t)(j) * ldb]
  if (tid < 2) s_abort[tid] = 0;
  __syncthreads();
  int step = 0;  // over all sweeps of this CTA, the same in every warp

  if (warp == NW) {  // ---- Householder warp (norms in FP64) ----
    for (int64_t s = blockIdx.x; s < n - 1; s += gridDim.x) {
      const int64_t ns = sb_nsteps(s, n, B);
      for (int64_t k = 0; k < ns; ++k, ++step) {
        bar_sync(kBarX, NT + 32);  // xs is complete
        double tail = 0.0;
        for (int j = 1 + lane; j < B; j += 32) tail += (double)xs[j] * (double)xs[j];
        tail = warp_sum(tail);
        const double x0 = (double)xs[0];
        double beta = x0, tu = 0.0, inv = 0.0;
        if (tail > 0.0) {
          if (sizeof(T) == 4) householder_scalars_f32(x0, tail, lane, &beta, &tu, &inv);
          else householder_scalars(x0, tail, lane, &beta, &tu, &inv);
          if (tu == 0.0) inv = 0.0;
        }
        if (lane == 0) {
          s_hh[0] = beta;
          s_hh[1] = tu;
          s_hh[2] = inv;
          a.rtau[s * a.kmax + k] = tu;
          // the entry sweep s+1 reads at step k-2: one word, so nothing to order
          sb_publish(a.beta + s * a.kmax + k, (T)beta);
        }
        bar_sync(kBarReady, NT + 64);
        if (s_abort[step & 1]) return;
      }
    }
    return;
  }
  if (warp == NW + 1) {  // ---- release warp ----
    for (int64_t s = blockIdx.x; s < n - 1; s += gridDim.x) {
      const int64_t ns = sb_nsteps(s, n, B);
      for (int64_t k = 0; k < ns; ++k, ++step) {
        bar_sync(kBarReady, NT + 64);
        if (s_abort[step & 1]) return;
        bar_sync(kBarDone, NT + 32);  // the step's stores are issued
        if (lane == 0) st_release_gpu(a.progress + s, (int)(k + 1));  // orders the CTA's stores (after the barrier)
      }
    }
    return;
  }

  const bool active = tid < B * NG;
  const int t = tid % B, g = active ? tid / B : 0;
  T XF[C];
  for (int64_t s = blockIdx.x; s < n - 1; s += gridDim.x) {
    const int64_t ns = sb_nsteps(s, n, B);
    const int64_t ns_prev = (s > 0) ? sb_nsteps(s - 1, n, B) : 0;
    for (int64_t k = 0; k < ns; ++k, ++step) {
      const int64_t r0 = s + 1 + k * B;
      const int L = (int)((n - r0 < B) ? n - r0 : B);
      const int64_t r1 = r0 + L - 1;
      const int64_t c = (k == 0) ? s : r0 - B;
      const int nf = (int)(r0 - 1 - c);  // 0 at step 0, b - 1 after
      const int Lb = (int)((n - 1 - r1 < B) ? n - 1 - r1 : B);
      // ---- wait for sweep s-1 to have completed step k+1: every warp by itself ----
      if (s > 0) {
        const int need = (int)(k + 2 < ns_prev ? k + 2 : ns_prev);
        if (lane == 0) {
          const long long t0 = clock64();
          while (ld_acquire_gpu(a.progress + (s - 1)) < need)
            if (sb_give_up(a, t0)) {
              s_abort[step & 1] = 1;
              break;
            }
        }
        __syncwarp();
      }
      // ---- load (all of a thread's loads in flight together) ----
      if (k == 0) {
#pragma unroll
        for (int i = 0; i < C; ++i) XF[i] = T(0);
        if (active && g == 0) {
          if (t < L) XF[0] = __ldcg(&BAND(r0 + t, c));
          xs[t] = XF[0];
        }
        bar_arrive(kBarX, NT + 32);
      }
      T Dr[C], Er[C];
#pragma unroll
      for (int i = 0; i < C; ++i) {
        const int u = g + NG * i;
        Dr[i] = (active && t < L && u <= t) ? __ldcg(&BAND(r0 + t, r0 + u)) : T(0);
        Er[i] = (active && t < Lb && u < L) ? __ldcg(&BAND(r1 + 1 + t, r0 + u)) : T(0);
      }
#pragma unroll
      for (int i = 0; i < C; ++i) {
        const int u = g + NG * i;
        if (active && u <= t) Ds[u + t * LDS] = Dr[i];
      }
      // the last entry of E is the subdiagonal value of sweep s-1's step k+2
      if (s > 0 && k + 2 < ns_prev && t == B - 1 && g == (B - 1) % NG && active && Lb == B && L == B) {
        const T* word = a.beta + (s - 1) * a.kmax + k + 2;
        const long long t0 = clock64();
        while (!sb_published(word, &Er[C - 1]))
          if (sb_give_up(a, t0)) {
            s_abort[step & 1] = 1;
            break;
          }
      }
      bar_sync(kBarReady, NT + 64);  // the scalars, D's lower triangle and the abort flag
      if (s_abort[step & 1]) return;
#pragma unroll
      for (int i = 0; i < C; ++i) {
        const int u = g + NG * i;
        if (active && u > t) Dr[i] = Ds[t + u * LDS];  // upper triangle from the transpose
      }
      const double tu = s_hh[1];
      const T inv = (T)s_hh[2];
      const T vt = (t == 0) ? T(1) : xs[t] * inv;  // v, with v(0) = 1
      T vu[C];
#pragma unroll
      for (int i = 0; i < C; ++i) {
        const int u = g + NG * i;
        vu[i] = (u == 0) ? T(1) : xs[u] * inv;
      }
      if (active && g == 0) a.refl[((int64_t)s * a.kmax + k) * B + t] = vt;
      // ---- partial sums: F^T v (over rows), D v and E v (over columns), v^T D v ----
      {
        T pv[C];
#pragma unroll
        for (int i = 0; i < C; ++i) pv[i] = vt * XF[i];
        int idx;
        const T cs = sb_reduce_scatter<T, C, W>(pv, lane, &idx);
        if (active && (lane & (W / C - 1)) == 0) wpart[(t / W) % H][g + NG * idx] = cs;
      }
      T pp = T(0), ep = T(0);
#pragma unroll
      for (int i = 0; i < C; ++i) {
        pp += Dr[i] * vu[i];
        ep += Er[i] * vu[i];
      }
      if (active) {
        red_p[g][t] = pp;
        red_e[g][t] = ep;
      }
      {
        T kk = active ? vt * pp : T(0);
#pragma unroll
        for (int o = 16; o >= 1; o /= 2) kk += __shfl_xor_sync(0xffffffffu, kk, o);
        if (lane == 0) kpart[warp] = kk;
      }
      bar_sync(kBarWork, NT);
      // ---- full sums, once per row / column ----
      if (tid < B) {
        const T tuT = (T)tu;
        T ksum = T(0);
#pragma unroll
        for (int q = 0; q < NW; ++q) ksum += kpart[q];
        const T K = T(0.5) * tuT * tuT * ksum;  // tau/2 p^T v with p = tau D v
        const T vj = (tid == 0) ? T(1) : xs[tid] * inv;
        T ps = T(0), es = T(0), cs = T(0);
#pragma unroll
        for (int q = 0; q < NG; ++q) {
          ps += red_p[q][tid];
          es += red_e[q][tid];
        }
#pragma unroll
        for (int h = 0; h < H; ++h) cs += wpart[h][tid];
        wfull[tid] = tuT * ps - K * vj;
        eyfull[tid] = tuT * es;
        wqfull[tid] = tuT * cs;
      }
      bar_sync(kBarWork, NT);
      // ---- rank-one and rank-two updates in registers ----
      const T wt = wfull[t], eyt = eyfull[t];
      const T beta = (T)s_hh[0];  // before x: the Householder warp then overwrites the scalars
      Er[0] -= eyt * vu[0];
      if (k + 1 < ns) {  // the first column of E is the next step's x
        if (active && g == 0) xs[t] = Er[0];
        bar_arrive(kBarX, NT + 32);
      }
#pragma unroll
      for (int i = 0; i < C; ++i) {
        const int u = g + NG * i;
        XF[i] -= vt * wqfull[u];
        if (u <= t) Dr[i] -= vt * wfull[u] + wt * vu[i];  // only the stored triangle
        if (i > 0) Er[i] -= eyt * vu[i];
      }
      // ---- store x (annihilated), F and D's lower triangle; E moves on ----
      if (active && t < L) {
#pragma unroll
        for (int i = 0; i < C; ++i) {
          const int u = g + NG * i;
          if (u == 0) __stcg(&BAND(r0 + t, c), (t == 0) ? beta : T(0));
          else if (u <= nf) __stcg(&BAND(r0 + t, c + u), XF[i]);
          if (u <= t) __stcg(&BAND(r0 + t, r0 + u), Dr[i]);
        }
      }
#pragma unroll
      for (int i = 0; i < C; ++i) XF[i] = Er[i];
      bar_arrive(kBarDone, NT + 32);
    }
  }
#undef BAND
}

template <class T>
__global__ void band_diagonals(const T* band, int ldb, int64_t n, double* d, double* e) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  d[i] = band[i * ldb];
  if (i + 1 < n) e[i] = band[1 + i * ldb];
}

// Y <- Y Q2^T, i.e. Z <- Q2 Z on the transpose Y = Z^T (ld >= n), so that a
// row of Z is contiguous.  For each step k the reflectors H(s, k), s
// descending, act on a window of B rows of Z that slides up by one row per
// reflector.  A warp owns CPW = 32/P columns of Z; its lanes split the window
// into P parts of R = B/P rows each, held in registers: the dot product of a
// reflector with a column is a partial sum per part plus a butterfly over the
// P parts, and the slide moves one row per part boundary with a shuffle.  The
// CTA stages the reflectors of the next D steps in shared memory (double
// buffered) while it applies the current D; the rows entering the window are
// loaded one batch ahead.  Work: 4 L n flops per reflector of length L.
// Every CTA streams all the reflectors through its shared memory, so the
// CTA's warp count W sets the L2 traffic per column: 16 warps per CTA (one
// CTA per SM) halve it against 8 (two per SM), which matters once the
// columns fill the SMs (at n = 8810 in FP32, 68 against 93 ms for the
// kernel alone); with few columns, 8-warp CTAs spread over more SMs.
template <class T, int B, int P, int W>
__global__ void __launch_bounds__(W * 32, 16 / W)
q2t_apply_kernel(const T* __restrict__ refl, const double* __restrict__ rtau, int64_t n,
                 int64_t kmax, T* Y, int64_t ldy, int64_t ncols) {
  // D = R: a batch of D reflectors slides the window by one full register
  // rotation, and the sweep is padded with zero reflectors (tau = 0) to whole
  // batches, so every slide is unconditional and compiles to renaming.
  constexpr int Q2T_WARPS = W;
  constexpr int R = B / P, CPW = 32 / P, D = R, NT = Q2T_WARPS * 32;
  constexpr int PER = (D * B + NT - 1) / NT;  // staged doubles per thread
  __shared__ T vbuf[2][D][B];
  __shared__ T tbuf[2][D];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int part = lane / CPW, cl = lane % CPW;
  const int64_t col = ((int64_t)blockIdx.x * Q2T_WARPS + warp) * CPW + cl;
  const bool active = col < ncols;
  T* yc = Y + (active ? col : 0);
  const unsigned full = 0xffffffffu;

  for (int64_t k = 0; k < kmax; ++k) {
    const int64_t smax = n - 2 - k * B;
    if (smax < 0) break;
    const int64_t nbatch = (smax + D) / D;  // reflectors s = smax .. 0
    // stage a batch of reflectors (q = batch * D + j  <->  s = smax - q)
    auto fetch = [&](int64_t batch, T* vr, T* tr) {
      for (int e = 0; e < PER; ++e) {
        const int t = threadIdx.x + e * NT;
        T v = T(0);
        if (t < D * B) {
          const int j = t / B, c = t % B;
          const int64_t sj = smax - (batch * D + j);
          if (sj >= 0) v = __ldg(refl + (sj * kmax + k) * B + c);
        }
        vr[e] = v;
      }
      T tv = T(0);
      if (threadIdx.x < D) {
        const int64_t sj = smax - (batch * D + threadIdx.x);
        if (sj >= 0) tv = (T)__ldg(rtau + sj * kmax + k);
      }
      *tr = tv;
    };
    auto store = [&](int buf, const T* vr, T tr) {
      for (int e = 0; e < PER; ++e) {
        const int t = threadIdx.x + e * NT;
        if (t < D * B) vbuf[buf][t / B][t % B] = vr[e];
      }
      if (threadIdx.x < D) tbuf[buf][threadIdx.x] = tr;
    };
    T vr[PER], tr;
    fetch(0, vr, &tr);
    __syncthreads();  // previous k's readers are done with the buffers
    store(0, vr, tr);

    int64_t r0 = n - 1;  // window rows r0 .. r0 + B - 1 (rows >= n are zero)
    T w[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int64_t row = r0 + part * R + i;
      w[i] = (active && row < n) ? yc[row * ldy] : T(0);
    }
    T pf[D];  // rows entering the window during the current batch (part 0)
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const int64_t row = r0 - 1 - j;
      pf[j] = (part == 0 && active && row >= 1 + k * B) ? yc[row * ldy] : T(0);
    }
    __syncthreads();
    for (int64_t batch = 0; batch < nbatch; ++batch) {
      const int buf = (int)(batch & 1);
      const bool more = batch + 1 < nbatch;
      if (more) fetch(batch + 1, vr, &tr);
      T pn[D];  // rows for the next batch
#pragma unroll
      for (int j = 0; j < D; ++j) {
        const int64_t row = r0 - 1 - D - j;
        pn[j] = (more && part == 0 && active && row >= 1 + k * B) ? yc[row * ldy] : T(0);
      }
#pragma unroll
      for (int j = 0; j < D; ++j) {
        const T* v = &vbuf[buf][j][part * R];  // zero (with tau 0) past s = 0
        T d0 = T(0), d1 = T(0);
#pragma unroll
        for (int i = 0; i < R; i += 2) {
          d0 = fma(v[i], w[i], d0);
          if (i + 1 < R) d1 = fma(v[i + 1], w[i + 1], d1);
        }
        T dot = d0 + d1;
#pragma unroll
        for (int o = CPW; o < 32; o <<= 1) dot += __shfl_xor_sync(full, dot, o);
        const T f = tbuf[buf][j] * dot;
#pragma unroll
        for (int i = 0; i < R; ++i) w[i] = fma(-f, v[i], w[i]);
        {  // slide the window up by one row (rows above 1 + kB enter as zeros and are never written)
          const T out = w[R - 1];
          const int64_t leaving = r0 + B - 1;
          if (part == P - 1 && active && leaving < n) yc[leaving * ldy] = out;
          const T prev = __shfl_up_sync(full, out, CPW);
#pragma unroll
          for (int i = R - 1; i > 0; --i) w[i] = w[i - 1];
          w[0] = (part == 0) ? pf[j] : prev;
          --r0;
        }
      }
#pragma unroll
      for (int j = 0; j < D; ++j) pf[j] = pn[j];
      if (more) {
        store(buf ^ 1, vr, tr);
        __syncthreads();
      }
    }
#pragma unroll
    for (int i = 0; i < R; ++i) {  // flush the final window (rows 1 + kB ..)
      const int64_t row = r0 + part * R + i;
      if (active && row < n && row >= 1 + k * B) yc[row * ldy] = w[i];
    }
  }
}

// ---------------------------------------------------------------------------
// Y <- Y Q2^T in blocks (b = 32 and 64).  For one step k, B reflectors of
// consecutive sweeps s = qB .. qB + B - 1 act on 2B - 1 rows from
// base = 1 + kB + qB; their product H(qB) ... H(qB + B - 1) is I - V T V^T with
// V(i + t, i) = v_i(t), a parallelogram, and T upper triangular.  The factor
// -U = -V T (stored by columns of 2B rows) is formed once per block by
// q2_factor_kernel (as many steps at a time as the scratch holds); q2_block_kernel then streams the blocks: a CTA owns NCB
// columns of Z, keeps the 2B rows of the window in shared memory, and for each
// block forms W = V^T Z and Z += (-U) W as two small products in registers.
// The next block's window is B rows higher: the upper half becomes the lower
// one, the finished lower half goes to global memory and the rows that enter
// (fetched a block ahead) take its place.
//
// Why: applied one by one, every reflector costs a dot product over the lanes
// that share a column (three shuffles) and a one-row slide, a serial chain of
// some 190 ns per reflector at n = 8810, 16 % of the FP32 pipe; in blocks the
// FMAs are independent and run in packed pairs, for 1.4 times the flops (the
// factor U fills the parallelogram; the loops skip its zero corners).  What
// bounds them now is the shared-memory bandwidth (1.5 to 2 bytes per FMA at
// 8 x 4 and 4 x 4 outputs a thread) and the latency of eight warps an SM.
// GB300, the whole stage: FP32 n = 8810, b = 64 112 -> 68 ms (of which the
// factors some 9), n = 3001 12.1 -> 5 ms; FP64 n = 2304, b = 32 79 -> 39 ms,
// n = 751 8.6 -> 4.8 ms, bound by the FP64 pipe.
// ---------------------------------------------------------------------------
template <class T>
struct Pair2;  // two values along the rows of an operand, multiplied by one broadcast value
template <>
struct Pair2<float> {
  unsigned long long v;
  static __device__ __forceinline__ Pair2 of(float a, float b) {
    Pair2 p;
    asm("mov.b64 %0, {%1, %2};" : "=l"(p.v) : "f"(a), "f"(b));
    return p;
  }
  __device__ __forceinline__ void get(float* a, float* b) const {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(*a), "=f"(*b) : "l"(v));
  }
  __device__ __forceinline__ void fma(const Pair2& x, const Pair2& y) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(v) : "l"(x.v), "l"(y.v));
  }
};
template <>
struct Pair2<double> {
  double x, y;
  static __device__ __forceinline__ Pair2 of(double a, double b) { return Pair2{a, b}; }
  __device__ __forceinline__ void get(double* a, double* b) const { *a = x, *b = y; }
  __device__ __forceinline__ void fma(const Pair2& p, const Pair2& q) {
    x = ::fma(p.x, q.x, x);
    y = ::fma(p.y, q.y, y);
  }
};

// Blocks of step k start at k N0 - k (k - 1) / 2, N0 = ceil((n - 1) / B).
__host__ __device__ inline int64_t q2_block_offset(int64_t k, int64_t N0) { return k * N0 - k * (k - 1) / 2; }

template <int B>
constexpr size_t q2_factor_smem() {
  return sizeof(double) * (3 * B * (B + 1));
}

// One CTA per block: V from the reflectors, G = V^T V, T by the column
// recurrence T(0:i, i) = -tau_i T(0:i, 0:i) G(0:i, i), and -U = -V T, all in FP64
// (-U is rounded once, so the block is orthogonal to the rounding of its
// factors; the FP64 work, some n^2 b / 8 FMAs, is a few per cent of the stage).
template <class T, int B>
__global__ void __launch_bounds__(256) q2_factor_kernel(const T* __restrict__ refl, const double* __restrict__ rtau,
                                                        int64_t n, int64_t kmax, int64_t N0, int64_t first,
                                                        T* __restrict__ ut) {  // blocks from `first` on
  extern __shared__ __align__(128) unsigned char q2_smem[];
  constexpr int LD = B + 1;
  double* Ts = reinterpret_cast<double*>(q2_smem);
  double* G = Ts + B * LD;
  double* V = G + B * LD;  // V[i][t] (converted once: a conversion costs the FP64 pipe as much as an FMA)
  __shared__ double tau[B];
  const int tid = threadIdx.x;
  // block index -> (k, q): row k of the triangle has N0 - k blocks
  const int64_t blk = first + blockIdx.x;
  int64_t k = (int64_t)((2.0 * N0 + 1.0 - sqrt((2.0 * N0 + 1.0) * (2.0 * N0 + 1.0) - 8.0 * (double)blk)) * 0.5);
  if (k < 0) k = 0;
  while (k > 0 && q2_block_offset(k, N0) > blk) --k;
  while (q2_block_offset(k + 1, N0) <= blk) ++k;
  const int64_t q = blk - q2_block_offset(k, N0), smax = n - 2 - k * B;
  for (int e = tid; e < B * B; e += 256) {
    const int64_t s = q * B + e / B;
    V[(e / B) * LD + e % B] = (s <= smax) ? (double)refl[(s * kmax + k) * B + e % B] : 0.0;
  }
  if (tid < B) tau[tid] = (q * B + tid <= smax) ? rtau[(q * B + tid) * kmax + k] : 0.0;
  __syncthreads();
  for (int e = tid; e < B * B; e += 256) {
    const int i = e % B, j = e / B, o = j - i;  // i < j: rows j .. i + B - 1
    Ts[i * LD + j] = 0.0;
    if (o <= 0) continue;
    double sum = 0.0;
    for (int t = 0; t < B - o; ++t) sum = ::fma(V[j * LD + t], V[i * LD + t + o], sum);
    G[i * LD + j] = sum;
  }
  __syncthreads();
  // row i of T by four lanes: T(i, j) = -tau_j sum_{i <= p < j} T(i, p) G(p, j)
  if (tid < 4 * B) {
    const int i = tid >> 2, part = tid & 3;
    if (part == 0) Ts[i * LD + i] = tau[i];
    for (int j = 1; j < B; ++j) {
      double sum = 0.0;
      __syncwarp();
      if (i < j)
        for (int p = i + part; p < j; p += 4) sum = ::fma(Ts[i * LD + p], G[p * LD + j], sum);
      sum += __shfl_xor_sync(0xffffffffu, sum, 1);
      sum += __shfl_xor_sync(0xffffffffu, sum, 2);
      if (i < j && part == 0) Ts[i * LD + j] = -tau[j] * sum;
    }
  }
  __syncthreads();
  // -U(r, i) = -sum_{i' <= i, 0 <= r - i' < B} V(r, i') T(i', i), stored [i][r]
  T* out = ut + (int64_t)blockIdx.x * (2 * B * B);
  for (int e = tid; e < 2 * B * B; e += 256) {
    const int r = e % (2 * B), i = e / (2 * B);
    const int lo = (r >= B) ? r - B + 1 : 0, hi = (r < i) ? r : i;
    double sum = 0.0;
    for (int p = lo; p <= hi; ++p) sum = ::fma(V[p * LD + r - p], Ts[p * LD + i], sum);
    out[e] = (T)(-sum);
  }
}

template <class T, int B, int NCB>
struct Q2Shape {
  static constexpr bool F32 = sizeof(T) == 4;
  static constexpr int RT = F32 ? 4 : 2;                       // rows per thread of each half (and of W)
  static constexpr int CT = F32 ? (NCB >= 32 ? 4 : 2) : 2;  // columns per thread
  static constexpr int NT = (B / RT) * (NCB / CT);             // threads
  static constexpr int LC = (NCB / CT < 8) ? NCB / CT : 8;     // lanes of a warp along the columns
  static constexpr int LDV = B + 16 / sizeof(T);
  static constexpr size_t SMEM = sizeof(T) * (2 * B * LDV + 2 * B * B + 2 * B * NCB + B * NCB);
};

template <class T, int N>
struct alignas(sizeof(T) * N) Vec {
  T v[N];
};

template <class T, int B, int NCB>
__global__ void __launch_bounds__(Q2Shape<T, B, NCB>::NT)
q2_block_kernel(const T* __restrict__ refl, const T* __restrict__ ut, int64_t n, int64_t kmax, int64_t N0, int64_t kbeg,
                int64_t kend, T* Y, int64_t ldy, int64_t ncols) {  // steps kbeg .. kend - 1; ut: where block 0's factor would be
  using Sh = Q2Shape<T, B, NCB>;
  using P = Pair2<T>;
  constexpr int RT = Sh::RT, CT = Sh::CT, NT = Sh::NT, LC = Sh::LC, LDV = Sh::LDV;
  constexpr int WC = (NCB / CT) / LC, LG = 32 / LC;
  constexpr int VPER = B * B / NT;
  extern __shared__ __align__(128) unsigned char q2_smem[];
  T* Us = reinterpret_cast<T*>(q2_smem);  // [B][2B]
  T* Vs = Us + 2 * B * B;                 // [2B][LDV], V(r, i)
  T* Zs = Vs + 2 * B * LDV;               // [2][B][NCB]
  T* Ws = Zs + 2 * B * NCB;               // [B][NCB]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g0 = (warp / WC) * LG, g = g0 + lane / LC;        // row group (warp's first, this thread's)
  const int c0 = ((warp % WC) * LC + lane % LC) * CT;         // first column of this thread in the tile
  const int64_t col = (int64_t)blockIdx.x * NCB + c0;
  const int nc = (int)((ncols - col >= CT) ? CT : (ncols > col ? ncols - col : 0));

  auto load_rows = [&](int64_t row0, T (&z)[RT][CT]) {  // rows row0 + g RT + q of the thread's columns
#pragma unroll
    for (int q = 0; q < RT; ++q) {
      const int64_t row = row0 + g * RT + q;
#pragma unroll
      for (int c = 0; c < CT; ++c) z[q][c] = (row < n && c < nc) ? Y[row * ldy + col + c] : T(0);
    }
  };
  auto store_rows = [&](int64_t row0, const T (&z)[RT][CT]) {
#pragma unroll
    for (int q = 0; q < RT; ++q) {
      const int64_t row = row0 + g * RT + q;
#pragma unroll
      for (int c = 0; c < CT; ++c)
        if (row < n && c < nc) Y[row * ldy + col + c] = z[q][c];
    }
  };
  auto put_half = [&](int half, const T (&z)[RT][CT]) {
#pragma unroll
    for (int q = 0; q < RT; ++q) {
      Vec<T, CT> o;
#pragma unroll
      for (int c = 0; c < CT; ++c) o.v[c] = z[q][c];
      *reinterpret_cast<Vec<T, CT>*>(&Zs[(half * B + g * RT + q) * NCB + c0]) = o;
    }
  };
  auto get_half = [&](int half, T (&z)[RT][CT]) {
#pragma unroll
    for (int q = 0; q < RT; ++q) {
      const Vec<T, CT> o = *reinterpret_cast<const Vec<T, CT>*>(&Zs[(half * B + g * RT + q) * NCB + c0]);
#pragma unroll
      for (int c = 0; c < CT; ++c) z[q][c] = o.v[c];
    }
  };
  auto fetch_v = [&](int64_t k, int64_t q, T (&v)[VPER]) {
    const int64_t smax = n - 2 - k * B;
#pragma unroll
    for (int e = 0; e < VPER; ++e) {
      const int p = tid + e * NT;
      const int64_t s = q * B + p / B;
      v[e] = (s <= smax) ? __ldg(refl + (s * kmax + k) * B + p % B) : T(0);
    }
  };
  auto put_v = [&](const T (&v)[VPER]) {
#pragma unroll
    for (int e = 0; e < VPER; ++e) {
      const int p = tid + e * NT, i = p / B, t = p % B;
      Vs[(i + t) * LDV + i] = v[e];
    }
  };
  auto fetch_u = [&](int64_t blk) {
    const T* src = ut + blk * (2 * B * B);
    T* dst = Us;
    constexpr int E = 16 / sizeof(T);
    for (int p = tid * E; p < 2 * B * B; p += NT * E)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst + p)),
                   "l"(src + p)
                   : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  for (int p = tid; p < 2 * B * LDV; p += NT) Vs[p] = T(0);  // the corners outside the parallelogram stay zero
  for (int64_t k = kbeg; k < kend; ++k) {
    const int64_t N = N0 - k, row_k = 1 + k * B;  // blocks N - 1 .. 0, block q starts at row row_k + q B
    if (N <= 0) break;
    __syncthreads();  // the previous step's rows are in global memory, the buffers are free
    T v[VPER], zn[RT][CT];
    fetch_v(k, N - 1, v);
    put_v(v);
    int top = 0;
    load_rows(row_k + (N - 1) * B, zn);
    put_half(0, zn);
    load_rows(row_k + N * B, zn);
    put_half(1, zn);
    for (int64_t q = N - 1; q >= 0; --q) {
      const bool more = q > 0;
      if (more) {
        fetch_v(k, q - 1, v);
        load_rows(row_k + (q - 1) * B, zn);
      }
      __syncthreads();
      fetch_u(q2_block_offset(k, N0) + q);  // last read before this barrier; lands while W is formed
      {  // W = V^T Z: rows i = g RT .. of W, over r = i .. i + B - 1 of the window
        P acc[RT / 2][CT];
#pragma unroll
        for (int a = 0; a < RT / 2; ++a)
#pragma unroll
          for (int c = 0; c < CT; ++c) acc[a][c] = P::of(T(0), T(0));
        const int lo = g0 * RT, hi = (g0 + LG) * RT + B - 1;  // r of the warp's rows
        const T* vp = Vs + g * RT;
        auto dot = [&](int r0, int r1, int half, int sub) {
          const T* zp = Zs + (half * B - sub) * NCB + c0;
#pragma unroll 4
          for (int r = r0; r < r1; ++r) {
            const Vec<T, RT> a = *reinterpret_cast<const Vec<T, RT>*>(vp + r * LDV);
            const Vec<T, CT> z = *reinterpret_cast<const Vec<T, CT>*>(zp + r * NCB);
#pragma unroll
            for (int c = 0; c < CT; ++c) {
              const P d = P::of(z.v[c], z.v[c]);
#pragma unroll
              for (int i = 0; i < RT / 2; ++i) acc[i][c].fma(P::of(a.v[2 * i], a.v[2 * i + 1]), d);
            }
          }
        };
        dot(lo, B, top, 0);
        dot(B, hi < 2 * B ? hi : 2 * B, top ^ 1, B);
#pragma unroll
        for (int i = 0; i < RT / 2; ++i) {
          Vec<T, CT> w0, w1;
#pragma unroll
          for (int c = 0; c < CT; ++c) acc[i][c].get(&w0.v[c], &w1.v[c]);
          T* wp = Ws + (g * RT + 2 * i) * NCB + c0;
          *reinterpret_cast<Vec<T, CT>*>(wp) = w0;
          *reinterpret_cast<Vec<T, CT>*>(wp + NCB) = w1;
        }
      }
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
      if (more) put_v(v);
      {  // Z += (-U) W: rows g RT .. of either half; the lower half starts at i = row + 1
        P at[RT / 2][CT], ab[RT / 2][CT];  // the change of Z, added to it once
#pragma unroll
        for (int i = 0; i < RT / 2; ++i)
#pragma unroll
          for (int c = 0; c < CT; ++c) at[i][c] = ab[i][c] = P::of(T(0), T(0));
        const T* up = Us + g * RT;
        const T* wp = Ws + c0;
        const int lo = g0 * RT + 1;  // smaller i have zeros in every lower row of this warp
        auto wdup = [&](int i, P (&d)[CT]) {
          const Vec<T, CT> w = *reinterpret_cast<const Vec<T, CT>*>(wp + i * NCB);
#pragma unroll
          for (int c = 0; c < CT; ++c) d[c] = P::of(w.v[c], w.v[c]);
        };
#pragma unroll 4
        for (int i = 0; i < lo; ++i) {
          P d[CT];
          wdup(i, d);
          const Vec<T, RT> u = *reinterpret_cast<const Vec<T, RT>*>(up + i * (2 * B));
#pragma unroll
          for (int c = 0; c < CT; ++c)
#pragma unroll
            for (int r = 0; r < RT / 2; ++r) at[r][c].fma(P::of(u.v[2 * r], u.v[2 * r + 1]), d[c]);
        }
#pragma unroll 4
        for (int i = lo; i < B; ++i) {
          P d[CT];
          wdup(i, d);
          const Vec<T, RT> u = *reinterpret_cast<const Vec<T, RT>*>(up + i * (2 * B));
          const Vec<T, RT> l = *reinterpret_cast<const Vec<T, RT>*>(up + i * (2 * B) + B);
#pragma unroll
          for (int c = 0; c < CT; ++c)
#pragma unroll
            for (int r = 0; r < RT / 2; ++r) {
              at[r][c].fma(P::of(u.v[2 * r], u.v[2 * r + 1]), d[c]);
              ab[r][c].fma(P::of(l.v[2 * r], l.v[2 * r + 1]), d[c]);
            }
        }
        T zt[RT][CT], zb[RT][CT];
        get_half(top, zt);
        get_half(top ^ 1, zb);
#pragma unroll
        for (int i = 0; i < RT / 2; ++i)
#pragma unroll
          for (int c = 0; c < CT; ++c) {
            T x, y;
            at[i][c].get(&x, &y);
            zt[2 * i][c] += x;
            zt[2 * i + 1][c] += y;
            ab[i][c].get(&x, &y);
            zb[2 * i][c] += x;
            zb[2 * i + 1][c] += y;
          }
        store_rows(row_k + (q + 1) * B, zb);
        if (more) {
          put_half(top, zt);
          put_half(top ^ 1, zn);  // only this thread reads or writes these entries between the barriers
        } else {
          store_rows(row_k + q * B, zt);
        }
      }
      top ^= 1;
    }
  }
}

// 32 x 32 tiled transpose: B(j, i) = A(i, j), A is rows x cols.
template <class T>
__global__ void transpose_kernel(const T* A, int64_t lda, T* Bm, int64_t ldb, int64_t rows,
                                 int64_t cols) {
  __shared__ T tile[32][33];
  const int64_t i0 = (int64_t)blockIdx.x * 32, j0 = (int64_t)blockIdx.y * 32;
  for (int t = threadIdx.y; t < 32; t += blockDim.y) {
    const int64_t i = i0 + threadIdx.x, j = j0 + t;
    if (i < rows && j < cols) tile[t][threadIdx.x] = A[i + j * lda];
  }
  __syncthreads();
  for (int t = threadIdx.y; t < 32; t += blockDim.y) {
    const int64_t j = j0 + threadIdx.x, i = i0 + t;
    if (i < rows && j < cols) Bm[j + i * ldb] = tile[threadIdx.x][t];
  }
}

}  // namespace

template <class T>
int stage2_take(Arena* ar, int64_t n, int b, Stage2T<T>* s) {
  s->kmax = (n >= 2) ? (n - 2) / b + 1 : 0;
  const int64_t nsw = (n >= 2) ? n - 1 : 0;
  s->refl = ar->take<T>(nsw * s->kmax * b);
  s->rtau = ar->take<double>(nsw * s->kmax);
  s->beta = nullptr;
  s->progress = ar->take<int>(n + 1);
  return 0;
}

template <class T, int B, int NG>
int sb2st_launch(fraclap_ctx* ctx, SbArgs<T> a, cudaStream_t st) {
  constexpr int NT = SbShape<B, NG>::NT + 64;  // and the Householder and release warps
  int per_sm = 0;
  FL_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sb2st_kernel<T, B, NG>, NT, 0));
  FL_CHECK(ctx, per_sm >= 1, FRACLAP_ERR_UNSUPPORTED, "sb2st: kernel does not fit on an SM");
  int64_t G = (int64_t)ctx->sm_count * per_sm;
  if (G > a.n - 1) G = a.n - 1;
  void* args[] = {&a};
  count_launch(ctx);
  FL_CUDA(ctx, cudaLaunchCooperativeKernel((void*)sb2st_kernel<T, B, NG>, dim3((unsigned)G), dim3(NT), args, 0, st));
  return 0;
}

template <class T>
int sb2st_run(fraclap_ctx* ctx, T* band, int64_t n, int b, double* d, double* e, Stage2T<T>* s,
              cudaStream_t st) {
  if (n >= 2) {
    FL_CUDA(ctx, cudaMemsetAsync(s->progress, 0, sizeof(int) * (n + 1), st));
    FL_CUDA(ctx, cudaMemsetAsync(s->beta, 0xFF, sizeof(T) * (n - 1) * s->kmax, st));
    FL_CUDA(ctx, cudaMemsetAsync(s->rtau, 0, sizeof(double) * (n - 1) * s->kmax, st));
    SbArgs<T> a{band, n, b, s->kmax, s->refl, s->rtau, s->progress, s->beta, ctx->d_status,
                ctx->wait_cycles};
    int rc = 0;
    switch (b) {
      case 4: rc = sb2st_launch<T, 4, 4>(ctx, a, st); break;
      case 8: rc = sb2st_launch<T, 8, 4>(ctx, a, st); break;
      case 16: rc = sb2st_launch<T, 16, 4>(ctx, a, st); break;
      case 32: rc = sb2st_launch<T, 32, 4>(ctx, a, st); break;
      case 64: rc = sb2st_launch<T, 64, 4>(ctx, a, st); break;
      default: FL_CHECK(ctx, false, FRACLAP_ERR_UNSUPPORTED, "sb2st: band width %d", b);
    }
    if (rc) return rc;
  }
  if (n >= 1) {
    band_diagonals<T><<<(unsigned)cdiv(n, 256), 256, 0, st>>>(band, 2 * b, n, d, e);
    count_launch(ctx);
    FL_CUDA(ctx, cudaGetLastError());
  }
  return 0;
}

template <class T>
int transpose_run(fraclap_ctx* ctx, const T* A, int64_t lda, T* Bm, int64_t ldb, int64_t rows,
                  int64_t cols, cudaStream_t st) {
  if (rows <= 0 || cols <= 0) return 0;
  dim3 grid((unsigned)cdiv(rows, 32), (unsigned)cdiv(cols, 32));
  FL_CHECK(ctx, grid.y <= 65535, FRACLAP_ERR_UNSUPPORTED, "transpose: too many columns");
  transpose_kernel<T><<<grid, dim3(32, 8), 0, st>>>(A, lda, Bm, ldb, rows, cols);
  count_launch(ctx);
  FL_CUDA(ctx, cudaGetLastError());
  return 0;
}

// The block factors, then the blocks on CTAs of NCB columns each.
template <class T, int B, int NCB>
int q2_blocks_launch(fraclap_ctx* ctx, const Stage2T<T>* s, int64_t n, int64_t ncols, T* Yt, int64_t ldy, T* ut,
                     int64_t ut_len, cudaStream_t st) {
  using Sh = Q2Shape<T, B, NCB>;
  const int64_t N0 = s->kmax, room = std::min<int64_t>(ut_len / (2 * B * B), INT32_MAX);  // N0 = ceil((n - 1) / B) = kmax
  FL_CHECK(ctx, room >= N0, FRACLAP_ERR_ALLOC, "q2 back-transformation: workspace too small");
  constexpr size_t fsm = q2_factor_smem<B>();
  FL_CUDA(ctx, cudaFuncSetAttribute(q2_factor_kernel<T, B>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fsm));
  FL_CUDA(ctx, cudaFuncSetAttribute(q2_block_kernel<T, B, NCB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)Sh::SMEM));
  for (int64_t k = 0; k < N0;) {
    const int64_t first = q2_block_offset(k, N0);
    int64_t e = k + 1;
    while (e < N0 && q2_block_offset(e + 1, N0) - first <= room) ++e;
    q2_factor_kernel<T, B><<<(unsigned)(q2_block_offset(e, N0) - first), 256, fsm, st>>>(s->refl, s->rtau, n, s->kmax, N0,
                                                                                        first, ut);
    count_launch(ctx);
    const T* block0 = reinterpret_cast<const T*>(reinterpret_cast<uintptr_t>(ut) - sizeof(T) * 2 * B * B * (size_t)first);
    q2_block_kernel<T, B, NCB><<<(unsigned)cdiv(ncols, NCB), Sh::NT, Sh::SMEM, st>>>(s->refl, block0, n, s->kmax, N0, k, e,
                                                                                     Yt, ldy, ncols);
    count_launch(ctx);
    k = e;
  }
  FL_CUDA(ctx, cudaGetLastError());
  return 0;
}

// Z <- Q2 Z (n x ncols, ld ldz), through the transposed copy Yt (ld >= ncols).
template <class T>
int q2_apply_run(fraclap_ctx* ctx, const Stage2T<T>* s, int64_t n, int b, T* Z, int64_t ldz,
                 int64_t ncols, T* Yt, int64_t ldy, T* ut, int64_t ut_len, cudaStream_t st) {
  if (n < 2 || ncols <= 0) return 0;
  FL_TRY(transpose_run<T>(ctx, Z, ldz, Yt, ldy, n, ncols, st));
  const int64_t sm = ctx->sm_count > 0 ? ctx->sm_count : 152;
  // FP64 at b = 64: with seven warps an SM the reflectors one by one keep the FP64
  // pipe busy too, for fewer operations (n = 7735 1333 ms against 1363, 4016 185
  // against 187; 2351 64 against 33)
  const bool single = sizeof(T) == 8 && b == 64 && cdiv(ncols, 4) >= 7 * sm;
  if ((b == 64 && ctx->q2_parts == 0 && !single) || b == 32) {
    // Columns per CTA: the fewest columns on the busiest SM, the wider CTA at a
    // tie (it reuses the factors more).  FP32, b = 64, 64 / 32 / 16 columns: n =
    // 7735 52.6 / 58.1 / 76.5 ms, 4741 20.3 / 15.1 / 16.3, 2740 6.8 / 5.1 / 5.5,
    // 1200 1.47 / 1.14 / 0.91.
    const auto cost = [&](int ncb) { return cdiv(cdiv(ncols, ncb), sm) * ncb; };
    int rc = 0;
    if constexpr (sizeof(T) == 8) {
      if (b == 64) rc = q2_blocks_launch<T, 64, 16>(ctx, s, n, ncols, Yt, ldy, ut, ut_len, st);
      else if (cost(16) <= cost(8)) rc = q2_blocks_launch<T, 32, 16>(ctx, s, n, ncols, Yt, ldy, ut, ut_len, st);
      else rc = q2_blocks_launch<T, 32, 8>(ctx, s, n, ncols, Yt, ldy, ut, ut_len, st);
    } else if (b == 64) {
      if (cost(64) <= cost(32) && cost(64) <= cost(16)) rc = q2_blocks_launch<T, 64, 64>(ctx, s, n, ncols, Yt, ldy, ut, ut_len, st);
      else if (cost(32) <= cost(16)) rc = q2_blocks_launch<T, 64, 32>(ctx, s, n, ncols, Yt, ldy, ut, ut_len, st);
      else rc = q2_blocks_launch<T, 64, 16>(ctx, s, n, ncols, Yt, ldy, ut, ut_len, st);
    } else {
      if (cost(32) <= cost(16)) rc = q2_blocks_launch<T, 32, 32>(ctx, s, n, ncols, Yt, ldy, ut, ut_len, st);
      else rc = q2_blocks_launch<T, 32, 16>(ctx, s, n, ncols, Yt, ldy, ut, ut_len, st);
    }
    if (rc) return rc;
    return transpose_run<T>(ctx, Yt, ldy, Z, ldz, ncols, n, st);
  }
  int cpw = 0;
  // parts per window at b = 64: 4 (16 rows per lane, 8 columns per warp),
  // 8 or 16 (fewer rows per lane, more warps over the same columns: the
  // kernel has ncols / (32 / P) warps in all, so small P leaves SMs idle).
  // Default 8: at n = 8810 in FP32 (8-warp CTAs) 123 ms against 140 (P = 4)
  // and 247 (P = 16, a barrier every four reflectors).
  const int parts64 = (ctx->q2_parts == 4 || ctx->q2_parts == 16) ? ctx->q2_parts : 8;
  // 16-warp CTAs once 8-warp CTAs would already cover every SM
  const auto wide = [&](int pp) { return cdiv(ncols, (int64_t)(32 / pp) * 8) >= ctx->sm_count; };
#define FL_Q2T_W(BB, PP, WW)                                                                         \
  {                                                                                                  \
    cpw = 32 / PP;                                                                                   \
    const int64_t grid = cdiv(ncols, (int64_t)cpw * WW);                                             \
    q2t_apply_kernel<T, BB, PP, WW><<<(unsigned)grid, WW * 32, 0, st>>>(s->refl, s->rtau, n, s->kmax, \
                                                                       Yt, ldy, ncols);              \
    count_launch(ctx);                                                                               \
  }
#define FL_Q2T(BB, PP)                    \
  if (b == BB && cpw == 0) {              \
    if (BB == 64 && wide(PP))             \
      FL_Q2T_W(BB, PP, 16)                \
    else                                  \
      FL_Q2T_W(BB, PP, 8)                 \
  }
  FL_Q2T(4, 1)
  FL_Q2T(8, 2)
  FL_Q2T(16, 4)
  if (b == 64) {
    if constexpr (sizeof(T) == 4) {  // FP64 windows of 16 rows would not fit the registers
      if (parts64 == 4) FL_Q2T(64, 4)
    }
    if (parts64 == 8) FL_Q2T(64, 8)
    if (parts64 == 16) FL_Q2T(64, 16)
    if (parts64 == 4) FL_Q2T(64, 8)  // FP64 asked for 4 parts: 8
  }
#undef FL_Q2T
#undef FL_Q2T_W
  FL_CHECK(ctx, cpw != 0, FRACLAP_ERR_UNSUPPORTED, "q2 back-transformation: band width %d not in {4, 8, 16, 32, 64}", b);
  FL_CUDA(ctx, cudaGetLastError());
  return transpose_run<T>(ctx, Yt, ldy, Z, ldz, ncols, n, st);
}

template int stage2_take<double>(Arena*, int64_t, int, Stage2T<double>*);
template int stage2_take<float>(Arena*, int64_t, int, Stage2T<float>*);
template int sb2st_run<double>(fraclap_ctx*, double*, int64_t, int, double*, double*, Stage2T<double>*, cudaStream_t);
template int sb2st_run<float>(fraclap_ctx*, float*, int64_t, int, double*, double*, Stage2T<float>*, cudaStream_t);
template int transpose_run<double>(fraclap_ctx*, const double*, int64_t, double*, int64_t, int64_t, int64_t, cudaStream_t);
template int transpose_run<float>(fraclap_ctx*, const float*, int64_t, float*, int64_t, int64_t, int64_t, cudaStream_t);
template int q2_apply_run<double>(fraclap_ctx*, const Stage2T<double>*, int64_t, int, double*, int64_t, int64_t, double*, int64_t, double*, int64_t, cudaStream_t);
template int q2_apply_run<float>(fraclap_ctx*, const Stage2T<float>*, int64_t, int, float*, int64_t, int64_t, float*, int64_t, float*, int64_t, cudaStream_t);

}  // namespace fraclap
