// MBAR (Shirts & Chodera 2008; "Estimation") by self-consistent iteration in log-sum-exp form.
//
// One iteration is four kernels on the stream:
//   1. log_denominators: for every sample n, log D_n = ln sum_k N_k exp(f_k - u_kn)   (one thread per n)
//   2. state_partials:   for every state i and a chunk of samples, the (max, sum) pair of
//                        exp(-u_in - log D_n)                                       (block per (chunk, i))
//   3. merge_chunks:     f_i <- -ln sum_n ..., the chunks' pairs of each state merged (one warp per state)
//   4. finalize:         gauge f_0 = 0, convergence flag                             (one block)
// Every kernel returns at once when the device flag says the iteration has converged, so the host
// can enqueue iterations in batches and poll the flag between batches.
//
// algdock_mbar's FP64 mode runs the same iteration on stored weights (see "FP64 on stored weights"
// below): the exponentials are formed once per solve instead of twice per iteration.
#include <limits.h>
#include <math.h>

#include <algorithm>
#include <mutex>
#include <string>

#include "internal.cuh"

namespace algdock {
namespace {

constexpr int kPartialThreads = 256;
// Samples per state_partials block: the largest power of two in [8192, 32768] that still gives a
// full wave of blocks (K x chunks >= 152 SMs x 8 resident blocks), so that large solves spread
// each block's merge over more loads and small ones keep every SM busy.
inline int64_t mbar_chunk(int K, int64_t N) {
  int64_t c = 32768;
  while (c > 8192 && (int64_t)K * ((N + c - 1) / c) < 152 * 8) c >>= 1;
  return c;
}

struct MbarState {
  int converged;
  int iters;
  int trip;    // weights path: the iteration left the range the stored weights are exact in
  int ticket;  // weights path: blocks of weight_update that have finished
};

// Online log-sum-exp accumulator: value = m + log(s).
struct Lse {
  double m, s;
};
__device__ inline void lse_add(Lse& a, double x) {
  if (x == -INFINITY) return;
  if (x <= a.m) {
    a.s += exp(x - a.m);
  } else {
    a.s = a.s * exp(a.m - x) + 1.0;
    a.m = x;
  }
}

// (float)v with the instruction's result, by integer operations where value and result are normal
// numbers (as widen).
__device__ __forceinline__ float narrow(double v) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const uint32_t t = (hi & 0x7fffffffu) - 0x38000000u;
  if (t - 0x00100000u >= 0x0fd00000u) return (float)v;
  uint32_t b = __funnelshift_l(lo, t, 3);
  b += (lo << 3) > 0x80000000u - (b & 1u);  // to nearest, ties to even
  return __uint_as_float(b | (hi & 0x80000000u));
}

// Precision mode 1, FP32 exponentials of FP64 arguments.  The FP64 pipe bounds it, so an element takes
// three operations there: x itself, its distance from the maximum (whose sign decides, as it is exact)
// and one multiply-add, s + e below the maximum and s e + 1 above it.  No branch: along a ladder the
// maximum rises at half of the states.  m starts at kLowest in place of -inf (an argument of -inf
// then adds nothing).
// K = 256, N = 1.0e6: 8.8 -> 4.3 ms an iteration, the same bits.
constexpr double kLowest = -1.7976931348623157e308;
__device__ __forceinline__ void lse_add_f32exp(Lse& a, double x) {
  const double d = x - a.m;
  const int hi = __double2hiint(d);
  const bool above = hi >= 0 && (hi | __double2loint(d)) != 0;
  const double e = widen(__expf(-fabsf(narrow(d))));
  a.s = fma(a.s, above ? e : 1.0, above ? 1.0 : e);
  a.m = above ? x : a.m;
}
template <int MODE>
__device__ __forceinline__ void lse_add_mode(Lse& a, double x) {
  if (MODE) lse_add_f32exp(a, x);
  else lse_add(a, x);
}
template <int MODE>
__device__ __forceinline__ Lse lse_none() { return Lse{MODE ? kLowest : -INFINITY, 0.0}; }
template <int MODE>
__device__ __forceinline__ void lse_end(Lse& a) {
  if (MODE && a.m == kLowest && a.s == 0.0) a.m = -INFINITY;
}
__device__ inline Lse lse_merge(Lse a, Lse b) {
  if (b.m == -INFINITY) return a;
  if (a.m == -INFINITY) return b;
  if (a.m >= b.m) return Lse{a.m, a.s + b.s * exp(b.m - a.m)};
  return Lse{b.m, b.s + a.s * exp(a.m - b.m)};
}

constexpr int kDenTile = 256;  // states whose ln N_k + f_k a block holds at a time
template <int MODE>
__global__ void log_denominators(int K, int64_t N, const double* __restrict__ u, const double* __restrict__ logNk,
                                 const double* __restrict__ f, double* logD, const MbarState* st) {
  if (st->converged) return;
  __shared__ double s_g[kDenTile];
  const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const double* col = u + min(n, N - 1);
  Lse a = lse_none<MODE>();
  // eight independent loads in flight, then the updates in the same order as one at a time
  constexpr int kAhead = 8;
  for (int k0 = 0; k0 < K; k0 += kDenTile) {
    const int kn = min(kDenTile, K - k0);
    __syncthreads();
    for (int k = threadIdx.x; k < kn; k += blockDim.x) s_g[k] = logNk[k0 + k] + f[k0 + k];
    __syncthreads();
    int k = 0;
    for (; k + kAhead <= kn; k += kAhead) {
      double v[kAhead];
#pragma unroll
      for (int j = 0; j < kAhead; ++j) v[j] = __ldg(col + (int64_t)(k0 + k + j) * N);
#pragma unroll
      for (int j = 0; j < kAhead; ++j) lse_add_mode<MODE>(a, s_g[k + j] - v[j]);
    }
    for (; k < kn; ++k) lse_add_mode<MODE>(a, s_g[k] - __ldg(col + (int64_t)(k0 + k) * N));
  }
  lse_end<MODE>(a);
  if (n < N) logD[n] = a.m + log(a.s);
}

template <int MODE>
__global__ void __launch_bounds__(kPartialThreads) state_partials(int64_t N, int64_t chunk_len,
                                                                  const double* __restrict__ u,
                                                                  const double* __restrict__ logD, double2* part,
                                                                  int n_chunks, const MbarState* st) {
  if (st->converged) return;
  const int i = blockIdx.y, chunk = blockIdx.x;
  const int64_t begin = (int64_t)chunk * chunk_len;
  const int64_t end = min(N, begin + chunk_len);
  Lse a = lse_none<MODE>();
  const double* ui = u + (int64_t)i * N;
  constexpr int kAhead = 8;
  const int64_t stride = blockDim.x;
  int64_t n = begin + threadIdx.x;
  for (; n + (kAhead - 1) * stride < end; n += kAhead * stride) {
    double v[kAhead], d[kAhead];
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
      v[j] = __ldg(ui + n + j * stride);
      d[j] = __ldg(logD + n + j * stride);
    }
#pragma unroll
    for (int j = 0; j < kAhead; ++j) lse_add_mode<MODE>(a, -v[j] - d[j]);
  }
  for (; n < end; n += stride) lse_add_mode<MODE>(a, -ui[n] - logD[n]);
  lse_end<MODE>(a);
  __shared__ double sm[kPartialThreads], ss[kPartialThreads];
  sm[threadIdx.x] = a.m;
  ss[threadIdx.x] = a.s;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      const Lse r = lse_merge(Lse{sm[threadIdx.x], ss[threadIdx.x]}, Lse{sm[threadIdx.x + w], ss[threadIdx.x + w]});
      sm[threadIdx.x] = r.m;
      ss[threadIdx.x] = r.s;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) part[(int64_t)i * n_chunks + chunk] = make_double2(sm[0], ss[0]);
}

// The gauge f_0 = 0 and the convergence test on f^new (formed by merge_chunks).
__global__ void finalize(int K, double* f, double* fnew, MbarState* st, double tol, int max_iter) {
  if (st->converged) return;
  __shared__ double s_delta[256];
  __syncthreads();
  const double f0 = fnew[0];
  double dmax = 0.0;
  for (int i = threadIdx.x; i < K; i += blockDim.x) {
    const double v = fnew[i] - f0;
    const double d = fabs(v - f[i]);
    dmax = (d > dmax || isnan(d)) ? d : dmax;
  }
  s_delta[threadIdx.x] = dmax;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      const double o = s_delta[threadIdx.x + w];
      if (o > s_delta[threadIdx.x] || isnan(o)) s_delta[threadIdx.x] = o;
    }
    __syncthreads();
  }
  for (int i = threadIdx.x; i < K; i += blockDim.x) f[i] = fnew[i] - f0;
  __syncthreads();
  if (threadIdx.x == 0) {
    st->iters += 1;
    if (s_delta[0] < tol) st->converged = 1;
    else if (st->iters >= max_iter) st->converged = 2;  // stop: not converged
  }
}

// ---------------------------------------------------------------- precision mode 2: FP32
// Every sample's column of u_kn is shifted once by its minimum s_n (in FP64) and stored as FP32,
// w_kn = u_kn - s_n.  The shift cancels exactly: log D_n and the state sums change by -s_n and +s_n
// in turn.  The iterations then run in FP32 (arguments, exponentials, Kahan-compensated sums),
// with FP64 only where the per-thread partial sums meet.  That halves the bytes read per
// iteration and removes FP64 work from the inner loops.
__global__ void shift_columns(int K, int64_t N, const double* __restrict__ u, float* w) {
  const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  double m = INFINITY;
  for (int k = 0; k < K; ++k) m = fmin(m, u[(int64_t)k * N + n]);
  if (!isfinite(m)) m = 0.0;
  for (int k = 0; k < K; ++k) w[(int64_t)k * N + n] = (float)(u[(int64_t)k * N + n] - m);
}

// Online log-sum-exp in FP32, value m + log(s - c) with the Kahan compensation c.  No branch: along a
// ladder the maximum rises at half of the states, so that a warp would take both sides.  Below the
// maximum y = e - c is added; above it the sum becomes s e + 1 and the compensation c e: one
// multiply-add with selected operands.  m starts at kLowestF in place of -inf (an argument of -inf
// then adds nothing).  exp(-|d|) is 2^(-|d| log2 e) on the base-two unit, where results below 2^-126
// are zero: against a sum of at least 1 they and what they leave in c are lost in any case.
// 256 states, 1.0e6 samples: 269 -> 164 us for the denominators (1.02 GB, 92 % of the copy rate), 251 ->
// 200 us for the states' sums, the same bits as with the branch.  Two samples or two states a
// thread, packed (300 us) or not (180, 230 us), were slower.
constexpr float kLowestF = -3.402823466e38f;
struct LseF {
  float m = kLowestF, s = 0.f, c = 0.f;
};
__device__ __forceinline__ void lsef_add(LseF& a, float x) {
  const float d = x - a.m;
  float e;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(-fabsf(d) * 1.4426950408889634f));
  const float y = e - a.c;
  const bool above = x > a.m;
  const float t = fmaf(a.s, above ? e : 1.f, above ? 1.f : y);
  const float c = (t - a.s) - y;
  a.c = above ? a.c * e : c;
  a.s = t;
  a.m = fmaxf(a.m, x);
}
__device__ __forceinline__ float lsef_max(const LseF& a) { return a.m == kLowestF && a.s == 0.f ? -INFINITY : a.m; }

// One (max, sum) pair from every thread's (m, s): the exact maximum M (a float), then
// sum_t s_t exp(m_t - M) with the factor in FP32 (about 1e-7 relative, independent between
// threads) and the sum in FP64, over the warp by shuffles and over the warps in shared memory.
// The result is valid in thread 0; every thread of the block must call it.
__device__ inline Lse block_merge_f32(float m, double s) {
  __shared__ float s_m[kPartialThreads / 32];
  __shared__ double s_s[kPartialThreads / 32];
  const unsigned full = 0xffffffffu;
  float wm = m;
  for (int o = 16; o > 0; o >>= 1) wm = fmaxf(wm, __shfl_xor_sync(full, wm, o));
  double t = (m == -INFINITY) ? 0.0 : s * (double)expf(m - wm);
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(full, t, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) {
    s_m[warp] = wm;
    s_s[warp] = t;
  }
  __syncthreads();
  Lse r{-INFINITY, 0.0};
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
    const float pm = lane < nw ? s_m[lane] : -INFINITY;
    const double ps = lane < nw ? s_s[lane] : 0.0;
    float bm = pm;
    for (int o = 16; o > 0; o >>= 1) bm = fmaxf(bm, __shfl_xor_sync(full, bm, o));
    double u = (pm == -INFINITY) ? 0.0 : ps * (double)expf(pm - bm);
    for (int o = 16; o > 0; o >>= 1) u += __shfl_xor_sync(full, u, o);
    r = Lse{bm == -INFINITY ? -INFINITY : (double)bm, u};
  }
  return r;
}

__global__ void log_denominators_f32(int K, int64_t N, const float* __restrict__ w, const double* __restrict__ logNk,
                                     const double* __restrict__ f, float* logD, const MbarState* st) {
  if (st->converged) return;
  extern __shared__ float g_k[];
  for (int k = threadIdx.x; k < K; k += blockDim.x) g_k[k] = (float)(logNk[k] + f[k]);
  __syncthreads();
  const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  LseF a;
  // sixteen independent loads in flight before the dependent log-sum-exp updates (each thread walks
  // its column; a warp's loads of one state are one coalesced row segment)
  constexpr int kAhead = 16;
  const float* col = w + n;
  int k = 0;
  for (; k + kAhead <= K; k += kAhead) {
    float v[kAhead];
#pragma unroll
    for (int j = 0; j < kAhead; ++j) v[j] = __ldg(col + (int64_t)(k + j) * N);
#pragma unroll
    for (int j = 0; j < kAhead; ++j) lsef_add(a, g_k[k + j] - v[j]);
  }
  for (; k < K; ++k) lsef_add(a, g_k[k] - __ldg(col + (int64_t)k * N));
  logD[n] = lsef_max(a) + logf(a.s - a.c);
}

__global__ void __launch_bounds__(kPartialThreads) state_partials_f32(int64_t N, int64_t chunk_len,
                                                                      const float* __restrict__ w,
                                                                      const float* __restrict__ logD, double2* part,
                                                                      int n_chunks, const MbarState* st) {
  if (st->converged) return;
  const int i = blockIdx.y, chunk = blockIdx.x;
  const int64_t begin = (int64_t)chunk * chunk_len;
  const int64_t end = min(N, begin + chunk_len);
  LseF a;
  const float* wi = w + (int64_t)i * N;
  // sixteen independent pairs of loads in flight per thread, then the dependent updates
  constexpr int kAhead = 16;
  const int64_t stride = blockDim.x;
  int64_t n = begin + threadIdx.x;
  for (; n + (kAhead - 1) * stride < end; n += kAhead * stride) {
    float v[kAhead], d[kAhead];
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
      v[j] = __ldg(wi + n + j * stride);
      d[j] = __ldg(logD + n + j * stride);
    }
#pragma unroll
    for (int j = 0; j < kAhead; ++j) lsef_add(a, -v[j] - d[j]);
  }
  for (; n < end; n += stride) lsef_add(a, -wi[n] - logD[n]);
  // block merge without FP64 exponentials (slow on this GPU): the exact maximum of the partials'
  // maxima, each partial rescaled by an FP32 exp of its (non-positive) offset, the rescaled sums
  // added in FP64; first within each warp, then over the warps
  const Lse r = block_merge_f32(lsef_max(a), (double)a.s - (double)a.c);
  if (threadIdx.x == 0) part[(int64_t)i * n_chunks + chunk] = make_double2(r.m, r.s);
}

// Each state's chunk pairs merged by one warp into f_i^new = -(M + ln S): lanes take every 32nd
// chunk, then a butterfly over the lanes.  F32 (precision mode 2, whose maxima are floats): the
// exact maximum, FP32 rescale factors and an FP64 sum.  Otherwise FP64 log-sum-exp merges (the
// merge is symmetric in its operands, so every lane ends with the same bits).  finalize then
// applies the gauge and the convergence test.
template <bool F32>
__global__ void merge_chunks(int K, int n_chunks, const double2* __restrict__ part, double* fnew,
                             const MbarState* st) {
  if (st->converged) return;
  const int i = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (i >= K) return;
  const unsigned full = 0xffffffffu;
  const double2* pi = part + (int64_t)i * n_chunks;
  if (F32) {
    float M = -INFINITY;
    for (int c = lane; c < n_chunks; c += 32) M = fmaxf(M, (float)pi[c].x);
    for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(full, M, o));
    double S = 0.0;
    if (M != -INFINITY)
      for (int c = lane; c < n_chunks; c += 32)
        if (pi[c].x != -INFINITY) S += pi[c].y * (double)expf((float)pi[c].x - M);
    for (int o = 16; o > 0; o >>= 1) S += __shfl_xor_sync(full, S, o);
    if (lane == 0) fnew[i] = M == -INFINITY ? INFINITY : -((double)M + log(S));
  } else {
    Lse a{-INFINITY, 0.0};
    for (int c = lane; c < n_chunks; c += 32) a = lse_merge(a, Lse{pi[c].x, pi[c].y});
    for (int o = 16; o > 0; o >>= 1) {
      const Lse b{__shfl_xor_sync(full, a.m, o), __shfl_xor_sync(full, a.s, o)};
      a = lse_merge(a, b);
    }
    if (lane == 0) fnew[i] = -(a.m + log(a.s));
  }
}

// Each state's chunk pairs merged into one (max, sum) pair (FP64 log-sum-exp merges, one warp per
// state), for MBAR sharded over samples: the pairs of all processes are merged on the host.
__global__ void merge_chunk_pairs(int K, int n_chunks, const double2* __restrict__ part, double2* out) {
  const int i = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (i >= K) return;
  const unsigned full = 0xffffffffu;
  const double2* pi = part + (int64_t)i * n_chunks;
  Lse a{-INFINITY, 0.0};
  for (int c = lane; c < n_chunks; c += 32) a = lse_merge(a, Lse{pi[c].x, pi[c].y});
  for (int o = 16; o > 0; o >>= 1) {
    const Lse b{__shfl_xor_sync(full, a.m, o), __shfl_xor_sync(full, a.s, o)};
    a = lse_merge(a, b);
  }
  if (lane == 0) out[i] = make_double2(a.m, a.s);
}

__global__ void init_state(int K, const int64_t* Nk, double* logNk, double* f, MbarState* st) {
  for (int k = threadIdx.x; k < K; k += blockDim.x) {
    logNk[k] = Nk[k] > 0 ? log((double)Nk[k]) : -INFINITY;
    f[k] = 0.0;
  }
  if (threadIdx.x == 0) {
    st->converged = 0;
    st->iters = 0;
    st->trip = 0;
    st->ticket = 0;
  }
}

// ---------------------------------------------------------------- FP64 on stored weights
// With W_kn = exp(g_k - u_kn - c_n) stored once, an iteration of f needs no exponential per
// element: with a_k = N_k exp(f_k - g_k),
//   D'_n = sum_k a_k W_kn,   f_k <- g_k - ln sum_n W_kn / D'_n
// (the shifts c_n cancel, and so does a factor common to all a_k).  Two FP64 multiply-adds per
// element and iteration remain, which is what bounds it: GB300 issues 2 FP64 lanes per clock and
// SM, so K = 128, N = 102400 cannot take less than 42 us an iteration (its 105 MB of weights take
// 15 us from HBM).  Measured: a solve of 43 iterations at that size 88.5 -> 3.85 ms (4.00 with one tile a
// block; two log-sum-exp passes with an FP64 exponential per element take 1455 us an iteration), and
// 25.9 -> 1.58 ms an iteration, the forming of the weights included, at K = 256, N = 1e6.
//
// Range.  c_n is the column's maximum, so the largest weight of a column is 1, D'_n is finite and only
// weights below 1e-308 of the largest are lost.  While the spread of f - g stays within kMaxSpread,
// D'_n >= N_k exp(-200) and the lost terms are below 1e-120 of any sum of at least kMinSum.  An
// iteration outside these limits is not applied (trip): the host then runs one log-sum-exp
// iteration from the same f, takes g = f and forms the weights again.  A ladder whose reduced
// energies span several hundred kT takes this turn once, at the start from f = 0.
constexpr int kWTile = 32;             // samples of a tile: W is stored [tile][K][32], zero past N
constexpr int kWStates = 32;           // states per warp at most
constexpr int kWMaxStates = 256;       // eight warps
constexpr double kMaxSpread = 200.0;   // of f - g
constexpr double kMinSum = 1e-150;     // of sum_n W_kn / D'_n

// One block per tile: lane = sample, each warp every eighth state.
__global__ void __launch_bounds__(256) build_weights(int K, int64_t N, const double* __restrict__ u,
                                                     const double* __restrict__ g, double* __restrict__ W) {
  __shared__ long long s_key[8][kWTile];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t n = (int64_t)blockIdx.x * kWTile + lane;
  const bool in = n < N;
  const double* col = u + (in ? n : N - 1);
  // the exact maximum, by integer comparisons: a shift rounded to the high word would be off by up to
  // 2^-20 of an offset common to the column, and the weights or D'_n could leave the range of a double
  long long key = LLONG_MIN;
  for (int k = warp; k < K; k += 8)
    key = max(key, order_key(__double_as_longlong(g[k] - __ldg(col + (int64_t)k * N))));
  s_key[warp][lane] = key;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 8; ++w) key = max(key, s_key[w][lane]);
  const double c = __longlong_as_double(order_key(key));
  double* out = W + (int64_t)blockIdx.x * K * kWTile + lane;
  for (int k = warp; k < K; k += 8)
    out[(int64_t)k * kWTile] = in ? exp((g[k] - __ldg(col + (int64_t)k * N)) - c) : 0.0;
}

// The sums of one iteration.  A block takes tiles blockIdx.x, + gridDim.x, ...: the tile goes to
// shared memory once and serves both passes, D'_n (each warp its states, then one warp adds the
// warps' parts) and the state sums, which stay in registers (lane = sample) over all the block's
// tiles.  Several blocks per SM, so that one loads while another computes; with STAGES = 2 (where two
// tiles a block leave room for three blocks) the next tile also loads during this one's passes.  The reduction of the 32
// accumulators over the lanes halves their number at each step (31 FP64 additions instead of 160:
// at 2 lanes per clock these count).  part[k][block].
template <int NW, int STAGES>
__global__ void __launch_bounds__(32 * NW) weight_pass(int K, int64_t N, const double* __restrict__ W,
                                                       const double* __restrict__ a, double* __restrict__ part,
                                                       const MbarState* st) {
  if (st->converged || st->trip) return;
  extern __shared__ __align__(16) double s_w[];  // STAGES tiles [K][32], then a [K]
  __shared__ double s_part[NW][kWTile];
  __shared__ double s_r[kWTile];
  double* s_a = s_w + STAGES * K * kWTile;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = (K + NW - 1) / NW;  // <= kWStates
  const int k0 = warp * per, kn = max(0, min(per, K - k0));
  for (int k = threadIdx.x; k < K; k += 32 * NW) s_a[k] = a[k];
  double acc[kWStates];
#pragma unroll
  for (int j = 0; j < kWStates; ++j) acc[j] = 0.0;
  const int64_t tiles = (N + kWTile - 1) / kWTile;
  const double* my_a = s_a + k0;
  auto load = [&](int64_t t, int stage) {
    if (t < tiles) {
      const char* src = (const char*)(W + t * K * kWTile);
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(s_w + stage * K * kWTile);
      for (int i = threadIdx.x; i < K * kWTile / 2; i += 32 * NW)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * i), "l"(src + 16 * i) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (STAGES == 2) load(blockIdx.x, 0);
  int stage = 0;
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x, stage ^= STAGES - 1) {
    const double* mine = s_w + (stage * K + k0) * kWTile + lane;
    load(STAGES == 2 ? t + gridDim.x : t, stage ^ (STAGES - 1));
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 1) : "memory");
    __syncthreads();
    double d0 = 0.0, d1 = 0.0;
#pragma unroll
    for (int j = 0; j < kWStates; j += 2) {
      if (j < kn) d0 = fma(my_a[j], mine[j * kWTile], d0);
      if (j + 1 < kn) d1 = fma(my_a[j + 1], mine[(j + 1) * kWTile], d1);
    }
    s_part[warp][lane] = d0 + d1;
    __syncthreads();
    if (warp == (int)(t % NW)) {
      double d = s_part[0][lane];
#pragma unroll
      for (int w = 1; w < NW; ++w) d += s_part[w][lane];
      s_r[lane] = t * kWTile + lane < N ? 1.0 / d : 0.0;
    }
    __syncthreads();
    const double r = s_r[lane];
#pragma unroll
    for (int j = 0; j < kWStates; ++j)
      if (j < kn) acc[j] = fma(mine[j * kWTile], r, acc[j]);
    __syncthreads();  // the tile and s_r are free again
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  // lane l ends with the sum of accumulator l over all lanes
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int j = 0; j < o; ++j) {
      const double give = up ? acc[j] : acc[j + o], keep = up ? acc[j + o] : acc[j];
      acc[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  if (lane < kn) part[(int64_t)(k0 + lane) * gridDim.x + blockIdx.x] = acc[0];
}

// Each state's block sums added by one warp; the last block to finish applies the gauge f_0 = 0, the
// limits above, the convergence test, and the factors a of the next iteration.
__global__ void __launch_bounds__(128) weight_update(int K, int n_part, const double* __restrict__ part,
                                                     const int64_t* __restrict__ Nk, const double* __restrict__ g,
                                                     double* f, double* fnew, double* a, MbarState* st, double tol,
                                                     int max_iter) {
  if (st->converged || st->trip) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int k = blockIdx.x * 4 + warp;
  if (k < K) {
    const double* p = part + (int64_t)k * n_part;
    double s = 0.0;
    for (int b = lane; b < n_part; b += 32) s += p[b];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    // a sum outside the limits (or NaN) becomes a NaN that trips below
    if (lane == 0) fnew[k] = s >= kMinSum && s <= 1.0 / kMinSum ? g[k] - log(s) : NAN;
  }
  __shared__ bool s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&st->ticket, 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // thread t holds states t and t + 128
  __shared__ double s_max[4], s_top[4], s_bot[4];
  const double f0 = __ldcg(fnew);
  double v[2], x[2], delta = 0.0, top = -INFINITY, bot = INFINITY;
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int i = threadIdx.x + 128 * j;
    v[j] = x[j] = 0.0;
    if (i >= K) continue;
    v[j] = __ldcg(fnew + i) - f0;
    x[j] = v[j] - g[i];
    const double d = fabs(v[j] - f[i]);
    delta = (d > delta || isnan(d)) ? d : delta;
    top = fmax(top, x[j]);
    bot = fmin(bot, x[j]);
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double d = __shfl_xor_sync(0xffffffffu, delta, o);
    delta = (d > delta || isnan(d)) ? d : delta;
    top = fmax(top, __shfl_xor_sync(0xffffffffu, top, o));
    bot = fmin(bot, __shfl_xor_sync(0xffffffffu, bot, o));
  }
  if (lane == 0) {
    s_max[warp] = delta;
    s_top[warp] = top;
    s_bot[warp] = bot;
  }
  __syncthreads();
  for (int w = 0; w < 4; ++w) {
    delta = (s_max[w] > delta || isnan(s_max[w])) ? s_max[w] : delta;
    top = fmax(top, s_top[w]);
    bot = fmin(bot, s_bot[w]);
  }
  const bool good = isfinite(delta) && top - bot <= kMaxSpread;
  if (good) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int i = threadIdx.x + 128 * j;
      if (i >= K) continue;
      f[i] = v[j];
      a[i] = (double)Nk[i] * exp(x[j] - top);
    }
  }
  if (threadIdx.x == 0) {
    st->ticket = 0;
    if (!good) {
      st->trip = 1;
    } else {
      st->iters += 1;
      if (delta < tol) st->converged = 1;
      else if (st->iters >= max_iter) st->converged = 2;
    }
  }
}

// g = f (or 0 at the start, where f is 0) and the factors that go with it; the trip is cleared.
__global__ void weight_base(int K, const int64_t* __restrict__ Nk, const double* __restrict__ f, double* g, double* a,
                            MbarState* st) {
  for (int k = threadIdx.x; k < K; k += blockDim.x) {
    g[k] = f[k];
    a[k] = (double)Nk[k];
  }
  if (threadIdx.x == 0) st->trip = 0;
}

// Blocks of a weight_pass launch: three per SM of four warps (two of eight), no more than tiles.
int weight_blocks(int K, int64_t N) {
  const int64_t tiles = (N + kWTile - 1) / kWTile;
  return (int)std::min<int64_t>(tiles, 152 * (K <= 128 ? 3 : 2));
}

// The two passes of a log-sum-exp iteration in FP64 or (mode 1) with FP32 exponentials.
void launch_passes(cudaStream_t s, int K, int64_t N, int64_t chunk_len, int n_chunks, const double* u,
                   const double* logNk, const double* f, double* logD, double2* part, const MbarState* st, int mode) {
  const unsigned blocks = (unsigned)((N + 255) / 256);
  const dim3 grid((unsigned)n_chunks, (unsigned)K);
  if (mode) {
    log_denominators<1><<<blocks, 256, 0, s>>>(K, N, u, logNk, f, logD, st);
    state_partials<1><<<grid, kPartialThreads, 0, s>>>(N, chunk_len, u, logD, part, n_chunks, st);
  } else {
    log_denominators<0><<<blocks, 256, 0, s>>>(K, N, u, logNk, f, logD, st);
    state_partials<0><<<grid, kPartialThreads, 0, s>>>(N, chunk_len, u, logD, part, n_chunks, st);
  }
}

size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

}  // namespace

// The weights path takes every state sampled (an unsampled state's weights have no bound) and up to
// 256 states.
bool mbar_takes_weights(int K, const int64_t* Nk_host) {
  if (K > kWMaxStates) return false;
  for (int k = 0; k < K; ++k)
    if (Nk_host[k] <= 0) return false;
  return true;
}
// Scratch of the weights path: the log-sum-exp solver's, then g[K] | a[K] | part[K][blocks] | W.
size_t mbar_weights_bytes(int K, int64_t N) {
  return (size_t)((N + kWTile - 1) / kWTile) * K * kWTile * sizeof(double);
}
size_t mbar_scratch_bytes(int K, int64_t N);
size_t mbar_scratch_bytes_weights(int K, int64_t N) {
  return align256(mbar_scratch_bytes(K, N)) + align256(16 * (size_t)K) +
         align256((size_t)K * weight_blocks(K, N) * sizeof(double)) + mbar_weights_bytes(K, N);
}

// Scratch layout (bytes): MbarState | logNk[K] | f[K] | fnew[K] | Nk[K] (int64) | part[K][n_chunks] | logD[N]
// (double; float in mode 2), then in mode 2 the shifted FP32 copy w[K][N] (256-byte aligned).
size_t mbar_scratch_bytes(int K, int64_t N) {
  const int64_t chunk_len = mbar_chunk(K, N);
  const int64_t n_chunks = (N + chunk_len - 1) / chunk_len;
  return 64 + 4 * (size_t)K * 8 + (size_t)K * n_chunks * 16 + (size_t)N * 8 + 256;
}
size_t mbar_scratch_bytes_mode(int K, int64_t N, int mode) {
  return mbar_scratch_bytes(K, N) + (mode == 2 ? (size_t)K * N * sizeof(float) + 256 : 0);
}

// One iteration's (max, sum) pair per state over these N samples, given the global N_k and the
// current f (host arrays): sum_n exp(-u_in - log D_n) = sum * exp(max), with log D_n over all K
// states as in the full solve.  Scratch: mbar_pairs_scratch_bytes(K, N).  pairs_host [K][2].
size_t mbar_pairs_scratch_bytes(int K, int64_t N) { return mbar_scratch_bytes(K, N) + 16 * (size_t)K + 256; }

cudaError_t mbar_local_pairs(cudaStream_t s, void* scratch, int K, int64_t N, const double* u_kn,
                             const int64_t* Nk_host, const double* f_host, int mode, double* pairs_host) {
  const int64_t chunk_len = mbar_chunk(K, N);
  const int64_t n_chunks = (N + chunk_len - 1) / chunk_len;
  char* p = (char*)scratch;
  MbarState* st = (MbarState*)p;
  double* logNk = (double*)(p + 64);
  double* f = logNk + K;
  double* fnew = f + K;
  int64_t* Nk = (int64_t*)(fnew + K);
  double2* part = (double2*)(Nk + K);
  double* logD = (double*)(part + (size_t)K * n_chunks);
  const size_t off = ((size_t)((char*)(logD + N) - p) + 255) & ~(size_t)255;
  double2* pairs = (double2*)(p + off);
  cudaError_t e = cudaMemcpyAsync(Nk, Nk_host, sizeof(int64_t) * K, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  init_state<<<1, 256, 0, s>>>(K, Nk, logNk, f, st);
  e = cudaMemcpyAsync(f, f_host, sizeof(double) * K, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  launch_passes(s, K, N, chunk_len, (int)n_chunks, u_kn, logNk, f, logD, part, st, mode);
  merge_chunk_pairs<<<(unsigned)((K * 32 + 255) / 256), 256, 0, s>>>(K, (int)n_chunks, part, pairs);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(pairs_host, pairs, sizeof(double2) * K, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  return e;
}

// Runs the solver on caller-provided scratch (mbar_scratch_bytes(K, N) bytes, 256-byte aligned).
// h_flag: kMbarFlagBytes of pinned host memory used to poll the device state.  weights: iterate on
// stored weights (mode 0, mbar_takes_weights; scratch mbar_scratch_bytes_weights).  Returns 0
// converged, 1 not converged, -1 on a CUDA error (then *err is set).
int mbar_run(cudaStream_t s, void* scratch, int K, int64_t N, const double* u_kn, const int64_t* Nk_host,
             double tol, int max_iter, int mode, bool weights, double* f_host, int* iters, int* h_flag,
             cudaError_t* err) {
  static_assert(sizeof(MbarState) <= kMbarFlagBytes, "the polled state fits the pinned words");
  MbarState* h_state = (MbarState*)h_flag;
  const int64_t chunk_len = mbar_chunk(K, N);
  const int64_t n_chunks = (N + chunk_len - 1) / chunk_len;
  char* p = (char*)scratch;
  MbarState* st = (MbarState*)p;
  double* logNk = (double*)(p + 64);
  double* f = logNk + K;
  double* fnew = f + K;
  int64_t* Nk = (int64_t*)(fnew + K);
  double2* part = (double2*)(Nk + K);
  double* logD = (double*)(part + (size_t)K * n_chunks);
  cudaError_t e = cudaMemcpyAsync(Nk, Nk_host, sizeof(int64_t) * K, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) { *err = e; return -1; }
  init_state<<<1, 256, 0, s>>>(K, Nk, logNk, f, st);
  const int threads = 256;
  const unsigned blocks_n = (unsigned)((N + threads - 1) / threads);
  const dim3 grid_p((unsigned)n_chunks, (unsigned)K);
  float* w32 = nullptr;
  if (mode == 2) {
    const size_t off = ((size_t)((char*)(logD + N) - (char*)scratch) + 255) & ~(size_t)255;
    w32 = (float*)((char*)scratch + off);
    shift_columns<<<blocks_n, threads, 0, s>>>(K, N, u_kn, w32);
    e = cudaFuncSetAttribute(log_denominators_f32, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kMaxBlockSmem);
    if (e != cudaSuccess) { *err = e; return -1; }
  }
  auto iterate = [&] {  // one log-sum-exp iteration
    if (mode == 2) {
      log_denominators_f32<<<blocks_n, threads, K * sizeof(float), s>>>(K, N, w32, logNk, f, (float*)logD, st);
      state_partials_f32<<<grid_p, kPartialThreads, 0, s>>>(N, chunk_len, w32, (const float*)logD, part, (int)n_chunks,
                                                            st);
    } else {
      launch_passes(s, K, N, chunk_len, (int)n_chunks, u_kn, logNk, f, logD, part, st, mode);
    }
    const unsigned merge_blocks = (unsigned)((K * 32 + 255) / 256);
    if (mode == 2)
      merge_chunks<true><<<merge_blocks, 256, 0, s>>>(K, (int)n_chunks, part, fnew, st);
    else
      merge_chunks<false><<<merge_blocks, 256, 0, s>>>(K, (int)n_chunks, part, fnew, st);
    finalize<<<1, 256, 0, s>>>(K, f, fnew, st, tol, max_iter);
  };
  auto poll = [&] {  // the device state into h_state
    cudaError_t q = cudaGetLastError();
    if (q == cudaSuccess) q = cudaMemcpyAsync(h_state, st, sizeof(MbarState), cudaMemcpyDeviceToHost, s);
    if (q == cudaSuccess) q = cudaStreamSynchronize(s);
    return q;
  };
  int done = 0;
  int issued = 0;
  int batch = 4;
  if (weights) {
    char* q = p + align256(mbar_scratch_bytes(K, N));
    double* g = (double*)q;
    double* a = g + K;
    double* wpart = (double*)(q + align256(16 * (size_t)K));
    const int blocks = weight_blocks(K, N);
    double* W = (double*)((char*)wpart + align256((size_t)K * blocks * sizeof(double)));
    const bool wide = K > 128;
    const size_t smem = (size_t)K * ((wide ? 1 : 2) * kWTile + 1) * sizeof(double);
    // the limit for the most states, whatever K: another thread's solve may set it between this and a launch
    e = cudaFuncSetAttribute(wide ? weight_pass<8, 1> : weight_pass<4, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)((wide ? kWMaxStates * (kWTile + 1) : 128 * (2 * kWTile + 1)) * sizeof(double)));
    if (e != cudaSuccess) { *err = e; return -1; }
    while (!done) {
      const int applied = issued;  // iterations applied when the weights were last formed
      weight_base<<<1, 256, 0, s>>>(K, Nk, f, g, a, st);
      build_weights<<<(unsigned)((N + kWTile - 1) / kWTile), 256, 0, s>>>(K, N, u_kn, g, W);
      for (bool trip = false; !done && !trip;) {
        for (int b = 0; b < batch && issued < max_iter; ++b, ++issued) {
          if (wide) weight_pass<8, 1><<<blocks, 256, smem, s>>>(K, N, W, a, wpart, st);
          else weight_pass<4, 2><<<blocks, 128, smem, s>>>(K, N, W, a, wpart, st);
          weight_update<<<(unsigned)((K + 3) / 4), 128, 0, s>>>(K, blocks, wpart, Nk, g, f, fnew, a, st, tol, max_iter);
        }
        e = poll();
        if (e != cudaSuccess) { *err = e; return -1; }
        trip = h_state->trip != 0;
        issued = trip ? h_state->iters : issued;
        done = h_state->converged != 0 || issued >= max_iter;
        if (batch < 64) batch *= 2;
      }
      if (done) break;
      const bool moved = issued > applied;
      iterate();
      ++issued;
      if (issued >= max_iter) done = 1;
      if (!moved && applied > 0) break;  // tripped twice in a row
    }
    batch = 4;
  }
  while (!done) {
    for (int b = 0; b < batch && issued < max_iter; ++b, ++issued) iterate();
    e = poll();
    if (e != cudaSuccess) { *err = e; return -1; }
    done = h_state->converged != 0 || issued >= max_iter;
    if (batch < 64) batch *= 2;
  }
  MbarState hs;
  e = cudaMemcpyAsync(&hs, st, sizeof(hs), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(f_host, f, sizeof(double) * K, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) { *err = e; return -1; }
  *iters = hs.iters;
  return hs.converged == 1 ? 0 : 1;
}

}  // namespace algdock

// ------------------------------------------------------------------ allocation-free MBAR
// Callers that must not allocate device memory - a host framework whose caching allocator owns
// all device memory and forbids direct cudaMalloc, or a service that reserves its whole memory
// budget at start-up - use algdock_mbar_noalloc.  Its scratch is this fixed array in the
// library's own device memory, present on every GPU that loads the library until the process
// exits.
namespace {

constexpr size_t kNoallocScratchBytes = (size_t)8 << 20;  // 8 MiB
constexpr int kNoallocMaxDevices = 64;

static __device__ __align__(256) unsigned char g_mbar_noalloc_scratch[kNoallocScratchBytes];

std::mutex g_noalloc_mu;
void* g_noalloc_ptr[kNoallocMaxDevices] = {};

// Device address of the scratch array on the current device.  In host code the array's name is
// only a host-side stand-in, so the address is looked up once per device (with that device
// current) and cached.
cudaError_t noalloc_scratch(int device, void** out) {
  if (device < 0 || device >= kNoallocMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[device]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_mbar_noalloc_scratch);
    if (e != cudaSuccess) return e;
    g_noalloc_ptr[device] = p;
  }
  *out = g_noalloc_ptr[device];
  return cudaSuccess;
}

}  // namespace

extern "C" algdock_status algdock_mbar_noalloc(algdock_ctx* c, int32_t K, int64_t N, const double* u_kn,
                                               const int64_t* N_k, double tol, int32_t max_iter,
                                               int32_t precision_mode, double* f_k, int32_t* iters) {
  if (!c) return ALGDOCK_E_INVALID;
  try {
    if (K < 1 || N < 1 || !u_kn || !N_k || !f_k || !iters || max_iter < 1 || !(tol > 0)) {
      c->err = "mbar_noalloc: bad arguments";
      return ALGDOCK_E_INVALID;
    }
    if (precision_mode != 0 && precision_mode != 1) {
      c->err = "mbar_noalloc: precision_mode must be 0 or 1 (mode 2 keeps an FP32 copy of u_kn, K*N*4 bytes, "
               "which the fixed scratch array does not hold; use algdock_mbar for mode 2)";
      return ALGDOCK_E_INVALID;
    }
    if (K > algdock::kMbarMaxStates) {
      c->err = "mbar_noalloc: K = " + std::to_string(K) + " exceeds the " + std::to_string(algdock::kMbarMaxStates) +
               " states one launch grid dimension can hold";
      return ALGDOCK_E_INVALID;
    }
    int64_t total = 0;
    for (int k = 0; k < K; ++k) {
      if (N_k[k] < 0) {
        c->err = "mbar_noalloc: negative N_k";
        return ALGDOCK_E_INVALID;
      }
      total += N_k[k];
    }
    if (total != N) {
      c->err = "mbar_noalloc: sum of N_k must equal N";
      return ALGDOCK_E_INVALID;
    }
    const size_t need = algdock::mbar_scratch_bytes(K, N);
    if (need > kNoallocScratchBytes) {
      c->err = "mbar_noalloc: K = " + std::to_string(K) + ", N = " + std::to_string(N) + " needs " +
               std::to_string(need) + " bytes of scratch, more than the fixed " +
               std::to_string(kNoallocScratchBytes) + "-byte buffer; use algdock_mbar";
      return ALGDOCK_E_INVALID;
    }
    cudaPointerAttributes attr;
    if (cudaPointerGetAttributes(&attr, u_kn) != cudaSuccess ||
        (attr.type != cudaMemoryTypeDevice && attr.type != cudaMemoryTypeManaged)) {
      cudaGetLastError();
      c->err = "mbar_noalloc: u_kn must be a device pointer";
      return ALGDOCK_E_INVALID;
    }
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != c->device) cudaSetDevice(c->device);
    void* scratch = nullptr;
    cudaError_t e = noalloc_scratch(c->device, &scratch);
    cudaError_t err = cudaSuccess;
    int it = 0;
    int r = -1;
    if (e == cudaSuccess) r = algdock::mbar_run(c->stream, scratch, K, N, u_kn, N_k, tol, max_iter, precision_mode, false,
                                                f_k, &it, c->h_flag, &err);
    else err = e;
    if (prev >= 0 && prev != c->device) cudaSetDevice(prev);
    *iters = it;
    if (r < 0) {
      c->err = std::string("mbar_noalloc: ") + cudaGetErrorString(err);
      return err == cudaErrorMemoryAllocation ? ALGDOCK_E_OOM : ALGDOCK_E_CUDA;
    }
    if (r == 1) {
      c->err = "mbar_noalloc: max_iter reached";
      return ALGDOCK_E_NOT_CONVERGED;
    }
    return ALGDOCK_OK;
  } catch (...) {
    try {
      c->err = "mbar_noalloc: host exception";
    } catch (...) {
    }
    return ALGDOCK_E_INVALID;
  }
}
