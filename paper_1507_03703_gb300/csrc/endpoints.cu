// End-point corrections of the thermodynamic cycle: the receptor-ligand interaction of the target
// force field, computed directly ("Thermodynamic Cycle": the target force field evaluates
// receptor-ligand interactions directly, the sampling force field by grid interpolation), and the
// Zwanzig free energy perturbation that carries milestone samples into the target force field
// ("Estimation": f_AB and f_DE by free energy perturbation).
#include <math.h>

#include "internal.cuh"

namespace algdock {
namespace {

constexpr int kTIMaxThreads = 256;                  // threads of a target-interaction block at most
constexpr int kRecPairTile = 128;                   // receptor atom pairs staged per shared-memory tile
constexpr int kFepThreads = 256;
constexpr int kFepMaxBlocks = 2 * 152;

// widen without its case for zero, which sums of terms hardly ever are: 1 % of the kernel's time.
__device__ __forceinline__ double widen_sum(float v) {
  const uint32_t b = __float_as_uint(v), m = b & 0x7fffffffu;
  if (m - 0x00800000u < 0x7f000000u)
    return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(b << 29));
  return (double)v;
}

// Each thread evaluates PER (configuration, atom) points against receptor atoms, two receptor atoms
// per paired instruction.  A block holds whole configurations (spb of them), so the
// per-configuration sums stay inside the block and are taken in a fixed order.  `groups` groups of
// T threads share the block's points: group g takes the receptor tiles g, g + groups, ...
// Receptor atoms j, j' = 2k, 2k + 1 (see ReceptorPair): x = x_hi + x_lo is the FP64
// coordinate, so that the difference (x_L - x_hi) - x_lo carries the rounding of the difference
// rather than of the coordinate.  Each term is FP32 (one approximate reciprocal; the floors of the
// attractive and electrostatic sums at 2 A are minima of the reciprocal powers, which equal the
// powers of max(r, 2)); a tile's terms are summed in FP32 and tiles in FP64.
// Bound: the FMA pipe, 15 lane-operations a pair term (2.7e12 terms/s); see kTIShapes for what the
// shape of the blocks gives.  At 16384 x 48 x 4000 1.84 -> 1.63 ms, 1.93e12 terms/s.
template <int PER>
__global__ void __launch_bounds__(kTIMaxThreads, 2) target_interaction_kernel(
    int64_t N, int na, int spb, int T, int groups, const float* __restrict__ x,
    const TargetFactors* __restrict__ lig_fac, const ReceptorPair* __restrict__ rec,
    const float2* __restrict__ rec_q, int n_pairs, double* __restrict__ psi) {
  extern __shared__ __align__(16) unsigned char ti_smem[];  // groups x (pairs, charges), then the energies
  const int g = threadIdx.x / T, tid = threadIdx.x - g * T;
  ReceptorPair* s_p = (ReceptorPair*)ti_smem + g * kRecPairTile;
  float2* s_q = (float2*)((ReceptorPair*)ti_smem + groups * kRecPairTile) + g * kRecPairTile;
  double* s_e = (double*)(ti_smem + groups * kRecPairTile * (sizeof(ReceptorPair) + sizeof(float2)));
  const int64_t s0 = (int64_t)blockIdx.x * spb;
  const int nsamp = (int)min((int64_t)spb, N - s0);
  const int npts = nsamp * na;
  const float* xb = x + 3 * (s0 * na);
  const float rmin2 = (float)(kRepulsiveMinDist * kRepulsiveMinDist);
  const float amin2_inv = (float)(1.0 / (kAttractiveMinDist * kAttractiveMinDist));
  const float amin6_inv = amin2_inv * amin2_inv * amin2_inv;
  f32x2 X[PER], Y[PER], Z[PER];
  double dr[PER], da[PER], de[PER];
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int p = tid + k * T;
    const bool v = p < npts;
    const float a = v ? xb[3 * p] : 0.f, b = v ? xb[3 * p + 1] : 0.f, c = v ? xb[3 * p + 2] : 0.f;
    X[k] = pack2(a, a);
    Y[k] = pack2(b, b);
    Z[k] = pack2(c, c);
    dr[k] = da[k] = de[k] = 0.0;
  }
  for (int round = 0; round < n_pairs; round += groups * kRecPairTile) {
    const int base = round + g * kRecPairTile;
    const int m = max(0, min(kRecPairTile, n_pairs - base));
    __syncthreads();
    for (int t = tid; t < m; t += T) {
      s_p[t] = rec[base + t];
      s_q[t] = rec_q[base + t];
    }
    __syncthreads();
    f32x2 fr[PER], fa[PER], fe[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) fr[k] = fa[k] = fe[k] = 0ull;
#pragma unroll 2
    for (int t = 0; t < m; ++t) {
      const ReceptorPair R = s_p[t];
      const float2 q = s_q[t];
      const f32x2 hx = pack2(R.c0.x, R.c0.y), hy = pack2(R.c0.z, R.c0.w), hz = pack2(R.c1.x, R.c1.y);
      const f32x2 lx = pack2(R.c1.z, R.c1.w), ly = pack2(R.c2.x, R.c2.y), lz = pack2(R.c2.z, R.c2.w);
      const f32x2 A = pack2(R.c3.x, R.c3.y), B = pack2(R.c3.z, R.c3.w), Q = pack2(q.x, q.y);
#pragma unroll
      for (int k = 0; k < PER; ++k) {
        const f32x2 dx = sub2(sub2(X[k], hx), lx), dy = sub2(sub2(Y[k], hy), ly), dz = sub2(sub2(Z[k], hz), lz);
        const f32x2 r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
        float ra, rb;
        unpack2(r2, ra, rb);
        const float ia = rcp_approx(fmaxf(ra, rmin2)), ib = rcp_approx(fmaxf(rb, rmin2));
        const f32x2 i2 = pack2(ia, ib);
        const f32x2 i6 = mul2(mul2(i2, i2), i2);
        fr[k] = fma2(A, mul2(i6, i6), fr[k]);
        float sa, sb;
        unpack2(i6, sa, sb);
        fa[k] = fma2(B, pack2(fminf(sa, amin6_inv), fminf(sb, amin6_inv)), fa[k]);
        fe[k] = fma2(Q, pack2(fminf(ia, amin2_inv), fminf(ib, amin2_inv)), fe[k]);
      }
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      float a, b;
      unpack2(fr[k], a, b);
      dr[k] += widen_sum(a) + widen_sum(b);
      unpack2(fa[k], a, b);
      da[k] += widen_sum(a) + widen_sum(b);
      unpack2(fe[k], a, b);
      de[k] += widen_sum(a) + widen_sum(b);
    }
  }
  // atom energy sqrt(A_i) LJr - sqrt(B_i) |LJa| + 332.0637 q_i elec, each group's share
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int p = tid + k * T;
    if (p < npts) {
      const TargetFactors f = lig_fac[p % na];
      s_e[g * PER * T + p] = f.sA * dr[k] - f.sB * da[k] + f.qC * de[k];
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < nsamp; k += groups * T) {  // up to 1024 configurations (one-atom ligands)
    double s = 0.0;
    for (int i = 0; i < na; ++i)
      for (int h = 0; h < groups; ++h) s += s_e[h * PER * T + k * na + i];
    psi[s0 + k] = s;
  }
}

// ------------------------------------------------------------------ FEP reduction
// Running log-sum-exp state of weights w = exp(-du): m = smallest du so far, s1 = sum exp(m - du),
// s2 = sum exp(2 (m - du)); m = +inf with s1 = s2 = 0 is the empty state.  du = +inf has weight 0;
// NaN and -inf are counted as invalid.
struct Lse {
  double m, s1, s2;
  int bad;
};

__device__ __forceinline__ void lse_add(Lse& a, double du) {
  if (isnan(du) || du == -INFINITY) {
    ++a.bad;
    return;
  }
  if (du == INFINITY) return;
  if (du < a.m) {
    const double r = a.s1 > 0.0 ? exp(du - a.m) : 0.0;
    a.s1 = a.s1 * r + 1.0;
    a.s2 = a.s2 * (r * r) + 1.0;
    a.m = du;
  } else {
    const double w = exp(a.m - du);
    a.s1 += w;
    a.s2 += w * w;
  }
}

__device__ __forceinline__ void lse_merge(Lse& a, const Lse& b) {
  a.bad += b.bad;
  if (!(b.s1 > 0.0)) return;
  if (!(a.s1 > 0.0)) {
    a.m = b.m;
    a.s1 = b.s1;
    a.s2 = b.s2;
    return;
  }
  const double m = fmin(a.m, b.m);
  const double ra = exp(m - a.m), rb = exp(m - b.m);
  a.s1 = a.s1 * ra + b.s1 * rb;
  a.s2 = a.s2 * (ra * ra) + b.s2 * (rb * rb);
  a.m = m;
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Block-wide merge: the exact minimum by integer comparisons, one factor exp(m - m_t) per thread,
// then sums in a fixed tree; the result is valid in thread 0.  GB300 issues 2 FP64 lanes per clock
// and SM, so the FP64 instructions count: a tree of pairwise merges takes two exponentials at each
// of its ten levels (44 us for 16384 samples with the launch of both kernels), this one in all.
__device__ Lse lse_block(Lse a) {
  constexpr int kWarps = kFepThreads / 32;
  __shared__ long long s_key[kWarps];
  __shared__ double s_1[kWarps], s_2[kWarps];
  __shared__ int s_bad[kWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  long long key = order_key(__double_as_longlong(a.m));
  for (int o = 16; o > 0; o >>= 1) key = min(key, __shfl_xor_sync(0xffffffffu, key, o));
  if (lane == 0) s_key[warp] = key;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kWarps; ++w) key = min(key, s_key[w]);
  const double m = __longlong_as_double(order_key(key));
  if (a.s1 > 0.0 && a.m > m) {
    const double r = exp(m - a.m);
    a.s1 *= r;
    a.s2 *= r * r;
  }
  a.s1 = warp_sum(a.s1);
  a.s2 = warp_sum(a.s2);
  a.bad = __reduce_add_sync(0xffffffffu, a.bad);
  if (lane == 0) {
    s_1[warp] = a.s1;
    s_2[warp] = a.s2;
    s_bad[warp] = a.bad;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a = Lse{m, s_1[0], s_2[0], s_bad[0]};
#pragma unroll
    for (int w = 1; w < kWarps; ++w) {
      a.s1 += s_1[w];
      a.s2 += s_2[w];
      a.bad += s_bad[w];
    }
  }
  return a;
}

// du_n = beta (u_t[n st] - u_s[n ss]) (u_s may be null: 0); each block merges a strided share.
__global__ void __launch_bounds__(kFepThreads) fep_partial_kernel(int64_t N, const double* __restrict__ ut, int64_t st,
                                                                  const double* __restrict__ us, int64_t ss,
                                                                  double beta, Lse* partial) {
  Lse a{INFINITY, 0.0, 0.0, 0};
  for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (int64_t)gridDim.x * blockDim.x) {
    const double d = ut[n * st] - (us ? us[n * ss] : 0.0);
    lse_add(a, beta * d);
  }
  a = lse_block(a);
  if (threadIdx.x == 0) partial[blockIdx.x] = a;
}

// out: f, sigma, n_eff, du_min, invalid count (as a double).
__global__ void __launch_bounds__(kFepThreads) fep_final_kernel(int64_t N, int n_part, const Lse* __restrict__ partial,
                                                                double* out) {
  Lse a{INFINITY, 0.0, 0.0, 0};
  for (int b = threadIdx.x; b < n_part; b += blockDim.x) lse_merge(a, partial[b]);
  a = lse_block(a);
  if (threadIdx.x == 0) {
    const double n = (double)N;
    if (a.s1 > 0.0) {
      const double n_eff = a.s1 * a.s1 / a.s2;
      out[0] = a.m - log(a.s1 / n);
      out[1] = N > 1 ? sqrt(fmax(n / n_eff - 1.0, 0.0) / (n - 1.0)) : NAN;
      out[2] = n_eff;
    } else {
      out[0] = INFINITY;
      out[1] = NAN;
      out[2] = 0.0;
    }
    out[3] = a.m;
    out[4] = (double)a.bad;
  }
}

struct TIShape {
  int per, threads, groups;
};

// The block shapes, and the rule that picks one: the least of max(pipe, chain) over the SM with most
// blocks.  Pipe: a receptor pair holds the FMA pipe of a warp's SM quarter for 30 cycles a point
// (15 paired instructions of two cycles) and 14 for the loop.  Chain: one warp alone takes 90 + 65
// a point, and about 16 warps overlap.  So large calls take four or three points a thread, whichever
// pads the blocks and the last SMs less, and small ones one point and several groups, down to a
// few warps per SM.  Microseconds at (configurations, atoms, receptor atoms), in the order 128
// threads of four points (the one shape before) -> 128 of three / two groups of 64 of three / four groups
// of 64 of three / two groups of 96 of one:
//   16384, 48, 4000   1858 -> 1683 / 1634 / 1762 / -    500, 10, 300     26 -> - / - / - / 12
//   10000, 70, 4000   1678 -> 1684 / - / - / -          1000, 20, 700    50 -> - / 26 / 25 / 23
//   3000, 33, 1200     122 -> 89 / 97 / - / -           2000, 13, 2500  163 -> - / 60 / 57 / 59
//   5000, 61, 300       76 -> 69 / - / - / -            500, 70, 4000   261 -> 172 / 155 / 155 / -
// Taken: two groups of 64 at the first and third, four points at the second, three points at the fourth; on
// the right two groups of 96, four groups of one point (not in the table), two groups of 96, four groups of 64.
// So the rule is up to 9 % from the best shape (97 for 89, 59 for 57).
constexpr TIShape kTIShapes[] = {{4, 128, 1}, {3, 128, 1}, {3, 64, 2}, {3, 64, 4}, {1, 96, 2}, {1, 64, 4}};

size_t ti_smem_bytes(const TIShape& h) {
  return (size_t)h.groups * (kRecPairTile * (sizeof(ReceptorPair) + sizeof(float2)) + h.per * h.threads * sizeof(double));
}

TIShape ti_shape(int64_t N, int na, int n_pairs) {
  TIShape best = kTIShapes[0];
  double least = INFINITY;
  for (const TIShape& h : kTIShapes) {
    const int spb = h.per * h.threads / na;
    if (spb < 1) continue;
    const int64_t per_sm = ((N + spb - 1) / spb + 151) / 152;
    const int rounds = (n_pairs + kRecPairTile * h.groups - 1) / (kRecPairTile * h.groups);
    const double pairs = min(n_pairs, rounds * kRecPairTile);
    const double warps = (double)per_sm * (h.threads / 32) * h.groups;
    const double pipe = warps / 4 * (30 * h.per + 14), chain = fmax(1.0, warps / 16) * (90 + 65 * h.per);
    const double t = pairs * fmax(pipe, chain);
    if (t < least) {
      least = t;
      best = h;
    }
  }
  return best;
}

template <int PER>
cudaError_t ti_launch(cudaStream_t s, const TIShape& h, int64_t N, int na, const float* x,
                      const TargetFactors* lig_fac, const ReceptorPair* rec, const float2* rec_q, int n_pairs,
                      double* psi) {
  const size_t smem = ti_smem_bytes(h);  // 43,008 bytes at most: no opt-in
  const int spb = h.per * h.threads / na;
  const int64_t blocks = (N + spb - 1) / spb;
  target_interaction_kernel<PER><<<(unsigned)blocks, h.threads * h.groups, smem, s>>>(
      N, na, spb, h.threads, h.groups, x, lig_fac, rec, rec_q, n_pairs, psi);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_target_interaction(cudaStream_t s, int64_t N, int na, const float* x, const TargetFactors* lig_fac,
                                      const ReceptorPair* rec, const float2* rec_q, int n_pairs, double* psi) {
  if (N <= 0) return cudaSuccess;
  const TIShape h = ti_shape(N, na, n_pairs);
  switch (h.per) {
    case 1: return ti_launch<1>(s, h, N, na, x, lig_fac, rec, rec_q, n_pairs, psi);
    case 3: return ti_launch<3>(s, h, N, na, x, lig_fac, rec, rec_q, n_pairs, psi);
    default: return ti_launch<4>(s, h, N, na, x, lig_fac, rec, rec_q, n_pairs, psi);
  }
}

size_t fep_scratch_bytes() { return sizeof(Lse) * kFepMaxBlocks + 8 * sizeof(double); }

cudaError_t launch_fep(cudaStream_t s, int64_t N, const double* ut, int64_t st, const double* us, int64_t ss,
                       double beta, void* scratch, double* out_dev) {
  Lse* part = (Lse*)scratch;
  const int64_t want = (N + kFepThreads - 1) / kFepThreads;  // one sample per thread up to 304 blocks
  const int blocks = (int)max((int64_t)1, min(want, (int64_t)kFepMaxBlocks));
  fep_partial_kernel<<<blocks, kFepThreads, 0, s>>>(N, ut, st, us, ss, beta, part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  fep_final_kernel<<<1, kFepThreads, 0, s>>>(N, blocks, part, out_dev);
  return cudaGetLastError();
}

}  // namespace algdock
