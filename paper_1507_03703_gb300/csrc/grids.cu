// Receptor grids: direct-sum construction and derivation of the interpolated lattices
// ("Thermodynamic Cycle": electrostatic and van der Waals grids, power-4 transform of the
// repulsive grid, soft tanh-capped grids).
#include <math.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "internal.cuh"

namespace algdock {
namespace {

constexpr int kBuildThreads = 128;
constexpr int kBuildTile = 128;      // receptor atom pairs staged per shared-memory tile
constexpr int kBuildNodes = 4;       // nodes per thread, spread along z
constexpr float kBuildMaxR2 = 8e37f;  // keeps the reciprocal normal and its refinement finite
// Nodes beyond kBuildFar of the origin, whose square FP32 does not hold, and atoms beyond three times that are
// taken to lie there: as far from all else, and hi + lo stays finite.
constexpr double kBuildFar = 2e19;

// s + e += a b: the rounded sum in s, its error (of the exact product) in e.
__device__ __forceinline__ void acc2(f32x2& s, f32x2& e, f32x2 a, f32x2 b) {
  const f32x2 t = fma2(a, b, s);
  e = add2(e, fma2(a, b, sub2(s, t)));
  s = t;
}
__device__ __forceinline__ double total2(f32x2 s, f32x2 e) {
  float sa, sb, ea, eb;
  unpack2(s, sa, sb);
  unpack2(e, ea, eb);
  const double v = (double)sa + (double)sb;
  return isfinite(v) ? v + ((double)ea + (double)eb) : v;  // an overflowed sum has no error term
}

// Direct sums, all in paired FP32 instructions (two receptor atoms each).  A thread takes four nodes
// of one column, so the x and y differences are shared, and `slices` groups of a block's threads share
// the receptor where the lattice alone would not fill the GPU.
//
// The differences are as exact as FP64 ones rounded to FP32: every coordinate (relative to the
// lattice origin) is hi + lo, with hi a multiple of a power of two such that every hi within 64 A of
// the lattice has at most 23 bits.  hi - hi is then exact, and one rounding remains, of the sum with
// lo - lo (an error of dx counts twelve times in r^-12).  LO: the nodes have a lo part; lattices of
// 0.25 or 0.5 A have none.  What dx lost in that rounding goes back into dx^2 (ex), and dz^2 comes last,
// as in the plain sum: shared by four nodes, this costs 3.5 % and keeps the error below that of FP32
// terms of FP64 differences (without it, it was up to 2 % above in the attractive grid).  The reciprocal
// takes one Newton step, and the floors of the attractive and electrostatic sums at 2 A are minima of the
// reciprocal powers.  The sums of thousands of terms (of mixed sign in the electrostatic grid) carry their
// rounding errors along (acc2): four instructions per channel, and exact products; only where a term
// exceeds the sum so far is part of the error lost.
//
// FP32-pipe bound: 22.5 paired instructions per two terms, of two cycles each, 4.8 ms for the 129^3
// lattice of a 4000-atom receptor.  Measured 7.36 ms, against 192 ms with FP64 differences and sums (6
// FP64 operations and 6 conversions a term on a pipe of 2 lanes per clock) and IEEE divisions.  Root mean
// square of the error against 64 bits, over 36 lattices and receptors, in units of 2^-24 of a node's sum of
// magnitudes, with those and here: repulsive 4.15, 3.87; attractive 0.960, 0.920; electrostatic 0.082, 0.076.
template <bool LO>
__global__ void __launch_bounds__(kBuildThreads) grid_build_kernel(
    int nx, int ny, int nz, int nq, int slices, double h, double quantum, int n_pairs,
    const ReceptorPair* __restrict__ rec, const float2* __restrict__ rec_q, float* ljr, float* lja, float* elec) {
  __shared__ ReceptorPair s_p[kBuildTile];
  __shared__ float2 s_q[kBuildTile];
  __shared__ double s_sum[kBuildThreads][3];
  const int width = kBuildThreads / slices;  // threads of a slice
  const int slice = threadIdx.x / width, tid = threadIdx.x % width;
  const int64_t item = (int64_t)blockIdx.x * width + tid;
  const int64_t n_items = (int64_t)nx * ny * nq;
  const bool active = item < n_items;
  // thread (i, j, q) of nx x ny x nq: nodes q, q + nq, q + 2 nq, q + 3 nq of column (i, j)
  const int i = (int)(item % nx), j = (int)((item / nx) % ny), q = (int)(item / ((int64_t)nx * ny));
  auto split = [&](int node, f32x2& hi, f32x2& lo) {
    const double p = fmin(h * node, kBuildFar);
    const float ph = (float)(rint(p / quantum) * quantum);
    const float pl = (float)(p - (double)ph);
    hi = pack2(ph, ph);
    lo = pack2(pl, pl);
  };
  f32x2 X, Xl, Y, Yl, Z[kBuildNodes], Zl[kBuildNodes];
  split(i, X, Xl);
  split(j, Y, Yl);
#pragma unroll
  for (int m = 0; m < kBuildNodes; ++m) split(q + m * nq, Z[m], Zl[m]);
  auto diff = [](f32x2 p, f32x2 pl, f32x2 a, f32x2 al) {
    return LO ? add2(sub2(p, a), sub2(pl, al)) : sub2(sub2(p, a), al);
  };
  auto diff_error = [](f32x2 d, f32x2 p, f32x2 pl, f32x2 a, f32x2 al) {  // exact less rounded difference
    return LO ? add2(sub2(sub2(p, a), d), sub2(pl, al)) : sub2(sub2(sub2(p, a), d), al);
  };
  const float rmin2 = (float)(kRepulsiveMinDist * kRepulsiveMinDist);
  const float amin2_inv = (float)(1.0 / (kAttractiveMinDist * kAttractiveMinDist));
  const float amin6_inv = amin2_inv * amin2_inv * amin2_inv;
  const f32x2 one = pack2(1.f, 1.f);
  constexpr f32x2 sign = 0x8000000080000000ull;
  f32x2 sr[kBuildNodes], er[kBuildNodes], sa[kBuildNodes], ea[kBuildNodes], se[kBuildNodes], ee[kBuildNodes];
#pragma unroll
  for (int m = 0; m < kBuildNodes; ++m) sr[m] = er[m] = sa[m] = ea[m] = se[m] = ee[m] = 0ull;
  for (int base = 0; base < n_pairs; base += kBuildTile) {
    const int n = min(kBuildTile, n_pairs - base);
    __syncthreads();
    for (int t = threadIdx.x; t < n; t += kBuildThreads) {
      s_p[t] = rec[base + t];
      s_q[t] = rec_q[base + t];
    }
    __syncthreads();
    const int end = active ? n * (slice + 1) / slices : 0;
    for (int t = n * slice / slices; t < end; ++t) {
      const ReceptorPair R = s_p[t];
      const float2 c = s_q[t];
      const f32x2 A = pack2(R.c3.x, R.c3.y), B = pack2(R.c3.z, R.c3.w), Q = pack2(c.x, c.y);
      const f32x2 hx = pack2(R.c0.x, R.c0.y), lx = pack2(R.c1.z, R.c1.w);
      const f32x2 dx = diff(X, Xl, hx, lx), ex = mul2(dx, diff_error(dx, X, Xl, hx, lx));
      const f32x2 dy = diff(Y, Yl, pack2(R.c0.z, R.c0.w), pack2(R.c2.x, R.c2.y));
      const f32x2 hz = pack2(R.c1.x, R.c1.y), lz = pack2(R.c2.z, R.c2.w);
      const f32x2 xy = fma2(dy, dy, fma2(dx, dx, add2(ex, ex)));
#pragma unroll
      for (int m = 0; m < kBuildNodes; ++m) {
        const f32x2 dz = diff(Z[m], Zl[m], hz, lz);
        float ra, rb;
        unpack2(fma2(dz, dz, xy), ra, rb);
        ra = fminf(fmaxf(ra, rmin2), kBuildMaxR2);
        rb = fminf(fmaxf(rb, rmin2), kBuildMaxR2);
        const f32x2 i0 = pack2(rcp_approx(ra), rcp_approx(rb));
        const f32x2 i2 = fma2(i0, fma2(pack2(ra, rb), i0 ^ sign, one), i0);
        const f32x2 i6 = mul2(mul2(i2, i2), i2);
        acc2(sr[m], er[m], A, mul2(i6, i6));
        float va, vb;
        unpack2(i6, va, vb);
        acc2(sa[m], ea[m], B, pack2(fminf(va, amin6_inv), fminf(vb, amin6_inv)));
        unpack2(i2, va, vb);
        acc2(se[m], ee[m], Q, pack2(fminf(va, amin2_inv), fminf(vb, amin2_inv)));  // 1/4 of eps(r) = 4r is in Q
      }
    }
  }
#pragma unroll
  for (int m = 0; m < kBuildNodes; ++m) {
    double r = total2(sr[m], er[m]), a = total2(sa[m], ea[m]), e = total2(se[m], ee[m]);
    if (slices > 1) {  // the slices' sums in order
      __syncthreads();
      s_sum[threadIdx.x][0] = r;
      s_sum[threadIdx.x][1] = a;
      s_sum[threadIdx.x][2] = e;
      __syncthreads();
      r = a = e = 0.0;
      for (int g = 0; g < slices; ++g) {
        r += s_sum[g * width + tid][0];
        a += s_sum[g * width + tid][1];
        e += s_sum[g * width + tid][2];
      }
    }
    const int k = q + m * nq;
    if (active && slice == 0 && k < nz) {
      const int64_t p = ((int64_t)k * ny + j) * nx + i;
      ljr[p] = (float)r;
      lja[p] = (float)(-a);
      elec[p] = (float)(kCoulomb * e);
    }
  }
}

// Derived lattices, computed in FP64 and rounded once to FP32.
// Node p's hard values go into its own x-pair record (first half) and into the record of its x - 1
// neighbour in the same row (second half); its soft values go into the (x, y) quad records of
// itself and of its x - 1, y - 1 and (x - 1, y - 1) neighbours in the same plane.  Halves that
// would hold a node past the last one of a row or column are zero (no cell starts there).
__global__ void grid_prepare_kernel(int64_t n, int nx, int ny, const float* __restrict__ ljr,
                                    const float* __restrict__ lja, const float* __restrict__ elec, double vmax_r,
                                    double vmax_e, float4* hard, float4* soft) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  double v = (double)ljr[p];
  if (!(v <= kRepulsiveNodeCap)) v = v > 0.0 ? kRepulsiveNodeCap : v;  // caps +inf as well
  if (!(v >= 0.0)) v = 0.0;
  const double e = (double)elec[p];
  const double root = pow(v, 0.25);
  const double soft_r = isinf(vmax_r) ? root : pow(vmax_r * tanh(v / vmax_r), 0.25);
  const double soft_e = isinf(vmax_e) ? e : vmax_e * tanh(e / vmax_e);
  const float4 h = make_float4((float)root, lja[p], elec[p], 0.f);
  const float2 sf = make_float2((float)soft_r, (float)soft_e);
  const int x = (int)(p % nx), y = (int)((p / nx) % ny);
  hard[2 * p] = h;
  if (x > 0) hard[2 * (p - 1) + 1] = h;
  if (x == nx - 1) hard[2 * p + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
  float2* q = (float2*)soft;  // 4 float2 per record: nodes (x, y), (x + 1, y), (x, y + 1), (x + 1, y + 1)
  const float2 zero = make_float2(0.f, 0.f);
  q[4 * p] = sf;
  if (x > 0) q[4 * (p - 1) + 1] = sf;
  if (y > 0) q[4 * (p - nx) + 2] = sf;
  if (x > 0 && y > 0) q[4 * (p - nx - 1) + 3] = sf;
  if (x == nx - 1) q[4 * p + 1] = q[4 * p + 3] = zero;
  if (y == ny - 1) q[4 * p + 2] = q[4 * p + 3] = zero;
}

// Peak rate of the interpolation's gathers, for the gather roofline (not a step of the method):
// each thread reads the 8 corners of cells drawn uniformly over the lattice (hard float4 corners,
// and with soft the float2 corners too, as one atom's interpolation does) and folds them into a
// sum that is stored only if it takes an impossible value, so that no load is dead.  Cells come
// from a per-thread xorshift stream mapped to [0, n - 1) by a multiply-shift (no division).
__device__ __forceinline__ uint32_t xorshift32(uint32_t& s) {
  s ^= s << 13;
  s ^= s >> 17;
  s ^= s << 5;
  return s;
}
__device__ __forceinline__ int below(uint32_t r, int n) { return (int)(((uint64_t)r * (uint32_t)n) >> 32); }

template <bool SOFT>
__global__ void __launch_bounds__(256) gather_probe_kernel(const float4* __restrict__ hard,
                                                           const float4* __restrict__ soft, int nx, int ny, int nz,
                                                           int64_t n_cells, uint32_t seed, float* sink) {
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  uint32_t st = (uint32_t)(tid * 2654435761u) ^ seed;
  st = st ? st : 0x9E3779B9u;
  const int64_t sy = nx, sz = (int64_t)nx * ny;
  float acc = 0.f;
  for (int64_t c = tid; c < n_cells; c += stride) {
    const int cx = below(xorshift32(st), nx - 1), cy = below(xorshift32(st), ny - 1),
              cz = below(xorshift32(st), nz - 1);
    const int64_t b = cz * sz + cy * sy + cx;
    // the cell's records, as the interpolation reads them: four 32-byte hard x-pair records and
    // (with SOFT) two 32-byte soft quad records
    float4 h0, h1, h2, h3, h4, h5, h6, h7;
    ldg_pair(hard + 2 * b, h0, h1);
    ldg_pair(hard + 2 * (b + sy), h2, h3);
    ldg_pair(hard + 2 * (b + sz), h4, h5);
    ldg_pair(hard + 2 * (b + sz + sy), h6, h7);
    acc += ((h0.x + h1.y) + (h2.z + h3.x)) + ((h4.y + h5.z) + (h6.x + h7.y));
    if (SOFT) {
      float4 s0, s1, s2, s3;
      ldg_pair(soft + 2 * b, s0, s1);
      ldg_pair(soft + 2 * (b + sz), s2, s3);
      acc += ((s0.x + s1.w) + (s2.x + s3.w)) + ((s0.z + s1.y) + (s2.z + s3.y));
    }
  }
  if (acc == -1.2345e-31f) sink[0] = acc;
}

}  // namespace

cudaError_t launch_grid_build(cudaStream_t s, const algdock_grid_desc& d, int n_rec, const double* xyz,
                              const double* rstar, const double* eps, const double* q, float* ljr, float* lja,
                              float* elec) {
  // Per-atom factors on the host (FP64), positions relative to the origin, then one upload.
  const int n_pairs = (n_rec + 1) / 2;
  const size_t np = (size_t)std::max(n_pairs, 1);
  std::vector<ReceptorPair> h_rec(np, ReceptorPair{});
  std::vector<float2> h_q(np, make_float2(0.f, 0.f));
  // the quantum of the hi parts: 2^-23 of the range the lattice and 64 A around it span
  const int n_max = std::max({d.n[0], d.n[1], d.n[2]});
  const double range = std::min(d.spacing * n_max + 64.0, kBuildFar);
  const double quantum = ldexp(1.0, std::ilogb(range) + 1 - 23);
  for (int j = 0; j < n_rec; ++j) {
    const double two_r = 2.0 * rstar[j];
    const double r6 = two_r * two_r * two_r * two_r * two_r * two_r;
    ReceptorPair& P = h_rec[j / 2];
    const bool odd = j & 1;
    float hi[3], lo[3];
    for (int a = 0; a < 3; ++a) {
      const double v = std::min(std::max(xyz[3 * (size_t)j + a] - d.origin[a], -3.0 * kBuildFar), 3.0 * kBuildFar);
      hi[a] = (float)(rint(v / quantum) * quantum);
      lo[a] = (float)(v - (double)hi[a]);
    }
    (odd ? P.c0.y : P.c0.x) = hi[0];
    (odd ? P.c0.w : P.c0.z) = hi[1];
    (odd ? P.c1.y : P.c1.x) = hi[2];
    (odd ? P.c1.w : P.c1.z) = lo[0];
    (odd ? P.c2.y : P.c2.x) = lo[1];
    (odd ? P.c2.w : P.c2.z) = lo[2];
    (odd ? P.c3.y : P.c3.x) = (float)(sqrt(eps[j]) * r6);
    (odd ? P.c3.w : P.c3.z) = (float)(sqrt(2.0 * eps[j]) * two_r * two_r * two_r);
    (odd ? h_q[j / 2].y : h_q[j / 2].x) = (float)(q[j] / 4.0);
  }
  bool lo = false;  // whether some node coordinate is no multiple of the quantum
  for (int i = 0; i < n_max && !lo; ++i) {
    const double p = std::min(d.spacing * i, kBuildFar);
    lo = !((double)(float)(rint(p / quantum) * quantum) == p);
  }
  void* d_rec = nullptr;
  const size_t bytes = np * (sizeof(ReceptorPair) + sizeof(float2));
  cudaError_t e = cudaMallocAsync(&d_rec, bytes, s);
  float2* d_q = (float2*)((ReceptorPair*)d_rec + np);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(d_rec, h_rec.data(), np * sizeof(ReceptorPair), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_q, h_q.data(), np * sizeof(float2), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // host staging buffers are freed below
  if (e == cudaSuccess) {
    const int nq = (d.n[2] + kBuildNodes - 1) / kBuildNodes;
    const int64_t items = (int64_t)d.n[0] * d.n[1] * nq;
    // four threads share a node's receptor where one each would leave fewer than eight blocks per SM
    const int slices = items >= (int64_t)152 * 8 * kBuildThreads ? 1 : 4;
    const int64_t blocks = (items * slices + kBuildThreads - 1) / kBuildThreads;
    auto k = lo ? grid_build_kernel<true> : grid_build_kernel<false>;
    k<<<(unsigned)blocks, kBuildThreads, 0, s>>>(d.n[0], d.n[1], d.n[2], nq, slices, d.spacing, quantum, n_pairs,
                                                 (const ReceptorPair*)d_rec, d_q, ljr, lja, elec);
    e = cudaGetLastError();
  }
  if (d_rec) cudaFreeAsync(d_rec, s);
  return e;
}

cudaError_t launch_grid_prepare(cudaStream_t s, size_t n_nodes, int nx, int ny, const float* ljr, const float* lja,
                                const float* elec, double vmax_r, double vmax_e, float4* hard, float4* soft) {
  const int threads = 256;
  const size_t blocks = (n_nodes + threads - 1) / threads;
  grid_prepare_kernel<<<(unsigned)blocks, threads, 0, s>>>((int64_t)n_nodes, nx, ny, ljr, lja, elec, vmax_r,
                                                            vmax_e, hard, soft);
  return cudaGetLastError();
}

}  // namespace algdock

namespace algdock {
cudaError_t launch_gather_probe(cudaStream_t s, const algdock_ctx& c, int64_t n_cells, bool soft, uint32_t seed,
                                float* sink) {
  const int threads = 256;
  const int blocks = 152 * 8;
  if (soft)
    gather_probe_kernel<true><<<blocks, threads, 0, s>>>(c.d_hard, c.d_soft, c.grid.nx, c.grid.ny, c.grid.nz, n_cells,
                                                          seed, sink);
  else
    gather_probe_kernel<false><<<blocks, threads, 0, s>>>(c.d_hard, c.d_soft, c.grid.nx, c.grid.ny, c.grid.nz,
                                                           n_cells, seed, sink);
  return cudaGetLastError();
}
}  // namespace algdock
