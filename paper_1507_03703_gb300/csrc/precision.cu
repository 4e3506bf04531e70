// The all-FP64 evaluation path: the energy components and forces of stored configurations with
// every operation in FP64, on FP64 lattices and FP64 parameters.  It is the FP64 arm of the
// precision study of the FP32 path (grid interaction, "Thermodynamic Cycle"; the ligand force
// field; the restraint, Eq. (binding_site); the state weights, Eq. (protocol)).
//
// GB300 issues 2 FP64 lanes per clock and SM (a warp instruction takes a scheduler 64 cycles), so
// the kernel is bound by the number of FP64 warp instructions and by nothing else.  One warp per
// configuration, with every stage laid out so that the lanes are full and each term is computed
// once:
//   1. bonded terms, one per lane, their forces to slots that are then added over the balanced
//      runs of the FP32 kernel's gather schedule;
//   2. nonbonded pairs, each unordered pair once: pair index p is (i, i + d mod n) with d = 1 + p/n,
//      i = p mod n, so 32 consecutive pairs have 32 different i and 32 different j, and the forces
//      on both are added in shared memory without conflict (a ligand of fewer than 32 atoms takes
//      one d at a time);
//   3. per atom: the five interpolated channels, edge differences along x, then y, then z.
// Reciprocal square roots take the place of square roots and divisions (the pair loop's from an
// FP32 seed by one third-order step), torsions the multiple-angle polynomials of cos(phi), sin(phi).  Where a
// rounding would count many times (a bond's length, R^2/r^2) one more step takes it out: the forces of bonds
// and of pairs are as close to extended precision as with square roots and divisions (1.5e-15 and 6.5e-16
// relative), their energies closer.
// 8192 configurations of 48 atoms take 1.23 ms.  With one thread per
// configuration (64 blocks, square roots, divisions, atan2, sincos, and forces added in global
// memory) they took 5.67 ms.  Two configurations per block or four make no difference at that size;
// two leave more blocks to a small one.
#include <math.h>

#include "internal.cuh"

namespace algdock {
namespace {

constexpr int kWarps64 = 2;  // configurations per block, fewer where their shared memory does not fit
constexpr size_t kMaxSmem64 = 227 * 1024;
constexpr unsigned kFull = 0xffffffffu;

struct V3 {
  double x, y, z;
};
__device__ inline V3 operator-(V3 a, V3 b) { return V3{a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ inline V3 operator+(V3 a, V3 b) { return V3{a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ inline V3 operator*(double s, V3 a) { return V3{s * a.x, s * a.y, s * a.z}; }
__device__ inline double dot3(V3 a, V3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ inline V3 cross3(V3 a, V3 b) { return V3{a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x}; }

__device__ inline double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// 1 / sqrt(v) and 1 / v from an FP32 seed y (error e = 1 - v y^2 about 2^-22, y^2 exact): y (1 + e/2 + 3 e^2/8)
// and y^2 (1 + e + e^2), whose errors 5 e^3/16 and e^3 are below FP64 rounding.  (The square of the root
// would carry its rounding twice, and r^-12 that twelve times.)
__device__ inline void reciprocals(double v, double& inv_root, double& inv) {
  const double y = (double)rsqrtf((float)v), y2 = y * y;
  const double e = fma(-v, y2, 1.0);
  inv_root = fma(y * e, fma(0.375, e, 0.5), y);
  inv = fma(y2, fma(e, e, e), y2);
}

// sqrt(v) from y = 1 / sqrt(v) by a Newton step: within 0.51 ulp, where v y is within 1.5 (a bond's stretch is a
// few hundredths of its length).  Zero and infinity are their own roots.
__device__ inline double sqrt_step(double v, double y) {
  const double r = v * y;
  return v > 0.0 && y > 0.0 ? fma(0.5 * y, fma(-r, r, v), r) : v;
}

// (c, s) / |(c, s)| where the sum of squares is zero, overflows or is not a number: (1, 0) for (0, 0), and the
// limit of the direction where a part is infinite, as the angle atan2(s, c) has it.
__device__ __noinline__ void direction(double& c, double& s) {
  double m = fmax(fabs(c), fabs(s));
  if (isinf(m)) {
    c = isinf(c) ? copysign(1.0, c) : 0.0 * c;
    s = isinf(s) ? copysign(1.0, s) : 0.0 * s;
    m = 1.0;
  }
  if (m > 0.0) {
    c /= m;
    s /= m;
    m = rsqrt(c * c + s * s);
    c *= m;
    s *= m;
  } else if (c == 0.0) {
    c = 1.0;
  }
}

// A warp's shared memory: positions [3][na], forces [3][na], bonded slots [3][n_slots + 1] (the last
// one zero).  A topology with more slots than fit (9000 and more; s null) adds its bonded forces
// by shared-memory atomics instead.
struct Warp64 {
  double *x, *f, *s;
  int na, ns;
  __device__ V3 pos(int i) const { return V3{x[i], x[na + i], x[2 * na + i]}; }
  __device__ V3 slot(int i) const { return V3{s[i], s[ns + i], s[2 * ns + i]}; }
  __device__ void put(int i, V3 v) const {
    s[i] = v.x;
    s[ns + i] = v.y;
    s[2 * ns + i] = v.z;
  }
  // the force of a bonded term's slot i on an atom
  __device__ void put(int i, int atom, V3 v) const {
    if (s) {
      put(i, v);
    } else {
      atomicAdd(f + atom, v.x);
      atomicAdd(f + na + atom, v.y);
      atomicAdd(f + 2 * na + atom, v.z);
    }
  }
};
__host__ __device__ inline int warp64_doubles(int na, int n_slots, bool slots) {
  return 6 * na + (slots ? 3 * (n_slots + 1) : 0);
}

// Trilinear value and gradient of lattice channel ch at p; coordinates outside the lattice are
// clamped to it, and the gradient along a clamped axis is zero.
struct Interp {
  int64_t b;
  double t[3];
  bool in[3];
};
__device__ inline Interp locate(const GridDev64& G, V3 p) {
  Interp I;
  const double o[3] = {G.ox, G.oy, G.oz}, q[3] = {p.x, p.y, p.z};
  const int n[3] = {G.nx, G.ny, G.nz};
  int c[3];
  for (int d = 0; d < 3; ++d) {
    double u = (q[d] - o[d]) / G.h;
    I.in[d] = true;
    if (!(u >= 0.0)) {
      u = 0.0;
      I.in[d] = false;
    }
    if (u > (double)(n[d] - 1)) {
      u = (double)(n[d] - 1);
      I.in[d] = false;
    }
    int ci = (int)floor(u);
    if (ci > n[d] - 2) ci = n[d] - 2;
    c[d] = ci;
    I.t[d] = u - ci;
  }
  I.b = ((int64_t)c[2] * G.ny + c[1]) * G.nx + c[0];
  return I;
}

// a (1 - t) + b t with both products, so that a large corner value far away in t leaves no error of
// its own size.
__device__ inline double lerp64(double a, double b, double t) { return fma(t, b, fma(-t, a, a)); }

// Value and gradient in lattice units from the corner values c[z][y][x].
__device__ inline double trilinear(const double (&c)[8], const double (&t)[3], V3& g) {
  const double d0 = c[1] - c[0], d1 = c[3] - c[2], d2 = c[5] - c[4], d3 = c[7] - c[6];
  const double a0 = lerp64(c[0], c[1], t[0]), a1 = lerp64(c[2], c[3], t[0]);
  const double a2 = lerp64(c[4], c[5], t[0]), a3 = lerp64(c[6], c[7], t[0]);
  const double y0 = a1 - a0, y1 = a3 - a2;
  const double b0 = lerp64(a0, a1, t[1]), b1 = lerp64(a2, a3, t[1]);
  const double x0 = fma(t[1], d1 - d0, d0), x1 = fma(t[1], d3 - d2, d2);
  g.z = b1 - b0;
  g.x = fma(t[2], x1 - x0, x0);
  g.y = fma(t[2], y1 - y0, y0);
  return lerp64(b0, b1, t[2]);
}

struct Eval64Args {
  int64_t N;
  Lig64 L;
  const double* P;        // the ligand's FP64 tables
  LigandLayout LL;        // of the FP32 blob, for its gather schedule
  const uint32_t* blob;
  GridDev64 G;
  const StateDev* states;
  int n_states;
  const int32_t* state_of;
  const float* x;
  double* force;
  double* comps;
  bool slots;             // the bonded slots are in shared memory
};

template <bool FORCES>
__global__ void __launch_bounds__(kWarps64 * 32) eval64_kernel(const Eval64Args A) {
  extern __shared__ double smem64[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t n = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
  if (n >= A.N) return;
  const Lig64& L = A.L;
  const int na = L.na, nb = L.nb, nang = L.nang, ntor = L.ntor, n_slots = A.LL.n_slots;
  Warp64 W;
  W.x = smem64 + (size_t)warp * warp64_doubles(na, n_slots, A.slots);
  W.f = W.x + 3 * na;
  W.s = A.slots ? W.f + 3 * na : nullptr;
  W.na = na;
  W.ns = n_slots + 1;
  double w_sg = 0.0, w_g = 0.0;
  if (A.state_of) {
    const int k = A.state_of[n];
    if ((unsigned)k < (unsigned)A.n_states) {
      w_sg = A.states[k].w_sg;
      w_g = A.states[k].w_g;
    }
  }
  const float* xin = A.x + n * na * 3;
  for (int i = lane; i < na; i += 32)
    for (int d = 0; d < 3; ++d) {
      W.x[d * na + i] = (double)xin[3 * i + d];
      if (FORCES) W.f[d * na + i] = 0.0;
    }
  if (FORCES && A.slots && lane == 0) W.put(n_slots, V3{0.0, 0.0, 0.0});
  __syncwarp();
  double e_lig = 0.0;
  // bonds: k (r - r0)^2
  for (int t = lane; t < nb; t += 32) {
    const double* b = A.P + L.off_bond + 4 * t;
    const int i = (int)b[0], j = (int)b[1];
    const V3 d = W.pos(i) - W.pos(j);
    const double r2 = dot3(d, d), inv_r = rsqrt(r2);
    const double dr = sqrt_step(r2, inv_r) - b[3];
    e_lig += b[2] * dr * dr;
    if (FORCES) {
      const V3 f = (-2.0 * b[2] * dr * inv_r) * d;
      W.put(t, i, f);
      W.put(nb + t, j, V3{-f.x, -f.y, -f.z});
    }
  }
  // angles: k (theta - theta0)^2, theta at the middle atom
  const int ab = 2 * nb;
  for (int t = lane; t < nang; t += 32) {
    const double* a = A.P + L.off_ang + 5 * t;
    const int i = (int)a[0], j = (int)a[1], k = (int)a[2];
    const V3 c0 = W.pos(j), u = W.pos(i) - c0, w = W.pos(k) - c0;
    const double lu2 = dot3(u, u), lw2 = dot3(w, w), inv_luw = rsqrt(lu2 * lw2);
    const double c = fmin(1.0, fmax(-1.0, dot3(u, w) * inv_luw));
    const double dth = acos(c) - a[4];
    e_lig += a[3] * dth * dth;
    if (FORCES) {
      // d theta / d u = -(w / luw - c u / lu2) / sin(theta), 1 / lu2 = lw2 / luw^2
      const double coef = 2.0 * a[3] * dth * rsqrt(fmax(1.0 - c * c, 1e-30));
      const double cx = coef * inv_luw, cc = cx * inv_luw * c;
      const V3 fi = cx * w - (cc * lw2) * u, fk = cx * u - (cc * lu2) * w;
      W.put(ab + t, i, fi);
      W.put(ab + nang + t, j, V3{-(fi.x + fk.x), -(fi.y + fk.y), -(fi.z + fk.z)});
      W.put(ab + 2 * nang + t, k, fk);
    }
  }
  // torsions: sum_n V_n/2 (1 + cos(n phi - gamma_n))
  const int tb = ab + 3 * nang;
  for (int t = lane; t < ntor; t += 32) {
    const double* q = A.P + L.off_tor + kTor64 * t;
    const int i = (int)q[0], j = (int)q[1], k = (int)q[2], l = (int)q[3];
    const V3 pj = W.pos(j), pk = W.pos(k);
    const V3 b1 = pj - W.pos(i), b2 = pk - pj, b3 = W.pos(l) - pk;
    const V3 n1 = cross3(b1, b2), n2 = cross3(b2, b3);
    const double lb22 = dot3(b2, b2), inv_lb2 = rsqrt(lb22), lb2 = sqrt_step(lb22, inv_lb2);
    // (cos phi, sin phi) is (n1.n2, |b2| b1.n2) normalised; collinear bonds have phi = 0
    const double cx = dot3(n1, n2), sx = lb2 * dot3(b1, n2);
    const double h2 = cx * cx + sx * sx, inv_h = rsqrt(h2);
    double c1 = cx * inv_h, s1 = sx * inv_h;
    if (!(h2 > 0.0 && inv_h > 0.0)) {
      c1 = cx;
      s1 = sx;
      direction(c1, s1);
    }
    const double c2 = 2.0 * c1 * c1 - 1.0, s2 = 2.0 * s1 * c1;
    const double c3 = c1 * (2.0 * c2 - 1.0), s3 = s1 * (2.0 * c2 + 1.0);
    const double *V = q + 4, *cg = q + 7, *sg = q + 10;
    e_lig += V[0] * (1.0 + c1 * cg[0] + s1 * sg[0]) + V[1] * (1.0 + c2 * cg[1] + s2 * sg[1]) +
             V[2] * (1.0 + c3 * cg[2] + s3 * sg[2]);
    if (FORCES) {
      const double dE = V[0] * (c1 * sg[0] - s1 * cg[0]) + 2.0 * V[1] * (c2 * sg[1] - s2 * cg[1]) +
                        3.0 * V[2] * (c3 * sg[2] - s3 * cg[2]);
      // forces: F_i = (dE lb2 / |n1|^2) n1, F_l = -(dE lb2 / |n2|^2) n2, and the middle atoms keep
      // the total force and torque zero
      const double i1 = rsqrt(fmax(dot3(n1, n1), 1e-60)), i2 = rsqrt(fmax(dot3(n2, n2), 1e-60));
      const double el = dE * lb2, inv_lb22 = inv_lb2 * inv_lb2;
      const V3 fi = (el * i1 * i1) * n1, fl = (-el * i2 * i2) * n2;
      const double p = dot3(b1, b2) * inv_lb22, r = dot3(b3, b2) * inv_lb22;
      W.put(tb + t, i, fi);
      W.put(tb + ntor + t, j, (-(1.0 + p)) * fi + r * fl);
      W.put(tb + 2 * ntor + t, k, p * fi + (-(1.0 + r)) * fl);
      W.put(tb + 3 * ntor + t, l, fl);
    }
  }
  __syncwarp();
  if (FORCES && A.slots) {
    // the slots of every atom over the lanes' balanced runs; each run's partial sums stay in place
    const uint2* gs = (const uint2*)(A.blob + A.LL.off_gs) + lane;
    V3 a{0.0, 0.0, 0.0};
    for (int j = 0; j < A.LL.gs_iters; ++j) {
      const uint2 w = __ldg(gs + 32 * j);
      const uint32_t e[4] = {w.x & 0xffffu, w.x >> 16, w.y & 0xffffu, w.y >> 16};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        a = a + W.slot(e[k] & 0x7fffu);
        if (e[k] & 0x8000u) {
          W.put(e[k] & 0x7fffu, a);
          a = V3{0.0, 0.0, 0.0};
        }
      }
    }
    __syncwarp();
  }
  // nonbonded pairs beyond 1-3 (excluded ones have R^2 < 0 and zero coefficients)
  {
    const int width = min(na, 32), n_pairs = na * (na - 1) / 2;
    const double* T = A.P + L.off_pair;
    double e12 = 0.0, e_el = 0.0;
    for (int p0 = 0; p0 < n_pairs; p0 += width) {
      const int p = p0 + lane;
      const bool on = lane < width && p < n_pairs;
      int i = 0, j = 0;
      V3 dx{0.0, 0.0, 0.0};
      double fr = 0.0;  // -dE/dr / r
      bool pair = false;
      if (on) {
        const int d = p / na;
        i = p - d * na;
        j = i + d + 1;
        j = j >= na ? j - na : j;
        const double R2 = __ldg(T + p), eps12 = __ldg(T + n_pairs + p), qq = __ldg(T + 2 * n_pairs + p);
        dx = W.pos(i) - W.pos(j);
        double r2 = dot3(dx, dx), y, y2;
        pair = __double2hiint(R2) >= 0;
        const bool none = !pair || __double2hiint(r2) == 0x7ff00000;  // excluded, or infinitely far apart
        r2 = none ? 1.0 : r2;
        reciprocals(r2, y, y2);
        if (none) y = y2 = 0.0;
        // R^2 / r^2 rounded once, by the remainder of the product with the rounded reciprocal
        double s2 = R2 * y2;
        s2 = fma(fma(-s2, r2, R2), y2, s2);
        const double s6 = s2 * s2 * s2, A12 = eps12 * s6, eel = qq * y;
        e12 = fma(A12, s6 - 2.0, e12);
        e_el += eel;
        if (FORCES) fr = fma(A12, s6 - 1.0, eel) * y2;
      }
      if (FORCES) {
        if (pair) {
          W.f[i] = fma(fr, dx.x, W.f[i]);
          W.f[na + i] = fma(fr, dx.y, W.f[na + i]);
          W.f[2 * na + i] = fma(fr, dx.z, W.f[2 * na + i]);
        }
        __syncwarp();
        if (pair) {
          W.f[j] = fma(-fr, dx.x, W.f[j]);
          W.f[na + j] = fma(-fr, dx.y, W.f[na + j]);
          W.f[2 * na + j] = fma(-fr, dx.z, W.f[2 * na + j]);
        }
        __syncwarp();
      }
    }
    e_lig += e12 * (1.0 / 12.0) + e_el;
  }
  // restraint on the centre of mass
  const double* atom = A.P + L.off_atom;
  V3 com{0.0, 0.0, 0.0};
  for (int i = lane; i < na; i += 32) com = com + __ldg(atom + 6 * i) * W.pos(i);
  com = V3{warp_sum(com.x), warp_sum(com.y), warp_sum(com.z)};
  const double inv_M = 1.0 / L.total_mass;
  const V3 dc = inv_M * com - V3{L.site[0], L.site[1], L.site[2]};
  const double d = sqrt(dot3(dc, dc));
  double e_rest = 0.0, c_rest = 0.0;
  if (d > L.d0) {
    const double ex = d - L.d0;
    e_rest = 0.5 * L.k_rest * ex * ex;
    c_rest = -L.k_rest * ex / d * inv_M;
  } else if (!(d <= L.d0)) {
    e_rest = d;  // NaN centre of mass
  }
  // grid terms: hard Psi_g = sA r^4 + sB a + q e, soft Psi_sg = sA sr^4 + q se
  double psi_g = 0.0, psi_sg = 0.0;
  const double inv_h = 1.0 / A.G.h;
  const int64_t sy = A.G.nx, sz = (int64_t)A.G.nx * A.G.ny;
  for (int i = lane; i < na; i += 32) {
    const double* ai = atom + 6 * i;
    const double m = __ldg(ai), q = __ldg(ai + 1), sA = __ldg(ai + 2), sB = __ldg(ai + 3);
    const Interp I = locate(A.G, W.pos(i));
    double c[3][8], r, v;
    V3 g, dg, dsg;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const double2* h = (const double2*)(A.G.hard + I.b + (k >> 2) * sz + ((k >> 1) & 1) * sy + (k & 1));
      const double2 ra = __ldg(h), e0 = __ldg(h + 1);
      c[0][k] = ra.x;
      c[1][k] = ra.y;
      c[2][k] = e0.x;
    }
    r = trilinear(c[0], I.t, g);
    dg = (4.0 * sA * r * r * r) * g;
    v = sA * (r * r) * (r * r);
    v += sB * trilinear(c[1], I.t, g);
    dg = dg + sB * g;
    v += q * trilinear(c[2], I.t, g);
    dg = dg + q * g;
    psi_g += v;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const double2 s = __ldg((const double2*)(A.G.soft + I.b + (k >> 2) * sz + ((k >> 1) & 1) * sy + (k & 1)));
      c[0][k] = s.x;
      c[1][k] = s.y;
    }
    r = trilinear(c[0], I.t, g);
    dsg = (4.0 * sA * r * r * r) * g;
    v = sA * (r * r) * (r * r);
    v += q * trilinear(c[1], I.t, g);
    dsg = dsg + q * g;
    psi_sg += v;
    if (FORCES) {
      const V3 f = (-w_g) * dg + (-w_sg) * dsg;
      V3 s = V3{W.f[i], W.f[na + i], W.f[2 * na + i]};
      if (c_rest != 0.0) s = s + (c_rest * m) * dc;
      if (A.slots) {
        const uint2 p = __ldg((const uint2*)(A.blob + A.LL.off_gp) + i);
        s = s + (W.slot(p.x & 0xffffu) + W.slot(p.x >> 16) + W.slot(p.y & 0xffffu) + W.slot(p.y >> 16));
      }
      double* out = A.force + (n * na + i) * 3;
      out[0] = s.x + (I.in[0] ? inv_h * f.x : 0.0);
      out[1] = s.y + (I.in[1] ? inv_h * f.y : 0.0);
      out[2] = s.z + (I.in[2] ? inv_h * f.z : 0.0);
    }
  }
  e_lig = warp_sum(e_lig);
  psi_sg = warp_sum(psi_sg);
  psi_g = warp_sum(psi_g);
  if (lane < 4) A.comps[4 * n + lane] = lane == 0 ? e_lig : (lane == 1 ? e_rest : (lane == 2 ? psi_sg : psi_g));
}

__global__ void grid_prepare64_kernel(int64_t n, const double* __restrict__ ljr, const double* __restrict__ lja,
                                      const double* __restrict__ elec, double vmax_r, double vmax_e, Hard64* hard,
                                      Soft64* soft) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  double v = ljr[p];
  if (!(v <= kRepulsiveNodeCap)) v = v > 0.0 ? kRepulsiveNodeCap : v;  // caps +inf as well
  if (!(v >= 0.0)) v = 0.0;
  const double e = elec[p];
  hard[p] = Hard64{pow(v, 0.25), lja[p], e, 0.0};
  soft[p] = Soft64{isinf(vmax_r) ? pow(v, 0.25) : pow(vmax_r * tanh(v / vmax_r), 0.25),
                   isinf(vmax_e) ? e : vmax_e * tanh(e / vmax_e)};
}

}  // namespace

cudaError_t launch_grid_prepare64(cudaStream_t s, size_t n_nodes, const double* ljr, const double* lja,
                                  const double* elec, double vmax_r, double vmax_e, Hard64* hard, Soft64* soft) {
  const int threads = 256;
  grid_prepare64_kernel<<<(unsigned)((n_nodes + threads - 1) / threads), threads, 0, s>>>(
      (int64_t)n_nodes, ljr, lja, elec, vmax_r, vmax_e, hard, soft);
  return cudaGetLastError();
}

cudaError_t launch_eval64(cudaStream_t s, const algdock_ctx& c, int64_t N, const int32_t* state_of, const float* x,
                          double* force, double* comps) {
  if (N == 0) return cudaSuccess;
  const int na = c.lig.na, ns = c.lig.n_slots;
  const bool slots = force && sizeof(double) * warp64_doubles(na, ns, true) <= kMaxSmem64;
  const size_t per = sizeof(double) * warp64_doubles(na, ns, slots);
  int warps = kWarps64;
  while (warps * per > kMaxSmem64) warps /= 2;
  const size_t smem = warps * per;
  const Eval64Args A{N, c.lig64, c.d_lig64, c.lig, c.d_blob, c.grid64, c.d_states, c.K, state_of, x, force, comps,
                     slots};
  auto k = force ? eval64_kernel<true> : eval64_kernel<false>;
  // the limit itself, whatever the ligand: another thread's call may set it between this and the launch
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem64);
  if (e != cudaSuccess) return e;
  k<<<(unsigned)((N + warps - 1) / warps), warps * 32, smem, s>>>(A);
  return cudaGetLastError();
}

}  // namespace algdock
