// The fused HMC trial ("Sampling"): momentum draw, n_steps of velocity Verlet over the grid
// interaction energy ("Thermodynamic Cycle"), the ligand force field and the flat-bottom
// restraint (Eq. (binding_site)), then the Metropolis test on the total energy change.
//
// Layout: a team of warps per replica, one atom per lane (warp w of the team holds atoms 32w ..
// 32w+31; up to three warps).  Position, velocity and force of the atom stay in registers for the whole
// trajectory; the current positions are mirrored in the replica's shared-memory arrays so that
// every lane can read every atom.  The ligand's parameters and topology are staged once per CTA in
// shared memory.
//
// One force evaluation:
//   1. bonded terms, one term per lane of the team: each term's forces on its 2-4 atoms go to the
//      replica's shared-memory slots (role-major, so consecutive lanes write consecutive words);
//   2. the slots summed over balanced runs by one warp, while each warp does
//   3. the 8-corner gathers of the grid lattices for its atoms and
//   4. the nonbonded pairs of its atoms with every other atom (the pair type table marks excluded
//      and 1-4 pairs); when the last warp has at most 16 atoms, two lanes share an atom and split
//      the partner range;
//   5. the restraint on the warp-reduced centre of mass, and each atom's sum of all of these.
//
// The same sums in the same order as one warp holding all atoms (two or three per lane), which was
// the layout before: 128 registers and 16 warps per SM there, where a warp's idle lanes in the second
// and third pass, its long chain of stages and 38 instructions a pair without the pair table set the
// pace.  Teams keep 24 warps per SM in two blocks, run stages 2 to 4 beside each other and spread a
// few replicas over all SMs.  Measured (trials of 50 steps, bit-identical): 48 atoms, 8192 replicas
// 1852 -> 1596 us; 83 atoms, 1152 replicas 1100 -> 674 us; 60 atoms (no pair table), 4096 replicas
// 1924 -> 1334 us; 27 atoms, 8192 replicas 1025 -> 826 us; 16 replicas of 20 atoms, 20 steps, 96 -> 62 us.
// Every force is accumulated by one lane in a fixed order (no atomics), so results are
// deterministic.
#include <math.h>

#include <algorithm>

#include "internal.cuh"

namespace algdock {
namespace {

constexpr int kWarpsPerBlock = 4;
constexpr unsigned kFull = 0xffffffffu;

struct Lig {
  const float4* atom_a;  // (accel factor 4.184e-4/m, q, sqrt(A), sqrt(B))
  const float4* atom_b;  // (R*, sqrt(eps), m, sqrt(accel factor))
  const uint8_t* ptype;  // [j][i]: 0 nonbonded, 1 1-4, 2 excluded (and i == j)
  const float4* bond;
  const int4* ang_i;
  const float4* ang_p;
  const int4* tor_i;
  const float4* tor_v;
  const float4* tor_c;
  const float4* tor_s;
  const uint2* gs;  // gather schedule: [gs_iters][32] words of four 16-bit entries
  const uint2* gp;  // [na]: four 16-bit partial-sum slots per atom
  const float4* pair;   // [p][i]: records of atom i with partners 2p, 2p + 1 (only where the table is staged)
  // the HMC kernel without that table (stage_types): per partner pair (R*, R*', sqrt(eps), sqrt(eps)'),
  // the scales (LJ, LJ', Coulomb, Coulomb') of each combination of two pair types, and [p][i] the byte
  // offset of the pair's combination
  const float4* ppar;
  const float4* scale;
  const uint8_t* combo;
};

__device__ inline Lig bind_ligand(const uint32_t* s, const LigandLayout& L) {
  Lig g;
  g.atom_a = (const float4*)(s + L.off_atom_a);
  g.atom_b = (const float4*)(s + L.off_atom_b);
  g.ptype = (const uint8_t*)(s + L.off_ptype);
  g.bond = (const float4*)(s + L.off_bond);
  g.ang_i = (const int4*)(s + L.off_ang);
  g.ang_p = (const float4*)(s + L.off_ang + 4 * L.nang);
  g.tor_i = (const int4*)(s + L.off_tor);
  g.tor_v = (const float4*)(s + L.off_tor + 4 * L.ntor);
  g.tor_c = (const float4*)(s + L.off_tor + 8 * L.ntor);
  g.tor_s = (const float4*)(s + L.off_tor + 12 * L.ntor);
  g.gs = (const uint2*)(s + L.off_gs);
  g.gp = (const uint2*)(s + L.off_gp);
  g.pair = (const float4*)(s + L.off_pair);
  return g;
}

// The hardware's approximate reciprocal square root and quotient.  rsqrtf and __fdividef are the same
// instructions wrapped in a scaling of denormal arguments (three more instructions each, a tenth of
// the kernel's), which these take for zero.  Their arguments are squared distances, denormal only below
// 1.1e-19 A, and values with a floor; otherwise the results are the same bits.  Not so the product of a
// torsion's two squared normals, each with a floor: that is 1e-40 where all four atoms lie on a line.
__device__ __forceinline__ float rsqrt_fast(float v) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ float div_fast(float a, float b) {
  float r;
  asm("div.approx.ftz.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

__device__ inline double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}
__device__ inline float warp_sumf(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// Lattice coordinate of x along one axis.  x - o is formed exactly as s + e (two-sum), so the
// fractional offset keeps FP32 precision relative to the cell even far from the origin.
__device__ inline void axis_coord(float x, float o, float inv_h, int n, int& c, float& t, bool& inside) {
  const float a = x, b = -o;
  const float s = a + b;
  const float bb = s - a;
  const float e = (a - (s - bb)) + (b - bb);
  float u = s * inv_h;
  const float ue = e * inv_h;
  inside = true;
  float fl = floorf(u);
  float frac = (u - fl) + ue;
  if (!(u + ue >= 0.f)) {  // below the lattice, or NaN
    fl = 0.f;
    frac = 0.f;
    inside = false;
  } else if (!(fl + frac < (float)(n - 1))) {  // at or beyond the last node, including u = +inf
    fl = (float)(n - 2);
    frac = 1.f;
    if (u + ue > (float)(n - 1)) inside = false;
  } else if (frac >= 1.f) {  // ue pushed the offset into the next cell
    fl += 1.f;
    frac -= 1.f;
  } else if (frac < 0.f) {
    fl -= 1.f;
    frac += 1.f;
  }
  c = (int)fl;
  t = frac;
}

struct GridOut {
  float e_g, e_sg;   // Psi_g, Psi_sg contributions of this atom
  float fx, fy, fz;  // -(w_sg dPsi_sg + w_g dPsi_g)/dx
  bool outside;
};

// Trilinear value and gradient (in lattice units) of two channels at once from the 8 corner values
// c_zyx, in paired FP32 instructions: per channel, the edge differences along x and the values
// interpolated along x, then along y (with the y and x gradients), then along z.  Each half
// performs the operations of the one-channel interpolant in the same order.
struct Tri2 {
  f32x2 v, gx, gy, gz;
};
__device__ inline Tri2 tri2(f32x2 c000, f32x2 c001, f32x2 c010, f32x2 c011, f32x2 c100, f32x2 c101, f32x2 c110,
                            f32x2 c111, f32x2 tx, f32x2 ty, f32x2 tz) {
  const f32x2 d00 = sub2(c001, c000), d01 = sub2(c011, c010), d10 = sub2(c101, c100), d11 = sub2(c111, c110);
  const f32x2 a00 = fma2(tx, d00, c000), a01 = fma2(tx, d01, c010);
  const f32x2 a10 = fma2(tx, d10, c100), a11 = fma2(tx, d11, c110);
  const f32x2 by0 = sub2(a01, a00), by1 = sub2(a11, a10);
  const f32x2 b0 = fma2(ty, by0, a00), b1 = fma2(ty, by1, a10);
  const f32x2 bx0 = fma2(ty, sub2(d01, d00), d00), bx1 = fma2(ty, sub2(d11, d10), d10);
  Tri2 r;
  r.gz = sub2(b1, b0);
  r.v = fma2(tz, r.gz, b0);
  r.gx = fma2(tz, sub2(bx1, bx0), bx0);
  r.gy = fma2(tz, sub2(by1, by0), by0);
  return r;
}
__device__ inline f32x2 lo2(float4 c) { return pack2(c.x, c.y); }
__device__ inline f32x2 hi2(float4 c) { return pack2(c.z, c.w); }

// Grid energies and forces of one atom.  hard / soft select which lattices are read.  The hard
// lattice's channels run as the pairs (LJr^1/4, LJa) and (elec, 0), the soft lattice's as one pair.
__device__ inline GridOut grid_atom(const GridDev& G, float x, float y, float z, float sA, float sB, float q,
                                    bool hard, bool soft, float w_sg, float w_g) {
  GridOut o{0.f, 0.f, 0.f, 0.f, 0.f, false};
  int cx, cy, cz;
  float tx, ty, tz;
  bool ix, iy, iz;
  axis_coord(x, G.ox, G.inv_h, G.nx, cx, tx, ix);
  axis_coord(y, G.oy, G.inv_h, G.ny, cy, ty, iy);
  axis_coord(z, G.oz, G.inv_h, G.nz, cz, tz, iz);
  o.outside = !(ix && iy && iz);
  const float mx = ix ? G.inv_h : 0.f, my = iy ? G.inv_h : 0.f, mz = iz ? G.inv_h : 0.f;
  const int64_t sy = G.nx, sz = (int64_t)G.nx * G.ny;
  const int64_t b = (int64_t)cz * sz + (int64_t)cy * sy + cx;
  const f32x2 tx2 = pack2(tx, tx), ty2 = pack2(ty, ty), tz2 = pack2(tz, tz);
  f32x2 gx2 = 0ull, gy2 = 0ull, gz2 = 0ull;  // (sum of the weighted channel gradients) in two halves
  if (hard) {  // four x-pair records: corners (x, x+1) of each (y, z) edge in one 32-byte load
    float4 c000, c001, c010, c011, c100, c101, c110, c111;
    ldg_pair(G.hard + 2 * b, c000, c001);
    ldg_pair(G.hard + 2 * (b + sy), c010, c011);
    ldg_pair(G.hard + 2 * (b + sz), c100, c101);
    ldg_pair(G.hard + 2 * (b + sz + sy), c110, c111);
    const Tri2 ra = tri2(lo2(c000), lo2(c001), lo2(c010), lo2(c011), lo2(c100), lo2(c101), lo2(c110), lo2(c111), tx2,
                         ty2, tz2);
    const Tri2 e0 = tri2(hi2(c000), hi2(c001), hi2(c010), hi2(c011), hi2(c100), hi2(c101), hi2(c110), hi2(c111), tx2,
                         ty2, tz2);
    float rv, av, ev, zv;
    unpack2(ra.v, rv, av);
    unpack2(e0.v, ev, zv);
    const float r2 = rv * rv;
    o.e_g = sA * (r2 * r2) + sB * av + q * ev;
    if (w_g != 0.f) {
      const float cr = 4.f * sA * r2 * rv;
      const f32x2 kra = pack2(w_g * cr, w_g * sB), ke = pack2(w_g * q, 0.f);
      gx2 = fma2(kra, ra.gx, mul2(ke, e0.gx));
      gy2 = fma2(kra, ra.gy, mul2(ke, e0.gy));
      gz2 = fma2(kra, ra.gz, mul2(ke, e0.gz));
    }
  }
  if (soft) {  // two (x, y) quad records: the corners of the cell's lower and upper z face
    float4 e00, e01, e10, e11;
    ldg_pair(G.soft + 2 * b, e00, e01);
    ldg_pair(G.soft + 2 * (b + sz), e10, e11);
    const Tri2 re = tri2(lo2(e00), hi2(e00), lo2(e01), hi2(e01), lo2(e10), hi2(e10), lo2(e11), hi2(e11), tx2, ty2, tz2);
    float rv, ev;
    unpack2(re.v, rv, ev);
    const float r2 = rv * rv;
    o.e_sg = sA * (r2 * r2) + q * ev;
    if (w_sg != 0.f) {
      const f32x2 k = pack2(w_sg * (4.f * sA * r2 * rv), w_sg * q);
      gx2 = fma2(k, re.gx, gx2);
      gy2 = fma2(k, re.gy, gy2);
      gz2 = fma2(k, re.gz, gz2);
    }
  }
  float ga, gb;
  unpack2(gx2, ga, gb);
  o.fx = -(ga + gb) * mx;
  unpack2(gy2, ga, gb);
  o.fy = -(ga + gb) * my;
  unpack2(gz2, ga, gb);
  o.fz = -(ga + gb) * mz;
  return o;
}

struct Energies {
  float lig;    // bonded + nonbonded (pairs counted from both ends, halved)
  float rest;   // restraint
  float sg, g;  // grid terms
};

__device__ inline float3 sub(float4 a, float4 b) { return make_float3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ inline float dot(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ inline float3 cross(float3 a, float3 b) {
  return make_float3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__device__ inline void put(float4* sl, int s, float3 f) { sl[s] = make_float4(f.x, f.y, f.z, 0.f); }

// Step 1: bonded terms first, first + stride, ... of each kind, one per lane; per-role forces to
// the replica's float4 slots.
// Slots: bond t role r -> r*nb + t; angle -> 2nb + r*nang + t; torsion -> 2nb + 3nang + r*ntor + t.
template <bool ENERGY, bool FORCES = true>
__device__ inline float bonded_terms(const Lig& L, const LigandLayout& LL, const float4* xs, float4* sl, int first,
                                     int stride) {
  float e = 0.f;
  const int nb = LL.nb, nang = LL.nang, ntor = LL.ntor;
  for (int t = first; t < nb; t += stride) {  // k (r - r0)^2
    const float4 bp = L.bond[t];
    const float3 d = sub(xs[__float_as_int(bp.x)], xs[__float_as_int(bp.y)]);
    const float r2 = dot(d, d);
    const float inv_r = rsqrt_fast(r2);
    const float dr = r2 * inv_r - bp.w;
    if (ENERGY) e += bp.z * dr * dr;
    const float c = -2.f * bp.z * dr * inv_r;
    if (FORCES) put(sl, t, make_float3(c * d.x, c * d.y, c * d.z));
    if (FORCES) put(sl, nb + t, make_float3(-c * d.x, -c * d.y, -c * d.z));
  }
  const int ab = 2 * nb;
  for (int t = first; t < nang; t += stride) {  // k (theta - theta0)^2
    const int4 id = L.ang_i[t];
    const float4 ap = L.ang_p[t];
    const float3 u = sub(xs[id.x], xs[id.y]);
    const float3 w = sub(xs[id.z], xs[id.y]);
    const float lu2 = dot(u, u), lw2 = dot(w, w);
    const float inv_luw = rsqrt_fast(lu2 * lw2);
    const float c = fminf(1.f, fmaxf(-1.f, dot(u, w) * inv_luw));
    const float dth = acosf(c) - ap.y;
    if (ENERGY) e += ap.x * dth * dth;
    const float coef = 2.f * ap.x * dth * rsqrt_fast(fmaxf(1.f - c * c, 1e-12f));
    const float cu = div_fast(coef * c, lu2), cw = div_fast(coef * c, lw2), cx = coef * inv_luw;
    const float3 fa = make_float3(cx * w.x - cu * u.x, cx * w.y - cu * u.y, cx * w.z - cu * u.z);
    const float3 fc = make_float3(cx * u.x - cw * w.x, cx * u.y - cw * w.y, cx * u.z - cw * w.z);
    if (FORCES) put(sl, ab + t, fa);
    if (FORCES) put(sl, ab + nang + t, make_float3(-(fa.x + fc.x), -(fa.y + fc.y), -(fa.z + fc.z)));
    if (FORCES) put(sl, ab + 2 * nang + t, fc);
  }
  const int tb = ab + 3 * nang;
  for (int t = first; t < ntor; t += stride) {  // sum_n V_n/2 (1 + cos(n phi - gamma_n))
    const int4 id = L.tor_i[t];
    const float4 V = L.tor_v[t], cg = L.tor_c[t], sg = L.tor_s[t];
    const float3 b1 = sub(xs[id.y], xs[id.x]);
    const float3 b2 = sub(xs[id.z], xs[id.y]);
    const float3 b3 = sub(xs[id.w], xs[id.z]);
    const float3 n1 = cross(b1, b2), n2 = cross(b2, b3);
    const float lb22 = dot(b2, b2);
    const float inv_lb2 = rsqrt_fast(lb22);
    const float lb2 = lb22 * inv_lb2;
    const float n1s = fmaxf(dot(n1, n1), 1e-20f), n2s = fmaxf(dot(n2, n2), 1e-20f);
    const float inv = rsqrtf(n1s * n2s);       // finite also where both are at their floor
    const float cp = dot(n1, n2) * inv;        // cos phi
    const float sp = lb2 * dot(b1, n2) * inv;  // sin phi
    const float c2 = 2.f * cp * cp - 1.f, s2 = 2.f * sp * cp;
    const float c3 = cp * (4.f * cp * cp - 3.f), s3 = sp * (3.f - 4.f * sp * sp);
    if (ENERGY)
      e += V.x * (1.f + cp * cg.x + sp * sg.x) + V.y * (1.f + c2 * cg.y + s2 * sg.y) +
           V.z * (1.f + c3 * cg.z + s3 * sg.z);
    // dE/dphi = sum_n V_n/2 n (cos(n phi) sin g - sin(n phi) cos g)
    const float dE = V.x * (cp * sg.x - sp * cg.x) + 2.f * V.y * (c2 * sg.y - s2 * cg.y) +
                     3.f * V.z * (c3 * sg.z - s3 * cg.z);
    const float ai = div_fast(dE * lb2, n1s), al = -div_fast(dE * lb2, n2s);  // F_i = ai n1, F_l = al n2
    const float inv_lb22 = inv_lb2 * inv_lb2;
    const float p = dot(b1, b2) * inv_lb22, q = dot(b3, b2) * inv_lb22;
    const float3 fi = make_float3(ai * n1.x, ai * n1.y, ai * n1.z);
    const float3 fl = make_float3(al * n2.x, al * n2.y, al * n2.z);
    const float3 fj = make_float3(-(1.f + p) * fi.x + q * fl.x, -(1.f + p) * fi.y + q * fl.y,
                                  -(1.f + p) * fi.z + q * fl.z);
    const float3 fk = make_float3(p * fi.x - (1.f + q) * fl.x, p * fi.y - (1.f + q) * fl.y,
                                  p * fi.z - (1.f + q) * fl.z);
    if (FORCES) put(sl, tb + t, fi);
    if (FORCES) put(sl, tb + ntor + t, fj);
    if (FORCES) put(sl, tb + 2 * ntor + t, fk);
    if (FORCES) put(sl, tb + 3 * ntor + t, fl);
  }
  return e;
}

// Step 3: nonbonded pairs.  A pass covers atoms base .. base+31; a pass with at most 16 atoms gives
// each atom two lanes, which split the partner range and combine with one shuffle.  Adds the
// lane's energies to e2 and returns the force on atom base + lane (valid where that atom exists).
template <bool ENERGY>
__device__ inline float3 nonbonded_pass(const Lig& L, int na, int base, const float4* xs, float& e2) {
  const int lane = threadIdx.x & 31;
  const int m = na - base;
  const bool split = m <= 16;
  const int il = split ? (lane & 15) : lane;
  const int i = base + il;
  const bool act = il < m;
  // partners: all j; split: the low half-warp takes j = 0 .. h-1 upwards, the high half-warp
  // j = na-1 .. h downwards (opposite directions keep the two rows read per step in different
  // shared-memory banks)
  int jb = 0, cnt = na, dir = 1;
  if (split) {
    const int h = (na + 1) >> 1;
    jb = lane < 16 ? 0 : na - 1;
    cnt = lane < 16 ? h : na - h;
    dir = lane < 16 ? 1 : -1;
  }
  float fx = 0.f, fy = 0.f, fz = 0.f;
  if (act) {
    const float4 pi = xs[i];
    const float4 bi = L.atom_b[i];
    const float qi = (float)kCoulomb * pi.w, ri = bi.x, si = bi.y;
    const uint8_t* ty_col = L.ptype + i;
    for (int jj = 0; jj < cnt; ++jj) {
      const int j = jb + dir * jj;
      const float4 pj = xs[j];
      const float2 bj = *(const float2*)&L.atom_b[j];
      const uint32_t ty = ty_col[j * na];
      const bool excluded = ty == 2u;
      const float dx = pi.x - pj.x, dy = pi.y - pj.y, dz = pi.z - pj.z;
      const float r2 = excluded ? 1.f : fmaf(dx, dx, fmaf(dy, dy, dz * dz));
      const float inv_r = rsqrt_fast(r2);
      const float inv_r2 = inv_r * inv_r;
      const float R = ri + bj.x;
      const float s2 = R * R * inv_r2;
      const float s6 = s2 * s2 * s2;
      const float eps = excluded ? 0.f : (ty == 1u ? 0.5f : 1.f) * (si * bj.y);
      const float qq = excluded ? 0.f : (ty == 1u ? (float)(1.0 / 1.2) : 1.f) * (qi * pj.w);
      const float eel = qq * inv_r;
      const float fr = fmaf(12.f * eps, s6 * s6 - s6, eel) * inv_r2;
      fx = fmaf(fr, dx, fx);
      fy = fmaf(fr, dy, fy);
      fz = fmaf(fr, dz, fz);
      if (ENERGY) e2 += fmaf(eps, s6 * s6 - 2.f * s6, eel);
    }
  }
  if (split) {
    fx += __shfl_xor_sync(kFull, fx, 16);
    fy += __shfl_xor_sync(kFull, fy, 16);
    fz += __shfl_xor_sync(kFull, fz, 16);
  }
  return make_float3(fx, fy, fz);
}

// The forces of a full pass (more than 16 atoms), partners two at a time: the operations of
// nonbonded_pass in paired instructions up to the pair force, then both partners added in turn, so
// the sums are the same bits.  Pair types come as one byte per two partners, an offset into the
// table of their scales, in place of two bytes and their selects.  22 instructions a partner
// instead of 38.
__device__ inline float3 nonbonded_type_pass(const Lig& L, int na, int base, const float4* xs, const float* xp) {
  const int i = base + (threadIdx.x & 31);
  float fx = 0.f, fy = 0.f, fz = 0.f;
  if (i < na) {
    const float4 own = xs[i];
    const float2 b = *(const float2*)&L.atom_b[i];
    const float qc = (float)kCoulomb * own.w;
    const f32x2 X = pack2(own.x, own.x), Y = pack2(own.y, own.y), Z = pack2(own.z, own.z);
    const f32x2 Qi = pack2(qc, qc), Ri = pack2(b.x, b.x), Si = pack2(b.y, b.y), twelve = pack2(12.f, 12.f);
    constexpr f32x2 sign = 0x8000000080000000ull;
    const float4* pp = (const float4*)xp;
    const float4* par = L.ppar;
    const uint8_t* combo = L.combo + i;
#pragma unroll 2
    for (int p = (na + 1) >> 1; p > 0; --p) {
      const float4 q0 = pp[0];  // (x, x', y, y')
      const float4 q1 = pp[1];  // (z, z', q, q')
      const float4 s = *par;    // (R*, R*', sqrt(eps), sqrt(eps)')
      const float4 c = *(const float4*)((const char*)L.scale + *combo);
      pp += 2;
      ++par;
      combo += na;
      const f32x2 dx = sub2(X, pack2(q0.x, q0.y)), dy = sub2(Y, pack2(q0.z, q0.w));
      const f32x2 dz = sub2(Z, pack2(q1.x, q1.y));
      float ra, rb;
      unpack2(fma2(dx, dx, fma2(dy, dy, mul2(dz, dz))), ra, rb);
      ra = c.z == 0.f ? 1.f : ra;  // excluded (also i itself and the partner that completes an odd count)
      rb = c.w == 0.f ? 1.f : rb;
      const f32x2 inv_r = pack2(rsqrt_fast(ra), rsqrt_fast(rb));
      const f32x2 inv_r2 = mul2(inv_r, inv_r);
      const f32x2 R = add2(Ri, pack2(s.x, s.y));
      const f32x2 s2 = mul2(mul2(R, R), inv_r2);
      const f32x2 s6 = mul2(mul2(s2, s2), s2);
      const f32x2 eps = mul2(pack2(c.x, c.y), mul2(Si, pack2(s.z, s.w)));
      const f32x2 qq = mul2(pack2(c.z, c.w), mul2(Qi, pack2(q1.z, q1.w)));
      const f32x2 fr = mul2(fma2(mul2(twelve, eps), fma2(s6, s6, s6 ^ sign), mul2(qq, inv_r)), inv_r2);
      float fa, fb, da, db;
      unpack2(fr, fa, fb);
      unpack2(dx, da, db);
      fx = fmaf(fb, db, fmaf(fa, da, fx));
      unpack2(dy, da, db);
      fy = fmaf(fb, db, fmaf(fa, da, fy));
      unpack2(dz, da, db);
      fz = fmaf(fb, db, fmaf(fa, da, fz));
    }
  }
  return make_float3(fx, fy, fz);
}

// The energies of a pass (full or split) for atom base + lane, partners two at a time, as
// nonbonded_type_pass: the same terms added to e in the same order as nonbonded_pass.
__device__ inline void nonbonded_energy_pass(const Lig& L, int na, int base, const float4* xs, const float* xp,
                                             float& e) {
  const int lane = threadIdx.x & 31;
  const int m = na - base, P = (na + 1) >> 1;
  const bool split = m <= 16;
  const int i = base + (split ? (lane & 15) : lane);
  // split: the low half-warp takes j = 0 .. h-1 upwards, the high one j = na-1 .. h downwards; an odd
  // h leaves each half one partner of the middle pair
  const int h = (na + 1) >> 1;
  const bool down = split && lane >= 16;
  const int cnt = !split ? P : (down ? P - h / 2 : (h + 1) / 2);
  const int middle = split && (h & 1) ? h / 2 : -1;
  if (i >= na) return;
  const float4 own = xs[i];
  const float2 b = *(const float2*)&L.atom_b[i];
  const float qc = (float)kCoulomb * own.w;
  const f32x2 X = pack2(own.x, own.x), Y = pack2(own.y, own.y), Z = pack2(own.z, own.z);
  const f32x2 Qi = pack2(qc, qc), Ri = pack2(b.x, b.x), Si = pack2(b.y, b.y), minus_two = pack2(-2.f, -2.f);
  int p = down ? P - 1 : 0;
  const int step = down ? -1 : 1;
#pragma unroll 2
  for (int k = 0; k < cnt; ++k, p += step) {
    const float4 q0 = ((const float4*)xp)[2 * p];      // (x, x', y, y')
    const float4 q1 = ((const float4*)xp)[2 * p + 1];  // (z, z', q, q')
    const float4 s = L.ppar[p];                        // (R*, R*', sqrt(eps), sqrt(eps)')
    const float4 c = *(const float4*)((const char*)L.scale + L.combo[p * na + i]);
    const f32x2 dx = sub2(X, pack2(q0.x, q0.y)), dy = sub2(Y, pack2(q0.z, q0.w));
    const f32x2 dz = sub2(Z, pack2(q1.x, q1.y));
    float ra, rb;
    unpack2(fma2(dx, dx, fma2(dy, dy, mul2(dz, dz))), ra, rb);
    ra = c.z == 0.f ? 1.f : ra;  // excluded (also i itself and the partner that completes an odd count)
    rb = c.w == 0.f ? 1.f : rb;
    const f32x2 inv_r = pack2(rsqrt_fast(ra), rsqrt_fast(rb));
    const f32x2 inv_r2 = mul2(inv_r, inv_r);
    const f32x2 R = add2(Ri, pack2(s.x, s.y));
    const f32x2 s2 = mul2(mul2(R, R), inv_r2);
    const f32x2 s6 = mul2(mul2(s2, s2), s2);
    const f32x2 eps = mul2(pack2(c.x, c.y), mul2(Si, pack2(s.z, s.w)));
    const f32x2 qq = mul2(pack2(c.z, c.w), mul2(Qi, pack2(q1.z, q1.w)));
    const f32x2 lj = fma2(s6, s6, mul2(minus_two, s6));
    float ea, eb;
    unpack2(fma2(eps, lj, mul2(qq, inv_r)), ea, eb);
    if (p == middle) {  // the other half-warp's partner adds nothing here
      ea = down ? 0.f : ea;
      eb = down ? eb : 0.f;
    }
    e += down ? eb : ea;
    e += down ? ea : eb;
  }
}

template <int APL>
__device__ inline void nonbonded(const Lig& L, int na, const float4* xs, float (&F)[APL][3], float& el) {
  const int lane = threadIdx.x & 31;
  float e2 = 0.f;
#pragma unroll
  for (int a = 0; a < APL; ++a) {
    const int m = na - 32 * a;
    if (m <= 0) break;
    const float3 f = nonbonded_pass<true>(L, na, 32 * a, xs, e2);
    if (lane < m) {
      F[a][0] += f.x;
      F[a][1] += f.y;
      F[a][2] += f.z;
    }
  }
  el += 0.5f * e2;
}

// Step 3 from the pair table: the same passes and lane layout as `nonbonded`, with each pair's
// scaled coefficients read from the table (12 eps_ij s_LJ, 332 q_i q_j s_el; zero for excluded
// pairs and i == j) instead of being formed from per-atom parameters and the pair type.
// R_ij = R*_i + R*_j (Lorentz-Berthelot) is formed in registers.  r^2 is floored at 0.01 A^2 so
// that a zero record meets finite powers (i == j): (R_ij / r)^12 stays below 1e20 for R_ij <= 4 A.
//
// Partners come two at a time (j = 2p, 2p + 1), and the two terms share paired FP32 instructions:
// the positions are read from the pair-interleaved mirror xp (8 floats per partner pair:
// x, x', y, y', z, z', R*, R*'), the coefficients from one 16-byte record per atom and partner
// pair, so that every operand pair arrives in one aligned register pair.  An odd na ends with a
// zero partner (zero position and radius, zero records).  Each half accumulates its own forces and
// energy; the halves are added at the end of a pass.
constexpr float kPairMinR2 = 1.0e-2f;

// Writes atom i's coordinates into the pair-interleaved mirror.
__device__ inline void put_pair_pos(float* xp, int i, float x, float y, float z) {
  float* b = xp + 8 * (i >> 1) + (i & 1);
  b[0] = x;
  b[2] = y;
  b[4] = z;
}

template <bool ENERGY, int UNROLL>
__device__ inline float3 nonbonded_table_pass(const Lig& L, int na, int base, const float4* xs, const float* xp,
                                              f32x2& e2) {
  const int lane = threadIdx.x & 31;
  const int P = (na + 1) >> 1;
  const f32x2 one = pack2(1.f, 1.f), two = pack2(2.f, 2.f), twelfth = pack2(1.f / 12.f, 1.f / 12.f);
  const int m = na - base;
  const bool split = m <= 16;
  const int il = split ? (lane & 15) : lane;
  const int i = base + il;
  const bool act = il < m;
  int pb = 0, cnt = P, dir = 1;
  if (split) {
    const int h = (P + 1) >> 1;
    pb = lane < 16 ? 0 : P - 1;
    cnt = lane < 16 ? h : P - h;
    dir = lane < 16 ? 1 : -1;
  }
  f32x2 fx2 = 0ull, fy2 = 0ull, fz2 = 0ull;
  if (act) {
    const float4 own = xs[i];  // (x, y, z, R*_i) in the table path
    const f32x2 X = pack2(own.x, own.x), Y = pack2(own.y, own.y), Z = pack2(own.z, own.z);
    const f32x2 Ri = pack2(own.w, own.w);
    const float4* rec = L.pair + (size_t)pb * na + i;
    const float4* pp = (const float4*)xp + 2 * pb;
    const int rstep = dir * na, pstep = 2 * dir;
#pragma unroll UNROLL
    for (int jj = 0; jj < cnt; ++jj) {
      const float4 q0 = pp[0];  // (x, x', y, y')
      const float4 q1 = pp[1];  // (z, z', R*, R*')
      const float4 t = *rec;    // (e, e', c, c')
      pp += pstep;
      rec += rstep;
      const f32x2 dx = sub2(X, pack2(q0.x, q0.y)), dy = sub2(Y, pack2(q0.z, q0.w));
      const f32x2 dz = sub2(Z, pack2(q1.x, q1.y));
      float ra, rb;
      unpack2(fma2(dx, dx, fma2(dy, dy, mul2(dz, dz))), ra, rb);
      const f32x2 inv_r = pack2(rsqrt_fast(fmaxf(ra, kPairMinR2)), rsqrt_fast(fmaxf(rb, kPairMinR2)));
      const f32x2 R = add2(Ri, pack2(q1.z, q1.w));
      const f32x2 inv_r2 = mul2(inv_r, inv_r);
      const f32x2 s2 = mul2(mul2(R, R), inv_r2);
      const f32x2 s6 = mul2(mul2(s2, s2), s2);
      const f32x2 e = pack2(t.x, t.y);
      const f32x2 eel = mul2(pack2(t.z, t.w), inv_r);
      const f32x2 fr = mul2(fma2(e, mul2(s6, sub2(s6, one)), eel), inv_r2);
      fx2 = fma2(fr, dx, fx2);
      fy2 = fma2(fr, dy, fy2);
      fz2 = fma2(fr, dz, fz2);
      if (ENERGY) e2 = add2(e2, fma2(mul2(e, twelfth), mul2(s6, sub2(s6, two)), eel));
    }
  }
  float fx, fy, fz, ha, hb;
  unpack2(fx2, fx, ha);
  fx += ha;
  unpack2(fy2, fy, ha);
  fy += ha;
  unpack2(fz2, fz, hb);
  fz += hb;
  if (split) {
    fx += __shfl_xor_sync(kFull, fx, 16);
    fy += __shfl_xor_sync(kFull, fy, 16);
    fz += __shfl_xor_sync(kFull, fz, 16);
  }
  return make_float3(fx, fy, fz);
}

// Step 2a: the bonded forces gathered over the lanes' balanced runs of the atom-sorted slot list
// (the gather schedule): each lane adds its run in order and stores the partial sum of every atom
// it ends in that atom's last slot of the run.
__device__ inline void gather_runs(const Lig& L, const LigandLayout& LL, float4* sl) {
  const int lane = threadIdx.x & 31;
  float ax = 0.f, ay = 0.f, az = 0.f;
  const uint2* gs = L.gs + lane;
  for (int j = 0; j < LL.gs_iters; ++j) {
    const uint2 w = gs[32 * j];
    const uint32_t e[4] = {w.x & 0xffffu, w.x >> 16, w.y & 0xffffu, w.y >> 16};
    float4 v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = sl[e[k] & 0x7fffu];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      ax += v[k].x;
      ay += v[k].y;
      az += v[k].z;
      if (e[k] & 0x8000u) {
        sl[e[k] & 0x7fffu] = make_float4(ax, ay, az, 0.f);
        ax = ay = az = 0.f;
      }
    }
  }
}

// Restraint energy of the summed m x.
__device__ inline float restraint_energy(const LigandLayout& LL, float mx, float my, float mz) {
  const float invM = 1.f / LL.total_mass;
  const float dx = mx * invM - LL.site[0], dy = my * invM - LL.site[1], dz = mz * invM - LL.site[2];
  const float d = sqrtf(dx * dx + dy * dy + dz * dz);
  if (d > LL.d0) {
    const float ex = d - LL.d0;
    return 0.5f * LL.k_rest * ex * ex;
  }
  return d <= LL.d0 ? 0.f : d;  // NaN centre of mass: make the energy NaN
}

// Energies and the forces on the lane's atoms of one configuration by one warp, lane l holding atoms l,
// l+32, l+64.  xs holds all positions (x, y, z, q); sl is the warp's bonded-slot scratch (n_slots + 1
// float4, the last zero).
template <int APL>
__device__ inline void evaluate(const LigandLayout& LL, const Lig& L, const GridDev& G, const float4* xs, float4* sl,
                                const float (&x)[APL][3], const float (&mass)[APL], float (&F)[APL][3], float w_sg,
                                float w_g, Energies& en) {
  const int lane = threadIdx.x & 31;
  const int na = LL.na;
  float el = bonded_terms<true>(L, LL, xs, sl, lane, 32);
  __syncwarp();
  gather_runs(L, LL, sl);
  __syncwarp();
  float eg = 0.f, esg = 0.f;
  float mx = 0.f, my = 0.f, mz = 0.f;
#pragma unroll
  for (int a = 0; a < APL; ++a) {
    const int i = lane + 32 * a;
    F[a][0] = F[a][1] = F[a][2] = 0.f;
    if (i >= na) continue;
    const float4 pa = L.atom_a[i];
    mx += mass[a] * x[a][0];
    my += mass[a] * x[a][1];
    mz += mass[a] * x[a][2];
    const GridOut go = grid_atom(G, x[a][0], x[a][1], x[a][2], pa.z, pa.w, pa.y, true, true, w_sg, w_g);
    F[a][0] += go.fx;
    F[a][1] += go.fy;
    F[a][2] += go.fz;
    eg += go.e_g;
    esg += go.e_sg;
    {  // the atom's partial sums, in run order
      const uint2 p = L.gp[i];
      const float4 q0 = sl[p.x & 0xffffu], q1 = sl[p.x >> 16], q2 = sl[p.y & 0xffffu], q3 = sl[p.y >> 16];
      F[a][0] += ((q0.x + q1.x) + q2.x) + q3.x;
      F[a][1] += ((q0.y + q1.y) + q2.y) + q3.y;
      F[a][2] += ((q0.z + q1.z) + q2.z) + q3.z;
    }
  }
  nonbonded<APL>(L, na, xs, F, el);
  // restraint on the centre of mass
  mx = warp_sumf(mx);
  my = warp_sumf(my);
  mz = warp_sumf(mz);
  const float invM = 1.f / LL.total_mass;
  const float dx = mx * invM - LL.site[0], dy = my * invM - LL.site[1], dz = mz * invM - LL.site[2];
  const float d = sqrtf(dx * dx + dy * dy + dz * dz);
  float er = 0.f;
  if (d > LL.d0) {
    const float ex = d - LL.d0;
    er = 0.5f * LL.k_rest * ex * ex;
    const float c = -LL.k_rest * ex / d * invM;
#pragma unroll
    for (int a = 0; a < APL; ++a) {
      const int i = lane + 32 * a;
      if (i >= na) continue;
      F[a][0] += c * mass[a] * dx;
      F[a][1] += c * mass[a] * dy;
      F[a][2] += c * mass[a] * dz;
    }
  } else if (!(d <= LL.d0)) {  // NaN centre of mass: make the energy NaN
    er = d;
  }
  en.lig = el;
  en.rest = lane == 0 ? er : 0.f;
  en.sg = esg;
  en.g = eg;
}

// The four components summed over the warp.  The butterfly's pairs, with two of the four sums (then
// one) kept per lane at the first steps: 6 FP64 additions a lane instead of 20, the same sums.
__device__ inline void reduce_components(const Energies& e, double c[4]) {
  const int lane = threadIdx.x & 31;
  const double lig = (double)e.lig, rest = (double)e.rest, sg = (double)e.sg, g = (double)e.g;
  const bool h16 = lane & 16, h8 = lane & 8;
  const double k0 = (h16 ? sg : lig) + __shfl_xor_sync(kFull, h16 ? lig : sg, 16);
  const double k1 = (h16 ? g : rest) + __shfl_xor_sync(kFull, h16 ? rest : g, 16);
  double v = (h8 ? k1 : k0) + __shfl_xor_sync(kFull, h8 ? k0 : k1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
#pragma unroll
  for (int j = 0; j < 4; ++j) c[j] = __shfl_sync(kFull, v, 8 * j);
}

// U_k = ((U_L + U_I) + w_sg Psi_sg) + w_g Psi_g, a zero weight dropping its term.
__device__ inline double weighted(const double c[4], double w_sg, double w_g) {
  double e = __dadd_rn(c[0], c[1]);
  if (w_sg != 0.0) e = __dadd_rn(e, __dmul_rn(w_sg, c[2]));
  if (w_g != 0.0) e = __dadd_rn(e, __dmul_rn(w_g, c[3]));
  return e;
}

__device__ inline void stage_ligand(uint32_t* s, const uint32_t* __restrict__ blob, int words) {
  const uint4* src = (const uint4*)blob;
  uint4* dst = (uint4*)s;
  for (int i = threadIdx.x; i < words / 4; i += blockDim.x) dst[i] = src[i];
}

// Shared memory of one replica: 32*APL float4 positions, the pair-interleaved mirror of the pair loop
// (32*APL * 4 floats), the bonded-slot scratch (n_slots + 1 float4, the last a zero slot) and, for a
// team of warps, what they exchange.  A block holds the ligand blob and one such area per replica
// (of the energy kernel: per warp, without the mirror and the exchange area, which is also what the
// rule on the pair table counts, with the mirror where the table is).
__host__ __device__ inline int scratch_words(const LigandLayout& L) { return 4 * (L.n_slots + 1); }
__host__ __device__ inline int warp_words(const LigandLayout& L, int apl, bool table) {
  return (table ? 8 : 4) * 32 * apl + scratch_words(L);
}
struct TeamExchange {
  f32x2 lane[32];                // per-lane values on their way to the first warp
  float rx, ry, rz, rc, re;      // restraint: displacement, force factor, energy
  int accept;
  unsigned long long replica[2];
};
constexpr int kTeamWords = (sizeof(TeamExchange) + 15) / 16 * 4;
__host__ __device__ inline int replica_words(const LigandLayout& L, int apl) {
  return warp_words(L, apl, true) + (apl > 1 ? kTeamWords : 0);
}
// Staged tables of a block: the blob with the pair table, or without it the pair-type tables after it.
__host__ __device__ inline int combo_words(const LigandLayout& L) { return (((L.na + 1) / 2) * L.na + 15) / 16 * 4; }
__host__ __device__ inline int staged_words(const LigandLayout& L, bool table) {
  return table ? L.words_pair : L.words + 4 * ((L.na + 1) / 2) + 64 + combo_words(L);
}

struct WarpSmem {
  float4* xs;
  float* xp;   // pair-interleaved positions and R* (pair table) or charges
  float4* sl;  // bonded-force slots
  TeamExchange* ex;
};
template <int APL, bool MIRROR>
__device__ inline WarpSmem warp_smem(uint32_t* p, const LigandLayout& LL) {
  float* xp = MIRROR ? (float*)(p + 4 * 32 * APL) : nullptr;
  float4* sl = (float4*)(p + (MIRROR ? 8 : 4) * 32 * APL);
  return WarpSmem{(float4*)p, xp, sl, (TeamExchange*)(p + warp_words(LL, APL, MIRROR))};
}

// The pair-type tables (Lig::ppar, scale, combo) from the staged blob, by the whole block.
__device__ inline void stage_types(uint32_t* s, const LigandLayout& LL, Lig& L) {
  const int na = LL.na, P = (na + 1) / 2;
  float4* par = (float4*)(s + LL.words);
  float4* scale = par + P;
  uint8_t* combo = (uint8_t*)(scale + 16);
  const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int p = threadIdx.x; p < P; p += blockDim.x) {
    const float4 a = L.atom_b[2 * p], b = 2 * p + 1 < na ? L.atom_b[2 * p + 1] : none;
    par[p] = make_float4(a.x, b.x, a.y, b.y);
  }
  for (int e = threadIdx.x; e < 16; e += blockDim.x) {
    auto lj = [](int ty) { return ty == 0 ? 1.f : (ty == 1 ? 0.5f : 0.f); };
    auto el = [](int ty) { return ty == 0 ? 1.f : (ty == 1 ? (float)(1.0 / 1.2) : 0.f); };
    scale[e] = make_float4(lj(e & 3), lj(e >> 2), el(e & 3), el(e >> 2));
  }
  for (int e = threadIdx.x; e < P * na; e += blockDim.x) {
    const int p = e / na, i = e - p * na;
    const int ta = L.ptype[2 * p * na + i], tb = 2 * p + 1 < na ? L.ptype[(2 * p + 1) * na + i] : 2;
    combo[e] = (uint8_t)(16 * (ta | tb << 2));
  }
  L.ppar = par;
  L.scale = scale;
  L.combo = combo;
}

struct HmcArgs {
  GridDev G;
  LigandLayout LL;
  const uint32_t* blob;
  const StateDev* states;
  int n_states;
  int64_t n_rep;
  const int32_t* state_of;
  float* x;
  double* comps;
  double* dH;
  uint8_t* acc;
  int n_steps;
  uint64_t seed;
  uint32_t cycle;
  int64_t rep_offset;
  int64_t* counters;
  // batches only: the ligand records, this launch's work items (one per block) and the position
  // stride of a replica (atoms)
  const BatchLigand* bligs;
  const BatchItem* items;
  int x_stride;
  unsigned long long* work;  // single-ligand launches: replicas handed out so far (zero at launch), or NULL
};

// The warps of a replica's team: warp w of W holds atoms 32w .. 32w+31.
template <int W>
__device__ __forceinline__ void team_sync(int team) {
  if (W == 1) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(team), "n"(32 * W) : "memory");
}

// One force evaluation by the team, with the positions published.  The pieces and the order of
// every sum are those of one warp holding all atoms; the pieces that do not depend on one another
// run in different warps:
//   - bonded terms over all the team's lanes; then
//   - the last warp, which has the fewest atoms, adds the slots over the balanced runs and forms the
//     centre of mass, while each warp does its atoms' grid terms and pairs; then
//   - each warp adds up its atoms' forces.
// An energy evaluation (the first and the last of a trial) also sums energies per lane in the order
// of one warp: the first warp takes all bonded terms, and the pair and grid sums of a lane pass
// through the warps in turn.  Its results are valid in the first warp.
template <int W, bool ENERGY, bool TABLE, int UNROLL>
__device__ __forceinline__ void team_evaluate(const LigandLayout& LL, const Lig& L, const GridDev& G,
                                              const WarpSmem& ws, int w, int team, const float (&x)[3], float mass,
                                              float (&F)[3], float w_sg, float w_g, float invM, float d0_safe2,
                                              Energies& en, int& outside) {
  const int lane = threadIdx.x & 31;
  const int na = LL.na;
  const int i = 32 * w + lane;
  const bool own = i < na;
  float el = 0.f;
  if (ENERGY) {
    if (w == 0) el = bonded_terms<true>(L, LL, ws.xs, ws.sl, lane, 32);
  } else {
    bonded_terms<false>(L, LL, ws.xs, ws.sl, i, 32 * W);
  }
  team_sync<W>(team);
  float rx, ry, rz, rc = 0.f, er = 0.f;
  if (w == W - 1) {
    gather_runs(L, LL, ws.sl);
    float mx = 0.f, my = 0.f, mz = 0.f;
    if (W == 1) {
      if (own) {
        mx += mass * x[0];
        my += mass * x[1];
        mz += mass * x[2];
      }
    } else {
#pragma unroll
      for (int a = 0; a < W; ++a) {
        const int j = lane + 32 * a;
        if (j >= na) continue;
        const float m = L.atom_b[j].z;
        const float4 p = ws.xs[j];
        mx += m * p.x;
        my += m * p.y;
        mz += m * p.z;
      }
    }
    mx = warp_sumf(mx);
    my = warp_sumf(my);
    mz = warp_sumf(mz);
    rx = mx * invM - LL.site[0], ry = my * invM - LL.site[1], rz = mz * invM - LL.site[2];
    const float d2 = rx * rx + ry * ry + rz * rz;
    if (!(d2 < d0_safe2)) {  // not clearly inside
      const float d = sqrtf(d2);
      if (d > LL.d0) {
        const float ex = d - LL.d0;
        er = 0.5f * LL.k_rest * ex * ex;
        rc = -LL.k_rest * ex / d * invM;
      } else if (!(d <= LL.d0)) {  // NaN centre of mass: make the energy NaN
        er = d;
      }
    }
    if (W > 1 && lane == 0) {
      ws.ex->rx = rx;
      ws.ex->ry = ry;
      ws.ex->rz = rz;
      ws.ex->rc = rc;
      ws.ex->re = er;
    }
  }
  const bool hard = ENERGY || w_g != 0.f;
  const bool soft = ENERGY || w_sg != 0.f;
  float eg = 0.f, esg = 0.f;
  F[0] = F[1] = F[2] = 0.f;
  if (own && (hard || soft)) {
    const float4 pa = L.atom_a[i];
    const GridOut go = grid_atom(G, x[0], x[1], x[2], pa.z, pa.w, pa.y, hard, soft, w_sg, w_g);
    F[0] += go.fx;
    F[1] += go.fy;
    F[2] += go.fz;
    eg += go.e_g;
    esg += go.e_sg;
    outside += go.outside ? 1 : 0;
  }
  float3 f = make_float3(0.f, 0.f, 0.f);
  if (!ENERGY || W == 1) {
    f32x2 e2 = 0ull;
    float e1 = 0.f;
    if (TABLE) {
      if (32 * w < na) f = nonbonded_table_pass<ENERGY, UNROLL>(L, na, 32 * w, ws.xs, ws.xp, e2);
    } else if (!ENERGY && na - 32 * w > 16) {
      f = nonbonded_type_pass(L, na, 32 * w, ws.xs, ws.xp);
    } else if (32 * w < na) {
      f = nonbonded_pass<ENERGY>(L, na, 32 * w, ws.xs, e1);
    }
    if (ENERGY) {
      float ea = e1, eb = 0.f;
      if (TABLE) unpack2(e2, ea, eb);
      el += 0.5f * (TABLE ? ea + eb : e1);
    }
  } else {
    for (int a = 0; a < W; ++a) {
      if (w == a && 32 * a < na) {
        f32x2 e2 = a > 0 ? ws.ex->lane[lane] : 0ull;
        if (TABLE) {
          f = nonbonded_table_pass<true, 1>(L, na, 32 * a, ws.xs, ws.xp, e2);
        } else {
          float e1, pad;
          unpack2(e2, e1, pad);
          f = nonbonded_pass<true>(L, na, 32 * a, ws.xs, e1);
          e2 = pack2(e1, 0.f);
        }
        ws.ex->lane[lane] = e2;
      }
      team_sync<W>(team);
    }
    if (w == 0) {
      float ea, eb;
      unpack2(ws.ex->lane[lane], ea, eb);
      el += 0.5f * (TABLE ? ea + eb : ea);
    }
    for (int a = 1; a < W; ++a) {
      team_sync<W>(team);
      if (w == a) ws.ex->lane[lane] = pack2(eg, esg);
      team_sync<W>(team);
      if (w == 0) {
        float v, u;
        unpack2(ws.ex->lane[lane], v, u);
        eg += v;
        esg += u;
      }
    }
  }
  team_sync<W>(team);  // partial sums and restraint
  if (W > 1) {
    rx = ws.ex->rx;
    ry = ws.ex->ry;
    rz = ws.ex->rz;
    rc = ws.ex->rc;
    if (ENERGY) er = ws.ex->re;
  }
  if (own) {
    // the atom's partial sums, in run order
    const uint2 p = L.gp[i];
    const float4 q0 = ws.sl[p.x & 0xffffu], q1 = ws.sl[p.x >> 16], q2 = ws.sl[p.y & 0xffffu], q3 = ws.sl[p.y >> 16];
    F[0] += ((q0.x + q1.x) + q2.x) + q3.x;
    F[1] += ((q0.y + q1.y) + q2.y) + q3.y;
    F[2] += ((q0.z + q1.z) + q2.z) + q3.z;
    F[0] += f.x;
    F[1] += f.y;
    F[2] += f.z;
    if (rc != 0.f) {
      F[0] += rc * mass * rx;
      F[1] += rc * mass * ry;
      F[2] += rc * mass * rz;
    }
  }
  if (ENERGY) {
    en.lig = el;
    en.rest = lane == 0 ? er : 0.f;
    en.sg = esg;
    en.g = eg;
  }
}

// Sum of the atoms' m v^2 (in the first warp): a lane's atoms in order, then over the lanes.  t: the
// calling lane's v^2.
template <int W>
__device__ __forceinline__ double team_kinetic(const Lig& L, int na, const WarpSmem& ws, int w, int team, float mass,
                                               float t) {
  const int lane = threadIdx.x & 31;
  float* buf = (float*)ws.ex->lane;
  if (W > 1) {
    if (w > 0) buf[32 * (w - 1) + lane] = t;
    team_sync<W>(team);
    if (w > 0) return 0.0;
  }
  float kin = 0.f;
  if (lane < na) kin += mass * t;
#pragma unroll
  for (int a = 1; a < W; ++a) {
    const int j = lane + 32 * a;
    if (j < na) kin += L.atom_b[j].z * buf[32 * (a - 1) + lane];
  }
  return warp_sum((double)kin);
}

// One HMC trial of replica r by the calling team: momenta, n_steps of velocity Verlet, the
// Metropolis test, and the write-back of an accepted trial.  ws: the replica's shared-memory arrays
// (the zero partner of an odd atom count and the zero slot are already there).
template <int W, bool TABLE, bool BATCH, int UNROLL>
__device__ __forceinline__ void hmc_trial(const HmcArgs& A, const LigandLayout& LL, const Lig& L, const WarpSmem& ws,
                                          int w, int team, int64_t r) {
  const int lane = threadIdx.x & 31;
  float4* xs = ws.xs;
  float* xp = ws.xp;
  const int na = LL.na;
  const int i = 32 * w + lane;
  const bool own = i < na;
  const int64_t xstride = BATCH ? A.x_stride : na;
  const int k = A.state_of[r];
  if ((unsigned)k >= (unsigned)A.n_states) {  // invalid state index: leave the replica untouched
    if (w == 0 && lane == 0) {
      if (A.dH) A.dH[r] = __longlong_as_double(0x7ff8000000000000ll);
      if (A.acc) A.acc[r] = 0;
    }
    return;
  }
  const StateDev* st = A.states + k;
  const float dt = st->dt, hdt = 0.5f * dt;
  const float w_sg = st->w_sg_f, w_g = st->w_g_f;
  const uint32_t rid = (uint32_t)(A.rep_offset + r);
  const float invM = 1.f / LL.total_mass;
  // below this square the centre of mass is inside the restraint's flat bottom whatever the rounding
  const float d0_safe2 = LL.d0 > 0.f ? LL.d0 * LL.d0 * 0.999f : 0.f;

  float x[3] = {0.f, 0.f, 0.f}, v[3] = {0.f, 0.f, 0.f}, F[3];
  float mass = 0.f, accel = 0.f;  // the atom's mass and force-to-acceleration factor
  // the fourth component: the charge for the pair-type loop, R*_i for the table loop (which
  // reads the partners' positions and radii from the pair-interleaved mirror)
  float fourth = 0.f;
  if (own) {
    const float* src = A.x + (r * xstride + i) * 3;
    x[0] = src[0];
    x[1] = src[1];
    x[2] = src[2];
    const U4 o = philox(A.seed, (uint32_t)i, rid, A.cycle, kPurposeMomentum);
    // Box-Muller: u1 in (0, 1] from 23 bits + 1/2, u2 in [0, 1) from 23 bits (exact in FP32)
    const float u1 = ((float)(o.x >> 9) + 0.5f) * (1.0f / 8388608.0f);
    const float u2 = (float)(o.y >> 9) * (1.0f / 8388608.0f);
    const float u3 = ((float)(o.z >> 9) + 0.5f) * (1.0f / 8388608.0f);
    const float u4 = (float)(o.w >> 9) * (1.0f / 8388608.0f);
    const float rr1 = sqrtf(-2.f * logf(u1)), rr2 = sqrtf(-2.f * logf(u3));
    float s1, c1, s2, c2;
    sincospif(2.f * u2, &s1, &c1);
    sincospif(2.f * u4, &s2, &c2);
    const float4 pb = L.atom_b[i];
    const float4 pa = L.atom_a[i];
    mass = pb.z;
    accel = pa.x;
    const float sd = st->sqrt_kT * pb.w;  // sqrt(kT * 4.184e-4 / m)
    v[0] = rr1 * c1 * sd;
    v[1] = rr1 * s1 * sd;
    v[2] = rr2 * c2 * sd;
    fourth = TABLE ? pb.x : pa.y;
    xs[i] = make_float4(x[0], x[1], x[2], fourth);
    put_pair_pos(xp, i, x[0], x[1], x[2]);
    xp[8 * (i >> 1) + 6 + (i & 1)] = fourth;
  }
  const double mv0 = team_kinetic<W>(L, na, ws, w, team, mass, v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
  team_sync<W>(team);
  int outside = 0;
  Energies en;
  double c[4] = {0.0, 0.0, 0.0, 0.0}, U0 = 0.0, U1 = 0.0;
  for (int s = 0;; ++s) {  // s steps done up to the force evaluation
    if (s == 0 || s == A.n_steps) {
      team_evaluate<W, true, TABLE, 1>(LL, L, A.G, ws, w, team, x, mass, F, w_sg, w_g, invM, d0_safe2,
                                      en, outside);
      if (w == 0) {
        reduce_components(en, c);
        U1 = weighted(c, st->w_sg, st->w_g);
        if (s == 0) {  // the starting components go out now (a rejected trial leaves them); only U0 stays live
          U0 = U1;
          if (lane < 4) A.comps[r * 4 + lane] = lane == 0 ? c[0] : (lane == 1 ? c[1] : (lane == 2 ? c[2] : c[3]));
        }
      }
    } else {
      team_evaluate<W, false, TABLE, UNROLL>(LL, L, A.G, ws, w, team, x, mass, F, w_sg, w_g, invM,
                                            d0_safe2, en, outside);
    }
    if (own && s > 0) {
#pragma unroll
      for (int d = 0; d < 3; ++d) v[d] = fmaf(hdt * accel, F[d], v[d]);
    }
    if (s == A.n_steps) break;
    // every warp has finished reading the previous positions (the evaluation's last barrier)
    if (own) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        v[d] = fmaf(hdt * accel, F[d], v[d]);
        x[d] = fmaf(dt, v[d], x[d]);
      }
      xs[i] = make_float4(x[0], x[1], x[2], fourth);
      put_pair_pos(xp, i, x[0], x[1], x[2]);
    }
    team_sync<W>(team);  // positions published; the bonded slots of the last evaluation read
  }
  const double mv1 = team_kinetic<W>(L, na, ws, w, team, mass, v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
  bool accept = false;
  if (w == 0) {
    const double dH = fma(0.5 * kKineticToKcal, mv1, U1) - fma(0.5 * kKineticToKcal, mv0, U0);
    const U4 o = philox(A.seed, 0u, rid, A.cycle, kPurposeAccept);
    const double u = uniform53(o.x, o.y);
    accept = u < exp(-dH / st->kT);
    if (accept && A.n_steps > 0 && lane < 4)
      A.comps[r * 4 + lane] = lane == 0 ? c[0] : (lane == 1 ? c[1] : (lane == 2 ? c[2] : c[3]));
    if (lane == 0) {
      if (A.dH) A.dH[r] = dH;
      if (A.acc) A.acc[r] = accept ? 1 : 0;
      if (A.counters) {
        if (accept) atomicAdd((unsigned long long*)&A.counters[ALGDOCK_CNT_ACCEPTED], 1ull);
        if (!isfinite(dH)) atomicAdd((unsigned long long*)&A.counters[ALGDOCK_CNT_NONFINITE], 1ull);
      }
      if (W > 1) ws.ex->accept = accept;
    }
  }
  if (W > 1) {
    team_sync<W>(team);
    accept = ws.ex->accept;
  }
  if (accept && own) {  // a rejected trial leaves the stored positions and components as they were
    float* dst = A.x + (r * xstride + i) * 3;
    dst[0] = x[0];
    dst[1] = x[1];
    dst[2] = x[2];
  }
  if (A.counters) {
    const int out_total = __reduce_add_sync(kFull, outside);
    if (lane == 0 && out_total)
      atomicAdd((unsigned long long*)&A.counters[ALGDOCK_CNT_OUTSIDE], (unsigned long long)out_total);
  }
}

// A team of APL warps per replica, one atom per lane; a block holds the ligand's tables and up to
// SLOTS replicas (blockDim.x / (32 APL) of them, fewer where their shared memory does not fit).
// MINB blocks per SM.  At 48 atoms two blocks of 6 replicas take 1596 us, one of 12 1685, of 10 1770, of
// 8 1769, of 16 (64 registers) 1810: more warps wait on the shared-memory pipe (70 % busy) instead.
// TABLE: the pair table is staged with the blob.
// BATCH: the block's ligand and replicas come from its work item (a run of consecutive replicas of
// one ligand of a multi-ligand batch) and positions are stored x_stride atoms apart.
// Otherwise each team runs one replica (team t of block b replica t gridDim.x + b) or, with A.work
// set, the blocks are persistent: each team takes replicas from the work
// counter until all n_rep are handed out, highest index first (the coupling leg, whose trials
// gather the lattices, before the cheaper warming leg), so that no SM idles while another still
// runs a last wave of blocks.  Which team runs a replica does not change its result.
template <int APL, int SLOTS, bool TABLE, bool BATCH = false, int MINB = 1>
__global__ void __launch_bounds__(SLOTS * APL * 32, MINB) hmc_kernel(const HmcArgs A) {
  constexpr int kUnroll = APL == 1 ? 4 : (SLOTS * APL > 24 ? 1 : 2);  // of the table pair loop
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ LigandLayout s_ll;
  const uint32_t* blob = A.blob;
  if (BATCH) {
    const BatchItem it = A.items[blockIdx.x];
    if (threadIdx.x == 0) s_ll = A.bligs[it.lig].LL;
    blob = A.blob + A.bligs[it.lig].blob_off;
    __syncthreads();
  }
  const LigandLayout& LL = BATCH ? s_ll : A.LL;
  const int staged = staged_words(LL, TABLE);
  stage_ligand(smem, blob, TABLE ? LL.words_pair : LL.words);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // A warp's scheduler is its index mod 4.  Teams of two swap their roles every other pair of teams,
  // so that each scheduler gets as many first warps (more atoms) as last ones.
  const int team = warp / APL, w = (APL == 2 ? warp + (team >> 1) : warp) % APL;
  const int slots = (int)blockDim.x / (32 * APL);
  const int na = LL.na;
  const WarpSmem ws = warp_smem<APL, true>(smem + staged + team * replica_words(LL, APL), LL);
  if (w == 0 && lane == 0) {
    ws.sl[LL.n_slots] = make_float4(0.f, 0.f, 0.f, 0.f);  // the zero slot
    if (na & 1) {  // the zero partner that completes the last pair
      put_pair_pos(ws.xp, na, 0.f, 0.f, 0.f);
      ws.xp[8 * (na >> 1) + 7] = 0.f;
    }
  }
  __syncthreads();
  Lig L = bind_ligand(smem, LL);
  if (!TABLE) {
    stage_types(smem, LL, L);
    __syncthreads();
  }
  if (BATCH) {
    const BatchItem it = A.items[blockIdx.x];
    for (int j = team; j < it.count; j += slots) {
      const int64_t r = it.r0 + j;
      if (r < A.n_rep) hmc_trial<APL, TABLE, BATCH, kUnroll>(A, LL, L, ws, w, team, r);
    }
    return;
  }
  if (!A.work) {
    const int64_t r = (int64_t)team * gridDim.x + blockIdx.x;
    if (r < A.n_rep) hmc_trial<APL, TABLE, BATCH, kUnroll>(A, LL, L, ws, w, team, r);
    return;
  }
  for (int it = 0;; it ^= 1) {
    unsigned long long t = 0;
    if (w == 0 && lane == 0) t = atomicAdd(A.work, 1ull);
    if (APL == 1) {
      t = __shfl_sync(kFull, t, 0);
    } else {  // two words in turn: the next is written while a slow warp may still read this one
      if (w == 0 && lane == 0) ws.ex->replica[it] = t;
      team_sync<APL>(team);
      t = ws.ex->replica[it];
    }
    if (t >= (unsigned long long)A.n_rep) break;
    hmc_trial<APL, TABLE, BATCH, kUnroll>(A, LL, L, ws, w, team, A.n_rep - 1 - (int64_t)t);
  }
}

// Energies and forces of stored configurations, one warp each; comps may be NULL.
struct EvalArgs {
  GridDev G;
  LigandLayout LL;
  const uint32_t* blob;
  const StateDev* states;
  int n_states;
  int64_t N;
  const int32_t* state_of;
  const float* x;
  float* force;
  double* comps;
};

template <int APL>
__global__ void __launch_bounds__(kWarpsPerBlock * 32) eval_kernel(const EvalArgs A) {
  extern __shared__ __align__(16) uint32_t smem[];
  stage_ligand(smem, A.blob, A.LL.words);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n = (int64_t)blockIdx.x * kWarpsPerBlock + warp;
  if (n >= A.N) return;
  const Lig L = bind_ligand(smem, A.LL);
  const WarpSmem ws = warp_smem<APL, false>(smem + A.LL.words + warp * warp_words(A.LL, APL, false), A.LL);
  if (lane == 0) ws.sl[A.LL.n_slots] = make_float4(0.f, 0.f, 0.f, 0.f);  // the zero slot
  const int na = A.LL.na;
  const int k = A.state_of[n];
  if ((unsigned)k >= (unsigned)A.n_states) return;  // invalid state index: no output
  const float w_sg = A.states[k].w_sg_f, w_g = A.states[k].w_g_f;
  float x[APL][3], F[APL][3], mass[APL];
#pragma unroll
  for (int a = 0; a < APL; ++a) {
    const int i = lane + 32 * a;
    if (i < na) {
      const float* src = A.x + (n * na + i) * 3;
      x[a][0] = src[0];
      x[a][1] = src[1];
      x[a][2] = src[2];
      mass[a] = L.atom_b[i].z;
      ws.xs[i] = make_float4(x[a][0], x[a][1], x[a][2], L.atom_a[i].y);
    } else {
      x[a][0] = x[a][1] = x[a][2] = mass[a] = 0.f;
    }
  }
  __syncwarp();
  Energies en;
  evaluate<APL>(A.LL, L, A.G, ws.xs, ws.sl, x, mass, F, w_sg, w_g, en);
  double c[4];
  reduce_components(en, c);
#pragma unroll
  for (int a = 0; a < APL; ++a) {
    const int i = lane + 32 * a;
    if (i < na) {
      float* dst = A.force + (n * na + i) * 3;
      dst[0] = F[a][0];
      dst[1] = F[a][1];
      dst[2] = F[a][2];
    }
  }
  if (A.comps && lane < 4) A.comps[n * 4 + lane] = c[lane];
}

// Energies only: no bonded force slots, grid gradients or pair forces, so a warp's shared memory is its
// positions (twice) and 32 warps fit an SM (498 us for 102400 configurations of 48 atoms and their u_kn at
// 128 states; 24 warps 518, 16 warps 567; 791 with one staging of the ligand per four configurations, one
// partner at a time and u_kn in a launch of its own).  Persistent blocks stage the ligand once.  A block
// takes tiles of 8 * per consecutive configurations, `per` to a warp, and, with u_kn, forms their reduced
// energies at k_count states from k_begin while other blocks evaluate: u_kn is FP64 work (5
// operations an element on a pipe of 2 lanes per clock, 105 us for 128 x 102400), the evaluation FP32.
constexpr int kEnergyWarps = 8, kEnergyPer = 4;
struct EnergyArgs {
  GridDev G;
  LigandLayout LL;
  const uint32_t* blob;
  const StateDev* states;
  int64_t N;
  int per;
  const float* x;
  double* comps;  // may be NULL with u_kn
  double* u_kn;   // may be NULL
  int k_begin, k_count;
};

template <int APL>
__global__ void __launch_bounds__(kEnergyWarps * 32, 4) energy_kernel(const EnergyArgs A) {
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ double s_c[kEnergyWarps * kEnergyPer][4];
  const LigandLayout& LL = A.LL;
  const int na = LL.na;
  stage_ligand(smem, A.blob, LL.words);
  __syncthreads();
  Lig L = bind_ligand(smem, LL);
  stage_types(smem, LL, L);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float4* xs = (float4*)(smem + staged_words(LL, false) + warp * 8 * 32 * APL);
  float* xp = (float*)(xs + 32 * APL);
  if ((na & 1) && lane == 0) {  // the zero partner that completes the last pair
    put_pair_pos(xp, na, 0.f, 0.f, 0.f);
    xp[8 * (na >> 1) + 7] = 0.f;
  }
  __syncthreads();
  const int tile_n = kEnergyWarps * A.per, shift = 31 - __clz(tile_n);  // a power of two
  const int64_t tiles = (A.N + tile_n - 1) / tile_n;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    for (int j = 0; j < A.per; ++j) {
      const int slot = warp * A.per + j;
      const int64_t n = tile * tile_n + slot;
      if (n >= A.N) break;
      __syncwarp();  // the previous configuration's reads are done
      float mx = 0.f, my = 0.f, mz = 0.f, eg = 0.f, esg = 0.f;
#pragma unroll
      for (int a = 0; a < APL; ++a) {
        const int i = lane + 32 * a;
        if (i >= na) continue;
        const float* src = A.x + (n * na + i) * 3;
        const float x = src[0], y = src[1], z = src[2], q = L.atom_a[i].y;
        xs[i] = make_float4(x, y, z, q);
        put_pair_pos(xp, i, x, y, z);
        xp[8 * (i >> 1) + 6 + (i & 1)] = q;
      }
      __syncwarp();
      float el = bonded_terms<true, false>(L, LL, xs, nullptr, lane, 32);
#pragma unroll
      for (int a = 0; a < APL; ++a) {
        const int i = lane + 32 * a;
        if (i >= na) continue;
        const float4 p = xs[i], pa = L.atom_a[i];
        const float m = L.atom_b[i].z;
        mx += m * p.x;
        my += m * p.y;
        mz += m * p.z;
        const GridOut go = grid_atom(A.G, p.x, p.y, p.z, pa.z, pa.w, pa.y, true, true, 0.f, 0.f);
        eg += go.e_g;
        esg += go.e_sg;
      }
      float e2 = 0.f;
#pragma unroll
      for (int a = 0; a < APL; ++a)
        if (32 * a < na) nonbonded_energy_pass(L, na, 32 * a, xs, xp, e2);
      el += 0.5f * e2;
      Energies en;
      en.lig = el;
      en.sg = esg;
      en.g = eg;
      mx = warp_sumf(mx);
      my = warp_sumf(my);
      mz = warp_sumf(mz);
      en.rest = lane == 0 ? restraint_energy(LL, mx, my, mz) : 0.f;
      double c[4];
      reduce_components(en, c);
      if (lane < 4) {
        const double v = lane == 0 ? c[0] : (lane == 1 ? c[1] : (lane == 2 ? c[2] : c[3]));
        if (A.comps) A.comps[n * 4 + lane] = v;
        s_c[slot][lane] = v;
      }
    }
    if (!A.u_kn) continue;
    __syncthreads();
    for (int e = threadIdx.x; e < tile_n * A.k_count; e += kEnergyWarps * 32) {
      const int k = e >> shift, slot = e & (tile_n - 1);
      const int64_t n = tile * tile_n + slot;
      const StateDev& st = A.states[A.k_begin + k];
      if (n < A.N) A.u_kn[(int64_t)k * A.N + n] = __dmul_rn(st.beta, weighted(s_c[slot], st.w_sg, st.w_g));
    }
    __syncthreads();
  }
}

// u < exp(z), decided by an FP32 exponential where it is clear: at |z| <= 40 that is within 1e-5 of
// exp(z), and an FP64 exponential is some 30 dependent FP64 instructions.
__device__ inline bool below_exp(double u, double z) {
  if (z >= 0.0) return u < 1.0 || u < exp(z);
  if (z > -40.0) {
    const float e = expf((float)z), v = (float)u;
    if (v < 0.9999f * e) return true;
    if (v > 1.0001f * e) return false;
  }
  return u < exp(z);
}

// External-coordinate moves ("Sampling"): for a replica whose state has alpha < alpha_max, n_moves
// moves, each a uniformly random rotation about the centre of mass (the unit quaternion of three
// uniforms by Shoemake's construction) and a Gaussian translation of sigma per dimension, accepted
// by the Metropolis test on the state's energy.  One warp per replica.  A rigid move leaves the
// intramolecular energy unchanged, so U_L is carried over and only the grid terms and the
// restraint of the moved pose are evaluated (both lattices, so all four components stay current).
// Philox counter {d, replica, cycle * n_moves + move, 5}: d = 0 the quaternion's uniforms, d = 1
// the translation (Box-Muller), d = 2 the accept uniform.
struct ExtArgs {
  GridDev G;
  LigandLayout LL;
  const uint32_t* blob;  // the ligand blob in global memory (read through the cache)
  const StateDev* states;
  int n_states;
  int64_t n_rep;
  const int32_t* state_of;
  float* x;
  double* comps;
  int n_moves;
  double alpha_max;
  float sigma;
  uint64_t seed;
  uint64_t cycle;
  int64_t rep_offset;
  int32_t* accepted;
  int64_t* counters;
};

template <int APL>
__global__ void __launch_bounds__(kWarpsPerBlock * 32) external_kernel(const ExtArgs A) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t r = (int64_t)blockIdx.x * kWarpsPerBlock + warp;
  if (r >= A.n_rep) return;
  const int k = A.state_of[r];
  if ((unsigned)k >= (unsigned)A.n_states) return;
  const StateDev st = A.states[k];
  if (!(st.alpha < A.alpha_max)) return;  // also the warming leg's NaN
  const Lig L = bind_ligand(A.blob, A.LL);
  const int na = A.LL.na;
  const uint32_t rid = (uint32_t)(A.rep_offset + r);
  float x[APL][3], sA[APL], sB[APL], q[APL], m[APL];
#pragma unroll
  for (int a = 0; a < APL; ++a) {
    const int i = lane + 32 * a;
    const bool own = i < na;
    const float4 pa = own ? L.atom_a[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    m[a] = own ? L.atom_b[i].z : 0.f;
    q[a] = pa.y;
    sA[a] = pa.z;
    sB[a] = pa.w;
#pragma unroll
    for (int d = 0; d < 3; ++d) x[a][d] = own ? A.x[(r * na + i) * 3 + d] : 0.f;
  }
  double c0[4];
  {
    const double mine = lane < 4 ? A.comps[r * 4 + lane] : 0.0;
#pragma unroll
    for (int c = 0; c < 4; ++c) c0[c] = __shfl_sync(kFull, mine, c);
  }
  const float invM = 1.f / A.LL.total_mass;
  const double u0 = weighted(c0, st.w_sg, st.w_g);
  int n_acc = 0, outside = 0;
  double u_cur = u0;
  // Few replicas take these moves (one of 128 states at paper scale), so a launch waits for one
  // warp's chain of moves.  Out of that chain: the moves' random numbers (one move per lane, 32 at a
  // time), the FP64 exponential, the wait for one pass's lattice loads before the next pass's.  20
  // moves of 64 replicas of 48 atoms: 143 -> 68 us.
  float rot[9], shift_s[2], shift_c[3];  // rotation; the translation's products sigma r and their cosines
  double uni = 0.0;                      // accept uniform
  for (int mv = 0; mv < A.n_moves; ++mv) {
    if ((mv & 31) == 0 && mv + lane < A.n_moves) {
      const uint32_t ctr = (uint32_t)(A.cycle * (uint64_t)A.n_moves + (uint64_t)(mv + lane));
      // rotation
      const U4 rq = philox(A.seed, 0u, rid, ctr, kPurposeExternal);
      const float u1 = (float)(rq.x >> 9) * (1.0f / 8388608.0f);
      const float u2 = (float)(rq.y >> 9) * (1.0f / 8388608.0f);
      const float u3 = (float)(rq.z >> 9) * (1.0f / 8388608.0f);
      const float s1 = sqrtf(1.f - u1), s2 = sqrtf(u1);
      float sn2, cs2, sn3, cs3;
      sincospif(2.f * u2, &sn2, &cs2);
      sincospif(2.f * u3, &sn3, &cs3);
      const float qx = s1 * sn2, qy = s1 * cs2, qz = s2 * sn3, qw = s2 * cs3;
      rot[0] = 1.f - 2.f * (qy * qy + qz * qz), rot[1] = 2.f * (qx * qy - qz * qw), rot[2] = 2.f * (qx * qz + qy * qw);
      rot[3] = 2.f * (qx * qy + qz * qw), rot[4] = 1.f - 2.f * (qx * qx + qz * qz), rot[5] = 2.f * (qy * qz - qx * qw);
      rot[6] = 2.f * (qx * qz - qy * qw), rot[7] = 2.f * (qy * qz + qx * qw), rot[8] = 1.f - 2.f * (qx * qx + qy * qy);
      // translation: Box-Muller on 23-bit uniforms, as for the momenta
      const U4 rt = philox(A.seed, 1u, rid, ctr, kPurposeExternal);
      const float ua = ((float)(rt.x >> 9) + 0.5f) * (1.0f / 8388608.0f), ub = (float)(rt.y >> 9) * (1.0f / 8388608.0f);
      const float uc = ((float)(rt.z >> 9) + 0.5f) * (1.0f / 8388608.0f), ud = (float)(rt.w >> 9) * (1.0f / 8388608.0f);
      float sb, cb, sd_, cd;
      sincospif(2.f * ub, &sb, &cb);
      sincospif(2.f * ud, &sd_, &cd);
      shift_s[0] = A.sigma * sqrtf(-2.f * logf(ua)), shift_s[1] = A.sigma * sqrtf(-2.f * logf(uc));
      shift_c[0] = cb, shift_c[1] = sb, shift_c[2] = cd;
      const U4 ra4 = philox(A.seed, 2u, rid, ctr, kPurposeExternal);
      uni = uniform53(ra4.x, ra4.y);
    }
    const int src = mv & 31;
    const float R00 = __shfl_sync(kFull, rot[0], src), R01 = __shfl_sync(kFull, rot[1], src),
                R02 = __shfl_sync(kFull, rot[2], src), R10 = __shfl_sync(kFull, rot[3], src),
                R11 = __shfl_sync(kFull, rot[4], src), R12 = __shfl_sync(kFull, rot[5], src),
                R20 = __shfl_sync(kFull, rot[6], src), R21 = __shfl_sync(kFull, rot[7], src),
                R22 = __shfl_sync(kFull, rot[8], src);
    const float sab = __shfl_sync(kFull, shift_s[0], src), scd = __shfl_sync(kFull, shift_s[1], src);
    const float tx = sab * __shfl_sync(kFull, shift_c[0], src), ty = sab * __shfl_sync(kFull, shift_c[1], src),
                tz = scd * __shfl_sync(kFull, shift_c[2], src);
    const double u_acc = __shfl_sync(kFull, uni, src);
    // centre of mass, moved pose, its grid terms and restraint
    float cx = 0.f, cy = 0.f, cz = 0.f;
#pragma unroll
    for (int a = 0; a < APL; ++a) {
      cx += m[a] * x[a][0];
      cy += m[a] * x[a][1];
      cz += m[a] * x[a][2];
    }
    cx = warp_sumf(cx) * invM;
    cy = warp_sumf(cy) * invM;
    cz = warp_sumf(cz) * invM;
    float y[APL][3];
    float eg = 0.f, esg = 0.f, mx = 0.f, my = 0.f, mz = 0.f;
    int out_mv = 0;
#pragma unroll
    for (int a = 0; a < APL; ++a) {
      const float vx = x[a][0] - cx, vy = x[a][1] - cy, vz = x[a][2] - cz;
      y[a][0] = cx + (R00 * vx + R01 * vy + R02 * vz) + tx;
      y[a][1] = cy + (R10 * vx + R11 * vy + R12 * vz) + ty;
      y[a][2] = cz + (R20 * vx + R21 * vy + R22 * vz) + tz;
      // without a branch, so that the lattice loads of all passes are in flight together
      const bool own = lane + 32 * a < na;
      const GridOut go = grid_atom(A.G, y[a][0], y[a][1], y[a][2], sA[a], sB[a], q[a], true, true, 0.f, 0.f);
      eg += own ? go.e_g : 0.f;
      esg += own ? go.e_sg : 0.f;
      out_mv += own && go.outside ? 1 : 0;
      mx += m[a] * y[a][0];
      my += m[a] * y[a][1];
      mz += m[a] * y[a][2];
    }
    mx = warp_sumf(mx);
    my = warp_sumf(my);
    mz = warp_sumf(mz);
    const float dx = mx * invM - A.LL.site[0], dy = my * invM - A.LL.site[1], dz = mz * invM - A.LL.site[2];
    const float d = sqrtf(dx * dx + dy * dy + dz * dz);
    float er = 0.f;
    if (d > A.LL.d0) {
      const float ex = d - A.LL.d0;
      er = 0.5f * A.LL.k_rest * ex * ex;
    } else if (!(d <= A.LL.d0)) {
      er = d;
    }
    double c1[4];
    c1[0] = c0[0];
    c1[1] = (double)er;
    // both grid sums over the warp: the butterfly's pairs, one of the two sums per lane
    const bool high = lane & 16;
    double v = (double)(high ? eg : esg) + __shfl_xor_sync(kFull, (double)(high ? esg : eg), 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    c1[2] = __shfl_sync(kFull, v, 0);
    c1[3] = __shfl_sync(kFull, v, 16);
    const double u1e = weighted(c1, st.w_sg, st.w_g);
    const bool acc = below_exp(u_acc, -st.beta * (u1e - u_cur));
    outside += out_mv;
    if (acc) {
#pragma unroll
      for (int a = 0; a < APL; ++a)
#pragma unroll
        for (int dd = 0; dd < 3; ++dd) x[a][dd] = y[a][dd];
#pragma unroll
      for (int c = 0; c < 4; ++c) c0[c] = c1[c];
      u_cur = u1e;
      ++n_acc;
    }
  }
#pragma unroll
  for (int a = 0; a < APL; ++a) {
    const int i = lane + 32 * a;
    if (i < na)
#pragma unroll
      for (int d = 0; d < 3; ++d) A.x[(r * na + i) * 3 + d] = x[a][d];
  }
  if (lane < 4) A.comps[r * 4 + lane] = lane == 0 ? c0[0] : (lane == 1 ? c0[1] : (lane == 2 ? c0[2] : c0[3]));
  if (lane == 0) {
    if (A.accepted) A.accepted[r] += n_acc;
    if (A.counters) {
      if (n_acc) atomicAdd((unsigned long long*)&A.counters[ALGDOCK_CNT_ACCEPTED], (unsigned long long)n_acc);
    }
  }
  if (A.counters) {
    const int out_total = __reduce_add_sync(kFull, outside);
    if (lane == 0 && out_total)
      atomicAdd((unsigned long long*)&A.counters[ALGDOCK_CNT_OUTSIDE], (unsigned long long)out_total);
  }
}

// u_kn[k][n] from stored components (k over k_count states from k_begin).
__global__ void ukn_kernel(const StateDev* __restrict__ states, int k_begin, int k_count, int64_t N,
                           const double* __restrict__ comps, double* u_kn) {
  const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  double c[4];
  const double2 c01 = *(const double2*)(comps + 4 * n), c23 = *(const double2*)(comps + 4 * n + 2);
  c[0] = c01.x;
  c[1] = c01.y;
  c[2] = c23.x;
  c[3] = c23.y;
  for (int k = blockIdx.y; k < k_count; k += gridDim.y) {
    const StateDev st = states[k_begin + k];
    u_kn[(int64_t)k * N + n] = __dmul_rn(st.beta, weighted(c, st.w_sg, st.w_g));
  }
}

int atoms_per_lane(int na) { return na <= 32 ? 1 : (na <= 64 ? 2 : 3); }

size_t block_smem(const LigandLayout& L, int apl, int wpb = kWarpsPerBlock, bool table = false) {
  return ((size_t)(table ? L.words_pair : L.words) + (size_t)wpb * warp_words(L, apl, table)) * 4;
}

constexpr int kTableWarps = 16;  // replicas per block of the pair-table HMC kernel
// Replicas per block of a one-ligand launch, with and without the pair table, by atoms per lane (warps
// per team).  Up to 4 replicas per SM of 33-64 atoms take the kernel with 126 registers instead of 80
// (32 replicas of 48 atoms: 166 us against 193); from there on the one with 24 warps per SM.
constexpr int kTable1 = 5, kTable2 = 6, kTable2Few = 4, kType1 = 16, kType2 = 4, kType3 = 8;
// Two warps a replica, with more replicas than two blocks of kTable2 hold per SM but no more than one of 16
// does: one block of 16 takes them at once, where the two would need a second round for a few.  45 atoms,
// 1900 replicas, 50 steps: 547 -> 401 us (534 with one warp a replica).
constexpr int kTable2Wave = 16;

// Dynamic shared memory of an HMC block of `slots` replicas, and the most of at most `slots` that a
// limit holds (at least one).
size_t team_smem(const LigandLayout& L, int apl, int slots, bool table) {
  return ((size_t)staged_words(L, table) + (size_t)slots * replica_words(L, apl)) * 4;
}
int team_slots(const LigandLayout& L, int apl, int slots, bool table, size_t limit) {
  while (slots > 1 && team_smem(L, apl, slots, table) > limit) --slots;
  return slots;
}

template <typename Kernel, typename Args>
cudaError_t launch_templated(Kernel k1, Kernel k2, Kernel k3, int apl, size_t smem, int64_t items, cudaStream_t s,
                             const Args& A, int wpb = kWarpsPerBlock) {
  Kernel k = apl == 1 ? k1 : (apl == 2 ? k2 : k3);
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxBlockSmem);
  if (e != cudaSuccess) return e;
  const int64_t blocks = (items + wpb - 1) / wpb;
  k<<<(unsigned)blocks, wpb * 32, smem, s>>>(A);
  return cudaGetLastError();
}

}  // namespace

bool hmc_uses_table(const LigandLayout& L) {
  const int apl = atoms_per_lane(L.na);
  return apl <= 2 && block_smem(L, apl, kTableWarps, true) <= kMaxBlockSmem;
}

cudaError_t launch_hmc(cudaStream_t s, const algdock_ctx& c, int64_t n_rep, const int32_t* state_of, float* x,
                       double* comps, double* dH, uint8_t* acc, int n_steps, uint64_t seed, uint64_t cycle,
                       int64_t rep_offset, int64_t* counters) {
  if (n_rep == 0) return cudaSuccess;
  HmcArgs A{c.grid, c.lig, c.d_blob, c.d_states, c.K, n_rep, state_of, x, comps, dH, acc, n_steps, seed,
            (uint32_t)cycle, rep_offset, counters, nullptr, nullptr, 0, nullptr};
  const int apl = atoms_per_lane(c.lig.na);
  // the pair table where a block of 16 replicas can stage it (up to 64 atoms with a small topology);
  // otherwise the pair-type path
  const bool table = hmc_uses_table(c.lig);
  void (*k)(const HmcArgs);
  int most;
  int sms = 0;
  cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c.device);
  if (e != cudaSuccess) return e;
  if (table && apl == 2 && n_rep <= (int64_t)kTable2Few * sms) {
    k = hmc_kernel<2, kTable2Few, true>;
    most = kTable2Few;
  } else if (table && apl == 2 && n_rep > (int64_t)2 * kTable2 * sms && n_rep <= (int64_t)kTable2Wave * sms) {
    k = hmc_kernel<2, kTable2Wave, true>;
    most = kTable2Wave;
  } else if (table) {
    k = apl == 1 ? hmc_kernel<1, kTable1, true, false, 4> : hmc_kernel<2, kTable2, true, false, 2>;
    most = apl == 1 ? kTable1 : kTable2;
  } else {
    k = apl == 1 ? hmc_kernel<1, kType1, false>
                 : (apl == 2 ? hmc_kernel<2, kType2, false, false, 2> : hmc_kernel<3, kType3, false>);
    most = apl == 1 ? kType1 : (apl == 2 ? kType2 : kType3);
  }
  int slots = team_slots(c.lig, apl, most, table, kMaxBlockSmem), per_sm = 0;
  size_t smem = team_smem(c.lig, apl, slots, table);
  e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxBlockSmem);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, slots * apl * 32, smem);
  if (e != cudaSuccess) return e;
  // As many blocks as fit on the device at once.  Replicas that fill their teams once or twice are
  // spread evenly over them; what fills them more than once comes from the work counter.
  const int64_t fit = (int64_t)std::max(per_sm, 1) * sms;
  const int64_t rounds = (n_rep + fit * slots - 1) / (fit * slots);
  if (rounds <= 2) slots = (int)((n_rep + rounds * fit - 1) / (rounds * fit));
  smem = team_smem(c.lig, apl, slots, table);
  if (rounds > 1) {
    A.work = c.d_work;
    e = cudaMemsetAsync(c.d_work, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
  }
  const int64_t blocks = std::min(n_rep, fit);
  const int threads = slots * apl * 32;
  k<<<(unsigned)blocks, threads, smem, s>>>(A);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ multi-ligand batches
size_t batch_block_smem(const LigandLayout& L, int apl, int wpb, bool table) { return block_smem(L, apl, wpb, table); }
size_t batch_team_smem(const LigandLayout& L, int apl, int slots, bool table) {
  return team_smem(L, apl, slots, table);
}

// Launch shapes tried for a class: pair-table blocks of 16 or 8 replicas, or 4-replica blocks
// without the table (classes 0 and 1); 8-replica table blocks or 4 without (2); 4 or 8 replicas
// without the table (3).
int batch_candidates(int cls, int* wpb, bool* table) {
  if (cls == 3) {
    wpb[0] = 4, table[0] = false;
    wpb[1] = 8, table[1] = false;
    return 2;
  }
  if (cls == 2) {
    wpb[0] = 8, table[0] = true;
    wpb[1] = kWarpsPerBlock, table[1] = false;
    return 2;
  }
  wpb[0] = kTableWarps, table[0] = true;
  wpb[1] = 8, table[1] = true;
  wpb[2] = kWarpsPerBlock, table[2] = false;
  return 3;
}

namespace {
using HmcKernel = void (*)(const HmcArgs);
HmcKernel batch_kernel(int apl, int wpb, bool table) {
  if (apl == 1) {
    if (table) return wpb == kTableWarps ? hmc_kernel<1, kTableWarps, true, true> : hmc_kernel<1, 8, true, true>;
    return hmc_kernel<1, kWarpsPerBlock, false, true>;
  }
  if (apl == 2) {
    if (table) return wpb == kTableWarps ? hmc_kernel<2, kTableWarps, true, true> : hmc_kernel<2, 8, true, true>;
    return hmc_kernel<2, kWarpsPerBlock, false, true>;
  }
  return wpb == 8 ? hmc_kernel<3, 8, false, true> : hmc_kernel<3, kWarpsPerBlock, false, true>;
}
}  // namespace

size_t batch_smem_limit(int apl, int wpb, bool table) {
  int dev = 0, optin = 0;
  cudaFuncAttributes fa;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      cudaFuncGetAttributes(&fa, batch_kernel(apl, wpb, table)) != cudaSuccess)
    return 0;
  return (size_t)optin > fa.sharedSizeBytes ? (size_t)optin - fa.sharedSizeBytes : 0;
}

bool batch_uses_table16(const LigandLayout& L) {
  const int apl = atoms_per_lane(L.na);
  return apl <= 2 && block_smem(L, apl, kTableWarps, true) <= batch_smem_limit(apl, kTableWarps, true);
}

cudaError_t batch_set_attributes(const algdock_ctx& c) {
  for (int k = 0; k < kBatchClasses; ++k) {
    const BatchClass& B = c.batch_cls[k];
    if (B.n_items == 0) continue;
    cudaError_t e = cudaFuncSetAttribute(batch_kernel(kClassApl[k], B.wpb, B.table),
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)batch_smem_limit(kClassApl[k], B.wpb, B.table));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// One kernel per class (only_class >= 0: that class alone).  With more than one
// class the launches go to the context's side streams, forked from and joined back to s, so that
// they overlap (and capture into one graph with parallel branches).
cudaError_t launch_hmc_batch(cudaStream_t s, const algdock_ctx& c, const int32_t* state_of, float* x, double* comps,
                             double* dH, uint8_t* acc, int n_steps, uint64_t seed, uint64_t cycle, int64_t rep_offset,
                             int64_t* counters, int only_class) {
  HmcArgs A{c.grid, LigandLayout{}, c.d_batch_blob, c.d_states, c.K, c.batch_n_rep, state_of, x, comps, dH, acc,
            n_steps, seed, (uint32_t)cycle, rep_offset, counters, c.d_batch, nullptr, c.batch_x_stride, nullptr};
  int active[kBatchClasses], n_active = 0;
  for (int k = 0; k < kBatchClasses; ++k)
    if (c.batch_cls[k].n_items > 0 && (only_class < 0 || only_class == k)) active[n_active++] = k;
  if (n_active == 0) return cudaSuccess;
  cudaError_t e = cudaSuccess;
  if (n_active > 1) e = cudaEventRecord(c.batch_fork, s);
  for (int t = 0; t < n_active && e == cudaSuccess; ++t) {
    const int k = active[t];
    const BatchClass& B = c.batch_cls[k];
    cudaStream_t st = s;
    if (n_active > 1) {
      st = c.batch_side[k];
      e = cudaStreamWaitEvent(st, c.batch_fork, 0);
      if (e != cudaSuccess) break;
    }
    A.items = B.d_items;
    batch_kernel(kClassApl[k], B.wpb, B.table)
        <<<(unsigned)B.n_items, B.slots * kClassApl[k] * 32, B.smem, st>>>(A);
    e = cudaGetLastError();
    if (e == cudaSuccess && n_active > 1) {
      e = cudaEventRecord(c.batch_join[k], st);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(s, c.batch_join[k], 0);
    }
  }
  return e;
}

// Components of N configurations (comps, or NULL) and, with u_kn, their reduced energies at k_count
// states from k_begin.
cudaError_t launch_evaluate(cudaStream_t s, const algdock_ctx& c, int64_t N, const float* x, double* comps, int k_begin,
                            int k_count, double* u_kn) {
  if (N == 0) return cudaSuccess;
  const int apl = atoms_per_lane(c.lig.na);
  void (*k)(const EnergyArgs) = apl == 1 ? energy_kernel<1> : (apl == 2 ? energy_kernel<2> : energy_kernel<3>);
  const size_t smem = 4 * ((size_t)staged_words(c.lig, false) + (size_t)kEnergyWarps * 8 * 32 * apl);
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)(kMaxBlockSmem - sizeof(double[kEnergyWarps * kEnergyPer][4])));
  int per_sm = 0, sms = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kEnergyWarps * 32, smem);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c.device);
  if (e != cudaSuccess) return e;
  const int64_t fit = (int64_t)std::max(per_sm, 1) * sms;
  // several configurations per warp (longer rows of u_kn) once every block still has a few tiles
  const int per = N >= 4 * fit * kEnergyWarps * kEnergyPer ? kEnergyPer : 1;
  const int64_t tiles = (N + kEnergyWarps * per - 1) / (kEnergyWarps * per);
  const EnergyArgs A{c.grid, c.lig, c.d_blob, c.d_states, N, per, x, comps, k_count > 0 ? u_kn : nullptr, k_begin,
                     k_count};
  k<<<(unsigned)std::min(tiles, fit), kEnergyWarps * 32, smem, s>>>(A);
  return cudaGetLastError();
}

cudaError_t launch_energy_force(cudaStream_t s, const algdock_ctx& c, int64_t N, const int32_t* state_of,
                                const float* x, float* force, double* comps) {
  if (N == 0) return cudaSuccess;
  EvalArgs A{c.grid, c.lig, c.d_blob, c.d_states, c.K, N, state_of, x, force, comps};
  const int apl = atoms_per_lane(c.lig.na);
  return launch_templated(eval_kernel<1>, eval_kernel<2>, eval_kernel<3>, apl, block_smem(c.lig, apl), N, s, A);
}

cudaError_t launch_external(cudaStream_t s, const algdock_ctx& c, int64_t n_rep, const int32_t* state_of, float* x,
                            double* comps, int n_moves, double alpha_max, float sigma, uint64_t seed, uint64_t cycle,
                            int64_t rep_offset, int32_t* accepted, int64_t* counters) {
  if (n_rep == 0 || n_moves == 0) return cudaSuccess;
  ExtArgs A{c.grid, c.lig, c.d_blob, c.d_states, c.K, n_rep, state_of, x, comps, n_moves, alpha_max, sigma, seed,
            cycle, rep_offset, accepted, counters};
  const int apl = atoms_per_lane(c.lig.na);
  const unsigned blocks = (unsigned)((n_rep + kWarpsPerBlock - 1) / kWarpsPerBlock);
  if (apl == 1) external_kernel<1><<<blocks, kWarpsPerBlock * 32, 0, s>>>(A);
  else if (apl == 2) external_kernel<2><<<blocks, kWarpsPerBlock * 32, 0, s>>>(A);
  else external_kernel<3><<<blocks, kWarpsPerBlock * 32, 0, s>>>(A);
  return cudaGetLastError();
}

cudaError_t launch_ukn(cudaStream_t s, const algdock_ctx& c, int64_t N, const double* comps, int k_begin,
                       int k_count, double* u_kn) {
  if (N == 0 || k_count == 0) return cudaSuccess;
  const int threads = 256;
  dim3 grid((unsigned)((N + threads - 1) / threads), (unsigned)min(k_count, 64));
  ukn_kernel<<<grid, threads, 0, s>>>(c.d_states, k_begin, k_count, N, comps, u_kn);
  return cudaGetLastError();
}

}  // namespace algdock
