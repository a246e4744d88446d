// Device functions of the fused stream-collide update: neighbour addressing,
// the pull stream with the mask's boundary rules, moments, equilibrium, BGK
// and KBC collisions and the exact-difference body force.
//
// All arithmetic is FP32 on deviations df_i = f_i - w_i (rho0 = 1):
//   rho = 1 + sum_i df_i                       (Eq. 6)
//   j   = sum_i c_i df_i, u = j / rho          (Eq. 7; sum_i c_i w_i = 0)
//   df_i^eq = w_i [drho + rho (3 c.u + 4.5 (c.u)^2 - 1.5 u.u)]   (Eq. 5)
#pragma once
#include "lane_math.cuh"
#include "lattice.cuh"
#include "xlb_types.h"

namespace xlb {

enum Collision { COLL_NONE = 0, COLL_BGK = 1, COLL_KBC = 2 };

// Periodic neighbour coordinates of one cell: xo[k] = x + k - 1 wrapped, and
// rb[b][c] = row offset of (y + b - 1, z + c - 1) wrapped.  The source of
// direction i is xo[1 - cx] + rb[1 - cy][1 - cz].  Cell indices are 32-bit
// (the library caps a lattice at 2^31 - 1 cells); plane offsets are 64-bit.
struct Nbr {
  int xo[3];
  int rb[3][3];
};

__device__ __forceinline__ int wrap_m(int v, int n) { return v == 0 ? n - 1 : v - 1; }
__device__ __forceinline__ int wrap_p(int v, int n) { return v == n - 1 ? 0 : v + 1; }

__device__ __forceinline__ void make_nbr(Nbr& nb, int x, int y, int z, int nx, int ny, int nz) {
  nb.xo[0] = wrap_m(x, nx);
  nb.xo[1] = x;
  nb.xo[2] = wrap_p(x, nx);
  const int ys[3] = {wrap_m(y, ny), y, wrap_p(y, ny)};
  const int zs[3] = {nz > 1 ? wrap_m(z, nz) : 0, z, nz > 1 ? wrap_p(z, nz) : 0};
#pragma unroll
  for (int b = 0; b < 3; ++b)
#pragma unroll
    for (int c = 0; c < 3; ++c) nb.rb[b][c] = nx * (ys[b] + ny * zs[c]);
}

template <int Q>
__device__ __forceinline__ int src_index(const Nbr& nb, int i) {
  return nb.xo[1 - Lattice<Q>::c(i, 0)] + nb.rb[1 - Lattice<Q>::c(i, 1)][1 - Lattice<Q>::c(i, 2)];
}

template <int Q>
__device__ __forceinline__ void moments(const float (&df)[Q], float& drho, float (&j)[3]) {
  drho = 0.f;
  j[0] = j[1] = j[2] = 0.f;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    drho += df[i];
    if (Lattice<Q>::c(i, 0)) j[0] += Lattice<Q>::c(i, 0) * df[i];
    if (Lattice<Q>::c(i, 1)) j[1] += Lattice<Q>::c(i, 1) * df[i];
    if (Lattice<Q>::c(i, 2)) j[2] += Lattice<Q>::c(i, 2) * df[i];
  }
}

// Moments of order 0, 1 and 2 of the deviations in one pass over the pairs
// (i, opp(i)): their sum carries the even moments, their difference the odd.
// M = sum_i c_ia c_ib df_i, stored xx yy zz xy xz yz.
template <int Q, typename T>
__device__ __forceinline__ void moments_kbc(const T (&df)[Q], T& drho, T (&j)[3], T (&M)[6]) {
  constexpr int D = Lattice<Q>::D;
  drho = df[0];
  bool fj[3] = {true, true, true}, fm[6] = {true, true, true, true, true, true};
  auto acc = [](T& s, bool& first, int c, T x) {
    s = first ? x : (c > 0 ? vadd(s, x) : vsub(s, x));
    first = false;
  };
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    if (opposite<Q>(i) > i) {
      const T sp = vadd(df[i], df[opposite<Q>(i)]), dm = vsub(df[i], df[opposite<Q>(i)]);
      const int cx = Lattice<Q>::c(i, 0), cy = Lattice<Q>::c(i, 1), cz = D == 3 ? Lattice<Q>::c(i, 2) : 0;
      drho = vadd(drho, sp);
      if (cx) acc(j[0], fj[0], cx, dm);
      if (cy) acc(j[1], fj[1], cy, dm);
      if (cz) acc(j[2], fj[2], cz, dm);
      if (cx) acc(M[0], fm[0], 1, sp);
      if (cy) acc(M[1], fm[1], 1, sp);
      if (cz) acc(M[2], fm[2], 1, sp);
      if (cx * cy) acc(M[3], fm[3], cx * cy, sp);
      if (cx * cz) acc(M[4], fm[4], cx * cz, sp);
      if (cy * cz) acc(M[5], fm[5], cy * cz, sp);
    }
  }
}

// Bracket of Eq. 5 without the leading 1: 3 c.u + 4.5 (c.u)^2 - 1.5 u.u
template <int Q>
__device__ __forceinline__ float eq_poly(int i, const float (&u)[3], float usq) {
  float cu = 0.f;
  if (Lattice<Q>::c(i, 0)) cu += Lattice<Q>::c(i, 0) * u[0];
  if (Lattice<Q>::c(i, 1)) cu += Lattice<Q>::c(i, 1) * u[1];
  if (Lattice<Q>::c(i, 2)) cu += Lattice<Q>::c(i, 2) * u[2];
  return cu * (3.0f + 4.5f * cu) - 1.5f * usq;
}

// Deviations f_i^eq(rho, u) - w_i of an initial state, before storage rounds them.
// Every rounding is spelled out: the kernels that form f_0 (the initialisation and
// the first update, for every storage type) must agree to the bit, or 16-bit storage
// rounds some values apart.
template <int Q>
__device__ __forceinline__ void init_deviations(float rho, const float (&u)[3], float (&df)[Q]) {
  const float usq = __fmaf_rn(u[2], u[2], __fmaf_rn(u[1], u[1], __fmul_rn(u[0], u[0])));
  const float drho = __fsub_rn(rho, 1.0f), b = __fmul_rn(1.5f, usq);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    float cu = 0.f;
#pragma unroll
    for (int a = 0; a < Lattice<Q>::D; ++a)
      if (Lattice<Q>::c(i, a)) cu = __fmaf_rn((float)Lattice<Q>::c(i, a), u[a], cu);
    const float x = __fmaf_rn(cu, __fmaf_rn(4.5f, cu, 3.0f), -b);
    df[i] = __fmul_rn(weight<Q>(i), __fmaf_rn(rho, x, drho));
  }
}

// c_i . u
template <int Q>
__device__ __forceinline__ float cdot(int i, const float (&u)[3]) {
  float cu = 0.f;
  if (Lattice<Q>::c(i, 0)) cu += Lattice<Q>::c(i, 0) * u[0];
  if (Lattice<Q>::c(i, 1)) cu += Lattice<Q>::c(i, 1) * u[1];
  if (Lattice<Q>::c(i, 2)) cu += Lattice<Q>::c(i, 2) * u[2];
  return cu;
}

// Pull: df_i(x) = h_i(x - c_i), periodic (Eq. 2).  Sources on a boundary face
// (StepParams::face) take the rule instead, chosen before any load so that
// each direction is still exactly one load:
//   WALL: h_opp(i)(x);  LID: h_opp(i)(x) + 2 w_i rho_w (c_i . u_w) / cs^2;
//   EQ: f_i^eq(rho_w, u_w) (no load);  FWALL: the plain pull.
// WALL / LID / EQ sources elsewhere hold ghost values (k_boundary).

// Bit i of the result: c_i has component v on the axis (i >= 1).
template <int Q>
__host__ __device__ constexpr uint32_t dir_bits(int axis, int v) {
  uint32_t m = 0;
  for (int i = 1; i < Q; ++i)
    if (Lattice<Q>::c(i, axis) == v) m |= 1u << i;
  return m;
}

// Directions of one cell whose source lies on a boundary face, one bit each:
// they load the cell's own opposite population (own); of those, lid adds the
// moving wall's term and eq takes the equilibrium value.  WALL wins where planes meet,
// then FWALL (a plain pull).
struct FaceDirs {
  uint32_t own, lid, eq;
};

// The directions `at` gives for each face: the source lies on that plane.
__device__ __forceinline__ FaceDirs face_dirs(const StepParams& p, const uint32_t (&at)[6]) {
  uint32_t wall = 0u, fw = 0u, lid = 0u, eq = 0u;
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    // the types are the same for the whole launch
    const int t = p.face[f];
    if (t == WALL) wall |= at[f];
    if (t == FWALL) fw |= at[f];
    if (t == LID) lid |= at[f];
    if (t == EQ) eq |= at[f];
  }
  fw |= wall;
  FaceDirs d;
  d.lid = lid & ~fw;
  d.eq = eq & ~fw;
  d.own = wall | d.lid | d.eq;
  return d;
}

// Rule a source takes, from the three axes' face types of its coordinates:
// WALL wins; then a source on an FWALL plane is pulled plainly (0); else LID
// / EQ (at most one of the two meets; verified on the host).  FW = false
// compiles the form for lattices without FWALL faces.
template <bool FW = true>
__device__ __forceinline__ int face_combine(int a, int b, int c) {
  if (a == WALL || b == WALL || c == WALL) return WALL;
  if (FW && (a == FWALL || b == FWALL || c == FWALL)) return 0;
  return a | b | c;
}

// Full-way bounce-back (Section 3.5): the collision of an FWALL cell sends
// every population back where it came from, f*_i = f_opp(i).
template <int Q>
__device__ __forceinline__ void reverse_populations(float (&df)[Q]) {
#pragma unroll
  for (int i = 1; i < Q; ++i)
    if (i < opposite<Q>(i)) {
      const float t = df[i];
      df[i] = df[opposite<Q>(i)];
      df[opposite<Q>(i)] = t;
    }
}

// Returns, with FW, whether the cell itself lies on an FWALL face plane (its
// own coordinates then count as near a face, so that only warps holding such
// cells evaluate it).
// With `outlet` (a cell of an OUTLET plane x = nx - 1 that copies the pull of
// x - 1 in the directions c_x = -1, nb.xo[2] then being x itself) the face
// rules of those directions take the populations of x - 1.
template <int Q, typename S, bool FW = true>
__device__ __forceinline__ bool pull_periodic(const S* src, const StepParams& p, const Nbr& nb,
                                              int self, int x, int y, int z, float (&df)[Q], bool outlet = false) {
  // next to a face plane, or on it (a superset: its directions follow below)
  bool near_x = false, near_y = false, near_z = false;
  if (p.has_faces) {
    near_x = (p.face[0] | p.face[1]) != 0 && (x <= 1 || x >= p.nx - 2);
    near_y = (p.face[2] | p.face[3]) != 0 && (y <= 1 || y >= p.ny - 2);
    near_z = (p.face[4] | p.face[5]) != 0 && (z <= 1 || z >= p.nz - 2);
  }
  const S* base = src;
  // warp-uniform choice: a warp with no lane next to a face loads plainly;
  // otherwise every lane picks each address branch-free, so either way the
  // warp issues one round of Q independent loads
  if (!__any_sync(__activemask(), near_x || near_y || near_z)) {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      df[i] = Store<S>::ld(base + src_index<Q>(nb, i));
      base += p.plane;
    }
    return false;
  }
  // per face, the directions whose source is on it: a source coordinate v - c
  // equal to the face's
  uint32_t at[6] = {0u, 0u, 0u, 0u, 0u, 0u};
  const int lx = p.nx - 1, ly = p.ny - 1, lz = p.nz - 1;
  if (near_x) {
    const int xm = nb.xo[0], xp = nb.xo[2];  // xp: x + 1, or x itself (outlet)
    at[0] = (xm == 0 ? dir_bits<Q>(0, 1) : 0u) | (x == 0 ? dir_bits<Q>(0, 0) : 0u) | (xp == 0 ? dir_bits<Q>(0, -1) : 0u);
    at[1] = (xm == lx ? dir_bits<Q>(0, 1) : 0u) | (x == lx ? dir_bits<Q>(0, 0) : 0u) | (xp == lx ? dir_bits<Q>(0, -1) : 0u);
  }
  if (near_y) {
    const int ym = wrap_m(y, p.ny), yp = wrap_p(y, p.ny);
    at[2] = (ym == 0 ? dir_bits<Q>(1, 1) : 0u) | (y == 0 ? dir_bits<Q>(1, 0) : 0u) | (yp == 0 ? dir_bits<Q>(1, -1) : 0u);
    at[3] = (ym == ly ? dir_bits<Q>(1, 1) : 0u) | (y == ly ? dir_bits<Q>(1, 0) : 0u) | (yp == ly ? dir_bits<Q>(1, -1) : 0u);
  }
  if (Lattice<Q>::D == 3 && p.nz > 1 && near_z) {
    const int zm = wrap_m(z, p.nz), zp = wrap_p(z, p.nz);
    at[4] = (zm == 0 ? dir_bits<Q>(2, 1) : 0u) | (z == 0 ? dir_bits<Q>(2, 0) : 0u) | (zp == 0 ? dir_bits<Q>(2, -1) : 0u);
    at[5] = (zm == lz ? dir_bits<Q>(2, 1) : 0u) | (z == lz ? dir_bits<Q>(2, 0) : 0u) | (zp == lz ? dir_bits<Q>(2, -1) : 0u);
  }
  const FaceDirs d = face_dirs(p, at);
  // all loads first (addresses chosen branch-free, the two planes of a pair
  // (i, opp(i)) at hand), adjustments after, so the Q loads stay in flight
  // together
  df[0] = Store<S>::ld(src + self);
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    if (opposite<Q>(i) > i) {
      const int k = opposite<Q>(i);
      const S* pi = src + (long long)i * p.plane;
      const S* pk = src + (long long)k * p.plane;
      const bool bi = d.own >> i & 1, bk = d.own >> k & 1;
      const int si = (Lattice<Q>::c(i, 0) == -1 && outlet) ? self - 1 : self;
      const int sk = (Lattice<Q>::c(k, 0) == -1 && outlet) ? self - 1 : self;
      df[i] = Store<S>::ld((bi ? pk : pi) + (bi ? si : src_index<Q>(nb, i)));
      df[k] = Store<S>::ld((bk ? pi : pk) + (bk ? sk : src_index<Q>(nb, k)));
    }
  }
  if (d.lid | d.eq) {
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      if (d.eq >> i & 1) df[i] = p.eq_df[i];
      if (d.lid >> i & 1) df[i] = __fadd_rn(df[i], p.lid_term[i]);
    }
  }
  // where a WALL face meets an FWALL plane the cell is WALL and its slots are
  // never read, so reversing it as well is harmless
  return FW && ((x == 0 && p.face[0] == FWALL) || (x == p.nx - 1 && p.face[1] == FWALL) ||
                (y == 0 && p.face[2] == FWALL) || (y == p.ny - 1 && p.face[3] == FWALL) ||
                (p.nz > 1 && ((z == 0 && p.face[4] == FWALL) || (z == p.nz - 1 && p.face[5] == FWALL))));
}

// Velocity boundaries at INLET cells, with inward normal n = sign e_axis
// (StepParams::inlet_axis / inlet_sign; +x, an inflow, by default; with a
// velocity parallel to the wall they are a moving wall).  The unknown
// populations are those entering the fluid through the boundary, c_i.n = +1.
// The velocity is StepParams::inlet_u, or the cell's entry of
// StepParams::inlet_field (a velocity profile) when that is set.
template <int Q>
__device__ __forceinline__ void inlet_velocity(const StepParams& p, int self, float (&u)[3]) {
  u[0] = p.inlet_u[0];
  u[1] = p.inlet_u[1];
  u[2] = p.inlet_u[2];
  if (p.inlet_field) {
    const long long n = (long long)p.nx * p.ny * p.nz;
    u[0] = p.inlet_field[self];
    u[1] = p.inlet_field[n + self];
    u[2] = Lattice<Q>::D == 3 ? p.inlet_field[2 * n + self] : 0.f;
  }
}

// c_i . n for the inlet normal
template <int Q>
__device__ __forceinline__ int inlet_cn(const StepParams& p, int i) {
  const int c = p.inlet_axis == 0 ? Lattice<Q>::c(i, 0) : (p.inlet_axis == 1 ? Lattice<Q>::c(i, 1) : Lattice<Q>::c(i, 2));
  return p.inlet_sign * c;
}

// rho = [sum_{c.n=0} f_i + 2 sum_{c.n=-1} f_i] / (1 - u.n); in deviations the
// rest parts of the numerator sum to exactly 1.
template <int Q>
__device__ __forceinline__ float inlet_density(const StepParams& p, const float (&df)[Q], const float (&u)[3]) {
  float s = 1.0f;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int cn = inlet_cn<Q>(p, i);
    if (cn == 0) s += df[i];
    if (cn == -1) s += 2.0f * df[i];
  }
  const float un = p.inlet_sign * (p.inlet_axis == 0 ? u[0] : (p.inlet_axis == 1 ? u[1] : u[2]));
  return s / (1.0f - un);
}

// Zou-He: each unknown f_i = f_opp(i) + f_i^eq - f_opp(i)^eq = f_opp(i) + 6 w_i rho (c_i . u).
template <int Q>
__device__ __forceinline__ void zou_he_inlet(const StepParams& p, int self, float (&df)[Q]) {
  float u[3];
  inlet_velocity<Q>(p, self, u);
  const float rho = inlet_density<Q>(p, df, u);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    if (inlet_cn<Q>(p, i) == 1) {
      float cu = Lattice<Q>::c(i, 0) * u[0] + Lattice<Q>::c(i, 1) * u[1];
      if (Lattice<Q>::D == 3) cu += Lattice<Q>::c(i, 2) * u[2];
      df[i] = df[opposite<Q>(i)] + 6.0f * weight<Q>(i) * rho * cu;
    }
  }
}

// Regularized velocity boundary (Latt et al. 2008; the other inflow rule
// Section 4.3 names, and the regularized lid of Section 4.2): rho as for
// Zou-He; non-equilibrium parts of the known populations, those of the
// unknown ones by bounce-back; Pi = sum_i c_i c_i f^neq_i; every population
// becomes f_i = f_i^eq(rho, u) + w_i / (2 cs^4) (c_i c_i - cs^2 I) : Pi.
template <int Q>
__device__ __forceinline__ void regularized_inlet(const StepParams& p, int self, float (&df)[Q]) {
  float u[3];
  inlet_velocity<Q>(p, self, u);
  const float rho = inlet_density<Q>(p, df, u);
  const float usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  // equilibrium deviations f_i^eq - w_i, then the non-equilibrium parts
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const float eqd = weight<Q>(i) * (rho - 1.0f) + weight<Q>(i) * rho * eq_poly<Q>(i, u, usq);
    df[i] -= eqd;  // df now holds f^neq_i
  }
#pragma unroll
  for (int i = 0; i < Q; ++i)
    if (inlet_cn<Q>(p, i) == 1) df[i] = df[opposite<Q>(i)];
  float pxx = 0.f, pyy = 0.f, pzz = 0.f, pxy = 0.f, pxz = 0.f, pyz = 0.f;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const float cx = Lattice<Q>::c(i, 0), cy = Lattice<Q>::c(i, 1), cz = Lattice<Q>::c(i, 2);
    pxx += cx * cx * df[i];
    pyy += cy * cy * df[i];
    pzz += cz * cz * df[i];
    pxy += cx * cy * df[i];
    pxz += cx * cz * df[i];
    pyz += cy * cz * df[i];
  }
  constexpr float cs2 = 1.0f / 3.0f;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const float cx = Lattice<Q>::c(i, 0), cy = Lattice<Q>::c(i, 1), cz = Lattice<Q>::c(i, 2);
    float qpi = (cx * cx - cs2) * pxx + (cy * cy - cs2) * pyy + 2.0f * cx * cy * pxy;
    if (Lattice<Q>::D == 3) qpi += (cz * cz - cs2) * pzz + 2.0f * (cx * cz * pxz + cy * cz * pyz);
    const float eqd = weight<Q>(i) * (rho - 1.0f) + weight<Q>(i) * rho * eq_poly<Q>(i, u, usq);
    df[i] = eqd + 4.5f * weight<Q>(i) * qpi;  // 1 / (2 cs^4) = 4.5
  }
}

// The velocity boundary of an INLET cell, by the chosen scheme.
template <int Q>
__device__ __forceinline__ void inlet_rule(const StepParams& p, int self, float (&df)[Q]) {
  if (p.inlet_regularized)
    regularized_inlet<Q>(p, self, df);
  else
    zou_he_inlet<Q>(p, self, df);
}

// Post-stream populations of a fluid-like or FWALL cell.  The pull applies
// the face rules and reads the ghost values that every other WALL / LID / EQ
// source carries (see k_boundary), i.e. the bounce-back, moving-wall and
// equilibrium rules; INLET cells then rebuild their c_x = +1 populations by
// Zou-He and OUTLET cells copy their c_x = -1 populations from the pull at
// x - 1 (zero-gradient outflow).
template <int Q, typename S>
__device__ __forceinline__ void pull_cell(const S* src, const StepParams& p, int x, int y, int z,
                                          int type, const Nbr& nb, float (&df)[Q]) {
  const int self = x + p.nx * (y + p.ny * z);
  pull_periodic<Q, S>(src, p, nb, self, x, y, z, df);
  if (type == INLET) inlet_rule<Q>(p, self, df);
  if (type == OUTLET) {
    const int xl = wrap_m(x, p.nx);
    Nbr nl;
    make_nbr(nl, xl, y, z, p.nx, p.ny, p.nz);
    float dl[Q];
    pull_periodic<Q, S>(src, p, nl, self - x + xl, xl, y, z, dl);
#pragma unroll
    for (int i = 0; i < Q; ++i)
      if (Lattice<Q>::c(i, 0) == -1) df[i] = dl[i];
  }
}

// The collision code below walks the rest direction and the pairs
// (i, opp(i)), i < opp(i): with a = 3 c_i.u and b = 4.5 (c_i.u)^2 - 1.5 u.u
// the bracket of Eq. 5 is b + a for i and b - a for opp(i), and every even
// function of c (the KBC shear part, the second moments) is shared.

// c_i . u, i < opp(i): the first non-zero component is +1
template <int Q, typename T>
__device__ __forceinline__ T vdot(int i, const T (&u)[3]) {
  const int cx = Lattice<Q>::c(i, 0), cy = Lattice<Q>::c(i, 1), cz = Lattice<Q>::D == 3 ? Lattice<Q>::c(i, 2) : 0;
  T s = cx ? u[0] : (cy ? u[1] : u[2]);
  if (cx && cy) s = cy > 0 ? vadd(s, u[1]) : vsub(s, u[1]);
  if ((cx || cy) && cz) s = cz > 0 ? vadd(s, u[2]) : vsub(s, u[2]);
  return s;
}

template <int Q, typename T>
__device__ __forceinline__ T vnorm2(const T (&u)[3]) {
  const T s = vfma(u[0], u[0], vmul(u[1], u[1]));
  return Lattice<Q>::D == 3 ? vfma(u[2], u[2], s) : s;
}

// Exact-difference body force: df_i += f_i^eq(rho, u + F/rho) - f_i^eq(rho, u).
template <int Q, typename T>
__device__ __forceinline__ void add_force(T (&df)[Q], T rho, T ir, const T (&u)[3], T usq, const float (&F)[3]) {
  T v[3];
#pragma unroll
  for (int a = 0; a < Lattice<Q>::D; ++a) v[a] = vfma(vset<T>(F[a]), ir, u[a]);
  const T dsq = vmul(vset<T>(-1.5f), vsub(vnorm2<Q>(v), usq));
  df[0] = vfma(vmul(vset<T>(weight<Q>(0)), rho), dsq, df[0]);
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    if (opposite<Q>(i) > i) {
      const T cu = vdot<Q>(i, u), cv = vdot<Q>(i, v);
      const T e = vfma(vset<T>(4.5f), vfma(cv, cv, vmul(vneg(cu), cu)), dsq), o = vsub(cv, cu);
      const T wr = vmul(vset<T>(weight<Q>(i)), rho);
      df[i] = vfma(wr, vfma(vset<T>(3.0f), o, e), df[i]);
      df[opposite<Q>(i)] = vfma(wr, vfma(vset<T>(-3.0f), o, e), df[opposite<Q>(i)]);
    }
  }
}

// BGK (Eq. 3) on one cell (T = float) or two (T = F2), in place on deviations:
// df_i += omega (df_i^eq - df_i), then the body force.
template <int Q, typename T>
__device__ __forceinline__ void collide_bgk(T (&df)[Q], const StepParams& p) {
  T drho = df[0], j[3];
#pragma unroll
  for (int i = 1; i < Q; ++i) drho = vadd(drho, df[i]);
#pragma unroll
  for (int a = 0; a < Lattice<Q>::D; ++a) {
    bool first = true;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      const int c = Lattice<Q>::c(i, a);
      if (c == 0) continue;
      j[a] = first ? df[i] : (c > 0 ? vadd(j[a], df[i]) : vsub(j[a], df[i]));
      first = false;
    }
  }
  const T rho = vadd(vset<T>(1.0f), drho);
  const T ir = vrcp(rho);
  T u[3];
#pragma unroll
  for (int a = 0; a < Lattice<Q>::D; ++a) u[a] = vmul(j[a], ir);
  const T usq = vnorm2<Q>(u);
  const T b0 = vmul(vset<T>(-1.5f), usq);  // b of the rest direction (c = 0)
  // df + omega (w x - df) as df - omega (df - w x), the same value
  const T nom = vset<T>(-p.omega);
  df[0] = vfma(nom, vfma(vset<T>(-weight<Q>(0)), vfma(rho, b0, drho), df[0]), df[0]);
  const T r3 = vmul(rho, vset<T>(3.0f)), n3 = vneg(r3);
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    if (opposite<Q>(i) > i) {
      const int k = opposite<Q>(i);
      const T cu = vdot<Q>(i, u);
      const T bb = vfma(rho, vfma(vmul(vset<T>(4.5f), cu), cu, b0), drho);
      const T nw = vset<T>(-weight<Q>(i));
      df[i] = vfma(nom, vfma(nw, vfma(r3, cu, bb), df[i]), df[i]);
      df[k] = vfma(nom, vfma(nw, vfma(n3, cu, bb), df[k]), df[k]);
    }
  }
  if (p.has_force) add_force<Q>(df, rho, ir, u, usq, p.F);
}

// KBC shear population ds_i, i < opp(i), from hd = D_aa / 2 (a = x, y, z) and
// qo = Pi_ab / 4 (ab = xy, xz, yz) and their negatives nqo; directions with
// one or two non-zero components (it is zero on the others).
template <int Q, typename T>
__device__ __forceinline__ T kbc_ds(int i, const T (&hd)[3], const T (&qo)[3], const T (&nqo)[3]) {
  const int cx = Lattice<Q>::c(i, 0), cy = Lattice<Q>::c(i, 1), cz = Lattice<Q>::D == 3 ? Lattice<Q>::c(i, 2) : 0;
  if (nnz<Q>(i) == 1) return cx ? hd[0] : (cy ? hd[1] : hd[2]);
  const int k = cx && cy ? 0 : (cx && cz ? 1 : 2), c = cx && cy ? cx * cy : (cx && cz ? cx * cz : cy * cz);
  return c > 0 ? qo[k] : nqo[k];
}

// KBC (Karlin, Bosch, Chikatamarla 2014) on one cell (T = float) or two
// (T = F2): f^neq = ds + dh, beta = omega / 2,
//   gamma = 1/beta - (2 - 1/beta) <ds|dh> / <dh|dh>,  <a|b> = sum a_i b_i / f_i^eq,
//   f_i <- f_i - beta (2 ds_i + gamma dh_i)
// where ds carries the deviatoric second moments of f^neq on the natural
// moment basis: ds_i = D_aa / 2 for c_i = +-e_a, ds_i = c_ia c_ib Pi_ab / 4
// for c_i with two non-zero components a, b, and 0 otherwise
// (D_aa = Pi_aa - tr(Pi) / d).
// The second moments of f^neq come from those of the deviations (moments_kbc)
// and the closed form of the equilibrium's: on these lattices
// sum_i c_ia c_ib f_i^eq = rho (d_ab / 3 + u_a u_b), so
//   P_ab = M_ab - rho u_a u_b - d_ab drho / 3.
// One pass then turns df into f^neq and forms <ds|dh> and <dh|dh>, with
// dh = f^neq - ds; with them the update reads
//   df_i <- df_i^eq + (1 - beta gamma) f^neq_i - beta (2 - gamma) ds_i.
template <int Q, typename T>
__device__ __forceinline__ void collide_kbc(T (&df)[Q], const StepParams& p) {
  constexpr int D = Lattice<Q>::D;
  T drho, j[3], M[6];
  moments_kbc<Q>(df, drho, j, M);
  const T rho = vadd(vset<T>(1.0f), drho), ir = vrcp(rho);
  T u[3];
#pragma unroll
  for (int a = 0; a < D; ++a) u[a] = vmul(j[a], ir);
  const T usq = vnorm2<Q>(u);
  const T b0 = vmul(vset<T>(-1.5f), usq);  // b of the rest direction (c = 0)
  const T nrho = vneg(rho);
  T nru[3], P[3], S;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    nru[a] = vmul(nrho, u[a]);
    P[a] = vfma(drho, vset<T>(-1.0f / 3.0f), vfma(nru[a], u[a], M[a]));
    S = a == 0 ? P[0] : vadd(S, P[a]);
  }
  T hd[3], qo[3], nqo[3];
#pragma unroll
  for (int a = 0; a < D; ++a) hd[a] = vmul(vset<T>(0.5f), vfma(S, vset<T>(-1.0f / D), P[a]));
#pragma unroll
  for (int k = 0; k < (D == 3 ? 3 : 1); ++k) {
    const int a = k == 2 ? 1 : 0, b = k == 0 ? 1 : 2;
    qo[k] = vmul(vset<T>(0.25f), vfma(nru[a], u[b], M[3 + k]));
    nqo[k] = vneg(qo[k]);
  }
  // <a|b> = sum a_i b_i / f_i^eq with f_i^eq = w_i rho (1 + b +- a); the
  // common 1/rho cancels in gamma, and one reciprocal serves a pair:
  // 1 / (X +- a) = (X -+ a) / (X^2 - a^2).  The rest direction has ds = 0.
  const T e0 = vmul(vset<T>(weight<Q>(0)), vfma(rho, b0, drho));
  df[0] = vsub(df[0], e0);
  T hh = vmul(vmul(df[0], df[0]),
              vdiv_fast(vset<T>(1.0f / weight<Q>(0)), vadd(vset<T>(1.0f), b0)));
  T sh = vset<T>(0.0f);
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    if (opposite<Q>(i) > i) {
      const int k = opposite<Q>(i);
      const T cu = vdot<Q>(i, u), nw = vset<T>(-weight<Q>(i));
      const T bq = vfma(vmul(vset<T>(4.5f), cu), cu, b0), a3 = vmul(vset<T>(3.0f), cu);
      const T bb = vfma(rho, bq, drho);
      const T fi = vfma(nw, vfma(rho, a3, bb), df[i]), fk = vfma(nw, vfma(nrho, a3, bb), df[k]);
      df[i] = fi;
      df[k] = fk;
      const T X = vadd(vset<T>(1.0f), bq);
      const T rc = vdiv_fast(vset<T>(1.0f / weight<Q>(i)), vfma(X, X, vmul(vneg(a3), a3)));
      const T ri = vmul(vsub(X, a3), rc), rk = vmul(vadd(X, a3), rc);
      T hi = fi, hk = fk;
      if (nnz<Q>(i) < 3) {
        const T s = kbc_ds<Q>(i, hd, qo, nqo);
        hi = vsub(fi, s);
        hk = vsub(fk, s);
        sh = vfma(s, vfma(hi, ri, vmul(hk, rk)), sh);
      }
      hh = vfma(vmul(hi, hi), ri, vfma(vmul(hk, hk), rk, hh));
    }
  }
  const float beta = 0.5f * p.omega, ib = 1.0f / beta;
  // (a uniform stream takes no division: 0 / 0 cost the FP32 / FP16 sphere from
  // rest 3% / 4% of an update, and a harmless divisor chosen instead 1% of any)
  const T gamma = vsub_div_unless_less(vset<T>(2.0f), ib, vmul(vset<T>(2.0f - ib), sh), hh,
                                       vmul(vset<T>(1e-20f), rho));
  const T a1 = vfma(vset<T>(-beta), gamma, vset<T>(1.0f));
  const T na2 = vmul(vset<T>(-beta), vsub(vset<T>(2.0f), gamma));
  df[0] = vfma(a1, df[0], e0);
  const T r3 = vmul(rho, vset<T>(3.0f)), n3 = vneg(r3);
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    if (opposite<Q>(i) > i) {
      const int k = opposite<Q>(i);
      const T cu = vdot<Q>(i, u), w = vset<T>(weight<Q>(i));
      const T bb = vfma(rho, vfma(vmul(vset<T>(4.5f), cu), cu, b0), drho);
      T si = vmul(a1, df[i]), sk = vmul(a1, df[k]);
      if (nnz<Q>(i) < 3) {
        const T nsd = vmul(na2, kbc_ds<Q>(i, hd, qo, nqo));
        si = vfma(a1, df[i], nsd);
        sk = vfma(a1, df[k], nsd);
      }
      df[i] = vfma(w, vfma(r3, cu, bb), si);
      df[k] = vfma(w, vfma(n3, cu, bb), sk);
    }
  }
  if (p.has_force) add_force<Q>(df, rho, ir, u, usq, p.F);
}

// Collision C of Eq. 1 on one fluid-like cell, in place on deviations.
template <int Q, int COLL, typename T>
__device__ __forceinline__ void collide(T (&df)[Q], const StepParams& p) {
  if constexpr (COLL == COLL_BGK) collide_bgk<Q>(df, p);
  if constexpr (COLL == COLL_KBC) collide_kbc<Q>(df, p);
}

}  // namespace xlb
