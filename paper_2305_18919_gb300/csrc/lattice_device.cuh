// Lattice-Boltzmann passes, device code: the fused pull stream-collide over the whole lattice (Eqs. 9-10
// with Guo forcing and half-way bounce-back), the velocity gather at the active interface
// tiles (the velocity step of Sec. III), and the read-back / initialisation helpers.
//
// Populations are stored as deviations f_i - w_i rho0 ("shifted"), structure of arrays
// [19][nz][ny][nx] with x fastest. The state array holds post-collision populations of
// the previous step; a pull reads f_i(x - c_i) from it, which is the streaming step.
// Right after initialisation the state holds post-streaming populations ("fresh") and the
// first collision reads them in place. The storage type S may be narrower than the
// arithmetic type `real` (FP16 / BF16 storage with FP32 arithmetic), see Storage below.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <string.h>

#include <cmath>
#include <type_traits>

#include "iblb_internal.cuh"

#ifndef IBLB_RO
#define IBLB_RO __restrict__
#endif

namespace iblb {
namespace {

// Coefficients of the collision (see collide below), formed on the host in double and rounded
// once: la, ld (momentum), ba, bd, b0 (density and trace) and qa, qd (second order) of the axis,
// diagonal and rest directions.
template <typename real>
struct CollideCoef {
  real omc, nom;      // 1 - omega, -omega
  real la, ld;        // 3 w omega
  real ba, bd, b0;    // w omega
  real qa, qd;        // 4.5 w omega
  real m0, ma, md;    // weights of stored populations in the moments (16-bit storage)
  real Fh[3];         // g/2:            u = (j + g/2)/rho
  real Kc[3];         // (2 tau - 1/2) g: K = j + (2 tau - 1/2) g
  real Lc[3];         // g/omega:        L = j + g/omega
  real ga[3], gd[3];  // 3 w g of the axis and diagonal directions (FP32, see collide)
};

// Coefficients of the active-tile correction (in the arithmetic's units, see Correction).
template <typename real>
struct CorrectionCoef {
  real ba, bd, b0, qa, qd;  // as in CollideCoef
  real la, ld;              // 3 w
  real kappa;               // 2 tau - 1/2
  real Gh[3];               // g/2:              u0 = (J - g/2)/rho
  real Kt[3];               // (2 tau - 3/2) g:  K0 = J + (2 tau - 3/2) g
};

template <typename real>
struct LatParams {
  int nx, ny, nz, has_walls;
  int ntx, nty;
  size_t ncell;
  real rho0;
  real g[3];         // uniform body force
  real wb[19];       // 6 w_i rho0 (c_i . u_bottom): moving-wall term, bottom wall
  real wt[19];       // same for the top wall
  CollideCoef<real> cc;
  CorrectionCoef<real> ct;
};

// The collision's coefficients. Rounding them one by one would make the collision gain or lose
// mass and momentum in proportion to the state, step after step; so the ones that are free are
// taken from the ones already rounded, such that the sums over the 19 directions come out:
//   sum of the momentum terms  2 la + 8 ld = om,   sum of the density terms 6 ba + 12 bd + b0 = om
// exactly, with om the relaxation rate that the f term applies (FP32: f - om f with om as
// rounded; FP64 and 16-bit storage: (1 - om) f, om = 1 - (1 - om as rounded)): ld and bd are
// taken as multiples of an eighth of om's last place, which leaves la and b0 representable.
// `scale` is 0 for plain storage, else K of the 16-bit units g_i = (f_i - w_i rho0) K / w_i,
// where the weights cancel.
template <typename real>
CollideCoef<real> collide_coef(const Ctx &c, double scale) {
  CollideCoef<real> k;
  const double tau = c.tau;
  k.nom = (real)(-1.0 / tau);
  k.omc = (real)(1.0 - 1.0 / tau);
  const bool delta = sizeof(real) == 4 && scale == 0.0;  // f - om f (see collide)
  double om = delta ? -(double)k.nom : 1.0 - (double)k.omc;
  if (!(om > 0.0)) om = 1.0 / tau;  // 1/tau below the last place of 1: the f term keeps all of f
  if (scale != 0.0) {
    k.la = k.ld = (real)(3.0 * scale * om);
    k.ba = k.bd = k.b0 = (real)(scale * om);
    k.qa = k.qd = (real)(4.5 * scale * om);
    k.m0 = (real)(1.0 / (3.0 * scale));
    k.ma = (real)(1.0 / (18.0 * scale));
    k.md = (real)(1.0 / (36.0 * scale));
  } else {
    const double step = std::ldexp(1.0, std::ilogb(om) - (sizeof(real) == 4 ? 23 : 52) - 3);
    k.ld = (real)(std::rint(om / 12.0 / step) * step);
    k.la = (real)((om - 8.0 * (double)k.ld) / 2.0);
    k.bd = (real)(std::rint(om / 36.0 / step) * step);
    k.ba = (real)(2.0 * (double)k.bd);
    k.b0 = (real)(om - 24.0 * (double)k.bd);
    k.qd = (real)(om / 8.0);
    k.qa = (real)(2.0 * (double)k.qd);
    k.m0 = k.ma = k.md = (real)1;
  }
  for (int a = 0; a < 3; a++) {
    k.Fh[a] = (real)(0.5 * c.g[a]);
    k.Kc[a] = (real)((2.0 * tau - 0.5) * c.g[a]);
    k.Lc[a] = (real)(c.g[a] / om);
    k.ga[a] = (real)(c.g[a] / 6.0);
    k.gd[a] = (real)(c.g[a] / 12.0);
  }
  return k;
}

template <typename real>
CorrectionCoef<real> correction_coef(const Ctx &c) {
  CorrectionCoef<real> k;
  const double om = 1.0 / c.tau;
  k.bd = (real)(om / 36.0);
  k.ba = (real)(om / 18.0);
  k.b0 = (real)(om / 3.0);
  k.qd = (real)(om / 8.0);
  k.qa = (real)(om / 4.0);
  k.ld = (real)(1.0 / 12.0);
  k.la = (real)(1.0 / 6.0);
  k.kappa = (real)(2.0 * c.tau - 0.5);
  for (int a = 0; a < 3; a++) {
    k.Gh[a] = (real)(0.5 * c.g[a]);
    k.Kt[a] = (real)((2.0 * c.tau - 1.5) * c.g[a]);
  }
  return k;
}

template <typename real>
LatParams<real> lat_params(const Ctx &c) {
  LatParams<real> p;
  p.nx = c.nx; p.ny = c.ny; p.nz = c.nz; p.has_walls = c.has_walls;
  p.ntx = c.ntx; p.nty = c.nty;
  p.ncell = c.ncell;
  p.rho0 = (real)c.rho0;
  for (int k = 0; k < 3; k++) p.g[k] = (real)c.g[k];
  for (int i = 0; i < Q; i++) {
    double cb = cx(i) * c.ub[0] + cy(i) * c.ub[1] + cz(i) * c.ub[2];
    double ct = cx(i) * c.ut[0] + cy(i) * c.ut[1] + cz(i) * c.ut[2];
    p.wb[i] = (real)(6.0 * wgt(i) * c.rho0 * cb);
    p.wt[i] = (real)(6.0 * wgt(i) * c.rho0 * ct);
  }
  p.cc = collide_coef<real>(c, c.precision == IBLB_FP16 ? 1024.0 : c.precision == IBLB_BF16 ? 1.0 : 0.0);
  p.ct = correction_coef<real>(c);
  return p;
}

// n / d for 0 <= n < 2^31 and a fixed d >= 1, by one multiplication (d >= 2): with 2^(l-1) < d <= 2^l and
// m = floor(2^(31+l) / d) + 1 (below 2^32), m d exceeds 2^(31+l) by at most 2^l, which shifts
// n m / 2^(31+l) from n / d by less than 1 / d: the floor is the same.
struct FastDiv {
  unsigned m;
  int shift;
  int d;
  __device__ __forceinline__ int div(int n) const {
    return d == 1 ? n : (int)(__umulhi((unsigned)n, m) >> shift);
  }
};
FastDiv fast_div(int d) {
  int l = 1;
  while ((1ll << l) < d) l++;
  FastDiv f;
  f.m = (unsigned)(((1ull << (31 + l)) / (unsigned)d) + 1ull);
  f.shift = l - 1;
  f.d = d;
  return f;
}

// Node groups of the fluid layers in memory order (a group: the nodes of one thread).
struct FlatGroups {
  FastDiv per_row, ny;  // groups per lattice row, rows per layer
  int n;                // groups in all
  __device__ __forceinline__ void at(int g, int &gx, int &y, int &z) const {
    const int row = per_row.div(g);
    gx = g - row * per_row.d;
    z = ny.div(row);
    y = row - z * ny.d;
  }
};
FlatGroups flat_groups(int per_row, int ny, int layers) {
  return FlatGroups{fast_div(per_row), fast_div(ny), per_row * ny * layers};
}

// Storage of the shifted populations. Population i is stored as g_i = (f_i - w_i rho0) k_i
// in type S and used as f_i - w_i rho0 in type `real`. For float and double k_i = 1. For the
// 16-bit types (arithmetic stays FP32) k_i = K / w_i: the deviations of the 19 directions
// then share one scale, about |drho| + 3 |c.u|, and with K = 1024 the FP16 values sit well
// inside its normal range (6.1e-5 .. 65504), so each keeps FP16's 11-bit significand. BF16
// has FP32's exponent range and needs no shift (K = 1).
template <typename S>
struct Storage;
template <>
struct Storage<double> {
  using V2 = double2;
  static constexpr double K = 0.0;  // 0: stored unscaled
};
template <>
struct Storage<float> {
  using V2 = float2;
  static constexpr double K = 0.0;
};
template <>
struct Storage<__half> {
  using V2 = __half2;
  static constexpr double K = 1024.0;
};
template <>
struct Storage<__nv_bfloat16> {
  using V2 = __nv_bfloat162;
  static constexpr double K = 1.0;
};

// k_i and 1 / k_i
template <typename S>
__host__ __device__ constexpr double kscale(int i) {
  return Storage<S>::K == 0.0 ? 1.0 : Storage<S>::K / wgt(i);
}
template <typename S>
__host__ __device__ constexpr double kinv(int i) {
  return Storage<S>::K == 0.0 ? 1.0 : wgt(i) / Storage<S>::K;
}

__device__ __forceinline__ float widen(float v) { return v; }
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ float widen(__half v) { return __half2float(v); }
__device__ __forceinline__ float widen(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ void widen2(float2 v, float &a, float &b) { a = v.x; b = v.y; }
__device__ __forceinline__ void widen2(double2 v, double &a, double &b) { a = v.x; b = v.y; }
__device__ __forceinline__ void widen2(__half2 v, float &a, float &b) {
  a = __low2float(v);
  b = __high2float(v);
}
__device__ __forceinline__ void widen2(__nv_bfloat162 v, float &a, float &b) {
  a = __low2float(v);
  b = __high2float(v);
}

// Rounding of `real` values to the storage type (round to nearest even).
template <typename S>
struct Narrow;
template <>
struct Narrow<float> {
  __device__ static float one(float v) { return v; }
  __device__ static float2 two(float a, float b) { return make_float2(a, b); }
};
template <>
struct Narrow<double> {
  __device__ static double one(double v) { return v; }
  __device__ static double2 two(double a, double b) { return make_double2(a, b); }
};
template <>
struct Narrow<__half> {
  __device__ static __half one(float v) { return __float2half_rn(v); }
  __device__ static __half2 two(float a, float b) { return __floats2half2_rn(a, b); }
};
template <>
struct Narrow<__nv_bfloat16> {
  __device__ static __nv_bfloat16 one(float v) { return __float2bfloat16_rn(v); }
  __device__ static __nv_bfloat162 two(float a, float b) { return __floats2bfloat162_rn(a, b); }
};

// The deviation f_i - w_i rho0 stored at element `idx` of array p (population i).
template <typename real, typename S>
__device__ __forceinline__ real dev(const S *IBLB_RO p, int i, size_t idx) {
  return real(widen(p[idx])) * real(kinv<S>(i));
}

// Loads of the shell-velocity pass, whose pulled rows are scattered over the lattice: the
// prefetch-size qualifier bounds each L2 fill from DRAM to 64 bytes (a plain load brings a
// whole 128-byte line for a 4-byte access). The pass runs beside the full-lattice pass, which
// gets the DRAM bandwidth saved (256^3: 23.6 MB against 37.4 MB per launch).
#define IBLB_SCATTER_LD "ld.global.L2::64B"
#ifndef IBLB_SCATTER_ASM
#define IBLB_SCATTER_ASM asm
#endif
__device__ __forceinline__ float ld_scattered(const float *p) {
  float v;
  IBLB_SCATTER_ASM(IBLB_SCATTER_LD ".f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ double ld_scattered(const double *p) {
  double v;
  IBLB_SCATTER_ASM(IBLB_SCATTER_LD ".f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ __half ld_scattered(const __half *p) {
  unsigned short v;
  IBLB_SCATTER_ASM(IBLB_SCATTER_LD ".b16 %0, [%1];" : "=h"(v) : "l"(p));
  return __ushort_as_half(v);
}
__device__ __forceinline__ __nv_bfloat16 ld_scattered(const __nv_bfloat16 *p) {
  unsigned short v;
  IBLB_SCATTER_ASM(IBLB_SCATTER_LD ".b16 %0, [%1];" : "=h"(v) : "l"(p));
  return __ushort_as_bfloat16(v);
}
__device__ __forceinline__ float2 ld_scattered(const float2 *p) {
  float2 v;
  IBLB_SCATTER_ASM(IBLB_SCATTER_LD ".v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ double2 ld_scattered(const double2 *p) {
  double2 v;
  IBLB_SCATTER_ASM(IBLB_SCATTER_LD ".v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ __half2 ld_scattered(const __half2 *p) {
  unsigned v;
  IBLB_SCATTER_ASM(IBLB_SCATTER_LD ".b32 %0, [%1];" : "=r"(v) : "l"(p));
  __half2 h;
  memcpy(&h, &v, sizeof(v));
  return h;
}
__device__ __forceinline__ __nv_bfloat162 ld_scattered(const __nv_bfloat162 *p) {
  unsigned v;
  IBLB_SCATTER_ASM(IBLB_SCATTER_LD ".b32 %0, [%1];" : "=r"(v) : "l"(p));
  __nv_bfloat162 h;
  memcpy(&h, &v, sizeof(v));
  return h;
}

// dev() through ld_scattered
template <typename real, typename S>
__device__ __forceinline__ real dev_scattered(const S *IBLB_RO p, int i, size_t idx) {
  return real(widen(ld_scattered(p + idx))) * real(kinv<S>(i));
}

// Single roundings that the compiler does not fuse, so that every kernel that collides a node
// gives the same bits.
__device__ __forceinline__ float add_(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_(double a, double b) { return __dmul_rn(a, b); }

// Pull the 19 post-streaming populations of fluid node (x, y, z) from post-collision array
// `fp`. A link whose source is a wall node is bounced back: the opposite post-collision
// population of the same node plus the moving-wall term.
template <typename real, typename S, bool SCATTERED = false>
__device__ __forceinline__ void pull(const S *IBLB_RO fp, const LatParams<real> &P, int x,
                                     int y, int z, real f[Q]) {
  const int xm = x == 0 ? P.nx - 1 : x - 1, xp = x == P.nx - 1 ? 0 : x + 1;
  const int ym = y == 0 ? P.ny - 1 : y - 1, yp = y == P.ny - 1 ? 0 : y + 1;
  int zm = z - 1, zp = z + 1;
  if (!P.has_walls) {
    zm = z == 0 ? P.nz - 1 : zm;
    zp = z == P.nz - 1 ? 0 : zp;
  }
  const bool wall_below = P.has_walls && zm == 0;
  const bool wall_above = P.has_walls && zp == P.nz - 1;
  const size_t plane = (size_t)P.nx * P.ny;
  // source offsets along each axis, indexed by 1 - c (c = +1 -> minus side, c = -1 -> plus side)
  const size_t zo[3] = {(size_t)zm * plane, (size_t)z * plane, (size_t)zp * plane};
  const size_t yo[3] = {(size_t)ym * P.nx, (size_t)y * P.nx, (size_t)yp * P.nx};
  const int xo[3] = {xm, x, xp};
  const size_t n = zo[1] + yo[1] + x;
#pragma unroll
  for (int i = 0; i < Q; i++) {
    // (opposite directions have the same weight, so population i's scale serves both)
    const bool bounce = (cz(i) > 0 && wall_below) || (cz(i) < 0 && wall_above);
    const size_t idx = bounce ? (size_t)opp(i) * P.ncell + n
                              : (size_t)i * P.ncell + zo[1 - cz(i)] + yo[1 - cy(i)] + xo[1 - cx(i)];
    f[i] = SCATTERED ? dev_scattered<real>(fp, i, idx) : dev<real>(fp, i, idx);
    if (bounce) f[i] = add_(f[i], cz(i) > 0 ? P.wb[i] : P.wt[i]);
  }
}

// Force density (body force and interface) of the node pair (x0, x0 + 1) from the active-tile
// table; the two nodes lie in one tile.
template <typename real>
__device__ __forceinline__ void tile_force_pair(const int *IBLB_RO tile_slot,
                                                const Vec4<real> *IBLB_RO Fslot,
                                                const LatParams<real> &P, int x0, int y, int z,
                                                real Fa[3], real Fb[3]) {
#pragma unroll
  for (int k = 0; k < 3; k++) Fa[k] = Fb[k] = P.g[k];
  if (tile_slot == nullptr) return;
  const int s = tile_slot[((z >> 2) * P.nty + (y >> 2)) * P.ntx + (x0 >> 2)];
  if (s < 0) return;
  const Vec4<real> *F = Fslot + (size_t)s * TILE_CELLS + (x0 & 3) + 4 * (y & 3) + 16 * (z & 3);
  const Vec4<real> fa = F[0], fb = F[1];
  Fa[0] += fa.x;
  Fa[1] += fa.y;
  Fa[2] += fa.z;
  Fb[0] += fb.x;
  Fb[1] += fb.y;
  Fb[2] += fb.z;
}

__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }

// 1/a and 1/b of two nodes' densities. FP64 divides cost an order of magnitude more than an
// FP64 multiply-add, so the two share one reciprocal, 1/(ab), by Newton's iteration
// r <- r + r (1 - x r) from a float seed (relative error 2^-23, then 2^-46, then rounding);
// outside the seed's range they are plain divisions. u enters the collision only at second order.
__device__ __forceinline__ float reciprocal(float a) { return 1.0f / a; }
__device__ __forceinline__ double reciprocal(double a) {
  const float s = (float)a;
  if (!(s > 1e-30f && s < 1e30f)) return 1.0 / a;
  double r = (double)(1.0f / s);
  r = fma(r, fma(-a, r, 1.0), r);
  return fma(r, fma(-a, r, 1.0), r);
}
__device__ __forceinline__ void reciprocals(double a, double b, double &ra, double &rb) {
  const double x = mul_(a, b);
  const float s = (float)x;
  if (s > 1e-30f && s < 1e30f) {
    double r = (double)(1.0f / s);
    r = fma(r, fma(-x, r, 1.0), r);
    r = fma(r, fma(-x, r, 1.0), r);
    ra = mul_(r, b);
    rb = mul_(r, a);
  } else {  // also a node whose density is zero or not finite: the other keeps its own
    ra = 1.0 / a;
    rb = 1.0 / b;
  }
}

// Density and momentum of a node's shifted populations: rho = rho0 + sum f, j = sum c f (the
// rest-state part carries no momentum), from the sums and differences of opposite directions.
template <typename real>
__device__ __forceinline__ void node_moments(const real f[Q], real &drho, real j[3]) {
  real s[9], d[9];
#pragma unroll
  for (int p = 0; p < 9; p++) {
    s[p] = add_(f[2 * p + 1], f[2 * p + 2]);
    d[p] = add_(f[2 * p + 1], -f[2 * p + 2]);
  }
  drho = add_(add_(f[0], add_(add_(s[0], s[1]), s[2])),
              add_(add_(add_(s[3], s[4]), add_(s[5], s[6])), add_(s[7], s[8])));
  j[0] = add_(d[0], add_(add_(d[3], d[4]), add_(d[5], d[6])));
  j[1] = add_(d[1], add_(add_(d[3], -d[4]), add_(d[7], d[8])));
  j[2] = add_(d[2], add_(add_(d[5], -d[6]), add_(d[7], -d[8])));
}

// One population after the collision: its relaxed value plus the equilibrium part P and the
// momentum part l v. FP64: (1 - omega) f + P + l v; FP32: f + (P - omega f + l v), whose
// rounding stays in proportion to omega at large tau.
__device__ __forceinline__ double relaxed(double f, double P, double l, double v,
                                          const CollideCoef<double> &k) {
  return fma(l, v, fma(k.omc, f, P));
}
__device__ __forceinline__ float relaxed(float f, float P, float l, float v,
                                         const CollideCoef<float> &k) {
  return __fadd_rn(f, fmaf(l, v, fmaf(k.nom, f, P)));
}
// the rest population: no momentum part
__device__ __forceinline__ double relaxed(double f, double P, const CollideCoef<double> &k) {
  return fma(k.omc, f, P);
}
__device__ __forceinline__ float relaxed(float f, float P, const CollideCoef<float> &k) {
  return __fadd_rn(f, fmaf(k.nom, f, P));
}

// BGK collision with Guo forcing (Eqs. 9-10) of one node's shifted populations f in place, with
// the uniform force g (FORCE; without it the force terms vanish), given 1/rho. With
// u = (j + g/2)/rho the momentum rho u is j + g/2 itself, so the equilibrium's linear term needs
// no velocity and no density, and the linear parts of equilibrium and source join:
//   omega 3 w c.(rho u) + (1 - omega/2) 3 w c.g           = omega 3 w c.L,  L = j + g/omega;
// likewise the second-order parts, with K = j + (2 tau - 1/2) g:
//   omega 4.5 w rho (c.u)^2 + (1 - omega/2) 9 w (c.g)(c.u)  = omega 4.5 w (c.u)(c.K),
//   omega 1.5 w rho u^2 + (1 - omega/2) 3 w u.g             = omega 1.5 w u.K,
// so f*_i = (1 - omega) f_i + w omega (drho - 1.5 u.K) + 4.5 w omega (c.u)(c.K) +- 3 w omega c.L,
// where the directions of an axis or of a coordinate plane share their second-order term: about
// 120 operations instead of 250. FP64 passes are bound by the FP64 units (2 lanes per cycle and
// SM; ncu: 84 % busy): 128^3 on all SMs 506 us against 867, 32^3 13.1 against 32.1 (there the
// flat node groups halve it as well), 256^3 3.98 ms against 6.85. The FP32 pass stays at the
// copy bandwidth (256^3: 366 us); 16-bit storage, 256^3 BF16 on 112 SMs 223 us against 229.
// The rounding of u enters at second order only, where a form with rho u rounds it into the
// linear term: u of the 256^3 FP32 run is 1.2e-7 off 64 bits after 40 steps, against 3.6e-7.
// FP32 with a force keeps 3 w c.g out of the momentum part and adds it beside the smaller
// equilibrium part: rounding j + g/omega, the same way at a node step after step, would change the
// force by as much as the last place of j (24x20x18, g = 2e-6, u about 1e-3: u after 500 steps 8e-8
// off 64 bits against 5.6e-6, and 3.6e-6 with the source added to each population by itself).
template <bool FORCE, typename real>
__device__ __forceinline__ void collide(real f[Q], real drho, const real j[3], real ir,
                                        const CollideCoef<real> &k) {
  constexpr bool apart = FORCE && sizeof(real) == 4;
  real u[3], K[3], L[3];
#pragma unroll
  for (int a = 0; a < 3; a++) {
    u[a] = mul_(FORCE ? add_(j[a], k.Fh[a]) : j[a], ir);
    K[a] = FORCE ? add_(j[a], k.Kc[a]) : j[a];
    L[a] = FORCE && !apart ? add_(j[a], k.Lc[a]) : j[a];
  }
  const real qxx = mul_(u[0], K[0]), qyy = mul_(u[1], K[1]), qzz = mul_(u[2], K[2]);
  const real s = fma_(real(-1.5), add_(add_(qxx, qyy), qzz), drho);
  f[0] = relaxed(f[0], mul_(k.b0, s), k);
  const real pa = mul_(k.ba, s), pd = mul_(k.bd, s);
  const real qk[3] = {qxx, qyy, qzz};
#pragma unroll
  for (int a = 0; a < 3; a++) {
    const real P = fma_(k.qa, qk[a], pa);
    f[2 * a + 1] = relaxed(f[2 * a + 1], apart ? add_(P, k.ga[a]) : P, k.la, L[a], k);
    f[2 * a + 2] = relaxed(f[2 * a + 2], apart ? add_(P, -k.ga[a]) : P, -k.la, L[a], k);
  }
#pragma unroll
  for (int p = 0; p < 3; p++) {  // planes xy, xz, yz: directions 7 + 4 p .. 10 + 4 p
    const int a = p == 2 ? 1 : 0, b = p == 0 ? 1 : 2, i = 7 + 4 * p;
    const real P = fma_(k.qd, add_(qk[a], qk[b]), pd);
    // the mixed term u_a K_b + u_b K_a (twice u_a K_b without a force)
    const real m = FORCE ? fma_(u[a], K[b], mul_(u[b], K[a])) : mul_(u[a], K[b]);
    const real qm = FORCE ? k.qd : k.qa;
    const real Pp = fma_(qm, m, P), Pm = fma_(-qm, m, P);
    const real lp = add_(L[a], L[b]), lm = add_(L[a], -L[b]);
    const real gp = add_(k.gd[a], k.gd[b]), gm = add_(k.gd[a], -k.gd[b]);
    f[i] = relaxed(f[i], apart ? add_(Pp, gp) : Pp, k.ld, lp, k);
    f[i + 1] = relaxed(f[i + 1], apart ? add_(Pp, -gp) : Pp, -k.ld, lp, k);
    f[i + 2] = relaxed(f[i + 2], apart ? add_(Pm, gm) : Pm, k.ld, lm, k);
    f[i + 3] = relaxed(f[i + 3], apart ? add_(Pm, -gm) : Pm, -k.ld, lm, k);
  }
}

// The collision of the two nodes a and b of a pair.
template <bool FORCE, typename real>
__device__ __forceinline__ void collide_pair(real a[Q], real b[Q], const LatParams<real> &P) {
  real da, db, ja[3], jb[3], ia, ib;
  if constexpr (sizeof(real) == 4) {  // one after the other: fewer registers
    node_moments(a, da, ja);
    collide<FORCE>(a, da, ja, real(1) / add_(P.rho0, da), P.cc);
    node_moments(b, db, jb);
    collide<FORCE>(b, db, jb, real(1) / add_(P.rho0, db), P.cc);
  } else {
    node_moments(a, da, ja);
    node_moments(b, db, jb);
    reciprocals(add_(P.rho0, da), add_(P.rho0, db), ia, ib);
    collide<FORCE>(a, da, ja, ia, P.cc);
    collide<FORCE>(b, db, jb, ib, P.cc);
  }
}

// Post-streaming populations a (node x0) and b (node x0 + 1) of two fluid nodes, x0 even,
// from post-collision array `fin` (FIRST: `fin` already holds post-streaming populations,
// read in place). Populations that do not move along x are one aligned 2-wide load; a link
// whose source is a wall node is bounced back (opposite population of the same node plus the
// moving-wall term).
template <typename real, typename S, bool FIRST>
__device__ __forceinline__ void load_pair(const S *IBLB_RO fin, const LatParams<real> &P,
                                          int x0, int y, int z, real a[Q], real b[Q]) {
  using V2 = typename Storage<S>::V2;
  const size_t plane = (size_t)P.nx * P.ny;
  const size_t n = (size_t)z * plane + (size_t)y * P.nx + x0;
  if (FIRST) {
#pragma unroll
    for (int i = 0; i < Q; i++) {
      widen2(*reinterpret_cast<const V2 *>(fin + (size_t)i * P.ncell + n), a[i], b[i]);
      a[i] *= real(kinv<S>(i));
      b[i] *= real(kinv<S>(i));
    }
    return;
  }
  const int xm = x0 == 0 ? P.nx - 1 : x0 - 1;   // source of node x0 for c_x = +1
  const int xp = x0 + 2 == P.nx ? 0 : x0 + 2;   // source of node x0 + 1 for c_x = -1
  const int ym = y == 0 ? P.ny - 1 : y - 1, yp = y == P.ny - 1 ? 0 : y + 1;
  int zm = z - 1, zp = z + 1;
  if (!P.has_walls) {
    zm = z == 0 ? P.nz - 1 : zm;
    zp = z == P.nz - 1 ? 0 : zp;
  }
  const bool wall_below = P.has_walls && zm == 0;
  const bool wall_above = P.has_walls && zp == P.nz - 1;
  const size_t zo[3] = {(size_t)zm * plane, (size_t)z * plane, (size_t)zp * plane};
  const size_t yo[3] = {(size_t)ym * P.nx, (size_t)y * P.nx, (size_t)yp * P.nx};
#pragma unroll
  for (int i = 0; i < Q; i++) {
    if ((cz(i) > 0 && wall_below) || (cz(i) < 0 && wall_above)) {
      widen2(*reinterpret_cast<const V2 *>(fin + (size_t)opp(i) * P.ncell + n), a[i], b[i]);
      const real wall = cz(i) > 0 ? P.wb[i] : P.wt[i];
      a[i] = add_(a[i] * real(kinv<S>(opp(i))), wall);
      b[i] = add_(b[i] * real(kinv<S>(opp(i))), wall);
      continue;
    }
    const S *row = fin + (size_t)i * P.ncell + zo[1 - cz(i)] + yo[1 - cy(i)];
    if (cx(i) == 0) {
      widen2(*reinterpret_cast<const V2 *>(row + x0), a[i], b[i]);
    } else if (cx(i) > 0) {
      a[i] = widen(row[xm]);
      b[i] = widen(row[x0]);
    } else {
      a[i] = widen(row[x0 + 1]);
      b[i] = widen(row[xp]);
    }
    a[i] *= real(kinv<S>(i));
    b[i] *= real(kinv<S>(i));
  }
}

template <typename real, typename S>
__device__ __forceinline__ void store_pair(S *IBLB_RO fout, const LatParams<real> &P,
                                           size_t n, const real a[Q], const real b[Q]) {
  using V2 = typename Storage<S>::V2;
#pragma unroll
  for (int i = 0; i < Q; i++)
    *reinterpret_cast<V2 *>(fout + (size_t)i * P.ncell + n) =
        Narrow<S>::two(a[i] * real(kscale<S>(i)), b[i] * real(kscale<S>(i)));
}

// Two-wide FP32 arithmetic (one packed instruction per operation on sm_100 and later):
// lane x belongs to the first node of a pair, lane y to the second.
__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, dup(-1.0f), a); }

// The collision of `collide` for a node pair held in the scaled storage units of a 16-bit type,
// g_i = (f_i - w_i rho0) K / w_i: the moments weigh g_i by w_i / K, and in the update the weights
// cancel, so every direction has the coefficients
//   g*_i = (1 - omega) g_i + omega K (drho - 1.5 u.K) + 4.5 omega K (c.u)(c.K) +- 3 omega K c.L.
template <bool FORCE>
__device__ __forceinline__ void collide_pair_scaled(float2 g[Q], const LatParams<float> &P) {
  const CollideCoef<float> &k = P.cc;
  float2 s[9], d[9];
#pragma unroll
  for (int p = 0; p < 9; p++) {
    s[p] = add2(g[2 * p + 1], g[2 * p + 2]);
    d[p] = sub2(g[2 * p + 1], g[2 * p + 2]);
  }
  const float2 ma = dup(k.ma), md = dup(k.md);
  const float2 sa = add2(add2(s[0], s[1]), s[2]);
  const float2 sd = add2(add2(add2(s[3], s[4]), add2(s[5], s[6])), add2(s[7], s[8]));
  const float2 drho = fma2(md, sd, fma2(ma, sa, mul2(dup(k.m0), g[0])));
  float2 j[3];
  j[0] = fma2(ma, d[0], mul2(md, add2(add2(d[3], d[4]), add2(d[5], d[6]))));
  j[1] = fma2(ma, d[1], mul2(md, add2(sub2(d[3], d[4]), add2(d[7], d[8]))));
  j[2] = fma2(ma, d[2], mul2(md, add2(sub2(d[5], d[6]), sub2(d[7], d[8]))));
  const float2 rho = add2(dup(P.rho0), drho);
  const float2 ir = make_float2(__frcp_rn(rho.x), __frcp_rn(rho.y));
  float2 u[3], K[3], L[3];
#pragma unroll
  for (int a = 0; a < 3; a++) {
    u[a] = mul2(FORCE ? add2(j[a], dup(k.Fh[a])) : j[a], ir);
    K[a] = FORCE ? add2(j[a], dup(k.Kc[a])) : j[a];
    L[a] = FORCE ? add2(j[a], dup(k.Lc[a])) : j[a];
  }
  const float2 q[3] = {mul2(u[0], K[0]), mul2(u[1], K[1]), mul2(u[2], K[2])};
  const float2 tr = fma2(dup(-1.5f), add2(add2(q[0], q[1]), q[2]), drho);
  const float2 base = mul2(dup(k.bd), tr);
  const float2 omc = dup(k.omc), qd = dup(k.qd), l = dup(k.ld), nl = dup(-k.ld);
  g[0] = fma2(omc, g[0], base);
#pragma unroll
  for (int a = 0; a < 3; a++) {
    const float2 Pq = fma2(qd, q[a], base);
    g[2 * a + 1] = fma2(l, L[a], fma2(omc, g[2 * a + 1], Pq));
    g[2 * a + 2] = fma2(nl, L[a], fma2(omc, g[2 * a + 2], Pq));
  }
  const float2 qm = dup(FORCE ? k.qd : 2.0f * k.qd), nqm = dup(FORCE ? -k.qd : -2.0f * k.qd);
#pragma unroll
  for (int p = 0; p < 3; p++) {
    const int a = p == 2 ? 1 : 0, b = p == 0 ? 1 : 2, i = 7 + 4 * p;
    const float2 Pq = fma2(qd, add2(q[a], q[b]), base);
    const float2 m = FORCE ? fma2(u[a], K[b], mul2(u[b], K[a])) : mul2(u[a], K[b]);
    const float2 Pp = fma2(qm, m, Pq), Pm = fma2(nqm, m, Pq);
    const float2 lp = add2(L[a], L[b]), lm = sub2(L[a], L[b]);
    g[i] = fma2(l, lp, fma2(omc, g[i], Pp));
    g[i + 1] = fma2(nl, lp, fma2(omc, g[i + 1], Pp));
    g[i + 2] = fma2(l, lm, fma2(omc, g[i + 2], Pm));
    g[i + 3] = fma2(nl, lm, fma2(omc, g[i + 3], Pm));
  }
}

template <typename V2>
__device__ __forceinline__ float2 widen_pair(V2 v);
template <>
__device__ __forceinline__ float2 widen_pair(__half2 v) { return __half22float2(v); }
template <>
__device__ __forceinline__ float2 widen_pair(__nv_bfloat162 v) { return __bfloat1622float2(v); }
template <typename V2>
__device__ __forceinline__ V2 narrow_pair(float2 v);
template <>
__device__ __forceinline__ __half2 narrow_pair(float2 v) { return __float22half2_rn(v); }
template <>
__device__ __forceinline__ __nv_bfloat162 narrow_pair(float2 v) { return __float22bfloat162_rn(v); }

// Reinterpret 32 bits as a pair of 16-bit storage values, and back.
template <typename V2>
__device__ __forceinline__ V2 as_pair(unsigned int u) {
  V2 v;
  memcpy(&v, &u, sizeof(v));
  return v;
}
template <typename V2>
__device__ __forceinline__ unsigned int as_bits(V2 v) {
  unsigned int u;
  memcpy(&u, &v, sizeof(u));
  return u;
}

// K1 for 16-bit storage: each thread owns four nodes x0 .. x0 + 3 (x0 a multiple of 4), so
// every population row is one aligned 8-byte load (plus one 2-byte load of the neighbouring
// node for the directions that move along x) and every store one 8-byte store: half the
// memory instructions of the two-node form and twice the bytes in flight per thread, which a
// 2-byte type needs to keep HBM busy. The loaded rows stay packed in registers (`lo` holds
// nodes x0, x0 + 1, `hi` nodes x0 + 2, x0 + 3) and are widened one node pair at a time for
// the collision; the results are packed back in place.
// `After`: applied to the packed results lo, hi before they are stored.
template <typename S, bool FIRST, bool FORCE, typename After>
__device__ __forceinline__ void quad_nodes(const S *IBLB_RO fin, S *IBLB_RO fout,
                                           const LatParams<float> &P, int x0, int y, int z,
                                           After after) {
  using V2 = typename Storage<S>::V2;
  const size_t plane = (size_t)P.nx * P.ny;
  const size_t n = (size_t)z * plane + (size_t)y * P.nx + x0;
  unsigned int lo[Q], hi[Q];  // packed pairs (x0, x0 + 1) and (x0 + 2, x0 + 3)
  bool bounced[Q];            // population i comes from the wall: add the wall term
  if (FIRST) {
#pragma unroll
    for (int i = 0; i < Q; i++) {
      const uint2 v = *reinterpret_cast<const uint2 *>(fin + (size_t)i * P.ncell + n);
      lo[i] = v.x;
      hi[i] = v.y;
      bounced[i] = false;
    }
  } else {
    const int xm = x0 == 0 ? P.nx - 1 : x0 - 1;   // source of node x0 for c_x = +1
    const int xp = x0 + 4 == P.nx ? 0 : x0 + 4;   // source of node x0 + 3 for c_x = -1
    const int ym = y == 0 ? P.ny - 1 : y - 1, yp = y == P.ny - 1 ? 0 : y + 1;
    int zm = z - 1, zp = z + 1;
    if (!P.has_walls) {
      zm = z == 0 ? P.nz - 1 : zm;
      zp = z == P.nz - 1 ? 0 : zp;
    }
    const bool wall_below = P.has_walls && zm == 0;
    const bool wall_above = P.has_walls && zp == P.nz - 1;
    const size_t zo[3] = {(size_t)zm * plane, (size_t)z * plane, (size_t)zp * plane};
    const size_t yo[3] = {(size_t)ym * P.nx, (size_t)y * P.nx, (size_t)yp * P.nx};
#pragma unroll
    for (int i = 0; i < Q; i++) {
      bounced[i] = (cz(i) > 0 && wall_below) || (cz(i) < 0 && wall_above);
      if (bounced[i]) {
        const uint2 v = *reinterpret_cast<const uint2 *>(fin + (size_t)opp(i) * P.ncell + n);
        lo[i] = v.x;
        hi[i] = v.y;
        continue;
      }
      const S *row = fin + (size_t)i * P.ncell + zo[1 - cz(i)] + yo[1 - cy(i)];
      const uint2 v = *reinterpret_cast<const uint2 *>(row + x0);  // nodes x0 .. x0 + 3
      if (cx(i) == 0) {
        lo[i] = v.x;
        hi[i] = v.y;
      } else if (cx(i) > 0) {  // sources x0 - 1 .. x0 + 2
        const unsigned int e = *reinterpret_cast<const unsigned short *>(row + xm);
        lo[i] = __byte_perm(e, v.x, 0x5410);
        hi[i] = __byte_perm(v.x, v.y, 0x5432);
      } else {  // sources x0 + 1 .. x0 + 4
        const unsigned int e = *reinterpret_cast<const unsigned short *>(row + xp);
        lo[i] = __byte_perm(v.x, v.y, 0x5432);
        hi[i] = __byte_perm(v.y, e, 0x5432);
      }
    }
  }
#pragma unroll
  for (int h = 0; h < 2; h++) {  // node pairs (x0, x0 + 1), (x0 + 2, x0 + 3)
    unsigned int *pk = h ? hi : lo;
    float2 g[Q];
#pragma unroll
    for (int i = 0; i < Q; i++) {
      g[i] = widen_pair(as_pair<V2>(pk[i]));
      if (bounced[i]) {  // stored units: the wall term times k_i
        const float wall = (cz(i) > 0 ? P.wb[i] : P.wt[i]) * float(kscale<S>(i));
        g[i] = add2(g[i], dup(wall));
      }
    }
    collide_pair_scaled<FORCE>(g, P);
#pragma unroll
    for (int i = 0; i < Q; i++) pk[i] = as_bits(narrow_pair<V2>(g[i]));
  }
  after(lo, hi);
#pragma unroll
  for (int i = 0; i < Q; i++)
    *reinterpret_cast<uint2 *>(fout + (size_t)i * P.ncell + n) = make_uint2(lo[i], hi[i]);
}

// no step after the collision
struct Nothing {
  __device__ __forceinline__ void operator()(unsigned int *, unsigned int *) const {}
};

template <typename real, typename S>
struct StreamArgs {
  const S *fin;
  S *fout;
  LatParams<real> P;
  FlatGroups G;  // node groups of the context
  int z0;        // first fluid layer
  int force;     // the body force is non-zero
  const int *tile_slot;        // the interface force of the step, by active tile (null: no mesh)
  const Vec4<real> *Fslot;
};

// K1t: the fluid nodes of the active tiles with body + interface force. Runs after K1 of the
// same step and corrects K1's result there in place. The collision (BGK with Guo forcing,
// Eqs. 9-10) keeps rho and turns the momentum j into j + Ft (Ft the total force), so K1's
// output f0 at a node (the collision with the body force g alone) gives rho = rho0 + sum f0
// and j = J - g, J = sum c f0, without the pre-collision populations. K1t therefore reads and
// writes only each node's own populations, no pulled neighbours.
// Its work list is the node pairs (x0, x0 + 1), x0 even, that hold a node of some vertex's
// stencil, appended by the spreading's gather pass (K4b) as slot * 32 + pair. Nodes without force
// keep K1's result, which is already final. A thread takes a listed pair, or one node of it: long
// lists are bound by the scattered rows' accesses, which the pair halves (96 wetting boxes: 1.29
// ms per step against 1.36), short ones by one thread's chain, which the node halves (32^3 FP64 in
// the fused kernel: 6.8 us against 11.5). Both give the same bits.
template <typename real, typename S>
struct TilesArgs {
  S *fout;
  const int *slot_tile, *pair_list, *npairs_ptr;
  const Vec4<real> *Fslot;
  LatParams<real> P;
  int max_pairs;
};

// f (deviations, after the collision with the body force g alone) becomes the collision with
// g + F. In the collision's form (see collide) the interface force F shifts u by h = F/(2 rho),
// K by e = (2 tau - 1/2) F and L by F/omega, so the second-order products u_a K_b change by
//   D_ab = u0_a e_b + h_a K1_b,   K1 = K0 + e,
// and the populations by w omega (-1.5 tr D) + 4.5 w omega c.D c +- 3 w c.F.
template <typename real>
__device__ __forceinline__ void apply_force(real f[Q], real drho, const real J[3], real ir,
                                            const real F[3], const CorrectionCoef<real> &k) {
  real u0[3], h[3], e[3], K1[3], D[3];
  const real hr = mul_(real(0.5), ir);
#pragma unroll
  for (int a = 0; a < 3; a++) {
    u0[a] = mul_(add_(J[a], -k.Gh[a]), ir);
    h[a] = mul_(F[a], hr);
    e[a] = mul_(F[a], k.kappa);
    K1[a] = add_(add_(J[a], k.Kt[a]), e[a]);
    D[a] = fma_(u0[a], e[a], mul_(h[a], K1[a]));
  }
  const real s = mul_(real(-1.5), add_(add_(D[0], D[1]), D[2]));
  f[0] = fma_(k.b0, s, f[0]);
  const real pa = mul_(k.ba, s), pd = mul_(k.bd, s);
#pragma unroll
  for (int a = 0; a < 3; a++) {
    const real P = fma_(k.qa, D[a], pa);
    f[2 * a + 1] = add_(f[2 * a + 1], fma_(k.la, F[a], P));
    f[2 * a + 2] = add_(f[2 * a + 2], fma_(-k.la, F[a], P));
  }
#pragma unroll
  for (int p = 0; p < 3; p++) {  // planes xy, xz, yz
    const int a = p == 2 ? 1 : 0, b = p == 0 ? 1 : 2, i = 7 + 4 * p;
    const real m = add_(fma_(u0[a], e[b], mul_(h[a], K1[b])), fma_(u0[b], e[a], mul_(h[b], K1[a])));
    const real P = fma_(k.qd, add_(D[a], D[b]), pd);
    const real Pp = fma_(k.qd, m, P), Pm = fma_(-k.qd, m, P);
    const real lp = add_(F[a], F[b]), lm = add_(F[a], -F[b]);
    f[i] = add_(f[i], fma_(k.ld, lp, Pp));
    f[i + 1] = add_(f[i + 1], fma_(-k.ld, lp, Pp));
    f[i + 2] = add_(f[i + 2], fma_(k.ld, lm, Pm));
    f[i + 3] = add_(f[i + 3], fma_(-k.ld, lm, Pm));
  }
}

// apply_force at one node (deviations f after K1's collision) with its interface force.
template <typename real>
__device__ __forceinline__ void correct_node(real f[Q], const Vec4<real> &F, const LatParams<real> &P) {
  const real Fk[3] = {F.x, F.y, F.z};
  real drho, J[3];
  node_moments(f, drho, J);
  apply_force(f, drho, J, reciprocal(add_(P.rho0, drho)), Fk, P.ct);
}
template <typename real>
__device__ __forceinline__ bool any_force(const Vec4<real> &F) {
  return F.x != real(0) || F.y != real(0) || F.z != real(0);
}

template <bool PAIR, typename real, typename S>
__device__ __forceinline__ void tiles_body(const TilesArgs<real, S> &A, int first, int stride) {
  S *IBLB_RO fout = A.fout;
  const int *IBLB_RO slot_tile = A.slot_tile;
  const int *IBLB_RO pair_list = A.pair_list;
  const Vec4<real> *IBLB_RO Fslot = A.Fslot;
  const LatParams<real> P = A.P;  // held in registers: the loop below is latency-bound
  constexpr int N = PAIR ? 2 : 1;  // nodes of a thread
  const int items = (PAIR ? 1 : 2) * min(*A.npairs_ptr, A.max_pairs);
  for (int k = first; k < items; k += stride) {
    const int e = pair_list[PAIR ? k : k >> 1];
    const int s = e >> 5;                                    // slot, and the first node in the tile
    const int cell = 2 * (e & 31) + (PAIR ? 0 : k & 1);
    Vec4<real> Fv[N];
    bool any = false;
#pragma unroll
    for (int m = 0; m < N; m++) {
      Fv[m] = Fslot[(size_t)s * TILE_CELLS + cell + m];
      any |= any_force(Fv[m]);
    }
    const int t = slot_tile[s];
    const int tx = t % P.ntx, ty = (t / P.ntx) % P.nty, tz = t / (P.ntx * P.nty);
    const int x0 = tx * TILE + (cell & 3), y = ty * TILE + ((cell >> 2) & 3);
    const int z = tz * TILE + (cell >> 4);
    if (z >= P.nz || (P.has_walls && (z == 0 || z == P.nz - 1))) continue;
    const size_t n = (size_t)z * P.nx * P.ny + (size_t)y * P.nx + x0;
    real f[N][Q];
#pragma unroll
    for (int i = 0; i < Q; i++) {
      const S *row = fout + (size_t)i * P.ncell + n;
      if constexpr (PAIR) {
        widen2(*reinterpret_cast<const typename Storage<S>::V2 *>(row), f[0][i], f[1][i]);
        f[0][i] *= real(kinv<S>(i));
        f[1][i] *= real(kinv<S>(i));
      } else {
        f[0][i] = real(widen(*row)) * real(kinv<S>(i));
      }
    }
    if (!any) continue;
#pragma unroll
    for (int m = 0; m < N; m++) correct_node(f[m], Fv[m], P);
    if constexpr (PAIR) {
      store_pair(fout, P, n, f[0], f[1]);
    } else {
#pragma unroll
      for (int i = 0; i < Q; i++)
        fout[(size_t)i * P.ncell + n] = Narrow<S>::one(f[0][i] * real(kscale<S>(i)));
    }
  }
}

// K1 and K1t in one: node group (gx, y, z) of the lattice pass, its active-tile nodes corrected
// before they are stored, rounded to the storage type in between as in the two passes, so that
// the results are theirs bit for bit. For passes that start after the step's force is complete.
template <typename real, typename S, bool FORCE>
__device__ __forceinline__ void forced_group(const StreamArgs<real, S> &A, int gx, int y, int z) {
  constexpr int N = sizeof(S) == 2 ? 4 : 2;  // nodes of the group, all in one tile row
  const LatParams<real> &P = A.P;
  const int x0 = N * gx;
  int slot = -1;
  if (A.tile_slot) slot = A.tile_slot[((z >> 2) * P.nty + (y >> 2)) * P.ntx + (x0 >> 2)];
  const Vec4<real> *F = A.Fslot + ((x0 & 3) + 4 * (y & 3) + 16 * (z & 3));
  if constexpr (sizeof(S) == 2) {
    using V2 = typename Storage<S>::V2;
    quad_nodes<S, false, FORCE>(A.fin, A.fout, P, x0, y, z, [&](unsigned int *lo, unsigned int *hi) {
      if (slot < 0) return;
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const Vec4<real> Fa = F[(size_t)slot * TILE_CELLS + 2 * h];
        const Vec4<real> Fb = F[(size_t)slot * TILE_CELLS + 2 * h + 1];
        if (!any_force(Fa) && !any_force(Fb)) continue;
        unsigned int *pk = h ? hi : lo;
        real a[Q], b[Q];
#pragma unroll
        for (int i = 0; i < Q; i++) {
          widen2(as_pair<V2>(pk[i]), a[i], b[i]);
          a[i] *= real(kinv<S>(i));
          b[i] *= real(kinv<S>(i));
        }
        correct_node(a, Fa, P);
        correct_node(b, Fb, P);
#pragma unroll
        for (int i = 0; i < Q; i++)
          pk[i] = as_bits(Narrow<S>::two(a[i] * real(kscale<S>(i)), b[i] * real(kscale<S>(i))));
      }
    });
  } else {
    real a[Q], b[Q];
    load_pair<real, S, false>(A.fin, P, x0, y, z, a, b);
    collide_pair<FORCE>(a, b, P);
    if (slot >= 0) {
      const Vec4<real> Fa = F[(size_t)slot * TILE_CELLS], Fb = F[(size_t)slot * TILE_CELLS + 1];
      if (any_force(Fa)) correct_node(a, Fa, P);
      if (any_force(Fb)) correct_node(b, Fb, P);
    }
    store_pair(A.fout, P, (size_t)z * P.nx * P.ny + (size_t)y * P.nx + x0, a, b);
  }
}

// K1b: velocity after streaming at the nodes the interpolation reads: the nodes of the pairs
// that K4b listed (every fluid node of a vertex's stencil, and its pair partner); one thread
// per node of a listed pair. u = (j + (g + F)/2)/rho, the velocity of the forced collision
// (Eq. 10 with Guo's forcing). The wall layers, which the interpolation takes from the wall
// velocities, are never listed.
template <typename real, typename S>
struct ShellArgs {
  const S *fpost;
  const int *slot_tile, *pair_list, *npairs_ptr;
  const Vec4<real> *Fslot;
  Vec4<real> *Uslot;
  LatParams<real> P;
  int max_pairs;
};

template <typename real, typename S>
__device__ __forceinline__ void shell_body(const ShellArgs<real, S> &A, int first, int stride) {
  const S *IBLB_RO fpost = A.fpost;
  const int *IBLB_RO slot_tile = A.slot_tile;
  const int *IBLB_RO pair_list = A.pair_list;
  const Vec4<real> *IBLB_RO Fslot = A.Fslot;
  Vec4<real> *IBLB_RO Uslot = A.Uslot;
  const LatParams<real> P = A.P;
  const int nodes = 2 * min(*A.npairs_ptr, A.max_pairs);
  for (int k = first; k < nodes; k += stride) {
    const int e = pair_list[k >> 1];
    const int s = e >> 5, cell = 2 * (e & 31) + (k & 1);
    const int t = slot_tile[s];
    const int tx = t % P.ntx, ty = (t / P.ntx) % P.nty, tz = t / (P.ntx * P.nty);
    const int x = tx * TILE + (cell & 3), y = ty * TILE + ((cell >> 2) & 3),
              z = tz * TILE + (cell >> 4);
    if (z >= P.nz || (P.has_walls && (z == 0 || z == P.nz - 1))) continue;
    real f[Q];
    pull<real, S, true>(fpost, P, x, y, z, f);
    real drho, j[3];
    node_moments(f, drho, j);
    const Vec4<real> Fs = Fslot[(size_t)s * TILE_CELLS + cell];
    const real Fk[3] = {Fs.x, Fs.y, Fs.z};
    const real rho_hi = P.rho0 + drho;
    const real rho_lo = (P.rho0 - rho_hi) + drho;
    const real r1 = real(1) / rho_hi;
    const real inv_rho = r1 * (real(1) - rho_lo * r1);
    Vec4<real> uv;
    uv.x = (j[0] + real(0.5) * (P.g[0] + Fk[0])) * inv_rho;
    uv.y = (j[1] + real(0.5) * (P.g[1] + Fk[1])) * inv_rho;
    uv.z = (j[2] + real(0.5) * (P.g[2] + Fk[2])) * inv_rho;
    uv.w = real(0);
    Uslot[(size_t)s * TILE_CELLS + cell] = uv;
  }
}

// Node groups of K1's direct kernels: pairs along x, four nodes with 16-bit storage.
template <typename S>
FlatGroups k1_groups(const Ctx &c) {
  return flat_groups(c.nx / (sizeof(S) == 2 ? 4 : 2), c.ny, c.has_walls ? c.nz - 2 : c.nz);
}

// Argument records of K1t and K1b for the step that starts from c's current state (K1t pulls
// from f[cur] into f[cur ^ 1]; K1b reads the array that step writes, `fpost`).
template <typename real, typename S>
TilesArgs<real, S> tiles_args(const Ctx &c) {
  TilesArgs<real, S> a;
  a.fout = (S *)c.f[c.cur ^ 1];
  a.slot_tile = c.slot_tile[c.map];
  a.pair_list = c.pair_list;
  a.npairs_ptr = c.counters + 5;
  a.Fslot = (const Vec4<real> *)c.Fslot[c.map];
  a.P = lat_params<real>(c);
  a.max_pairs = 32 * c.max_slots;
  return a;
}
template <typename real, typename S>
ShellArgs<real, S> shell_args(const Ctx &c, const void *fpost) {
  ShellArgs<real, S> a;
  a.fpost = (const S *)fpost;
  a.slot_tile = c.slot_tile[c.map];
  a.pair_list = c.pair_list;
  a.npairs_ptr = c.counters + 5;
  a.Fslot = (const Vec4<real> *)c.Fslot[c.map];
  a.Uslot = (Vec4<real> *)c.Uslot;
  a.P = lat_params<real>(c);
  a.max_pairs = 32 * c.max_slots;
  return a;
}
template <typename real, typename S>
StreamArgs<real, S> stream_args(const Ctx &c) {
  StreamArgs<real, S> a;
  a.fin = (const S *)c.f[c.cur];
  a.fout = (S *)c.f[c.cur ^ 1];
  a.P = lat_params<real>(c);
  a.z0 = c.has_walls ? 1 : 0;
  a.G = k1_groups<S>(c);
  a.force = c.g[0] != 0.0 || c.g[1] != 0.0 || c.g[2] != 0.0;
  a.tile_slot = c.nv ? c.tile_slot[c.map] : nullptr;
  a.Fslot = (const Vec4<real> *)c.Fslot[c.map];
  return a;
}

}  // namespace
}  // namespace iblb
