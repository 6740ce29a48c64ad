// Discrete adjoint of the coupled IB-LB step (Sec. III), in double precision: gradients of an
// observable of the final vertex positions with respect to the interface parameters
// theta = (alpha1, alpha2, alpha3, eps) of Eqs. 2 and 19. The forward run is that of the
// context, FP64 or FP32; with FP32 the reverse pass linearises the double-precision step about
// the recomputed FP32 trajectory.
//
// One forward step n maps (P_n, q_n) to (P_{n+1}, q_{n+1}), P being the post-collision
// populations the pull scheme keeps between steps:
//   phi   = phi(q_n; theta)                          nodal forces, Eqs. 16-19
//   F(x)  = sum_v phi_v W(x - q_v)                   spreading on the fluid nodes, Eqs. 13-15
//   P'(x) = C(pull(P_n)(x), g + F(x))                BGK + Guo collision of the streamed state
//   u(x)  = (sum_i c_i pull(P')(x)_i + (g+F)/2)/rho  velocity after streaming
//   q_{n+1,v} = q_{n,v} + sum_x u(x) W(x - q_v)      interpolation and Euler update, Eqs. 11-12
// The reverse step applies the transposed Jacobians in the opposite order:
//   interpolation^T (including the derivative of the Peskin weights in q), the velocity
//   moments^T, the collision^T with the streaming^T (a permutation of (node, direction)
//   pairs: every adjoint population is written exactly once, no atomics), spreading^T, and
//   the transposed force Jacobian dphi/dq, which is symmetric (phi = -grad E) and is applied
//   as a forward-mode (dual number) derivative of the face forces along the adjoint force.
//   The forces are linear in alpha and eps, so dphi/dtheta is the force with one parameter
//   set to 1 and the others to 0.
// The trajectory is recorded as checkpoints every K steps; the reverse pass recomputes each
// segment forward from its checkpoint with the ordinary step, so the recomputed states are
// the recorded ones bit for bit.
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "lattice_device.cuh"

namespace iblb {
namespace {

// --- device helpers --------------------------------------------------------------------
//
// FP64 issues at 1/64 of the FP32 rate on this GPU, two lanes per cycle and SM whatever the number
// of active lanes: the kernels count double operations, and give each pass enough warps to use
// every SM's unit.

struct FaceArgs {
  int nf;
  const int *faces;
  const double *fref;  // [nf][4]: H11, H12, H22, A0
  double centre[3];
  double alpha[3], eps, xi;
  int lj;  // wall force on and the lattice has walls
  double zb, zt;
};

__device__ __forceinline__ double dot3(const double a[3], const double b[3]) {
  return fma(a[0], b[0], fma(a[1], b[1], a[2] * b[2]));
}
__device__ __forceinline__ void cross3(const double a[3], const double b[3], double o[3]) {
  o[0] = fma(a[1], b[2], -a[2] * b[1]);
  o[1] = fma(a[2], b[0], -a[0] * b[2]);
  o[2] = fma(a[0], b[1], -a[1] * b[0]);
}
__device__ __forceinline__ double warp_sum(double x) {
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
// Sum of the n values at p by one warp (every lane gets it), in a fixed order.
__device__ __forceinline__ double warp_total(const double *__restrict__ p, int n) {
  double s[4] = {0, 0, 0, 0};
  for (int k0 = 0; k0 < n; k0 += 128)
#pragma unroll
    for (int c = 0; c < 4; c++) {
      const int k = k0 + 32 * c + (threadIdx.x & 31);
      if (k < n) s[c] += p[k];
    }
  return warp_sum((s[0] + s[1]) + (s[2] + s[3]));
}

// Metric of a face and the Skalak energy's coefficients (Eq. 2, readings R4, R5): the strain
// forces are -dE/da = -(paa a + pab b) on corner 1, -dE/db = -(pab a + pbb b) on corner 2 and
// their opposite on corner 0, with eI = 2 dE/dI1 and eL = 2 dE/dL / det G.
struct Strain {
  double G11, G12, G22, id, L;  // metric, 1/det G, ln(det G / det G0)
  double eI, eL, paa, pab, pbb;
};
__device__ __forceinline__ Strain strain_of(const FaceArgs &A, const double a[3], const double b[3],
                                            const double H[4]) {
  Strain s;
  s.G11 = dot3(a, a);
  s.G12 = dot3(a, b);
  s.G22 = dot3(b, b);
  const double det = fma(s.G11, s.G22, -s.G12 * s.G12);
  s.id = 1.0 / det;
  s.L = log(det / (4.0 * H[3] * H[3]));
  s.eI = A.alpha[2] * H[3];
  s.eL = H[3] * fma(0.5 * (A.alpha[0] + A.alpha[1]), s.L, A.alpha[0] - A.alpha[2]) * s.id;
  s.paa = fma(s.eI, H[0], s.eL * s.G22);
  s.pab = fma(s.eI, H[1], -s.eL * s.G12);
  s.pbb = fma(s.eI, H[2], s.eL * s.G11);
  return s;
}
// Lennard-Jones force along z of both wall planes on a centroid at height gz (Eq. 19, readings
// R6-R8) per 48 eps, and its derivative in gz: with s = (xi/dz)^6, (s^2 - s/2)/dz and
// (-13 s^2 + 3.5 s)/dz^2.
__device__ __forceinline__ void lj_pair(const FaceArgs &A, double gz, double &f, double &df) {
  f = df = 0.0;
  for (int w = 0; w < 2; w++) {
    const double r = 1.0 / (gz - (w == 0 ? A.zb : A.zt));
    const double x = A.xi * r, x2 = x * x, s6 = x2 * x2 * x2;
    f = fma(fma(s6, s6, -0.5 * s6), r, f);
    df = fma(s6 * fma(-13.0, s6, 3.5), r * r, df);
  }
}

// Forward pass over faces at positions q: corner forces fc [nf][9], volume gradient share
// (a x b)/6 per corner fn [nf][3] and per warp of 32 faces their share of V, vpart.
__global__ void adj_face_value_kernel(FaceArgs A, const double *__restrict__ q,
                                      double *__restrict__ fc, double *__restrict__ fn,
                                      double *__restrict__ vpart) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  double V = 0.0;
  if (j < A.nf) {
    double x[3][3];
    for (int c = 0; c < 3; c++)
      for (int k = 0; k < 3; k++) x[c][k] = q[3 * A.faces[3 * j + c] + k];
    double a[3], b[3], r0[3], n[3];
    for (int k = 0; k < 3; k++) {
      a[k] = x[1][k] - x[0][k];
      b[k] = x[2][k] - x[0][k];
      r0[k] = x[0][k] - A.centre[k];
    }
    const Strain s = strain_of(A, a, b, A.fref + 4 * j);
    double fz = 0.0;
    if (A.lj) {
      double f, df;
      lj_pair(A, (x[0][2] + x[1][2] + x[2][2]) * (1.0 / 3.0), f, df);
      fz = 16.0 * A.eps * f;  // a third to each corner
    }
    double *o = fc + 9 * (size_t)j;
    for (int k = 0; k < 3; k++) {
      const double ga = fma(s.paa, a[k], s.pab * b[k]), gb = fma(s.pab, a[k], s.pbb * b[k]);
      const double w = k == 2 ? fz : 0.0;
      o[k] = ga + gb + w;
      o[3 + k] = w - ga;
      o[6 + k] = w - gb;
    }
    cross3(a, b, n);
    for (int k = 0; k < 3; k++) fn[3 * (size_t)j + k] = n[k] * (1.0 / 6.0);
    V = dot3(r0, n) * (1.0 / 6.0);  // r0 . (r1 x r2) = r0 . (a x b)
  }
  V = warp_sum(V);
  if ((threadIdx.x & 31) == 0 && j < A.nf) vpart[j >> 5] = V;
}

// Derivative pass over faces along the tangent t (the adjoint force lambda_phi):
// d(corner forces) fj [nf][9], d((a x b)/6) dn [nf][3], and per warp of 32 faces the sums of
// ((a x b)/6) . (t0 + t1 + t2), a share of grad V . t, and of t . dphi/dtheta_k: part [5][warps].
// The strain forces' derivative follows from the metric's, dG = (2 a.ta, a.tb + b.ta, 2 b.tb) and
// d det = dG11 G22 + G11 dG22 - 2 G12 dG12; the forces are linear in each parameter and their
// component along t is -(eI (H : dG)/2 + eL d det / 2), so the four parameter derivatives need no
// further pass.
__global__ void adj_face_tangent_kernel(FaceArgs A, const double *__restrict__ q,
                                        const double *__restrict__ t, double *__restrict__ fj,
                                        double *__restrict__ dn, double *__restrict__ part) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x, warps = (A.nf + 31) / 32;
  double sum[5] = {0, 0, 0, 0, 0};
  if (j < A.nf) {
    double x[3][3], u[3][3];
    for (int c = 0; c < 3; c++)
      for (int k = 0; k < 3; k++) {
        const int v = A.faces[3 * j + c];
        x[c][k] = q[3 * v + k];
        u[c][k] = t[3 * v + k];
      }
    double a[3], b[3], ta[3], tb[3];
    for (int k = 0; k < 3; k++) {
      a[k] = x[1][k] - x[0][k];
      b[k] = x[2][k] - x[0][k];
      ta[k] = u[1][k] - u[0][k];
      tb[k] = u[2][k] - u[0][k];
    }
    const double *H = A.fref + 4 * j;
    const double A0 = H[3];
    const Strain s = strain_of(A, a, b, H);
    const double hG11 = dot3(a, ta), dG12 = dot3(a, tb) + dot3(b, ta), hG22 = dot3(b, tb);
    const double hdet = fma(hG11, s.G22, fma(s.G11, hG22, -s.G12 * dG12));  // d det / 2
    const double dL = 2.0 * hdet * s.id;
    const double deL = s.id * dL * A0 * 0.5 * (A.alpha[0] + A.alpha[1]) - s.eL * dL;
    const double dpaa = fma(deL, s.G22, 2.0 * s.eL * hG22);
    const double dpab = -fma(deL, s.G12, s.eL * dG12);
    const double dpbb = fma(deL, s.G11, 2.0 * s.eL * hG11);
    double f = 0.0, df = 0.0, tz = 0.0, dfz = 0.0;
    if (A.lj) {
      tz = (u[0][2] + u[1][2] + u[2][2]) * (1.0 / 3.0);
      lj_pair(A, (x[0][2] + x[1][2] + x[2][2]) * (1.0 / 3.0), f, df);
      dfz = 16.0 * A.eps * df * tz;
    }
    double *o = fj + 9 * (size_t)j;
    for (int k = 0; k < 3; k++) {
      const double ga = fma(dpaa, a[k], fma(s.paa, ta[k], fma(dpab, b[k], s.pab * tb[k])));
      const double gb = fma(dpab, a[k], fma(s.pab, ta[k], fma(dpbb, b[k], s.pbb * tb[k])));
      const double w = k == 2 ? dfz : 0.0;
      o[k] = ga + gb + w;
      o[3 + k] = w - ga;
      o[6 + k] = w - gb;
    }
    double n[3], c1[3], c2[3], ts[3];
    cross3(a, b, n);
    cross3(ta, b, c1);
    cross3(a, tb, c2);
    for (int k = 0; k < 3; k++) {
      dn[3 * (size_t)j + k] = (c1[k] + c2[k]) * (1.0 / 6.0);
      ts[k] = u[0][k] + u[1][k] + u[2][k];
    }
    sum[0] = dot3(n, ts) * (1.0 / 6.0);
    const double SI = fma(H[0], hG11, fma(H[1], dG12, H[2] * hG22));
    sum[1] = -A0 * fma(0.25, s.L, 0.5) * dL;   // alpha1
    sum[2] = -A0 * 0.25 * s.L * dL;            // alpha2
    sum[3] = A0 * fma(0.5, dL, -SI);           // alpha3
    sum[4] = 48.0 * f * tz;                    // eps
  }
  for (int k = 0; k < 5; k++) {
    const double v = warp_sum(sum[k]);
    if ((threadIdx.x & 31) == 0 && j < A.nf) part[(size_t)k * warps + (j >> 5)] = v;
  }
}

struct VolArgs {
  int on;
  double kV, V0;
};

// Peskin's 4-point function (Eq. 15, reading R2) on the four nodes floor(p) - 1 .. floor(p) + 2 and
// its derivative with respect to p: with r = p - floor(p) and s = sqrt(1 + 4r - 4r^2) the weights
// are (3-2r-s)/8, (3-2r+s)/8, (1+2r+s)/8, (1+2r-s)/8, and s' = (2 - 4r)/s.
struct Stencil {
  int base[3];
  int pad;
  double w[3][4], dw[3][4];
};
__device__ __forceinline__ void stencil_axis(double p, int &base, double w[4], double dw[4]) {
  const double fl = floor(p);
  base = (int)fl - 1;
  const double r = p - fl;
  const double s = sqrt(fma(4.0 * r, 1.0 - r, 1.0));
  const double ds = (2.0 - 4.0 * r) / s;
  const double lo = fma(-2.0, r, 3.0), hi = fma(2.0, r, 1.0);
  w[0] = 0.125 * (lo - s);
  w[1] = 0.125 * (lo + s);
  w[2] = 0.125 * (hi + s);
  w[3] = 0.125 * (hi - s);
  dw[0] = 0.125 * (-2.0 - ds);
  dw[1] = 0.125 * (-2.0 + ds);
  dw[2] = 0.125 * (2.0 + ds);
  dw[3] = 0.125 * (2.0 - ds);
}

constexpr int kFaceThreads = 32, kVertexThreads = 64;

// Forward pass over vertices: phi_v, the sum over the faces at v of the corner forces
// - kV (V - V0)/V0 dV/dq_v, and the stencil of v. Each block sums the volume's partials itself.
// A thread per (vertex, coordinate).
__global__ void __launch_bounds__(kVertexThreads) adj_vertex_value_kernel(
    int nv, int nwarps, const int *__restrict__ vf_start, const int *__restrict__ vf_list,
    const double *__restrict__ corner, const double *__restrict__ fn,
    const double *__restrict__ vpart, VolArgs va, const double *__restrict__ q,
    double *__restrict__ phi, Stencil *__restrict__ st) {
  __shared__ double s_coef;
  if (threadIdx.x < 32) {
    const double V = warp_total(vpart, nwarps);
    if (threadIdx.x == 0) s_coef = va.on ? va.kV * (V - va.V0) / va.V0 : 0.0;
  }
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double f = 0, g = 0;
  if (i < 3 * nv) {
    const int v = i / 3, k = i - 3 * v;
    for (int e = vf_start[v]; e < vf_start[v + 1]; e++) {
      const int fcr = vf_list[e];  // face * 3 + corner
      f += corner[3 * (size_t)fcr + k];
      g += fn[3 * (size_t)(fcr / 3) + k];
    }
    double w[4], dw[4];
    int base;
    stencil_axis(q[i], base, w, dw);
    Stencil &s = st[v];
    s.base[k] = base;
    for (int d = 0; d < 4; d++) {
      s.w[k][d] = w[d];
      s.dw[k][d] = dw[d];
    }
  }
  __syncthreads();
  if (i < 3 * nv) phi[i] = fma(-s_coef, g, f);
}

// Derivative pass over vertices: lam_q_v += the tangent of phi_v along lambda_phi,
//   d(corner forces) - kV/V0 [(V - V0) d(dV/dq_v) + (grad V . t) dV/dq_v];
// block 0 also adds the step's parameter derivatives to grad. A thread per (vertex, coordinate).
__global__ void __launch_bounds__(kVertexThreads) adj_vertex_tangent_kernel(
    int nv, int nwarps, const int *__restrict__ vf_start, const int *__restrict__ vf_list,
    const double *__restrict__ corner, const double *__restrict__ fn, const double *__restrict__ dn,
    const double *__restrict__ vpart, const double *__restrict__ part, VolArgs va,
    double *__restrict__ lam_q, double *__restrict__ grad) {
  __shared__ double s_coef, s_coef2;
  if (threadIdx.x < 32) {
    const double V = warp_total(vpart, nwarps);
    if (threadIdx.x == 0) s_coef = va.on ? va.kV * (V - va.V0) / va.V0 : 0.0;
    if (blockIdx.x == 0)
      for (int k = 0; k < 2; k++) {
        const double p = warp_total(part + (size_t)(1 + k) * nwarps, nwarps);
        if (threadIdx.x == 0) grad[k] += p;
      }
  } else {
    const double d = warp_total(part, nwarps);
    if (threadIdx.x == 32) s_coef2 = va.on ? va.kV / va.V0 * d : 0.0;
    if (blockIdx.x == 0)
      for (int k = 2; k < 4; k++) {
        const double p = warp_total(part + (size_t)(1 + k) * nwarps, nwarps);
        if (threadIdx.x == 32) grad[k] += p;
      }
  }
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double f = 0, g = 0, dg = 0;
  if (i < 3 * nv) {
    const int v = i / 3, k = i - 3 * v;
    for (int e = vf_start[v]; e < vf_start[v + 1]; e++) {
      const int fcr = vf_list[e];
      f += corner[3 * (size_t)fcr + k];
      g += fn[3 * (size_t)(fcr / 3) + k];
      dg += dn[3 * (size_t)(fcr / 3) + k];
    }
  }
  __syncthreads();
  if (i < 3 * nv) lam_q[i] += fma(-s_coef2, g, fma(-s_coef, dg, f));
}

// --- immersed-boundary transposes ------------------------------------------------------

struct LatArgs {
  int nx, ny, nz, walls;
  size_t ncell;
  FastDiv dx, dy;             // by nx, by ny
  double rho0, omega, gamma;  // 1/tau, 1 - 1/(2 tau)
  double g[3];
  int has_g;                  // the body force is not zero
  double ub[3], ut[3];        // wall velocities
  double wb[19], wt[19];      // moving-wall terms of the bounce-back (deviation units)
};

// z kind of a node: 0 fluid, 1 bottom wall, 2 top wall, -1 beyond the array (reading R9).
__device__ __forceinline__ int zkind(int z, const LatArgs &L) {
  if (!L.walls) return 0;
  if (z < 0 || z >= L.nz) return -1;
  if (z == 0) return 1;
  if (z == L.nz - 1) return 2;
  return 0;
}
__device__ __forceinline__ int wrapi(int a, int n) {
  if ((unsigned)a < (unsigned)n) return a;
  const int r = a % n;
  return r < 0 ? r + n : r;
}

// A node and its neighbours' offsets along each axis, at 1 - c for a source x - c.
struct Node {
  size_t n, zo[3], yo[3];
  int xo[3], z;
  bool below, above;  // a link up starts at the bottom wall, one down at the top wall
};
__device__ __forceinline__ Node node_at(size_t n, const LatArgs &L) {
  Node d;
  d.n = n;
  // (node numbers beyond 2^31 take the plain division)
  const size_t row = n < ((size_t)1 << 31) ? (size_t)L.dx.div((int)n) : n / L.nx;
  const int x = (int)(n - row * L.nx);
  const int z = row < ((size_t)1 << 31) ? L.dy.div((int)row) : (int)(row / L.ny);
  const int y = (int)(row - (size_t)z * L.ny);
  d.z = z;
  d.xo[0] = x == 0 ? L.nx - 1 : x - 1;
  d.xo[1] = x;
  d.xo[2] = x == L.nx - 1 ? 0 : x + 1;
  d.yo[0] = (size_t)(y == 0 ? L.ny - 1 : y - 1) * L.nx;
  d.yo[1] = (size_t)y * L.nx;
  d.yo[2] = (size_t)(y == L.ny - 1 ? 0 : y + 1) * L.nx;
  const size_t plane = (size_t)L.nx * L.ny;
  d.zo[0] = (size_t)(z == 0 ? L.nz - 1 : z - 1) * plane;
  d.zo[1] = (size_t)z * plane;
  d.zo[2] = (size_t)(z == L.nz - 1 ? 0 : z + 1) * plane;
  d.below = L.walls && z == 1;
  d.above = L.walls && z == L.nz - 2;
  return d;
}
// Source of the pulled population i at node d: element index into P (i-th array); a link from a
// wall bounces back: population opp(i) at the same node, plus the wall term.
__device__ __forceinline__ bool bounced(const Node &d, int i) {
  return (cz(i) > 0 && d.below) || (cz(i) < 0 && d.above);
}
__device__ __forceinline__ size_t pull_source(const Node &d, int i, const LatArgs &L) {
  if (bounced(d, i)) return (size_t)opp(i) * L.ncell + d.n;
  return (size_t)i * L.ncell + d.zo[1 - cz(i)] + d.yo[1 - cy(i)] + d.xo[1 - cx(i)];
}

// Post-streaming populations (deviations) at a fluid node from the post-collision populations P
// as stored, in the arithmetic type A of the forward state: double for FP64 contexts; float for
// FP32 contexts, whose forward step ran in float (the reverse pass linearises the double-precision
// step about that trajectory; its rho and u are formed in float, like the forward step's, and the
// adjoint arithmetic itself stays double).
template <typename A, typename T>
__device__ __forceinline__ void pull_dev(const T *__restrict__ P, const Node &d, const LatArgs &L,
                                         A f[Q]) {
#pragma unroll
  for (int i = 0; i < Q; i++) {
    f[i] = (A)P[pull_source(d, i, L)];
    if (bounced(d, i)) f[i] += (A)(cz(i) > 0 ? L.wb[i] : L.wt[i]);
  }
}

// Velocity (Guo shift with the total force Ft) of deviations f; returns rho.
template <typename A>
__device__ __forceinline__ A velocity(const A f[Q], const A Ft[3], A rho0, A u[3]) {
  A drho, j[3];
  node_moments(f, drho, j);
  const A rho = rho0 + drho;
  const A ir = reciprocal(rho);
  for (int k = 0; k < 3; k++) u[k] = (j[k] + A(0.5) * Ft[k]) * ir;
  return rho;
}

// Velocity and density after streaming at a node.
struct alignas(32) NodeU {
  double x, y, z, rho;
};

// The per-vertex passes run sixteen lanes per vertex: lane l holds the stencil row (dy, dz) =
// (l & 3, l >> 2), its four nodes along x one after another. Two rows' factors are shared by all
// four nodes, so a vertex costs a third of the FP64 instructions of a lane per node pair.
struct Row {
  int v, z, kind;
  size_t base;   // of node (0, y, z)
  double wy, wz, dwy, dwz;
};
__device__ __forceinline__ Row row_of(const Stencil &s, int v, const LatArgs &L) {
  Row r;
  const int l = threadIdx.x & 15, dy = l & 3, dz = l >> 2;
  r.v = v;
  r.z = s.base[2] + dz;
  r.kind = zkind(r.z, L);
  r.base = ((size_t)wrapi(r.z, L.nz) * L.ny + wrapi(s.base[1] + dy, L.ny)) * L.nx;
  r.wy = s.w[1][dy];
  r.wz = s.w[2][dz];
  r.dwy = s.dw[1][dy];
  r.dwz = s.dw[2][dz];
  return r;
}
// Sum over the sixteen lanes of a vertex.
__device__ __forceinline__ double half_sum(double x) {
  for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
// Sums over the sixteen lanes of a vertex of 2 N values: the first step exchanges halves of the
// values between two halves of the lanes, so each lane goes on with N of them. Lanes with
// (l & 8) == 0 return the sums of v[0 .. N-1], the others of v[N .. 2N-1].
template <int N>
__device__ __forceinline__ void half_sums(const double v[2 * N], double out[N]) {
  const bool up = threadIdx.x & 8;
#pragma unroll
  for (int k = 0; k < N; k++) {
    const double other = __shfl_xor_sync(0xffffffffu, up ? v[k] : v[N + k], 8);
    out[k] = (up ? v[N + k] : v[k]) + other;
  }
  for (int o = 4; o > 0; o >>= 1)
#pragma unroll
    for (int k = 0; k < N; k++) out[k] += __shfl_xor_sync(0xffffffffu, out[k], o);
}

// Spreading at q_n onto the fluid nodes (Eq. 13): F += W phi, and the nodes' marks are set. F and
// the marks are zero on entry: the spreading transpose that last used them cleared them.
__global__ void adj_spread_kernel(int nv, const Stencil *__restrict__ st,
                                  const double *__restrict__ phi, LatArgs L, double *__restrict__ F,
                                  unsigned char *__restrict__ mark) {
  const int v = (blockIdx.x * blockDim.x + threadIdx.x) >> 4;
  if (v >= nv) return;
  const Stencil &s = st[v];
  const Row r = row_of(s, v, L);
  if (r.kind != 0) return;  // wall layer: force dropped; beyond: skipped
  const double wyz = r.wy * r.wz;
  const double ph[3] = {wyz * phi[3 * v], wyz * phi[3 * v + 1], wyz * phi[3 * v + 2]};
  for (int dx = 0; dx < 4; dx++) {
    const size_t n = r.base + wrapi(s.base[0] + dx, L.nx);
    const double w = s.w[0][dx];
    mark[n] = 1;
    for (int k = 0; k < 3; k++) atomicAdd(&F[3 * n + k], w * ph[k]);
  }
}

// Velocity and density after streaming at the marked nodes, U = (u, rho), from the post-collision
// populations P_{n+1} and the step's total force g + F.
template <typename T>
__global__ void adj_moments_kernel(const T *__restrict__ P, const double *__restrict__ F,
                                   const unsigned char *__restrict__ mark, LatArgs L,
                                   NodeU *__restrict__ U) {
  const size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (n >= L.ncell || !mark[n]) return;
  const Node d = node_at(n, L);
  using A = T;  // the forward state's arithmetic type
  A f[Q], u[3];
  pull_dev<A>(P, d, L, f);
  const A Ft[3] = {(A)(L.g[0] + F[3 * n]), (A)(L.g[1] + F[3 * n + 1]), (A)(L.g[2] + F[3 * n + 2])};
  const A rho = velocity<A>(f, Ft, (A)L.rho0, u);
  U[n] = NodeU{(double)u[0], (double)u[1], (double)u[2], (double)rho};
}

// Interpolation^T: lam_qn_v = lam_v + sum_x (u(x) . lam_v) dW/dq_v, and lam_u(x) += W lam_v
// on the fluid nodes, with u(x) the velocity of the step (the wall velocity on wall layers).
__global__ void adj_interp_t_kernel(int nv, const Stencil *__restrict__ st,
                                    const double *__restrict__ lam, const NodeU *__restrict__ U,
                                    LatArgs L, double *__restrict__ lam_qn,
                                    double *__restrict__ lam_u) {
  const int v = (blockIdx.x * blockDim.x + threadIdx.x) >> 4;
  double c[3] = {0, 0, 0}, l[3] = {0, 0, 0};
  if (v < nv) {
    const Stencil &s = st[v];
    const Row r = row_of(s, v, L);
    for (int k = 0; k < 3; k++) l[k] = lam[3 * v + k];
    if (r.kind >= 0) {
      const double wyz = r.wy * r.wz;
      double p = 0.0, dp = 0.0;  // sum over x of (u . lam) wx, (u . lam) dwx
      if (r.kind > 0) {
        const double *uw = r.kind == 1 ? L.ub : L.ut;
        const double ul = dot3(uw, l);
        for (int dx = 0; dx < 4; dx++) {
          p = fma(ul, s.w[0][dx], p);
          dp = fma(ul, s.dw[0][dx], dp);
        }
      } else {
        const double lw[3] = {wyz * l[0], wyz * l[1], wyz * l[2]};
        for (int dx = 0; dx < 4; dx++) {
          const size_t n = r.base + wrapi(s.base[0] + dx, L.nx);
          const NodeU un = U[n];
          const double u[3] = {un.x, un.y, un.z};
          const double ul = dot3(u, l), w = s.w[0][dx];
          p = fma(ul, w, p);
          dp = fma(ul, s.dw[0][dx], dp);
          for (int k = 0; k < 3; k++) atomicAdd(&lam_u[3 * n + k], w * lw[k]);
        }
      }
      c[0] = dp * wyz;
      c[1] = p * (r.dwy * r.wz);
      c[2] = p * (r.wy * r.dwz);
    }
  }
  for (int k = 0; k < 3; k++) c[k] = half_sum(c[k]);
  const int k = threadIdx.x & 15;
  if (v < nv && k < 3) lam_qn[3 * v + k] = k == 0 ? l[0] + c[0] : k == 1 ? l[1] + c[1] : l[2] + c[2];
}

// Velocity moments^T at the marked nodes with lam_u != 0: the adjoint of each pulled population,
// (c_i - u) . lam_u / rho, added to its source in lam_P (its force part, lam_u / (2 rho), is added
// by the collision transpose, which also clears lam_u).
__global__ void adj_velocity_t_kernel(const double *__restrict__ lam_u,
                                      const unsigned char *__restrict__ mark,
                                      const NodeU *__restrict__ U, LatArgs L,
                                      double *__restrict__ lam_P) {
  const size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (n >= L.ncell || !mark[n]) return;
  const double lu[3] = {lam_u[3 * n], lam_u[3 * n + 1], lam_u[3 * n + 2]};
  if (lu[0] == 0.0 && lu[1] == 0.0 && lu[2] == 0.0) return;
  const Node d = node_at(n, L);
  const NodeU un = U[n];
  const double ir = reciprocal(un.rho);
  const double l[3] = {lu[0] * ir, lu[1] * ir, lu[2] * ir};
  const double u[3] = {un.x, un.y, un.z};
  const double m = -dot3(u, l);
#pragma unroll
  for (int i = 0; i < Q; i++) {
    double a = m;
    if (cx(i)) a += cx(i) > 0 ? l[0] : -l[0];
    if (cy(i)) a += cy(i) > 0 ? l[1] : -l[1];
    if (cz(i)) a += cz(i) > 0 ? l[2] : -l[2];
    lam_P[pull_source(d, i, L)] += a;  // each (source, direction) has one puller
  }
}

// Collision^T and streaming^T at every fluid node. mu = lam_P1 at the node is the adjoint of
// the post-collision populations out_i = f_i - omega (f_i - feq_i(rho, u)) + S_i(u, F) of the
// pulled pre-collision f (BGK with Guo forcing). With the moments of mu,
//   m0 = sum w_i mu_i, m1 = sum w_i mu_i c_i, M2 = sum w_i mu_i c_i c_i^T, N = 9 M2 - 3 m0 I,
// the vector-Jacobian product is
//   lam_f_j = (1 - omega) mu_j + A - b . u + b . c_j,
//   A = omega (m0 + u . (3 m1 + N u / 2))                  (d/d rho)
//   b = omega G + gamma N Ft / rho,  G = 3 m1 + N u        (d/d u, over rho)
//   lam_F = b / 2 + gamma G                                 (d/d F)
// (u depends on f through (sum c f + Ft/2)/rho; Ft = g + F). lam_f_j goes to the source of
// the pulled population (a permutation: written once). lam_F is needed at the marked nodes only,
// and Ft is zero elsewhere without a body force. The velocity-moment transpose of step n+1 adds
// lam_u / (2 rho_{n+1}) to lam_F here, and lam_u is cleared for the next step. About 135 double
// operations per node (the moments scaled by 36, opposite directions in pairs) against 220.
template <typename T>
__global__ void __launch_bounds__(128) adj_collide_t_kernel(
    const double *__restrict__ lam_P1, const T *__restrict__ Pn, const double *__restrict__ F,
    const unsigned char *__restrict__ mark, const NodeU *__restrict__ U1,
    double *__restrict__ lam_u, LatArgs L, int fresh, double *__restrict__ lam_P0,
    double *__restrict__ lam_F) {
  const size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (n >= L.ncell) return;
  const Node d = node_at(n, L);
  if (zkind(d.z, L) != 0) return;
  using A = T;  // the forward state's arithmetic type
  const bool marked = mark[n];
  A f[Q], ua[3];
  if (fresh) {
#pragma unroll
    for (int i = 0; i < Q; i++) f[i] = (A)Pn[(size_t)i * L.ncell + n];
  } else {
    pull_dev<A>(Pn, d, L, f);
  }
  double mu[Q];
#pragma unroll
  for (int i = 0; i < Q; i++) mu[i] = lam_P1[(size_t)i * L.ncell + n];
  double Ft[3] = {L.g[0], L.g[1], L.g[2]};
  if (marked)
    for (int k = 0; k < 3; k++) Ft[k] += F[3 * n + k];
  const A Fta[3] = {(A)Ft[0], (A)Ft[1], (A)Ft[2]};
  const A rho = velocity<A>(f, Fta, (A)L.rho0, ua);
  const double u[3] = {(double)ua[0], (double)ua[1], (double)ua[2]};
  // 36 times the moments
  double s[9], e[9];
#pragma unroll
  for (int p = 0; p < 9; p++) {
    s[p] = mu[2 * p + 1] + mu[2 * p + 2];
    e[p] = mu[2 * p + 1] - mu[2 * p + 2];
  }
  const double pxy = s[3] + s[4], pxz = s[5] + s[6], pyz = s[7] + s[8];
  const double M0 = fma(12.0, mu[0], fma(2.0, s[0] + s[1] + s[2], pxy + pxz + pyz));
  const double c0 = M0 * (-1.0 / 12.0);
  const double Nxx = fma(0.25, fma(2.0, s[0], pxy + pxz), c0);
  const double Nyy = fma(0.25, fma(2.0, s[1], pxy + pyz), c0);
  const double Nzz = fma(0.25, fma(2.0, s[2], pxz + pyz), c0);
  const double Nxy = 0.25 * (s[3] - s[4]), Nxz = 0.25 * (s[5] - s[6]), Nyz = 0.25 * (s[7] - s[8]);
  const double t[3] = {fma(2.0, e[0], (e[3] + e[4]) + (e[5] + e[6])) * (1.0 / 12.0),  // 3 m1
                       fma(2.0, e[1], (e[3] - e[4]) + (e[7] + e[8])) * (1.0 / 12.0),
                       fma(2.0, e[2], (e[5] - e[6]) + (e[7] - e[8])) * (1.0 / 12.0)};
  const double Nu[3] = {fma(Nxx, u[0], fma(Nxy, u[1], Nxz * u[2])),
                        fma(Nxy, u[0], fma(Nyy, u[1], Nyz * u[2])),
                        fma(Nxz, u[0], fma(Nyz, u[1], Nzz * u[2]))};
  double G[3], b[3], acc = M0 * (1.0 / 36.0);
  for (int k = 0; k < 3; k++) {
    acc = fma(u[k], fma(0.5, Nu[k], t[k]), acc);
    G[k] = t[k] + Nu[k];
    b[k] = L.omega * G[k];
  }
  if (marked || L.has_g) {
    const double gr = L.gamma * reciprocal((double)rho);
    b[0] = fma(gr, fma(Nxx, Ft[0], fma(Nxy, Ft[1], Nxz * Ft[2])), b[0]);
    b[1] = fma(gr, fma(Nxy, Ft[0], fma(Nyy, Ft[1], Nyz * Ft[2])), b[1]);
    b[2] = fma(gr, fma(Nxz, Ft[0], fma(Nyz, Ft[1], Nzz * Ft[2])), b[2]);
  }
  if (marked) {
    double lf[3];
    for (int k = 0; k < 3; k++) lf[k] = fma(0.5, b[k], L.gamma * G[k]);
    const double lu[3] = {lam_u[3 * n], lam_u[3 * n + 1], lam_u[3 * n + 2]};
    if (lu[0] != 0.0 || lu[1] != 0.0 || lu[2] != 0.0) {
      const double h = 0.5 * reciprocal(U1[n].rho);
      for (int k = 0; k < 3; k++) {
        lf[k] = fma(lu[k], h, lf[k]);
        lam_u[3 * n + k] = 0.0;
      }
    }
    for (int k = 0; k < 3; k++) lam_F[3 * n + k] = lf[k];
  }
  double s0 = L.omega * acc;
  for (int k = 0; k < 3; k++) s0 = fma(-u[k], b[k], s0);
  const double om1 = 1.0 - L.omega;
  mu[0] = fma(om1, mu[0], s0);
#pragma unroll
  for (int i = 1; i < Q; i += 2) {  // c.b changes sign between opposite directions
    double cb = 0.0;
    if (cx(i)) cb = cx(i) > 0 ? b[0] : -b[0];
    if (cy(i)) cb = cx(i) ? (cy(i) > 0 ? cb + b[1] : cb - b[1]) : (cy(i) > 0 ? b[1] : -b[1]);
    if (cz(i)) cb = cx(i) || cy(i) ? (cz(i) > 0 ? cb + b[2] : cb - b[2]) : (cz(i) > 0 ? b[2] : -b[2]);
    mu[i] = fma(om1, mu[i], s0 + cb);
    mu[i + 1] = fma(om1, mu[i + 1], s0 - cb);
  }
#pragma unroll
  for (int i = 0; i < Q; i++)  // a permutation: written once
    lam_P0[fresh ? (size_t)i * L.ncell + n : pull_source(d, i, L)] = mu[i];
}

// Spreading^T: lam_phi_v = sum_x W lam_F(x) over the fluid nodes, and
// lam_qn_v += sum_x (phi_v . lam_F(x)) dW/dq_v. With row sums over x, a = sum wx lam_F and
// d = sum dwx lam_F, a row gives wy wz a, and wy wz phi.d, dwy wz phi.a, wy dwz phi.a. The step's
// force field F and the marks are no longer needed afterwards: cleared here for the next step that
// uses them.
__global__ void adj_spread_t_kernel(int nv, const Stencil *__restrict__ st,
                                    const double *__restrict__ phi, const double *__restrict__ lam_F,
                                    LatArgs L, double *__restrict__ lam_phi,
                                    double *__restrict__ lam_qn, double *__restrict__ F,
                                    unsigned char *__restrict__ mark) {
  const int v = (blockIdx.x * blockDim.x + threadIdx.x) >> 4;
  double c[6] = {0, 0, 0, 0, 0, 0};
  if (v < nv) {
    const Stencil &s = st[v];
    const Row r = row_of(s, v, L);
    if (r.kind == 0) {
      double a[3] = {0, 0, 0}, g[3] = {0, 0, 0};
      for (int dx = 0; dx < 4; dx++) {
        const size_t n = r.base + wrapi(s.base[0] + dx, L.nx);
        const double w = s.w[0][dx], dw = s.dw[0][dx];
        for (int k = 0; k < 3; k++) {
          const double lf = lam_F[3 * n + k];
          a[k] = fma(w, lf, a[k]);
          g[k] = fma(dw, lf, g[k]);
          F[3 * n + k] = 0.0;
        }
        mark[n] = 0;
      }
      const double ph[3] = {phi[3 * v], phi[3 * v + 1], phi[3 * v + 2]};
      const double pa = dot3(ph, a), wyz = r.wy * r.wz;
      for (int k = 0; k < 3; k++) c[k] = wyz * a[k];
      c[3] = wyz * dot3(ph, g);
      c[4] = pa * (r.dwy * r.wz);
      c[5] = pa * (r.wy * r.dwz);
    }
  }
  double o[3];
  half_sums<3>(c, o);
  if (v >= nv) return;
  const int k = threadIdx.x & 7;
  const double x = k == 0 ? o[0] : k == 1 ? o[1] : o[2];
  if (k < 3) {
    if (threadIdx.x & 8) lam_qn[3 * v + k] += x;
    else lam_phi[3 * v + k] = x;
  }
}

// --- host side ---------------------------------------------------------------------------

// What the forward pieces of a reverse step leave for its transposes; two sets, so that those of
// the next reverse step are prepared on a stream of their own beside this step's transposes.
struct Pieces {
  double *fc = nullptr, *fn = nullptr, *vpart = nullptr, *phi = nullptr, *F = nullptr;
  unsigned char *mark = nullptr;  // [ncell] node of some vertex's stencil (fluid)
  NodeU *U = nullptr;             // [ncell] velocity and density after streaming, marked nodes
  Stencil *st = nullptr;          // [nv] stencils of the step's positions
  cudaEvent_t ready = nullptr, free = nullptr;
};

struct Adjoint {
  int nsteps = 0, every = 0, first_fresh = 0;
  bool recorded = false;              // the checkpoints hold a whole run
  bool work = false;                  // the work arrays are there
  std::vector<void *> ck_P;           // populations at steps 0, K, 2K, ..., nsteps (storage type)
  std::vector<double *> ck_q;         // positions at the same steps
  std::vector<void *> seg_P;          // states of the segment being reversed (storage type)
  std::vector<double *> seg_q;
  double *lam_P[2] = {nullptr, nullptr};
  double *lam_q = nullptr, *lam_qn = nullptr, *lam_phi = nullptr, *lam_F = nullptr,
         *lam_u = nullptr;
  double *fj = nullptr, *dn = nullptr, *part = nullptr, *grad = nullptr;
  Pieces pieces[2];
  cudaStream_t side = nullptr;        // stream of the forward pieces
};

// Free the work arrays of a gradient (also a part of them, after a failed allocation).
void free_work(Adjoint *a) {
  auto f = [](auto *&p) {
    if (p) cudaFree(p);
    p = nullptr;
  };
  if (a->side) cudaStreamSynchronize(a->side);
  f(a->lam_P[0]); f(a->lam_P[1]); f(a->lam_q); f(a->lam_qn); f(a->lam_phi); f(a->lam_F);
  f(a->lam_u); f(a->fj); f(a->dn); f(a->part); f(a->grad);
  for (Pieces &p : a->pieces) {
    f(p.fc); f(p.fn); f(p.vpart); f(p.phi); f(p.F); f(p.mark); f(p.U); f(p.st);
    if (p.ready) cudaEventDestroy(p.ready);
    if (p.free) cudaEventDestroy(p.free);
    p.ready = p.free = nullptr;
  }
  if (a->side) cudaStreamDestroy(a->side);
  a->side = nullptr;
  a->work = false;
}

void free_all(Adjoint *a) {
  free_work(a);
  for (void *p : a->ck_P) cudaFree(p);
  for (double *p : a->ck_q) cudaFree(p);
  for (size_t m = 1; m < a->seg_P.size(); m++) cudaFree(a->seg_P[m]);  // ([0] is a checkpoint)
  for (double *p : a->seg_q) cudaFree(p);
  delete a;
}

int afail(Ctx &c, int code, const std::string &m) {
  c.err = m;
  return code;
}

// (the error is taken: the next launch's check would find it)
#define ADJ_TRY(c, expr)                                                                   \
  do {                                                                                     \
    cudaError_t e_ = (expr);                                                               \
    if (e_ != cudaSuccess) {                                                               \
      cudaGetLastError();                                                                  \
      return iblb::afail((c), e_ == cudaErrorMemoryAllocation ? IBLB_ENOMEM : IBLB_ECUDA,   \
                   std::string(#expr) + ": " + cudaGetErrorString(e_));                    \
    }                                                                                      \
  } while (0)

cudaError_t dmalloc(double **p, size_t n) {
  *p = nullptr;
  return cudaMalloc((void **)p, (n ? n : 1) * sizeof(double));
}

// Make P hold nP population states and q hold nq positions, keeping what is there.
int resize_states(Ctx &c, std::vector<void *> &P, std::vector<double *> &q, int nP, int nq) {
  while ((int)P.size() > nP) {
    cudaFree(P.back());
    P.pop_back();
  }
  while ((int)q.size() > nq) {
    cudaFree(q.back());
    q.pop_back();
  }
  while ((int)P.size() < nP) {
    void *p = nullptr;
    ADJ_TRY(c, cudaMalloc(&p, (size_t)Q * c.ncell * c.pop_size));
    P.push_back(p);
  }
  while ((int)q.size() < nq) {
    double *p = nullptr;
    ADJ_TRY(c, dmalloc(&p, (size_t)3 * c.nv));
    q.push_back(p);
  }
  return 0;
}

FaceArgs face_args(const Ctx &c) {
  FaceArgs A;
  A.nf = c.nf;
  A.faces = c.faces;
  A.fref = c.fref;
  for (int k = 0; k < 3; k++) {
    A.centre[k] = c.centre[k];
    A.alpha[k] = c.iface.alpha[k];
  }
  A.eps = c.iface.eps;
  A.xi = c.iface.xi;
  A.lj = c.iface.wall_force_on && c.has_walls;
  A.zb = 0.5;
  A.zt = c.nz - 1.5;
  return A;
}

LatArgs lat_args(const Ctx &c) {
  LatArgs L;
  L.nx = c.nx; L.ny = c.ny; L.nz = c.nz; L.walls = c.has_walls;
  L.ncell = c.ncell;
  L.dx = fast_div(c.nx);
  L.dy = fast_div(c.ny);
  L.has_g = c.g[0] != 0.0 || c.g[1] != 0.0 || c.g[2] != 0.0;
  L.rho0 = c.rho0;
  L.omega = 1.0 / c.tau;
  L.gamma = 1.0 - 0.5 / c.tau;
  for (int k = 0; k < 3; k++) {
    L.g[k] = c.g[k];
    L.ub[k] = c.ub[k];
    L.ut[k] = c.ut[k];
  }
  for (int i = 0; i < Q; i++) {
    const double cb = cx(i) * c.ub[0] + cy(i) * c.ub[1] + cz(i) * c.ub[2];
    const double ct = cx(i) * c.ut[0] + cy(i) * c.ut[1] + cz(i) * c.ut[2];
    L.wb[i] = 6.0 * wgt(i) * c.rho0 * cb;
    L.wt[i] = 6.0 * wgt(i) * c.rho0 * ct;
  }
  return L;
}

// A checkpoint: the populations as stored (so that restoring them continues bit for bit) and
// the positions.
int snapshot_raw(Ctx &c, void *P, double *q) {
  ADJ_TRY(c, cudaMemcpyAsync(P, c.f[c.cur], (size_t)Q * c.ncell * c.pop_size,
                             cudaMemcpyDeviceToDevice, c.stream));
  ADJ_TRY(c, cudaMemcpyAsync(q, c.q, (size_t)3 * c.nv * sizeof(double), cudaMemcpyDeviceToDevice,
                             c.stream));
  return 0;
}

// n steps queued with the health check of iblb_step at their end
int run_steps(Ctx &c, int n) {
  ADJ_TRY(c, cudaMemsetAsync(c.counters + 3, 0, sizeof(int), c.stream));
  if (int rc = enqueue_steps(c, n)) return rc;
  int hw = 0;
  ADJ_TRY(c, cudaMemcpyAsync(&hw, c.counters + 3, sizeof(int), cudaMemcpyDeviceToHost, c.stream));
  ADJ_TRY(c, cudaStreamSynchronize(c.stream));
  return health_status(c, hw);
}

// Recompute a segment from checkpoint `s`: `len` steps, state m + 1 written by its step straight
// into seg_P[m + 1] (the step reads one population array and writes the other, and these two are
// lent to the context in place of its own), positions copied to seg_q; everything queued, one
// health check at the end. State 0 is the checkpoint itself.
int recompute_segment(Ctx &c, Adjoint *a, int s, int len, int fresh) {
  void *const own[2] = {c.f[0], c.f[1]};
  a->seg_P[0] = a->ck_P[s];
  ADJ_TRY(c, cudaMemsetAsync(c.counters + 3, 0, sizeof(int), c.stream));
  int rc = restore_positions(c, a->ck_q[s], fresh);
  for (int m = 0; m < len && rc == 0; m++) {
    cudaError_t e = cudaMemcpyAsync(a->seg_q[m], c.q, (size_t)3 * c.nv * sizeof(double),
                                    cudaMemcpyDeviceToDevice, c.stream);
    if (e != cudaSuccess) rc = afail(c, IBLB_ECUDA, cudaGetErrorString(e));
    c.f[c.cur] = a->seg_P[m];
    c.f[c.cur ^ 1] = a->seg_P[m + 1];
    if (rc == 0) rc = enqueue_steps(c, 1);
  }
  c.f[0] = own[0];
  c.f[1] = own[1];
  if (rc) return rc;
  int hw = 0;
  ADJ_TRY(c, cudaMemcpyAsync(&hw, c.counters + 3, sizeof(int), cudaMemcpyDeviceToHost, c.stream));
  ADJ_TRY(c, cudaStreamSynchronize(c.stream));
  return health_status(c, hw);
}

int face_warps(const Ctx &c) { return (c.nf + 31) / 32; }

// Allocate the work arrays of a gradient; what a failure leaves is for free_work.
int allocate_work(Ctx &c, Adjoint *a) {
  const size_t pn = (size_t)Q * c.ncell, qn = (size_t)3 * c.nv;
  ADJ_TRY(c, dmalloc(&a->lam_P[0], pn));
  ADJ_TRY(c, dmalloc(&a->lam_P[1], pn));
  ADJ_TRY(c, dmalloc(&a->lam_q, qn));
  ADJ_TRY(c, dmalloc(&a->lam_qn, qn));
  ADJ_TRY(c, dmalloc(&a->lam_phi, qn));
  ADJ_TRY(c, dmalloc(&a->lam_F, 3 * c.ncell));
  ADJ_TRY(c, dmalloc(&a->lam_u, 3 * c.ncell));
  ADJ_TRY(c, dmalloc(&a->fj, (size_t)9 * c.nf));
  ADJ_TRY(c, dmalloc(&a->dn, (size_t)3 * c.nf));
  ADJ_TRY(c, dmalloc(&a->part, (size_t)5 * face_warps(c)));
  ADJ_TRY(c, dmalloc(&a->grad, 4));
  for (Pieces &p : a->pieces) {
    ADJ_TRY(c, dmalloc(&p.fc, (size_t)9 * c.nf));
    ADJ_TRY(c, dmalloc(&p.fn, (size_t)3 * c.nf));
    ADJ_TRY(c, dmalloc(&p.vpart, (size_t)face_warps(c)));
    ADJ_TRY(c, dmalloc(&p.phi, qn));
    ADJ_TRY(c, dmalloc(&p.F, 3 * c.ncell));
    ADJ_TRY(c, cudaMalloc((void **)&p.mark, c.ncell));
    ADJ_TRY(c, cudaMalloc((void **)&p.U, c.ncell * sizeof(NodeU)));
    ADJ_TRY(c, cudaMalloc((void **)&p.st, (size_t)c.nv * sizeof(Stencil)));
    ADJ_TRY(c, cudaEventCreateWithFlags(&p.ready, cudaEventDisableTiming));
    ADJ_TRY(c, cudaEventCreateWithFlags(&p.free, cudaEventDisableTiming));
  }
  ADJ_TRY(c, cudaStreamCreateWithFlags(&a->side, cudaStreamNonBlocking));
  a->work = true;
  return 0;
}

// Forward pieces of reverse step n at q_n, on the side stream: forces, volume, stencils, the
// spread force field, the moments of P_{n+1}. They depend on the recomputed states only.
template <typename T>
int forward_pieces(Ctx &c, Adjoint *a, Pieces &p, const double *qn, const T *Pn1) {
  const LatArgs L = lat_args(c);
  const VolArgs va{c.iface.volume_force_on, c.iface.kV, c.V0};
  const unsigned gf = (unsigned)((c.nf + kFaceThreads - 1) / kFaceThreads);
  const unsigned gv = (unsigned)((3L * c.nv + kVertexThreads - 1) / kVertexThreads);
  const unsigned gw = (unsigned)((16L * c.nv + 127) / 128);  // sixteen lanes per vertex
  const unsigned gn = (unsigned)((c.ncell + 255) / 256);
  cudaStream_t st = a->side;
  ADJ_TRY(c, cudaStreamWaitEvent(st, p.free, 0));
  adj_face_value_kernel<<<gf, kFaceThreads, 0, st>>>(face_args(c), qn, p.fc, p.fn, p.vpart);
  adj_vertex_value_kernel<<<gv, kVertexThreads, 0, st>>>(c.nv, face_warps(c), c.vf_start, c.vf_list,
                                                         p.fc, p.fn, p.vpart, va, qn, p.phi, p.st);
  adj_spread_kernel<<<gw, 128, 0, st>>>(c.nv, p.st, p.phi, L, p.F, p.mark);
  adj_moments_kernel<T><<<gn, 256, 0, st>>>(Pn1, p.F, p.mark, L, p.U);
  ADJ_TRY(c, cudaGetLastError());
  ADJ_TRY(c, cudaEventRecord(p.ready, st));
  return 0;
}

// Reverse step n: a->lam_q (of q_{n+1}) and a->lam_P[1] (of P_{n+1}) become those of q_n, P_n
// in a->lam_qn and a->lam_P[0] (swapped by the caller). Pn are stored populations (T). No scratch
// field needs clearing: F, the marks and lam_u are zero between steps (cleared by their last
// readers), lam_P0 is overwritten at every fluid node, lam_F at every marked one.
template <typename T>
int reverse_step(Ctx &c, Adjoint *a, Pieces &p, const T *Pn, const double *qn, int fresh) {
  const LatArgs L = lat_args(c);
  const VolArgs va{c.iface.volume_force_on, c.iface.kV, c.V0};
  const unsigned gf = (unsigned)((c.nf + kFaceThreads - 1) / kFaceThreads);
  const unsigned gv = (unsigned)((3L * c.nv + kVertexThreads - 1) / kVertexThreads);
  const unsigned gw = (unsigned)((16L * c.nv + 127) / 128);
  cudaStream_t st = c.stream;
  ADJ_TRY(c, cudaStreamWaitEvent(st, p.ready, 0));
  // interpolation^T, velocity^T, collision^T and streaming^T, spreading^T
  adj_interp_t_kernel<<<gw, 128, 0, st>>>(c.nv, p.st, a->lam_q, p.U, L, a->lam_qn, a->lam_u);
  adj_velocity_t_kernel<<<(unsigned)((c.ncell + 255) / 256), 256, 0, st>>>(a->lam_u, p.mark, p.U, L,
                                                                          a->lam_P[1]);
  adj_collide_t_kernel<T><<<(unsigned)((c.ncell + 127) / 128), 128, 0, st>>>(
      a->lam_P[1], Pn, p.F, p.mark, p.U, a->lam_u, L, fresh, a->lam_P[0], a->lam_F);
  adj_spread_t_kernel<<<gw, 128, 0, st>>>(c.nv, p.st, p.phi, a->lam_F, L, a->lam_phi, a->lam_qn, p.F,
                                          p.mark);
  // force Jacobian^T along lam_phi, and the parameter derivatives (added to grad)
  adj_face_tangent_kernel<<<gf, kFaceThreads, 0, st>>>(face_args(c), qn, a->lam_phi, a->fj, a->dn,
                                                       a->part);
  adj_vertex_tangent_kernel<<<gv, kVertexThreads, 0, st>>>(c.nv, face_warps(c), c.vf_start, c.vf_list,
                                                           a->fj, p.fn, a->dn, p.vpart, a->part, va,
                                                           a->lam_qn, a->grad);
  ADJ_TRY(c, cudaGetLastError());
  ADJ_TRY(c, cudaEventRecord(p.free, st));
  return 0;
}

// The reverse steps of a recomputed segment of len steps (seg_P[0] fresh: the run's first state).
template <typename T>
int reverse_segment(Ctx &c, Adjoint *a, int len, int first_fresh) {
  // the side stream starts after the recomputed states (and after what last used the pieces)
  for (Pieces &p : a->pieces) ADJ_TRY(c, cudaEventRecord(p.free, c.stream));
  auto prepare = [&](int m) {
    return forward_pieces<T>(c, a, a->pieces[m & 1], a->seg_q[m], (const T *)a->seg_P[m + 1]);
  };
  if (int rc = prepare(len - 1)) return rc;
  for (int m = len - 1; m >= 0; m--) {
    if (m > 0)
      if (int rc = prepare(m - 1)) return rc;
    if (int rc = reverse_step<T>(c, a, a->pieces[m & 1], (const T *)a->seg_P[m], a->seg_q[m],
                                 m == 0 && first_fresh))
      return rc;
    std::swap(a->lam_q, a->lam_qn);
    std::swap(a->lam_P[0], a->lam_P[1]);
  }
  return 0;
}

}  // namespace

void adjoint_free(Ctx &c) {
  if (c.adj) free_all((Adjoint *)c.adj);
  c.adj = nullptr;
}

}  // namespace iblb

using iblb::Ctx;

extern "C" {

int iblb_adjoint_record(iblb_ctx *h, int32_t nsteps, int32_t every) {
  if (!h) return IBLB_EINVAL;
  Ctx &c = h->c;
  if (c.precision != IBLB_FP64 && c.precision != IBLB_FP32)
    return iblb::afail(c, IBLB_EINVAL, "the adjoint needs an IBLB_FP64 or IBLB_FP32 context");
  if (c.nv == 0) return iblb::afail(c, IBLB_EINVAL, "no mesh has been added");
  if (nsteps < 1 || every < 1) return iblb::afail(c, IBLB_EINVAL, "nsteps and every must be >= 1");
  if (int rc = iblb::settle_health(c)) return rc;  // a failure of earlier iblb_step_async steps
  // the arrays of an earlier recording serve again (its states change in number only): allocating
  // and freeing them took 2 ms of a 60-step gradient. Released by iblb_adjoint_release.
  const int step = every < nsteps ? every : nsteps;
  const int nck = (nsteps + step - 1) / step + 1;
  if (!c.adj) c.adj = new iblb::Adjoint();
  auto *a = (iblb::Adjoint *)c.adj;
  a->recorded = false;
  int rc = iblb::resize_states(c, a->ck_P, a->ck_q, nck, nck);
  if (rc == IBLB_ENOMEM && (a->work || a->seg_P.size() > 1 || !a->seg_q.empty())) {
    // without the last gradient's arrays
    iblb::adjoint_free(c);
    c.adj = a = new iblb::Adjoint();
    rc = iblb::resize_states(c, a->ck_P, a->ck_q, nck, nck);
  }
  if (rc) return rc;
  a->nsteps = nsteps;
  a->every = step;
  a->first_fresh = c.fresh;
  ADJ_TRY(c, cudaStreamSynchronize(c.stream));
  if (int rc = iblb::snapshot_raw(c, a->ck_P[0], a->ck_q[0])) return rc;
  int done = 0;
  for (int k = 1; k < nck; k++) {
    const int n = nsteps - done < a->every ? nsteps - done : a->every;
    if (int rc = iblb::run_steps(c, n)) return rc;
    done += n;
    if (int rc = iblb::snapshot_raw(c, a->ck_P[k], a->ck_q[k])) return rc;
  }
  ADJ_TRY(c, cudaStreamSynchronize(c.stream));
  a->recorded = true;
  return IBLB_OK;
}

int iblb_adjoint_gradient(iblb_ctx *h, const double *dJdq, double *dJdtheta) {
  if (!h || !dJdq || !dJdtheta) return IBLB_EINVAL;
  Ctx &c = h->c;
  auto *a = (iblb::Adjoint *)c.adj;
  if (!a || !a->recorded)
    return iblb::afail(c, IBLB_EINVAL, "no trajectory recorded (iblb_adjoint_record)");
  if (int rc = iblb::settle_health(c)) return rc;
  const size_t pn = (size_t)iblb::Q * c.ncell, qn = (size_t)3 * c.nv;
  // work arrays (kept for later calls)
  if (!a->work)
    if (int rc = iblb::allocate_work(c, a)) {
      iblb::free_work(a);
      return rc;
    }
  // states 1 .. every of a segment and the positions 0 .. every - 1
  if (a->seg_P.empty()) a->seg_P.push_back(nullptr);
  if (int rc = iblb::resize_states(c, a->seg_P, a->seg_q, a->every + 1, a->every)) return rc;
  ADJ_TRY(c, cudaMemcpyAsync(a->lam_q, dJdq, qn * sizeof(double), cudaMemcpyHostToDevice, c.stream));
  ADJ_TRY(c, cudaMemsetAsync(a->lam_P[0], 0, pn * sizeof(double), c.stream));
  ADJ_TRY(c, cudaMemsetAsync(a->lam_P[1], 0, pn * sizeof(double), c.stream));
  // zero between reverse steps (each step leaves them so)
  for (iblb::Pieces &p : a->pieces) {
    ADJ_TRY(c, cudaMemsetAsync(p.F, 0, 3 * c.ncell * sizeof(double), c.stream));
    ADJ_TRY(c, cudaMemsetAsync(p.mark, 0, c.ncell, c.stream));
  }
  ADJ_TRY(c, cudaMemsetAsync(a->lam_u, 0, 3 * c.ncell * sizeof(double), c.stream));
  ADJ_TRY(c, cudaMemsetAsync(a->grad, 0, 4 * sizeof(double), c.stream));
  const int nseg = (int)a->ck_P.size() - 1;
  int rc = 0;
  for (int s = nseg - 1; s >= 0 && rc == 0; s--) {
    const int first = s * a->every;
    const int len = (a->nsteps - first) < a->every ? a->nsteps - first : a->every;
    const int first_fresh = s == 0 && a->first_fresh;
    rc = iblb::recompute_segment(c, a, s, len, first_fresh);
    if (rc == 0)
      rc = c.pop_size == sizeof(double) ? iblb::reverse_segment<double>(c, a, len, first_fresh)
                                        : iblb::reverse_segment<float>(c, a, len, first_fresh);
  }
  // back to the end of the recorded run, also after a failure: the recomputed states were lent to the
  // context, whose own arrays hold older ones
  const std::string why = c.err;
  const int back = iblb::restore_state(c, a->ck_P[nseg], a->ck_q[nseg], 0);
  if (rc) {
    c.err = why;
    return rc;
  }
  if (back) return back;
  ADJ_TRY(c, cudaMemcpyAsync(dJdtheta, a->grad, 4 * sizeof(double), cudaMemcpyDeviceToHost, c.stream));
  ADJ_TRY(c, cudaStreamSynchronize(c.stream));
  return IBLB_OK;
}

int iblb_adjoint_release(iblb_ctx *h) {
  if (!h) return IBLB_EINVAL;
  cudaStreamSynchronize(h->c.stream);
  iblb::adjoint_free(h->c);
  return IBLB_OK;
}

}  // extern "C"
