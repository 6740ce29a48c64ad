// Interface passes, device code: per-face forces (Eqs. 2, 17-19) with the double-precision volume sum,
// per-vertex gathering into nodal forces (Eq. 16) and binning by 4x4x4 source tile,
// spreading by owner-computes gather over the binned vertices (Eq. 13), interpolation and
// the Euler update (Eqs. 11-12). The active tiles of a step are marked beside its face forces.
//
// Arithmetic runs in the population type `real` (float or double); vertex positions, the
// enclosed volume V and V - V0 are always double.
#pragma once

#include <math.h>
#include <string.h>

#include "iblb_internal.cuh"

// Pointers that a kernel only reads, or that nothing else in it aliases: true of the kernels that
// are one pass each, not of the fused step kernel, whose passes read what earlier ones wrote (it
// defines this empty).
#ifndef IBLB_RO
#define IBLB_RO __restrict__
#endif

namespace iblb {
namespace {

struct Dims {
  int nx, ny, nz, has_walls, ntx, nty, ntz, max_slots;
  double zb, zt;              // wall planes
  double inx, iny, inz;       // 1/nx, 1/ny, 1/nz
};

Dims dims_of(const Ctx &c) {
  Dims d;
  d.nx = c.nx; d.ny = c.ny; d.nz = c.nz; d.has_walls = c.has_walls;
  d.ntx = c.ntx; d.nty = c.nty; d.ntz = c.ntz; d.max_slots = c.max_slots;
  d.zb = 0.5;
  d.zt = c.nz - 1.5;
  d.inx = 1.0 / c.nx;
  d.iny = 1.0 / c.ny;
  d.inz = 1.0 / c.nz;
  return d;
}

// i reduced to [0, n).
__device__ __forceinline__ int wrap_index(int i, int n) {
  if ((unsigned)i >= (unsigned)n) {
    i += i < 0 ? n : -n;
    if ((unsigned)i >= (unsigned)n) {  // positions are stored unwrapped
      i %= n;
      i += i < 0 ? n : 0;
    }
  }
  return i;
}

// Base node floor(p) - 1 of the delta stencil of coordinate p on an axis of n nodes, and
// r = p - floor(p). Periodic axes: the base in [0, n); a walled axis: not wrapped. Integer work
// but for one conversion each way and one subtraction (FP64 issues at 1/64 of the FP32 rate);
// the stencil and the tile marking take the same base.
__device__ __forceinline__ int stencil_base(double p, int n, double inv_n, bool periodic, double &r) {
  if ((__double2hiint(p) & 0x7fffffff) >= 0x41d00000)  // |p| >= 2^30 or no number
    p = periodic ? p - n * floor(p * inv_n) : fmin(fmax(p, -8.0), n + 8.0);
  const int i = __double2int_rd(p);
  r = p - (double)i;
  return periodic ? wrap_index(i - 1, n) : i - 1;
}

__device__ __forceinline__ float log_(float v) { return logf(v); }
__device__ __forceinline__ double log_(double v) { return log(v); }
__device__ __forceinline__ float sqrt_(float v) { return sqrtf(v); }
__device__ __forceinline__ double sqrt_(double v) { return sqrt(v); }

// Lennard-Jones force along z on a centroid at signed height dz above a wall plane (Eq. 19;
// d points from the wall foot point to the centroid).
template <typename real>
__device__ __forceinline__ real lj_fz(real dz, real eps48, real xi) {
  const real inv_d2 = real(1) / (dz * dz);
  const real s2 = xi * xi * inv_d2;
  const real s6 = s2 * s2 * s2;
  return eps48 * (s6 * s6 - real(0.5) * s6) * dz * inv_d2;
}

// Tiles covered along one axis by the stencil of coordinate p: t0 (lower) and t1 (upper,
// equal to t0 when the four nodes fall in one tile); `ok1` tells whether t1 is a distinct
// tile that exists. Periodic axes wrap; along a walled z axis tiles beyond the lattice are
// skipped (valid flags).
struct AxisTiles {
  int t0, t1;
  bool ok0, ok1;
};

// of an axis of n nodes (nt tiles)
__device__ __forceinline__ AxisTiles axis_tiles(double p, int n, int nt, double inv_n, bool periodic) {
  AxisTiles a;
  double r;
  const int b = stencil_base(p, n, inv_n, periodic, r);
  a.t0 = b >> 2;  // (arithmetic shift: floors)
  a.t1 = (b + 3) >> 2;
  if (periodic) {
    a.t1 = a.t1 >= nt ? a.t1 - nt : a.t1;
    a.ok0 = true;
    a.ok1 = a.t1 != a.t0;  // a short periodic axis may wrap onto the same tile
  } else {
    a.ok0 = a.t0 >= 0 && a.t0 < nt;
    a.ok1 = a.t1 != a.t0 && a.t1 >= 0 && a.t1 < nt;
  }
  return a;
}

// Tile e (bit k picks the upper tile along axis k) of the stencil described by ax, or -1.
__device__ __forceinline__ int stencil_tile(const AxisTiles ax[3], int e, const Dims &D) {
  int t[3];
  for (int k = 0; k < 3; k++) {
    const bool up = (e >> k) & 1;
    if (up ? !ax[k].ok1 : !ax[k].ok0) return -1;
    t[k] = up ? ax[k].t1 : ax[k].t0;
  }
  return (t[2] * D.nty + t[1]) * D.ntx + t[0];
}

// A tile map: the active tiles of one step's positions. Marked by the face pass of that step.
struct TileMap {
  int *tile_slot, *slot_tile, *nslots, *slot_count, *out_src, *health;
};

// Vertices that one warp marks.
constexpr int kMarkVertices = 8;

// Mark the tiles of the stencils of eight vertices by one warp (called together): lane l takes
// vertex v0 + l / 4 and, l % 4 = k < 3, its axis k; each lane then claims two of the vertex's (up
// to 8) tiles. The first claimant of a tile takes a new slot; a plain read first keeps the many
// vertices of an already-claimed tile off the atomics, and a lane's two claims are in flight
// together.
__device__ __forceinline__ void mark_vertices(const double *IBLB_RO q, int nv, int v0, const Dims &D,
                                              const TileMap &M) {
  const int lane = threadIdx.x & 31, k = lane & 3, v = v0 + (lane >> 2);
  int t0 = 0, t1 = 0, flags = 0;  // bit 0 / 1: ok0 / ok1 of the axis; bit 2: a number
  if (v < nv && k < 3) {
    const double p = q[3 * (size_t)v + k];
    if (p == p) {
      const int n = k == 0 ? D.nx : k == 1 ? D.ny : D.nz;
      const int nt = k == 0 ? D.ntx : k == 1 ? D.nty : D.ntz;
      const double inv = k == 0 ? D.inx : k == 1 ? D.iny : D.inz;
      const AxisTiles ax = axis_tiles(p, n, nt, inv, k < 2 || !D.has_walls);
      t0 = ax.t0;
      t1 = ax.t1;
      flags = (ax.ok0 ? 1 : 0) | (ax.ok1 ? 2 : 0) | 4;
    }
  }
  AxisTiles ax[3];
  int all = 4;
  for (int a = 0; a < 3; a++) {
    ax[a].t0 = __shfl_sync(0xffffffffu, t0, a, 4);
    ax[a].t1 = __shfl_sync(0xffffffffu, t1, a, 4);
    const int fl = __shfl_sync(0xffffffffu, flags, a, 4);
    ax[a].ok0 = fl & 1;
    ax[a].ok1 = fl & 2;
    all &= fl;
  }
  if (!all) return;  // (also beyond the last vertex)
  int t[2], won[2];
  for (int h = 0; h < 2; h++) {
    t[h] = stencil_tile(ax, k + 4 * h, D);
    won[h] = t[h] >= 0 && *(volatile int *)&M.tile_slot[t[h]] == -1;
  }
  for (int h = 0; h < 2; h++)
    if (won[h]) won[h] = atomicCAS(&M.tile_slot[t[h]], -1, -2) == -1;
  if (!(won[0] | won[1])) return;
  int s = atomicAdd(M.nslots, won[0] + won[1]);
  for (int h = 0; h < 2; h++) {
    if (!won[h]) continue;
    if (s < D.max_slots) {
      M.slot_tile[s] = t[h];
      M.slot_count[s] = 0;
      int4 *o = reinterpret_cast<int4 *>(M.out_src + 8 * (size_t)s);
      o[0] = o[1] = make_int4(-1, -1, -1, -1);
      atomicExch(&M.tile_slot[t[h]], s);
    } else {
      atomicOr(M.health, H_CAPACITY);
    }
    s++;
  }
}

// Per-face reference data in the population type, stored by component ([FGEO][nf]): A, B
// (edges), X0 - c, the reference centroid height above the bottom and the top wall plane, a
// pad, and the reference metric inverse H11, H12, H22 with the reference area A0 (rounded
// once on the host).
constexpr int FGEO = 16;

// Interface parameters of the face kernel, rounded once to the population type on the host
// (FP64 issues at 1/64 of the FP32 rate on this GPU: no per-face conversions).
template <typename real>
struct FaceParams {
  real a3;        // alpha3
  real cL0, cL1;  // 0.5 (alpha1 - alpha3), 0.25 (alpha1 + alpha2)
  real eps48, xi;
  int wall_on;
};

// K3a: one thread per face, in the population type. Writes the strain + wall force of each
// corner, the face's contribution (a x b)/6 to the volume gradient of each of its corners,
// and one partial sum per warp of V_j - V0_j, the change of the face's share of the volume.
// With reset != 0 (a step) it also marks the tile map of the current positions and clears the one
// that the previous step used. The marking runs beside the faces, by warps of its own: at the end
// of the interpolation its two rounds of atomics were the longest chain of the step.
//
// V_j = (x0 - c) . (a x b) / 6 for a fixed point c. Written with the displacements
// u_k = x_k - X_k from the reference shape (da = u1 - u0, db = u2 - u0, reference edges A, B)
// the change is
//   6 (V_j - V0_j) = u0 . (a x b) + (X0 - c) . (da x b + A x db),
// a sum of terms proportional to the displacement, so float arithmetic loses nothing to the
// cancellation between V and V0 (the per-warp partials are summed in double).
template <typename real>
struct FaceArgs {
  int nf;
  const int *faces;
  const Vec4<real> *disp;
  const real *fgeo;
  Vec4<real> *fcontrib, *fnorm;
  double *vol_partial;
  FaceParams<real> fp;
  Dims D;
  int *other_tile_slot;
  const int *other_slot_tile, *other_nslots;
  int reset;
  TileMap map;           // with reset: the map of the current positions, marked by this pass
  const double *q;
  int nv;
  int *ovf_count;
  unsigned *spill_bits;  // [spill_words] cleared here, before the vertex kernel bins
  int spill_words;
};

// Threads per block of K3a and K3b: few, so that a mesh of some thousand faces and vertices
// spreads over all SMs of the chain (each SM's FP64 unit and each warp's chain of loads, not
// memory, set their time): K3a of 81920 faces on 24 SMs 19 us against 27 with 256-thread blocks.
template <typename real>
struct FaceThreads {
  static constexpr int value = sizeof(real) == 4 ? 128 : 64;
};
constexpr int kVertexThreads = 128;

// Warps of K3a: one per kMarkVertices vertices to mark, then one per 32 faces.
template <typename real>
__device__ __forceinline__ int mark_warps(const FaceArgs<real> &A) {
  return A.reset ? (A.nv + kMarkVertices - 1) / kMarkVertices : 0;
}

// K3a for the warps first / 32, first / 32 + stride / 32, ... (`first`: of this thread; a warp's 32
// threads hold 32 consecutive ones and call it together).
template <typename real>
__device__ __forceinline__ void face_body(const FaceArgs<real> &A, int first, int stride) {
  const int nf = A.nf;
  const int *IBLB_RO faces = A.faces;
  const Vec4<real> *IBLB_RO disp = A.disp;
  const real *IBLB_RO fgeo = A.fgeo;
  Vec4<real> *IBLB_RO fcontrib = A.fcontrib;
  Vec4<real> *IBLB_RO fnorm = A.fnorm;
  double *IBLB_RO vol_partial = A.vol_partial;
  const FaceParams<real> fp = A.fp;
  const Dims D = A.D;
  const int lane = threadIdx.x & 31;
  const int marks = mark_warps(A), warps = marks + (nf + 31) / 32;
  for (int w = first >> 5; w < warps; w += stride >> 5) {
  if (w < marks) {
    mark_vertices(A.q, A.nv, kMarkVertices * w, D, A.map);
    continue;
  }
  const int j = 32 * (w - marks) + lane;
  real dvj = 0;
  if (j < nf) {
    const int iv[3] = {faces[3 * j], faces[3 * j + 1], faces[3 * j + 2]};
    real u[3][3];
    for (int c = 0; c < 3; c++) {
      const Vec4<real> d = disp[iv[c]];
      u[c][0] = d.x;
      u[c][1] = d.y;
      u[c][2] = d.z;
    }
    // A, B, X0 - c, centroid heights above the walls, pad, H11 H12 H22 A0; stored by
    // component ([FGEO][nf]), so that each load of a warp reads one contiguous row
    real geo[FGEO];
#pragma unroll
    for (int k = 0; k < FGEO; k++) geo[k] = k == 11 ? real(0) : fgeo[(size_t)k * nf + j];
    real A[3], B[3], X0c[3], da[3], db[3], a[3], b[3];
    for (int k = 0; k < 3; k++) {
      A[k] = geo[k];
      B[k] = geo[3 + k];
      X0c[k] = geo[6 + k];
      da[k] = u[1][k] - u[0][k];
      db[k] = u[2][k] - u[0][k];
      a[k] = A[k] + da[k];
      b[k] = B[k] + db[k];
    }
    const real H11 = geo[12], H12 = geo[13], H22 = geo[14], A0 = geo[15];
    const real G11 = a[0] * a[0] + a[1] * a[1] + a[2] * a[2];
    const real G12 = a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
    const real G22 = b[0] * b[0] + b[1] * b[1] + b[2] * b[2];
    const real detG = G11 * G22 - G12 * G12;
    const real L = log_(detG / (real(4) * A0 * A0));  // log(I2 + 1), det G0 = 4 A0^2
    // dE/da = paa a + pab b and dE/db = pab a + pbb b, with I1 = H11 G11 + 2 H12 G12 + H22 G22 - 2
    // and L = log det G + const
    const real eI = fp.a3 * A0;                                          // 2 dE/dI1
    const real eL = real(2) * A0 * (fp.cL0 + fp.cL1 * L) / detG;          // 2 dE/dL / det G
    const real paa = eI * H11 + eL * G22;
    const real pab = eI * H12 - eL * G12;
    const real pbb = eI * H22 + eL * G11;
    real f0[3], f1[3], f2[3];
    for (int k = 0; k < 3; k++) {
      const real ga = paa * a[k] + pab * b[k];
      const real gb = pab * a[k] + pbb * b[k];
      f1[k] = -ga;
      f2[k] = -gb;
      f0[k] = ga + gb;
    }
    if (fp.wall_on && D.has_walls) {
      // centroid height above each wall plane: reference height (from the set-up, in double)
      // plus the mean displacement
      const real uz = (u[0][2] + u[1][2] + u[2][2]) * real(1.0 / 3.0);
      const real third = (lj_fz<real>(geo[9] + uz, fp.eps48, fp.xi) +
                          lj_fz<real>(geo[10] + uz, fp.eps48, fp.xi)) *
                         real(1.0 / 3.0);
      f0[2] += third;
      f1[2] += third;
      f2[2] += third;
    }
    Vec4<real> *fc = fcontrib + 3 * (size_t)j;
    fc[0] = Vec4<real>{f0[0], f0[1], f0[2], real(0)};
    fc[1] = Vec4<real>{f1[0], f1[1], f1[2], real(0)};
    fc[2] = Vec4<real>{f2[0], f2[1], f2[2], real(0)};
    // For a closed surface the gradient of V at vertex i does not depend on the point about
    // which the tetrahedra are taken; with that point at x_i every face around i contributes
    // (a x b)/6, the same edge cross product for all three corners.
    const real n[3] = {a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2],
                       a[0] * b[1] - a[1] * b[0]};
    const real m[3] = {da[1] * b[2] - da[2] * b[1] + A[1] * db[2] - A[2] * db[1],
                       da[2] * b[0] - da[0] * b[2] + A[2] * db[0] - A[0] * db[2],
                       da[0] * b[1] - da[1] * b[0] + A[0] * db[1] - A[1] * db[0]};
    const real sixth = real(1.0 / 6.0);
    fnorm[j] = Vec4<real>{n[0] * sixth, n[1] * sixth, n[2] * sixth, real(0)};
    dvj = (u[0][0] * n[0] + u[0][1] * n[1] + u[0][2] * n[2] + X0c[0] * m[0] + X0c[1] * m[1] +
           X0c[2] * m[2]) * sixth;
  }
  // the warp's sum of V_j - V0_j in the population type, by a fixed shuffle tree
  real dw = dvj;
  for (int o = 16; o > 0; o >>= 1) dw += __shfl_down_sync(0xffffffffu, dw, o);
  if (lane == 0) vol_partial[j >> 5] = (double)dw;
  }
  if (first == 0) {
    A.ovf_count[0] = 0;  // vertices beyond their bucket (a count only)
    A.ovf_count[2] = 0;  // number of source tiles (counters[4])
    A.ovf_count[3] = 0;  // listed force pairs (counters[5]), appended by K4b
  }
  for (int w = first; w < A.spill_words; w += stride) A.spill_bits[w] = 0u;
  if (A.reset) {
    const int n_other = min(*A.other_nslots, D.max_slots);
    for (int s = first; s < n_other; s += stride) A.other_tile_slot[A.other_slot_tile[s]] = -1;
  }
}

template <typename real>
__global__ void __launch_bounds__(FaceThreads<real>::value) face_kernel(const FaceArgs<real> A) {
  face_body(A, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

template <typename real>
__global__ void __launch_bounds__(FaceThreads<real>::value) face_kernel_multi(
    const FaceArgs<real> *__restrict__ all, const int *__restrict__ start, int n) {
  const MultiBlock m = multi_block(start, n);
  face_body(all[m.inst], m.block * blockDim.x + threadIdx.x, m.nblocks * blockDim.x);
}

// kV (V - V0)/V0 from the per-warp partial sums of V - V0, by one warp in a fixed order;
// also returns V.
__device__ __forceinline__ double volume_coef(const double *IBLB_RO part, int n, double V0,
                                              double kV, int volume_on, double *V_out) {
  double s[4] = {0.0, 0.0, 0.0, 0.0};  // four chains of additions per lane
  for (int k0 = 0; k0 < n; k0 += 128)
#pragma unroll
    for (int c = 0; c < 4; c++) {
      const int k = k0 + 32 * c + (threadIdx.x & 31);
      if (k < n) s[c] += part[k];
    }
  double dv = (s[0] + s[1]) + (s[2] + s[3]);
  for (int o = 16; o > 0; o >>= 1) dv += __shfl_down_sync(0xffffffffu, dv, o);
  dv = __shfl_sync(0xffffffffu, dv, 0);
  if (V_out) *V_out = V0 + dv;
  return volume_on ? kV * dv / V0 : 0.0;
}

// One-dimensional Peskin weights of the four nodes floor(p)-1 .. floor(p)+2 (Eq. 15).
// With r = p - floor(p) and s = sqrt(1 + 4r - 4r^2) the four branches reduce to
// (3-2r-s)/8, (3-2r+s)/8, (1+2r+s)/8, (1+2r-s)/8, which sum to one.
template <typename real>
__device__ __forceinline__ void peskin_weights(real r, real w[4]) {
  const real s = sqrt_(real(1) + real(4) * r - real(4) * r * r);
  w[0] = (real(3) - real(2) * r - s) * real(0.125);
  w[1] = (real(3) - real(2) * r + s) * real(0.125);
  w[2] = (real(1) + real(2) * r + s) * real(0.125);
  w[3] = (real(1) + real(2) * r - s) * real(0.125);
}

// Faces around a vertex gathered with all loads in flight (icosphere valences are 5 and 6).
constexpr int GATHER_UNROLL = 8;

// K3b: four lanes per vertex. Gathers, in face order, the strain + wall force of the vertex's
// corners (phi, Eq. 16 without the volume term) and its volume gradient g = dV/dq_i; the
// volume term -kV (V - V0)/V0 g is added where the force is used (spreading, read-back),
// after V is complete. Then the delta stencil of the vertex and its binning into the source
// tile (the tile that holds its base node).
struct VolumeParams {
  double V0, kV;
  int volume_on, vol_blocks;
};

template <typename real>
struct VertexArgs {
  int nv;
  const int *vf_start, *vf_list;
  const Vec4<real> *fcontrib, *fnorm;
  const double *q;
  Vec4<real> *phi, *gvol;
  StencilRec<real> *stencil;
  int bin;
  const int *tile_slot;
  int *slot_count, *bucket, *ovf_count, *src_slot, *nsources, *health, *zero_counter;
  unsigned *spill_bits;  // bit i: vertex i did not fit in its tile's bucket
  const double *vol_partial;  // per-warp V_j - V0_j partials of the face kernel
  VolumeParams vp;
  real *vcoef;                // out: kV (V - V0)/V0 for the spreading pass
  Dims D;
};

// The step's scalars, by one warp: the volume-force coefficient (the spreading pass reads it),
// the volume health check, and the other map's tile counter zeroed.
template <typename real>
__device__ __forceinline__ void volume_task(const VertexArgs<real> &A) {
  double V;
  const real coef = (real)volume_coef(A.vol_partial, A.vp.vol_blocks, A.vp.V0, A.vp.kV,
                                      A.vp.volume_on, &V);
  if ((threadIdx.x & 31) == 0) {
    if (A.zero_counter) *A.zero_counter = 0;
    *A.vcoef = coef;
    if (!(fabs(V / A.vp.V0 - 1.0) <= 0.05)) atomicOr(A.health, H_VOLUME);
  }
}

// K3b for lane `gid`: vertex gid / 4; lane k = gid % 4 < 3 gathers component k of its forces and
// finds the stencil along axis k, lane 0 then bins the vertex. A third of the serial FP64 work and
// of the loads per lane of one lane per vertex, whose chain set the pass's time where the vertices
// are few (fused step, with the lighter grid barrier, against one lane per vertex: 32^3 FP64, 642
// vertices, 47.6 us against 53; 24^3 FP32 23 against 28; 64^3, 2562 vertices, 31 against 35); with
// many the two are equal (128x128x96, 10242 vertices, 64.9 against 65). A warp's 32 lanes are
// consecutive and call it together.
template <typename real>
__device__ __forceinline__ void vertex_body(const VertexArgs<real> &A, int gid) {
  const int *IBLB_RO vf_start = A.vf_start;
  const int *IBLB_RO vf_list = A.vf_list;
  const real *IBLB_RO fcontrib = reinterpret_cast<const real *>(A.fcontrib);  // [3 nf][4]
  const real *IBLB_RO fnorm = reinterpret_cast<const real *>(A.fnorm);        // [nf][4]
  const double *IBLB_RO q = A.q;
  const Dims D = A.D;
  const int i = gid >> 2, k = gid & 3;
  const bool mine = i < A.nv && k < 3;
  int base = 0;
  if (mine) {
    const int e0 = vf_start[i], e1 = vf_start[i + 1];
    const double p = A.bin ? q[3 * (size_t)i + k] : 0.0;
    real F = 0, g = 0;
    for (int eb = e0; eb < e1; eb += GATHER_UNROLL) {
      int fcs[GATHER_UNROLL];
#pragma unroll
      for (int u = 0; u < GATHER_UNROLL; u++) fcs[u] = eb + u < e1 ? vf_list[eb + u] : -1;
#pragma unroll
      for (int u = 0; u < GATHER_UNROLL; u++) {  // (no branch between the loads: all in flight)
        const int fc = max(fcs[u], 0);            // face * 3 + corner
        const real f = fcontrib[4 * (size_t)fc + k], n = fnorm[4 * (size_t)(fc / 3) + k];
        F += fcs[u] < 0 ? real(0) : f;
        g += fcs[u] < 0 ? real(0) : n;
      }
    }
    reinterpret_cast<real *>(A.phi + i)[k] = F;
    reinterpret_cast<real *>(A.gvol + i)[k] = g;
    if (A.bin) {
      double r;
      const int n = k == 0 ? D.nx : k == 1 ? D.ny : D.nz;
      const double inv = k == 0 ? D.inx : k == 1 ? D.iny : D.inz;
      base = stencil_base(p, n, inv, k < 2 || !D.has_walls, r);
      real w[4];
      peskin_weights<real>((real)r, w);
      StencilRec<real> &rec = A.stencil[i];
      rec.base[k] = base;
#pragma unroll
      for (int d = 0; d < 4; d++) rec.w[k][d] = w[d];
    }
  }
  if (!A.bin) return;
  const int by = __shfl_sync(0xffffffffu, base, 1, 4), bz_ = __shfl_sync(0xffffffffu, base, 2, 4);
  if (!mine || k != 0) return;
  const int bz = min(max(bz_, 0), D.nz - 1);
  const int t = ((bz >> 2) * D.nty + (by >> 2)) * D.ntx + (base >> 2);
  const int s = A.tile_slot[t];
  if (s < 0) {
    atomicOr(A.health, H_CAPACITY);
    return;
  }
  const int rank = atomicAdd(&A.slot_count[s], 1);
  if (rank == 0) A.src_slot[atomicAdd(A.nsources, 1)] = s;  // first vertex: the tile gets a region
  if (rank < BUCKET_CAP) {
    A.bucket[(size_t)s * BUCKET_CAP + rank] = i;
  } else {
    // which vertices end up in the bucket depends on the order of the atomics; the spread
    // pass therefore adds every vertex of a tile that spilled in vertex-index order
    atomicAdd(A.ovf_count, 1);
    atomicOr(&A.spill_bits[i >> 5], 1u << (i & 31));
  }
}

// Block `bid` of K3b: the first takes the scalars, the others a vertex per four threads.
template <typename real>
__device__ __forceinline__ void vertex_block(const VertexArgs<real> &A, int bid) {
  if (bid == 0) {
    if (threadIdx.x < 32) volume_task(A);
    return;
  }
  vertex_body(A, (bid - 1) * blockDim.x + threadIdx.x);
}

template <typename real>
__global__ void __launch_bounds__(kVertexThreads) vertex_kernel(const VertexArgs<real> A) {
  vertex_block(A, blockIdx.x);
}

template <typename real>
__global__ void __launch_bounds__(kVertexThreads) vertex_kernel_multi(
    const VertexArgs<real> *__restrict__ all, const int *__restrict__ start, int n) {
  const MultiBlock m = multi_block(start, n);
  vertex_block(all[m.inst], m.block);
}

// Spreading works on regions: the stencils of the vertices binned in a source tile S (base
// node in S) cover the 7x7x7 nodes S_lo .. S_lo + 6.
constexpr int REGION = 7;
constexpr int REGION_NODES = REGION * REGION * REGION;
// Threads per block of K4a: one block per source tile, one bucket entry per thread.
constexpr int kSourceThreads = BUCKET_CAP;
static_assert(kSourceThreads == 128, "four warps: one per z plane of a stencil");

// w[d] for a run-time d in 0..3 without indexing a local array.
template <typename real>
__device__ __forceinline__ real pick4(const real w[4], int d) {
  return d == 0 ? w[0] : d == 1 ? w[1] : d == 2 ? w[2] : w[3];
}

// K4a: spreading, first pass (Eq. 13). One block of four warps per source tile S: its bucket is
// sorted by vertex index (rank by comparison, at most 128 entries) and the vertices' stencil
// records and forces (completed with the volume term -kV (V - V0)/V0 dV/dq) are staged in shared
// memory in that order. Of the 7x7x7 region of S warp w owns the z planes w and w + 4, of which
// every vertex's stencil covers exactly one; a half warp adds the 16 nodes of that plane, the
// lower half for the even vertices, the upper half for the odd ones into a copy of its own (no
// atomics, no waiting between warps). The two copies are added and written out, and the region's
// index is pushed to the (up to 8) tiles T = S + {0,1}^3 it overlaps. The time is the chain of
// additions into shared memory, a quarter as long as with one warp per tile, whose lanes added two
// nodes of every vertex one vertex after the other (10242 vertices on 64 SMs: 9.3 us against 12.5;
// 96 wetting boxes 134 us against 180; 40962 vertices on 24 SMs, where the SMs are full: 89 both).
// A tile with more than 128 vertices (its bucket holds 128 of them, chosen by the order of the
// binning atomics) marks its bucket's vertices in the spill bitmap, which already holds its
// spilled ones, and adds all of its vertices in increasing vertex index instead, found by a
// scan of the bitmap. Either way the order of summation depends only on the vertex set.
template <typename real>
struct SourceArgs {
  const int *tile_slot, *slot_tile, *nsources_ptr, *slot_count, *src_slot, *bucket;
  unsigned *spill_bits;
  int spill_words, max_sources;
  const StencilRec<real> *stencil;
  const Vec4<real> *phi, *gvol;
  const real *vcoef;  // kV (V - V0)/V0, written by the vertex kernel of the step
  Vec4<real> *Rslot;
  int *out_src;
  Dims D;
};

// One vertex's plane of nodes added by a half warp: base (bx, by, bz) in the region, weights w
// (x, y, z), force f. Lane l of the half owns the node (l & 3, l >> 2) of the plane.
template <typename real>
__device__ __forceinline__ void add_plane(Vec4<real> *region, int plane, int l, int bx, int by,
                                          int bz, const real *wx, const real *wy, const real *wz,
                                          real fx, real fy, real fz) {
  const int dz = (plane - bz) & 3, rz = bz + dz;  // the stencil's plane that this warp owns
  if (rz < 0 || rz >= REGION) return;             // beyond the lattice in z
  const int dx = l & 3, dy = l >> 2;
  const real w = wx[dx] * wy[dy] * wz[dz];
  Vec4<real> &o = region[(rz * REGION + by + dy) * REGION + bx + dx];
  Vec4<real> v = o;
  v.x += w * fx;
  v.y += w * fy;
  v.z += w * fz;
  v.w = real(1);  // a stencil node of some vertex (the interpolation reads it)
  o = v;
}

// Words of the spill bitmap that a warp scans per round (at most 8: list entries are a byte).
constexpr int kScanWords = 8;

// Shared memory of one group of kSourceThreads threads of K4a.
template <typename real>
struct SourceShared {
  Vec4<real> region[2][REGION_NODES];
  Vec4<real> f[BUCKET_CAP];
  real w[BUCKET_CAP][12];
  int b[BUCKET_CAP];
  int v[BUCKET_CAP];
  unsigned char list[kSourceThreads / 32][32 * kScanWords];  // of a spilled tile: see below
  int listed[kSourceThreads / 32];
};

// Barrier of the kSourceThreads threads of group `g` of a block.
__device__ __forceinline__ void group_barrier(int g) {
  asm volatile("barrier.cta.sync %0, %1;" ::"r"(1 + g), "n"(kSourceThreads) : "memory");
}

// A vertex's record, completed with the volume term, to place r of the stage of source tile S. Its base
// is relative to S_lo (x, y wrapped into [0, n) by the vertex kernel): x, y in 0..3, z in -4..3 (below 0
// only at a wall), in a byte each.
template <typename real>
__device__ __forceinline__ void stage_record(SourceShared<real> &sh, int r, const StencilRec<real> &rec,
                                             const Vec4<real> &pv, const Vec4<real> &gv, real coef,
                                             int Sx, int Sy, int Sz) {
  for (int k = 0; k < 4; k++) {
    sh.w[r][k] = rec.w[0][k];
    sh.w[r][4 + k] = rec.w[1][k];
    sh.w[r][8 + k] = rec.w[2][k];
  }
  sh.f[r] = Vec4<real>{pv.x - coef * gv.x, pv.y - coef * gv.y, pv.z - coef * gv.z, real(0)};
  const int bz = max(rec.base[2] - Sz, -4);
  sh.b[r] = (rec.base[0] - Sx) | (rec.base[1] - Sy) << 8 | (bz + 4) << 16;
}
// Add the n staged vertices, the tile's rank-th and following: even ranks by the lower half warp.
template <typename real>
__device__ __forceinline__ void add_staged(SourceShared<real> &sh, int n, int rank, int warp, int half,
                                           int l16) {
  for (int c0 = 0; c0 < n; c0 += 2) {
    const int c = c0 + ((half ^ rank) & 1);
    if (c < n) {
      const int b = sh.b[c];
      const Vec4<real> f = sh.f[c];
      add_plane(sh.region[half], warp, l16, b & 255, (b >> 8) & 255, (b >> 16) - 4, sh.w[c],
                sh.w[c] + 4, sh.w[c] + 8, f.x, f.y, f.z);
    }
    __syncwarp();
  }
}

// A tile that spilled: mark its bucket's vertices too, then add every vertex of the tile in
// increasing index (bitmap words read through L2, where the atomics are performed). A round
// scans the next kScanWords words of each of the four warps, which list the tile's vertices
// among them in a row each; the rows, one after the other, are staged and added like a bucket.
// (With every warp scanning all words, and a vertex's record read when its turn came, a tile
// was a chain of memory latencies. 96^3 FP32 with 40962 vertices on a sphere of radius 20, whose
// tiles nearly all spill: 411 us per step against 1026, by the separate kernels 232 against 606;
// radius 16, 275 against 762.)
template <typename real>
__device__ __forceinline__ void spread_spilled(const SourceArgs<real> &A, SourceShared<real> &sh, int g,
                                               int tid, int v, int t) {
  unsigned *spill_bits = A.spill_bits;
  const StencilRec<real> *stencil = A.stencil;
  const Dims &D = A.D;
  const real coef = *A.vcoef;
  const int lane = tid & 31, warp = tid >> 5, half = lane >> 4, l16 = lane & 15;
  const int tsx = t % D.ntx, tsy = (t / D.ntx) % D.nty, tsz = t / (D.ntx * D.nty);
  atomicOr(&spill_bits[v >> 5], 1u << (v & 31));
  group_barrier(g);
  int rank = 0;
  for (int wb = 0; wb < A.spill_words; wb += kScanWords * (kSourceThreads / 32)) {
    const int w0 = wb + kScanWords * warp;
    const unsigned words =
        lane < kScanWords && w0 + lane < A.spill_words ? __ldcg(&spill_bits[w0 + lane]) : 0u;
    int n = 0;
#pragma unroll 1
    for (int k0 = 0; k0 < kScanWords; k0 += 2) {  // (two words' loads in flight: few registers)
      bool mine[2];
#pragma unroll
      for (int k = 0; k < 2; k++) {
        mine[k] = (__shfl_sync(0xffffffffu, words, k0 + k) >> lane) & 1u;
        if (mine[k]) {
          const StencilRec<real> &rl = stencil[(w0 + k0 + k) * 32 + lane];
          mine[k] = (rl.base[0] >> 2) == tsx && (rl.base[1] >> 2) == tsy &&
                    (min(max(rl.base[2], 0), D.nz - 1) >> 2) == tsz;
        }
      }
#pragma unroll
      for (int k = 0; k < 2; k++) {
        const unsigned members = __ballot_sync(0xffffffffu, mine[k]);
        if (mine[k])
          sh.list[warp][n + __popc(members & ((1u << lane) - 1u))] =
              (unsigned char)(32 * (k0 + k) + lane);
        n += __popc(members);
      }
    }
    if (lane == 0) sh.listed[warp] = n;
    group_barrier(g);
    const int e1 = sh.listed[0], e2 = e1 + sh.listed[1], e3 = e2 + sh.listed[2];
    const int total = e3 + sh.listed[3];
    for (int c0 = 0; c0 < total; c0 += kSourceThreads) {
      const int e = c0 + tid, m = min(total - c0, kSourceThreads);
      if (tid < m) {
        const int row = (e >= e1) + (e >= e2) + (e >= e3);
        const int at = e - (row == 0 ? 0 : row == 1 ? e1 : row == 2 ? e2 : e3);
        const int vm = 32 * (wb + kScanWords * row) + sh.list[row][at];
        stage_record(sh, tid, stencil[vm], A.phi[vm], A.gvol[vm], coef, tsx * TILE, tsy * TILE,
                     tsz * TILE);
      }
      group_barrier(g);
      add_staged(sh, m, rank, warp, half, l16);
      rank += m;
      group_barrier(g);  // the stage and the lists are written again
    }
    if (total == 0) group_barrier(g);
  }
}
// The same as a function of its own, where inlining it slows code that it does not touch: the kernel of
// a whole step in FP64 (128^3 562 us per step inlined, 552 so) and FP32 (112^3 63.3, 61.3), but not
// in 16 bits (128^3 57.5 inlined, 60.3 so).
template <typename real>
__device__ __noinline__ void spread_spilled_call(const SourceArgs<real> &A, SourceShared<real> &sh, int g,
                                                 int tid, int v, int t) {
  spread_spilled(A, sh, g, tid, v, t);
}

// K4a for the source tiles bid, bid + nb, ..., by group `g` of its block (thread tid of it).
// CALL: spilled tiles by a call.
template <bool CALL, typename real>
__device__ __forceinline__ void spread_source_body(const SourceArgs<real> &A, SourceShared<real> &sh,
                                                   int bid, int nb, int g, int tid) {
  const int *IBLB_RO tile_slot = A.tile_slot;
  const int *IBLB_RO slot_tile = A.slot_tile;
  const int *IBLB_RO slot_count = A.slot_count;
  const int *IBLB_RO bucket = A.bucket;
  unsigned *spill_bits = A.spill_bits;
  const StencilRec<real> *IBLB_RO stencil = A.stencil;
  const Vec4<real> *IBLB_RO phi = A.phi;
  const Vec4<real> *IBLB_RO gvol = A.gvol;
  int *IBLB_RO out_src = A.out_src;
  const Dims D = A.D;
  const int nsources = min(*A.nsources_ptr, A.max_sources);
  const int lane = tid & 31, warp = tid >> 5;
  const int half = lane >> 4, l16 = lane & 15;
  const real coef = *A.vcoef;
  for (int reg = bid; reg < nsources; reg += nb) {
    const int s = A.src_slot[reg];
    const int cnt = slot_count[s];
    const int t = slot_tile[s];
    const int *bk = bucket + (size_t)s * BUCKET_CAP;
    const int v = tid < cnt ? bk[tid] : 0x7fffffff;
    for (int k = tid; k < 2 * REGION_NODES; k += kSourceThreads)
      sh.region[0][k] = Vec4<real>{0, 0, 0, 0};
    const int tsx = t % D.ntx, tsy = (t / D.ntx) % D.nty, tsz = t / (D.ntx * D.nty);
    const int Sx = tsx * TILE, Sy = tsy * TILE, Sz = tsz * TILE;
    // push the region to the tiles it overlaps: T = S + e, seen from T as source e
    if (tid >= kSourceThreads - 8) {
      const int e = tid & 7;
      int ux = tsx + (e & 1), uy = tsy + ((e >> 1) & 1), uz = tsz + (e >> 2);
      ux = ux >= D.ntx ? ux - D.ntx : ux;
      uy = uy >= D.nty ? uy - D.nty : uy;
      bool ok = true;
      if (uz >= D.ntz) {
        if (D.has_walls) ok = false;
        uz -= D.ntz;
      }
      if (ok) {
        const int slot_t = tile_slot[(uz * D.nty + uy) * D.ntx + ux];
        if (slot_t >= 0) out_src[8 * (size_t)slot_t + e] = reg;
      }
    }
    if (cnt <= BUCKET_CAP) {
      // sort the bucket by vertex index and stage the records in that order
      StencilRec<real> rec;
      Vec4<real> pv, gv;
      sh.v[tid] = v;
      if (tid < cnt) {
        rec = stencil[v];
        pv = phi[v];
        gv = gvol[v];
      }
      group_barrier(g);
      if (tid < cnt) {
        int r = 0;
        for (int m = 0; m < cnt; m++) r += sh.v[m] < v;
        stage_record(sh, r, rec, pv, gv, coef, Sx, Sy, Sz);
      }
      group_barrier(g);
      add_staged(sh, cnt, 0, warp, half, l16);
    } else if constexpr (CALL) {
      spread_spilled_call(A, sh, g, tid, v, t);
    } else {
      spread_spilled(A, sh, g, tid, v, t);
    }
    group_barrier(g);
    Vec4<real> *out = A.Rslot + (size_t)reg * REGION_NODES;
    for (int k = tid; k < REGION_NODES; k += kSourceThreads) {
      const Vec4<real> a = sh.region[0][k], b = sh.region[1][k];
      out[k] = Vec4<real>{a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w};
    }
    group_barrier(g);  // the region is cleared for the next tile
  }
}

template <typename real>
__global__ void __launch_bounds__(kSourceThreads)
    spread_source_kernel(const __grid_constant__ SourceArgs<real> A) {
  __shared__ SourceShared<real> sh;
  spread_source_body<sizeof(real) == 8>(A, sh, blockIdx.x, gridDim.x, 0, threadIdx.x);
}

// (seven blocks per SM, in FP64 four: a few registers fewer than it would take)
template <typename real>
__global__ void __launch_bounds__(kSourceThreads, sizeof(real) == 4 ? 7 : 4) spread_source_kernel_multi(
    const SourceArgs<real> *__restrict__ all, const int *__restrict__ start, int n) {
  const MultiBlock m = multi_block(start, n);
  __shared__ SourceShared<real> sh;
  spread_source_body<sizeof(real) == 8>(all[m.inst], sh, m.block, m.nblocks, 0, threadIdx.x);
}

// K4b: spreading, second pass. One 64-thread block per active tile T (grid-stride), thread =
// node (lx, ly, lz): the force is the sum, in the fixed order e = 0..7, of the regions of the
// source tiles S = T - e pushed by K4a; the node sits at (l + 4 e) in S's region. On a
// periodic axis only 4 nodes long S - e and S coincide and the two terms are the node's two
// images in the region. Force landing on a wall layer is dropped. K4a marks each region
// node that lies in a vertex's stencil (w = 1); K4b lists the node pairs holding such a node,
// the work of the active-tile correction (K1t) and of the shell velocity (K1b).
template <typename real>
struct GatherArgs {
  const int *slot_tile, *nslots_ptr, *out_src;
  const Vec4<real> *Rslot;
  Vec4<real> *Fslot;
  int *pair_list, *npairs;  // node pairs (x even, x + 1) in some vertex's stencil, for K1t, K1b
  Dims D;
};

// K4b for the active tiles bid, bid + nb, ..., by 64 threads (two warps; tid: thread of them).
template <typename real>
__device__ __forceinline__ void spread_gather_body(const GatherArgs<real> &A, int bid, int nb, int tid) {
  const int *IBLB_RO slot_tile = A.slot_tile;
  const int *IBLB_RO out_src = A.out_src;
  const Vec4<real> *IBLB_RO Rslot = A.Rslot;
  Vec4<real> *IBLB_RO Fslot = A.Fslot;
  const Dims D = A.D;
  const int nslots = min(*A.nslots_ptr, D.max_slots);
  const int lx = tid & 3, ly = (tid >> 2) & 3, lz = tid >> 4;
  for (int b = bid; b < nslots; b += nb) {
    const int4 *src4 = reinterpret_cast<const int4 *>(out_src + 8 * (size_t)b);
    const int4 lo = src4[0], hi = src4[1];
    const int src[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
    real f[3] = {0, 0, 0};
    bool stencil_node = false;
    Vec4<real> r[8];
#pragma unroll
    for (int e = 0; e < 8; e++) {
      const int rx = lx + 4 * (e & 1), ry = ly + 4 * ((e >> 1) & 1), rz = lz + 4 * (e >> 2);
      const bool in = src[e] >= 0 && rx < REGION && ry < REGION && rz < REGION;
      r[e] = Vec4<real>{0, 0, 0, 0};
      if (in) r[e] = Rslot[(size_t)src[e] * REGION_NODES + (rz * REGION + ry) * REGION + rx];
    }
#pragma unroll
    for (int e = 0; e < 8; e++) {
      f[0] += r[e].x;
      f[1] += r[e].y;
      f[2] += r[e].z;
      stencil_node |= r[e].w != real(0);
    }
    const int Z = (slot_tile[b] / (D.ntx * D.nty)) * TILE + lz;
    const bool drop = D.has_walls && (Z == 0 || Z >= D.nz - 1);
    Vec4<real> o;
    o.x = drop ? real(0) : f[0];
    o.y = drop ? real(0) : f[1];
    o.z = drop ? real(0) : f[2];
    o.w = real(0);
    Fslot[(size_t)b * TILE_CELLS + tid] = o;
    // list the pairs (tid even, tid + 1) of this warp of which either node is a fluid node of
    // some vertex's stencil (every node that can carry a force, and every node the
    // interpolation reads off the wall layers): one atomic per warp, entries in pair order
    // within the warp
    const unsigned m = __ballot_sync(0xffffffffu, stencil_node && !drop);
    const unsigned pm = (m | (m >> 1)) & 0x55555555u;  // bit 2k: pair k is listed
    const int lane = tid & 31;
    int base = 0;
    if (lane == 0 && pm) base = atomicAdd(A.npairs, __popc(pm));
    base = __shfl_sync(0xffffffffu, base, 0);
    if ((pm >> lane) & 1u)
      A.pair_list[base + __popc(pm & ((1u << lane) - 1u))] = 32 * b + (tid >> 1);
  }
}

template <typename real>
__global__ void __launch_bounds__(64) spread_gather_kernel(const GatherArgs<real> A) {
  spread_gather_body(A, blockIdx.x, gridDim.x, threadIdx.x);
}

template <typename real>
__global__ void __launch_bounds__(64) spread_gather_kernel_multi(
    const GatherArgs<real> *__restrict__ all, const int *__restrict__ start, int n) {
  const MultiBlock m = multi_block(start, n);
  spread_gather_body(all[m.inst], m.block, m.nblocks, threadIdx.x);
}

// K2: interpolation (Eq. 11) and the Euler update (Eq. 12); 4 lanes per vertex, lane dz
// sums the 16 nodes of its z-plane of the stencil, the 4 planes are summed by shuffles; lane k
// then adds the update to coordinate k of the double position. One lane per axis issues a third of
// the FP64 instructions of one lane per vertex (an FP64 instruction holds the SM's FP64 unit for 16
// cycles however few lanes take part): 10242 vertices on 64 SMs 12.8 us against 17.2, 40962 on 24
// SMs 88 against 127, 96 wetting boxes 108 against 262.
// The delta-weight accumulation of a vertex is carried at double precision in every
// precision (VertexSum): each stencil row's four products w_x u (one x row of a tile, in the
// arithmetic type) is added to the vertex's sum with its weight w_y w_z, and the four planes'
// sums are added across the lanes, without rounding the sum back to float.
template <typename real>
struct VertexSum;

// FP64 contexts: a plain double sum.
template <>
struct VertexSum<double> {
  double s[3] = {0.0, 0.0, 0.0};
  __device__ __forceinline__ void add_prod(int k, double a, double b) { s[k] += a * b; }
  __device__ __forceinline__ void set(int k, double x) { s[k] = x; }
  __device__ __forceinline__ void add_lanes(int o) {
    for (int k = 0; k < 3; k++) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
  }
  // component k of a run-time k
  __device__ __forceinline__ double value(int k) const { return k == 0 ? s[0] : k == 1 ? s[1] : s[2]; }
};

// Float contexts: the sum is a pair of floats hi + lo (double-float arithmetic), kept exact
// up to rounding at about 2^-44 of the sum with the error-free transformations of Dekker
// (the product a b = p + e, e by a fused multiply-add) and Knuth (TwoSum: s + err = x + y).
// This is as accurate as a double sum of the same float products; on GB300 double arithmetic
// runs at 1/64 of the float rate, and the double form lengthened the 16-bit step. The _rn
// intrinsics keep the compiler from fusing the steps the transformations rely on.
template <>
struct VertexSum<float> {
  float hi[3] = {0.f, 0.f, 0.f}, lo[3] = {0.f, 0.f, 0.f};
  __device__ __forceinline__ void add(int k, float x, float xerr) {
    const float s = __fadd_rn(hi[k], x);
    const float bp = __fsub_rn(s, hi[k]);
    const float err = __fadd_rn(__fsub_rn(hi[k], __fsub_rn(s, bp)), __fsub_rn(x, bp));
    hi[k] = s;
    lo[k] = __fadd_rn(lo[k], __fadd_rn(err, xerr));
  }
  __device__ __forceinline__ void add_prod(int k, float a, float b) {
    const float p = __fmul_rn(a, b);
    add(k, p, __fmaf_rn(a, b, -p));
  }
  __device__ __forceinline__ void set(int k, double x) {
    hi[k] = __double2float_rn(x);
    lo[k] = __double2float_rn(x - (double)hi[k]);
  }
  // the same result in every lane of the butterfly: the addition is commutative and TwoSum's
  // error term is exact
  __device__ __forceinline__ void add_lanes(int o) {
    for (int k = 0; k < 3; k++) {
      const float h = __shfl_xor_sync(0xffffffffu, hi[k], o);
      const float l = __shfl_xor_sync(0xffffffffu, lo[k], o);
      lo[k] = __fadd_rn(lo[k], l);
      add(k, h, 0.f);
    }
  }
  __device__ __forceinline__ double value(int k) const {
    const float h = k == 0 ? hi[0] : k == 1 ? hi[1] : hi[2];
    const float l = k == 0 ? lo[0] : k == 1 ? lo[1] : lo[2];
    return (double)h + (double)l;
  }
};

template <typename real>
struct InterpArgs {
  int nv;
  const StencilRec<real> *stencil;
  const int *tile_slot;
  const Vec4<real> *Uslot;
  double *q, *qdot;
  const double *xref;
  Vec4<real> *disp;
  double3 ub, ut;
  Dims D;
  int *health;
};

// K2's sum over plane dz of vertex v's stencil.
template <typename real>
__device__ __forceinline__ void interp_plane(const InterpArgs<real> &A, int v, int dz,
                                             VertexSum<real> &acc) {
  const StencilRec<real> *IBLB_RO stencil = A.stencil;
  const int *IBLB_RO tile_slot = A.tile_slot;
  const Vec4<real> *IBLB_RO Uslot = A.Uslot;
  int *IBLB_RO health = A.health;
  const double3 ub = A.ub, ut = A.ut;
  const Dims &D = A.D;
  {
    const StencilRec<real> rec = stencil[v];
    int Z = rec.base[2] + dz;
    if (!D.has_walls) Z = Z >= D.nz ? Z - D.nz : Z;
    if (Z >= 0 && Z < D.nz) {
      const real wz = pick4(rec.w[2], dz);
      if (D.has_walls && (Z == 0 || Z == D.nz - 1)) {
        const double3 w = Z == 0 ? ub : ut;
        const double sxy =
            ((double)rec.w[0][0] + (double)rec.w[0][1] + (double)rec.w[0][2] + (double)rec.w[0][3]) *
            ((double)rec.w[1][0] + (double)rec.w[1][1] + (double)rec.w[1][2] + (double)rec.w[1][3]) *
            (double)wz;
        acc.set(0, sxy * w.x);
        acc.set(1, sxy * w.y);
        acc.set(2, sxy * w.z);
      } else {
        // the 4 stencil nodes along x (and along y) fall in at most two tiles: look up the
        // (up to) four tile slots of this z-plane once
        int X[4], Y[4];
        for (int d = 0; d < 4; d++) {
          const int xx = rec.base[0] + d, yy = rec.base[1] + d;
          X[d] = xx >= D.nx ? xx - D.nx : xx;
          Y[d] = yy >= D.ny ? yy - D.ny : yy;
        }
        const int tzrow = (Z >> 2) * D.nty;
        int sl[2][2];
        for (int iy = 0; iy < 2; iy++)
          for (int ix = 0; ix < 2; ix++)
            sl[iy][ix] = tile_slot[(tzrow + (Y[3 * iy] >> 2)) * D.ntx + (X[3 * ix] >> 2)];
        // an unmarked tile (only after a capacity failure) counts as at rest; checked ahead of the
        // loads, so that no branch stands between them and they are all in flight at once
        if (min(min(sl[0][0], sl[0][1]), min(sl[1][0], sl[1][1])) < 0) atomicOr(health, H_CAPACITY);
#pragma unroll
        for (int dy = 0; dy < 4; dy++) {
          const bool uy = (Y[dy] >> 2) != (Y[0] >> 2);
          const int crow = 4 * (Y[dy] & 3) + 16 * (Z & 3);
          const int s0 = uy ? sl[1][0] : sl[0][0], s1 = uy ? sl[1][1] : sl[0][1];
          Vec4<real> u[4];
#pragma unroll
          for (int dx = 0; dx < 4; dx++) {
            const int sidx = (X[dx] >> 2) != (X[0] >> 2) ? s1 : s0;
            u[dx] = Uslot[(size_t)max(sidx, 0) * TILE_CELLS + (X[dx] & 3) + crow];
            if (sidx < 0) u[dx] = Vec4<real>{0, 0, 0, 0};
          }
          real r3[3] = {0, 0, 0};
#pragma unroll
          for (int dx = 0; dx < 4; dx++) {
            const real w = rec.w[0][dx];
            r3[0] += w * u[dx].x;
            r3[1] += w * u[dx].y;
            r3[2] += w * u[dx].z;
          }
          const real wyz = rec.w[1][dy] * wz;
          acc.add_prod(0, wyz, r3[0]);
          acc.add_prod(1, wyz, r3[1]);
          acc.add_prod(2, wyz, r3[2]);
        }
      }
    }
  }
}

// K2 for N vertices per four lanes: lane `gid` takes plane gid % 4 of the vertices gid / 4,
// gid / 4 + step, ... A warp's 32 lanes are consecutive and call it together. With N = 2 the two
// vertices' loads are in flight together, for a grid that has fewer lanes than the mesh asks for.
template <int N, typename real>
__device__ __forceinline__ void interp_body(const InterpArgs<real> &A, int gid, int step) {
  const Dims &D = A.D;
  const int dz = gid & 3;
  // lane k < 3 of a vertex updates coordinate k: its position is read ahead
  double qk[N], xk[N];
  VertexSum<real> acc[N];
#pragma unroll
  for (int m = 0; m < N; m++) {
    const int v = (gid >> 2) + m * step;
    const bool axis = v < A.nv && dz < 3;
    qk[m] = axis ? A.q[3 * (size_t)v + dz] : 0.0;
    xk[m] = axis ? A.xref[3 * (size_t)v + dz] : 0.0;
  }
#pragma unroll
  for (int m = 0; m < N; m++) {
    const int v = (gid >> 2) + m * step;
    if (v < A.nv) interp_plane(A, v, dz, acc[m]);
  }
  // sum of the 4 planes (fixed butterfly order)
  for (int o = 2; o > 0; o >>= 1)
#pragma unroll
    for (int m = 0; m < N; m++) acc[m].add_lanes(o);
#pragma unroll
  for (int m = 0; m < N; m++) {
    const int v = (gid >> 2) + m * step;
    if (v >= A.nv || dz >= 3) continue;
    const double qd = acc[m].value(dz);
    const double pn = qk[m] + qd;
    A.qdot[3 * (size_t)v + dz] = qd;
    A.q[3 * (size_t)v + dz] = pn;
    int h = 0;
    if (!(fabs(qd) < 0.1)) h |= (qd == qd) ? H_FAST : H_NAN;
    if (dz == 2 && D.has_walls && (pn - D.zb < 0.05 || D.zt - pn < 0.05)) h |= H_WALL;
    if (h) atomicOr(A.health, h);
    reinterpret_cast<real *>(A.disp + v)[dz] = (real)(pn - xk[m]);
  }
}

// Threads per block of K2.
constexpr int kInterpThreads = 128;

template <typename real>
__global__ void __launch_bounds__(kInterpThreads) interp_kernel(const InterpArgs<real> A) {
  interp_body<1>(A, blockIdx.x * blockDim.x + threadIdx.x, 0);
}

template <typename real>
__global__ void __launch_bounds__(kInterpThreads) interp_kernel_multi(
    const InterpArgs<real> *__restrict__ all, const int *__restrict__ start, int n) {
  const MultiBlock m = multi_block(start, n);
  interp_body<1>(all[m.inst], m.block * blockDim.x + threadIdx.x, 0);
}

// Displacement from the reference shape, after setting vertices; one thread per coordinate.
template <typename real>
__global__ void displacement_kernel(int nv, const double *__restrict__ q,
                                    const double *__restrict__ xref, Vec4<real> *__restrict__ disp) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < 3 * nv) reinterpret_cast<real *>(disp + i / 3)[i % 3] = (real)(q[i] - xref[i]);
}

template <typename real>
__global__ void expand_force_kernel(const int *__restrict__ slot_tile, const int *__restrict__ nslots,
                                    const Vec4<real> *__restrict__ Fslot, Dims D,
                                    double *__restrict__ F) {
  const int n = min(*nslots, D.max_slots);
  for (int b = blockIdx.x; b < n; b += gridDim.x) {
    const int t = slot_tile[b];
    const int tx = t % D.ntx, ty = (t / D.ntx) % D.nty, tz = t / (D.ntx * D.nty);
    const int c = threadIdx.x;
    const int X = tx * TILE + (c & 3), Y = ty * TILE + ((c >> 2) & 3), Z = tz * TILE + (c >> 4);
    if (Z >= D.nz) continue;
    const size_t node = ((size_t)Z * D.ny + Y) * D.nx + X;
    const Vec4<real> f = Fslot[(size_t)b * TILE_CELLS + c];
    F[3 * node] = (double)f.x;
    F[3 * node + 1] = (double)f.y;
    F[3 * node + 2] = (double)f.z;
  }
}

// Nodal force of Eq. 16, phi - kV (V - V0)/V0 dV/dq, in double for read-back.
template <typename real>
__global__ void combine_forces_kernel(int nv, const Vec4<real> *__restrict__ phi,
                                      const Vec4<real> *__restrict__ gvol,
                                      const double *__restrict__ vol_partial, VolumeParams vp,
                                      double *__restrict__ out) {
  __shared__ double s_coef;
  if (threadIdx.x < 32) {
    const double coef = volume_coef(vol_partial, vp.vol_blocks, vp.V0, vp.kV, vp.volume_on, nullptr);
    if (threadIdx.x == 0) s_coef = coef;
  }
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nv) return;
  const real coef = (real)s_coef;
  const Vec4<real> p = phi[i], g = gvol[i];
  out[3 * (size_t)i] = (double)(p.x - coef * g.x);
  out[3 * (size_t)i + 1] = (double)(p.y - coef * g.y);
  out[3 * (size_t)i + 2] = (double)(p.z - coef * g.z);
}

VolumeParams volume_params(const Ctx &c) {
  VolumeParams vp;
  vp.V0 = c.V0;
  vp.kV = c.iface.kV;
  vp.volume_on = c.iface.volume_force_on;
  vp.vol_blocks = c.vol_blocks;
  return vp;
}

// The tile map of the context's current positions.
TileMap tile_map(const Ctx &c) {
  return TileMap{c.tile_slot[c.map], c.slot_tile[c.map], c.counters + c.map, c.slot_count,
                 c.out_src[c.map], c.counters + 3};
}

// Argument records of the step kernels for context c as it is now (its cur and map), shared by
// the single-context launches and the batched ones.
template <typename real>
FaceArgs<real> face_args(const Ctx &c, int reset) {
  FaceArgs<real> a;
  const double *al = c.iface.alpha;
  a.fp.a3 = (real)al[2];
  a.fp.cL0 = (real)(0.5 * (al[0] - al[2]));
  a.fp.cL1 = (real)(0.25 * (al[0] + al[1]));
  a.fp.eps48 = (real)(48.0 * c.iface.eps);
  a.fp.xi = (real)c.iface.xi;
  a.fp.wall_on = c.iface.wall_force_on;
  const int other = c.map ^ 1;
  a.nf = c.nf;
  a.faces = c.faces;
  a.disp = (const Vec4<real> *)c.disp;
  a.fgeo = (const real *)c.fgeo;
  a.fcontrib = (Vec4<real> *)c.fcontrib;
  a.fnorm = (Vec4<real> *)c.fnorm;
  a.vol_partial = c.vol_partial;
  a.D = dims_of(c);
  a.other_tile_slot = c.tile_slot[other];
  a.other_slot_tile = c.slot_tile[other];
  a.other_nslots = c.counters + other;
  a.reset = reset;
  a.map = tile_map(c);
  a.q = c.q;
  a.nv = c.nv;
  a.ovf_count = c.counters + 2;
  a.spill_bits = c.spill_bits;
  a.spill_words = c.spill_words;
  return a;
}
template <typename real>
int face_blocks(const Ctx &c, int reset) {
  const int warps = (c.nf + 31) / 32 + (reset ? (c.nv + kMarkVertices - 1) / kMarkVertices : 0);
  return (32 * warps + FaceThreads<real>::value - 1) / FaceThreads<real>::value;
}

template <typename real>
VertexArgs<real> vertex_args(const Ctx &c, int bin) {
  VertexArgs<real> a;
  a.nv = c.nv;
  a.vf_start = c.vf_start;
  a.vf_list = c.vf_list;
  a.fcontrib = (const Vec4<real> *)c.fcontrib;
  a.fnorm = (const Vec4<real> *)c.fnorm;
  a.q = c.q;
  a.phi = (Vec4<real> *)c.phi;
  a.gvol = (Vec4<real> *)c.gvol;
  a.stencil = (StencilRec<real> *)c.stencil;
  a.bin = bin;
  a.tile_slot = c.tile_slot[c.map];
  a.slot_count = c.slot_count;
  a.bucket = c.bucket;
  a.ovf_count = c.counters + 2;
  a.spill_bits = c.spill_bits;
  a.src_slot = c.src_slot;
  a.nsources = c.counters + 4;
  a.health = c.counters + 3;
  a.zero_counter = bin == 2 ? c.counters + (c.map ^ 1) : nullptr;
  a.vol_partial = c.vol_partial;
  a.vp = volume_params(c);
  a.vcoef = (real *)c.vcoef;
  a.D = dims_of(c);
  return a;
}
// the first block takes the volume coefficient
int vertex_blocks(const Ctx &c) { return (int)((4L * c.nv + kVertexThreads - 1) / kVertexThreads) + 1; }

template <typename real>
SourceArgs<real> source_args(const Ctx &c) {
  SourceArgs<real> a;
  a.tile_slot = c.tile_slot[c.map];
  a.slot_tile = c.slot_tile[c.map];
  a.nsources_ptr = c.counters + 4;
  a.max_sources = c.max_sources;
  a.slot_count = c.slot_count;
  a.src_slot = c.src_slot;
  a.bucket = c.bucket;
  a.spill_bits = c.spill_bits;
  a.spill_words = c.spill_words;
  a.stencil = (const StencilRec<real> *)c.stencil;
  a.phi = (const Vec4<real> *)c.phi;
  a.gvol = (const Vec4<real> *)c.gvol;
  a.vcoef = (const real *)c.vcoef;
  a.Rslot = (Vec4<real> *)c.Rslot;
  a.out_src = c.out_src[c.map];
  a.D = dims_of(c);
  return a;
}
// persistent grids sized to the SMs the interface chain runs on; in a batch (no partition,
// many contexts side by side) to the context's expected active tiles instead, about half of
// them source tiles: a block per source tile
template <typename real>
int source_blocks(const Ctx &c, bool batched) {
  const int sms = c.ib_sms > 0 ? c.ib_sms : c.sm_count;
  int g = batched ? (c.tile_estimate + 3) / 4 : sms * (sizeof(real) == 4 ? 10 : 5);
  if (g > c.max_sources) g = c.max_sources;
  return g < 1 ? 1 : g;
}

template <typename real>
GatherArgs<real> gather_args(const Ctx &c) {
  GatherArgs<real> a;
  a.slot_tile = c.slot_tile[c.map];
  a.nslots_ptr = c.counters + c.map;
  a.out_src = c.out_src[c.map];
  a.Rslot = (const Vec4<real> *)c.Rslot;
  a.Fslot = (Vec4<real> *)c.Fslot[c.map];
  a.pair_list = c.pair_list;
  a.npairs = c.counters + 5;
  a.D = dims_of(c);
  return a;
}
int gather_blocks(const Ctx &c, bool batched) {
  const int sms = c.ib_sms > 0 ? c.ib_sms : c.sm_count;
  int g = batched ? (c.tile_estimate + 1) / 2 : sms * 16;  // batched: a block per two tiles
  if (g > c.max_slots) g = c.max_slots;
  return g < 1 ? 1 : g;
}

template <typename real>
InterpArgs<real> interp_args(const Ctx &c) {
  InterpArgs<real> a;
  a.nv = c.nv;
  a.stencil = (const StencilRec<real> *)c.stencil;
  a.tile_slot = c.tile_slot[c.map];
  a.Uslot = (const Vec4<real> *)c.Uslot;
  a.q = c.q;
  a.qdot = c.qdot;
  a.xref = c.xref;
  a.disp = (Vec4<real> *)c.disp;
  a.ub = make_double3(c.ub[0], c.ub[1], c.ub[2]);
  a.ut = make_double3(c.ut[0], c.ut[1], c.ut[2]);
  a.D = dims_of(c);
  a.health = c.counters + 3;
  return a;
}
int interp_blocks(const Ctx &c) { return (int)((4L * c.nv + kInterpThreads - 1) / kInterpThreads); }

}  // namespace
}  // namespace iblb
