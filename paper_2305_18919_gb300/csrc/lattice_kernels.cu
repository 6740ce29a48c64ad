// Lattice kernels of the step: the stream-collide pass (direct and staged through shared memory),
// launches of the passes in lattice_device.cuh, one context or many per launch, and the read-back
// and initialisation kernels.
#include "lattice_device.cuh"

namespace iblb {
namespace {

// K1: fused stream-collide of every fluid node with the uniform body force only (FORCE: the
// body force is non-zero). The nodes of active interface tiles are collided again by K1t with
// their interface force, so this pass does not wait for the interface chain of the step.
// Each thread owns the two nodes (x0, x0 + 1), x0 even: populations that do not move along x
// and every store are one aligned 2-wide access, and the address arithmetic is shared.
// Each block covers (part of) one lattice row, or with FLAT the next blockDim.x pairs in memory
// order: rows that are no whole number of warps would leave lanes idle (nx = 132: 66 pairs in 96
// lanes, 45 us per pass of 132 x 100 x 77; nx = 32: 16 pairs in 32).
// fin and fout carry no __restrict__: launched early, the kernel is there while the one before it
// still writes fin, and `const __restrict__` would promise that nothing does. The loads, all after
// the wait, are those of load_pair.
template <typename real>
struct K1MinBlocks {  // FP32: 72 registers, 28 warps per SM (64 registers spill and are no faster)
  static constexpr int value = sizeof(real) == 4 ? 7 : 1;
};

template <typename real, typename S, bool FIRST, bool FORCE, bool FLAT>
__global__ void __launch_bounds__(128, K1MinBlocks<real>::value) stream_collide_kernel(
    const S *fin, S *fout, const LatParams<real> P, int z0, const FlatGroups G) {
  int x0, y, z;
  pdl_let_next();
  pdl_wait();
  if (FLAT) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= G.n) return;
    G.at(g, x0, y, z);
    x0 *= 2;
    z += z0;
  } else {
    x0 = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    y = blockIdx.y;
    z = blockIdx.z + z0;
  }
  real a[Q], b[Q];  // populations of nodes x0 and x0 + 1
  load_pair<real, S, FIRST>(fin, P, x0, y, z, a, b);
  collide_pair<FORCE>(a, b, P);
  store_pair(fout, P, (size_t)z * P.nx * P.ny + (size_t)y * P.nx + x0, a, b);
}

// (its threads always take the quads in memory order)
template <typename S, bool FIRST, bool FORCE>
__global__ void __launch_bounds__(128) stream_collide_quad_kernel(const S *fin, S *fout,
                                                                  const LatParams<float> P,
                                                                  int z0, const FlatGroups G) {
  pdl_let_next();
  pdl_wait();
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= G.n) return;
  int gx, y, z;
  G.at(g, gx, y, z);
  quad_nodes<S, FIRST, FORCE>(fin, fout, P, 4 * gx, y, z + z0, Nothing());
}

// --- K1s: stream-collide with the pulled rows staged in shared memory by bulk copies ----------
//
// A unit of work is R lattice rows (y0 .. y0 + R - 1 at one z). The pulled populations of a
// unit are whole x-rows of the population array: population i of row (y, z) streams from row
// (y - c_iy, z - c_iz), or, for a link from a wall node, is population opp(i) of row (y, z)
// itself. A producer warp copies those 19 R rows into a shared-memory stage with cp.async.bulk,
// their completion counted in bytes on the stage's `full` mbarrier; NC compute warps read the
// nodes from the stage (the periodic x wrap is an index into the row), collide them and store
// the results straight to global memory, then release the stage on its `empty` mbarrier. D
// stages rotate, so the bytes in flight per SM are set by shared memory, not by registers.
// Every wait is bounded: a wait that gives up records H_TIMEOUT in the health word and the
// block returns once the producer has waited (again bounded) for its own copies in flight.

__device__ __forceinline__ unsigned smem_addr(const void *p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned long long *bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(unsigned long long *bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long *bar, unsigned parity) {
  unsigned done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return done != 0;
}
// Non-blocking test for the completion of the phase of parity `parity`.
__device__ __forceinline__ bool mbar_test_wait(unsigned long long *bar, unsigned parity) {
  unsigned done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return done != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
constexpr unsigned long long kDrainWaitNs = 1000000000ull;  // the wait for copies in flight
constexpr int kStageWaitPolls = 1 << 26;                     // polls before any wait gives up
// Wait for the completion of the phase of parity `parity`; false if the wait gave up (after
// limit_ns nanoseconds of the global timer) or another warp of the block raised `abort_flag`
// meanwhile. limit_ns = 0: one non-blocking test.
__device__ __forceinline__ bool mbar_wait(unsigned long long *bar, unsigned parity,
                                          const volatile int *abort_flag,
                                          unsigned long long limit_ns) {
  if (limit_ns == 0) return mbar_test_wait(bar, parity);
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  for (int k = 0; k < kStageWaitPolls; k++) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag || global_ns() - t0 > limit_ns) return false;
  }
  return false;
}
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// Bulk copy of `bytes` (a multiple of 16; both addresses 16-byte aligned) from global to
// shared memory, completing `bytes` transactions on mbarrier `bar`.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, unsigned bytes,
                                         unsigned long long *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// Shape of the staged pass: units of R rows, D stages of R * 19 rows of nx values each.
struct StageGeom {
  int z0;            // first fluid layer
  int units_per_z;   // ny / R
  int nunits;        // units_per_z * fluid layers
  int R, D;
  int stage_elems;   // R * 19 * nx
  unsigned long long wait_ns;  // limit of a wait for a stage or for a free stage
};

// Bytes ahead of the first stage: the 2 D mbarriers and the abort flag.
constexpr int kStageHeader = 256;

// Row (z, wall flags) of a unit. Links from a wall exist only on the first and last fluid
// layer, and they are the same for every row of the unit.
struct UnitRows {
  int z, y0, zm, zp;
  bool wall_below, wall_above;
};
template <typename real>
__device__ __forceinline__ UnitRows unit_rows(int unit, const LatParams<real> &P,
                                              const StageGeom &G) {
  UnitRows u;
  u.z = G.z0 + unit / G.units_per_z;
  u.y0 = (unit % G.units_per_z) * G.R;
  u.zm = u.z - 1;
  u.zp = u.z + 1;
  if (!P.has_walls) {
    u.zm = u.z == 0 ? P.nz - 1 : u.zm;
    u.zp = u.z == P.nz - 1 ? 0 : u.zp;
  }
  u.wall_below = P.has_walls && u.zm == 0;
  u.wall_above = P.has_walls && u.zp == P.nz - 1;
  return u;
}

// Signs of c_iy and c_iz as bit masks over i, for run-time direction indices.
__host__ __device__ constexpr unsigned dir_mask(int axis, int sign) {
  unsigned m = 0;
  for (int i = 0; i < Q; i++) {
    const int c = axis == 1 ? cy(i) : cz(i);
    if (c == sign) m |= 1u << i;
  }
  return m;
}
constexpr unsigned kYPos = dir_mask(1, 1), kYNeg = dir_mask(1, -1);
constexpr unsigned kZPos = dir_mask(2, 1), kZNeg = dir_mask(2, -1);
__device__ __forceinline__ int dir_c(unsigned pos, unsigned neg, int i) {
  return (int)((pos >> i) & 1u) - (int)((neg >> i) & 1u);
}

// Producer lanes: queue the copies of `unit` into `stage` (lane 0 has armed `full` with the
// byte count). The stage holds [19][R][nx] values: block i is population i of lattice rows
// y0 .. y0 + R - 1 as pulled, or population opp(i) of those rows for a link from the wall. The
// R source rows of a population are consecutive rows of one plane, so one copy brings them,
// or two where they wrap around y.
template <typename S>
__device__ __forceinline__ void stage_issue(const S *__restrict__ fin, S *stage,
                                            unsigned long long *full, const UnitRows &u,
                                            const LatParams<float> &P, const StageGeom &G,
                                            int lane) {
  if (lane >= Q) return;
  const int i = lane;
  const unsigned row_bytes = (unsigned)(P.nx * sizeof(S));
  const size_t plane = (size_t)P.nx * P.ny;
  const int ciy = dir_c(kYPos, kYNeg, i);
  const int ciz = dir_c(kZPos, kZNeg, i);
  S *dst = stage + (size_t)i * G.R * P.nx;
  if ((ciz > 0 && u.wall_below) || (ciz < 0 && u.wall_above)) {
    const size_t src = (size_t)opp(i) * P.ncell + (size_t)u.z * plane + (size_t)u.y0 * P.nx;
    bulk_g2s(dst, fin + src, G.R * row_bytes, full);
    return;
  }
  const int zs = ciz > 0 ? u.zm : (ciz < 0 ? u.zp : u.z);
  const S *pop = fin + (size_t)i * P.ncell + (size_t)zs * plane;
  const int ys = u.y0 - ciy;  // source of row y0; rows ys .. ys + R - 1 follow (mod ny)
  if (ys < 0) {               // row y0 = 0 pulls from row ny - 1
    bulk_g2s(dst, pop + (size_t)(P.ny - 1) * P.nx, row_bytes, full);
    if (G.R > 1) bulk_g2s(dst + P.nx, pop, (G.R - 1) * row_bytes, full);
  } else if (ys + G.R > P.ny) {  // the last row of the unit pulls from row 0
    if (G.R > 1) bulk_g2s(dst, pop + (size_t)ys * P.nx, (G.R - 1) * row_bytes, full);
    bulk_g2s(dst + (size_t)(G.R - 1) * P.nx, pop, row_bytes, full);
  } else {
    bulk_g2s(dst, pop + (size_t)ys * P.nx, G.R * row_bytes, full);
  }
}

// Compute lanes, FP32 storage: the node pair (x0, x0 + 1) of one lattice row, whose pulled
// population i is the stage row rows + i * stride, collided and stored at node n of fout.
template <bool FORCE>
__device__ __forceinline__ void staged_pair(const float *rows, int stride, int x0,
                                            const UnitRows &u, const LatParams<float> &P,
                                            float *__restrict__ fout, size_t n) {
  const int xm = x0 == 0 ? P.nx - 1 : x0 - 1;  // source of node x0 for c_x = +1
  const int xp = x0 + 2 == P.nx ? 0 : x0 + 2;  // source of node x0 + 1 for c_x = -1
  float a[Q], b[Q];
#pragma unroll
  for (int i = 0; i < Q; i++) {
    const float *row = rows + i * stride;
    if ((cz(i) > 0 && u.wall_below) || (cz(i) < 0 && u.wall_above)) {
      const float2 v = *reinterpret_cast<const float2 *>(row + x0);
      const float wall = cz(i) > 0 ? P.wb[i] : P.wt[i];
      a[i] = v.x + wall;
      b[i] = v.y + wall;
    } else if (cx(i) == 0) {
      const float2 v = *reinterpret_cast<const float2 *>(row + x0);
      a[i] = v.x;
      b[i] = v.y;
    } else if (cx(i) > 0) {
      a[i] = row[xm];
      b[i] = row[x0];
    } else {
      a[i] = row[x0 + 1];
      b[i] = row[xp];
    }
  }
  collide_pair<FORCE>(a, b, P);
  store_pair(fout, P, n, a, b);
}

// Compute lanes, 16-bit storage: the four nodes x0 .. x0 + 3 (as in K1's 16-bit form, with
// the rows read from the stage).
template <typename S, bool FORCE>
__device__ __forceinline__ void staged_quad(const S *rows, int stride, int x0, const UnitRows &u,
                                            const LatParams<float> &P, S *__restrict__ fout,
                                            size_t n) {
  using V2 = typename Storage<S>::V2;
  const int xm = x0 == 0 ? P.nx - 1 : x0 - 1;  // source of node x0 for c_x = +1
  const int xp = x0 + 4 == P.nx ? 0 : x0 + 4;  // source of node x0 + 3 for c_x = -1
  unsigned int lo[Q], hi[Q];
#pragma unroll
  for (int i = 0; i < Q; i++) {
    const S *row = rows + i * stride;
    const uint2 v = *reinterpret_cast<const uint2 *>(row + x0);
    const bool bounced = (cz(i) > 0 && u.wall_below) || (cz(i) < 0 && u.wall_above);
    if (bounced || cx(i) == 0) {
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
#pragma unroll
  for (int h = 0; h < 2; h++) {  // node pairs (x0, x0 + 1), (x0 + 2, x0 + 3)
    unsigned int *pk = h ? hi : lo;
    float2 g[Q];
#pragma unroll
    for (int i = 0; i < Q; i++) {
      g[i] = widen_pair(as_pair<V2>(pk[i]));
      if ((cz(i) > 0 && u.wall_below) || (cz(i) < 0 && u.wall_above)) {
        const float wall = (cz(i) > 0 ? P.wb[i] : P.wt[i]) * float(kscale<S>(i));
        g[i] = add2(g[i], dup(wall));
      }
    }
    collide_pair_scaled<FORCE>(g, P);
#pragma unroll
    for (int i = 0; i < Q; i++) pk[i] = as_bits(narrow_pair<V2>(g[i]));
  }
#pragma unroll
  for (int i = 0; i < Q; i++)
    *reinterpret_cast<uint2 *>(fout + (size_t)i * P.ncell + n) = make_uint2(lo[i], hi[i]);
}

// Compute lanes, 16-bit storage, two nodes x0, x0 + 1 (x0 even): one 4-byte word per row,
// plus the neighbouring 2-byte value for the directions that move along x; the node pair is
// collided exactly as each pair of the four-node form.
template <typename S, bool FORCE>
__device__ __forceinline__ void staged_pair16(const S *rows, int stride, int x0, const UnitRows &u,
                                              const LatParams<float> &P, S *__restrict__ fout,
                                              size_t n) {
  using V2 = typename Storage<S>::V2;
  const int xm = x0 == 0 ? P.nx - 1 : x0 - 1;  // source of node x0 for c_x = +1
  const int xp = x0 + 2 == P.nx ? 0 : x0 + 2;  // source of node x0 + 1 for c_x = -1
  float2 g[Q];
#pragma unroll
  for (int i = 0; i < Q; i++) {
    const S *row = rows + i * stride;
    const unsigned int w = *reinterpret_cast<const unsigned int *>(row + x0);
    const bool bounced = (cz(i) > 0 && u.wall_below) || (cz(i) < 0 && u.wall_above);
    unsigned int pr;
    if (bounced || cx(i) == 0) {
      pr = w;
    } else if (cx(i) > 0) {  // sources x0 - 1, x0
      const unsigned int e = *reinterpret_cast<const unsigned short *>(row + xm);
      pr = __byte_perm(e, w, 0x5410);
    } else {  // sources x0 + 1, x0 + 2
      const unsigned int e = *reinterpret_cast<const unsigned short *>(row + xp);
      pr = __byte_perm(w, e, 0x5432);
    }
    g[i] = widen_pair(as_pair<V2>(pr));
    if (bounced) {  // stored units: the wall term times k_i
      const float wall = (cz(i) > 0 ? P.wb[i] : P.wt[i]) * float(kscale<S>(i));
      g[i] = add2(g[i], dup(wall));
    }
  }
  collide_pair_scaled<FORCE>(g, P);
#pragma unroll
  for (int i = 0; i < Q; i++)
    *reinterpret_cast<unsigned int *>(fout + (size_t)i * P.ncell + n) = as_bits(narrow_pair<V2>(g[i]));
}

// Launch bound of the staged kernel: 8 compute warps and the copying warp with four nodes per
// lane (the four-node form needs ~170 registers), 16 + 1 warps with two.
__host__ __device__ constexpr int staged_threads(int npt) { return npt == 4 ? 288 : 544; }

// K1s: persistent staged stream-collide (not the first step of a run). blockDim.x = 32 (NC + 1)
// (NC <= 8 with NPT = 4, <= 16 with NPT = 2): warps 0 .. NC-1 compute, warp NC produces. Block
// b takes units b, b + gridDim.x, ... NPT nodes per compute lane: 2 for FP32, 2 or 4 for 16-bit
// storage.
template <typename S, bool FORCE, int NPT>
__global__ void __launch_bounds__(staged_threads(NPT), 1) stream_collide_staged_kernel(
    const S *__restrict__ fin, S *__restrict__ fout, const LatParams<float> P,
    const StageGeom G, int *__restrict__ health) {
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned long long *full = reinterpret_cast<unsigned long long *>(smem);
  unsigned long long *empty = full + G.D;
  volatile int *abort_flag = reinterpret_cast<volatile int *>(empty + G.D);
  S *stages = reinterpret_cast<S *>(smem + kStageHeader);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int NC = (blockDim.x >> 5) - 1;
  if (threadIdx.x == 0) {
    for (int s = 0; s < G.D; s++) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, NC);
    }
    *abort_flag = 0;
    fence_barrier_init();
  }
  __syncthreads();
  const int my_units = G.nunits > (int)blockIdx.x
                           ? (G.nunits - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x
                           : 0;
  if (warp == NC) {  // producer
    int issued = 0;
    for (int k = 0; k < my_units; k++) {
      const int s = k % G.D;
      if (k >= G.D) {  // stage s is free once every compute warp released unit k - D
        bool ok = true;
        if (lane == 0) ok = mbar_wait(empty + s, ((k / G.D) - 1) & 1, abort_flag, G.wait_ns);
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok) {
          if (lane == 0) {
            *abort_flag = 1;
            atomicOr(health, H_TIMEOUT);
          }
          break;
        }
      }
      const UnitRows u = unit_rows(blockIdx.x + k * gridDim.x, P, G);
      S *stage = stages + (size_t)s * G.stage_elems;
      if (lane == 0) {
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(full + s, (unsigned)(G.R * Q * P.nx * sizeof(S)));
      }
      __syncwarp();
      stage_issue(fin, stage, full + s, u, P, G, lane);
      issued = k + 1;
    }
    // copies still in flight land before the block exits: those of the last D units issued
    // (a unit before them was waited for by every compute warp before its stage was reused)
    if (lane == 0) {
      const int no_abort = 0;
      for (int k = issued - G.D < 0 ? 0 : issued - G.D; k < issued; k++)
        if (!mbar_wait(full + k % G.D, (k / G.D) & 1, &no_abort, kDrainWaitNs))
          atomicOr(health, H_TIMEOUT);
    }
    return;
  }
  // compute warps
  const int per_row = P.nx / NPT;
  const size_t plane = (size_t)P.nx * P.ny;
  for (int k = 0; k < my_units; k++) {
    const int s = k % G.D;
    if (!__all_sync(0xffffffffu, mbar_wait(full + s, (k / G.D) & 1, abort_flag, G.wait_ns))) {
      if (lane == 0) {
        *abort_flag = 1;
        atomicOr(health, H_TIMEOUT);
      }
      return;
    }
    const UnitRows u = unit_rows(blockIdx.x + k * gridDim.x, P, G);
    const S *stage = stages + (size_t)s * G.stage_elems;
    for (int w = warp * 32 + lane; w < G.R * per_row; w += NC * 32) {
      const int r = w / per_row, x0 = NPT * (w - r * per_row);
      const size_t n = (size_t)u.z * plane + (size_t)(u.y0 + r) * P.nx + x0;
      if constexpr (sizeof(S) == 2 && NPT == 4)
        staged_quad<S, FORCE>(stage + (size_t)r * P.nx, G.R * P.nx, x0, u, P, fout, n);
      else if constexpr (sizeof(S) == 2)
        staged_pair16<S, FORCE>(stage + (size_t)r * P.nx, G.R * P.nx, x0, u, P, fout, n);
      else
        staged_pair<FORCE>(stage + (size_t)r * P.nx, G.R * P.nx, x0, u, P, fout, n);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(empty + s);
  }
}

// K1 over many contexts in one launch (the batched ensemble; never the first, in-place step):
// each thread takes one node group in memory order, a pair (x0, x0 + 1) or, with 16-bit
// storage, four nodes x0 .. x0 + 3, and runs the very code of the single-context kernels on it,
// so each context's populations come out bit for bit as from those.
// Blocks per SM of the batched pass, run as a persistent grid over its blocks. A pass that does not
// fill the SMs leaves room for the interface kernels of the other streams, which then run beside
// it instead of after it (96 wetting boxes, ms per step: with the interface force taken in, on
// three lanes, 1.162 with 6, 1.178 with 4 or 3; without it, beside a partitioned chain, 1.317 with
// 4, 1.402 with 6).
constexpr int k1_multi_per_sm(bool forced) { return forced ? 6 : 4; }

// Blocks per SM that the registers are bounded for with FP32 storage; the others would spill.
template <typename real, typename S>
struct MultiMinBlocks {
  static constexpr int value = sizeof(real) == 4 && sizeof(S) == 4 ? 4 : 1;
};

// FORCED: with the interface force of the step (forced_group), else the body force only.
template <typename real, typename S, bool FORCED>
__global__ void __launch_bounds__(128, MultiMinBlocks<real, S>::value) stream_collide_kernel_multi(
    const StreamArgs<real, S> *__restrict__ all, const int *__restrict__ start, int n) {
  __shared__ int s_start[kMultiMax + 1];
  pdl_let_next();
  for (int k = threadIdx.x; k <= n; k += blockDim.x) s_start[k] = start[k];
  __syncthreads();
  pdl_wait();
  const int total = s_start[n];
  for (int vb = blockIdx.x; vb < total; vb += gridDim.x) {
    const MultiBlock m = multi_block_of(s_start, n, vb);
    const StreamArgs<real, S> &A = all[m.inst];
    const int g = m.block * blockDim.x + threadIdx.x;
    if (g >= A.G.n) continue;
    int gx, y, z;
    A.G.at(g, gx, y, z);
    z += A.z0;
    if constexpr (FORCED) {
      if (A.force) forced_group<real, S, true>(A, gx, y, z);
      else forced_group<real, S, false>(A, gx, y, z);
    } else if constexpr (sizeof(S) == 2) {
      if (A.force) quad_nodes<S, false, true>(A.fin, A.fout, A.P, 4 * gx, y, z, Nothing());
      else quad_nodes<S, false, false>(A.fin, A.fout, A.P, 4 * gx, y, z, Nothing());
    } else {
      const int x0 = 2 * gx;
      real a[Q], b[Q];
      load_pair<real, S, false>(A.fin, A.P, x0, y, z, a, b);
      if (A.force) collide_pair<true>(a, b, A.P);
      else collide_pair<false>(a, b, A.P);
      store_pair(A.fout, A.P, (size_t)z * A.P.nx * A.P.ny + (size_t)y * A.P.nx + x0, a, b);
    }
  }
}

// Threads per block of K1t: few, so that a short list spreads over all SMs (the kernel's time
// there is one pair's chain of loads and arithmetic).
constexpr int kTilesThreads = 64;

template <typename real, typename S>
__global__ void __launch_bounds__(kTilesThreads) stream_collide_tiles_kernel(const TilesArgs<real, S> A) {
  tiles_body<true>(A, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

template <typename real, typename S>
__global__ void __launch_bounds__(kTilesThreads, sizeof(real) == 4 ? 8 : 1) stream_collide_tiles_kernel_multi(
    const TilesArgs<real, S> *__restrict__ all, const int *__restrict__ start, int n) {
  const MultiBlock m = multi_block(start, n);
  tiles_body<true>(all[m.inst], m.block * blockDim.x + threadIdx.x, m.nblocks * blockDim.x);
}

template <typename real, typename S>
__global__ void __launch_bounds__(128) shell_velocity_kernel(const ShellArgs<real, S> A) {
  shell_body<real, S>(A, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

template <typename real, typename S>
__global__ void __launch_bounds__(128) shell_velocity_kernel_multi(
    const ShellArgs<real, S> *__restrict__ all, const int *__restrict__ start, int n) {
  const MultiBlock m = multi_block(start, n);
  shell_body<real, S>(all[m.inst], m.block * blockDim.x + threadIdx.x, m.nblocks * blockDim.x);
}

// rho - rho0 and u of one node for the read-back, in double.
//
// FP64 contexts compute in double, with one residual correction of each quotient by the
// reciprocal. Float contexts carry every value as an unevaluated pair of floats hi + lo: sums by
// TwoSum (Knuth: the exact error of each addition, six float operations), quotients by one
// residual step (Dekker), about 2^-45 of the value, and widen the pair once at the end. One FP64
// operation takes the issue slots of 64 float operations on this GPU; in double, the sums and
// quotients of a node took 18 times as long as its bytes.

// (double)f by moving its bits: zeros and normal floats, the conversion instruction otherwise.
__device__ __forceinline__ double widened(float f) {
  const unsigned u = __float_as_uint(f), sign = u & 0x80000000u, mag = u ^ sign;
  if (mag == 0u) return __hiloint2double((int)sign, 0);
  if (mag - 0x00800000u >= 0x7f000000u) return (double)f;  // subnormal, infinite or NaN
  return __hiloint2double((int)(sign | ((mag >> 3) + 0x38000000u)), (int)(mag << 29));
}

template <typename real>
struct Pair;  // a value of the read-back's arithmetic
template <>
struct Pair<double> {
  double v;
  __device__ __forceinline__ explicit Pair(double f) : v(f) {}
  __device__ __forceinline__ void add(double f) { v = add_(v, f); }
  __device__ __forceinline__ double value() const { return v; }
};
template <>
struct Pair<float> {
  float hi, lo;
  __device__ __forceinline__ explicit Pair(float f, float e = 0.0f) : hi(f), lo(e) {}
  __device__ __forceinline__ void add(float f) {
    const float s = __fadd_rn(hi, f), b = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(f, b)));
    hi = s;
  }
  __device__ __forceinline__ double value() const {  // (the error of inf is no number)
    return isfinite(hi) ? widened(hi) + widened(lo) : (double)hi;
  }
};

// u = j / (rho0 + drho) of the two nodes of a pair.
__device__ __forceinline__ void field_quotients(const Pair<double> &ma, const Pair<double> &mb,
                                                const Pair<double> ja[3], const Pair<double> jb[3],
                                                double rho0, double ua[3], double ub[3]) {
  const double ra = rho0 + ma.v, rb = rho0 + mb.v;
  double ia, ib;
  reciprocals(ra, rb, ia, ib);
#pragma unroll
  for (int k = 0; k < 3; k++) {
    ua[k] = mul_(ja[k].v, ia);
    ub[k] = mul_(jb[k].v, ib);
    // (no residual of an infinity; the exponent's bits cost no FP64 issue slot)
    if ((__double2hiint(ua[k]) & 0x7ff00000) != 0x7ff00000)
      ua[k] = fma(fma(-ua[k], ra, ja[k].v), ia, ua[k]);
    if ((__double2hiint(ub[k]) & 0x7ff00000) != 0x7ff00000)
      ub[k] = fma(fma(-ub[k], rb, jb[k].v), ib, ub[k]);
  }
}
__device__ __forceinline__ void field_quotient(const Pair<float> &m, const Pair<float> j[3],
                                               double rho0, double u[3]) {
  const float r0 = (float)rho0, r0e = (float)(rho0 - (double)r0);
  Pair<float> r(r0, __fadd_rn(r0e, m.lo));
  r.add(m.hi);
  const float rh = __fadd_rn(r.hi, r.lo), rl = __fsub_rn(r.lo, __fsub_rn(rh, r.hi));
  const float inv = 1.0f / rh;
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const float jh = __fadd_rn(j[k].hi, j[k].lo);
    const float jl = __fsub_rn(j[k].lo, __fsub_rn(jh, j[k].hi));
    const float q = __fmul_rn(jh, inv);
    // jh - q rh is a float (q is jh / rh to within two roundings), the fused form gives it
    const float res = __fadd_rn(__fmaf_rn(-q, rh, jh), __fmaf_rn(-q, rl, jl));
    u[k] = Pair<float>(q, __fmul_rn(res, inv)).value();
  }
}
__device__ __forceinline__ void field_quotients(const Pair<float> &ma, const Pair<float> &mb,
                                                const Pair<float> ja[3], const Pair<float> jb[3],
                                                double rho0, double ua[3], double ub[3]) {
  field_quotient(ma, ja, rho0, ua);
  field_quotient(mb, jb, rho0, ub);
}

// drho and the momentum j (with half the force F) of one node; m and j hold f[0] and f[1], f[3],
// f[5] on entry.
__device__ __forceinline__ void field_sums(const double f[Q], const double F[3], Pair<double> &m,
                                           Pair<double> j[3]) {
  double jd[3];
  node_moments(f, m.v, jd);
#pragma unroll
  for (int k = 0; k < 3; k++) j[k].v = F[k] != 0.0 ? fma(0.5, F[k], jd[k]) : jd[k];
}
__device__ __forceinline__ void field_sums(const float f[Q], const float F[3], Pair<float> &m,
                                           Pair<float> j[3]) {
#pragma unroll
  for (int i = 1; i < Q; i++) {
    m.add(f[i]);
    if (cx(i) && i != 1) j[0].add(cx(i) > 0 ? f[i] : -f[i]);
    if (cy(i) && i != 3) j[1].add(cy(i) > 0 ? f[i] : -f[i]);
    if (cz(i) && i != 5) j[2].add(cz(i) > 0 ? f[i] : -f[i]);
  }
#pragma unroll
  for (int k = 0; k < 3; k++)
    if (F[k] != 0.0f) j[k].add(0.5f * F[k]);
}

// rho and u of every node of the current post-streaming state (read-back, not on the step). A
// thread per node pair: the pair's populations as the stream-collide pass loads them, 16-byte
// stores. 256^3 FP32: 0.370 ms (0.72 of the copy bandwidth) against 4.81 ms with a thread per
// node in double; FP16 0.388 against 4.82; 128^3 FP64, bound by the FP64 units, 0.30 against 0.56.
struct FieldsArgs {
  double3 ub, ut;
  double rho0;
  double *rho, *u;
};

template <typename real, typename S, bool FRESH>
__global__ void __launch_bounds__(128) fields_kernel(const S *__restrict__ fstate,
                                                     const int *__restrict__ tile_slot,
                                                     const Vec4<real> *__restrict__ Fslot,
                                                     const LatParams<real> P, const FieldsArgs A,
                                                     const FlatGroups G) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= G.n) return;
  int x0, y, z;
  G.at(g, x0, y, z);
  x0 *= 2;
  const size_t n = ((size_t)z * P.ny + y) * P.nx + x0;
  double2 rho, u[3];
  if (P.has_walls && (z == 0 || z == P.nz - 1)) {
    const double3 w = z == 0 ? A.ub : A.ut;
    rho = make_double2(A.rho0, A.rho0);
    u[0] = make_double2(w.x, w.y);
    u[1] = make_double2(w.z, w.x);
    u[2] = make_double2(w.y, w.z);
  } else {
    real a[Q], b[Q];
    load_pair<real, S, FRESH>(fstate, P, x0, y, z, a, b);
    real Fa[3], Fb[3];
    tile_force_pair(tile_slot, Fslot, P, x0, y, z, Fa, Fb);
    Pair<real> ma(a[0]), mb(b[0]);
    Pair<real> ja[3] = {Pair<real>(a[1]), Pair<real>(a[3]), Pair<real>(a[5])};
    Pair<real> jb[3] = {Pair<real>(b[1]), Pair<real>(b[3]), Pair<real>(b[5])};
    field_sums(a, Fa, ma, ja);
    field_sums(b, Fb, mb, jb);
    double ua[3], ub[3];
    field_quotients(ma, mb, ja, jb, A.rho0, ua, ub);
    rho = make_double2(A.rho0 + ma.value(), A.rho0 + mb.value());
    u[0] = make_double2(ua[0], ua[1]);
    u[1] = make_double2(ua[2], ub[0]);
    u[2] = make_double2(ub[1], ub[2]);
  }
  // the caller's buffers are doubles: 16-byte stores where they are aligned to them
  double *ro = A.rho + n, *uo = A.u + 3 * n;
  if ((((size_t)A.rho | (size_t)A.u) & 15) == 0) {
    *reinterpret_cast<double2 *>(ro) = rho;
#pragma unroll
    for (int k = 0; k < 3; k++) reinterpret_cast<double2 *>(uo)[k] = u[k];
  } else {
    ro[0] = rho.x;
    ro[1] = rho.y;
#pragma unroll
    for (int k = 0; k < 3; k++) {
      uo[2 * k] = u[k].x;
      uo[2 * k + 1] = u[k].y;
    }
  }
}

template <typename real, typename S>
__global__ void populations_kernel(const S *__restrict__ fstate, int fresh,
                                   const LatParams<real> P, double rho0,
                                   double *__restrict__ f_out) {
  const size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (n >= P.ncell) return;
  const int x = (int)(n % P.nx), y = (int)((n / P.nx) % P.ny), z = (int)(n / ((size_t)P.nx * P.ny));
  if (P.has_walls && (z == 0 || z == P.nz - 1)) {
    for (int i = 0; i < Q; i++) f_out[(size_t)i * P.ncell + n] = 0.0;
    return;
  }
  real f[Q];
  if (fresh) {
    for (int i = 0; i < Q; i++) f[i] = dev<real>(fstate, i, (size_t)i * P.ncell + n);
  } else {
    pull(fstate, P, x, y, z, f);
  }
  for (int i = 0; i < Q; i++) f_out[(size_t)i * P.ncell + n] = wgt(i) * rho0 + (double)f[i];
}

template <typename real, typename S>
__global__ void init_equilibrium_kernel(S *__restrict__ fstate, const LatParams<real> P,
                                        double rho0, const double *__restrict__ rho_in,
                                        const double *__restrict__ u_in) {
  const size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (n >= P.ncell) return;
  const int z = (int)(n / ((size_t)P.nx * P.ny));
  const bool wall = P.has_walls && (z == 0 || z == P.nz - 1);
  const double rho = rho_in[n];
  const double ux = u_in[3 * n], uy = u_in[3 * n + 1], uz = u_in[3 * n + 2];
  const double uu = ux * ux + uy * uy + uz * uz;
  for (int i = 0; i < Q; i++) {
    const double cu = cx(i) * ux + cy(i) * uy + cz(i) * uz;
    const double v = wgt(i) * ((rho - rho0) + rho * (3.0 * cu + 4.5 * cu * cu - 1.5 * uu));
    fstate[(size_t)i * P.ncell + n] = Narrow<S>::one(wall ? real(0) : (real)(v * kscale<S>(i)));
  }
}

// Without a mesh the pass follows the last step's on its stream, and is launched early (64^3 FP32
// 6.5 us per step against 8.4, 132x100x77 24.9 against 27.4, 84x68x64 FP16 5.5 against 8.4); with
// one it waits for events. Not in FP64, where the blocks that arrive early crowd the SMs that are
// free first and then share their FP64 units (32^3: 31 us against 14.5).
bool follows_itself(const Ctx &c) { return c.nv == 0 && c.pop_size < 8; }

// Threads per block of K1's flat kernels: what the tuner chose, as the threads of that many
// lattice rows (whole warps, at most 128), else 128, or 64 with FP64 arithmetic, whose small
// lattices spread more evenly over the SMs (the pass is bound by each SM's FP64 units).
template <typename S>
int k1_flat_threads(const Ctx &c, int per_row) {
  if (c.k1_rows <= 0) return sizeof(S) == 8 ? 64 : 128;
  const int t = (per_row * k1_block_rows(c) + 31) / 32 * 32;
  return t < 128 ? t : 128;
}

template <typename S>
cudaError_t stream_collide_quad_t(Ctx &c, int first, cudaStream_t st) {
  const LatParams<float> P = lat_params<float>(c);
  const int z0 = c.has_walls ? 1 : 0;
  const FlatGroups G = k1_groups<S>(c);
  const int block = k1_flat_threads<S>(c, G.per_row.d), grid = (G.n + block - 1) / block;
  const S *fin = (const S *)c.f[c.cur];
  S *fout = (S *)c.f[c.cur ^ 1];
  const bool force = c.g[0] != 0.0 || c.g[1] != 0.0 || c.g[2] != 0.0;
  auto *kern = first ? (force ? stream_collide_quad_kernel<S, true, true>
                              : stream_collide_quad_kernel<S, true, false>)
                     : (force ? stream_collide_quad_kernel<S, false, true>
                              : stream_collide_quad_kernel<S, false, false>);
  return launch_after(follows_itself(c), kern, dim3(grid), block, st, fin, fout, P, z0, G);
}

// Nodes per compute lane of the staged pass: 2 for FP32; for 16-bit storage k1_nodes, by
// default kStageNodes16.
template <typename S>
int staged_nodes(const Ctx &c) {
  if (sizeof(S) != 2) return 2;
  return c.k1_nodes > 0 ? c.k1_nodes : kStageNodes16;
}

// Shape of the staged pass on context c (false where it does not apply: a row of the storage
// type that is not a whole number of 16-byte blocks, or too little shared memory for two
// stages). R lattice rows per unit (`rows`, or by default as many as keep one population's
// copy within kStageCopyBytes): the copies are few and large, which the copy engine needs.
template <typename S>
bool stage_geom(const Ctx &c, int stages, int rows, StageGeom &G, size_t &smem) {
  const int NPT = staged_nodes<S>(c);
  const size_t row_bytes = (size_t)c.nx * sizeof(S);
  if (row_bytes % 16 != 0 || c.nx % NPT != 0) return false;
  auto fits = [&](int r, int d) { return kStageHeader + (size_t)d * r * Q * row_bytes <= (size_t)c.smem_optin; };
  int R = rows;
  if (R <= 0) {
    R = 1;
    while (R < 16 && c.ny % (2 * R) == 0 && 2 * R * row_bytes <= kStageCopyBytes && fits(2 * R, 2))
      R *= 2;
  }
  if (c.ny % R != 0 || !fits(R, 2)) return false;
  const size_t stage_bytes = (size_t)R * Q * row_bytes;
  int D = stages;
  while (D > 2 && !fits(R, D)) D--;
  G.z0 = c.has_walls ? 1 : 0;
  G.units_per_z = c.ny / R;
  G.nunits = G.units_per_z * (c.has_walls ? c.nz - 2 : c.nz);
  G.R = R;
  G.D = D;
  G.stage_elems = R * Q * c.nx;
  G.wait_ns = c.stage_wait_ns;
  smem = kStageHeader + D * stage_bytes;
  return true;
}

template <typename S, bool FORCE, int NPT>
cudaError_t launch_staged(Ctx &c, const StageGeom &G, size_t smem, int nc, cudaStream_t st) {
  auto kern = stream_collide_staged_kernel<S, FORCE, NPT>;
  if (32 * (nc + 1) > staged_threads(NPT)) nc = staged_threads(NPT) / 32 - 1;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // one block per SM of the lattice partition (of all SMs without a mesh), each working through
  // its share of the units
  const int sms = c.green[0] && c.nv ? c.lat_sms : c.sm_count;
  const int grid = G.nunits < sms ? G.nunits : sms;
  kern<<<grid, 32 * (nc + 1), smem, st>>>((const S *)c.f[c.cur], (S *)c.f[c.cur ^ 1],
                                          lat_params<float>(c), G, c.counters + 3);
  return cudaGetLastError();
}

// The kind of stream-collide kernel asked for, resolved for storage type S: AUTO takes the
// staged kernel for 16-bit storage, where it is the faster one (for FP32 the direct kernel
// already runs at the copy bandwidth).
template <typename S>
bool staged_kind(const Ctx &c) {
  if (sizeof(S) == 8 || c.k1_kind == IBLB_STREAM_COLLIDE_DIRECT) return false;
  return c.k1_kind == IBLB_STREAM_COLLIDE_STAGED || sizeof(S) == 2;
}

template <typename real, typename S>
bool uses_staged_t(const Ctx &c) {
  StageGeom G;
  size_t smem = 0;
  return staged_kind<S>(c) &&
         stage_geom<S>(c, c.k1_stages > 0 ? c.k1_stages : kStages, c.k1_unit_rows, G, smem);
}

// K1 through the staged kernel where it applies; *used tells whether it did.
template <typename real, typename S>
cudaError_t stream_collide_staged_t(Ctx &c, cudaStream_t st, bool *used) {
  *used = false;
  if constexpr (sizeof(S) == 8) {
    return cudaSuccess;
  } else {
    const int nc = c.k1_warps > 0 ? c.k1_warps : kStageWarps;
    const int stages = c.k1_stages > 0 ? c.k1_stages : kStages;
    StageGeom G;
    size_t smem = 0;
    if (!staged_kind<S>(c) || !stage_geom<S>(c, stages, c.k1_unit_rows, G, smem))
      return cudaSuccess;
    *used = true;
    const bool force = c.g[0] != 0.0 || c.g[1] != 0.0 || c.g[2] != 0.0;
    if constexpr (sizeof(S) == 2)
      if (staged_nodes<S>(c) == 4)
        return force ? launch_staged<S, true, 4>(c, G, smem, nc, st)
                     : launch_staged<S, false, 4>(c, G, smem, nc, st);
    return force ? launch_staged<S, true, 2>(c, G, smem, nc, st)
                 : launch_staged<S, false, 2>(c, G, smem, nc, st);
  }
}

template <typename real, typename S>
cudaError_t stream_collide_t(Ctx &c, int first, cudaStream_t st) {
  if (!first) {
    bool used = false;
    const cudaError_t e = stream_collide_staged_t<real, S>(c, st, &used);
    if (used) return e;
  }
  if constexpr (sizeof(S) == 2) {
    return stream_collide_quad_t<S>(c, first, st);
  } else {
    const LatParams<real> P = lat_params<real>(c);
    const int z0 = c.has_walls ? 1 : 0;
    const FlatGroups G = k1_groups<S>(c);
    const int per_row = G.per_row.d;
    // a block per row where a row is a whole number of warps, at least two of them, and of
    // 128-thread blocks (it saves the flat form's index arithmetic), else the flat form
    const bool rows = c.k1_rows <= 1 && (per_row <= 128 ? per_row >= 64 && per_row % 32 == 0
                                                        : per_row % 128 == 0);
    const int block = rows ? (per_row < 128 ? per_row : 128) : k1_flat_threads<S>(c, per_row);
    const dim3 grid = rows ? dim3(per_row / block, c.ny, c.has_walls ? c.nz - 2 : c.nz)
                           : dim3((G.n + block - 1) / block);
    const S *fin = (const S *)c.f[c.cur];
    S *fout = (S *)c.f[c.cur ^ 1];
    const bool force = c.g[0] != 0.0 || c.g[1] != 0.0 || c.g[2] != 0.0;
    auto launch = [&](auto first_c, auto force_c, auto flat_c) {
      return launch_after(follows_itself(c),
                          stream_collide_kernel<real, S, decltype(first_c)::value,
                                                decltype(force_c)::value, decltype(flat_c)::value>,
                          grid, block, st, fin, fout, P, z0, G);
    };
    using T = std::true_type;
    using F = std::false_type;
    if (first) {
      if (force) return rows ? launch(T(), T(), F()) : launch(T(), T(), T());
      return rows ? launch(T(), F(), F()) : launch(T(), F(), T());
    }
    if (force) return rows ? launch(F(), T(), F()) : launch(F(), T(), T());
    return rows ? launch(F(), F(), F()) : launch(F(), F(), T());
  }
}

// a thread per listed pair; single context: eight 64-thread blocks per SM (about 78k pairs
// in one pass); in a batch a block per four of the context's expected active tiles
int tiles_blocks(const Ctx &c, bool batched) {
  int grid = batched ? (c.tile_estimate + 3) / 4 : c.sm_count * 8;
  if (grid > c.max_slots) grid = c.max_slots;
  return grid < 1 ? 1 : grid;
}

// a thread per node of a listed pair, 128 per block; single context: sixteen blocks per SM of
// the partition it runs on; in a batch a block per two of the context's expected active tiles
int shell_blocks(const Ctx &c, bool batched) {
  const int sms = c.ib_sms > 0 ? c.ib_sms : c.sm_count;
  int grid = batched ? (c.tile_estimate + 1) / 2 : sms * 16;
  if (grid > c.max_slots) grid = c.max_slots;
  return grid < 1 ? 1 : grid;
}

template <typename real, typename S>
cudaError_t stream_collide_tiles_t(Ctx &c, int first, cudaStream_t st) {
  const int grid = tiles_blocks(c, false);
  (void)first;  // K1t corrects K1's output in place, whatever K1 read
  stream_collide_tiles_kernel<real, S><<<grid, kTilesThreads, 0, st>>>(tiles_args<real, S>(c));
  return cudaGetLastError();
}

template <typename real, typename S>
cudaError_t shell_velocity_t(Ctx &c, cudaStream_t st) {
  shell_velocity_kernel<real, S><<<shell_blocks(c, false), 128, 0, st>>>(
      shell_args<real, S>(c, c.f[c.cur]));
  return cudaGetLastError();
}

template <typename T>
void append_record(std::vector<unsigned char> &bytes, const T &rec) {
  const size_t off = bytes.size();
  bytes.resize(off + sizeof(T));
  memcpy(bytes.data() + off, &rec, sizeof(T));
}

template <typename real, typename S>
int lattice_multi_record_t(const Ctx &c, MultiKernel k, std::vector<unsigned char> &bytes) {
  switch (k) {
    case MK_FORCED:
    case MK_STREAM_COLLIDE: {
      const StreamArgs<real, S> a = stream_args<real, S>(c);
      append_record(bytes, a);
      const int b = (a.G.n + 127) / 128;
      return b < 1 ? 1 : b;
    }
    case MK_TILES: append_record(bytes, tiles_args<real, S>(c)); return tiles_blocks(c, true);
    case MK_SHELL:
      append_record(bytes, shell_args<real, S>(c, c.f[c.cur ^ 1]));
      return shell_blocks(c, true);
    default: return -1;
  }
}

template <typename real, typename S>
cudaError_t lattice_launch_multi_t(MultiKernel k, const MultiLaunch &m, cudaStream_t s) {
  switch (k) {
    case MK_FORCED:
    case MK_STREAM_COLLIDE: {
      static int sms = 0;
      if (!sms && cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, 0) != cudaSuccess)
        sms = 0;
      const int cap = k1_multi_per_sm(k == MK_FORCED) * sms;
      const int grid = cap > 0 && m.blocks > cap ? cap : m.blocks;
      const auto *args = (const StreamArgs<real, S> *)m.args;
      return k == MK_FORCED
                 ? launch_after(m.early, stream_collide_kernel_multi<real, S, true>, grid, 128, s, args, m.start, m.n)
                 : launch_after(m.early, stream_collide_kernel_multi<real, S, false>, grid, 128, s, args, m.start, m.n);
    }
    case MK_TILES:
      return launch_after(m.early, stream_collide_tiles_kernel_multi<real, S>, m.blocks, kTilesThreads, s,
                          (const TilesArgs<real, S> *)m.args, m.start, m.n);
    case MK_SHELL:
      return launch_after(m.early, shell_velocity_kernel_multi<real, S>, m.blocks, 128, s,
                          (const ShellArgs<real, S> *)m.args, m.start, m.n);
    default:
      return cudaErrorInvalidValue;
  }
}

template <typename real, typename S>
cudaError_t fields_t(Ctx &c, double *rho_dev, double *u_dev) {
  const FlatGroups G = flat_groups(c.nx / 2, c.ny, c.nz);
  const int block = 128, grid = (G.n + block - 1) / block;
  FieldsArgs A;
  A.ub = make_double3(c.ub[0], c.ub[1], c.ub[2]);
  A.ut = make_double3(c.ut[0], c.ut[1], c.ut[2]);
  A.rho0 = c.rho0;
  A.rho = rho_dev;
  A.u = u_dev;
  // the force of the last spreading step lives in the map that step used
  const int *ts = (c.nv && c.have_force) ? c.tile_slot[c.map ^ 1] : nullptr;
  const S *f = (const S *)c.f[c.cur];
  const Vec4<real> *F = (const Vec4<real> *)c.Fslot[c.map ^ 1];
  const LatParams<real> P = lat_params<real>(c);
  if (c.fresh) fields_kernel<real, S, true><<<grid, block, 0, c.stream>>>(f, ts, F, P, A, G);
  else fields_kernel<real, S, false><<<grid, block, 0, c.stream>>>(f, ts, F, P, A, G);
  return cudaGetLastError();
}

template <typename real, typename S>
cudaError_t populations_t(Ctx &c, double *f_dev) {
  const int blocks = (int)((c.ncell + 255) / 256);
  populations_kernel<real, S><<<blocks, 256, 0, c.stream>>>(
      (const S *)c.f[c.cur], c.fresh, lat_params<real>(c), c.rho0, f_dev);
  return cudaGetLastError();
}

template <typename real, typename S>
cudaError_t init_equilibrium_t(Ctx &c, const double *rho_dev, const double *u_dev) {
  const int blocks = (int)((c.ncell + 255) / 256);
  init_equilibrium_kernel<real, S><<<blocks, 256, 0, c.stream>>>(
      (S *)c.f[c.cur], lat_params<real>(c), c.rho0, rho_dev, u_dev);
  return cudaGetLastError();
}

}  // namespace

int k1_block_rows(const Ctx &c) {
  // a block is at most 128 threads (the kernels' launch bound); ny is a multiple of 4, so
  // every row count 1, 2, 4 divides it
  const int per_row = c.pop_size == 2 ? c.nx / 4 : c.nx / 2;
  const int bx = per_row < 128 ? per_row : 128;
  int rows = c.k1_rows > 0 ? c.k1_rows : 1;
  while (rows > 1 && bx * rows > 128) rows /= 2;
  return rows;
}

// Dispatch on the context's precision: (arithmetic, storage) = (double, double) for FP64,
// (float, float) for FP32, (float, half) for FP16 and (float, bfloat16) for BF16.
#define IBLB_DISPATCH(c, FN, ...)                                         \
  switch ((c).precision) {                                                \
    case IBLB_FP64: return FN<double, double>(__VA_ARGS__);               \
    case IBLB_FP16: return FN<float, __half>(__VA_ARGS__);                \
    case IBLB_BF16: return FN<float, __nv_bfloat16>(__VA_ARGS__);         \
    default: return FN<float, float>(__VA_ARGS__);                        \
  }

bool stream_collide_staged(const Ctx &c) { IBLB_DISPATCH(c, uses_staged_t, c) }

int lattice_multi_record(const Ctx &c, MultiKernel k, std::vector<unsigned char> &bytes) {
  IBLB_DISPATCH(c, lattice_multi_record_t, c, k, bytes)
}

cudaError_t lattice_launch_multi(int precision, MultiKernel k, const MultiLaunch &m,
                                 cudaStream_t s) {
  switch (precision) {
    case IBLB_FP64: return lattice_launch_multi_t<double, double>(k, m, s);
    case IBLB_FP16: return lattice_launch_multi_t<float, __half>(k, m, s);
    case IBLB_BF16: return lattice_launch_multi_t<float, __nv_bfloat16>(k, m, s);
    default: return lattice_launch_multi_t<float, float>(k, m, s);
  }
}

cudaError_t launch_stream_collide(Ctx &c, int first, cudaStream_t s) {
  IBLB_DISPATCH(c, stream_collide_t, c, first, s)
}

cudaError_t launch_stream_collide_tiles(Ctx &c, int first, cudaStream_t s) {
  IBLB_DISPATCH(c, stream_collide_tiles_t, c, first, s)
}

cudaError_t launch_shell_velocity(Ctx &c, cudaStream_t s) { IBLB_DISPATCH(c, shell_velocity_t, c, s) }

cudaError_t launch_fields(Ctx &c, double *rho_dev, double *u_dev) {
  IBLB_DISPATCH(c, fields_t, c, rho_dev, u_dev)
}

cudaError_t launch_populations(Ctx &c, double *f_dev) { IBLB_DISPATCH(c, populations_t, c, f_dev) }

cudaError_t launch_init_equilibrium(Ctx &c, const double *rho_dev, const double *u_dev) {
  IBLB_DISPATCH(c, init_equilibrium_t, c, rho_dev, u_dev)
}

}  // namespace iblb
