// The whole coupled step as one cooperative kernel, for lattices whose step is bound by the chain
// of small passes rather than by the lattice pass.
//
// On a small or ordinary lattice the step is a chain of seven short passes (face forces, vertex
// gather, two spreading passes, active-tile correction, shell velocity, interpolation), each a few
// microseconds of latency; as kernels of their own they also pay a launch gap of 1.5 to 3 us
// between any two, and only the SMs of the interface partition work on them. Here the passes run
// as phases of one resident grid, with a barrier of the grid between two of them, and a launch
// advances many steps. The device code of the phases is that of the separate kernels, so the
// results are the same bit for bit.
//
// Half of the blocks (one per SM of those that the grid is sized for, fused_sms) run the interface phases. The other half run the lattice pass of
// the same step meanwhile (it needs the previous step's populations only); a block of the first
// half that is done with the spreading helps with what is left of the lattice pass. Both halves
// then correct the active tiles, after which the second half starts the next step's lattice pass
// while the first finishes this step's interpolation:
//
//   interface blocks: face | vertex | source | gather | (lattice) || tiles || shell | interp | face ...
//   lattice blocks:   lattice pass .............................. || tiles || next lattice pass ....
//                     (| barrier of the interface blocks, || barrier of all blocks)
//
// The grid is launched cooperatively (all blocks resident). Every wait is bounded: a barrier that
// does not complete within the context's limit (iblb_set_barrier_wait_limit) sets H_TIMEOUT and an
// abort flag that ends every block. A launch that finds H_TIMEOUT set, by one queued before it, does
// nothing; the host empties the tile maps, which an abort leaves half marked, when it reads the word.
#define IBLB_RO               // phases read what earlier phases of the same kernel wrote
#define IBLB_SCATTER_ASM asm volatile
#include "ib_device.cuh"
#include "lattice_device.cuh"

namespace iblb {
namespace {

// Control words of a launch, zero between launches (the last block to leave clears them).
struct FusedControl {
  unsigned chain;     // arrivals at the interface blocks' barriers
  unsigned all;       // arrivals at the barriers of all blocks
  unsigned left;      // blocks that have left
  int abort;          // a wait gave up: every block returns
  int next[2];        // next chunk of the lattice pass, per parity of the step
};
static_assert(sizeof(FusedControl) <= kFusedControlBytes, "control words");

// Arguments of a step's phases, for each parity of the steps (cur and map alternate).
template <typename real, typename S>
struct FusedStep {
  FaceArgs<real> face;
  VertexArgs<real> vertex;
  SourceArgs<real> source;
  GatherArgs<real> gather;
  StreamArgs<real, S> stream;
  TilesArgs<real, S> tiles;
  ShellArgs<real, S> shell;
  InterpArgs<real> interp;
};
template <typename real, typename S>
struct FusedArgs {
  FusedStep<real, S> step[2];
  FusedControl *ctl;
  int *health;
  unsigned long long wait_ns;
  int nsteps, nchain;
};

// Threads per block and resident blocks per SM: float, 256 threads at 128 registers; double, 128
// threads with the registers that its longest phase (the correction of a node pair) wants.
template <typename real>
struct FusedShape {
  static constexpr int threads = sizeof(real) == 4 ? 256 : 128;
  static constexpr int per_sm = 2;
};

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Whether an earlier launch gave up (called by every thread of the block; one answer for all).
__device__ __forceinline__ bool gave_up(const int *health) {
  __shared__ int s_word;
  if (threadIdx.x == 0) s_word = *(const volatile int *)health;
  __syncthreads();
  return s_word & H_TIMEOUT;
}

// Wait until `target` blocks have arrived on *ctr, this one included (called by every thread of the
// block). False if the wait gave up (after wait_ns; 0: after one test) or another block's did.
__device__ __forceinline__ bool grid_barrier(unsigned *ctr, unsigned target, FusedControl *ctl,
                                             int *health, unsigned long long wait_ns) {
  __shared__ int s_go;
  __syncthreads();
  if (threadIdx.x == 0) {
    // (release and acquire at the GPU's scope, cumulative over the block by its barriers: no full
    // fences, each a microsecond's part of a barrier that a step passes seven times)
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(ctr) : "memory");
    int go = 1;
    if ((int)(ld_acquire(ctr) - target) < 0) {
      const unsigned long long t0 = now_ns();
      for (int k = 0;; k++) {
        if ((int)(ld_acquire(ctr) - target) >= 0) break;
        if ((k & 63) == 63 || wait_ns == 0) {
          if (*(volatile int *)&ctl->abort) go = 0;
          if (go && now_ns() - t0 >= wait_ns) {
            atomicOr(health, H_TIMEOUT);
            atomicExch(&ctl->abort, 1);
            go = 0;
          }
          if (!go) break;
        }
      }
    }
    s_go = go;
  }
  __syncthreads();
  return s_go != 0;
}

// The last block to leave clears the control words for the next launch.
__device__ __forceinline__ void leave_grid(FusedControl *ctl) {
  __syncthreads();
  if (threadIdx.x != 0) return;
  __threadfence();
  if (atomicAdd(&ctl->left, 1u) == gridDim.x - 1) {
    ctl->chain = 0;
    ctl->all = 0;
    ctl->abort = 0;
    ctl->next[0] = ctl->next[1] = 0;
    __threadfence();
    ctl->left = 0;
  }
}

// Node group g of the lattice pass (K1, body force only).
template <typename real, typename S>
__device__ __forceinline__ void lattice_group(const StreamArgs<real, S> &A, int g) {
  int gx, y, z;
  A.G.at(g, gx, y, z);
  z += A.z0;
  if constexpr (sizeof(S) == 2) {
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

// The lattice pass of a step (K1, body force only): blocks take chunks of one node group per
// thread until none is left. The next chunk's number is fetched while the current one is worked on.
template <typename real, typename S>
__device__ __forceinline__ void lattice_chunks(const StreamArgs<real, S> &A, int *next) {
  __shared__ int s_chunk[2];
  const int nt = blockDim.x;
  const int chunks = (A.G.n + nt - 1) / nt;
  __syncthreads();
  if (threadIdx.x == 0) s_chunk[0] = atomicAdd(next, 1);
  __syncthreads();
  for (int k = 0;; k++) {
    const int c = s_chunk[k & 1];
    if (c >= chunks) break;
    if (threadIdx.x == 0) s_chunk[(k & 1) ^ 1] = atomicAdd(next, 1);
    const int g = c * nt + threadIdx.x;
    if (g < A.G.n) lattice_group(A, g);
    __syncthreads();
  }
}

template <typename real, typename S>
__device__ __forceinline__ void fused_steps(const FusedArgs<real, S> &P, SourceShared<real> *sh) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  const int nchain = P.nchain;
  const bool chain = (int)blockIdx.x < nchain;
  FusedControl *ctl = P.ctl;
  // items go to the threads warp by warp, the warps dealt to the blocks in turn, so that a short
  // list spreads over all of them
  const int chain_first = ((tid >> 5) * nchain + blockIdx.x) * 32 + lane, chain_stride = nchain * nt;
  const int all_first = ((tid >> 5) * gridDim.x + blockIdx.x) * 32 + lane,
            all_stride = gridDim.x * nt;
  unsigned n_chain = 0, n_all = 0;  // arrivals expected at the next barrier
#define CHAIN_BARRIER() \
  if (!grid_barrier(&ctl->chain, n_chain += nchain, ctl, P.health, P.wait_ns)) return
#define ALL_BARRIER() \
  if (!grid_barrier(&ctl->all, n_all += gridDim.x, ctl, P.health, P.wait_ns)) return
  for (int s = 0; s < P.nsteps; s++) {
    const FusedStep<real, S> &A = P.step[s & 1];
    if (chain) {
      face_body(A.face, chain_first, chain_stride);
      CHAIN_BARRIER();
      if ((int)blockIdx.x == nchain - 1 && tid >= nt - 32) volume_task(A.vertex);
      for (int g = chain_first; g - lane < 4 * A.vertex.nv; g += chain_stride) vertex_body(A.vertex, g);
      CHAIN_BARRIER();
      const int g = tid / kSourceThreads, ng = nt / kSourceThreads;
      spread_source_body<sizeof(S) != 2>(A.source, sh[g], blockIdx.x + g * nchain, ng * nchain, g,
                                         tid % kSourceThreads);
      CHAIN_BARRIER();
      const int h = tid / TILE_CELLS, nh = nt / TILE_CELLS;
      spread_gather_body(A.gather, blockIdx.x + h * nchain, nh * nchain, tid % TILE_CELLS);
    }
    lattice_chunks(A.stream, &ctl->next[s & 1]);
    ALL_BARRIER();
    if (blockIdx.x == 0 && tid == 0) ctl->next[s & 1] = 0;  // used again two steps on
    tiles_body<false>(A.tiles, all_first, all_stride);
    ALL_BARRIER();
    if (chain) {
      shell_body<real, S>(A.shell, chain_first, chain_stride);
      CHAIN_BARRIER();
      if (4 * A.interp.nv <= chain_stride) {
        interp_body<1>(A.interp, chain_first, 0);
      } else {  // two vertices at a time per lane
        for (int g0 = chain_first; g0 - lane < 4 * A.interp.nv; g0 += 2 * chain_stride)
          interp_body<2>(A.interp, g0, chain_stride >> 2);
      }
      if (s + 1 < P.nsteps) CHAIN_BARRIER();
    }
  }
#undef CHAIN_BARRIER
#undef ALL_BARRIER
}

template <typename real, typename S>
__global__ void __launch_bounds__(FusedShape<real>::threads, FusedShape<real>::per_sm)
    fused_step_kernel(const __grid_constant__ FusedArgs<real, S> P) {
  __shared__ SourceShared<real> sh[FusedShape<real>::threads / kSourceThreads];
  if (!gave_up(P.health)) fused_steps(P, sh);
  leave_grid(P.ctl);
}

// Steps of a lattice without a mesh: the lattice pass alone, a barrier between two steps. Groups
// go to the threads of the grid in memory order, round after round.
template <typename real, typename S>
struct LatticeSteps {
  StreamArgs<real, S> step[2];
  FusedControl *ctl;
  int *health;
  unsigned long long wait_ns;
  int nsteps;
};
// (FP32 and 16-bit storage: FP64 is faster by the separate passes.) Blocks of 128 threads per SM: what
// the pass's registers allow.
template <typename S>
struct LatticeShape {
  static constexpr int per_sm = sizeof(S) == 2 ? 4 : 7;
};

template <typename real, typename S>
__global__ void __launch_bounds__(128, LatticeShape<S>::per_sm)
    lattice_steps_kernel(const __grid_constant__ LatticeSteps<real, S> P) {
  unsigned n_all = 0;
  const int nsteps = gave_up(P.health) ? 0 : P.nsteps;
  for (int s = 0; s < nsteps; s++) {
    const StreamArgs<real, S> &A = P.step[s & 1];
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < A.G.n; g += gridDim.x * blockDim.x)
      lattice_group(A, g);
    if (s + 1 < nsteps &&
        !grid_barrier(&P.ctl->all, n_all += gridDim.x, P.ctl, P.health, P.wait_ns))
      break;
  }
  leave_grid(P.ctl);
}

template <typename real, typename S>
cudaError_t launch_lattice_steps_t(Ctx &c, int nsteps, cudaStream_t st) {
  LatticeSteps<real, S> a;
  for (int p = 0; p < 2; p++) {
    c.cur ^= p;
    a.step[p] = stream_args<real, S>(c);
    c.cur ^= p;
  }
  a.ctl = (FusedControl *)c.fused_ctl;
  a.health = c.counters + 3;
  a.wait_ns = c.barrier_wait_ns;
  a.nsteps = nsteps;
  const int need = (a.step[0].G.n + 127) / 128, room = LatticeShape<S>::per_sm * c.sm_count;
  void *params[] = {&a};
  return cudaLaunchCooperativeKernel((const void *)lattice_steps_kernel<real, S>,
                                     dim3(need < room ? need : room), dim3(128), params, 0, st);
}

// SMs that a step's grid is sized for. A small lattice has too little work for all of them, and its
// barriers are the cheaper the fewer blocks meet there: half of the SMs, from 40^3 (FP64) and 64^3 nodes
// down, with up to 4096 vertices. What that leaves free serves other contexts: us per step and context
// on half / on all SMs, one context alone and two at once, 24^3 FP32 24.4 / 24.5 and 12.5 / 24.2, 48^3
// 26.6 / 27.5 and 13.7 / 27.2, 64^3 26.7 / 28.7 and 15.2 / 29.0, 32^3 FP64 38.2 / 42.7 and 20.6 / 42.6;
// above the line 96^3 FP32 49.9 / 41.8, 48^3 FP64 61.4 / 52.1, 64^3 FP32 with 10242 vertices 53.5 / 46.5.
int fused_sms(const Ctx &c) {
  const size_t nodes = (size_t)1 << (c.pop_size == 8 ? 16 : 18);
  return c.ncell <= nodes && c.nv <= 4096 ? (c.sm_count + 1) / 2 : c.sm_count;
}

template <typename real, typename S>
cudaError_t launch_fused_t(Ctx &c, int nsteps, cudaStream_t st) {
  if (c.nv == 0) {
    if constexpr (sizeof(real) == 4) return launch_lattice_steps_t<real, S>(c, nsteps, st);
    return cudaErrorInvalidValue;  // (no FP64 lattice without a mesh comes here)
  }
  FusedArgs<real, S> a;
  const int cur = c.cur, map = c.map;
  for (int p = 0; p < 2; p++) {
    c.cur = cur ^ p;
    c.map = map ^ p;
    FusedStep<real, S> &s = a.step[p];
    s.face = face_args<real>(c, 1);
    s.vertex = vertex_args<real>(c, 2);
    s.source = source_args<real>(c);
    s.gather = gather_args<real>(c);
    s.stream = stream_args<real, S>(c);
    s.tiles = tiles_args<real, S>(c);
    s.shell = shell_args<real, S>(c, c.f[c.cur ^ 1]);
    s.interp = interp_args<real>(c);
  }
  c.cur = cur;
  c.map = map;
  a.ctl = (FusedControl *)c.fused_ctl;
  a.health = c.counters + 3;
  a.wait_ns = c.barrier_wait_ns;
  a.nsteps = nsteps;
  a.nchain = fused_sms(c);
  void *params[] = {&a};
  // (two blocks per SM always fit: the launch bound limits their registers, and each has 42 KB of
  // shared memory; a caller's context with fewer SMs than the device refuses the launch)
  return cudaLaunchCooperativeKernel((const void *)fused_step_kernel<real, S>,
                                     dim3(FusedShape<real>::per_sm * a.nchain),
                                     dim3(FusedShape<real>::threads), params, 0, st);
}

}  // namespace

cudaError_t launch_fused_steps(Ctx &c, int nsteps, cudaStream_t s) {
  switch (c.precision) {
    case IBLB_FP64: return launch_fused_t<double, double>(c, nsteps, s);
    case IBLB_FP16: return launch_fused_t<float, __half>(c, nsteps, s);
    case IBLB_BF16: return launch_fused_t<float, __nv_bfloat16>(c, nsteps, s);
    default: return launch_fused_t<float, float>(c, nsteps, s);
  }
}

}  // namespace iblb
