// Interface kernels of the step: launches of the passes in ib_device.cuh, one context or many per
// launch, and the small kernels of the read-back calls.
#include "ib_device.cuh"

namespace iblb {
namespace {

// Standalone marking of the current positions (a read of the spread field between steps).
__global__ void mark_kernel(int nv, const double *IBLB_RO q, Dims D, TileMap M) {
  mark_vertices(q, nv, kMarkVertices * ((blockIdx.x * blockDim.x + threadIdx.x) >> 5), D, M);
}

__global__ void volume_sum_kernel(const double *__restrict__ part, int n, double V0,
                                  double *__restrict__ out) {
  double V;
  volume_coef(part, n, V0, 0.0, 0, &V);
  if (threadIdx.x == 0) *out = V;
}

template <typename real>
cudaError_t face_forces_t(Ctx &c, int reset, cudaStream_t st) {
  face_kernel<real><<<face_blocks<real>(c, reset), FaceThreads<real>::value, 0, st>>>(face_args<real>(c, reset));
  return cudaGetLastError();
}

template <typename real>
cudaError_t vertex_forces_t(Ctx &c, int bin, cudaStream_t st) {
  vertex_kernel<real><<<vertex_blocks(c), kVertexThreads, 0, st>>>(vertex_args<real>(c, bin));
  return cudaGetLastError();
}

template <typename real>
cudaError_t spread_t(Ctx &c, cudaStream_t st) {
  spread_source_kernel<real><<<source_blocks<real>(c, false), kSourceThreads, 0, st>>>(
      source_args<real>(c));
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  spread_gather_kernel<real><<<gather_blocks(c, false), TILE_CELLS, 0, st>>>(gather_args<real>(c));
  return cudaGetLastError();
}

template <typename real>
cudaError_t interp_t(Ctx &c, cudaStream_t st) {
  interp_kernel<real><<<interp_blocks(c), kInterpThreads, 0, st>>>(interp_args<real>(c));
  return cudaGetLastError();
}

template <typename T>
void append_record(std::vector<unsigned char> &bytes, const T &rec) {
  const size_t off = bytes.size();
  bytes.resize(off + sizeof(T));
  memcpy(bytes.data() + off, &rec, sizeof(T));
}

template <typename real>
int ib_multi_record_t(const Ctx &c, MultiKernel k, std::vector<unsigned char> &bytes) {
  switch (k) {
    case MK_FACE: append_record(bytes, face_args<real>(c, 1)); return face_blocks<real>(c, 1);
    case MK_VERTEX: append_record(bytes, vertex_args<real>(c, 2)); return vertex_blocks(c);
    case MK_SOURCE: append_record(bytes, source_args<real>(c)); return source_blocks<real>(c, true);
    case MK_GATHER: append_record(bytes, gather_args<real>(c)); return gather_blocks(c, true);
    case MK_INTERP: append_record(bytes, interp_args<real>(c)); return interp_blocks(c);
    default: return -1;
  }
}

template <typename real>
cudaError_t ib_launch_multi_t(MultiKernel k, const MultiLaunch &m, cudaStream_t s) {
  switch (k) {
    case MK_FACE:
      return launch_after(m.early, face_kernel_multi<real>, m.blocks, FaceThreads<real>::value, s,
                          (const FaceArgs<real> *)m.args, m.start, m.n);
    case MK_VERTEX:
      return launch_after(m.early, vertex_kernel_multi<real>, m.blocks, kVertexThreads, s,
                          (const VertexArgs<real> *)m.args, m.start, m.n);
    case MK_SOURCE:
      return launch_after(m.early, spread_source_kernel_multi<real>, m.blocks, kSourceThreads, s,
                          (const SourceArgs<real> *)m.args, m.start, m.n);
    case MK_GATHER:
      return launch_after(m.early, spread_gather_kernel_multi<real>, m.blocks, TILE_CELLS, s,
                          (const GatherArgs<real> *)m.args, m.start, m.n);
    case MK_INTERP:
      return launch_after(m.early, interp_kernel_multi<real>, m.blocks, kInterpThreads, s,
                          (const InterpArgs<real> *)m.args, m.start, m.n);
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace

int ib_multi_record(const Ctx &c, MultiKernel k, std::vector<unsigned char> &bytes) {
  return c.precision == IBLB_FP64 ? ib_multi_record_t<double>(c, k, bytes)
                                  : ib_multi_record_t<float>(c, k, bytes);
}

cudaError_t ib_launch_multi(int precision, MultiKernel k, const MultiLaunch &m, cudaStream_t s) {
  return precision == IBLB_FP64 ? ib_launch_multi_t<double>(k, m, s)
                                : ib_launch_multi_t<float>(k, m, s);
}

size_t stencil_record_bytes(const Ctx &c) {
  return c.precision == IBLB_FP64 ? sizeof(StencilRec<double>) : sizeof(StencilRec<float>);
}

cudaError_t launch_face_forces(Ctx &c, int reset_other_map, cudaStream_t s) {
  return c.precision == IBLB_FP64 ? face_forces_t<double>(c, reset_other_map, s)
                                  : face_forces_t<float>(c, reset_other_map, s);
}

// bin: 0 forces only; 1 forces + stencil + binning; 2 as 1 and also zero the other map's
// tile counter (inside a step, after that map was cleared by the face kernel).
cudaError_t launch_vertex_forces(Ctx &c, int bin, cudaStream_t s) {
  c.health_clear = 0;  // (the volume check)
  return c.precision == IBLB_FP64 ? vertex_forces_t<double>(c, bin, s)
                                  : vertex_forces_t<float>(c, bin, s);
}

cudaError_t launch_spread(Ctx &c, cudaStream_t s) {
  return c.precision == IBLB_FP64 ? spread_t<double>(c, s) : spread_t<float>(c, s);
}

cudaError_t launch_interpolate_advect(Ctx &c, cudaStream_t s) {
  return c.precision == IBLB_FP64 ? interp_t<double>(c, s) : interp_t<float>(c, s);
}

cudaError_t launch_mark(Ctx &c) {
  c.health_clear = 0;
  const int warps = (c.nv + kMarkVertices - 1) / kMarkVertices;
  mark_kernel<<<(32 * warps + 127) / 128, 128, 0, c.stream>>>(c.nv, c.q, dims_of(c), tile_map(c));
  return cudaGetLastError();
}

cudaError_t launch_displacement(Ctx &c) {
  const int blocks = (3 * c.nv + 127) / 128;
  if (c.precision == IBLB_FP64)
    displacement_kernel<double><<<blocks, 128, 0, c.stream>>>(c.nv, c.q, c.xref, (Vec4<double> *)c.disp);
  else
    displacement_kernel<float><<<blocks, 128, 0, c.stream>>>(c.nv, c.q, c.xref, (Vec4<float> *)c.disp);
  return cudaGetLastError();
}

cudaError_t launch_expand_force(Ctx &c, double *F_dev) {
  int grid = c.sm_count * 8;
  if (grid > c.max_slots) grid = c.max_slots;
  if (grid < 1) grid = 1;
  if (c.precision == IBLB_FP64)
    expand_force_kernel<double><<<grid, TILE_CELLS, 0, c.stream>>>(
        c.slot_tile[c.map], c.counters + c.map, (const Vec4<double> *)c.Fslot[c.map], dims_of(c), F_dev);
  else
    expand_force_kernel<float><<<grid, TILE_CELLS, 0, c.stream>>>(
        c.slot_tile[c.map], c.counters + c.map, (const Vec4<float> *)c.Fslot[c.map], dims_of(c), F_dev);
  return cudaGetLastError();
}

cudaError_t launch_phi_to_double(Ctx &c, double *phi_dev) {
  const int blocks = (c.nv + 255) / 256;
  if (c.precision == IBLB_FP64)
    combine_forces_kernel<double><<<blocks, 256, 0, c.stream>>>(
        c.nv, (const Vec4<double> *)c.phi, (const Vec4<double> *)c.gvol, c.vol_partial,
        volume_params(c), phi_dev);
  else
    combine_forces_kernel<float><<<blocks, 256, 0, c.stream>>>(
        c.nv, (const Vec4<float> *)c.phi, (const Vec4<float> *)c.gvol, c.vol_partial,
        volume_params(c), phi_dev);
  return cudaGetLastError();
}

cudaError_t launch_volume(Ctx &c, double *V_dev) {
  volume_sum_kernel<<<1, 32, 0, c.stream>>>(c.vol_partial, c.vol_blocks, c.V0, V_dev);
  return cudaGetLastError();
}

}  // namespace iblb
