// FP32 instantiation of the BdG product kernels.
#include "apply2_f32.cuh"

namespace bdg {

static cudaError_t row_f32(const ApplyArgs<float>& g, cudaStream_t s) {
  switch (g.grid->n[g.grid->dim - 1]) {
    case 8: return launch_row<8, float>(g, s);
    case 16: return launch_row<16, float>(g, s);
    case 32: return launch_row2<32>(g, s);
    case 64: return launch_row2<64>(g, s);
    case 128: return launch_row2<128>(g, s);
    case 256: return launch_row2<256>(g, s);
    case 512: return launch_row2<512>(g, s);
    case 1024: return launch_row2<1024>(g, s);
    default: return cudaErrorInvalidValue;
  }
}

static cudaError_t axis_f32(const ApplyArgs<float>& g, int ax, cudaStream_t s) {
  switch (g.grid->n[ax]) {
    case 8: return launch_axis<8, float>(g, ax, s);
    case 16: return launch_axis<16, float>(g, ax, s);
    case 32: return launch_axis2<32>(g, ax, s);
    case 64: return launch_axis2<64>(g, ax, s);
    case 128: return launch_axis2<128>(g, ax, s);
    case 256: return launch_axis2<256>(g, ax, s);
    case 512: return launch_axis2<512>(g, ax, s);
    case 1024: return launch_axis2<1024>(g, ax, s);
    default: return cudaErrorInvalidValue;
  }
}

template <>
cudaError_t apply_launch<float>(const ApplyArgs<float>& g, cudaStream_t s) {
  if (g.nvec <= 0) return cudaSuccess;
  cudaError_t e = row_f32(g, s);
  for (int ax = g.grid->dim - 2; e == cudaSuccess && ax >= 0; --ax) e = axis_f32(g, ax, s);
  return e;
}

}  // namespace bdg
