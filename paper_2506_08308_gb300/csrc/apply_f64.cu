// FP64 instantiation of the BdG product kernels.
#include "apply_spread.cuh"

namespace bdg {

typedef double R;

// Lines of all components and vectors up to which four points per thread are
// faster (FEW_LINES, fft_spread.cuh), one pass at a time.
static bool few_lines(const ApplyArgs<R>& g, int n) {
  return g.grid->npts / n * 6 * g.nvec <= FEW_LINES;
}

static cudaError_t row_full(const ApplyArgs<R>& g, cudaStream_t s) {
  BDG_DISPATCH_N(g.grid->n[g.grid->dim - 1], launch_row, g, s)
}
static cudaError_t row_spread(const ApplyArgs<R>& g, cudaStream_t s) {
  BDG_DISPATCH_N(g.grid->n[g.grid->dim - 1], launch_row_spread, g, s)
}
static cudaError_t axis_full(const ApplyArgs<R>& g, int ax, cudaStream_t s) {
  BDG_DISPATCH_N(g.grid->n[ax], launch_axis, g, ax, s)
}
static cudaError_t axis_spread(const ApplyArgs<R>& g, int ax, cudaStream_t s) {
  BDG_DISPATCH_N(g.grid->n[ax], launch_axis_spread, g, ax, s)
}

template <>
cudaError_t apply_launch<double>(const ApplyArgs<double>& g, cudaStream_t s) {
  if (g.nvec <= 0) return cudaSuccess;
  const int last = g.grid->dim - 1;
  cudaError_t e = few_lines(g, g.grid->n[last]) ? row_spread(g, s) : row_full(g, s);
  for (int ax = last - 1; e == cudaSuccess && ax >= 0; --ax)
    e = few_lines(g, g.grid->n[ax]) ? axis_spread(g, ax, s) : axis_full(g, ax, s);
  return e;
}

}  // namespace bdg
