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

// Axes of 128 and 256 points go to the tensor cores above 2048 lines (64
// tiles of 32; apply_digits.cu).  Measured per product, before -> digits:
// 256^2 x 32 UV 3097 -> 1052 us, x 48 FG 4414 -> 1319, x 4 FG 435 -> 168 (full
// FFTs); x 2 FG (3072 lines) 226 -> 95, 128^2 x 4 FG 114 -> 58 (spread FFTs);
// 256^2 x 1 (1536 lines) 119, with digits 145: a tile takes 30 (N = 128) or 60
// us whether or not every SM has one.
constexpr long long DIGIT_LINES = 2048;
static bool digits(const ApplyArgs<R>& g, int ax) {
  return g.kdig[ax] && g.grid->npts / g.grid->n[ax] * 6 * g.nvec > DIGIT_LINES;
}

template <>
cudaError_t apply_launch<double>(const ApplyArgs<double>& g, cudaStream_t s) {
  if (g.nvec <= 0) return cudaSuccess;
  const int last = g.grid->dim - 1;
  cudaError_t e;
  if (digits(g, last)) {
    e = couple_launch(g, s);
    if (e == cudaSuccess) e = axis_digits_launch(g, last, s);
  } else {
    e = few_lines(g, g.grid->n[last]) ? row_spread(g, s) : row_full(g, s);
  }
  for (int ax = last - 1; e == cudaSuccess && ax >= 0; --ax) {
    if (digits(g, ax)) e = axis_digits_launch(g, ax, s);
    else e = few_lines(g, g.grid->n[ax]) ? axis_spread(g, ax, s) : axis_full(g, ax, s);
  }
  return e;
}

}  // namespace bdg
