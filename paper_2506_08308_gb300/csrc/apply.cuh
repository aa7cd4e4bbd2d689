// Launch interface of the BdG product kernels.
#pragma once

#include "common.cuh"

namespace bdg {

template <typename R>
struct ApplyArgs {
  const Grid* grid;
  const typename CT<R>::T* x;
  typename CT<R>::T* y;
  int nvec;
  int mode;                         // BDG_UV or BDG_FG
  const typename CT<R>::Q* phiv;    // (phi_1, phi_0, phi_-1, V) per node
  const typename CT<R>::T* tw[3];   // per-axis twiddles W_N^r
  R kscale[3];                      // 1/2 (2 pi / len_a)^2 / n_a per axis
  Coupling<R> cp;
  // FP64 axes of 128 and 256 points (apply_digits.cu): digit tables, their
  // exponents, and 1/2 (2 pi / len_a)^2; no table: NULL
  const uint8_t* kdig[3];
  int kexp[3];
  double kfac[3];
};

template <typename R>
cudaError_t apply_launch(const ApplyArgs<R>& g, cudaStream_t s);

// The FP64 product's passes in integer digits on the tensor cores.
bool axis_digits_supported(int n);
cudaError_t axis_digits_table(int n, uint8_t** out, int* kexp, cudaStream_t s);  // *out: cudaMalloc
cudaError_t couple_launch(const ApplyArgs<double>& g, cudaStream_t s);           // y = C x
cudaError_t axis_digits_launch(const ApplyArgs<double>& g, int ax, cudaStream_t s);

}  // namespace bdg
