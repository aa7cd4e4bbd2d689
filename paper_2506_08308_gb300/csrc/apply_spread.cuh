// FP64 BdG product for few lines, four points per thread (fft_spread.cuh):
// the row pass (last axis and coupling) and the strided passes of
// apply_impl.cuh with one group of lines of one component per CTA.
#pragma once

#include "apply_impl.cuh"
#include "fft_spread.cuh"

namespace bdg {

// Coupling of one component at one node: row j of A and B (see the head of
// apply_impl.cuh) times the six components x[0], x[np], ...
template <typename R, typename Q>
__device__ __forceinline__ typename CT<R>::T couple_row(const Q pv, const Coupling<R>& cp, int c, int mode,
                                                        const typename CT<R>::T* __restrict__ x, long long np) {
  typedef typename CT<R>::T T;
  const R a = (R)pv.x, b = (R)pv.y, m = (R)pv.z, V = (R)pv.w;
  const R bn = cp.beta_n, bs = cp.beta_s;
  const int j = c < 3 ? c : c - 3;
  R A[3], B[3];
  if (j == 1) {
    const R b2 = b * b, am = a * m;
    const R rho = a * a + b2 + m * m;
    A[0] = bn * a * b + bs * b * (a + 2 * m);
    A[1] = V + cp.d0 + bn * (rho + b2) + bs * (rho - b2);
    A[2] = bn * b * m + bs * b * (2 * a + m);
    B[0] = (bn + bs) * a * b;
    B[1] = bn * b2 + 2 * bs * am;
    B[2] = (bn + bs) * b * m;
  } else {
    // rows 0 and 2 are each other's mirror image: e is the component's own
    // field, o the opposite one
    const R e = j == 0 ? a : m, o = j == 0 ? m : a;
    const R e2 = e * e, b2 = b * b, o2 = o * o, am = a * m;
    const R off = bn * e * b + bs * b * (e + 2 * o), far = (bn - bs) * am;
    const R boff = (bn + bs) * e * b, bfar = bn * am + bs * (b2 - am);
    const R d = V + (j == 0 ? cp.d1 : cp.dm) + bn * (2 * e2 + b2 + o2) + bs * (2 * e2 + b2 - o2);
    A[0] = j == 0 ? d : far;
    A[1] = off;
    A[2] = j == 0 ? far : d;
    B[0] = j == 0 ? (bn + bs) * e2 : bfar;
    B[1] = boff;
    B[2] = j == 0 ? bfar : (bn + bs) * e2;
  }
  T y = mk((R)0, (R)0);
  if (mode == BDG_UV) {
    const T* own = c < 3 ? x : x + 3 * np;      // A acts on the component's own half, B on the other
    const T* oth = c < 3 ? x + 3 * np : x;
#pragma unroll
    for (int k = 0; k < 3; ++k) y = cfma(own[k * np], A[k], y);
#pragma unroll
    for (int k = 0; k < 3; ++k) y = cfma(oth[k * np], B[k], y);
    return c < 3 ? y : mk(-y.x, -y.y);
  }
  const R sg = c < 3 ? (R)1 : (R)-1;
  const T* own = c < 3 ? x : x + 3 * np;
#pragma unroll
  for (int k = 0; k < 3; ++k) y = cfma(own[k * np], A[k] + sg * B[k], y);
  return y;
}

// The first FT threads transform WARP_LINES rows of component c, the other FT
// form the coupling of the same points meanwhile.
template <int N, typename R>
__global__ void __launch_bounds__(2 * Spread<N, typename CT<R>::T>::FT)
    k_row_spread(const typename CT<R>::T* __restrict__ x, typename CT<R>::T* __restrict__ y, int nunits, int row_bits,
                 long long npts, const typename CT<R>::Q* __restrict__ phiv, const typename CT<R>::T* __restrict__ twg,
                 Coupling<R> cp, R kscale, int mode) {
  typedef typename CT<R>::T T;
  typedef Spread<N, T> L;
  constexpr int TH = L::TH, WL = L::WARP_LINES, FT = L::FT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* ex = reinterpret_cast<T*>(smem_raw);  // [WL][2 N]
  T* cbuf = ex + WL * 2 * N;               // [WL][N]
  const int c = blockIdx.x % 6, tid = threadIdx.x;
  const bool fft = tid < FT;
  const int i = fft ? tid : tid - FT, l = i / TH, t = i - l * TH;
  const int u = (int)(blockIdx.x / 6) * WL + l;
  const bool on = u < nunits;
  const long long node = (long long)((on ? u : 0) & ((1 << row_bits) - 1)) * N + t;
  const long long vec = ((on ? u : 0) >> row_bits) * 6 * npts;
  const T* xl = x + vec + node;
  T a[4];
  if (fft) {
    L f;
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] = xl[c * npts + TH * k];
    f.load_twiddles(t, twg);
    T* e = ex + l * 2 * N;
    auto go = [&](auto sync) {
      f.template run<-1>(a, t, e, sync);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int kk = kidx<N>(t + TH * k);
        a[k] = a[k] * (kscale * (R)(kk * kk));
      }
      f.template run<1>(a, t, e, sync);
    };
    if constexpr (FT == 32) go(SpreadWarp());
    else go(SpreadBar<FT>());
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      cbuf[l * N + t + TH * k] = couple_row<R>(phiv[node + TH * k], cp, c, mode, xl + TH * k, npts);
  }
  __syncthreads();
  if (fft && on) {
    const R sg = (mode == BDG_UV && c >= 3) ? (R)-1 : (R)1;
    T* yl = y + vec + c * npts + node;
#pragma unroll
    for (int k = 0; k < 4; ++k) yl[TH * k] = cfma(a[k], sg, cbuf[l * N + t + TH * k]);
  }
}

// y += s_c T_a x along a strided axis: WARP_LINES adjacent lines per CTA
template <int N, typename R>
__global__ void __launch_bounds__(Spread<N, typename CT<R>::T>::FT)
    k_axis_spread(const typename CT<R>::T* __restrict__ x, typename CT<R>::T* __restrict__ y, long long npts,
                  long long st, int comp_bits, int st_bits, const typename CT<R>::T* __restrict__ twg, R kscale,
                  int mode) {
  typedef typename CT<R>::T T;
  typedef Spread<N, T> L;
  constexpr int TH = L::TH, WL = L::WARP_LINES, FT = L::FT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* ex = reinterpret_cast<T*>(smem_raw);  // [WL][2 N]
  const int l = threadIdx.x % WL, t = threadIdx.x / WL;
  const long long line = (long long)blockIdx.x * WL + l;     // the lines of all components, then vectors
  const int vc = (int)(line >> comp_bits);
  const long long in = line & ((1LL << comp_bits) - 1);      // line within the component
  const long long base = vc * npts + (in >> st_bits) * (N * st) + (in & (st - 1)) + t * st;
  T a[4];
  L f;
#pragma unroll
  for (int k = 0; k < 4; ++k) a[k] = x[base + TH * k * st];
  f.load_twiddles(t, twg);
  T* e = ex + l * 2 * N;
  auto go = [&](auto sync) {
    f.template run<-1>(a, t, e, sync);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int kk = kidx<N>(t + TH * k);
      a[k] = a[k] * (kscale * (R)(kk * kk));
    }
    f.template run<1>(a, t, e, sync);
  };
  T yv[4];
  if constexpr (FT == 32) go(SpreadWarp());
  else go(SpreadBar<FT>());
  const R sg = (mode == BDG_UV && vc % 6 >= 3) ? (R)-1 : (R)1;
#pragma unroll
  for (int k = 0; k < 4; ++k) yv[k] = y[base + TH * k * st];
#pragma unroll
  for (int k = 0; k < 4; ++k) y[base + TH * k * st] = cfma(a[k], sg, yv[k]);
}

template <int N, typename R>
static cudaError_t launch_row_spread(const ApplyArgs<R>& g, cudaStream_t s) {
  typedef Spread<N, typename CT<R>::T> L;
  const size_t sm = sizeof(typename CT<R>::T) * (size_t)L::WARP_LINES * 3 * N;
  cudaError_t e = allow_dynamic_smem((const void*)k_row_spread<N, R>, sm);
  if (e != cudaSuccess) return e;
  const int ax = g.grid->dim - 1;
  const long long rows = g.grid->npts / N, nunits = rows * g.nvec;
  const long long groups = (nunits + L::WARP_LINES - 1) / L::WARP_LINES;
  k_row_spread<N, R><<<(unsigned)(groups * 6), 2 * L::FT, sm, s>>>(g.x, g.y, (int)nunits, log2i(rows), g.grid->npts,
                                                                   g.phiv, g.tw[ax], g.cp, g.kscale[ax], g.mode);
  return cudaGetLastError();
}

template <int N, typename R>
static cudaError_t launch_axis_spread(const ApplyArgs<R>& g, int ax, cudaStream_t s) {
  typedef Spread<N, typename CT<R>::T> L;
  long long st = 1;
  for (int a = ax + 1; a < g.grid->dim; ++a) st *= g.grid->n[a];
  const size_t sm = sizeof(typename CT<R>::T) * (size_t)L::WARP_LINES * 2 * N;
  cudaError_t e = allow_dynamic_smem((const void*)k_axis_spread<N, R>, sm);
  if (e != cudaSuccess) return e;
  const long long lines = g.grid->npts / N;   // per component
  k_axis_spread<N, R><<<(unsigned)((lines * 6 * g.nvec + L::WARP_LINES - 1) / L::WARP_LINES), L::FT, sm, s>>>(
      g.x, g.y, g.grid->npts, st, log2i(lines), log2i(st), g.tw[ax], g.kscale[ax], g.mode);
  return cudaGetLastError();
}

}  // namespace bdg
