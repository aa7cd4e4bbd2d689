// FP32 BdG product with two lines per thread (fft2.cuh): the same two kinds
// of passes as in apply_impl.cuh, for lines of 32 points and more.
//
// What bounds them: at one line per thread the row pass was bound by issue
// slots and the strided pass waited on shared memory and scalar arithmetic
// (256^2, 48 vectors: 118 + 89 us).  With pairs the same transforms take
// about half the arithmetic instructions; the row pass now runs its FMA pipe
// at 54 % and reads x a second time from L2 instead of keeping it in shared
// memory (54 KB per CTA, three CTAs per SM), the strided pass runs at 74 % of
// the DRAM peak.  Measured per call, before -> after: 256^2 x 48 FG 206 ->
// 134 us, 512^2 x 12 345 -> 194 us, 1024^2 x 3 381 -> 237 us, 128^3 x 16
// 2810 -> 2054 us, 64 x 128 x 5 11.3 -> 9.7 us, 1-D 256 x 24 7.7 -> 6.7 us:
// faster at every size it covers, so that the one-line kernels serve FP32
// only for N = 8 and 16, whose lines would leave a pair kernel's warps idle.
#pragma once

#include "apply_impl.cuh"
#include "fft2.cuh"

namespace bdg {

struct Sym3x2 {  // a symmetric 3 x 3 matrix at two nodes
  V2 d0, d1, d2, o01, o12, o02;
};
// rows of the matrices of the first (second) node times x
template <bool SECOND>
__device__ __forceinline__ void mul3(const Sym3x2& m, const float2* x, float2* y) {
  Sym3<float> s;
  s.d0 = SECOND ? hi(m.d0) : lo(m.d0); s.d1 = SECOND ? hi(m.d1) : lo(m.d1); s.d2 = SECOND ? hi(m.d2) : lo(m.d2);
  s.o01 = SECOND ? hi(m.o01) : lo(m.o01); s.o12 = SECOND ? hi(m.o12) : lo(m.o12); s.o02 = SECOND ? hi(m.o02) : lo(m.o02);
  y[0] = sym3_row0(s, x[0], x[1], x[2]);
  y[1] = sym3_row1(s, x[0], x[1], x[2]);
  y[2] = sym3_row2(s, x[0], x[1], x[2]);
}
// all six components of the coupling at the first (second) node; A, B are the
// blocks in the UV form, A + B and A - B in the FG form.  For the last three
// components of the UV form the negative of the coupling.
template <bool SECOND>
__device__ __forceinline__ void couple(const Sym3x2& A, const Sym3x2& B, int mode, const float2* v, float2* w) {
  if (mode == BDG_UV) {
    float2 t[3];
    mul3<SECOND>(A, v, w);
    mul3<SECOND>(B, v + 3, t);
#pragma unroll
    for (int c = 0; c < 3; ++c) w[c] = w[c] + t[c];
    mul3<SECOND>(B, v, w + 3);
    mul3<SECOND>(A, v + 3, t);
#pragma unroll
    for (int c = 0; c < 3; ++c) w[3 + c] = w[3 + c] + t[c];
  } else {
    mul3<SECOND>(A, v, w);
    mul3<SECOND>(B, v + 3, w + 3);
  }
}

// coupling_blocks at two nodes
__device__ __forceinline__ void coupling_blocks2(float4 p, float4 q, const Coupling<float>& cp, Sym3x2& A, Sym3x2& B) {
  const V2 a = pk(p.x, q.x), b = pk(p.y, q.y), c = pk(p.z, q.z), V = pk(p.w, q.w);
  const V2 bn = dup(cp.beta_n), bs = dup(cp.beta_s), bnbs = dup(cp.beta_n + cp.beta_s);
  const V2 a2 = a * a, b2 = b * b, c2 = c * c, ac = a * c, ab = a * b, bc = b * c;
  const V2 rho = a2 + b2 + c2, sum = a + c;
  A.d0 = fma2(bn, rho + a2, fma2(bs, a2 + a2 + b2 - c2, V + dup(cp.d1)));
  A.d1 = fma2(bn, rho + b2, fma2(bs, a2 + c2, V + dup(cp.d0)));
  A.d2 = fma2(bn, rho + c2, fma2(bs, c2 + c2 + b2 - a2, V + dup(cp.dm)));
  A.o01 = fma2(bn, ab, bs * (b * (sum + c)));
  A.o12 = fma2(bn, bc, bs * (b * (sum + a)));
  A.o02 = dup(cp.beta_n - cp.beta_s) * ac;
  B.d0 = bnbs * a2;
  B.d1 = fma2(bn, b2, bs * (ac + ac));
  B.d2 = bnbs * c2;
  B.o01 = bnbs * ab;
  B.o12 = bnbs * bc;
  B.o02 = fma2(bn, ac, bs * (b2 - ac));
}
__device__ __forceinline__ Sym3x2 operator+(const Sym3x2& A, const Sym3x2& B) {
  return Sym3x2{A.d0 + B.d0, A.d1 + B.d1, A.d2 + B.d2, A.o01 + B.o01, A.o12 + B.o12, A.o02 + B.o02};
}
__device__ __forceinline__ Sym3x2 operator-(const Sym3x2& A, const Sym3x2& B) {
  return Sym3x2{A.d0 - B.d0, A.d1 - B.d1, A.d2 - B.d2, A.o01 - B.o01, A.o12 - B.o12, A.o02 - B.o02};
}

// Row pass: last axis + coupling.  Warp c of the six transforms component c
// of 2 RP grid rows, rows r and r + RP in one thread (RP = 32 / N1); the
// transforms land in shared memory in place of their exchange area, and a
// pointwise phase over (row pair, point) reads x again (it comes from L1/L2)
// for the coupling and writes all six components of y.
// exchange area of a line pair in 16-byte elements; with N1 = 4 a quarter
// warp holds two line pairs, kept half a bank cycle apart
template <int N>
constexpr int row2_area() {
  typedef Line2<N, WarpSync> L;
  return L::N1 == 4 ? (L::AREA + 7) / 8 * 8 + 4 : L::AREA;
}
template <int N>
__global__ void __launch_bounds__(192, N <= 256 ? 3 : 2)
    k_row2(const float2* __restrict__ x, float2* __restrict__ y, int nunits, int row_bits, long long npts,
           const float4* __restrict__ phiv, const float2* __restrict__ twg, Coupling<float> cp, float kscale, int mode) {
  typedef Line2<N, WarpSync> L;
  constexpr int N1 = L::N1, N2 = L::N2, RP = 32 / N1, NT = 192;
  constexpr int LS = row2_area<N>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2* buf = reinterpret_cast<C2*>(smem_raw);                 // [6][RP][LS]
  float2* tw = reinterpret_cast<float2*>(buf + 6 * RP * LS);  // [N]
  const int tid = threadIdx.x;
  const int u0 = (int)blockIdx.x * (2 * RP), row_mask = (1 << row_bits) - 1;
  {
    const int lane = tid & 31, c = tid >> 5, r = lane / N1, t = lane - r * N1;
    C2* ex = buf + (c * RP + r) * LS;
    const int ua = u0 + r, ub = ua + RP;
    const float2* xa = x + ((ua >> row_bits) * 6 + c) * npts + (ua & row_mask) * N + t;
    const float2* xb = x + ((ub >> row_bits) * 6 + c) * npts + (ub & row_mask) * N + t;
    const float2 z = make_float2(0.f, 0.f);
    float2 p[N2], q[N2];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) {
      p[n2] = ua < nunits ? xa[N1 * n2] : z;
      q[n2] = ub < nunits ? xb[N1 * n2] : z;
    }
    L::load_twiddles(tw, twg);
    __syncthreads();
    L::fwdA(p, q, t, ex, tw, WarpSync());
    L::mid(t, ex, kscale, WarpSync());
    C2 a[N2];
    L::invA(a, t, ex, tw);
    __syncwarp();   // the line's exchange area has been read by all its threads
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) ex[t + N1 * n2] = a[n2];
  }
  __syncthreads();
  for (int p = tid; p < RP * N; p += NT) {
    const int r = p / N, i = p - r * N;
    const int ua = u0 + r;
    if (ua >= nunits) break;
    const bool two = ua + RP < nunits;
    const int ub = two ? ua + RP : ua;
    const int na = (ua & row_mask) * N + i, nb = (ub & row_mask) * N + i;
    const long long oa = (ua >> row_bits) * 6 * npts + na, ob = (ub >> row_bits) * 6 * npts + nb;
    const float2* xa = x + oa;
    const float2* xb = x + ob;
    float2 va[6], vb[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      va[c] = xa[c * npts];
      vb[c] = xb[c * npts];
    }
    Sym3x2 A, B;
    coupling_blocks2(phiv[na], phiv[nb], cp, A, B);
    if (mode != BDG_UV) {
      const Sym3x2 P = A + B;
      B = A - B;
      A = P;
    }
    float2 wa[6], wb[6];
    couple<false>(A, B, mode, va, wa);
    couple<true>(A, B, mode, vb, wb);
    float2* ya = y + oa;
    float2* yb = y + ob;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const C2 f = buf[(c * RP + r) * LS + i];
      const float g = c >= 3 && mode == BDG_UV ? -1.f : 1.f;   // y = g (T x + w)
      ya[c * npts] = make_float2(g * (lo(f.x) + wa[c].x), g * (lo(f.y) + wa[c].y));
      if (two) yb[c * npts] = make_float2(g * (hi(f.x) + wb[c].x), g * (hi(f.y) + wb[c].y));
    }
  }
}

// Strided-axis pass y += s_c T_a x: W adjacent lines per CTA, lines w and
// w + W/2 in one thread; thread (w, j): w = tid % (W/2), j = tid / (W/2).
// tile_bits: log2 of the tiles per component; inner_bits: of st / W.
template <int N, int W>
constexpr int axis2_area() {  // eight (four) neighbouring w of a quarter warp on different banks
  constexpr int A = Line2<N, BlockSync>::AREA;
  return W >= 16 ? A | 1 : (A + 7) / 8 * 8 + 2;
}
template <int N, int W>
__global__ void __launch_bounds__(W / 2 * Split<N>::N1, N <= 256 ? 512 / (W / 2 * Split<N>::N1) : 1)
    k_axis2(const float2* __restrict__ x, float2* __restrict__ y, long long npts, long long st, int tile_bits,
            int inner_bits, const float2* __restrict__ twg, float kscale, int mode) {
  typedef Line2<N, BlockSync> L;
  constexpr int N1 = L::N1, N2 = L::N2, H = W / 2, LS = axis2_area<N, W>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2* exb = reinterpret_cast<C2*>(smem_raw);               // [H][LS]
  float2* tw = reinterpret_cast<float2*>(exb + H * LS);    // [N]
  const int tid = threadIdx.x;
  // from the last vector to the first: what the pass before wrote last is still in L2
  const unsigned bid = gridDim.x - 1 - blockIdx.x;
  const int vc = bid >> tile_bits;  // vector*6 + component
  const int tile = bid & ((1u << tile_bits) - 1);
  const int outer = tile >> inner_bits, inner0 = (tile & ((1 << inner_bits) - 1)) * W;
  const int w = tid % H, j = tid / H;
  const long long base = vc * npts + outer * (N * st) + inner0 + w + j * st;
  const float2* xl = x + base;
  {
    float2 p[N2], q[N2];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) {
      p[n2] = xl[N1 * n2 * st];
      q[n2] = xl[N1 * n2 * st + H];
    }
    L::load_twiddles(tw, twg);
    __syncthreads();
    L::fwdA(p, q, j, exb + w * LS, tw, BlockSync());
  }
  L::mid(j, exb + w * LS, kscale, BlockSync());
  C2 a[N2];
  L::invA(a, j, exb + w * LS, tw);
  const float sg = (mode == BDG_UV && vc % 6 >= 3) ? -1.f : 1.f;
  float2* yl = y + base;
  // y in batches of YB rows, all loads of a batch before its stores
  constexpr int YB = N2 < 8 ? N2 : 8;
#pragma unroll
  for (int n0 = 0; n0 < N2; n0 += YB) {
    float2 u[YB], v[YB];
#pragma unroll
    for (int k = 0; k < YB; ++k) {
      u[k] = yl[N1 * (n0 + k) * st];
      v[k] = yl[N1 * (n0 + k) * st + H];
    }
#pragma unroll
    for (int k = 0; k < YB; ++k) {
      const C2 r = a[n0 + k];
      yl[N1 * (n0 + k) * st] = make_float2(fmaf(lo(r.x), sg, u[k].x), fmaf(lo(r.y), sg, u[k].y));
      yl[N1 * (n0 + k) * st + H] = make_float2(fmaf(hi(r.x), sg, v[k].x), fmaf(hi(r.y), sg, v[k].y));
    }
  }
}

template <int N>
static cudaError_t launch_row2(const ApplyArgs<float>& g, cudaStream_t s) {
  constexpr int RP = 32 / Split<N>::N1;
  const size_t sm = sizeof(C2) * 6 * RP * row2_area<N>() + sizeof(float2) * N;
  cudaError_t e = allow_dynamic_smem((const void*)k_row2<N>, sm);
  if (e != cudaSuccess) return e;
  const int ax = g.grid->dim - 1;
  const long long rows_per_vec = g.grid->npts / N, nunits = rows_per_vec * g.nvec;
  k_row2<N><<<(unsigned)((nunits + 2 * RP - 1) / (2 * RP)), 192, sm, s>>>(
      g.x, g.y, (int)nunits, log2i(rows_per_vec), g.grid->npts, g.phiv, g.tw[ax], g.cp, g.kscale[ax], g.mode);
  return cudaGetLastError();
}

template <int N, int W>
static cudaError_t launch_axis2_w(const ApplyArgs<float>& g, int ax, long long st, cudaStream_t s) {
  const size_t sm = sizeof(C2) * (size_t)(W / 2) * axis2_area<N, W>() + sizeof(float2) * N;
  cudaError_t e = allow_dynamic_smem((const void*)k_axis2<N, W>, sm);
  if (e != cudaSuccess) return e;
  const long long tiles = g.grid->npts / ((long long)N * W);
  k_axis2<N, W><<<(unsigned)(tiles * 6 * g.nvec), W / 2 * Split<N>::N1, sm, s>>>(g.x, g.y, g.grid->npts, st, log2i(tiles),
                                                                              log2i(st / W), g.tw[ax], g.kscale[ax], g.mode);
  return cudaGetLastError();
}

template <int N>
static cudaError_t launch_axis2(const ApplyArgs<float>& g, int ax, cudaStream_t s) {
  long long st = 1;
  for (int a = ax + 1; a < g.grid->dim; ++a) st *= g.grid->n[a];
  if (st >= 16) return launch_axis2_w<N, 16>(g, ax, st, s);
  return launch_axis2_w<N, 8>(g, ax, st, s);
}

}  // namespace bdg
