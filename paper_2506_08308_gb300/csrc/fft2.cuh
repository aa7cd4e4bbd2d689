// Line FFTs of fft.cuh for two lines per thread in packed FP32.
//
// sm_103a issues add/sub/mul/fma on pairs of FP32 values (f32x2) in one slot
// at the same FLOP rate as two scalar instructions, so a transform that is
// bound by issue slots runs with half the arithmetic instructions when every
// operand is a pair.  The pair is (line 0, line 1): a complex value holds
// the two real parts in one 64-bit register pair and the two imaginary parts
// in another, all butterflies, twiddles and k-space factors act on both
// lines alike, and no instruction ever has to swap halves.  Every operation
// and its order are those of the scalar transform.
#pragma once

#include "fft.cuh"

namespace bdg {

struct V2 {  // two FP32 values in one register pair
  unsigned long long v;
};
__device__ __forceinline__ V2 pk(float a, float b) {
  V2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ V2 dup(float a) { return pk(a, a); }
__device__ __forceinline__ float lo(V2 a) { return __uint_as_float((unsigned)a.v); }
__device__ __forceinline__ float hi(V2 a) { return __uint_as_float((unsigned)(a.v >> 32)); }
__device__ __forceinline__ V2 operator+(V2 a, V2 b) {
  V2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ V2 operator-(V2 a, V2 b) {
  V2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ V2 operator*(V2 a, V2 b) {
  V2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ V2 fma2(V2 a, V2 b, V2 c) {
  V2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

struct __align__(16) C2 {  // one complex value of each of the two lines
  V2 x, y;                 // real parts, imaginary parts
};
__device__ __forceinline__ C2 operator+(C2 a, C2 b) { return C2{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ C2 join(float2 a, float2 b) { return C2{pk(a.x, b.x), pk(a.y, b.y)}; }
__device__ __forceinline__ float2 line0(C2 a) { return make_float2(lo(a.x), lo(a.y)); }
__device__ __forceinline__ float2 line1(C2 a) { return make_float2(hi(a.x), hi(a.y)); }

// d exp(i DIR 2 pi q / 32) for 0 < q < 16, q != 8.  Products with constants
// run in scalar instructions: those take the constant as an immediate, where
// a packed one wants it duplicated in a register pair.
template <int DIR>
__device__ __forceinline__ C2 rot_pair(C2 d, int q) {
  const double c = cos32(q), s = DIR * sin32(q);
  const float cf = (float)c, sf = (float)s;
  if ((q & 7) == 4) {  // |c| = |s|
    const V2 p = c * s > 0 ? d.x - d.y : d.x + d.y, m = c * s > 0 ? d.x + d.y : d.y - d.x;
    // (c, s) signs: ++ p = x - y, m = y + x; +- p = x + y, m = y - x; -+ and -- the same negated
    return C2{pk(lo(p) * cf, hi(p) * cf), pk(lo(m) * cf, hi(m) * cf)};
  }
  return C2{pk(fmaf(lo(d.x), cf, -lo(d.y) * sf), fmaf(hi(d.x), cf, -hi(d.y) * sf)),
            pk(fmaf(lo(d.x), sf, lo(d.y) * cf), fmaf(hi(d.x), sf, hi(d.y) * cf))};
}
// (u - v) exp(i DIR 2 pi q / 32), 0 <= q < 16; the quarter turn is folded
// into the order of the subtractions
template <int DIR>
__device__ __forceinline__ C2 rot_diff(C2 u, C2 v, int q) {
  if (q == 8) return DIR > 0 ? C2{v.y - u.y, u.x - v.x} : C2{u.y - v.y, v.x - u.x};
  const C2 d{u.x - v.x, u.y - v.y};
  return q == 0 ? d : rot_pair<DIR>(d, q);
}

template <int NR, int SPAN, int DIR>
struct DifStage<NR, SPAN, DIR, C2> {
  __device__ __forceinline__ static void run(C2 (&a)[NR]) {
#pragma unroll
    for (int blk = 0; blk < NR; blk += 2 * SPAN) {
#pragma unroll
      for (int j = 0; j < SPAN; ++j) {
        const C2 u = a[blk + j], v = a[blk + j + SPAN];
        a[blk + j] = u + v;
        a[blk + j + SPAN] = rot_diff<DIR>(u, v, j * (32 / (2 * SPAN)));
      }
    }
    DifStage<NR, SPAN / 2, DIR, C2>::run(a);
  }
};
template <int NR, int DIR>
struct DifStage<NR, 0, DIR, C2> {
  __device__ __forceinline__ static void run(C2 (&)[NR]) {}
};

// Forward DFT of size NR of two lines held apart (p: line 0, q: line 1).  The
// first stage runs in scalar instructions that write straight into the pairs:
// the same FMA-pipe time, and no instructions spent on pairing the operands.
template <int NR>
__device__ __forceinline__ void dft_reg_split(const float2 (&p)[NR], const float2 (&q)[NR], C2 (&a)[NR]) {
  constexpr int H = NR / 2;
  C2 b[NR];
#pragma unroll
  for (int j = 0; j < H; ++j) {
    b[j] = C2{pk(p[j].x + p[j + H].x, q[j].x + q[j + H].x), pk(p[j].y + p[j + H].y, q[j].y + q[j + H].y)};
    const int r = j * (32 / NR);
    if (r == 8) {  // -i (u - v)
      b[j + H] = C2{pk(p[j].y - p[j + H].y, q[j].y - q[j + H].y), pk(p[j + H].x - p[j].x, q[j + H].x - q[j].x)};
    } else {
      const C2 d{pk(p[j].x - p[j + H].x, q[j].x - q[j + H].x), pk(p[j].y - p[j + H].y, q[j].y - q[j + H].y)};
      b[j + H] = r == 0 ? d : rot_pair<-1>(d, r);
    }
  }
  DifStage<NR, NR / 4, -1, C2>::run(b);
  BitRevCopy<NR, 0, C2>::run(b, a);
}

// Line<N> for two lines per thread.  tw holds W_N^{t k1} at [k1 * N1 + t]
// (threads of a warp read neighbouring entries, where the natural order
// [(t k1) mod N] puts the even k1 on few banks).  The exchange area of a line
// pair keeps element (t, k1) at t (N2 + 1) + k1: conflict-free both ways with
// addresses known at compile time up to one base.  Twiddles multiply in
// scalar instructions, which take the factors unpaired.
template <int N, typename Sync>
struct Line2 {
  static constexpr int N1 = Split<N>::N1, N2 = Split<N>::N2, S = N2 / N1;
  static constexpr int P = N2 + 1, AREA = N1 * P;

  __device__ __forceinline__ static void load_twiddles(float2* tw, const float2* __restrict__ twg) {
    for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = twg[((i % N1) * (i / N1)) & (N - 1)];
  }
  // a W (DIR < 0) or a conj(W) (DIR > 0)
  template <int DIR>
  __device__ __forceinline__ static C2 twiddle(C2 a, float2 w) {
    const float s = DIR < 0 ? w.y : -w.y;
    return C2{pk(fmaf(lo(a.x), w.x, -lo(a.y) * s), fmaf(hi(a.x), w.x, -hi(a.y) * s)),
              pk(fmaf(lo(a.x), s, lo(a.y) * w.x), fmaf(hi(a.x), s, hi(a.y) * w.x))};
  }
  // p[n2], q[n2] = the two lines at t + N1 n2  ->  exchange area
  __device__ __forceinline__ static void fwdA(const float2 (&p)[N2], const float2 (&q)[N2], int t, C2* ex,
                                              const float2* tw, Sync sync) {
    C2 a[N2];
    dft_reg_split<N2>(p, q, a);
    C2* e = ex + t * P;
    e[0] = a[0];
#pragma unroll
    for (int k1 = 1; k1 < N2; ++k1) e[k1] = twiddle<-1>(a[k1], tw[k1 * N1 + t]);
    sync();
  }
  // forward stage B, the multiplier ks (signed wavenumber)^2, inverse stage B
  __device__ __forceinline__ static void mid(int t, C2* ex, float ks, Sync sync) {
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const int k1 = t + N1 * s;
      C2* e = ex + k1;
      C2 b[N1];
#pragma unroll
      for (int j = 0; j < N1; ++j) b[j] = e[j * P];
      dft_reg<N1, -1>(b);
#pragma unroll
      for (int k2 = 0; k2 < N1; ++k2) {
        // slot k = k1 + N2 k2 < N/2 exactly when k2 < N1/2
        const float kf = (float)k1 + (float)(k2 < N1 / 2 ? N2 * k2 : N2 * k2 - N);
        const V2 m = dup(ks * (kf * kf));
        b[k2] = C2{b[k2].x * m, b[k2].y * m};
      }
      dft_reg<N1, +1>(b);
#pragma unroll
      for (int j = 0; j < N1; ++j) e[j * P] = b[j];
    }
    sync();
  }
  // exchange area -> a[n2] = (unnormalized inverse)[t + N1 n2]
  __device__ __forceinline__ static void invA(C2 (&a)[N2], int t, const C2* ex, const float2* tw) {
    const C2* e = ex + t * P;
    a[0] = e[0];
#pragma unroll
    for (int k1 = 1; k1 < N2; ++k1) a[k1] = twiddle<1>(e[k1], tw[k1 * N1 + t]);
    dft_reg<N2, +1>(a);
  }
};

}  // namespace bdg
