// Line FFTs for few lines: four points per thread.
//
// The four-step lines of fft.cuh put 8 to 32 points on a thread.  With FP64
// at two multiply-adds per clock and SM (a warp instruction takes 64 clocks
// of its quarter of the SM), a problem of a few hundred lines then sits on a
// few SMs: 144 lines of 256 points are 72 warps, on 12 CTAs.  Here a line of
// N points is N/4 threads, so that the same work reaches four times as many
// SM quarters and each thread's chain is a quarter as long.  Stockham radix-4
// stages (a last radix-2 stage for N = 2 4^k) exchange through shared memory;
// thread t holds points t + (N/4) k before and after the forward and the
// inverse transform, so a k-space multiplier needs no reordering.
#pragma once

#include "common.cuh"

namespace bdg {

// Lines (of all vectors and components) up to which a pass runs this way.
// Measured, FP64 product, full (fft.cuh) -> spread: 144 lines of 256 (1-D, 24
// vectors) 66 -> 9.7 us, 1-D 1024 x 24 155 -> 32 us, 64^2 x 1 42 -> 15 us,
// 64^2 x 12 (4608 lines) 77 -> 72 us, x 24 (9216) 125 -> 136 us, 128^2 x 4
// (3072) 123 -> 114 us, x 12 (9216) 279 -> 313 us, 256^2 x 2 (3072) 252 -> 226
// us, 32^3 x 1 (6144) 61 -> 65 us.  Beyond, the FP64 pipes are busy either way
// and the radix-4 stages' extra twiddles cost about 10 %.
constexpr long long FEW_LINES = 5000;

struct SpreadWarp {  // the line's threads are in one warp
  __device__ __forceinline__ void operator()() const { __syncwarp(); }
};
template <int THREADS>
struct SpreadBar {  // they are the first THREADS of the CTA
  __device__ __forceinline__ void operator()() const { asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory"); }
};

template <int N, typename T>
struct Spread {
  typedef decltype(T().x) R;
  static constexpr int TH = N / 4;                                   // threads per line
  static constexpr int LOG = N == 8 ? 3 : N == 16 ? 4 : N == 32 ? 5 : N == 64 ? 6 : N == 128 ? 7 : N == 256 ? 8 : N == 512 ? 9 : 10;
  static constexpr int NS = LOG / 2;                                 // radix-4 stages
  static constexpr bool R2 = LOG % 2;                                // and a radix-2 stage
  static constexpr int NT = R2 ? NS : NS - 1;                        // stages with twiddles
  static constexpr int WARP_LINES = TH < 32 ? 32 / TH : 1;           // lines of a group of threads
  static constexpr int FT = WARP_LINES * TH;                         // threads of the group

  T w[NT][3];  // twiddles of this thread's butterflies

  __device__ __forceinline__ void load_twiddles(int t, const T* __restrict__ tw) {
#pragma unroll
    for (int i = 0; i < NT; ++i) {
      const int s = 1 << (2 * i), ps = t & ~(s - 1);  // p s with p = t / s
#pragma unroll
      for (int k = 1; k < 4; ++k) w[i][k - 1] = tw[(ps * k) & (N - 1)];
    }
  }
  // DIR = -1 forward, +1 inverse (unnormalized); ex: 2 N values
  template <int DIR, typename Sync>
  __device__ __forceinline__ void run(T (&a)[4], int t, T* ex, Sync sync) const {
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      const T p = a[0] + a[2], m = a[0] - a[2], q = a[1] + a[3], d = a[1] - a[3];
      const T j = DIR < 0 ? mk(d.y, -d.x) : mk(-d.y, d.x);  // DIR i (a1 - a3)
      a[0] = p + q;
      a[1] = m + j;
      a[2] = p - q;
      a[3] = m - j;
      if (i < NT) {
#pragma unroll
        for (int k = 1; k < 4; ++k) a[k] = DIR < 0 ? cmul(a[k], w[i < NT ? i : 0][k - 1]) : cmulc(a[k], w[i < NT ? i : 0][k - 1]);
      }
      if (i + 1 < NS || R2) {
        const int s = 1 << (2 * i);
        T* b = ex + (i & 1) * N;
        T* o = b + (t & (s - 1)) + 4 * (t & ~(s - 1));
#pragma unroll
        for (int k = 0; k < 4; ++k) o[k * s] = a[k];
        sync();
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] = b[t + TH * k];
      }
    }
    if (R2) {
      const T u0 = a[0] + a[2], u2 = a[0] - a[2], u1 = a[1] + a[3], u3 = a[1] - a[3];
      a[0] = u0; a[1] = u1; a[2] = u2; a[3] = u3;
    }
    if ((NS - 1 + (R2 ? 1 : 0)) & 1) sync();  // an odd number of exchanges: the next run starts in the half read last
  }
};

}  // namespace bdg
