// FP64 BdG product for many lines of 128 or 256 points: the spectral Laplacian
// of each axis as a matrix product on the tensor cores, exact in integer
// digits (digits.cuh), and the pointwise coupling in a kernel of its own.
//
// Along one axis -1/2 d^2/dx^2 is the real symmetric circulant kappa K with
// K[0] = (N^2 + 2) / 12 and K[m] = (-1)^m / (2 sin^2(pi m / N)), the inverse
// transform of k^2 (eq. laplace_approx; the Nyquist mode counts (N/2)^2), and
// kappa = 1/2 (2 pi / len)^2.  FP64 arithmetic runs at two multiply-adds per
// clock and SM on this part, and the FFT passes are bound by it (about 27
// instructions per real value and axis).  Here a line is cut into seven 8-bit
// digits against its own largest exponent, the table K likewise, and the 34
// digit products of the eight leading weights are summed exactly by
// tcgen05.mma (K = 128 terms); the eight sums of a value are put together in
// 64-bit integers, and one FP64 multiply-add per value adds the result to y.
// Lines of 256 points are folded first: sums and differences of the points n
// and n + 128 meet a circulant and a skew-circulant of 128 points each, which
// halves the products and costs integer additions only.
//
// What is lost: up to a unit of 2^-55 of the line's largest value, half one of 2^-55 of
// K[0]'s power of two, and the weights past the eighth -- below the rounding of the FFTs
// (2^-53 at each of its stages).  Against extended precision, relative to the
// result, one axis, digits / FFT: noise 2.0e-16 / 2.9e-16 (N = 256), 2.1e-16 /
// 2.7e-16 (128), noise under a Gaussian 2.3e-16 / 2.9e-16, smooth functions
// (whose result is a small difference) 1.1e-13 / 1.9e-13.
//
// 256^2, 32 vectors, UV: 3097 us with FFTs -> 1052 us: 370 us per axis (a tile
// of 64 real lines takes 14 us of MMAs, each bound by its 6 KB of operands at
// 128 bytes per clock, and about 20 of integer work at 1.7 instructions a
// clock, one after the other: tensor memory and shared memory hold one block
// at a time), 310 us of coupling at 90 % of the FP64 pipe (FG, 24 vectors: 136 us).
//
// One CTA of sixteen warps per SM, 32 complex (64 real) lines a tile: the
// warps load, fold and cut the digits of a block of 128 x 64 values (MMA B
// operand, MN-major, core matrices 144 bytes apart so that both ways of
// walking a tile store without bank conflicts); the table's digits (A operand,
// 128 x 16 per chunk, 28 KB) stream through a ring of three stages from L2;
// 8 weights x 64 lines fill the tensor memory.
#include <cmath>

#include "apply.cuh"
#include "apply_impl.cuh"
#include "digits.cuh"

namespace bdg {

namespace {

constexpr int ND = 7, NW = 8;            // digits per value, weights kept
constexpr int BLK = 128;                 // points of a block
constexpr int LINES = 64;                // real lines of a tile
constexpr int CORE = 144;                // bytes from core matrix to core matrix along the lines
constexpr int X_TILE = BLK / 8 * (LINES / 8) * CORE;      // one digit of a block
constexpr int T_DIGIT = BLK * 16 * 2;                     // one digit of a table chunk (16 points)
constexpr int T_CHUNK = ND * T_DIGIT;
constexpr int STAGES = 3, CHUNKS = BLK / 16;
constexpr int THREADS = 512;
constexpr int SMEM = ND * X_TILE + STAGES * T_CHUNK + 8 * (2 * STAGES + 1) + 8 + LINES * 12;

__device__ __forceinline__ void bulk_load(void* dst, const void* src, int bytes, uint64_t* bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// Digits of a pair of folded values, |X| < 2^56: the top one, up to 256 in
// size, is biased by 512, the others by 128 (see digit_pairs).
__device__ __forceinline__ void folded_digits(long long x, long long y, uint32_t (&d)[ND]) {
  const unsigned long long bias = 0x0200808080808080ull;
  const unsigned long long u = (unsigned long long)x + bias, v = (unsigned long long)y + bias;
  const unsigned ul = (unsigned)u, uh = (unsigned)(u >> 32), vl = (unsigned)v, vh = (unsigned)(v >> 32);
  auto put = [&](int k, uint32_t w, unsigned short off) {
    const __half2 h = __hsub2(*reinterpret_cast<__half2*>(&w), __half2half2(__ushort_as_half(off)));
    d[k] = *reinterpret_cast<const uint32_t*>(&h);
  };
  put(0, __byte_perm(uh, vh, 0x7632) | 0x64006400u, 0x6600);  // 1024 + 512
  put(1, (__byte_perm(uh, vh, 0x0501) & 0x00FF00FFu) | 0x64006400u, 0x6480);
  put(2, (__byte_perm(uh, vh, 0x0400) & 0x00FF00FFu) | 0x64006400u, 0x6480);
#pragma unroll
  for (int k = 3; k < ND; ++k)
    put(k, (__byte_perm(ul, vl, (6 - k) | ((10 - k) << 8)) & 0x00FF00FFu) | 0x64006400u, 0x6480);
}

// The eight weight sums of one result, in units of the sixth weight (rounded
// there): |c0..c2| < 2^22 by the table (its top digits are few), all below
// 2^24, integers.
__device__ __forceinline__ long long weigh(const float (&c)[NW]) {
  auto small = [](float v) { return __float_as_int(v + 12582912.f) - 0x4B400000; };  // 1.5 2^23
  const int a = (small(c[0]) << 8) + small(c[1]);
  const int b = (small(c[2]) << 8) + __float2int_rn(c[3]);
  const int e = (__float2int_rn(c[4]) << 8) + __float2int_rn(c[5]);
  const int f = __float2int_rn(c[6]) + ((__float2int_rn(c[7]) + 128) >> 8);
  const long long hi = (long long)(((unsigned long long)(unsigned)(a + (b >> 16)) << 32) | ((unsigned)b << 16));
  return hi + e + ((f + 128) >> 8);
}

// v 2^(top - TOP) as a double (round to nearest, away from zero in the ties)
// without the FP64 pipe; |v| < 2^62
constexpr int TOP = 1085;
__device__ __forceinline__ double to_double(long long v, int top) {
  const int s = (int)(v >> 63);
  const unsigned long long m = (unsigned long long)((v ^ (long long)s) - (long long)s);
  const int lz = __clzll((long long)m);  // 2 .. 64
  const unsigned long long n = (m << (lz & 63)) + 0x400;        // leading bit at 63, half a unit of bit 11 added
  unsigned long long bits = ((unsigned long long)(unsigned)(top - lz) << 52) + (n >> 11);  // (the leading bit adds one)
  if (n < 0x400ull) bits = (unsigned long long)(unsigned)(top + 2 - lz) << 52;                 // a carry out of bit 63
  if (m == 0) bits = 0;
  return __longlong_as_double((long long)(bits | ((unsigned long long)(unsigned)s << 63 & 0x8000000000000000ull)));
}

// y += s_c T x along one axis of N points with stride st (st = 1: the last
// axis).  Complex lines are numbered component by component; comp_bits:
// log2 of the lines per component, st_bits of st.
template <int N>
__global__ void __launch_bounds__(THREADS, 1)
    k_axis_digits(const double2* __restrict__ x, double2* __restrict__ y, long long npts, long long st, int comp_bits,
                  int st_bits, long long nlines, const uint8_t* __restrict__ table, double kfac, int kexp, int mode) {
  constexpr int NB = N / BLK;   // blocks of a line
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t* xd = smem;
  uint8_t* td = smem + ND * X_TILE;
  uint64_t* full = reinterpret_cast<uint64_t*>(td + STAGES * T_CHUNK);
  uint64_t* empty = full + STAGES;
  uint64_t* done = empty + STAGES;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  int* bad = reinterpret_cast<int*>(tmem_slot + 1);          // a wait ran out: the results become NaN
  unsigned* ex = reinterpret_cast<unsigned*>(tmem_slot + 2);  // [LINES] largest magnitudes
  double* sc = reinterpret_cast<double*>(ex + LINES);       // [LINES] scale of the result
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;

  if (warp == 0) tmem_alloc(tmem_slot, 512);
  if (tid == 0) {
    *bad = 0;
    for (int s = 0; s < STAGES; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&full[s])) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[s])) : "memory");
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(done)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t idesc = mma_idesc_f16(BLK, LINES, true, true);
  bool lost = false;
  unsigned chunk = 0, blocks = 0;   // table chunks and blocks so far
  const long long ntiles = (nlines + LINES / 2 - 1) / (LINES / 2);
  const unsigned nchunks = (unsigned)((ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x) * NB * CHUNKS;  // of this CTA
  // loads of the table run STAGES chunks ahead of the MMAs, over the ends of
  // blocks and tiles (one thread of warp 1)
  auto load_chunk = [&](unsigned at) {
    if (at >= nchunks) return;
    const unsigned s = at % STAGES;
    // the MMAs that read this stage STAGES chunks ago are done (a fresh barrier's other phase counts as complete)
    if (!mma_wait(&empty[s], ((at / STAGES) & 1) ^ 1)) lost = true;
    bulk_load(td + s * T_CHUNK, table + (size_t)(at % (NB * CHUNKS)) * T_CHUNK, T_CHUNK, &full[s]);
  };
  if (warp == 1) {
    if (elect_one())
      for (unsigned c = 0; c < STAGES; ++c) load_chunk(c);
    __syncwarp();
  }

  // a task is four complex lines at one point of the block; neighbouring
  // threads take neighbouring points (last axis) or neighbouring lines
  const int g = st == 1 ? tid >> 6 : tid & 7, n0 = st == 1 ? tid & 63 : tid >> 3;
  // first element of complex line l of a tile
  auto line_base = [&](long long tile, int l) {
    long long ln = tile * (LINES / 2) + l;
    if (ln >= nlines) ln = nlines - 1;
    const long long vc = ln >> comp_bits, in = ln & ((1LL << comp_bits) - 1);
    return vc * npts + (in >> st_bits) * (N * st) + (in & (st - 1));
  };
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    if (tid < LINES) ex[tid] = 0;
    double2 v[2][4][NB];
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const double2* p = x + line_base(tile, 4 * g + l) + n0 * st;
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int b = 0; b < NB; ++b) v[q][l][b] = p[(64 * q + BLK * b) * st];
    }
    __syncthreads();
    // largest magnitude of every real line
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      unsigned mr = 0, mi = 0;
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          mr = max(mr, magnitude(v[q][l][b].x));
          mi = max(mi, magnitude(v[q][l][b].y));
        }
      if (st == 1) {
        mr = __reduce_max_sync(0xffffffffu, mr);
        mi = __reduce_max_sync(0xffffffffu, mi);
      } else {
#pragma unroll
        for (int o = 8; o < 32; o <<= 1) {
          mr = max(mr, __shfl_xor_sync(0xffffffffu, mr, o));
          mi = max(mi, __shfl_xor_sync(0xffffffffu, mi, o));
        }
      }
      if (st == 1 ? lane == 0 : lane < 8) {
        atomicMax(&ex[8 * g + 2 * l], mr);
        atomicMax(&ex[8 * g + 2 * l + 1], mi);
      }
    }
    __syncthreads();
    // tiny lines (digits.cuh) among the tile's are cut times 2^GROW; their
    // scales hold that factor too, and the integer results its inverse
    const bool rare = __any_sync(0xffffffffu, is_tiny<double>(ex[lane]) || is_tiny<double>(ex[lane + 32]));
    auto tiny = [&](int line) { return rare && is_tiny<double>(ex[line]); };
    auto top_of = [&](int line) { return tiny(line) ? TOP - Tiny<double>::GROW : TOP; };
    if (tid < LINES) {
      const int e = biased_exponent<double>(ex[tid]) + (tiny(tid) ? Tiny<double>::GROW : 0);
      const long long ln = min(tile * (LINES / 2) + tid / 2, nlines - 1);
      const double sg = mode == BDG_UV && (int)((ln >> comp_bits) % 6) >= 3 ? -kfac : kfac;
      sc[tid] = e >= 2047 ? (double)NAN : e == 0 ? 0.0 : scalbn(sg, e + kexp - 1076);
    }
    // fixed point, folded: block 0 the sums, block 1 the differences
    long long X[NB][2][4][2];
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const int lr = 8 * g + 2 * l, li = lr + 1;
      int er = (int)ex[lr], ei = (int)ex[li];
      auto grow = [&](int& e, auto part) {
        e = (biased_exponent<double>(e) + Tiny<double>::GROW) << 20;
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
          for (int b = 0; b < NB; ++b) part(v[q][l][b]) *= Tiny<double>::FACTOR;
      };
      if (tiny(lr)) grow(er, [](double2& z) -> double& { return z.x; });
      if (tiny(li)) grow(ei, [](double2& z) -> double& { return z.y; });
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        long long r[NB], i[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          r[b] = to_fixed<7>(v[q][l][b].x, er);
          i[b] = to_fixed<7>(v[q][l][b].y, ei);
        }
        if constexpr (NB == 2) {
          X[0][q][l][0] = r[0] + r[1];
          X[1][q][l][0] = r[0] - r[1];
          X[0][q][l][1] = i[0] + i[1];
          X[1][q][l][1] = i[0] - i[1];
        } else {
          X[0][q][l][0] = r[0];
          X[0][q][l][1] = i[0];
        }
      }
    }
    const int quarter = warp & 3, cg = (warp >> 2) * 16;   // read-back: outputs 32 quarter + lane, 16 real lines
    long long c0[16], c1[16];   // results at points j and (N = 256) j + 128
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      // (the last block's MMAs and read-backs are behind the barrier at the end of the loop)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        uint32_t d[4][ND];
#pragma unroll
        for (int l = 0; l < 4; ++l) folded_digits(X[b][q][l][0], X[b][q][l][1], d[l]);
        const int n = n0 + 64 * q;
        uint8_t* o = xd + ((n >> 3) * (LINES / 8) + g) * CORE + (n & 7) * 16;
#pragma unroll
        for (int k = 0; k < ND; ++k)
          *reinterpret_cast<uint4*>(o + k * X_TILE) = make_uint4(d[0][k], d[1][k], d[2][k], d[3][k]);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncthreads();
      if (warp == 1) {
        if (elect_one())
          for (int c = 0; c < CHUNKS; ++c) load_chunk(chunk + c + STAGES);
        __syncwarp();
      } else if (warp == 0) {
        tc_fence_after();
        const bool leader = elect_one();
        for (int c = 0; c < CHUNKS; ++c) {
          const unsigned at = chunk + c, s = at % STAGES;
          if (!mma_wait(&full[s], (at / STAGES) & 1)) lost = true;
          tc_fence_after();
          if (leader) {
            const uint64_t dt = mma_desc(smem_u32(td + s * T_CHUNK), BLK / 8 * 128, 128);
            const uint64_t dx = mma_desc(smem_u32(xd) + c * 2 * (LINES / 8) * CORE, (LINES / 8) * CORE, CORE);
#pragma unroll
            for (int i = 0; i < ND; ++i)       // table digit
#pragma unroll
              for (int j = 0; j < ND && i + j < NW; ++j)
                mma_f16(tmem + (uint32_t)((i + j) * LINES), dt + ((i * T_DIGIT) >> 4), dx + ((j * X_TILE) >> 4), idesc,
                        !(c == 0 && (i == 0 || (i == 1 && j == ND - 1))));
            mma_commit(&empty[s]);
            if (c == CHUNKS - 1) mma_commit(done);
          }
          __syncwarp();
        }
      }
      chunk += CHUNKS;
      if (b == 0 && tile + gridDim.x < ntiles) {  // the next tile's values come to L2 meanwhile
        for (int l = 0; l < 4; ++l) {
          const double2* p = x + line_base(tile + gridDim.x, 4 * g + l) + n0 * st;
#pragma unroll
          for (int q = 0; q < N / 64; ++q) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + 64 * q * st));
        }
      }
      if (!mma_wait(done, blocks & 1)) lost = true;
      ++blocks;
      tc_fence_after();
      const uint32_t ta = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)cg;
#pragma unroll
      for (int q = 0; q < 16; q += 4) {
        float w[NW][4];
#pragma unroll
        for (int k = 0; k < NW; ++k) tmem_ld4(ta + (uint32_t)(k * LINES + q), w[k]);
        tmem_ld_wait();
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const float c[NW] = {w[0][p], w[1][p], w[2][p], w[3][p], w[4][p], w[5][p], w[6][p], w[7][p]};
          const long long r = weigh(c);
          if (b == 0) c0[q + p] = r;
          else {  // the differences' block: result pair
            const long long s = c0[q + p];
            c0[q + p] = s + r;
            c1[q + p] = s - r;
          }
        }
      }
      tc_fence_before();
      if (lost) *bad = 1;
      __syncthreads();   // digits and accumulators may be overwritten
    }
    // results at points j and j + 128 of eight complex lines
    const int j = 32 * quarter + lane;
    if (st == 1) {  // neighbouring lanes hold neighbouring elements of y
#pragma unroll
      for (int q = 0; q < 16; q += 2) {
        const int l = (cg + q) / 2;
        if (tile * (LINES / 2) + l >= nlines) continue;
        double2* p = y + line_base(tile, l) + j;
        const double sr = *bad ? (double)NAN : sc[cg + q], si = *bad ? (double)NAN : sc[cg + q + 1];
        double2 u = *p;
        double2 w = NB == 2 ? p[BLK] : u;
        const int tr = top_of(cg + q), ti = top_of(cg + q + 1);
        *p = make_double2(fma(to_double(c0[q], tr), sr, u.x), fma(to_double(c0[q + 1], ti), si, u.y));
        if constexpr (NB == 2)
          p[BLK] = make_double2(fma(to_double(c1[q], tr), sr, w.x), fma(to_double(c1[q + 1], ti), si, w.y));
      }
    } else {        // through shared memory, where the digits were: lanes to neighbouring lines
      long long* stage = reinterpret_cast<long long*>(xd);   // [128 points][32 lines][re, im], lines swizzled
      const bool on = tile * (LINES / 2) + lane < nlines;
      double2* p = y + line_base(tile, lane);
      const double sr = *bad ? (double)NAN : sc[2 * lane], si = *bad ? (double)NAN : sc[2 * lane + 1];
      const int tr = top_of(2 * lane), ti = top_of(2 * lane + 1);
#pragma unroll
      for (int h = 0; h < NB; ++h) {
        if (h) __syncthreads();
#pragma unroll
        for (int q = 0; q < 16; q += 2) {
          const int l = (cg + q) / 2;
          *reinterpret_cast<longlong2*>(stage + 2 * (j * 32 + (l ^ lane))) =
              h ? make_longlong2(c1[q], c1[q + 1]) : make_longlong2(c0[q], c0[q + 1]);
        }
        __syncthreads();
        if (on) {
          constexpr int RB = 4;   // rows in flight
          for (int n = warp; n < BLK; n += 16 * RB) {
            double2 u[RB];
#pragma unroll
            for (int r = 0; r < RB; ++r) u[r] = p[(h * BLK + n + 16 * r) * st];
#pragma unroll
            for (int r = 0; r < RB; ++r) {
              const int m = n + 16 * r;
              const longlong2 c = *reinterpret_cast<const longlong2*>(stage + 2 * (m * 32 + (lane ^ (m & 31))));
              p[(h * BLK + m) * st] = make_double2(fma(to_double(c.x, tr), sr, u[r].x), fma(to_double(c.y, ti), si, u[r].y));
            }
          }
        }
      }
    }
    __syncthreads();   // sc, ex
  }
  // (after a lost wait, MMAs and a table load may still run: both are waited for once more, bounded)
  if (__syncthreads_or(lost) && nchunks > 0) {
    mma_wait(done, (blocks - 1) & 1);
    for (int s = 0; s < STAGES; ++s) mma_wait(&full[s], (((nchunks - 1 - s) / STAGES) & 1));
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_free(tmem, 512);
}

// acc + row r of m times x
__device__ __forceinline__ double2 row_fma(double m0, double m1, double m2, const double2 (&x)[3], double2 acc) {
  return cfma(x[2], m2, cfma(x[1], m1, cfma(x[0], m0, acc)));
}
__device__ __forceinline__ void mul3_add(const Sym3<double>& m, const double2 (&x)[3], double2 (&y)[3]) {
  y[0] = row_fma(m.d0, m.o01, m.o02, x, y[0]);
  y[1] = row_fma(m.o01, m.d1, m.o12, x, y[1]);
  y[2] = row_fma(m.o02, m.o12, m.d2, x, y[2]);
}

// y = C x: the pointwise coupling of all six components, one thread per node
// and up to VECS vectors, for which the node's 21 coefficients are formed
// once.  The UV form sums A u + B v and B u + A v as they stand: half the
// products would do with (A + B) / 2 and (A - B) / 2 on u + v and u - v, but the
// small B u would then be a difference of two terms of the size of A u.  The
// CTAs of all nodes, then of all groups of vectors, lie along x (gridDim.y ends
// at 65535 groups, about a million vectors); node_bits: log2 of the node blocks.
constexpr int VECS = 16;
__global__ void __launch_bounds__(128) k_couple(const double2* __restrict__ x, double2* __restrict__ y, long long npts,
                                                int node_bits, int nvec, const dquad* __restrict__ phiv,
                                                Coupling<double> cp, int mode) {
  const long long i = (long long)(blockIdx.x & ((1u << node_bits) - 1)) * 128 + threadIdx.x;
  Sym3<double> A, B;   // UV: the blocks; FG: A + B and A - B
  coupling_blocks<double>(phiv[i], cp, A, B);
  if (mode != BDG_UV) {
    const Sym3<double> P = sym_add(A, B, 1.0);
    B = sym_add(A, B, -1.0);
    A = P;
  }
  const int v0 = (int)(blockIdx.x >> node_bits) * VECS, v1 = min(nvec, v0 + VECS);
  for (int v = v0; v < v1; ++v) {
    const double2* p = x + (long long)v * 6 * npts + i;
    double2* o = y + (long long)v * 6 * npts + i;
    double2 a[3], b[3], f[3], g[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      a[c] = p[c * npts];
      b[c] = p[(3 + c) * npts];
      f[c] = g[c] = make_double2(0.0, 0.0);
    }
    mul3_add(A, a, f);
    if (mode == BDG_UV) {
      mul3_add(B, b, f);
      mul3_add(B, a, g);
      mul3_add(A, b, g);
#pragma unroll
      for (int c = 0; c < 3; ++c) g[c] = make_double2(-g[c].x, -g[c].y);
    } else {
      mul3_add(B, b, g);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      o[c * npts] = f[c];
      o[(3 + c) * npts] = g[c];
    }
  }
}

// Fixed-point table values T[block][m] for the points' distance m (block 1 is
// skew: T[-m] = -T[128 - m]).
struct TableValues {
  long long t[2][BLK];
};
// the table's digits as the MMA reads them: [block][chunk of 16 points n][digit]
// [n group of 8][j group of 8][n][j], FP16
__global__ void __launch_bounds__(256) k_table(const __grid_constant__ TableValues tv, int blocks, __half* __restrict__ out) {
  const int total = blocks * CHUNKS * 16 * BLK;
  for (int e = blockIdx.x * 256 + threadIdx.x; e < total; e += gridDim.x * 256) {
    const int j = e % BLK, n = e / BLK % BLK, b = e / (BLK * BLK);
    const int m = j - n;
    long long t = tv.t[b][m < 0 ? m + BLK : m];
    if (m < 0 && b == 1) t = -t;
    const unsigned long long u = (unsigned long long)t + 0x80808080808080ull;
    const int c = n / 16, n8 = n / 8 % 2;
    __half* o = out + (size_t)(b * CHUNKS + c) * (T_CHUNK / 2) + (n8 * (BLK / 8) + j / 8) * 64 + (n % 8) * 8 + j % 8;
#pragma unroll
    for (int k = 0; k < ND; ++k) {
      const int d = (int)(k == 0 ? u >> 48 : (u >> (8 * (ND - 1 - k))) & 0xFF) - 128;
      o[k * (T_DIGIT / 2)] = __int2half_rn(d);
    }
  }
}

}  // namespace

bool axis_digits_supported(int n) { return n == 128 || n == 256; }

// K[m] = (1/n) sum_k k^2 cos(2 pi k m / n), the Nyquist mode counted once, 0 <= m < n
static long double kernel_value(int n, int m) {
  if (m == 0) return ((long double)n * n + 2) / 12;
  const long double sn = sinl(3.14159265358979323846264338327950288L * m / n);
  return (m % 2 ? -1.0L : 1.0L) / (2 * sn * sn);
}

cudaError_t axis_digits_table(int n, uint8_t** out, int* kexp, cudaStream_t s) {
  *out = nullptr;
  const int blocks = n / BLK;
  cudaError_t e = cudaMalloc((void**)out, (size_t)blocks * CHUNKS * T_CHUNK);
  if (e != cudaSuccess) return e;
  TableValues tv;
  *kexp = 0;
  const long double top = blocks == 2 ? 0.5L * (kernel_value(n, 0) + fabsl(kernel_value(n, BLK))) : kernel_value(n, 0);
  while (ldexpl(1.0L, *kexp) <= top) ++*kexp;
  for (int m = 0; m < BLK; ++m) {
    const long double a = kernel_value(n, m), b = blocks == 2 ? kernel_value(n, m + BLK) : 0.0L;
    tv.t[0][m] = llroundl(ldexpl(blocks == 2 ? 0.5L * (a + b) : a, 55 - *kexp));
    tv.t[1][m] = llroundl(ldexpl(0.5L * (a - b), 55 - *kexp));
  }
  k_table<<<64, 256, 0, s>>>(tv, blocks, (__half*)*out);
  return cudaGetLastError();
}

cudaError_t couple_launch(const ApplyArgs<double>& g, cudaStream_t s) {
  const long long nodes = g.grid->npts / 128;   // (an axis of 128 or 256 points: a power of two, no remainder)
  const long long ctas = nodes * ((g.nvec + VECS - 1LL) / VECS);
  k_couple<<<(unsigned)ctas, 128, 0, s>>>(g.x, g.y, g.grid->npts, log2i(nodes), g.nvec, g.phiv, g.cp, g.mode);
  return cudaGetLastError();
}

template <int N>
static cudaError_t launch(const ApplyArgs<double>& g, int ax, cudaStream_t s) {
  cudaError_t e = allow_dynamic_smem((const void*)k_axis_digits<N>, SMEM);
  if (e != cudaSuccess) return e;
  long long st = 1;
  for (int a = ax + 1; a < g.grid->dim; ++a) st *= g.grid->n[a];
  const long long per = g.grid->npts / N, nlines = per * 6 * g.nvec, tiles = (nlines + LINES / 2 - 1) / (LINES / 2);
  k_axis_digits<N><<<(unsigned)(tiles < 152 ? tiles : 152), THREADS, SMEM, s>>>(
      g.x, g.y, g.grid->npts, st, log2i(per), log2i(st), nlines, g.kdig[ax], g.kfac[ax], g.kexp[ax], g.mode);
  return cudaGetLastError();
}

cudaError_t axis_digits_launch(const ApplyArgs<double>& g, int ax, cudaStream_t s) {
  return g.grid->n[ax] == 128 ? launch<128>(g, ax, s) : launch<256>(g, ax, s);
}

}  // namespace bdg
