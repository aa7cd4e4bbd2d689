// Tall-skinny Gram G = A^T B of two pair blocks on the tensor cores
// (tcgen05.mma kind::f16, accumulators in tensor memory), from exact digits
// (digits.cuh): FP64 accuracy with seven digits per element (34 digit
// products), FP32 accuracy with four (10).
//
// A CTA owns a tile of 128 x NT real columns and a range of row chunks of
// CHUNK = 256 rows.  Every column has one exponent per chunk (k_col_exp),
// against which its values are cut into digits; within a chunk the products
// of each digit weight add up in one FP32 accumulator, exactly for the four
// leading weights (256 rows x 4 pairs x 2^14 = 2^24), to 2^-24 of a part
// below 2^-32 of the result for the others.  After a chunk the accumulators
// are read back.  FP64 accuracy: the weights are put together in a 64-bit
// integer, in units of 2^-54 of the product of the columns' largest values, and
// added to an FP64 sum per output in registers.  (In one double-float sum, the
// weights from the fourth on in one float, what 256 rows lost was 2^-47 of that
// product, and of 288 FP64 solves of 64^2 problems 38 levelled off above their
// tolerance of 1e-10; 18 with double-float Grams, one or two now.)  FP32 accuracy: the
// leading three weights error-free into a double-float sum.  The CTA writes its
// sums as FP64, and the CTAs' partial sums are added in FP64 in a fixed order.
//
// Digits are relative to the largest value of 256 rows, so their error is small
// beside |a| |b| but not always beside sum |a b|: columns whose large parts lie
// apart have a small sum that the rounding of those parts covers.  A checked
// Gram (CHECK) therefore forms, per output, what the digits may have lost and a
// 14-bit estimate of sum |a b|: the leading digits' absolute values are one more
// digit tile and one more accumulator, and k_col_exp adds up |x| of every column
// and chunk.  An element is off by at most a unit, 2^-55 of its column's largest
// value a^, so a chunk by 2^-55 (a^ sum |b| + b^ sum |a|); outputs for which that
// exceeds 2^-49 of the estimate in all are marked, and the caller forms them in
// double-float (gram_pairs_checked).  Random columns and functions on the same
// support stay below by a factor of six and more.
//
// Why: a double-float multiply-add is 15 FP32 instructions, so the same
// contraction in double-float is bound by the FP32 pipe at 5 TFLOP/s (and
// measured at 3).  Here the arithmetic is 34 (10) FP16 products per
// multiply-add on the tensor cores, and cutting the digits about 30 integer
// instructions per element and tile.  72 x 72 pairs of 196608 rows: 2627 -> 648
// us, 711 with the check and the calls that follow it (66 us are the pass over the
// exponents, 571 and 614 the products), error 5e-15 -> 6e-16 of |G|; 24 x 24: 534
// -> 147 and 172 us.  Columns that all lie apart pay for both ways: 3340 us.  A
// stage of 32 rows takes about 5000 clocks there, 3080 of them MMAs (70, each bound
// by its 5.5 KB of operands at 128 bytes per clock); the rest is cutting that they
// do not cover.
//
// Operand tiles are MN-major without swizzle: a core matrix holds 8 rows (K)
// of 8 neighbouring real columns (16 bytes), so that a thread that has one
// row of four complex columns stores 16 bytes per digit, a warp reads 32
// consecutive rows of a column and its stores cover whole bank cycles.
#include <algorithm>

#include "blas.cuh"
#include "digits.cuh"

namespace bdg {

namespace {

constexpr int TM = 128;      // A real columns per CTA (MMA M)
constexpr int TBK = 32;      // rows per pipeline stage (two MMA K steps of 16)
constexpr int PWARPS = 16;   // warps that cut digits and read back; one more issues the MMAs
constexpr int TTHREADS = 32 * (PWARPS + 1);
constexpr int CHUNK = 256;   // rows per exponent and per read-back
constexpr int STEPS = CHUNK / TBK;
// digit weights kept: with seven digits the eighth as well, whose pairs would
// otherwise be the largest error
template <int ND> constexpr int weights() { return ND == 7 ? ND + 1 : ND; }
// stages in flight: what shared memory holds
template <int ND> constexpr int stages() { return ND == 7 ? 2 : 3; }
inline int padded8(int cols) { return (cols + 7) / 8 * 8; }

// 2^e as a float for e <= 0, 0 below the normal range
__device__ __forceinline__ float pow2_neg(int e) { return e < -126 ? 0.f : __int_as_float((e + 127) << 23); }
// |x| 2^(1022 - emax), by its bits (a subnormal counts as zero)
__device__ __forceinline__ float fraction(double x, int emax) {
  const unsigned hi = (unsigned)__double2hiint(x);
  const int e = (int)(hi >> 20) & 0x7FF;
  if (e == 0) return 0.f;
  return __uint_as_float(0x3F800000u | (__funnelshift_l((unsigned)__double2loint(x), hi, 3) & 0x7FFFFFu)) *
         pow2_neg(e - 1 - emax);
}

// A column's entry in the table of exponents: the biased exponent of its largest
// value in the chunk, with TINY_BIT where that is a tiny one (digits.cuh).
constexpr int TINY_BIT = 0x1000;
__device__ __forceinline__ int exponent_in(int entry) { return entry & (TINY_BIT - 1); }

// exps[chunk * ld + 2 c + part]: the entries of the column's real and imaginary
// parts; one warp per chunk and complex column, the columns up to ld (2 cols
// rounded up to 8) are zero.  sums (SUMS, FP64 blocks), laid out alike: the sum of
// |x| in units of the power of two above the largest value, and half a unit.
template <typename R, bool SUMS>
__global__ void __launch_bounds__(256) k_col_exp(PairBlock<R> X, int nchunks, int ld, short* __restrict__ exps,
                                                 float* __restrict__ sums) {
  typedef typename CT<R>::T T;
  const int warp = (int)((blockIdx.x * 256LL + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  const int c = warp / nchunks, chunk = warp - c * nchunks;
  if (2 * c >= ld) return;
  auto entry = [](unsigned m) { return biased_exponent<R>(m) | (is_tiny<R>(m) ? TINY_BIT : 0); };
  if (c >= X.cols) {
    if (lane == 0) {
      *reinterpret_cast<short2*>(exps + (long long)chunk * ld + 2 * c) = make_short2(0, 0);
      if (SUMS) *reinterpret_cast<float2*>(sums + (long long)chunk * ld + 2 * c) = make_float2(0.f, 0.f);
    }
    return;
  }
  const T* p = X.p + (long long)c * X.ld + (long long)chunk * CHUNK;
  const int rows = (int)min((long long)CHUNK, X.n - (long long)chunk * CHUNK);
  unsigned mx = 0, my = 0;
  T v[CHUNK / 32];
#pragma unroll
  for (int k = 0; k < CHUNK / 32; ++k) {
    const int r = lane + 32 * k;
    v[k] = mk((R)0, (R)0);
    if (r < rows) v[k] = p[r];
    mx = max(mx, magnitude(v[k].x));
    my = max(my, magnitude(v[k].y));
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  my = __reduce_max_sync(0xffffffffu, my);
  if (lane == 0) *reinterpret_cast<short2*>(exps + (long long)chunk * ld + 2 * c) = make_short2((short)entry(mx), (short)entry(my));
  if constexpr (SUMS) {
    float sx = 0.f, sy = 0.f;
#pragma unroll
    for (int k = 0; k < CHUNK / 32; ++k) {
      sx += fraction(v[k].x, biased_exponent<double>(mx));
      sy += fraction(v[k].y, biased_exponent<double>(my));
    }
    for (int o = 16; o > 0; o >>= 1) {
      sx += __shfl_xor_sync(0xffffffffu, sx, o);
      sy += __shfl_xor_sync(0xffffffffu, sy, o);
    }
    if (lane == 0) *reinterpret_cast<float2*>(sums + (long long)chunk * ld + 2 * c) = make_float2(sx + 0.5f, sy + 0.5f);
  }
}

// v 2^(e - 40) as a double for |v| < 2^62 and e <= 0 (0 for e < -900), rounded to
// nearest, without the FP64 pipe
__device__ __forceinline__ double chunk_value(long long v, int e) {
  const int s = (int)(v >> 63);
  const unsigned long long m = (unsigned long long)((v ^ (long long)s) - (long long)s);
  const int lz = __clzll((long long)m);                                 // 2 .. 64
  const unsigned long long n = (m << (lz & 63)) + 0x400;
  unsigned long long bits = ((unsigned long long)(unsigned)(1045 - lz + e) << 52) + (n >> 11);   // (the leading bit adds one)
  if (n < 0x400ull) bits = (unsigned long long)(unsigned)(1047 - lz + e) << 52;                  // a carry out of bit 63
  if (m == 0 || e < -900) bits = 0;
  return __longlong_as_double((long long)(bits | ((unsigned long long)(unsigned)s << 63 & 0x8000000000000000ull)));
}

// Work of one producer warp in every stage: four complex columns, 32 rows.
// Columns past the block's last are read from the last one: their digits land
// in rows (columns) of the tile that nothing reads.
template <typename R>
struct RowTask {
  const typename CT<R>::T* p;  // first column, the lane's row of the next load
  long long ld;                // column stride, 0 past the last column
  int c1, c2, c3;              // columns 1..3 in units of ld
  const short* e;              // exponents of the chunk of the next load
  typename CT<R>::T v[4];
  uint4 ev;                    // eight exponents (shorts)
  __device__ __forceinline__ void start(const PairBlock<R>& X, const short* exps, int c0, long long r) {
    const int last = X.cols - 1 - c0;
    p = X.p + (long long)c0 * X.ld + r;
    ld = X.ld;
    c1 = min(1, last);
    c2 = min(2, last);
    c3 = min(3, last);
    e = exps + 2 * c0;
  }
  __device__ __forceinline__ void load(bool in) {
    ev = *reinterpret_cast<const uint4*>(e);
    if (in) {
      v[0] = p[0];
      v[1] = p[c1 * ld];
      v[2] = p[c2 * ld];
      v[3] = p[c3 * ld];
    } else {
      v[0] = v[1] = v[2] = v[3] = mk((R)0, (R)0);
    }
    p += TBK;
  }
};
// digits of eight real columns at one row: 16 bytes per digit tile (and, with
// CHECK, one more of the leading digits' absolute values)
template <typename R, int ND, bool CHECK>
__device__ __forceinline__ void store_task(RowTask<R>& x, uint8_t* base, uint32_t tile_bytes) {
  unsigned e[4] = {x.ev.x, x.ev.y, x.ev.z, x.ev.w};
  constexpr unsigned LO = TINY_BIT, HI = (unsigned)TINY_BIT << 16;
  if ((e[0] | e[1] | e[2] | e[3]) & (LO | HI)) {   // (all lanes have the same columns)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (e[q] & LO) x.v[q].x *= Tiny<R>::FACTOR;
      if (e[q] & HI) x.v[q].y *= Tiny<R>::FACTOR;
      e[q] += (e[q] & LO ? Tiny<R>::GROW : 0) + (e[q] & HI ? Tiny<R>::GROW << 16 : 0);
    }
  }
  uint32_t d[4][ND];
#pragma unroll
  for (int q = 0; q < 4; ++q)
    digit_pairs<ND>(to_fixed<ND>(x.v[q].x, (int)(e[q] << 20)), to_fixed<ND>(x.v[q].y, (int)(e[q] << 4)), d[q]);
#pragma unroll
  for (int k = 0; k < ND; ++k)
    *reinterpret_cast<uint4*>(base + k * tile_bytes) = make_uint4(d[0][k], d[1][k], d[2][k], d[3][k]);
  if (CHECK) {
    constexpr uint32_t M = 0x7FFF7FFFu;
    *reinterpret_cast<uint4*>(base + ND * tile_bytes) = make_uint4(d[0][0] & M, d[1][0] & M, d[2][0] & M, d[3][0] & M);
  }
}

__device__ __forceinline__ void bar_init(uint64_t* bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// v 2^e without the FP64 pipe, on which a few instructions per output cost a
// short Gram more than its products
__device__ __forceinline__ double times_pow2(double v, int e) {
  const int f = (int)(__double2hiint(v) >> 20 & 0x7FF);
  if (f == 0 || f == 2047 || f + e < 1 || f + e > 2046) return scalbn(v, e);
  return __hiloint2double(__double2hiint(v) + (e << 20), __double2loint(v));
}
__device__ __forceinline__ double widened(float v) {
  const unsigned b = __float_as_uint(v), m = b & 0x7FFFFFFFu;
  if (m < 0x00800000u || m >= 0x7F800000u) return (double)v;
  return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + (896u << 20))), (int)(m << 29));
}

// part[group][i][j] for a tile of mw <= 128 x nw <= NT real columns over the chunks of blockIdx.z.  Sixteen producer warps cut the digits of
// the next stage while one thread issues the MMAs of the last; the read-back
// of a chunk comes after the next chunk's first stage is in place.  A wait
// that runs out writes NaN.  With CHECK, room, laid out like part, gets the
// estimate of sum |a b| less 2^49 times the bound of the error (see the head).
template <typename R, int ND, int NT, bool CHECK>
__global__ void __launch_bounds__(TTHREADS, 1)
    k_gram_digits(PairBlock<R> A, PairBlock<R> B, const short* __restrict__ expA, const short* __restrict__ expB, int ldea,
              int ldeb, int mw, int nw, int nchunks, int chunks_per_group, double* __restrict__ part,
              const float* __restrict__ sumA, const float* __restrict__ sumB, double* __restrict__ room, int* any) {
  constexpr int NW = weights<ND>(), TSTAGES = stages<ND>(), TILES = ND + CHECK, ACC = (NW + CHECK) * NT;
  constexpr uint32_t A_TILE = TM * TBK * 2, B_TILE = NT * TBK * 2, STAGE = TILES * (A_TILE + B_TILE);
  constexpr uint32_t NCOLS = ACC <= 32 ? 32 : ACC <= 64 ? 64 : ACC <= 128 ? 128 : ACC <= 256 ? 256 : 512;
  static_assert(ACC <= 512 && NT % 16 == 0, "one accumulator per digit weight");
  constexpr int NQ = NT / 4;  // output columns per thread
  extern __shared__ __align__(1024) uint8_t smem[];
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + TSTAGES * STAGE);
  uint64_t* empty = full + TSTAGES;
  uint64_t* acc_full = empty + TSTAGES;
  uint64_t* acc_free = acc_full + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_free + 1);
  int* ra = reinterpret_cast<int*>(tmem_slot + 2);  // [TM] largest exponents of the group's chunks
  int* rb = ra + TM;                                // [NT]
  // (the shuffle tells the compiler that the warp index is uniform)
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int i0 = blockIdx.x * mw, j0 = blockIdx.y * nw;
  const int Q2 = 2 * B.cols, i1 = min(2 * A.cols, i0 + mw), j1 = min(Q2, j0 + nw);
  const int ch0 = blockIdx.z * chunks_per_group, ch1 = min(nchunks, ch0 + chunks_per_group);

  if (warp == PWARPS) tmem_alloc(tmem_slot, NCOLS);
  if (CHECK && tid == 0 && blockIdx.x + blockIdx.y + blockIdx.z == 0) *any = 0;   // (the reduction sets it)
  if (tid == 0) {
    for (int s = 0; s < TSTAGES; ++s) {
      bar_init(&full[s], PWARPS);
      bar_init(&empty[s], 1);
    }
    bar_init(acc_full, 1);
    bar_init(acc_free, PWARPS);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int c = tid; c < TM + NT; c += TTHREADS) {
    const bool isA = c < TM;
    const int col = isA ? i0 + c : j0 + c - TM, ld = isA ? ldea : ldeb;
    const short* e = isA ? expA : expB;
    int m = 0;
    if (col < (isA ? i1 : j1))
      for (int ch = ch0; ch < ch1; ++ch) m = max(m, exponent_in(e[(long long)ch * ld + col]));
    (isA ? ra : rb)[isA ? c : c - TM] = m;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int nsteps = max(0, ch1 - ch0) * STEPS;
  bool lost = false;

  if (warp == PWARPS) {
    const uint32_t idesc = mma_idesc_f16(TM, NT, true, true);
    const bool leader = elect_one();
    for (int step = 0; step < nsteps; ++step) {
      const int st = step % TSTAGES, u = step / TSTAGES;
      if (!mma_wait(&full[st], (uint32_t)(u & 1))) lost = true;
      // accumulators of the chunk before have been read back
      if (step % STEPS == 0 && step > 0 && !mma_wait(acc_free, (uint32_t)((step / STEPS - 1) & 1))) lost = true;
      tc_fence_after();
      if (leader) {
        const uint32_t sa = smem_u32(smem + st * STAGE), sb = sa + TILES * A_TILE;
        const uint64_t da = mma_desc(sa, (TM / 8) * 128, 128), db = mma_desc(sb, (NT / 8) * 128, 128);
        const bool first = step % STEPS == 0;
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {
          auto mma = [&](int acc, int i, int j, bool accumulate) {
            mma_f16(tmem + (uint32_t)(acc * NT), da + ((i * A_TILE + kk * 2 * (TM / 8) * 128) >> 4),
                    db + ((j * B_TILE + kk * 2 * (NT / 8) * 128) >> 4), idesc, accumulate);
          };
#pragma unroll
          for (int i = 0; i < ND; ++i)
#pragma unroll
            for (int j = 0; j < ND && i + j < NW; ++j)
              mma(i + j, i, j, !(first && kk == 0 && (i == 0 || (j == ND - 1 && i + j >= ND && i == NW - ND))));
          if (CHECK) mma(NW, ND, ND, !(first && kk == 0));
        }
        mma_commit(&empty[st]);
        if (step % STEPS == STEPS - 1) mma_commit(acc_full);
      }
      __syncwarp();
    }
  } else {
    // tasks of a stage: groups of four complex columns of A, then of B, one or
    // two to a warp.  The loads of a task are issued a stage ahead.
    const int na = (i1 - i0 + 7) / 8, nt = na + (j1 - j0 + 7) / 8;
    RowTask<R> x[2];
    const long long r_first = (long long)ch0 * CHUNK + lane;
    auto start = [&](int q) {
      const int t = warp + PWARPS * q;
      if (t < na) x[q].start(A, expA + (long long)ch0 * ldea, i0 / 2 + 4 * t, r_first);
      else if (t < nt) x[q].start(B, expB + (long long)ch0 * ldeb, j0 / 2 + 4 * (t - na), r_first);
    };
    auto fetch = [&](int step, int q) {
      const int t = warp + PWARPS * q;
      if (t >= nt || step >= nsteps) return;
      if (step % STEPS == 0 && step > 0) x[q].e += t < na ? ldea : ldeb;
      x[q].load(r_first + (long long)step * TBK < A.n);
    };
    constexpr bool FP64 = ND == 7;
    float hi[NQ], lo[NQ];   // the sums of FP32 accuracy,
    double sum[NQ];         // and of FP64 accuracy,
    float rm[NQ];           // and their room, relative to the group's largest values
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      hi[q] = lo[q] = rm[q] = 0.f;
      sum[q] = 0.0;
    }
    const int quarter = warp & 3, jq = (warp >> 2) * NQ;
    const int row = 32 * quarter + lane;
    const uint32_t tlane = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)jq;
    auto read_back = [&](int chunk) {  // chunk of this group
      if (!mma_wait(acc_full, (uint32_t)(chunk & 1))) lost = true;
      tc_fence_after();
      const int ch = ch0 + chunk;
      // (a column of zeros in the chunk has no digits that mean anything)
      const int xa = i0 + row < i1 ? exponent_in(expA[(long long)ch * ldea + i0 + row]) : 0;
      const int ea = xa ? xa - ra[row] : -4096;
      const float fa = pow2_neg(ea);
      const float sa = CHECK && i0 + row < i1 ? sumA[(long long)ch * ldea + i0 + row] : 0.f;
#pragma unroll
      for (int c0 = 0; c0 < NQ; c0 += 4) {
        float v[NW][4], va[4], sb[4];
        if (CHECK) tmem_ld4(tlane + (uint32_t)(NW * NT + c0), va);
#pragma unroll
        for (int w = 0; w < NW; ++w) tmem_ld4(tlane + (uint32_t)(w * NT + c0), v[w]);
        int e[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int xb = j0 + jq + c0 + q < j1 ? exponent_in(expB[(long long)ch * ldeb + j0 + jq + c0 + q]) : 0;
          e[q] = xb ? xb - rb[jq + c0 + q] : -4096;
          sb[q] = CHECK && j0 + jq + c0 + q < j1 ? sumB[(long long)ch * ldeb + j0 + jq + c0 + q] : 0.f;
        }
        tmem_ld_wait();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (CHECK)
            rm[c0 + q] = fmaf(fa * pow2_neg(e[q]), fmaf(va[q], 0x1p-14f, -0x1p-6f * (sa + sb[q])), rm[c0 + q]);
          if constexpr (FP64) {
            // in units of the sixth weight (rounded there); the weights are integers below 2^25,
            // the leading two (top digits are at most 64) not above 2^22
            int i[NW];
#pragma unroll
            for (int w = 0; w < NW; ++w)
              i[w] = w < 2 ? __float_as_int(v[w][q] + 12582912.f) - 0x4B400000 : __float2int_rn(v[w][q]);
            const long long top = ((long long)i[0] << 40) + ((long long)i[1] << 32);
            const long long mid = ((long long)i[2] << 24) + ((long long)i[3] << 16);
            const int below = NW > 7 ? i[6] + ((i[NW - 1] + 128) >> 8) : i[6];
            sum[c0 + q] += chunk_value(top + mid + ((long long)i[4] << 8) + i[5] + ((below + 128) >> 8), ea + e[q]);
          } else {
            const float g = fa * pow2_neg(e[q]);
            // three leading weights by error-free sums, the rest in one float
            float s = hi[c0 + q], err = 0.f;
#pragma unroll
            for (int w = 0; w < 3; ++w) {
              const float t = v[w][q] * (g * (w == 0 ? 1.f : w == 1 ? 0x1p-8f : 0x1p-16f));
              const float n = __fadd_rn(s, t), b = __fsub_rn(n, s);
              err = __fadd_rn(err, __fadd_rn(__fsub_rn(s, __fsub_rn(n, b)), __fsub_rn(t, b)));
              s = n;
            }
            float tail = v[NW - 1][q];
#pragma unroll
            for (int w = NW - 2; w >= 3; --w) tail = fmaf(tail, 0x1p-8f, v[w][q]);
            const float l = __fadd_rn(lo[c0 + q], fmaf(tail, g * 0x1p-24f, err));
            const float n = __fadd_rn(s, l);
            lo[c0 + q] = __fsub_rn(l, __fsub_rn(n, s));
            hi[c0 + q] = n;
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) bar_arrive(acc_free);
    };
    auto produce = [&](int step, int q) {
      const int st = step % TSTAGES, t = warp + PWARPS * q;
      if (t >= nt) return;
      // core matrix (row group lane / 8, column group g) at ((lane / 8) groups + g) 128, 16 bytes per row
      uint8_t* base = t < na ? smem + st * STAGE + ((lane >> 3) * (TM / 8) + t) * 128
                             : smem + st * STAGE + TILES * A_TILE + ((lane >> 3) * (NT / 8) + t - na) * 128;
      store_task<R, ND, CHECK>(x[q], base + (lane & 7) * 16, t < na ? A_TILE : B_TILE);
    };
    start(0);
    start(1);
    fetch(0, 0);
    fetch(0, 1);
    for (int step = 0; step < nsteps; ++step) {
      const int st = step % TSTAGES;
      // the MMAs that read this stage (committed TSTAGES steps ago) are done
      if (step >= TSTAGES && !mma_wait(&empty[st], (uint32_t)((step / TSTAGES - 1) & 1))) lost = true;
      if (step > STEPS && step % STEPS == TSTAGES - 1) read_back(step / STEPS - 1);
      produce(step, 0);
      fetch(step + 1, 0);
      produce(step, 1);
      fetch(step + 1, 1);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) bar_arrive(&full[st]);
    }
    if (nsteps > 0) read_back(nsteps / STEPS - 1);
    const int i = i0 + row;
    if (i < i1) {
      const int er = ra[row];
      double* out = part + ((long long)blockIdx.z * 2 * A.cols + i) * Q2;
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const int j = j0 + jq + q;
        if (j >= j1) continue;
        const int e2 = rb[jq + q];
        const bool bad = lost || er >= 2047 || e2 >= 2047;  // infinities and NaN
        if (CHECK)
          room[((long long)blockIdx.z * 2 * A.cols + i) * Q2 + j] = bad ? 0.0 : times_pow2(widened(rm[q]), er + e2 - 2044);
        out[j] = bad ? (double)NAN : times_pow2(FP64 ? sum[q] : (double)hi[q] + (double)lo[q], product_unit<ND>(er, e2));
      }
    }
  }
  const bool any_lost = __syncthreads_or(lost) != 0;
  if (any_lost && warp != PWARPS && i0 + 32 * (warp & 3) + lane < i1) {  // a wait of another warp ran out
    double* out = part + ((long long)blockIdx.z * 2 * A.cols + i0 + 32 * (warp & 3) + lane) * Q2;
    for (int j = j0 + (warp >> 2) * NQ; j < min(j1, j0 + ((warp >> 2) + 1) * NQ); ++j) out[j] = (double)NAN;
    mma_wait(acc_full, (uint32_t)((nsteps / STEPS - 1) & 1));  // the MMAs may still run: wait, bounded
  }
  tc_fence_before();
  __syncthreads();
  if (warp == PWARPS) tmem_free(tmem, NCOLS);
}

// G[e] = sum over groups, in a fixed order: thread (x, y) of a 32 x 8 block
// sums groups y, y + 8, ... of output e (independent loads in flight), then
// the eight sums are added in order of y.  With CHECK, mask[e] says whether the
// room is below zero in all (a NaN has none to check), *any whether one is.
template <bool CHECK>
__global__ void __launch_bounds__(256) k_gram_digits_reduce(const double* __restrict__ part, int ngroups, int nout,
                                                        double* __restrict__ G, const double* __restrict__ room,
                                                        uint8_t* __restrict__ mask, int* any) {
  __shared__ double t[8][33], u[8][33];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + x;
  double s = 0.0, r = 0.0;
  if (e < nout)
#pragma unroll 4
    for (int c = y; c < ngroups; c += 8) {
      s += part[(long long)c * nout + e];
      if (CHECK) r += room[(long long)c * nout + e];
    }
  t[y][x] = s;
  if (CHECK) u[y][x] = r;
  __syncthreads();
  if (y == 0 && e < nout) {
    double g = t[0][x];
#pragma unroll
    for (int q = 1; q < 8; ++q) g += t[q][x];
    G[e] = g;
    if (CHECK) {
      for (int q = 1; q < 8; ++q) r += u[q][x];
      mask[e] = r < 0.0;
      if (r < 0.0) *any = 1;
    }
  }
}

struct Shape {
  int mt, nt, mw, nw, NT, nchunks, groups, cpg;
  size_t part_bytes, exp_bytes, sum_bytes;
  size_t bytes() const { return part_bytes * (sum_bytes ? 2 : 1) + exp_bytes + sum_bytes; }
};

// column tiles, row groups (one CTA per SM, fewer if the workspace holds
// fewer partial sums) and workspace of a Gram: partial sums (and their room),
// exponents (and sums of |x|)
template <int ND, bool CHECK = false>
Shape shape_of(int P, int Q, long long n, size_t ws_bytes = SIZE_MAX) {
  Shape s;
  const int P2 = 2 * P, Q2 = 2 * Q, cap = CHECK ? 48 : ND == 7 ? 64 : 128;   // (512 TMEM columns)
  s.mt = (P2 + TM - 1) / TM;
  s.nt = (Q2 + cap - 1) / cap;
  // tiles of equal width (the MMA takes 128 x NT columns whatever the tile holds)
  s.mw = padded8((P2 + s.mt - 1) / s.mt);
  s.nw = padded8((Q2 + s.nt - 1) / s.nt);
  s.NT = s.nw <= 16 ? 16 : s.nw <= 48 ? 48 : ND == 7 ? 64 : s.nw <= 80 ? 80 : 128;
  s.nchunks = (int)((n + CHUNK - 1) / CHUNK);
  // (16 bytes to spare for each array of partial sums, which the sizes below ask for)
  const size_t entries = (size_t)s.nchunks * (padded8(P2) + padded8(Q2));   // (a multiple of eight)
  s.exp_bytes = sizeof(short) * entries;
  s.sum_bytes = CHECK ? sizeof(float) * entries : 0;
  const size_t per = sizeof(double) * (size_t)P2 * Q2 * (CHECK ? 2 : 1), rest = s.exp_bytes + s.sum_bytes + (CHECK ? 32 : 16);
  const size_t fit = ws_bytes > rest ? (ws_bytes - rest) / per : 0;
  const int want = (int)std::max<size_t>(1, std::min<size_t>(152 / (s.mt * s.nt), fit));
  s.cpg = (s.nchunks + want - 1) / want;
  s.groups = (s.nchunks + s.cpg - 1) / s.cpg;
  s.part_bytes = (sizeof(double) * (size_t)s.groups * P2 * Q2 + 15) / 16 * 16;
  return s;
}

// where a checked Gram leaves its verdict
struct Verdict {
  uint8_t* mask;
  int* any;
};

template <typename R, int ND, int NT, bool CHECK>
cudaError_t launch(const PairBlock<R>& A, const PairBlock<R>& B, const Shape& h, void* ws, const Verdict& c, cudaStream_t s) {
  constexpr int TSTAGES = stages<ND>();
  const size_t smem = (size_t)TSTAGES * (ND + CHECK) * (TM + NT) * TBK * 2 + 8 * (2 * TSTAGES + 2) + 8 + sizeof(int) * (TM + NT);
  cudaError_t e = allow_dynamic_smem((const void*)k_gram_digits<R, ND, NT, CHECK>, smem);
  if (e != cudaSuccess) return e;
  const int lda = padded8(2 * A.cols), ldb = padded8(2 * B.cols);
  char* p = (char*)ws + h.part_bytes;
  double* room = CHECK ? (double*)p : nullptr;
  if (CHECK) p += h.part_bytes;
  short* ea = (short*)p;
  float* sa = CHECK ? (float*)(p + h.exp_bytes) : nullptr;
  const size_t b0 = (size_t)h.nchunks * lda;   // where B's entries begin
  k_gram_digits<R, ND, NT, CHECK><<<dim3(h.mt, h.nt, h.groups), TTHREADS, smem, s>>>(
      A, B, ea, ea + b0, lda, ldb, h.mw, h.nw, h.nchunks, h.cpg, (double*)ws, sa, CHECK ? sa + b0 : nullptr, room, c.any);
  return cudaGetLastError();
}

template <typename R, int ND, bool CHECK = false>
cudaError_t gram_digits(const PairBlock<R>& A, const PairBlock<R>& B, double* G_dev, void* ws, size_t ws_bytes,
                        cudaStream_t s, const Verdict& c = Verdict{nullptr, nullptr}) {
  if (A.n != B.n) return cudaErrorInvalidValue;
  const int P2 = 2 * A.cols, Q2 = 2 * B.cols;
  if (P2 == 0 || Q2 == 0) return cudaSuccess;
  if (A.n == 0) return cudaMemsetAsync(G_dev, 0, sizeof(double) * P2 * Q2, s);
  const Shape h = shape_of<ND, CHECK>(A.cols, B.cols, A.n, ws_bytes);
  if (ws_bytes < h.bytes()) return cudaErrorInvalidValue;
  const int lda = padded8(P2), ldb = padded8(Q2);
  const size_t b0 = (size_t)h.nchunks * lda;
  short* ea = (short*)((char*)ws + h.part_bytes * (CHECK ? 2 : 1));
  float* sa = CHECK ? (float*)((char*)ea + h.exp_bytes) : nullptr;
  k_col_exp<R, CHECK><<<(unsigned)(((long long)h.nchunks * (lda / 2) + 7) / 8), 256, 0, s>>>(A, h.nchunks, lda, ea, sa);
  k_col_exp<R, CHECK><<<(unsigned)(((long long)h.nchunks * (ldb / 2) + 7) / 8), 256, 0, s>>>(B, h.nchunks, ldb, ea + b0,
                                                                                              CHECK ? sa + b0 : nullptr);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (h.NT == 16) e = launch<R, ND, 16, CHECK>(A, B, h, ws, c, s);
  else if (h.NT == 48) e = launch<R, ND, 48, CHECK>(A, B, h, ws, c, s);
  else if constexpr (ND == 7 && !CHECK) e = launch<R, ND, 64, CHECK>(A, B, h, ws, c, s);
  else if constexpr (ND == 4) e = h.NT == 80 ? launch<R, ND, 80, CHECK>(A, B, h, ws, c, s) : launch<R, ND, 128, CHECK>(A, B, h, ws, c, s);
  if (e != cudaSuccess) return e;
  const int nout = P2 * Q2;
  k_gram_digits_reduce<CHECK><<<(nout + 31) / 32, 256, 0, s>>>((const double*)ws, h.groups, nout, G_dev,
                                                              (const double*)((const char*)ws + h.part_bytes), c.mask, c.any);
  return cudaGetLastError();
}

}  // namespace

size_t gram_digits_workspace_bytes(int P, int Q, long long n) {
  if (P <= 0 || Q <= 0 || n <= 0) return 0;
  return 16 + std::max(shape_of<4>(P, Q, n).bytes(), shape_of<7>(P, Q, n).bytes());
}

bool gram_digits_fits(int P, int Q, long long n, size_t ws_bytes) {
  return std::max(shape_of<4>(P, Q, n, ws_bytes).bytes(), shape_of<7>(P, Q, n, ws_bytes).bytes()) <= ws_bytes;
}

template <typename R>
cudaError_t gram_pairs_digits(const PairBlock<R>& A, const PairBlock<R>& B, int digits, double* G_dev, void* ws,
                              size_t ws_bytes, cudaStream_t s) {
  if constexpr (sizeof(R) == 8)
    if (digits > 4) return gram_digits<R, 7>(A, B, G_dev, ws, ws_bytes, s);
  return gram_digits<R, 4>(A, B, G_dev, ws, ws_bytes, s);
}

size_t gram_digits_checked_bytes(int P, int Q, long long n) { return 32 + shape_of<7, true>(P, Q, n).bytes(); }

cudaError_t gram_digits_checked(const PairBlock<double>& A, const PairBlock<double>& B, double* G_dev, void* ws,
                                size_t ws_bytes, uint8_t* mask, int* any, cudaStream_t s) {
  return gram_digits<double, 7, true>(A, B, G_dev, ws, ws_bytes, s, Verdict{mask, any});
}

template cudaError_t gram_pairs_digits<float>(const PairBlock<float>&, const PairBlock<float>&, int, double*, void*,
                                              size_t, cudaStream_t);
template cudaError_t gram_pairs_digits<double>(const PairBlock<double>&, const PairBlock<double>&, int, double*,
                                               void*, size_t, cudaStream_t);

}  // namespace bdg
