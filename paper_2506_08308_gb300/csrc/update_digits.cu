// FP64 block update Y = beta Y + alpha A C (tall A, small C) from exact integer
// digits on the tensor cores (digits.cuh).
//
// A tile is 128 rows.  Every row is written in fixed point against its own
// largest value over all columns, every column of C against its own (prepared
// once per call by k_update_table); seven 8-bit digits each, the eight leading
// digit weights (34 products) summed by tcgen05.mma over up to 160 real
// columns, put together in 64-bit integers and scaled by the two exponents.
// The error is that of cutting A's rows and C's columns at 2^-55 of their
// largest values, against 2^-48 per term in double-float (k_update_df, which
// spends 15 FP32 instructions on a multiply-add and is bound by them).
//
// Measured at 196608 rows (a 256^2 grid), pairs in -> out, double-float ->
// digits: 24 -> 24 323 -> 135 us, 48 -> 24 612 -> 200, 73 -> 24 874 -> 221,
// 72 -> 26 1138 -> 283, 16 -> 24 249 -> 143, 24 -> 8 127 -> 97; relative error
// (Frobenius, against extended precision) 6e-15..1e-14 -> 3e-16..4e-16.  73 -> 24
// moves 384 MB, 57 us at the copy rate.  What is left is the cutting of the
// digits (two fixed-point values and 14 halves per complex element) and the
// epilogue, which do not overlap: the accumulators take all of the TMEM columns
// at the widest outputs.
//
// Sixteen warps: a thread holds one row of every fourth group of four complex
// columns in registers, so that A is read once; the digits of 32 real columns
// at a time go to a ring of two stages (A operand, K-major: a core matrix is
// 8 rows of 16 bytes, which neighbouring lanes fill), C's digits follow from
// L2.  One warp issues the MMAs of a stage while the others cut the next.
#include <algorithm>

#include "blas.cuh"
#include "digits.cuh"

namespace bdg {

namespace {

constexpr int ND = 7, NW = 8;
constexpr int ROWS = 128, KC = 32;          // rows of a tile, real columns of a stage
constexpr int KMAX = 160;                   // real columns of A
constexpr int GROUPS = KMAX / KC;           // groups of four complex columns a thread holds
constexpr int A_DIGIT = ROWS * KC * 2, A_STAGE = ND * A_DIGIT;
constexpr int THREADS = 512;

// C's digits per stage: [digit][k group of 8][column group of 8][k][column]
template <int N> constexpr int c_digit() { return N * KC * 2; }

// One CTA per output column: exponent and digits of alpha C[:, j].
__global__ void __launch_bounds__(KMAX) k_update_table(const double* __restrict__ C, int ldc, int K, int kpad, int Q2,
                                                       int N, double alpha, __half* __restrict__ out,
                                                       short* __restrict__ exps) {
  __shared__ int emax;
  const int j = blockIdx.x, k = threadIdx.x;
  if (k == 0) emax = 0;
  __syncthreads();
  const double v = j < Q2 && k < K ? alpha * C[(long long)k * ldc + j] : 0.0;
  // (a subnormal coefficient counts as zero, and a zero as no value: no TINY case)
  const int ev = (__double2hiint(v) >> 20) & 0x7FF;
  atomicMax(&emax, ev);
  __syncthreads();
  if (k == 0) exps[j] = (short)emax;
  if (k >= kpad) return;
  const long long X = ev > 0 ? to_fixed<ND>(v, emax << 20) : 0;
  const unsigned long long u = (unsigned long long)X + 0x80808080808080ull;
  const int st = k / KC, k8 = k % KC / 8;
  __half* o = out + (size_t)st * ND * N * KC + (k8 * (N / 8) + j / 8) * 64 + (k % 8) * 8 + j % 8;
#pragma unroll
  for (int d = 0; d < ND; ++d)
    o[d * N * KC] = __int2half_rn((int)(d == 0 ? u >> 48 : (u >> (8 * (ND - 1 - d))) & 0xFF) - 128);
}

// sums of the eight weights in units of the sixth (rounded there).  All but the
// seventh are integers below 2^24 whatever the digits (160 terms x up to 6 pairs x
// 2^14); the seventh (7 pairs) may pass it from 147 real columns on and then be
// off by a unit, 2^-62 of the two largest values' product.
__device__ __forceinline__ long long weigh(const float (&c)[NW]) {
  int i[NW];
#pragma unroll
  for (int k = 0; k < NW; ++k) i[k] = __float2int_rn(c[k]);
  const long long hi = ((long long)i[0] << 40) + ((long long)i[1] << 32);
  const long long mid = ((long long)i[2] << 24) + ((long long)i[3] << 16);
  const long long low = ((long long)i[4] << 8) + i[5];
  return hi + mid + low + ((i[6] + ((i[7] + 128) >> 8) + 128) >> 8);
}

// v 2^e as a double, rounded to nearest, without the FP64 pipe where the
// result is a normal number
__device__ __forceinline__ double scaled(long long v, int e) {
  const int s = (int)(v >> 63);
  const unsigned long long m = (unsigned long long)((v ^ (long long)s) - (long long)s);
  if (m == 0) return 0.0;
  const int lz = __clzll((long long)m);
  const unsigned long long n = (m << lz) + 0x400;
  int field = 1085 - lz + e;                                     // (the leading bit adds one)
  unsigned long long frac = n >> 11;
  if (n < 0x400ull) {                                            // a carry out of bit 63
    frac = 0;
    field += 2;
  }
  if (field < 1 || field > 2040) return scalbn((double)v, e);
  return __longlong_as_double((long long)((((unsigned long long)(unsigned)field << 52) + frac) | ((unsigned long long)(unsigned)s << 63)));
}

template <int N>
__global__ void __launch_bounds__(THREADS, 1)
    k_update_digits(PairBlock<double> A, const uint8_t* __restrict__ table, const short* __restrict__ ec, int nst,
                    double beta, double2* __restrict__ Y, long long ldy, int Q, long long ntiles) {
  constexpr int C_STAGE = ND * c_digit<N>();
  constexpr uint32_t NCOLS = NW * N <= 128 ? 128 : NW * N <= 256 ? 256 : 512;
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t* cs = smem + 2 * A_STAGE;
  uint64_t* full = reinterpret_cast<uint64_t*>(cs + 2 * C_STAGE);  // C's digits of a stage are there
  uint64_t* empty = full + 2;                                      // the MMAs of a stage are done
  uint64_t* done = empty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  int* bad = reinterpret_cast<int*>(tmem_slot + 1);
  unsigned* er = reinterpret_cast<unsigned*>(bad + 1);             // [ROWS] largest magnitudes
  int* ecs = reinterpret_cast<int*>(er + ROWS);                                            // [N]
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  if (warp == 0) tmem_alloc(tmem_slot, NCOLS);
  if (tid == 0) {
    *bad = 0;
    for (int s = 0; s < 2; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&full[s])) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[s])) : "memory");
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(done)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int j = tid; j < N; j += THREADS) ecs[j] = ec[j];
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t idesc = mma_idesc_f16(ROWS, N, false, true);   // A K-major, C MN-major
  bool lost = false;
  unsigned at = 0, tiles = 0;   // stages and tiles so far

  const int row = tid & (ROWS - 1), qd = tid >> 7;   // this thread's groups: complex columns 16 s + 4 qd ..
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++tiles) {
    const long long r = tile * ROWS + row;
    const bool in = r < A.n;
    double2 v[GROUPS][4];
    unsigned m = 0;
#pragma unroll
    for (int s = 0; s < GROUPS; ++s)
#pragma unroll
      for (int l = 0; l < 4; ++l) {
        const int c = 16 * s + 4 * qd + l;
        v[s][l] = make_double2(0.0, 0.0);
        if (in && c < A.cols) v[s][l] = A.p[(long long)c * A.ld + r];
      }
    if (tid < ROWS) er[tid] = 0;
    __syncthreads();
#pragma unroll
    for (int s = 0; s < GROUPS; ++s)
#pragma unroll
      for (int l = 0; l < 4; ++l) m = max(m, max(magnitude(v[s][l].x), magnitude(v[s][l].y)));
    atomicMax(&er[row], m);
    __syncthreads();
    int e20 = (int)er[row];
    if (is_tiny<double>(e20)) {
      e20 = (biased_exponent<double>(e20) + Tiny<double>::GROW) << 20;
#pragma unroll
      for (int s = 0; s < GROUPS; ++s)
#pragma unroll
        for (int l = 0; l < 4; ++l) {
          v[s][l].x *= Tiny<double>::FACTOR;
          v[s][l].y *= Tiny<double>::FACTOR;
        }
    }
#pragma unroll
    for (int s = 0; s < GROUPS; ++s) {
      if (s >= nst) break;
      const unsigned st = at & 1;
      // the MMAs that read this stage two stages ago are done (a fresh barrier's other phase counts as complete)
      if (!mma_wait(&empty[st], ((at >> 1) & 1) ^ 1)) lost = true;
      if (warp == 1 && elect_one()) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&full[st])), "r"(C_STAGE) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         smem_u32(cs + st * C_STAGE)),
                     "l"(table + (size_t)s * C_STAGE), "r"(C_STAGE), "r"(smem_u32(&full[st]))
                     : "memory");
      }
      __syncwarp();
      uint32_t d[4][ND];
#pragma unroll
      for (int l = 0; l < 4; ++l) digit_pairs<ND>(to_fixed<ND>(v[s][l].x, e20), to_fixed<ND>(v[s][l].y, e20), d[l]);
      // core matrix (row group, k group qd): [k group][row group] of 128 bytes
      uint8_t* o = smem + st * A_STAGE + (qd * (ROWS / 8) + row / 8) * 128 + (row % 8) * 16;
#pragma unroll
      for (int k = 0; k < ND; ++k) *reinterpret_cast<uint4*>(o + k * A_DIGIT) = make_uint4(d[0][k], d[1][k], d[2][k], d[3][k]);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncthreads();
      if (warp == 0) {
        if (!mma_wait(&full[st], (at >> 1) & 1)) lost = true;
        tc_fence_after();
        if (elect_one()) {
          const uint64_t da = mma_desc(smem_u32(smem + st * A_STAGE), ROWS / 8 * 128, 128);
          const uint64_t dc = mma_desc(smem_u32(cs + st * C_STAGE), N / 8 * 128, 128);
#pragma unroll
          for (int kk = 0; kk < 2; ++kk)
#pragma unroll
            for (int i = 0; i < ND; ++i)
#pragma unroll
              for (int j = 0; j < ND && i + j < NW; ++j)
                mma_f16(tmem + (uint32_t)((i + j) * N), da + ((i * A_DIGIT + kk * 2 * (ROWS / 8) * 128) >> 4),
                        dc + ((j * c_digit<N>() + kk * 2 * (N / 8) * 128) >> 4), idesc,
                        !(s == 0 && kk == 0 && (i == 0 || (i == 1 && j == ND - 1))));
          mma_commit(&empty[st]);
          if (s == nst - 1) mma_commit(done);
        }
        __syncwarp();
      }
      ++at;
    }
    if (!mma_wait(done, tiles & 1)) lost = true;
    tc_fence_after();
    // rows 32 quarter + lane, N / 4 columns a warp
    constexpr int NQ = N / 4;
    const int quarter = warp & 3, jq = (warp >> 2) * NQ, orow = 32 * quarter + lane;
    const long long ro = tile * ROWS + orow;
    const int eo = biased_exponent<double>(er[orow]);
    if (lost) *bad = 1;
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NQ; c += 4) {
      float w[NW][4];
#pragma unroll
      for (int k = 0; k < NW; ++k) tmem_ld4(tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(k * N + jq + c), w[k]);
      tmem_ld_wait();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = jq + c + 2 * h, q = j / 2;
        if (q >= Q || ro >= A.n) continue;
        double z[2];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          const float cc[NW] = {w[0][2 * h + p], w[1][2 * h + p], w[2][2 * h + p], w[3][2 * h + p],
                                w[4][2 * h + p], w[5][2 * h + p], w[6][2 * h + p], w[7][2 * h + p]};
          const int e2 = ecs[j + p];
          z[p] = eo >= 2047 || e2 >= 2047 || *bad ? (double)NAN
                 : eo == 0 || e2 == 0             ? 0.0
                                                  : scaled(weigh(cc), eo + e2 - 2 * 1077 + 56);
        }
        double2* yp = Y + (long long)q * ldy + ro;
        if (beta != 0.0) {
          const double2 y = *yp;
          z[0] = fma(beta, y.x, z[0]);
          z[1] = fma(beta, y.y, z[1]);
        }
        *yp = make_double2(z[0], z[1]);
      }
    }
    tc_fence_before();
    __syncthreads();   // accumulators, exponents
    tc_fence_after();
  }
  if (__syncthreads_or(lost) && tiles > 0) {   // MMAs or a load may still run: wait once more, bounded
    mma_wait(done, (tiles - 1) & 1);
    for (unsigned s = 0; s < 2; ++s)
      if (at > s) mma_wait(&full[(at - 1 - s) & 1], ((at - 1 - s) >> 1) & 1);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_free(tmem, NCOLS);
}

template <int N>
cudaError_t launch(const PairBlock<double>& A, const uint8_t* table, const short* ec, int nst, double beta, double2* Y,
                   long long ldy, int Q, cudaStream_t s) {
  const size_t smem = 2 * (size_t)A_STAGE + 2 * (size_t)ND * c_digit<N>() + 8 * 5 + 8 + 4 * (ROWS + N);
  cudaError_t e = allow_dynamic_smem((const void*)k_update_digits<N>, smem);
  if (e != cudaSuccess) return e;
  const long long ntiles = (A.n + ROWS - 1) / ROWS;
  k_update_digits<N><<<(unsigned)std::min<long long>(ntiles, 152), THREADS, smem, s>>>(A, table, ec, nst, beta, Y, ldy, Q, ntiles);
  return cudaGetLastError();
}

}  // namespace

size_t update_digits_workspace_bytes() { return (size_t)ND * KMAX * 64 * 2 + 64 * sizeof(short); }

// Few rows leave most SMs without a tile, where both ways cost the same launch
// and table time: 8 -> 4 pairs take 15.3 us in double-float and 14.7 here at
// 8192 rows.  Narrower blocks than that are bound by reading A in either way and
// stay with the kernel that needs no table.
bool update_digits_pays(int P, int Q, long long n) {
  return 2 * P <= KMAX && 2 * Q <= 64 && P >= 8 && Q >= 4 && n >= 8192;
}

cudaError_t update_pairs_digits(const PairBlock<double>& A, const double* C_dev, int ldc, double beta, double2* Y,
                                long long ldy, int Q, void* ws, cudaStream_t s, double alpha) {
  const int K = 2 * A.cols, Q2 = 2 * Q, nst = (K + KC - 1) / KC, N = Q2 <= 16 ? 16 : Q2 <= 32 ? 32 : Q2 <= 48 ? 48 : 64;
  if (K > KMAX || Q2 > 64 || K == 0 || Q == 0) return cudaErrorInvalidValue;
  __half* table = (__half*)ws;
  short* ec = (short*)((char*)ws + (size_t)ND * KMAX * 64 * 2);
  k_update_table<<<N, KMAX, 0, s>>>(C_dev, ldc, K, nst * KC, Q2, N, alpha, table, ec);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const uint8_t* t = (const uint8_t*)table;
  if (N == 16) return launch<16>(A, t, ec, nst, beta, Y, ldy, Q, s);
  if (N == 32) return launch<32>(A, t, ec, nst, beta, Y, ldy, Q, s);
  if (N == 48) return launch<48>(A, t, ec, nst, beta, Y, ldy, Q, s);
  return launch<64>(A, t, ec, nst, beta, Y, ldy, Q, s);
}

}  // namespace bdg
