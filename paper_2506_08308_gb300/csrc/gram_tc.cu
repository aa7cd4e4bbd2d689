// Tall-skinny Gram G = A^T B of two pair blocks on the tensor cores
// (tcgen05.mma, accumulator in tensor memory).
//
// Every operand element x is split into three BF16 slices, x = x0 + x1 + x2
// (x0 the BF16 rounding of x, x1 of what x0 leaves, x2 of the rest), which
// holds x to about 2^-24.  Of the nine slice products the six whose weight
// reaches 2^-24 of the leading one are accumulated in FP32 by the MMA:
// x0 y0, x0 y1, x1 y0, x1 y1, x0 y2, x2 y0.  Each CTA sums a chunk of rows
// this way and writes its FP32 tile as FP64 partial sums; the chunks are
// summed in FP64.  The result has FP32 accuracy: about 1e-6 to 1e-5 of sum
// |a_k b_k|, most of it the truncation of the tensor cores' FP32 sums.  (The
// solver's Grams of this accuracy come from digits, gram_digits.cu.)
//
// What bounds it: one CTA used to load, split and multiply each 32-row stage
// in turn, and waited out a memory latency per stage (48 x 48 columns of
// 196608 FP64 rows: 288 us, 0.5 TB/s).  Eight or sixteen warps now load
// and split, two tasks ahead of their use, into a ring of stages, and one
// more issues the MMAs; the arithmetic and its order are unchanged, bit for bit,
// and the calls below went from 304 to 90 us (24 x 24 pairs, C128, 196608
// rows), 194 to 70 (C64), 559 to 363 (72 x 72, C128).  The row chunks, whose
// number the workspace gives, leave 96 CTAs there: the integer work of cutting
// FP64 values on those 96 SMs is what bounds it now.
//
// Layout of one pipeline stage in shared memory: for A (128 real columns)
// and B (NT real columns) three BF16 slice tiles of TBK = 32 rows each, MN-
// major without swizzle: a core matrix holds 8 rows of 8 neighbouring real
// columns (16 bytes a row), core matrix (k8, c8) at byte offset (k8 (cols / 8)
// + c8) 128.  A warp's task is four complex columns at 32 rows, one row a
// lane: 512-byte loads, 16-byte stores, no bank conflicts.  One MMA step
// covers 16 rows (two core matrices along K).
#include <cuda_bf16.h>

#include <algorithm>

#include "blas.cuh"
#include "digits.cuh"

namespace bdg {

namespace {

constexpr int TM = 128;          // A real columns per CTA (MMA M)
constexpr int TBK = 32;          // rows per pipeline stage (two MMA K steps of 16)
constexpr int TNMAX = 160;       // widest B tile (real columns, multiple of 16)
constexpr int NSLICE = 3;
constexpr int A_SLICE_BYTES = TM * TBK * 2;
// stages in flight, as many as the CTAs of an SM (two with eight producer
// warps, one with sixteen) have room for
__host__ __device__ constexpr int stages_of(int NT, int pwarps) { return (NT <= 48 ? 3 : 2) * (pwarps > 8 ? 2 : 1); }

// instruction descriptor of kind::f16: D FP32, A and B BF16, both MN-major
__device__ __forceinline__ uint32_t idesc_bf16(int M, int N) {
  return mma_idesc_f16(M, N, true, true) | (1u << 7) | (1u << 10);
}

// FP64 x cut to FP32 by its bits (24 significant bits, truncated; below the
// FP32 normal range 0, above it infinity, NaN kept): no FP64 arithmetic,
// which runs at a small fraction of the FP32 rate on this part.
__device__ __forceinline__ float cut_to_float(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned sign = hi & 0x80000000u, mag = hi & 0x7FFFFFFFu;
  if (mag - (897u << 20) < (254u << 20))  // exponents 897 .. 1150: the FP32 normal range
    return __uint_as_float((__funnelshift_l(lo, hi, 3) - (384u << 23)) | sign);  // (896 mod 512) off the 9 bits kept
  if (mag < (897u << 20)) return __uint_as_float(sign);
  const bool nan = (mag >> 20) == 0x7FFu && __funnelshift_l(lo, hi, 3) & 0x7FFFFFu;
  return __uint_as_float(sign | 0x7F800000u | (nan ? 0x400000u : 0u));
}
__device__ __forceinline__ float cut_to_float(float x) { return x; }

// the three BF16 slices of two values, packed (first value in the low half)
__device__ __forceinline__ void split3(float x, float y, uint32_t (&w)[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
    w[k] = *reinterpret_cast<const uint32_t*>(&h);
    if (k < 2) {
      x -= __uint_as_float(w[k] << 16);
      y -= __uint_as_float(w[k] & 0xFFFF0000u);
    }
  }
}

// Four complex columns of a block at one row (zero past the end).
template <typename R>
struct RowTask {
  typename CT<R>::T v[4];
};
template <typename R>
__device__ __forceinline__ void load_task(const PairBlock<R>& X, int c0, long long r, long long r_end, RowTask<R>& o) {
  const typename CT<R>::T* p = X.p + (long long)c0 * X.ld + r;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    o.v[q] = mk((R)0, (R)0);
    if (r < r_end && c0 + q < X.cols) o.v[q] = p[q * X.ld];
  }
}
// slices of eight real columns at one row: 16 bytes per slice tile
template <typename R>
__device__ __forceinline__ void store_task(const RowTask<R>& x, uint8_t* base, uint32_t slice_bytes) {
  uint32_t w[4][NSLICE];
#pragma unroll
  for (int q = 0; q < 4; ++q) split3(cut_to_float(x.v[q].x), cut_to_float(x.v[q].y), w[q]);
#pragma unroll
  for (int s = 0; s < NSLICE; ++s) *reinterpret_cast<uint4*>(base + s * slice_bytes) = make_uint4(w[0][s], w[1][s], w[2][s], w[3][s]);
}

// Partial Gram of one row chunk: part[chunk][i][j] for real columns
// i < 2 A.cols (128 per CTA along x), j < 2 B.cols <= NT.  A wait that runs
// out writes NaN into the tile (the caller sees a NaN Gram).
template <typename R, int PWARPS>
__global__ void __launch_bounds__(32 * (PWARPS + 1), PWARPS > 8 ? 1 : 2)
    k_gram_tc(PairBlock<R> A, PairBlock<R> B, int NT, long long crows, double* __restrict__ part) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int nstage = stages_of(NT, PWARPS);
  const uint32_t b_slice = (uint32_t)NT * TBK * 2;
  const uint32_t stage_bytes = NSLICE * (A_SLICE_BYTES + b_slice);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + nstage * stage_bytes);
  uint64_t* empty = full + nstage;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(empty + nstage);
  const uint32_t ncols = NT <= 32 ? 32u : NT <= 64 ? 64u : NT <= 128 ? 128u : 256u;
  const int i0 = blockIdx.x * TM;
  const long long r_begin = (long long)blockIdx.z * crows;
  const long long r_end = min(A.n, r_begin + crows);
  const int P2 = 2 * A.cols, Q2 = 2 * B.cols;

  if (warp == PWARPS) tmem_alloc(tmem_slot, ncols);
  if (tid == 0) {
    for (int s = 0; s < nstage; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&full[s])), "r"(PWARPS) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[s])) : "memory");
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  const int nsteps = r_end > r_begin ? (int)((r_end - r_begin + TBK - 1) / TBK) : 0;
  bool lost = false;
  if (warp == PWARPS) {
    const uint32_t idesc = idesc_bf16(TM, NT);
    const uint32_t lbo_a = (TM / 8) * 128, lbo_b = (uint32_t)(NT / 8) * 128;
    const bool leader = elect_one();
    int st = 0, ph = 0;
    for (int step = 0; step < nsteps; ++step) {
      if (!mma_wait(&full[st], (uint32_t)ph)) lost = true;
      tc_fence_after();
      if (leader) {
        const uint32_t sa = smem_u32(smem + st * stage_bytes), sb = sa + NSLICE * A_SLICE_BYTES;
        // slice pairs (A slice, B slice) whose weight reaches 2^-24 of the leading one
        const int pa[6] = {0, 0, 1, 1, 0, 2}, pb[6] = {0, 1, 0, 1, 2, 0};
#pragma unroll
        for (int p = 0; p < 6; ++p)
#pragma unroll
          for (int kk = 0; kk < 2; ++kk)
            mma_f16(tmem, mma_desc(sa + pa[p] * A_SLICE_BYTES + 2 * kk * lbo_a, lbo_a, 128),
                    mma_desc(sb + pb[p] * b_slice + 2 * kk * lbo_b, lbo_b, 128), idesc, step > 0 || p > 0 || kk > 0);
        mma_commit(&empty[st]);
      }
      __syncwarp();
      if (++st == nstage) { st = 0; ph ^= 1; }
    }
  } else {
    // tasks of a stage: groups of four complex columns of A, then of B; this
    // warp takes every PWARPS-th.  Rows of A's tile past the block's columns are
    // never written: they only reach rows of the result that nothing reads.
    const int na = (min(TM, P2 - i0) + 7) / 8, nt = na + (Q2 + 7) / 8;
    const int per = (nt + PWARPS - 1) / PWARPS;
    // items (step, q) in order, loads two items ahead
    int fs = 0, fq = 0;
    auto fetch = [&](RowTask<R>& x) {
      const int t = warp + PWARPS * fq;
      const long long r = r_begin + (long long)fs * TBK + lane;
      if (fs < nsteps) {
        if (t < na) load_task<R>(A, i0 / 2 + 4 * t, r, r_end, x);
        else if (t < nt) load_task<R>(B, 4 * (t - na), r, r_end, x);
      }
      if (++fq == per) { fq = 0; ++fs; }
    };
    int step = 0, q = 0, st = 0, ph = 1;   // (a fresh barrier's other phase counts as complete)
    auto produce = [&](RowTask<R>& x) {
      if (step >= nsteps) return;
      // the MMAs that read this stage nstage steps ago are done
      if (q == 0 && !mma_wait(&empty[st], (uint32_t)ph)) lost = true;
      const int t = warp + PWARPS * q;
      if (t < nt) {
        uint8_t* base = t < na ? smem + st * stage_bytes + ((lane >> 3) * (TM / 8) + t) * 128
                               : smem + st * stage_bytes + NSLICE * A_SLICE_BYTES + ((lane >> 3) * (NT / 8) + t - na) * 128;
        store_task<R>(x, base + (lane & 7) * 16, t < na ? (uint32_t)A_SLICE_BYTES : b_slice);
      }
      fetch(x);
      if (++q == per) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&full[st])) : "memory");
        q = 0;
        ++step;
        if (++st == nstage) { st = 0; ph ^= 1; }
      }
    };
    RowTask<R> x0, x1;
    fetch(x0);
    fetch(x1);
    for (int item = 0; item < nsteps * per; item += 2) {
      produce(x0);
      produce(x1);
    }
  }
  const int last = nsteps - 1;
  if (nsteps > 0 && !mma_wait(&empty[last % nstage], (uint32_t)((last / nstage) & 1))) lost = true;
  lost = __syncthreads_or(lost) != 0;
  tc_fence_after();
  if (warp < PWARPS) {
    const int quarter = warp & 3;  // a warp reads TMEM lanes 32 quarter .. 32 quarter + 31
    const int i = i0 + 32 * quarter + lane;
    double* out = part + (long long)blockIdx.z * P2 * Q2;
    for (int jc = (warp >> 2) * 4; jc < NT; jc += PWARPS) {
      float v[4] = {0.f, 0.f, 0.f, 0.f};
      if (nsteps > 0) {
        tmem_ld4(tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)jc, v);
        tmem_ld_wait();
      }
      if (i < P2) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (jc + q < Q2) out[(long long)i * Q2 + jc + q] = lost ? (double)NAN : (double)v[q];
      }
    }
  }
  if (lost && nsteps > 0) {
    // the MMAs may still run: wait (bounded) for the last commit before freeing their accumulator
    mma_wait(&empty[last % nstage], (uint32_t)((last / nstage) & 1));
  }
  tc_fence_before();
  __syncthreads();
  if (warp == PWARPS) tmem_free(tmem, ncols);
}

// G[e] = sum over chunks, in a fixed order: thread (x, y) of a 32 x 8 block
// sums chunks y, y + 8, ... of output e (independent loads in flight), then
// the eight sums are added in order of y.
__global__ void __launch_bounds__(256) k_gram_tc_reduce(const double* __restrict__ part, int nchunks, int nout,
                                                        double* __restrict__ G) {
  __shared__ double t[8][33];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + x;
  double s = 0.0;
  if (e < nout)
#pragma unroll 4
    for (int c = y; c < nchunks; c += 8) s += part[(long long)c * nout + e];
  t[y][x] = s;
  __syncthreads();
  if (y == 0 && e < nout) {
    double g = t[0][x];
#pragma unroll
    for (int q = 1; q < 8; ++q) g += t[q][x];
    G[e] = g;
  }
}

size_t tc_smem_bytes(int NT, int pwarps) {
  const int n = stages_of(NT, pwarps);
  return (size_t)n * NSLICE * (A_SLICE_BYTES + (size_t)NT * TBK * 2) + 16 * n + 16;
}

}  // namespace

bool gram_tc_supported(int P, int Q) { return P > 0 && Q > 0 && 2 * Q <= TNMAX; }

template <typename R>
cudaError_t gram_pairs_tc(const PairBlock<R>& A, const PairBlock<R>& B, double* G_dev, void* ws,
                          size_t ws_bytes, cudaStream_t s) {
  if (A.n != B.n) return cudaErrorInvalidValue;
  const int P2 = 2 * A.cols, Q2 = 2 * B.cols;
  if (P2 == 0 || Q2 == 0) return cudaSuccess;
  if (!gram_tc_supported(A.cols, B.cols)) return cudaErrorNotSupported;
  if (A.n == 0) return cudaMemsetAsync(G_dev, 0, sizeof(double) * P2 * Q2, s);
  const int NT = (Q2 + 15) / 16 * 16;
  const int mtiles = (P2 + TM - 1) / TM;
  const size_t per_chunk = sizeof(double) * (size_t)P2 * Q2;
  const long long cap = (long long)(ws_bytes / per_chunk);
  if (cap < 1) return cudaErrorInvalidValue;
  // two CTAs per SM (each holds two or three stages and 32 ... 256 TMEM columns)
  long long nch = std::min<long long>((2 * 152 + mtiles - 1) / mtiles, cap);
  nch = std::min<long long>(nch, (A.n + TBK - 1) / TBK);
  const long long crows = ((A.n + nch - 1) / nch + TBK - 1) / TBK * TBK;
  nch = (A.n + crows - 1) / crows;
  // few row chunks leave an SM with one CTA: then sixteen producer warps
  const bool wide = nch * mtiles <= 152;
  const size_t smem = tc_smem_bytes(NT, wide ? 16 : 8);
  auto kern = wide ? k_gram_tc<R, 16> : k_gram_tc<R, 8>;
  cudaError_t e = allow_dynamic_smem((const void*)kern, smem);
  if (e != cudaSuccess) return e;
  kern<<<dim3((unsigned)mtiles, 1, (unsigned)nch), 32 * (wide ? 17 : 9), smem, s>>>(A, B, NT, crows, (double*)ws);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const int nout = P2 * Q2;
  k_gram_tc_reduce<<<(nout + 31) / 32, 256, 0, s>>>((const double*)ws, (int)nch, nout, G_dev);
  return cudaGetLastError();
}

template cudaError_t gram_pairs_tc<float>(const PairBlock<float>&, const PairBlock<float>&, double*, void*, size_t,
                                          cudaStream_t);
template cudaError_t gram_pairs_tc<double>(const PairBlock<double>&, const PairBlock<double>&, double*, void*,
                                           size_t, cudaStream_t);

}  // namespace bdg
