// FP32 parallel cyclic Jacobi for the small symmetric eigenproblems of the
// Gram-Schmidt and Rayleigh-Ritz steps: round-robin ordering, each round
// rotates n/2 disjoint (p, q) planes, rows then columns.  Rotation of Golub &
// Van Loan (sym.schur2): tau = (a_qq - a_pp) / (2 a_pq),
// t = sign(tau) / (|tau| + sqrt(1 + tau^2)), c = 1/sqrt(1+t^2), s = t c.
// Output ascending eigenvalues and the matching columns of V (FP64 copies).
//
// Two kernels with the same arithmetic in the same order, one on one CTA
// (small n) and one on a cluster of eight (jacobi.cuh).
#include "jacobi.cuh"

namespace bdg {

namespace {

// the plane rotation that annihilates apq
__device__ __forceinline__ void rotation(float app, float apq, float aqq, float& c, float& s) {
  c = 1.f;
  s = 0.f;
  if (fabsf(apq) > 1e-30f && fabsf(apq) > 1e-9f * sqrtf(fabsf(app * aqq))) {
    const float tau = (aqq - app) / (2.f * apq);
    const float t = (tau >= 0.f ? 1.f : -1.f) / (fabsf(tau) + sqrtf(1.f + tau * tau));
    c = rsqrtf(1.f + t * t);
    s = t * c;
  }
}

__global__ void __launch_bounds__(1024) k_jacobi(int n, const double* __restrict__ Ag, int lda,
                                                 double* __restrict__ w, double* __restrict__ Vg,
                                                 int max_sweeps, float off_tol) {
  extern __shared__ float sm[];
  const int ld = n | 1;          // odd: V is rotated down its columns
  float* A = sm;                 // [n][ld]
  float* V = A + n * ld;         // [n][ld]
  float* cs = V + n * ld;        // [npair][2]
  int* pq = (int*)(cs + 2 * (n / 2 + 1));  // [npair][2]
  float* red = (float*)(pq + 2 * (n / 2 + 1));  // [64]
  const int tid = threadIdx.x, nt = blockDim.x;
  const int np2 = (n + 1) & ~1;  // even count including a dummy index
  const int npair = np2 / 2;
  for (int e = tid; e < n * n; e += nt) {
    const int i = e / n, j = e - i * n;
    A[i * ld + j] = (float)Ag[(long long)i * lda + j];
    V[i * ld + j] = (i == j) ? 1.f : 0.f;
  }
  __syncthreads();
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    // off-diagonal and total Frobenius norms
    float off = 0.f, tot = 0.f;
    for (int e = tid; e < n * n; e += nt) {
      const int i = e / n, j = e - i * n;
      const float v = A[i * ld + j];
      tot += v * v;
      if (i != j) off += v * v;
    }
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    if ((tid & 31) == 0) { red[tid >> 5] = off; red[32 + (tid >> 5)] = tot; }
    __syncthreads();
    if (tid == 0) {
      float so = 0.f, st = 0.f;
      for (int q = 0; q < (nt + 31) / 32; ++q) { so += red[q]; st += red[32 + q]; }
      red[0] = so;
      red[32] = st;
    }
    __syncthreads();
    const bool done = red[0] <= off_tol * red[32];
    __syncthreads();
    if (done) break;
    for (int r = 0; r < np2 - 1; ++r) {
      if (tid < npair) {
        const int k = tid;
        int p = (r + k) % (np2 - 1);
        int q = (k == 0) ? (np2 - 1) : (r - k + np2 - 1) % (np2 - 1);
        if (p > q) { const int t = p; p = q; q = t; }
        float c = 1.f, s = 0.f;
        if (q < n) {
          rotation(A[p * ld + p], A[p * ld + q], A[q * ld + q], c, s);
        } else {
          q = p;  // dummy: no rotation
        }
        pq[2 * k] = p;
        pq[2 * k + 1] = q;
        cs[2 * k] = c;
        cs[2 * k + 1] = s;
      }
      __syncthreads();
      // A <- J^T A J and V <- V J in one pass: a work item is the 2 x 2 block
      // (row pair k, column pair l) of A or the rows of V's column pair l.
      // Warps take row pairs (or V's column pairs), lanes column pairs (or
      // rows): no index division, and the row pair's indices and rotation
      // are broadcast loads.  A dummy pair (odd n) has p == q and c = 1,
      // s = 0, which makes its duplicate reads and writes agree.
      const int lane = tid & 31, warp = tid >> 5, nwarp = nt >> 5;
      for (int k = warp; k < npair; k += nwarp) {
        const int p = pq[2 * k], q = pq[2 * k + 1];
        const float ck = cs[2 * k], sk = cs[2 * k + 1];
        float* Ap = A + p * ld;
        float* Aq = A + q * ld;
        for (int l = lane; l < npair; l += 32) {
          const int u = pq[2 * l], v = pq[2 * l + 1];
          Block2<float> b{Ap[u], Ap[v], Aq[u], Aq[v]};
          b.rotate(ck, sk, cs[2 * l], cs[2 * l + 1]);
          Ap[u] = b.x00;
          Ap[v] = b.x01;
          Aq[u] = b.x10;
          Aq[v] = b.x11;
        }
      }
      for (int l = warp; l < npair; l += nwarp) {
        const int u = pq[2 * l], v = pq[2 * l + 1];
        if (u == v) continue;
        const float cl = cs[2 * l], sl = cs[2 * l + 1];
        for (int i = lane; i < n; i += 32) {
          const float vp = V[i * ld + u], vq = V[i * ld + v];
          V[i * ld + u] = minus2(cl, vp, sl, vq);
          V[i * ld + v] = plus2(sl, vp, cl, vq);
        }
      }
      __syncthreads();
    }
  }
  // ascending order by rank of the diagonal
  for (int j = tid; j < n; j += nt) {
    const float dj = A[j * ld + j];
    int rank = 0;
    for (int l = 0; l < n; ++l) {
      const float dl = A[l * ld + l];
      rank += (dl < dj) || (dl == dj && l < j);
    }
    w[rank] = (double)dj;
    for (int i = 0; i < n; ++i) Vg[(long long)i * n + rank] = (double)V[i * ld + j];
  }
}

// Random matrices of n = 64, 96, 128, 160, whole call: 544 -> 526, 1283 -> 863,
// 2543 -> 1620, 4597 -> 2087 us (k_jacobi -> here); what is left is the latency
// of a round, about a microsecond of it the barrier with the stores under way
// and the rotations' divisions and square roots.
constexpr int THREADS = 512;
__global__ void __cluster_dims__(JC, 1, 1) __launch_bounds__(THREADS)
    k_jacobi_cluster(int n, const double* __restrict__ Ag, int lda, double* __restrict__ w, double* __restrict__ Vg,
                     int max_sweeps, float off_tol) {
  __shared__ JShared<float, SMALL_MAX, THREADS> sh;
  __shared__ float diag[SMALL_MAX];
  __shared__ int ranks[SMALL_MAX];
  const int tid = threadIdx.x, cta = blockIdx.x;
  const int v0 = cta * n / JC, vrows = (cta + 1) * n / JC - v0;
  const int par = jacobi_sweeps(
      sh, n, cta, max_sweeps, [&](int i, int j) { return (float)Ag[(long long)i * lda + j]; }, rotation,
      [&](float off, float tot) { return off <= off_tol * tot; });
  // ascending order by rank of the diagonal, which the elements of the next round hold
  const int N2 = (n + 1) & ~1;
  if (tid < N2 / 2) {
    diag[tid] = sh.next[par][0][tid];
    diag[N2 - 1 - tid] = sh.next[par][2][tid];   // (round 0: positions pair k with N2 - 1 - k)
  }
  __syncthreads();
  for (int j = tid; j < n; j += THREADS) {
    const float dj = diag[j];
    int rank = 0;
    for (int l = 0; l < n; ++l) {
      const float dl = diag[l];
      rank += (dl < dj) || (dl == dj && l < j);
    }
    ranks[j] = rank;
    if (cta == 0) w[rank] = (double)dj;
  }
  __syncthreads();
  for (int e = tid; e < vrows * n; e += THREADS) {
    const int i = e / n, j = e - i * n;
    Vg[(long long)(v0 + i) * n + ranks[j]] = (double)sh.V[i * SMALL_MAX + j];
  }
}

// From this size on: k_jacobi is ahead at n = 48 (321 against 363 us) and 56
// (396, 420), level at 64.  (A CTA needs two positions: n >= 31.)
constexpr int JMIN = 64;

}  // namespace

cudaError_t jacobi_f32(int n, const double* A, int lda, double* w, double* V, cudaStream_t s) {
  if (n <= 0 || n > SMALL_MAX) return cudaErrorInvalidValue;
  // converged to off(A) <= 1e-12 |A|^2: the FP64 refinement needs a start
  // this close (a stop at 1e-7 left backward errors up to 5e-2)
  constexpr int max_sweeps = 30;
  constexpr float off_tol = 1e-12f;
  if (n >= JMIN) {
    k_jacobi_cluster<<<JC, THREADS, 0, s>>>(n, A, lda, w, V, max_sweeps, off_tol);
    return cudaGetLastError();
  }
  const size_t sm = sizeof(float) * (2 * (size_t)n * (n + 1) + 2 * (n / 2 + 1)) +
                    sizeof(int) * 2 * (n / 2 + 1) + sizeof(float) * 64;
  cudaError_t e = allow_dynamic_smem((const void*)k_jacobi, sm);
  if (e != cudaSuccess) return e;
  k_jacobi<<<1, 1024, sm, s>>>(n, A, lda, w, V, max_sweeps, off_tol);
  return cudaGetLastError();
}

}  // namespace bdg
