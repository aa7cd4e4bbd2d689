// Small dense FP64 kernels: GEMM, symmetric eigen-decomposition (FP32
// Jacobi + FP64 Ogita-Aishima refinement), scaling.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cmath>
#include <vector>

#include "dense.cuh"
#include "jacobi.cuh"

namespace bdg {

namespace {

// C = alpha op(A) op(B) + beta C on tiles of 8 x 16, a thread per element: its
// sum runs over k in order.  The FP64 pipe bounds a CTA (a warp's multiply-add
// takes 64 clocks of its SM quarter), so the tiles are small enough that the
// projected problems (n up to 160) reach every SM with a warp per quarter, and
// the next 16 steps of k load while these run.  A call (16 x 16 tiles without
// the loads ahead -> now): n = 72 10.4 -> 8.3 us, 96 12.5 -> 8.5, 140 16.6 ->
// 14.5, 160 18.7 -> 14.7.
constexpr int TM = 8, TB = 16;

__global__ void __launch_bounds__(TM* TB)
    k_dgemm(bool ta, bool tb, int m, int n, int k, double alpha, const double* __restrict__ A, int lda,
            const double* __restrict__ B, int ldb, double beta, double* __restrict__ C, int ldc) {
  __shared__ double sA[TM][TB + 1];
  __shared__ double sB[TB][TB + 1];
  const int tid = threadIdx.x, tx = tid % TB, ty = tid / TB;
  const int i0 = blockIdx.y * TM, j0 = blockIdx.x * TB;
  // the elements of a step that this thread loads, along the rows in memory
  const int ai = ta ? tid % TM : ty, al = ta ? tid / TM : tx;
  double va, vb[2];
  auto fetch = [&](int l0) {
    const int ii = i0 + ai, ll = l0 + al;
    va = 0.0;
    if (ii < m && ll < k) va = ta ? A[(long long)ll * lda + ii] : A[(long long)ii * lda + ll];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int bl = l0 + (tb ? tx : ty + TM * h), bj = j0 + (tb ? ty + TM * h : tx);
      vb[h] = 0.0;
      if (bl < k && bj < n) vb[h] = tb ? B[(long long)bj * ldb + bl] : B[(long long)bl * ldb + bj];
    }
  };
  fetch(0);
  double acc = 0.0;
  for (int l0 = 0; l0 < k; l0 += TB) {
    sA[ai][al] = va;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (tb) sB[tx][ty + TM * h] = vb[h];
      else sB[ty + TM * h][tx] = vb[h];
    }
    __syncthreads();
    if (l0 + TB < k) fetch(l0 + TB);
    const int steps = min(TB, k - l0);
    if (steps == TB) {
#pragma unroll
      for (int l = 0; l < TB; ++l) acc = fma(sA[ty][l], sB[l][tx], acc);
    } else {
      for (int l = 0; l < steps; ++l) acc = fma(sA[ty][l], sB[l][tx], acc);
    }
    __syncthreads();
  }
  const int i = i0 + ty, j = j0 + tx;
  if (i < m && j < n) {
    double* c = C + (long long)i * ldc + j;
    *c = beta == 0.0 ? alpha * acc : fma(alpha, acc, beta * *c);
  }
}

// One Ogita-Aishima correction (SIAM J. Sci. Comput. 2018), given R = X^T X
// and S = X^T A X: lam_i = s_ii / (1 - r_ii), with r = I - X^T X;
// E_ij = (s_ij + lam_j r_ij) / (lam_j - lam_i) for pairs the current X
// resolves, else r_ij / 2 (orthogonalization only).  A pair counts as
// resolved when its corrections are small, |E_ij|, |E_ji| < 1/100, and its gap is above
// the rounding level of S (16 eps sqrt(n) |A|_F).  The pairwise test replaces the
// paper's global threshold 2 (|S - diag(lam)| + |A| |R|), which for graded
// spectra lumps every eigenvalue below eps_32 |A| into one cluster and stalls
// the refinement there.  On entry R holds X^T X; E is written over S.
__global__ void __launch_bounds__(1024) k_oa_correction(int n, double* __restrict__ R,
                                                        double* __restrict__ S,
                                                        const double* __restrict__ anorm_p,
                                                        double* __restrict__ lam) {
  const double anorm = *anorm_p;
  const int tid = threadIdx.x, nt = blockDim.x;
  // Symmetrize both products first: X^T (A X) carries a rounding asymmetry of
  // about eps n |A|, and the antisymmetric part of S would enter the
  // correction as (s_ij - s_ji) / (lam_j - lam_i) -- a loss of orthogonality
  // of eps n |A| / gap for small, graded eigenvalues.
  for (int e = tid; e < n * n; e += nt) {
    const int i = e / n, j = e - i * n;
    if (i > j) continue;
    const double r = 0.5 * (R[e] + R[j * n + i]);
    const double sv = 0.5 * (S[e] + S[j * n + i]);
    R[e] = (i == j ? 1.0 : 0.0) - r;
    R[j * n + i] = R[e];
    S[e] = sv;
    S[j * n + i] = sv;
  }
  __syncthreads();
  for (int i = tid; i < n; i += nt) lam[i] = S[i * n + i] / (1.0 - R[i * n + i]);
  __syncthreads();
  const double floor_gap = 16.0 * 2.220446049250313e-16 * sqrt((double)n) * anorm;
  for (int e = tid; e < n * n; e += nt) {
    const int i = e / n, j = e - i * n;
    const double r = R[e];
    double ev = 0.5 * r;
    if (i != j) {
      // the test is symmetric in (i, j) so that E_ij + E_ji = r_ij holds for
      // every pair and the update stays orthogonal to first order
      const double num = S[e] + lam[j] * r;
      const double numt = S[e] + lam[i] * r;
      const double den = lam[j] - lam[i];
      if (fabs(den) > floor_gap && 100.0 * fmax(fabs(num), fabs(numt)) < fabs(den)) ev = num / den;
    }
    S[e] = ev;
  }
}

__global__ void k_frob(int n, const double* __restrict__ A, int lda, double* __restrict__ out) {
  __shared__ double red[32];
  double s = 0.0;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int i = e / n, j = e - i * n;
    const double v = A[(long long)i * lda + j];
    s += v * v;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < (int)(blockDim.x + 31) / 32; ++q) t += red[q];
    *out = sqrt(t);
  }
}

// sort (w, V columns) ascending after refinement (n small; one CTA)
__global__ void k_sort_eig(int n, const double* __restrict__ w, const double* __restrict__ V,
                           double* __restrict__ w2, double* __restrict__ V2) {
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    const double dj = w[j];
    int rank = 0;
    for (int l = 0; l < n; ++l) rank += (w[l] < dj) || (w[l] == dj && l < j);
    w2[rank] = dj;
    for (int i = 0; i < n; ++i) V2[(long long)i * n + rank] = V[(long long)i * n + j];
  }
}

__global__ void k_dscale(int m, int n, const double* __restrict__ A, int lda, const double* __restrict__ dl,
                         const double* __restrict__ dr, double* __restrict__ B, int ldb) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < m * n; e += gridDim.x * blockDim.x) {
    const int i = e / n, j = e - i * n;
    double v = A[(long long)i * lda + j];
    if (dl) v *= dl[i];
    if (dr) v *= dr[j];
    B[(long long)i * ldb + j] = v;
  }
}

__global__ void k_dsym(int n, double* A, int lda) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += gridDim.x * blockDim.x) {
    const int i = e / n, j = e - i * n;
    if (j >= i) continue;
    const double v = 0.5 * (A[(long long)i * lda + j] + A[(long long)j * lda + i]);
    A[(long long)i * lda + j] = v;
    A[(long long)j * lda + i] = v;
  }
}

__global__ void k_dzero(int m, int n, double* B, int ldb) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < m * n; e += gridDim.x * blockDim.x) {
    const int i = e / n, j = e - i * n;
    B[(long long)i * ldb + j] = 0.0;
  }
}

}  // namespace

cudaError_t dsym_small(int n, double* A, int lda, cudaStream_t s) {
  if (n <= 1) return cudaSuccess;
  k_dsym<<<(n * n + 255) / 256, 256, 0, s>>>(n, A, lda);
  return cudaGetLastError();
}

cudaError_t dzero_small(int m, int n, double* B, int ldb, cudaStream_t s) {
  if (m <= 0 || n <= 0) return cudaSuccess;
  k_dzero<<<(m * n + 255) / 256, 256, 0, s>>>(m, n, B, ldb);
  return cudaGetLastError();
}

cudaError_t dgemm_small(bool ta, bool tb, int m, int n, int k, double alpha, const double* A, int lda,
                        const double* B, int ldb, double beta, double* C, int ldc, cudaStream_t s) {
  if (m <= 0 || n <= 0) return cudaSuccess;
  dim3 grid((n + TB - 1) / TB, (m + TM - 1) / TM);
  k_dgemm<<<grid, TM * TB, 0, s>>>(ta, tb, m, n, k, alpha, A, lda, B, ldb, beta, C, ldc);
  return cudaGetLastError();
}

cudaError_t dscale_small(int m, int n, const double* A, int lda, const double* dl, const double* dr,
                         double* B, int ldb, cudaStream_t s) {
  if (m <= 0 || n <= 0) return cudaSuccess;
  k_dscale<<<(m * n + 255) / 256, 256, 0, s>>>(m, n, A, lda, dl, dr, B, ldb);
  return cudaGetLastError();
}


__global__ void k_add_diag(int n, double* A, int lda, double c) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) A[(long long)i * lda + i] += c;
}
// M = (3 I - G) / 2, one Newton-Schulz step toward (G)^-1/2 for G = V^T V near I
__global__ void k_newton_schulz(int n, double* G) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += gridDim.x * blockDim.x) {
    const int i = e / n, j = e - i * n;
    G[e] = (i == j ? 1.5 : 0.0) - 0.5 * G[e];
  }
}
__global__ void k_add_vec(int n, double* w, double c) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) w[i] += c;
}

size_t eigh_workspace_doubles(int n) { return (size_t)48 * n * n + 128 * n + 256; }

namespace {

// ---------------------------------------------------------------------------
// All clusters of an FP32 Jacobi basis resolved in one launch.  CTA b takes
// the run of columns [start, start + size) of V (n x n, ld n) with midpoint
// shift c: two FP64 Newton-Schulz steps orthonormalize the columns, the
// shifted projection G = Vs^T (A - c I) Vs (norm about half the run's
// spread) is diagonalized by parallel cyclic Jacobi in FP64 (rotations of
// Golub & Van Loan, round-robin pairs as in jacobi.cu), and the rotated
// columns and eigenvalues (ascending within the run) replace the old ones.
// ---------------------------------------------------------------------------
constexpr int RC_MAX_CLUSTERS = 96;   // runs of two or more columns: at most n / 2
constexpr int RC_NS_MAX = 48;         // wider runs keep the sequential path
struct ClusterList {
  int count;
  int start[RC_MAX_CLUSTERS];
  int size[RC_MAX_CLUSTERS];
  double shift[RC_MAX_CLUSTERS];
};

// The rotation that annihilates apq (above the rounding level tiny).  For
// |tau| > 2^28, sqrt(1 + tau^2) rounds to |tau| and 1 + t^2 to 1: the short
// form gives the same bits without two square roots and a division.
struct Rotation64 {
  double tiny;
  __device__ __forceinline__ void operator()(double app, double apq, double aqq, double& c, double& s) const {
    c = 1.0;
    s = 0.0;
    if (fabs(apq) > tiny) {
      const double tau = (aqq - app) / (2.0 * apq), at = fabs(tau), sg = tau >= 0.0 ? 1.0 : -1.0;
      if (at > 0x1p28 && at < 0x1p500) {
        s = sg / (at + at);
      } else {
        const double t = sg / (at + sqrt(1.0 + tau * tau));
        c = 1.0 / sqrt(1.0 + t * t);
        s = t * c;
      }
    }
  }
};

constexpr int RT = 256;   // threads of a CTA of the resolving kernels

// What both resolving kernels begin with, on one CTA: the run's columns of V
// orthonormalized in Vs, their shifted projection in G ([ns][ld]) and, for
// every thread, its Frobenius norm.  T: n x ns, Z: like G, red: 34 values.
__device__ double resolve_project(int n, const double* __restrict__ A, int lda, const double* V, int i0, int ns,
                                  double c, int ld, double* Vs, double* T, double* G, double* Z, double* red) {
  const int tid = threadIdx.x, nt = RT;
  for (int e = tid; e < n * ns; e += nt) {
    const int i = e / ns, j = e - i * ns;
    Vs[e] = V[(long long)i * n + i0 + j];
  }
  __syncthreads();
  // Vs <- Vs (3 I - Vs^T Vs) / 2, twice
  for (int it = 0; it < 2; ++it) {
    for (int e = tid; e < ns * ns; e += nt) {
      const int a = e / ns, b = e - a * ns;
      double sacc = 0.0;
      for (int i = 0; i < n; ++i) sacc = fma(Vs[i * ns + a], Vs[i * ns + b], sacc);
      G[a * ld + b] = (a == b ? 1.5 : 0.0) - 0.5 * sacc;
    }
    __syncthreads();
    for (int e = tid; e < n * ns; e += nt) {
      const int i = e / ns, b = e - i * ns;
      double sacc = 0.0;
      for (int a = 0; a < ns; ++a) sacc = fma(Vs[i * ns + a], G[a * ld + b], sacc);
      T[e] = sacc;
    }
    __syncthreads();
    for (int e = tid; e < n * ns; e += nt) Vs[e] = T[e];
    __syncthreads();
  }
  // T = (A - c I) Vs, G = Vs^T T symmetrized
  for (int e = tid; e < n * ns; e += nt) {
    const int i = e / ns, b = e - i * ns;
    const double* Ai = A + (long long)i * lda;
    double sacc = -c * Vs[i * ns + b];
    for (int k = 0; k < n; ++k) sacc = fma(Ai[k], Vs[k * ns + b], sacc);
    T[e] = sacc;
  }
  __syncthreads();
  for (int e = tid; e < ns * ns; e += nt) {
    const int a = e / ns, b = e - a * ns;
    double sacc = 0.0;
    for (int i = 0; i < n; ++i) sacc = fma(Vs[i * ns + a], T[i * ns + b], sacc);
    Z[a * ld + b] = sacc;
  }
  __syncthreads();
  double fro = 0.0;
  for (int e = tid; e < ns * ns; e += nt) {
    const int a = e / ns, b = e - a * ns;
    const double v = 0.5 * (Z[a * ld + b] + Z[b * ld + a]);
    G[a * ld + b] = v;
    fro += v * v;
  }
  for (int o = 16; o > 0; o >>= 1) fro += __shfl_xor_sync(0xffffffffu, fro, o);
  if ((tid & 31) == 0) red[tid >> 5] = fro;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int q = 0; q < nt / 32; ++q) t += red[q];
    red[32] = sqrt(t);
  }
  __syncthreads();
  return red[32];
}

size_t resolve_smem_bytes(int n, int ns) {
  const int np2 = (ns + 1) & ~1;
  return sizeof(double) * (2 * (size_t)n * ns + 2 * (size_t)ns * (ns | 1) + 4 * (size_t)np2 + 64) +
         sizeof(int) * (2 * (size_t)np2 + 2 * (size_t)ns + 8);
}

__global__ void __launch_bounds__(RT) k_resolve_clusters(int n, const double* __restrict__ A, int lda,
                                                         double* __restrict__ w, double* __restrict__ V,
                                                         ClusterList cl) {
  extern __shared__ double rsm[];
  const int i0 = cl.start[blockIdx.x], ns = cl.size[blockIdx.x];
  const double c = cl.shift[blockIdx.x];
  const int np2 = (ns + 1) & ~1, npair = np2 / 2;
  double* Vs = rsm;                       // [n][ns]
  double* T = Vs + (size_t)n * ns;        // [n][ns]
  const int ld = ns | 1;                  // odd: Z is rotated down its columns
  double* G = T + (size_t)n * ns;         // [ns][ld]
  double* Z = G + (size_t)ns * ld;        // [ns][ld]
  double* cs = Z + (size_t)ns * ld;       // [2][npair][2]: this round's rotations and the next's
  double* red = cs + 2 * np2;             // [64]
  int* pq = reinterpret_cast<int*>(red + 64);   // [2][npair][2]
  int* rank = pq + 2 * np2;               // [ns]
  const int tid = threadIdx.x, nt = RT;
  const double fro = resolve_project(n, A, lda, V, i0, ns, c, ld, Vs, T, G, Z, red);
  for (int e = tid; e < ns * ns; e += nt) Z[e / ns * ld + e % ns] = (e / ns == e % ns) ? 1.0 : 0.0;
  __syncthreads();
  const double tiny = 1e-18 * fro;
  const Rotation64 rotate{tiny};
  // parallel cyclic Jacobi in FP64
  for (int sweep = 0; sweep < 40; ++sweep) {
    double off = 0.0;
    for (int e = tid; e < ns * ns; e += nt) {
      const int a = e / ns, b = e - a * ns;
      const double v = G[a * ld + b];
      if (a != b) off += v * v;
    }
    for (int o = 16; o > 0; o >>= 1) off += __shfl_xor_sync(0xffffffffu, off, o);
    __syncthreads();
    if ((tid & 31) == 0) red[tid >> 5] = off;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int q = 0; q < (nt + 31) / 32; ++q) t += red[q];
      red[33] = t;
    }
    __syncthreads();
    if (!(red[33] > 1e-32 * fro * fro) || !(red[33] > tiny * tiny)) break;
    // The rotations of round r + 1 need the matrix of round r, but not Z: the
    // first warp forms them (a chain of divisions and square roots) while the
    // others rotate Z.  Per round the FP64 pipe of the SM bounds both parts.
    auto rotations = [&](int r, int set) {
      if (tid < npair) {
        const int k = tid;
        int p = (r + k) % (np2 - 1);
        int q = (k == 0) ? (np2 - 1) : (r - k + np2 - 1) % (np2 - 1);
        if (p > q) { const int t = p; p = q; q = t; }
        double cc = 1.0, ss = 0.0;
        if (q < ns) {
          rotate(G[p * ld + p], G[p * ld + q], G[q * ld + q], cc, ss);
        } else {
          q = p;
        }
        pq[set * np2 + 2 * k] = p;
        pq[set * np2 + 2 * k + 1] = q;
        cs[set * np2 + 2 * k] = cc;
        cs[set * np2 + 2 * k + 1] = ss;
      }
    };
    rotations(0, 0);
    for (int r = 0; r < np2 - 1; ++r) {
      const int* pqr = pq + (r & 1) * np2;
      const double* csr = cs + (r & 1) * np2;
      __syncthreads();
      for (int e = tid; e < npair * npair; e += nt) {
        const int k = e / npair, l = e - k * npair;
        const int p = pqr[2 * k], q = pqr[2 * k + 1], u = pqr[2 * l], v = pqr[2 * l + 1];
        Block2<double> x{G[p * ld + u], G[p * ld + v], G[q * ld + u], G[q * ld + v]};
        x.rotate(csr[2 * k], csr[2 * k + 1], csr[2 * l], csr[2 * l + 1]);
        G[p * ld + u] = x.x00;
        G[p * ld + v] = x.x01;
        G[q * ld + u] = x.x10;
        G[q * ld + v] = x.x11;
      }
      __syncthreads();
      if (tid < 32) {   // (npair <= 24 lanes of one warp)
        if (r + 1 < np2 - 1) rotations(r + 1, (r + 1) & 1);
      } else {
        for (int f = tid - 32; f < npair * ns; f += nt - 32) {
          const int l = f / ns, i = f - l * ns;
          const int u = pqr[2 * l], v = pqr[2 * l + 1];
          if (u == v) continue;
          const double cl_ = csr[2 * l], sl = csr[2 * l + 1];
          const double zp = Z[i * ld + u], zq = Z[i * ld + v];
          Z[i * ld + u] = minus2(cl_, zp, sl, zq);
          Z[i * ld + v] = plus2(sl, zp, cl_, zq);
        }
      }
    }
    __syncthreads();
  }
  // ascending order within the run, new columns Vs Z, eigenvalues + c
  for (int j = tid; j < ns; j += nt) {
    const double dj = G[j * ld + j];
    int rk = 0;
    for (int l = 0; l < ns; ++l) {
      const double dl = G[l * ld + l];
      rk += (dl < dj) || (dl == dj && l < j);
    }
    rank[j] = rk;
    w[i0 + rk] = dj + c;
  }
  __syncthreads();
  for (int e = tid; e < n * ns; e += nt) {
    const int i = e / ns, j = e - i * ns;
    double sacc = 0.0;
    for (int a = 0; a < ns; ++a) sacc = fma(Vs[i * ns + a], Z[a * ld + j], sacc);
    V[(long long)i * n + i0 + rank[j]] = sacc;
  }
}

// Wide runs on a cluster of eight CTAs (jacobi.cuh): the FP64 pipe of one SM
// bounds a round there, and the many sweeps of a run that is degenerate to
// working precision are serial.  Two runs of 48 such columns of n = 96: 9.9 ms
// on one CTA each, 3.84 here; two of 42 (n = 128), resolved in a few sweeps:
// whole eigensolve 9.8 -> 6.6 ms.  Narrower runs would leave a CTA of the
// cluster without its two pair positions.
constexpr int RC_WIDE = 32;
typedef JShared<double, RC_NS_MAX, RT> RShared;

size_t resolve_wide_smem_bytes(int n, int ns) {
  return sizeof(RShared) + sizeof(double) * (2 * (size_t)n * ns + 2 * (size_t)ns * (ns | 1) + 64 + (size_t)RC_NS_MAX) +
         sizeof(int) * (size_t)RC_NS_MAX;
}

__global__ void __cluster_dims__(JC, 1, 1) __launch_bounds__(RT)
    k_resolve_wide(int n, const double* __restrict__ A, int lda, double* __restrict__ w, double* __restrict__ V,
                   ClusterList cl) {
  extern __shared__ double rsm[];
  const int run = blockIdx.x / JC, cta = blockIdx.x % JC;
  const int i0 = cl.start[run], ns = cl.size[run], ld = ns | 1;
  const double c = cl.shift[run];
  RShared& sh = *reinterpret_cast<RShared*>(rsm);
  double* Vs = rsm + sizeof(RShared) / sizeof(double);   // [n][ns]
  double* T = Vs + (size_t)n * ns;                       // [n][ns]
  double* G = T + (size_t)n * ns;                        // [ns][ld]
  double* Z = G + (size_t)ns * ld;                       // [ns][ld]
  double* red = Z + (size_t)ns * ld;                     // [64]
  double* diag = red + 64;                               // [RC_NS_MAX]
  int* rank = reinterpret_cast<int*>(diag + RC_NS_MAX);  // [RC_NS_MAX]
  const int tid = threadIdx.x;
  const double fro = resolve_project(n, A, lda, V, i0, ns, c, ld, Vs, T, G, Z, red);   // (every CTA for itself)
  const double tiny = 1e-18 * fro;
  const int par = jacobi_sweeps(
      sh, ns, cta, 40, [&](int i, int j) { return G[i * ld + j]; }, Rotation64{tiny},
      [&](double off, double) { return !(off > 1e-32 * fro * fro) || !(off > tiny * tiny); });
  // the rows of Z to every CTA
  const int z0 = cta * ns / JC, zrows = (cta + 1) * ns / JC - z0;
  __syncthreads();
  for (int e = tid; e < zrows * ns; e += RT) {
    const int i = e / ns, j = e - i * ns;
    const uint32_t o = s_u32(Z + (z0 + i) * ld + j);
    const double v = sh.V[i * RC_NS_MAX + j];
    for (int d = 0; d < JC; ++d) put(at_cta(o, d), v);
  }
  // ascending order within the run, new columns Vs Z, eigenvalues + c
  const int np2 = (ns + 1) & ~1;
  if (tid < np2 / 2) {
    diag[tid] = sh.next[par][0][tid];
    if (np2 - 1 - tid < ns) diag[np2 - 1 - tid] = sh.next[par][2][tid];   // (round 0's pairs)
  }
  cluster_arrive();
  cluster_wait();
  for (int j = tid; j < ns; j += RT) {
    const double dj = diag[j];
    int rk = 0;
    for (int l = 0; l < ns; ++l) {
      const double dl = diag[l];
      rk += (dl < dj) || (dl == dj && l < j);
    }
    rank[j] = rk;
    if (cta == 0) w[i0 + rk] = dj + c;
  }
  __syncthreads();
  const int r0 = cta * n / JC, r1 = (cta + 1) * n / JC;
  for (int e = tid; e < (r1 - r0) * ns; e += RT) {
    const int i = r0 + e / ns, j = e % ns;
    double sacc = 0.0;
    for (int a = 0; a < ns; ++a) sacc = fma(Vs[i * ns + a], Z[a * ld + j], sacc);
    V[(long long)i * n + i0 + rank[j]] = sacc;
  }
}

// FP32 Jacobi start for A (n x n, lda) into (w, V), with clusters resolved
// by recursion.  FP32 separates eigenvalues only down to about 1e-7 max|w|;
// every run of consecutive eigenvalues closer than 1e-4 max|w| (a cluster
// around its midpoint c -- which includes the eigenvalues near zero of a
// graded matrix) is re-solved on the FP64 projection V_s^T (A - c I) V_s,
// whose norm is about the spread, and rotated back.  Runs are disjoint, so
// the workspace is reused from one to the next.
cudaError_t jacobi_multilevel(int n, const double* A, int lda, double* w, double* V, double* ws, int depth,
                              double floor, double shift, cudaStream_t s) {
  cudaError_t e;
  static const bool prof = getenv("BDG_PROFILE_EIGH") != nullptr;
  cudaEvent_t pj[2] = {};
  if (prof) {
    cudaEventCreate(&pj[0]);
    cudaEventCreate(&pj[1]);
    cudaEventRecord(pj[0], s);
  }
  if ((e = jacobi_f32(n, A, lda, w, V, s))) return e;
  if (prof) {
    cudaEventRecord(pj[1], s);
    cudaEventSynchronize(pj[1]);
    float t = 0;
    cudaEventElapsedTime(&t, pj[0], pj[1]);
    fprintf(stderr, "[bdg]   jacobi n %d depth %d %.3f ms\n", n, depth, t);
    cudaEventDestroy(pj[0]);
    cudaEventDestroy(pj[1]);
  }
  if (depth >= 4 || n < 2) return cudaSuccess;
  std::vector<double> hw(n);
  if ((e = cudaMemcpyAsync(hw.data(), w, sizeof(double) * n, cudaMemcpyDeviceToHost, s))) return e;
  if ((e = cudaStreamSynchronize(s))) return e;
  double amax = 0.0;
  for (double v : hw) amax = std::max(amax, std::fabs(v));
  if (!(amax > 0)) return cudaSuccess;
  if (depth == 0) floor *= amax;   // the caller's floor is relative at the top level
  const double tau = 1e-4 * amax;
  // runs of at most RC_NS_MAX columns are resolved by one launch (FP64
  // Jacobi per run); wider runs re-solve in turn on their projection
  ClusterList lists[2];   // narrow runs, wide ones
  int ns_max[2] = {0, 0};
  lists[0].count = lists[1].count = 0;
  for (int i0 = 0; i0 < n;) {
    int i1 = i0 + 1;
    while (i1 < n && hw[i1] - hw[i1 - 1] < tau) ++i1;
    const int ns = i1 - i0;
    // a run whose spread is at the FP64 rounding level -- of its own values
    // or of the whole matrix -- is degenerate to working precision: any
    // orthonormal basis of it is an eigenbasis and nothing is re-solved
    const double spread = hw[i1 - 1] - hw[i0];
    const double mag = std::max(std::fabs(hw[i0]), std::fabs(hw[i1 - 1]));
    const bool degenerate = spread <= 1e-12 * mag || spread <= 64 * 2.220446049250313e-16 * amax;
    // runs whose eigenvalues all lie below the caller's floor (|lambda| of the
    // original matrix) are not needed resolved: the caller discards them
    const double top = std::max(std::fabs(hw[i0] + shift), std::fabs(hw[i1 - 1] + shift));
    if (ns >= 2 && spread > 0 && !degenerate && !(top < floor) && ns <= RC_NS_MAX &&
        lists[ns >= RC_WIDE].count < RC_MAX_CLUSTERS) {
      ClusterList& cl = lists[ns >= RC_WIDE];
      cl.start[cl.count] = i0;
      cl.size[cl.count] = ns;
      cl.shift[cl.count] = 0.5 * (hw[i0] + hw[i1 - 1]);
      cl.count++;
      ns_max[ns >= RC_WIDE] = std::max(ns_max[ns >= RC_WIDE], ns);
    } else if (ns >= 2 && spread > 0 && !degenerate && !(top < floor)) {
      const double c = 0.5 * (hw[i0] + hw[i1 - 1]);  // midpoint: the shifted norm is half the spread
      double* Vs = ws;                         // n x ns
      double* AVs = Vs + (size_t)n * ns;       // n x ns
      double* As = AVs + (size_t)n * ns;       // ns x ns
      double* w2 = As + (size_t)ns * ns;       // ns
      double* V2 = w2 + ns + 8;                // ns x ns
      double* Vn = V2 + (size_t)ns * ns;       // n x ns
      double* rest = Vn + (size_t)n * ns;
      // V's columns i0 .. i1-1 are contiguous: gather with a strided copy
      if ((e = cudaMemcpy2DAsync(Vs, sizeof(double) * ns, V + i0, sizeof(double) * n, sizeof(double) * ns, n,
                                 cudaMemcpyDeviceToDevice, s)))
        return e;
      // FP64 orthonormalization of the FP32 columns (two Newton-Schulz
      // steps): with c != 0 the projection would otherwise carry
      // c (V^T V - I) ~ 1e-7 c, which can exceed the spread being resolved
      for (int it = 0; it < 2; ++it) {
        if ((e = dgemm_small(true, false, ns, ns, n, 1.0, Vs, ns, Vs, ns, 0.0, As, ns, s))) return e;
        k_newton_schulz<<<(ns * ns + 255) / 256, 256, 0, s>>>(ns, As);
        if ((e = cudaGetLastError())) return e;
        if ((e = dgemm_small(false, false, n, ns, ns, 1.0, Vs, ns, As, ns, 0.0, Vn, ns, s))) return e;
        if ((e = cudaMemcpyAsync(Vs, Vn, sizeof(double) * n * ns, cudaMemcpyDeviceToDevice, s))) return e;
      }
      if ((e = dgemm_small(false, false, n, ns, n, 1.0, A, lda, Vs, ns, 0.0, AVs, ns, s))) return e;
      if ((e = dgemm_small(true, false, ns, ns, n, 1.0, Vs, ns, AVs, ns, 0.0, As, ns, s))) return e;
      if ((e = dsym_small(ns, As, ns, s))) return e;
      k_add_diag<<<(ns + 127) / 128, 128, 0, s>>>(ns, As, ns, -c);
      if ((e = cudaGetLastError())) return e;
      if ((e = jacobi_multilevel(ns, As, ns, w2, V2, rest, depth + 1, floor, shift + c, s))) return e;
      k_add_vec<<<(ns + 127) / 128, 128, 0, s>>>(ns, w2, c);
      if ((e = cudaGetLastError())) return e;
      if ((e = dgemm_small(false, false, n, ns, ns, 1.0, Vs, ns, V2, ns, 0.0, Vn, ns, s))) return e;
      if ((e = cudaMemcpy2DAsync(V + i0, sizeof(double) * n, Vn, sizeof(double) * ns, sizeof(double) * ns, n,
                                 cudaMemcpyDeviceToDevice, s)))
        return e;
      if ((e = cudaMemcpyAsync(w + i0, w2, sizeof(double) * ns, cudaMemcpyDeviceToDevice, s))) return e;
    }
    i0 = i1;
  }
  if (prof && depth == 0)
    fprintf(stderr, "[bdg]   clusters n %d: %d batched (widest %d)\n", n, lists[0].count + lists[1].count,
            std::max(ns_max[0], ns_max[1]));
  if (lists[1].count > 0) {
    const size_t smr = resolve_wide_smem_bytes(n, ns_max[1]);
    if ((e = allow_dynamic_smem((const void*)k_resolve_wide, smr))) return e;
    k_resolve_wide<<<JC * lists[1].count, RT, smr, s>>>(n, A, lda, w, V, lists[1]);
    if ((e = cudaGetLastError())) return e;
  }
  if (lists[0].count > 0) {
    const size_t smr = resolve_smem_bytes(n, ns_max[0]);
    if ((e = allow_dynamic_smem((const void*)k_resolve_clusters, smr))) return e;
    k_resolve_clusters<<<lists[0].count, RT, smr, s>>>(n, A, lda, w, V, lists[0]);
    if ((e = cudaGetLastError())) return e;
  }
  return cudaSuccess;
}

}  // namespace

// ---------------------------------------------------------------------------
// Rank-revealing pivoted Cholesky (see dense.cuh), one CTA of 1024 threads:
// right-looking, the lower triangle of the working matrix S in shared memory;
// step k swaps the largest remaining diagonal to position k, forms column k of
// L and updates the trailing lower triangle.  The inverse X of L1 follows,
// right-looking as well, in the strictly upper triangle: row j,
// X_jc = acc_jc / L_jj, then acc_ic -= L_ij X_jc for all later rows i, from
// acc_ic = -L_ic / L_cc.  The FP64 pipe of the SM bounds both, n^3/3 multiply-
// adds, with the barriers: only one triangle is updated, warps take rows (of
// columns of X) and lanes run along them, and what lanes need of a column lies
// in a vector of its own.  Both triangles updated and X row by row -> now:
// n = 72 495 -> 389 us, 96 836 -> 569, 140 1330 -> 980, 160 2140 -> 1241, the
// same bits.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) k_pchol(int n, const double* __restrict__ A, int lda, double tol,
                                                double* __restrict__ L, double* __restrict__ M, int ldo,
                                                int* __restrict__ rank_dev) {
  extern __shared__ double psm[];
  double* S = psm;                           // [n][n]
  double* dinv = S + (size_t)n * n;          // [n]: 1 / L_ii
  double* diag = dinv + n;                   // [n]: remaining diagonal
  double* col = diag + n;                    // [n]: the step's column of L
  int* perm = reinterpret_cast<int*>(col + n);
  __shared__ double sh_d0;
  __shared__ int sh_p, sh_r;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarp = nt >> 5;
  for (int e = tid; e < n * n; e += nt) {
    const int i = e / n, j = e - i * n;
    if (j <= i) S[e] = A[(long long)i * lda + j];
  }
  for (int i = tid; i < n; i += nt) {
    perm[i] = i;
    diag[i] = A[(long long)i * lda + i];
  }
  if (tid == 0) sh_r = n;
  __syncthreads();
  if (tid < 32) {
    double m = 0.0;
    for (int i = tid; i < n; i += 32) m = fmax(m, diag[i]);
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (tid == 0) sh_d0 = m;
  }
  __syncthreads();
  const double dmin = tol * sh_d0;
  for (int k = 0; k < n; ++k) {
    if (tid < 32) {   // pivot: largest remaining diagonal (first index on ties)
      double m = -1.0;
      int p = k;
      for (int i = k + tid; i < n; i += 32) {
        const double d = diag[i];
        if (d > m) { m = d; p = i; }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const double m2 = __shfl_xor_sync(0xffffffffu, m, o);
        const int p2 = __shfl_xor_sync(0xffffffffu, p, o);
        if (m2 > m || (m2 == m && p2 < p)) { m = m2; p = p2; }
      }
      if (tid == 0) {
        sh_p = p;
        if (!(m > dmin) || !(sh_d0 > 0.0)) sh_r = k;
      }
    }
    __syncthreads();
    if (sh_r == k) break;
    const int p = sh_p;
    const double lkk = sqrt(diag[p]);
    // symmetric swap of rows / columns k and p in the lower triangle; row k is
    // column k of the trailing matrix
    if (p != k) {
      for (int j = tid; j < n; j += nt) {
        if (j == k || j == p) continue;
        double* x = S + (j < k ? k * n + j : j * n + k);
        double* y = S + (j < p ? p * n + j : j * n + p);
        const double t = *x;
        *x = *y;
        *y = t;
      }
      __syncthreads();
      if (tid == 0) {
        const int t = perm[k];
        perm[k] = perm[p];
        perm[p] = t;
        diag[p] = diag[k];
      }
    }
    for (int i = k + 1 + tid; i < n; i += nt) {
      const double c = S[i * n + k] / lkk;
      S[i * n + k] = c;
      col[i] = c;
    }
    if (tid == 0) S[k * n + k] = lkk;
    __syncthreads();
    // trailing update; the diagonal lives in its vector
    for (int i = k + 1 + warp; i < n; i += nwarp) {
      const double ci = col[i];
      for (int j = k + 1 + lane; j <= i; j += 32) {
        double* x = j < i ? S + i * n + j : diag + i;
        *x -= ci * col[j];
      }
    }
    __syncthreads();
  }
  const int r = sh_r;
  // L in the original row order: row perm[i] of L is row i of the factor
  for (int e = tid; e < n * n; e += nt) {
    const int i = e / n, c = e - i * n;
    L[(long long)perm[i] * ldo + c] = (c < r && c <= i) ? S[i * n + c] : 0.0;
    M[(long long)i * ldo + c] = 0.0;
  }
  for (int i = tid; i < r; i += nt) dinv[i] = 1.0 / S[i * n + i];
  __syncthreads();
  // X = L1^-1 (r x r, lower): X_ii in dinv, X_ic (c < i) at S[c * n + i]
  for (int c = warp; c < r; c += nwarp) {
    const double d = dinv[c];
    for (int i = c + 1 + lane; i < r; i += 32) S[c * n + i] = -S[i * n + c] * d;
  }
  __syncthreads();
  for (int j = 1; j < r; ++j) {
    for (int c = tid; c < j; c += nt) S[c * n + j] *= dinv[j];
    for (int i = j + 1 + tid; i < r; i += nt) col[i] = S[i * n + j];
    __syncthreads();
    for (int c = warp; c < j; c += nwarp) {
      const double x = S[c * n + j];
      for (int i = j + 1 + lane; i < r; i += 32) S[c * n + i] -= col[i] * x;
    }
    __syncthreads();
  }
  // M = P^T [L1^-T; 0]: row perm[i] (i < r) holds (L1^-T)_{i c} = X_{c i}
  for (int e = tid; e < r * r; e += nt) {
    const int i = e / r, c = e - i * r;
    M[(long long)perm[i] * ldo + c] = c == i ? dinv[i] : (c > i ? S[i * n + c] : 0.0);
  }
  if (tid == 0) *rank_dev = r;
}

// X = I, lam = diag(A): the start for nearly diagonal matrices
__global__ void k_identity_start(int n, const double* __restrict__ A, int lda, double* __restrict__ X,
                                 double* __restrict__ lam) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += gridDim.x * blockDim.x) {
    const int i = e / n, j = e - i * n;
    X[e] = i == j ? 1.0 : 0.0;
    if (i == j) lam[i] = A[(long long)i * lda + i];
  }
}

cudaError_t pchol(int n, const double* A, int lda, double tol, double* L, double* M, int ldo, int* rank_dev,
                  cudaStream_t s) {
  if (n <= 0 || n > SMALL_MAX || ldo < n) return cudaErrorInvalidValue;
  const size_t sm = sizeof(double) * ((size_t)n * n + 3 * (size_t)n) + sizeof(int) * (size_t)n;
  cudaError_t e = allow_dynamic_smem((const void*)k_pchol, sm);
  if (e != cudaSuccess) return e;
  k_pchol<<<1, 1024, sm, s>>>(n, A, lda, tol, L, M, ldo, rank_dev);
  return cudaGetLastError();
}

cudaError_t eigh(int n, const double* A, int lda, double* w, double* V, double* ws, int refine_steps,
                 cudaStream_t s, double floor_rel, bool from_identity) {
  if (n <= 0) return cudaSuccess;
  if (n > SMALL_MAX) return cudaErrorInvalidValue;
  cudaError_t e;
  double* X = ws;                 // n x n current eigenvectors
  double* X2 = X + n * n;         // n x n
  double* R = X2 + n * n;         // n x n
  double* S = R + n * n;          // n x n
  double* AX = S + n * n;         // n x n
  double* lam = AX + n * n;       // n
  double* lam2 = lam + n;         // n
  double* anorm = lam2 + n;       // 8
  double* rest = anorm + 8;
  // diagnostics (BDG_PROFILE_EIGH): device time of the start, the refinement
  // and the ordering of this call, printed per call
  static const bool prof = getenv("BDG_PROFILE_EIGH") != nullptr;
  cudaEvent_t pe[4] = {};
  if (prof)
    for (auto& x : pe) cudaEventCreate(&x);
  if (prof) cudaEventRecord(pe[0], s);
  if (from_identity) {
    k_identity_start<<<(n * n + 255) / 256, 256, 0, s>>>(n, A, lda, X, lam2);
    if ((e = cudaGetLastError())) return e;
  } else if ((e = jacobi_multilevel(n, A, lda, lam2, X, rest, 0, floor_rel, 0.0, s))) {
    return e;
  }
  if (prof) cudaEventRecord(pe[1], s);
  k_frob<<<1, 1024, 0, s>>>(n, A, lda, anorm);
  double* cur = X;
  double* nxt = X2;
  for (int it = 0; it < refine_steps; ++it) {
    if ((e = dgemm_small(true, false, n, n, n, 1.0, cur, n, cur, n, 0.0, R, n, s))) return e;
    if ((e = dgemm_small(false, false, n, n, n, 1.0, A, lda, cur, n, 0.0, AX, n, s))) return e;
    if ((e = dgemm_small(true, false, n, n, n, 1.0, cur, n, AX, n, 0.0, S, n, s))) return e;
    k_oa_correction<<<1, 1024, 0, s>>>(n, R, S, anorm, lam);
    if ((e = cudaGetLastError())) return e;
    // X <- X + X E
    if ((e = cudaMemcpyAsync(nxt, cur, sizeof(double) * n * n, cudaMemcpyDeviceToDevice, s))) return e;
    if ((e = dgemm_small(false, false, n, n, n, 1.0, cur, n, S, n, 1.0, nxt, n, s))) return e;
    double* t = cur; cur = nxt; nxt = t;
  }
  // Rotations driven by rounding noise (pairs just above the gap floor)
  // leave a second-order loss of orthogonality; two Newton-Schulz steps
  // X <- X (3 I - X^T X) / 2 remove it without rotating.
  for (int it = 0; refine_steps > 0 && it < 2; ++it) {
    if ((e = dgemm_small(true, false, n, n, n, 1.0, cur, n, cur, n, 0.0, R, n, s))) return e;
    k_newton_schulz<<<(n * n + 255) / 256, 256, 0, s>>>(n, R);
    if ((e = cudaGetLastError())) return e;
    if ((e = dgemm_small(false, false, n, n, n, 1.0, cur, n, R, n, 0.0, nxt, n, s))) return e;
    double* t = cur; cur = nxt; nxt = t;
  }
  if (prof) cudaEventRecord(pe[2], s);
  k_sort_eig<<<1, 256, 0, s>>>(n, refine_steps > 0 ? lam : lam2, cur, w, V);
  if (prof) {
    cudaEventRecord(pe[3], s);
    cudaEventSynchronize(pe[3]);
    float t0 = 0, t1 = 0, t2 = 0;
    cudaEventElapsedTime(&t0, pe[0], pe[1]);
    cudaEventElapsedTime(&t1, pe[1], pe[2]);
    cudaEventElapsedTime(&t2, pe[2], pe[3]);
    fprintf(stderr, "[bdg] eigh n %d %s start %.3f refine %.3f sort %.3f ms\n", n, from_identity ? "identity" : "jacobi",
            t0, t1, t2);
    for (auto& x : pe) cudaEventDestroy(x);
  }
  return cudaGetLastError();
}

}  // namespace bdg
