// FP32 parallel cyclic Jacobi for the small symmetric eigenproblems of the
// Gram-Schmidt and Rayleigh-Ritz steps: round-robin ordering, each round
// rotates n/2 disjoint (p, q) planes, rows then columns.  Rotation of Golub &
// Van Loan (sym.schur2): tau = (a_qq - a_pp) / (2 a_pq),
// t = sign(tau) / (|tau| + sqrt(1 + tau^2)), c = 1/sqrt(1+t^2), s = t c.
// Output ascending eigenvalues and the matching columns of V (FP64 copies).
//
// Two kernels with the same arithmetic in the same order, one on one CTA
// (small n) and one on a cluster of eight.
#include <algorithm>

#include "dense.cuh"

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

// One 2 x 2 block (rows p < q, columns u < v): rows first, then columns, as
// the two one-sided updates would do.
struct Block2 {
  float x00, x01, x10, x11;
  __device__ __forceinline__ void rotate(float ck, float sk, float cl, float sl) {
    const float r00 = ck * x00 - sk * x10, r01 = ck * x01 - sk * x11;
    const float r10 = sk * x00 + ck * x10, r11 = sk * x01 + ck * x11;
    x00 = cl * r00 - sl * r01;
    x01 = sl * r00 + cl * r01;
    x10 = cl * r10 - sl * r11;
    x11 = sl * r10 + cl * r11;
  }
};

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
          Block2 b{Ap[u], Ap[v], Aq[u], Aq[v]};
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
          V[i * ld + u] = cl * vp - sl * vq;
          V[i * ld + v] = sl * vp + cl * vq;
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

// ---------------------------------------------------------------------------
// The same on a cluster of eight CTAs.  One CTA is bound by the round: its
// shared-memory traffic and issue (n^2/4 blocks and n^2/2 rotations of V), a
// thousand rounds one after another.  Here a CTA
// holds the columns of A of its share of the round's pair positions, and its
// share of the rows of V.
//
// From round r to r + 1 the index at position k of the first kind ("P",
// (r + k) mod (n - 1)) moves to position k - 1 and that of the second kind
// ("Q", (r - k) mod (n - 1)) to k + 1; position 0's Q stays, and the two ends
// pass P to Q and Q to P.  Each kind's columns lie in a ring of one slot more
// than positions, so that a column which stays in the CTA does not move, and
// one that leaves is written by its update straight into the free slot of the
// neighbour (distributed shared memory).  Rows stay in the order of the index.
//
// The rotations of the next round need three elements per pair: the lanes that
// compute them send them to all eight CTAs, and every CTA forms all rotations
// itself: one cluster barrier a round, and V's rows (which need no exchange)
// are rotated while it completes.
//
// Results equal k_jacobi's bit for bit, but for the order of the sums in the
// stopping test.  Random matrices of n = 64, 96, 128, 160, whole call: 544 ->
// 519, 1283 -> 857, 2543 -> 1616, 4596 -> 2083 us (k_jacobi -> here); what is
// left is the latency of a round, about a microsecond of it the barrier with
// the stores under way and the rotations' divisions and square roots.
// ---------------------------------------------------------------------------
constexpr int JC = 8;                          // CTAs
constexpr int JT = 512;                        // threads of each
constexpr int JH = SMALL_MAX / 2;              // pairs
constexpr int JW = (JH + JC - 1) / JC;         // pair positions of a CTA
constexpr int JR = (SMALL_MAX + JC - 1) / JC;  // rows of V of a CTA
constexpr int JLD = SMALL_MAX;                 // rows of a column of A, columns of a row of V
// From this size on: k_jacobi is ahead at n = 48 (321 against 363 us) and 56
// (396, 420), level at 64.  (A CTA needs two positions: n >= 31.)
constexpr int JMIN = 64;

__device__ __forceinline__ uint32_t s_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t at_cta(uint32_t a, int cta) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(cta));
  return r;
}
__device__ __forceinline__ void put(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

struct JCol {        // a column of one of the CTA's pairs in a round
  const float* src;
  uint32_t dst;      // where it goes (shared::cluster address)
  int partner;       // row position of the next partner, if that is the smaller index: 2 position + (it is the larger
                     // of its present pair); -2 if not
  uint32_t diag;     // offsets in the next round's elements: its diagonal,
  uint32_t off;      // and the one with its partner
};

struct JShared {
  float P[(JW + 1) * JLD], Q[(JW + 1) * JLD], F[JLD];   // rings, and the Q of position 0
  float V[JR * JLD];
  float next[2][3][JH];   // app, apq, aqq of every pair, by the round's parity
  float2 cs[JH];
  JCol tab[2][JW][2];     // [parity][pair][smaller, larger index]
  float norm[JC][2];
  float red[2][JT / 32];
  float diag[SMALL_MAX];
  int rank[SMALL_MAX];
};

__global__ void __cluster_dims__(JC, 1, 1) __launch_bounds__(JT)
    k_jacobi_cluster(int n, const double* __restrict__ Ag, int lda, double* __restrict__ w, double* __restrict__ Vg,
                     int max_sweeps, float off_tol) {
  __shared__ JShared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int N2 = (n + 1) & ~1, H = N2 / 2, M1 = N2 - 1;   // odd n: index n is a dummy of zeros
  const int cta = blockIdx.x;
  const int a = cta * H / JC, b = (cta + 1) * H / JC, W = b - a;
  const int WL = cta > 0 ? a - (cta - 1) * H / JC : 0, WR = cta < JC - 1 ? (cta + 2) * H / JC - b : 0;
  const int v0 = cta * n / JC, vrows = (cta + 1) * n / JC - v0;

  // index of a position in round r
  auto index_at = [&](bool q, int k, int r) {
    const int x = !q ? r + k : r - k;
    return q && k == 0 ? M1 : x < 0 ? x + M1 : x >= M1 ? x - M1 : x;
  };
  // rounds so far, modulo the sizes of the rings
  struct Turn {
    int m, at;
    __device__ void next() { at = at + 1 == m ? 0 : at + 1; }
    __device__ int add(int x) const { return at + x >= m ? at + x - m : at + x; }   // (at + x) mod m, 0 <= x < m
    __device__ int sub(int x) const { return x >= at ? x - at : x - at + m; }       // (x - at) mod m
  };
  Turn tp{W + 1, 0}, tq{cta > 0 ? W + 1 : W, 0}, tl{WL + 1, 0}, tr{WR + 1, 0};
  auto slot = [&](bool q, int j) -> float* {   // column of local position j
    if (!q) return sh.P + tp.add(j) * JLD;
    if (cta > 0) return sh.Q + tq.sub(j) * JLD;
    return j == 0 ? sh.F : sh.Q + tq.sub(j - 1) * JLD;
  };
  // the column of kind q at local position j in round r: its entry in t
  auto describe = [&](int q, int j, int r, JCol (*t)[2]) {
    const int l = a + j, i = index_at(q, l, r);
    JCol c;
    c.src = slot(q, j);
    c.dst = s_u32(c.src);
    bool nq = q;   // where the column is in the next round
    int nk = l;
    if (q == 0) {
      if (l == 0) {
        nq = true;
        nk = 1;
        c.dst = s_u32(sh.Q + tq.sub(W - 1) * JLD);
      } else {
        nk = l - 1;
        if (j == 0) c.dst = at_cta(s_u32(sh.P + tl.add(WL) * JLD), cta - 1);
      }
    } else if (l > 0) {
      if (l == H - 1) {
        nq = false;
        c.dst = s_u32(sh.P + tp.add(W) * JLD);
      } else {
        nk = l + 1;
        if (j == W - 1) c.dst = at_cta(s_u32(sh.Q + tr.sub(WR) * JLD), cta + 1);
      }
    }
    // its partner there, and that index's present position
    const int y = index_at(!nq, nk, r + 1 == M1 ? 0 : r + 1);
    int ky = 0;
    bool qy = true;
    if (y != M1) {
      const int d = y >= r ? y - r : y - r + M1;
      qy = d >= H;
      ky = qy ? M1 - d : d;
    }
    c.partner = y < i ? 2 * ky + (y > index_at(!qy, ky, r)) : -2;
    c.diag = 4 * ((i < y ? 0 : 2 * JH) + nk);
    c.off = 4 * (JH + nk);
    t[j][i > index_at(!q, l, r)] = c;
  };

  for (int e = tid; e < 2 * W * N2; e += JT) {
    const int i = e / (2 * W), c = e - i * (2 * W), j = c >> 1;
    const int col = index_at(c & 1, a + j, 0);
    slot(c & 1, j)[i] = i < n && col < n ? (float)Ag[(long long)i * lda + col] : 0.f;
  }
  for (int e = tid; e < vrows * N2; e += JT) {
    const int i = e / N2, j = e - i * N2;
    sh.V[i * JLD + j] = v0 + i == j ? 1.f : 0.f;
  }
  if (tid < H) {
    const int x = index_at(false, tid, 0), y = index_at(true, tid, 0), p = min(x, y), q = max(x, y);
    sh.next[0][0][tid] = (float)Ag[(long long)p * lda + p];
    sh.next[0][1][tid] = q < n ? (float)Ag[(long long)p * lda + q] : 0.f;
    sh.next[0][2][tid] = q < n ? (float)Ag[(long long)q * lda + q] : 0.f;
  }
  if (tid < 2 * W) describe(tid & 1, tid >> 1, 0, sh.tab[0]);
  cluster_arrive();   // every CTA is there, with its columns
  cluster_wait();

  // this warp's share of a round: row (or column) positions 32 kc + lane, every ng-th pair or row of V
  const int KC = (H + 31) / 32, kc = warp % KC, ng = (JT / 32) / KC, wg = warp / KC;
  const int k = kc * 32 + lane;
  const bool on = k < H && wg < ng;
  int R = 0;   // rounds so far
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    float off = 0.f, tot = 0.f;
    for (int c = warp; c < 2 * W; c += JT / 32) {
      const float* col = slot(c & 1, c >> 1);
      const int ic = index_at(c & 1, a + (c >> 1), 0);   // (a sweep begins as round 0)
      for (int i = lane; i < N2; i += 32) {
        const float v = col[i];
        tot += v * v;
        if (i != ic) off += v * v;
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    if (lane == 0) { sh.red[0][warp] = off; sh.red[1][warp] = tot; }
    __syncthreads();
    if (tid < 2 * JC) {
      float t = 0.f;
      for (int q = 0; q < JT / 32; ++q) t += sh.red[tid & 1][q];
      put(at_cta(s_u32(&sh.norm[cta][tid & 1]), tid >> 1), t);
    }
    cluster_arrive();
    cluster_wait();
    off = tot = 0.f;
    for (int c = 0; c < JC; ++c) { off += sh.norm[c][0]; tot += sh.norm[c][1]; }
    if (off <= off_tol * tot) break;   // (the same sums in every CTA)
    for (int r = 0; r < M1; ++r, ++R) {
      const int par = R & 1;
      if (tid < H) {
        float c, s;
        rotation(sh.next[par][0][tid], sh.next[par][1][tid], sh.next[par][2][tid], c, s);
        sh.cs[tid] = make_float2(c, s);
      }
      __syncthreads();
      int p = 0, q = 0;
      float ck = 1.f, sk = 0.f;
      if (on) {
        const int x = index_at(false, k, r), y = index_at(true, k, r);
        p = min(x, y);
        q = max(x, y);
        ck = sh.cs[k].x;
        sk = sh.cs[k].y;
        const uint32_t nx = s_u32(sh.next[par ^ 1]);
        auto send = [&](uint32_t o, float v) {
#pragma unroll
          for (int d = 0; d < JC; ++d) put(at_cta(nx + o, d), v);
        };
        for (int j = wg; j < W; j += ng) {
          const JCol u = sh.tab[par][j][0], v = sh.tab[par][j][1];
          const float2 cl = sh.cs[a + j];
          Block2 x{u.src[p], v.src[p], u.src[q], v.src[q]};
          x.rotate(ck, sk, cl.x, cl.y);
          put(u.dst + 4 * p, x.x00);
          put(v.dst + 4 * p, x.x01);
          put(u.dst + 4 * q, x.x10);
          put(v.dst + 4 * q, x.x11);
          if (k == a + j) {
            send(u.diag, x.x00);
            send(v.diag, x.x11);
          }
          if (k == u.partner >> 1) send(u.off, u.partner & 1 ? x.x10 : x.x00);
          if (k == v.partner >> 1) send(v.off, v.partner & 1 ? x.x11 : x.x01);
        }
      }
      cluster_arrive();
      if (on && q < n)
        for (int i = wg; i < vrows; i += ng) {
          float* v = sh.V + i * JLD;
          const float vp = v[p], vq = v[q];
          v[p] = ck * vp - sk * vq;
          v[q] = sk * vp + ck * vq;
        }
      tp.next(), tq.next(), tl.next(), tr.next();
      if (tid >= JT - 32 && lane < 2 * W) describe(lane & 1, lane >> 1, r + 1 == M1 ? 0 : r + 1, sh.tab[par ^ 1]);
      cluster_wait();
    }
  }
  // ascending order by rank of the diagonal, which the elements of the next round hold
  if (tid < H) {
    const int x = index_at(false, tid, 0), y = index_at(true, tid, 0);
    sh.diag[min(x, y)] = sh.next[R & 1][0][tid];
    sh.diag[max(x, y)] = sh.next[R & 1][2][tid];
  }
  __syncthreads();
  for (int j = tid; j < n; j += JT) {
    const float dj = sh.diag[j];
    int rank = 0;
    for (int l = 0; l < n; ++l) {
      const float dl = sh.diag[l];
      rank += (dl < dj) || (dl == dj && l < j);
    }
    sh.rank[j] = rank;
    if (cta == 0) w[rank] = (double)dj;
  }
  __syncthreads();
  for (int e = tid; e < vrows * n; e += JT) {
    const int i = e / n, j = e - i * n;
    Vg[(long long)(v0 + i) * n + sh.rank[j]] = (double)sh.V[i * JLD + j];
  }
}

}  // namespace

cudaError_t jacobi_f32(int n, const double* A, int lda, double* w, double* V, cudaStream_t s) {
  if (n <= 0 || n > SMALL_MAX) return cudaErrorInvalidValue;
  // converged to off(A) <= 1e-12 |A|^2: the FP64 refinement needs a start
  // this close (a stop at 1e-7 left backward errors up to 5e-2)
  constexpr int max_sweeps = 30;
  constexpr float off_tol = 1e-12f;
  if (n >= JMIN) {
    k_jacobi_cluster<<<JC, JT, 0, s>>>(n, A, lda, w, V, max_sweeps, off_tol);
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
