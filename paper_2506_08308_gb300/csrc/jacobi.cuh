// Cyclic Jacobi on a cluster of eight CTAs (see jacobi.cu for the ordering).
#pragma once

#include <cstdint>

#include "dense.cuh"

namespace bdg {

namespace {

// c x - s y and s x + c y, with the products that are rounded before the sum
// fixed: the kernels that share a rotation agree bit for bit.
__device__ __forceinline__ float minus2(float c, float x, float s, float y) {
  return __fmaf_rn(c, x, -__fmul_rn(s, y));
}
__device__ __forceinline__ float plus2(float s, float x, float c, float y) {
  return __fmaf_rn(s, x, __fmul_rn(c, y));
}
__device__ __forceinline__ double minus2(double c, double x, double s, double y) {
  return __fma_rn(c, x, -__dmul_rn(s, y));
}
__device__ __forceinline__ double plus2(double s, double x, double c, double y) {
  return __fma_rn(s, x, __dmul_rn(c, y));
}

// One 2 x 2 block (rows p < q, columns u < v): rows first, then columns, as
// the two one-sided updates would do.
template <typename T>
struct Block2 {
  T x00, x01, x10, x11;
  __device__ __forceinline__ void rotate(T ck, T sk, T cl, T sl) {
    const T r00 = minus2(ck, x00, sk, x10), r01 = minus2(ck, x01, sk, x11);
    const T r10 = plus2(sk, x00, ck, x10), r11 = plus2(sk, x01, ck, x11);
    x00 = minus2(cl, r00, sl, r01);
    x01 = plus2(sl, r00, cl, r01);
    x10 = minus2(cl, r10, sl, r11);
    x11 = plus2(sl, r10, cl, r11);
  }
};

// ---------------------------------------------------------------------------
// One CTA is bound by the round: its shared-memory traffic and issue in FP32,
// its FP64 pipe in FP64 (n^2/4 blocks and n^2/2 rotations of V), a thousand
// rounds one after another.  Here a CTA holds the columns of A of its share of
// the round's pair positions, and its share of the rows of V.
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
// Results equal those of one CTA bit for bit, but for the order of the sums in
// the stopping test.
// ---------------------------------------------------------------------------
constexpr int JC = 8;   // CTAs of a cluster

__device__ __forceinline__ uint32_t s_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t at_cta(uint32_t a, int cta) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(cta));
  return r;
}
__device__ __forceinline__ void put(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void put(uint32_t a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <typename T>
struct JCol {        // a column of one of the CTA's pairs in a round
  const T* src;
  uint32_t dst;      // where it goes (shared::cluster address)
  int partner;       // row position of the next partner, if that is the smaller index: 2 position + (it is the larger
                     // of its present pair); -2 if not
  uint32_t diag;     // offsets in the next round's elements: its diagonal,
  uint32_t off;      // and the one with its partner
};

// n <= NMAX on NT threads a CTA
template <typename T, int NMAX, int NT>
struct JShared {
  static constexpr int JH = NMAX / 2;              // pairs
  static constexpr int JW = (JH + JC - 1) / JC;    // pair positions of a CTA
  static constexpr int JR = (NMAX + JC - 1) / JC;  // rows of V of a CTA
  static constexpr int JLD = NMAX;                 // rows of a column of A, columns of a row of V
  T P[(JW + 1) * JLD], Q[(JW + 1) * JLD], F[JLD];  // rings, and the Q of position 0
  T V[JR * JLD];
  T next[2][3][JH];       // app, apq, aqq of every pair, by the round's parity
  T cs[JH][2];
  JCol<T> tab[2][JW][2];  // [parity][pair][smaller, larger index]
  T norm[JC][2];
  T red[2][NT / 32];
};

// The sweeps on CTA `cta` of the cluster, for the matrix elem(i, j) of order n
// >= 31 (two positions a CTA): rotate(app, apq, aqq, c, s) gives the
// rotations, done(off, tot) the end, from the sums of squares off the diagonal
// and in all (the same values in every CTA).  Leaves this CTA's rows of V in
// sh.V, and returns the parity at which sh.next holds the diagonal (in the
// order of round 0).
template <typename T, int NMAX, int NT, class Elem, class Rotate, class Done>
__device__ int jacobi_sweeps(JShared<T, NMAX, NT>& sh, int n, int cta, int max_sweeps, Elem elem, Rotate rotate,
                             Done done) {
  constexpr int JH = NMAX / 2, JLD = NMAX;
  constexpr uint32_t SZ = sizeof(T);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int N2 = (n + 1) & ~1, H = N2 / 2, M1 = N2 - 1;   // odd n: index n is a dummy of zeros
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
  auto slot = [&](bool q, int j) -> T* {   // column of local position j
    if (!q) return sh.P + tp.add(j) * JLD;
    if (cta > 0) return sh.Q + tq.sub(j) * JLD;
    return j == 0 ? sh.F : sh.Q + tq.sub(j - 1) * JLD;
  };
  // the column of kind q at local position j in round r: its entry in t
  auto describe = [&](int q, int j, int r, JCol<T> (*t)[2]) {
    const int l = a + j, i = index_at(q, l, r);
    JCol<T> c;
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
    c.diag = SZ * ((i < y ? 0 : 2 * JH) + nk);
    c.off = SZ * (JH + nk);
    t[j][i > index_at(!q, l, r)] = c;
  };

  for (int e = tid; e < 2 * W * N2; e += NT) {
    const int i = e / (2 * W), c = e - i * (2 * W), j = c >> 1;
    const int col = index_at(c & 1, a + j, 0);
    slot(c & 1, j)[i] = i < n && col < n ? elem(i, col) : (T)0;
  }
  for (int e = tid; e < vrows * N2; e += NT) {
    const int i = e / N2, j = e - i * N2;
    sh.V[i * JLD + j] = v0 + i == j ? (T)1 : (T)0;
  }
  if (tid < H) {
    const int x = index_at(false, tid, 0), y = index_at(true, tid, 0), p = min(x, y), q = max(x, y);
    sh.next[0][0][tid] = elem(p, p);
    sh.next[0][1][tid] = q < n ? elem(p, q) : (T)0;
    sh.next[0][2][tid] = q < n ? elem(q, q) : (T)0;
  }
  if (tid < 2 * W) describe(tid & 1, tid >> 1, 0, sh.tab[0]);
  cluster_arrive();   // every CTA is there, with its columns
  cluster_wait();

  // this warp's share of a round: row (or column) positions 32 kc + lane, every ng-th pair or row of V
  const int KC = (H + 31) / 32, kc = warp % KC, ng = (NT / 32) / KC, wg = warp / KC;
  const int k = kc * 32 + lane;
  const bool on = k < H && wg < ng;
  int R = 0;   // rounds so far
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    T off = 0, tot = 0;
    for (int c = warp; c < 2 * W; c += NT / 32) {
      const T* col = slot(c & 1, c >> 1);
      const int ic = index_at(c & 1, a + (c >> 1), 0);   // (a sweep begins as round 0)
      for (int i = lane; i < N2; i += 32) {
        const T v = col[i];
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
      T t = 0;
      for (int q = 0; q < NT / 32; ++q) t += sh.red[tid & 1][q];
      put(at_cta(s_u32(&sh.norm[cta][tid & 1]), tid >> 1), t);
    }
    cluster_arrive();
    cluster_wait();
    off = tot = 0;
    for (int c = 0; c < JC; ++c) { off += sh.norm[c][0]; tot += sh.norm[c][1]; }
    if (done(off, tot)) break;   // (the same sums in every CTA)
    for (int r = 0; r < M1; ++r, ++R) {
      const int par = R & 1;
      if (tid < H) {
        T c, s;
        rotate(sh.next[par][0][tid], sh.next[par][1][tid], sh.next[par][2][tid], c, s);
        sh.cs[tid][0] = c;
        sh.cs[tid][1] = s;
      }
      __syncthreads();
      int p = 0, q = 0;
      T ck = 1, sk = 0;
      if (on) {
        const int x = index_at(false, k, r), y = index_at(true, k, r);
        p = min(x, y);
        q = max(x, y);
        ck = sh.cs[k][0];
        sk = sh.cs[k][1];
        const uint32_t nx = s_u32(sh.next[par ^ 1]);
        auto send = [&](uint32_t o, T v) {
#pragma unroll
          for (int d = 0; d < JC; ++d) put(at_cta(nx + o, d), v);
        };
        for (int j = wg; j < W; j += ng) {
          const JCol<T> u = sh.tab[par][j][0], v = sh.tab[par][j][1];
          Block2<T> x{u.src[p], v.src[p], u.src[q], v.src[q]};
          x.rotate(ck, sk, sh.cs[a + j][0], sh.cs[a + j][1]);
          put(u.dst + SZ * p, x.x00);
          put(v.dst + SZ * p, x.x01);
          put(u.dst + SZ * q, x.x10);
          put(v.dst + SZ * q, x.x11);
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
          T* v = sh.V + i * JLD;
          const T vp = v[p], vq = v[q];
          v[p] = minus2(ck, vp, sk, vq);
          v[q] = plus2(sk, vp, ck, vq);
        }
      tp.next(), tq.next(), tl.next(), tr.next();
      if (tid >= NT - 32 && lane < 2 * W) describe(lane & 1, lane >> 1, r + 1 == M1 ? 0 : r + 1, sh.tab[par ^ 1]);
      cluster_wait();
    }
  }
  return R & 1;
}

}  // namespace

}  // namespace bdg
