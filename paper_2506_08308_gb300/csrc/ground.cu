// Ground state on S_M (eq. groundDef) on the device, FP64.
//
// Phase 1, normalized gradient flow: with N(Phi) Phi the non-kinetic part of
// H Phi (eq. NLEP: trap, density, spin and Zeeman terms) and c = 1/tau +
// alpha, alpha >= max_x (V + (beta_n + |beta_s|) rho) + |p| + |q|,
//     (c - 1/2 Lap) Phi* = c Phi - N(Phi) Phi,   Phi <- P_SM(Phi*),
// the kinetic term implicit and diagonal in Fourier space (Section 3.1).
// Phase 2, inexact Newton on S_M: with the multipliers (mu + lambda S_z) of
// the least-squares fit H Phi ~ (mu + lambda S_z) Phi, solve
//     P H_+ P d = -P (H Phi - (mu + lambda S_z) Phi)
// by preconditioned CG on the tangent space {<Phi, d> = <S_z Phi, d> = 0}
// (P its projector, preconditioner P (c - 1/2 Lap)^-1 P), H_+ = A + B the
// Hessian of the Lagrangian (eqs. def_A + def_B at a real Phi), then
// Phi <- P_SM(Phi + d).  A Newton step that does not lower the residual
// hands back to 50 flow steps.
// Newton converges to any stationary point.  A converged state is therefore
// tested for negative curvature of the energy on S_M along the directions
// that move population between spin components; a saddle (e.g. the
// antiferromagnetic state when q > 0 makes the polar state lower) is left
// along that direction and the flow resumes (at most three times).
//
// P_SM scales the components, phi_j <- sigma_j phi_j, to mass 1 and
// magnetization M with sigma_1 sigma_-1 = sigma_0^2 (closed form).
//
// Spinors are kept as two complex planes, (phi_1, phi_-1) and (phi_0, 0): the
// Fourier operators are real and even, so they act on real and imaginary
// parts alike, and two planes of transforms serve the three components (the
// imaginary part of the second plane holds rounding only and is never read).
// A coarse grid's iteration is a chain of short kernels: every scalar of a
// step (the norms of P_SM, mu, the CG coefficients) is formed by the kernel
// that needs it from per-CTA partial sums, added in a fixed order, and the
// host reads one result record a step, one step behind the device: the next
// step is queued before the record of the last is looked at (its result is
// dropped if that record ends the phase).  The flow's own equation gives the
// Laplacian of its result, and a CG step carries -1/2 Lap p along with p, so
// that a step of either kind takes one k-space solve and no other transform.
// 64^2, about 1600 flow and 700 CG steps: 600 ms with three host waits, 16
// launches and five transform passes a flow step, 160 ms with one wait behind
// the device, seven launches and three passes, of which the passes take half;
// 256^2: 1.13 s -> 0.26 s.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "apply_impl.cuh"
#include "blas.cuh"
#include "kdiag.cuh"
#include "plan.cuh"

namespace bdg {
namespace {

// Small CTAs: an FP64 warp instruction holds its quarter of the SM for 64
// clocks, so a coarse grid's points go to as many SMs as there are.
constexpr int NT = 128;
constexpr int MAX_BLOCKS = 608;
constexpr int NSUM = 6;  // sums per partial record
unsigned nblk(long long n) {
  long long b = (n + NT - 1) / NT;
  return (unsigned)(b > MAX_BLOCKS ? MAX_BLOCKS : (b < 1 ? 1 : b));
}
#define GS_LOOP(i, n) \
  for (long long i = (long long)blockIdx.x * NT + threadIdx.x; i < (n); i += (long long)gridDim.x * NT)

struct GsCoef {
  double beta_n, beta_s, p, q;
};

// N(Phi) Phi (trap, density, spin and Zeeman terms).  For real Phi = (a, b,
// c): F_x = sqrt2 b (a + c), F_z = a^2 - c^2, F_y = 0, and (F.S) Phi = (b^2
// (a+c) + F_z a, b (a+c)^2, b^2 (a+c) - F_z c); Zeeman diag(q - p, 0, q + p).
__device__ __forceinline__ void nonkinetic(double a, double b, double c, double V, const GsCoef& k, double& n1,
                                           double& n0, double& nm) {
  const double rho = a * a + b * b + c * c, fz = a * a - c * c, s = a + c;
  const double w = V + k.beta_n * rho;
  n1 = w * a + k.beta_s * (b * b * s + fz * a) + (k.q - k.p) * a;
  n0 = w * b + k.beta_s * (b * s * s);
  nm = w * c + k.beta_s * (b * b * s - fz * c) + (k.q + k.p) * c;
}

// Block sums of Q per-thread values into part[q * gridDim.x + blockIdx.x].
template <int Q>
__device__ __forceinline__ void put_sums(const double (&v)[Q], double* __restrict__ part) {
  __shared__ double red[Q][NT / 32];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    double s = v[q];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[q][threadIdx.x >> 5] = s;
  }
  __syncthreads();
  if (threadIdx.x < Q) {
    double s = 0.0;
    for (int w = 0; w < NT / 32; ++w) s += red[threadIdx.x][w];
    part[threadIdx.x * gridDim.x + blockIdx.x] = s;
  }
  static_assert(Q <= NT, "one thread per quantity");
}
// Totals of Q quantities over nb partial sums, in a fixed order, in every CTA
// (the warps share the quantities).
template <int Q>
__device__ __forceinline__ void get_sums(const double* __restrict__ part, int nb, double (&t)[Q]) {
  __shared__ double tot[Q];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int q = warp; q < Q; q += NT / 32) {
    double s = 0.0;
    for (int b = lane; b < nb; b += 32) s += part[q * nb + b];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) tot[q] = s;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < Q; ++q) t[q] = tot[q];
  __syncthreads();  // the next call writes tot
}

// Result record of a flow step: 0 largest residual, 1..3 mu (1, 0, -1), 4
// set when no component can be scaled onto S_M.  Of a CG step: 5 (p, A p), 6
// (r, r).
constexpr int REC = 8;

// atomic max of non-negative doubles (NaN counts as the largest) through
// their bit patterns
__device__ void atomic_max_pos(double* addr, double v) {
  atomicMax(reinterpret_cast<unsigned long long*>(addr), (unsigned long long)__double_as_longlong(v));
}
__device__ void block_atomic_max(double v, double* out) {
  __shared__ double red[NT / 32];
  auto larger = [](double a, double b) { return isnan(a) || a > b ? a : b; };
  for (int o = 16; o > 0; o >>= 1) v = larger(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < NT / 32; ++q) v = larger(v, red[q]);
    atomic_max_pos(out, fabs(v));
  }
}

// |phi_j|^2 (plain grid sums) of components 1, 0, -1
__global__ void __launch_bounds__(NT) k_gs_norms(const double2* __restrict__ phi, long long np, double* part) {
  double v[3] = {0.0, 0.0, 0.0};
  GS_LOOP(i, np) {
    const double2 a = phi[i];
    const double b = phi[np + i].x;
    v[0] = fma(a.x, a.x, v[0]);
    v[1] = fma(b, b, v[1]);
    v[2] = fma(a.y, a.y, v[2]);
  }
  put_sums(v, part);
}

// Factors of P_SM from the sums of k_gs_norms: sum_j sigma_j^2 N_j = 1,
// sigma_1^2 N_1 - sigma_-1^2 N_-1 = M, sigma_1 sigma_-1 = sigma_0^2, N_j = h^d
// |phi_j|^2.  Clears the result record.
struct Scale3 {
  double s1, s0, sm;
};
__device__ __forceinline__ Scale3 project_factors(const double* part, int nb, double M, double cell, double* rec) {
  double N[3];
  get_sums(part, nb, N);
  const double N1 = N[0] * cell, N0 = N[1] * cell, Nm = N[2] * cell;
  const double sden = N0 + sqrt(M * M * N0 * N0 + 4.0 * (1.0 - M * M) * N1 * Nm);
  const double s = (1.0 - M * M) / sden;
  Scale3 f{0.0, sqrt(s), 0.0};
  if (N1 > 0) f.s1 = sqrt(fmax(1.0 + M - s * N0, 0.0) / (2.0 * N1));
  if (Nm > 0) f.sm = sqrt(fmax(1.0 - M - s * N0, 0.0) / (2.0 * Nm));
  if (N1 == 0 && Nm == 0) f.s0 = 1.0 / sqrt(N0);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    rec[0] = 0.0;
    rec[4] = sden > 0 ? 0.0 : 1.0;
  }
  return f;
}
__global__ void __launch_bounds__(NT) k_gs_project(double2* __restrict__ phi, long long np, const double* part, int nb,
                                                   double M, double cell, double* rec) {
  const Scale3 f = project_factors(part, nb, M, cell, rec);
  GS_LOOP(i, np) {
    const double2 a = phi[i];
    phi[i] = make_double2(a.x * f.s1, a.y * f.sm);
    phi[np + i] = make_double2(phi[np + i].x * f.s0, 0.0);
  }
}

// H phi = t + N(phi) phi at one point (t: -1/2 Lap phi there), and the sums
// (phi_j, (H phi)_j) and |phi_j|^2, j = 1, 0, -1
__device__ __forceinline__ void hphi_point(double2 p, double b, double2 t, double t0, double V, const GsCoef& k,
                                           double2& h, double& h0, double (&v)[6]) {
  double n1, n0, nm;
  nonkinetic(p.x, b, p.y, V, k, n1, n0, nm);
  h = make_double2(t.x + n1, t.y + nm);
  h0 = t0 + n0;
  v[0] = fma(p.x, h.x, v[0]);
  v[1] = fma(b, h0, v[1]);
  v[2] = fma(p.y, h.y, v[2]);
  v[3] = fma(p.x, p.x, v[3]);
  v[4] = fma(b, b, v[4]);
  v[5] = fma(p.y, p.y, v[5]);
}
// y: -1/2 Lap phi on entry, H phi on exit
__global__ void __launch_bounds__(NT) k_gs_hphi(const double2* __restrict__ phi, const double* __restrict__ V,
                                                long long np, GsCoef k, double2* __restrict__ y, double* part) {
  double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  GS_LOOP(i, np) {
    double2 h;
    double h0;
    hphi_point(phi[i], phi[np + i].x, y[i], y[np + i].x, V[i], k, h, h0, v);
    y[i] = h;
    y[np + i] = make_double2(h0, 0.0);
  }
  put_sums(v, part);
}
// The projection of a flow step together with H phi: phi* solves (c - 1/2
// Lap) phi* = rhs, so -1/2 Lap phi = sigma (rhs - c phi*) without transforms
// (to about eps c |phi|; close to convergence the transforms are taken).
__global__ void __launch_bounds__(NT) k_gs_project_h(double2* __restrict__ phi, const double2* __restrict__ rhs,
                                                     double c, const double* __restrict__ V, long long np, GsCoef k,
                                                     const double* part, int nb, double M, double cell,
                                                     double2* __restrict__ y, double* part_h, double* rec) {
  const Scale3 f = project_factors(part, nb, M, cell, rec);
  double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  GS_LOOP(i, np) {
    const double2 a = phi[i], r = rhs[i];
    const double a0 = phi[np + i].x, r0 = rhs[np + i].x;
    const double2 p = make_double2(a.x * f.s1, a.y * f.sm);
    const double b = a0 * f.s0;
    phi[i] = p;
    phi[np + i] = make_double2(b, 0.0);
    double2 h;
    double h0;
    hphi_point(p, b, make_double2(f.s1 * fma(-c, a.x, r.x), f.sm * fma(-c, a.y, r.y)), f.s0 * fma(-c, a0, r0), V[i], k,
               h, h0, v);
    y[i] = h;
    y[np + i] = make_double2(h0, 0.0);
  }
  put_sums(v, part_h);
}

// mu by eq. chem-formula from the sums of k_gs_hphi (vanishing components
// filled from mu_1 + mu_-1 = 2 mu_0), max |H phi - mu phi| into rec[0], and
// the right-hand side of the next flow step, rhs = cst phi - N(phi) phi.
__global__ void __launch_bounds__(NT) k_gs_residual(const double2* __restrict__ phi, const double2* __restrict__ hphi,
                                                    const double* __restrict__ V, long long np, GsCoef k,
                                                    const double* part, int nb, double cst, double2* __restrict__ rhs,
                                                    double* rec) {
  double v[6], mu[3];
  get_sums(part, nb, v);
  bool z[3];
  const double tiny = 1e-20 * (v[3] + v[4] + v[5]);  // vanishing components, relative to |Phi|^2
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    z[j] = v[3 + j] < tiny;
    mu[j] = z[j] ? (double)NAN : v[j] / v[3 + j];
  }
  if (z[1] && !z[0] && !z[2]) mu[1] = 0.5 * (mu[0] + mu[2]);
  else if (z[0] && z[2] && !z[1]) mu[0] = mu[2] = mu[1];
  else if (z[0] && !z[2] && !z[1]) mu[0] = 2 * mu[1] - mu[2];
  else if (z[2] && !z[0] && !z[1]) mu[2] = 2 * mu[1] - mu[0];
  if (blockIdx.x == 0 && threadIdx.x < 3) rec[1 + threadIdx.x] = threadIdx.x == 0 ? mu[0] : threadIdx.x == 1 ? mu[1] : mu[2];
  double m = 0.0;
  GS_LOOP(i, np) {
    const double2 p = phi[i], h = hphi[i];
    const double b = phi[np + i].x, h0 = hphi[np + i].x;
    const double r1 = fabs(h.x - mu[0] * p.x), r0 = fabs(h0 - mu[1] * b), rm = fabs(h.y - mu[2] * p.y);
    m = isnan(r1 + r0 + rm) ? (double)NAN : fmax(m, fmax(r1, fmax(r0, rm)));
    double n1, n0, nm;
    nonkinetic(p.x, b, p.y, V[i], k, n1, n0, nm);
    rhs[i] = make_double2(cst * p.x - n1, cst * p.y - nm);
    rhs[np + i] = make_double2(cst * b - n0, 0.0);
  }
  block_atomic_max(m, rec);
}
__global__ void __launch_bounds__(NT) k_gs_rhs(const double2* __restrict__ phi, const double* __restrict__ V,
                                               long long np, GsCoef k, double cst, double2* __restrict__ rhs) {
  GS_LOOP(i, np) {
    const double2 p = phi[i];
    const double b = phi[np + i].x;
    double n1, n0, nm;
    nonkinetic(p.x, b, p.y, V[i], k, n1, n0, nm);
    rhs[i] = make_double2(cst * p.x - n1, cst * p.y - nm);
    rhs[np + i] = make_double2(cst * b - n0, 0.0);
  }
}

// out[0] = max_x (V + (beta_n + |beta_s|) rho)
__global__ void __launch_bounds__(NT) k_gs_stab(const double2* __restrict__ phi, const double* __restrict__ V,
                                                long long np, double bsum, double* out) {
  double m = 0.0;
  GS_LOOP(i, np) {
    const double2 p = phi[i];
    const double b = phi[np + i].x;
    m = fmax(m, V[i] + bsum * (p.x * p.x + b * b + p.y * p.y));
  }
  block_atomic_max(m, out);
}

// up to six dot products over all components, as partial sums
struct DotSet {
  const double2* a[NSUM];
  const double2* b[NSUM];
};
template <int Q>
__global__ void __launch_bounds__(NT) k_gs_dots(DotSet d, long long np, double* part) {
  double v[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) v[q] = 0.0;
  GS_LOOP(i, np) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const double2 a = d.a[q][i], b = d.b[q][i];
      v[q] = fma(d.a[q][np + i].x, d.b[q][np + i].x, fma(a.y, b.y, fma(a.x, b.x, v[q])));
    }
  }
  put_sums(v, part);
}

// y = a x + b y over both planes (b = 0 does not read y)
__global__ void __launch_bounds__(NT) k_gs_axpby(long long len, double a, const double2* x, double b, double2* y) {
  GS_LOOP(e, len) {
    const double2 u = x[e];
    const double2 v = b != 0.0 ? y[e] : make_double2(0.0, 0.0);
    y[e] = make_double2(a * u.x + b * v.x, a * u.y + b * v.y);
  }
}

// r = m phi - H phi
__global__ void __launch_bounds__(NT) k_gs_negres(const double2* __restrict__ hphi, const double2* __restrict__ phi,
                                                  long long np, double m1, double m0, double mm,
                                                  double2* __restrict__ r) {
  GS_LOOP(i, np) {
    r[i] = make_double2(m1 * phi[i].x - hphi[i].x, mm * phi[i].y - hphi[i].y);
    r[np + i] = make_double2(m0 * phi[np + i].x - hphi[np + i].x, 0.0);
  }
}

// Directions that move population between the spin components of Phi = (a,
// b, c): kind 0: (0, (a + c) / sqrt2, 0) (from +-1 into 0), kind 1:
// (b, 0, b) / sqrt2 and kind 2: (b, 0, -b) / sqrt2 (from 0 into +-1).  At a
// stationary state that is not a minimum (e.g. the antiferromagnetic state
// (a, 0, a) when q > 0 makes the polar state lower) one of them has negative
// curvature.
__global__ void __launch_bounds__(NT) k_gs_transfer(const double2* __restrict__ phi, long long np, int kind,
                                                    double2* __restrict__ out) {
  const double h = 0.70710678118654752440;
  GS_LOOP(i, np) {
    const double2 p = phi[i];
    const double b = phi[np + i].x;
    out[i] = kind == 0 ? make_double2(0.0, 0.0) : make_double2(h * b, kind == 1 ? h * b : -h * b);
    out[np + i] = make_double2(kind == 0 ? h * (p.x + p.y) : 0.0, 0.0);
  }
}

// S_z Phi
__global__ void __launch_bounds__(NT) k_gs_sz(const double2* __restrict__ phi, long long np, double2* __restrict__ out) {
  GS_LOOP(i, np) {
    out[i] = make_double2(phi[i].x, -phi[i].y);
    out[np + i] = make_double2(0.0, 0.0);
  }
}

// Weighted-orthonormal basis of the normal directions of S_M (up to two).
struct Normal {
  const double2* z[2];
  const double2* tz[2];  // -1/2 Lap z
  int n;
  double cell;
};

// y = t + pointwise part of H_+ = A + B at phi with the multipliers in cp, on
// v (t: -1/2 Lap v, may be y); sums (v, y), (z_0, y), (z_1, y)
__global__ void __launch_bounds__(NT) k_gs_hplus(const double2* __restrict__ phi, const double* __restrict__ V,
                                                 long long np, Coupling<double> cp, const double2* __restrict__ v,
                                                 const double2* t, double2* y, Normal nz, double* part) {
  double s[3] = {0.0, 0.0, 0.0};
  GS_LOOP(i, np) {
    const double2 p = phi[i], x = v[i];
    const double x0 = v[np + i].x;
    Sym3<double> A, B;
    coupling_blocks<double>(dquad{p.x, phi[np + i].x, p.y, V[i]}, cp, A, B);
    const Sym3<double> P = sym_add(A, B, 1.0);
    const double2 tv = t[i];
    const double h1 = tv.x + (P.d0 * x.x + P.o01 * x0 + P.o02 * x.y);
    const double h0 = t[np + i].x + (P.o01 * x.x + P.d1 * x0 + P.o12 * x.y);
    const double hm = tv.y + (P.o02 * x.x + P.o12 * x0 + P.d2 * x.y);
    y[i] = make_double2(h1, hm);
    y[np + i] = make_double2(h0, 0.0);
    s[0] = fma(x0, h0, fma(x.y, hm, fma(x.x, h1, s[0])));
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (q < nz.n) {
        const double2 z = nz.z[q][i];
        s[1 + q] = fma(nz.z[q][np + i].x, h0, fma(z.y, hm, fma(z.x, h1, s[1 + q])));
      }
  }
  put_sums(s, part);
}

// CG update after A p = P H_+ p with the sums of k_gs_hplus: alpha = (r, z) /
// (p, A p); x += alpha p, r -= alpha A p; sum (r, r); rec[5] = (p, A p).
// rz: the partial record of (r, z) and its block count.
__global__ void __launch_bounds__(NT) k_gs_cg_xr(double2* __restrict__ x, double2* __restrict__ r,
                                                 const double2* __restrict__ p, const double2* __restrict__ ap,
                                                 long long np, Normal nz, const double* part, const double* rz, int nb,
                                                 double* part_rr, double* rec) {
  double s[3], t[1];
  get_sums(part, nb, s);
  get_sums(rz, nb, t);
  const double pap = s[0], a = pap > 0 ? t[0] / pap : 0.0;
  const double c0 = nz.n > 0 ? s[1] * nz.cell : 0.0, c1 = nz.n > 1 ? s[2] * nz.cell : 0.0;
  if (blockIdx.x == 0 && threadIdx.x == 0) rec[5] = pap;
  double v[1] = {0.0};
  GS_LOOP(e, 2 * np) {
    double2 q = ap[e];
    if (nz.n > 0) q = make_double2(fma(-c0, nz.z[0][e].x, q.x), fma(-c0, nz.z[0][e].y, q.y));
    if (nz.n > 1) q = make_double2(fma(-c1, nz.z[1][e].x, q.x), fma(-c1, nz.z[1][e].y, q.y));
    const double2 pv = p[e], xv = x[e], rv = r[e];
    x[e] = make_double2(fma(a, pv.x, xv.x), fma(a, pv.y, xv.y));
    const double2 n = make_double2(fma(-a, q.x, rv.x), fma(-a, q.y, rv.y));
    r[e] = n;
    v[0] = fma(n.x, n.x, v[0]);
    if (e < np) v[0] = fma(n.y, n.y, v[0]);
  }
  put_sums(v, part_rr);
}

// p <- P z + beta p with beta = (r, z) / (r, z)_old (first: beta = 0), from
// the sums (r, z), (z_0, z), (z_1, z); r is tangent, so (r, P z) = (r, z).
// Along with it tp = -1/2 Lap p: (c - 1/2 Lap) z = r gives -1/2 Lap z = r -
// c z.  rec[6] = (r, r) from part_rr (first: not set).
__global__ void __launch_bounds__(NT) k_gs_cg_p(double2* __restrict__ p, double2* __restrict__ tp,
                                                const double2* __restrict__ z, const double2* __restrict__ r, double c,
                                                long long np, Normal nz, const double* part, const double* rz_old,
                                                const double* part_rr, int nb, int first, double* rec) {
  double s[3], o[1], rr[1];
  get_sums(part, nb, s);
  get_sums(first ? part : rz_old, nb, o);
  get_sums(first ? part : part_rr, nb, rr);
  const double beta = first ? 0.0 : s[0] / o[0];
  const double c0 = nz.n > 0 ? s[1] * nz.cell : 0.0, c1 = nz.n > 1 ? s[2] * nz.cell : 0.0;
  if (!first && blockIdx.x == 0 && threadIdx.x == 0) rec[6] = rr[0];
  GS_LOOP(e, 2 * np) {
    double2 q = z[e];
    double2 t = make_double2(fma(-c, q.x, r[e].x), fma(-c, q.y, r[e].y));
    if (nz.n > 0) {
      q = make_double2(fma(-c0, nz.z[0][e].x, q.x), fma(-c0, nz.z[0][e].y, q.y));
      t = make_double2(fma(-c0, nz.tz[0][e].x, t.x), fma(-c0, nz.tz[0][e].y, t.y));
    }
    if (nz.n > 1) {
      q = make_double2(fma(-c1, nz.z[1][e].x, q.x), fma(-c1, nz.z[1][e].y, q.y));
      t = make_double2(fma(-c1, nz.tz[1][e].x, t.x), fma(-c1, nz.tz[1][e].y, t.y));
    }
    if (!first) {
      q = make_double2(fma(beta, p[e].x, q.x), fma(beta, p[e].y, q.y));
      t = make_double2(fma(beta, tp[e].x, t.x), fma(beta, tp[e].y, t.y));
    }
    p[e] = q;
    tp[e] = t;
  }
}

class GroundState {
 public:
  GroundState(bdg_plan_t plan, double M, cudaStream_t s) : plan_(plan), M_(M), s_(s) {
    np_ = plan->grid.npts;
    len_ = 2 * np_;
    nb_ = nblk(np_);
    cell_ = 1.0;
    for (int a = 0; a < plan->grid.dim; ++a) cell_ *= plan->grid.len[a] / plan->grid.n[a];
    k_.beta_n = plan->prm.beta_n;
    k_.beta_s = plan->prm.beta_s;
    k_.p = plan->prm.p;
    k_.q = plan->prm.q;
  }
  ~GroundState() {
    cudaStreamSynchronize(s_);   // a step queued ahead may still run
    for (void* p : bufs_) cudaFree(p);
    if (hrec_) cudaFreeHost(hrec_);
    for (auto e : ev_)
      if (e) cudaEventDestroy(e);
  }

  bdg_status init(const double* V, const double* phi0) {
    bdg_status st;
    const size_t vec = sizeof(double2) * (size_t)len_;
    if ((st = alloc(&V_, sizeof(double) * np_))) return st;
    double2** all[] = {&phi_[0], &phi_[1], &hphi_[0], &hphi_[1], &rhs_[0], &rhs_[1], &z_[0], &z_[1],
                       &tz_[0],  &tz_[1],  &cx_,      &cr_,      &cz_,     &cp_,     &tp_,   &cap_,  &trial_};
    for (double2** b : all)
      if ((st = alloc(b, vec))) return st;
    if ((st = alloc(&part_, sizeof(double) * PARTS * NSUM * MAX_BLOCKS)) || (st = alloc(&rec_, sizeof(double) * REC * 2)))
      return st;
    if (cudaMallocHost((void**)&hrec_, sizeof(double) * (REC * 2 + NSUM * MAX_BLOCKS)) != cudaSuccess) {
      cudaGetLastError();
      hrec_ = nullptr;
      return fail(plan_, BDG_ERR_NOMEM, "ground state: pinned allocation failed");
    }
    for (auto& e : ev_) BDG_CUDA_TRY(plan_, cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    BDG_CUDA_TRY(plan_, cudaMemcpyAsync(V_, V, sizeof(double) * np_, cudaMemcpyHostToDevice, s_));
    std::vector<double2> h(len_);
    for (long long i = 0; i < np_; ++i) {
      h[i] = make_double2(phi0[i], phi0[2 * np_ + i]);
      h[np_ + i] = make_double2(phi0[np_ + i], 0.0);
    }
    BDG_CUDA_TRY(plan_, cudaMemcpyAsync(phi_[0], h.data(), vec, cudaMemcpyHostToDevice, s_));
    BDG_CUDA_TRY(plan_, cudaStreamSynchronize(s_));
    cur_ = 0;
    return project(phi_[0], 0);
  }

  // the loop of phases 1 and 2; returns the residual through *res
  bdg_status run(double tol, int maxit, double* res, double mu[3], int* iters) {
    const double tau = 1.0, newton_start = 1e-3;
    int it = 0;
    double alpha = 0.0;
    bdg_status st = stab(phi_[cur_], &alpha);
    if (st) return st;
    double c = 1.0 / tau + alpha;
    if ((st = residual(phi_[cur_], cur_, c)) || (st = read(cur_, res, mu))) return st;
    int phase = 1, flow_left = 0, restarts = 0, flow_only = 0;
    double last = INFINITY;
    bool ahead = false;   // the flow step from cur_ is queued already
    while (it < maxit) {
      if (*res <= tol) {
        // a converged stationary state that is a saddle of the energy on S_M
        // is left along its negative-curvature direction and the flow resumes
        bool unstable = false;
        if (restarts >= 3) break;
        if ((st = stability(&unstable))) return st;
        if (!unstable) break;
        ++restarts;
        const double nphi = std::sqrt(dot1(phi_[cur_], phi_[cur_], &st));
        if (st) return st;
        k_gs_axpby<<<nblk(len_), NT, 0, s_>>>(len_, 1e-2 * nphi, cp_, 1.0, phi_[cur_]);
        BDG_CUDA_TRY(plan_, cudaGetLastError());
        if ((st = project(phi_[cur_], cur_)) || (st = residual(phi_[cur_], cur_, c)) || (st = read(cur_, res, mu)))
          return st;
        ahead = false;
        phase = 1;
        flow_left = 0;
        flow_only = 500;   // no Newton step until the unstable component has grown
        last = INFINITY;
        continue;
      }
      if (phase == 1 || flow_left > 0) {
        if (!ahead && (st = flow_step(cur_, c, *res))) return st;
        const int nxt = 1 - cur_;
        flow_left = flow_left > 0 ? flow_left - 1 : 0;
        ++it;
        // the step after this one, unless its c may change or it is not a flow step for certain
        ahead = it % 50 != 0 && it < maxit && (phase == 1 || flow_left > 0);
        if ((st = fetch(nxt))) return st;
        if (ahead && (st = flow_step(nxt, c, *res))) return st;
        if ((st = wait(nxt, res, mu))) return st;
        cur_ = nxt;
        if (it % 50 == 0) {
          if ((st = stab(phi_[cur_], &alpha))) return st;
          c = 1.0 / tau + alpha;
          if ((st = rhs(cur_, c))) return st;
          if (phase == 1 && flow_only == 0 && *res > 0.99 * last) phase = 2;
          last = *res;
        }
        const double mmax = std::max(std::fabs(mu[0]), std::max(std::fabs(mu[1]), std::fabs(mu[2])));
        if (flow_only > 0) {
          --flow_only;
          phase = 1;
        }
        if (phase == 1 && flow_only == 0 && *res < newton_start * (1.0 + mmax)) phase = 2;
      } else {
        // (a step queued ahead writes the other slot only, which the trial state may take over)
        ahead = false;
        int products = 0;
        if ((st = newton_step(c, &products))) return st;
        it += 1 + products;
        const int nxt = 1 - cur_;
        double rt, mt[3];
        BDG_CUDA_TRY(plan_, cudaMemcpyAsync(phi_[nxt], trial_, sizeof(double2) * len_, cudaMemcpyDeviceToDevice, s_));
        if ((st = project(phi_[nxt], nxt)) || (st = residual(phi_[nxt], nxt, c)) || (st = read(nxt, &rt, mt))) return st;
        if (rt < *res) {
          cur_ = nxt;
          *res = rt;
          for (int j = 0; j < 3; ++j) mu[j] = mt[j];
        } else {
          flow_left = 50;
        }
      }
      if (!std::isfinite(*res)) return fail(plan_, BDG_ERR_NAN, "ground state iteration produced NaN");
    }
    *iters = it;
    return BDG_OK;
  }

  bdg_status download(double* phi) {
    std::vector<double2> h(len_);
    BDG_CUDA_TRY(plan_, cudaMemcpyAsync(h.data(), phi_[cur_], sizeof(double2) * len_, cudaMemcpyDeviceToHost, s_));
    BDG_CUDA_TRY(plan_, cudaStreamSynchronize(s_));
    for (long long i = 0; i < np_; ++i) {
      phi[i] = h[i].x;
      phi[np_ + i] = h[np_ + i].x;
      phi[2 * np_ + i] = h[i].y;
    }
    return BDG_OK;
  }

 private:
  bdg_status alloc(void* pp, size_t bytes) {
    void** p = (void**)pp;
    if (cudaMalloc(p, bytes) != cudaSuccess) {
      cudaGetLastError();
      *p = nullptr;
      return fail(plan_, BDG_ERR_NOMEM, "ground state: device allocation failed");
    }
    bufs_.push_back(*p);
    return BDG_OK;
  }
  double* part(int i) { return part_ + (size_t)i * NSUM * MAX_BLOCKS; }

  // dot products summed on the host
  template <int Q>
  bdg_status dots(const DotSet& d, double (&out)[Q]) {
    k_gs_dots<Q><<<nb_, NT, 0, s_>>>(d, np_, part(PART_HOST));
    BDG_CUDA_TRY(plan_, cudaGetLastError());
    double* h = hrec_ + 2 * REC;
    BDG_CUDA_TRY(plan_, cudaMemcpyAsync(h, part(PART_HOST), sizeof(double) * Q * nb_, cudaMemcpyDeviceToHost, s_));
    BDG_CUDA_TRY(plan_, cudaStreamSynchronize(s_));
    for (int q = 0; q < Q; ++q) {
      out[q] = 0.0;
      for (unsigned b = 0; b < nb_; ++b) out[q] += h[(size_t)q * nb_ + b];
    }
    return BDG_OK;
  }
  double dot1(const double2* a, const double2* b, bdg_status* st) {
    DotSet d{};
    d.a[0] = a;
    d.b[0] = b;
    double v[1] = {0.0};
    *st = dots(d, v);
    return v[0];
  }

  KdArgs<double> kd(const double2* x, double2* y) {
    KdArgs<double> g;
    g.grid = &plan_->grid;
    g.x = x;
    g.y = y;
    g.nplanes = 2;
    for (int a = 0; a < 3; ++a) g.tw[a] = plan_->tw64[a];
    g.shift = 0.0;
    g.scale = 0.5;
    g.stream = s_;
    return g;
  }
  // y = (c - 1/2 Lap)^-1 x
  bdg_status kinetic_inverse(const double2* x, double2* y, double c) {
    KdArgs<double> g = kd(x, y);
    g.shift = c;
    BDG_CUDA_TRY(plan_, kdiag_launch<double>(g));
    return BDG_OK;
  }
  bdg_status laplacian(const double2* x, double2* y) {
    BDG_CUDA_TRY(plan_, laplacian_launch<double>(kd(x, y)));
    return BDG_OK;
  }

  // phi <- P_SM(phi), result record of `slot` cleared
  bdg_status project(double2* phi, int slot) {
    k_gs_norms<<<nb_, NT, 0, s_>>>(phi, np_, part(PART_NORM));
    k_gs_project<<<nb_, NT, 0, s_>>>(phi, np_, part(PART_NORM), nb_, M_, cell_, rec_ + slot * REC);
    BDG_CUDA_TRY(plan_, cudaGetLastError());
    return BDG_OK;
  }
  // record and next right-hand side of the projected state phi
  bdg_status residual(double2* phi, int slot, double c) {
    bdg_status st = laplacian(phi, hphi_[slot]);
    if (st) return st;
    k_gs_hphi<<<nb_, NT, 0, s_>>>(phi, V_, np_, k_, hphi_[slot], part(PART_H));
    k_gs_residual<<<nb_, NT, 0, s_>>>(phi, hphi_[slot], V_, np_, k_, part(PART_H), nb_, c, rhs_[slot], rec_ + slot * REC);
    BDG_CUDA_TRY(plan_, cudaGetLastError());
    return BDG_OK;
  }
  bdg_status rhs(int slot, double c) {
    k_gs_rhs<<<nb_, NT, 0, s_>>>(phi_[slot], V_, np_, k_, c, rhs_[slot]);
    BDG_CUDA_TRY(plan_, cudaGetLastError());
    return BDG_OK;
  }
  // one flow step from slot a into the other; with transforms for the
  // residual once that is below 1e-6
  bdg_status flow_step(int a, double c, double last_res) {
    const int b = 1 - a;
    bdg_status st = kinetic_inverse(rhs_[a], phi_[b], c);
    if (st) return st;
    if (last_res < 1e-6) {
      st = project(phi_[b], b);
      return st ? st : residual(phi_[b], b, c);
    }
    k_gs_norms<<<nb_, NT, 0, s_>>>(phi_[b], np_, part(PART_NORM));
    k_gs_project_h<<<nb_, NT, 0, s_>>>(phi_[b], rhs_[a], c, V_, np_, k_, part(PART_NORM), nb_, M_, cell_, hphi_[b],
                                       part(PART_H), rec_ + b * REC);
    k_gs_residual<<<nb_, NT, 0, s_>>>(phi_[b], hphi_[b], V_, np_, k_, part(PART_H), nb_, c, rhs_[b], rec_ + b * REC);
    BDG_CUDA_TRY(plan_, cudaGetLastError());
    return BDG_OK;
  }
  // result record of a slot: queue the copy, wait for it
  bdg_status fetch(int slot) {
    BDG_CUDA_TRY(plan_, cudaMemcpyAsync(hrec_ + slot * REC, rec_ + slot * REC, sizeof(double) * REC,
                                        cudaMemcpyDeviceToHost, s_));
    BDG_CUDA_TRY(plan_, cudaEventRecord(ev_[slot], s_));
    return BDG_OK;
  }
  bdg_status wait(int slot, double* res, double mu[3]) {
    BDG_CUDA_TRY(plan_, cudaEventSynchronize(ev_[slot]));
    const double* r = hrec_ + slot * REC;
    if (r[4] != 0.0) return fail(plan_, BDG_ERR_INVALID, "ground state: spinor has no admissible component");
    *res = r[0];
    for (int j = 0; j < 3; ++j) mu[j] = r[1 + j];
    return BDG_OK;
  }
  bdg_status read(int slot, double* res, double mu[3]) {
    bdg_status st = fetch(slot);
    return st ? st : wait(slot, res, mu);
  }

  bdg_status stab(const double2* phi, double* alpha) {
    double* d = part(PART_HOST);
    BDG_CUDA_TRY(plan_, cudaMemsetAsync(d, 0, sizeof(double), s_));
    k_gs_stab<<<nb_, NT, 0, s_>>>(phi, V_, np_, k_.beta_n + std::fabs(k_.beta_s), d);
    BDG_CUDA_TRY(plan_, cudaGetLastError());
    BDG_CUDA_TRY(plan_, cudaMemcpyAsync(hrec_ + 2 * REC, d, sizeof(double), cudaMemcpyDeviceToHost, s_));
    BDG_CUDA_TRY(plan_, cudaStreamSynchronize(s_));
    *alpha = hrec_[2 * REC] + std::fabs(k_.p) + std::fabs(k_.q);
    return BDG_OK;
  }

  Normal normal() const { return Normal{{z_[0], z_[1]}, {tz_[0], tz_[1]}, nz_, cell_}; }
  // P v = v - sum_i z_i <z_i, v>  (weighted inner product; z_i weighted-orthonormal)
  bdg_status tangent(double2* v) {
    if (nz_ == 0) return BDG_OK;
    DotSet d{};
    for (int i = 0; i < 2; ++i) {
      d.a[i] = z_[i < nz_ ? i : 0];
      d.b[i] = v;
    }
    double c[2];
    bdg_status st = dots(d, c);
    if (st) return st;
    for (int i = 0; i < nz_; ++i) k_gs_axpby<<<nblk(len_), NT, 0, s_>>>(len_, -c[i] * cell_, z_[i], 1.0, v);
    BDG_CUDA_TRY(plan_, cudaGetLastError());
    return BDG_OK;
  }

  // out = H_+ v at the current state with multipliers m3 from t = -1/2 Lap v (may be out);
  // sums (v, out), (z_i, out) in PART_AP
  bdg_status hplus(const double2* v, const double2* t, double2* out, const double m3[3]) {
    Coupling<double> cp;
    cp.beta_n = k_.beta_n;
    cp.beta_s = k_.beta_s;
    cp.d1 = k_.q - k_.p - m3[0];
    cp.d0 = -m3[1];
    cp.dm = k_.q + k_.p - m3[2];
    k_gs_hplus<<<nb_, NT, 0, s_>>>(phi_[cur_], V_, np_, cp, v, t, out, normal(), part(PART_AP));
    BDG_CUDA_TRY(plan_, cudaGetLastError());
    return BDG_OK;
  }

  // Multipliers m3 = mu + lambda S_z of the least-squares fit H Phi ~
  // (mu + lambda S_z) Phi at the current state and the weighted-orthonormal
  // basis z_ of span{Phi, S_z Phi} (the normal directions of S_M).
  bdg_status tangent_setup(double m3[3]) {
    const double2* phi = phi_[cur_];
    const double2* hphi = hphi_[cur_];
    k_gs_sz<<<nb_, NT, 0, s_>>>(phi, np_, z_[1]);
    BDG_CUDA_TRY(plan_, cudaGetLastError());
    DotSet d{};
    d.a[0] = phi; d.b[0] = phi;
    d.a[1] = phi; d.b[1] = z_[1];
    d.a[2] = z_[1]; d.b[2] = z_[1];
    d.a[3] = phi; d.b[3] = hphi;
    d.a[4] = z_[1]; d.b[4] = hphi;
    double g[5];
    bdg_status st = dots(d, g);
    if (st) return st;
    double mu, lam;
    const double det = g[0] * g[2] - g[1] * g[1];
    if (g[2] < 1e-300 || !(std::fabs(det) > 1e-30 * g[0] * g[2])) {
      mu = g[3] / g[0];
      lam = 0.0;
    } else {
      mu = (g[3] * g[2] - g[1] * g[4]) / det;
      lam = (g[0] * g[4] - g[1] * g[3]) / det;
    }
    m3[0] = mu + lam;
    m3[1] = mu;
    m3[2] = mu - lam;
    // weighted-orthonormal basis of span{Phi, S_z Phi}
    const double nphi = std::sqrt(cell_ * g[0]);
    k_gs_axpby<<<nblk(len_), NT, 0, s_>>>(len_, 1.0 / nphi, phi, 0.0, z_[0]);
    nz_ = 1;
    // z2 = S_z Phi - z1 <z1, S_z Phi>
    const double c12 = cell_ * g[1] / nphi;
    k_gs_axpby<<<nblk(len_), NT, 0, s_>>>(len_, -c12, z_[0], 1.0, z_[1]);
    BDG_CUDA_TRY(plan_, cudaGetLastError());
    const double n2 = std::sqrt(std::max(cell_ * dot1(z_[1], z_[1], &st), 0.0));
    if (st) return st;
    if (n2 > 1e-10 * nphi) {
      k_gs_axpby<<<nblk(len_), NT, 0, s_>>>(len_, 1.0 / n2, z_[1], 0.0, z_[1]);
      BDG_CUDA_TRY(plan_, cudaGetLastError());
      nz_ = 2;
    }
    return BDG_OK;
  }

  // Stability of a converged stationary state: the curvature
  // <d, P H_+ P d> / <d, d> of the energy on S_M along the population-transfer
  // directions (k_gs_transfer).  *unstable is set, and the unit direction of
  // most negative curvature left in cp_, when a curvature is below
  // -1e-9 (1 + max |mu|).
  bdg_status stability(bool* unstable) {
    *unstable = false;
    double m3[3];
    bdg_status st = tangent_setup(m3);
    if (st) return st;
    const double mmax = std::max(std::fabs(m3[0]), std::max(std::fabs(m3[1]), std::fabs(m3[2])));
    const double nphi = dot1(phi_[cur_], phi_[cur_], &st);
    if (st) return st;
    double best = -1e-9 * (1.0 + mmax);
    for (int kind = 0; kind < 3; ++kind) {
      k_gs_transfer<<<nb_, NT, 0, s_>>>(phi_[cur_], np_, kind, cz_);
      BDG_CUDA_TRY(plan_, cudaGetLastError());
      if ((st = tangent(cz_))) return st;
      const double dd = dot1(cz_, cz_, &st);
      if (st) return st;
      if (!(dd > 1e-16 * nphi)) continue;
      if ((st = laplacian(cz_, cap_)) || (st = hplus(cz_, cap_, cap_, m3)) || (st = tangent(cap_))) return st;
      const double kappa = dot1(cz_, cap_, &st) / dd;
      if (st) return st;
      if (kappa < best) {
        best = kappa;
        *unstable = true;
        k_gs_axpby<<<nblk(len_), NT, 0, s_>>>(len_, 1.0 / std::sqrt(dd), cz_, 0.0, cp_);
        BDG_CUDA_TRY(plan_, cudaGetLastError());
      }
    }
    return BDG_OK;
  }

  // z = T^-1 r and the sums (r, z), (z_i, z) into record `to`
  bdg_status precondition(double c, int to) {
    bdg_status st = kinetic_inverse(cr_, cz_, c);
    if (st) return st;
    DotSet d{};
    d.a[0] = cr_;
    for (int i = 0; i < 2; ++i) d.a[1 + i] = z_[i < nz_ ? i : 0];
    for (int i = 0; i < 3; ++i) d.b[i] = cz_;
    k_gs_dots<3><<<nb_, NT, 0, s_>>>(d, np_, part(to));
    BDG_CUDA_TRY(plan_, cudaGetLastError());
    return BDG_OK;
  }

  // one inexact Newton step from the current state, phi + x into trial_ (not
  // yet projected); *products = H_+ products
  bdg_status newton_step(double c, int* products) {
    const double eta = 1e-2;
    const int maxcg = 500;
    *products = 0;
    double m3[3];
    bdg_status st = tangent_setup(m3);
    if (st) return st;
    // b = -P r, r = H Phi - (mu + lambda S_z) Phi;  CG on P H_+ P x = b
    k_gs_negres<<<nb_, NT, 0, s_>>>(hphi_[cur_], phi_[cur_], np_, m3[0], m3[1], m3[2], cr_);
    BDG_CUDA_TRY(plan_, cudaGetLastError());
    if ((st = tangent(cr_))) return st;
    for (int i = 0; i < nz_; ++i)
      if ((st = laplacian(z_[i], tz_[i]))) return st;
    BDG_CUDA_TRY(plan_, cudaMemsetAsync(cx_, 0, sizeof(double2) * len_, s_));
    const double b0 = std::sqrt(dot1(cr_, cr_, &st));
    if (st) return st;
    int rz = PART_RZ;   // record of the current (r, z)
    if ((st = precondition(c, rz))) return st;
    k_gs_cg_p<<<nb_, NT, 0, s_>>>(cp_, tp_, cz_, cr_, c, np_, normal(), part(rz), nullptr, nullptr, nb_, 1, rec_);
    BDG_CUDA_TRY(plan_, cudaGetLastError());
    const int slot = 1 - cur_;   // its record is free
    for (int kcg = 0; kcg < maxcg && b0 > 0; ++kcg) {
      if ((st = hplus(cp_, tp_, cap_, m3))) return st;
      ++*products;
      k_gs_cg_xr<<<nb_, NT, 0, s_>>>(cx_, cr_, cp_, cap_, np_, normal(), part(PART_AP), part(rz), nb_, part(PART_RR),
                                     rec_ + slot * REC);
      BDG_CUDA_TRY(plan_, cudaGetLastError());
      const int nrz = PART_RZ + PART_RZ2 - rz;
      if ((st = precondition(c, nrz))) return st;
      k_gs_cg_p<<<nb_, NT, 0, s_>>>(cp_, tp_, cz_, cr_, c, np_, normal(), part(nrz), part(rz), part(PART_RR), nb_, 0,
                                    rec_ + slot * REC);
      BDG_CUDA_TRY(plan_, cudaGetLastError());
      rz = nrz;
      if ((st = fetch(slot))) return st;
      BDG_CUDA_TRY(plan_, cudaEventSynchronize(ev_[slot]));
      const double pap = hrec_[slot * REC + 5], rn = std::sqrt(hrec_[slot * REC + 6]);
      if (!(pap > 0) || rn <= eta * b0) break;
    }
    BDG_CUDA_TRY(plan_, cudaMemcpyAsync(trial_, phi_[cur_], sizeof(double2) * len_, cudaMemcpyDeviceToDevice, s_));
    k_gs_axpby<<<nblk(len_), NT, 0, s_>>>(len_, 1.0, cx_, 1.0, trial_);
    BDG_CUDA_TRY(plan_, cudaGetLastError());
    return BDG_OK;
  }

  enum { PART_NORM, PART_H, PART_AP, PART_RZ, PART_RZ2, PART_RR, PART_HOST, PARTS };

  bdg_plan_t plan_;
  double M_;
  cudaStream_t s_;
  long long np_ = 0, len_ = 0;
  unsigned nb_ = 1;
  double cell_ = 1.0;
  GsCoef k_{};
  std::vector<void*> bufs_;
  double* V_ = nullptr;
  // two states (the current one and the next), with H phi, the flow's
  // right-hand side and a result record each
  int cur_ = 0;
  double2 *phi_[2] = {nullptr, nullptr}, *hphi_[2] = {nullptr, nullptr}, *rhs_[2] = {nullptr, nullptr};
  double2* trial_ = nullptr;
  double2 *z_[2] = {nullptr, nullptr}, *tz_[2] = {nullptr, nullptr};
  int nz_ = 0;
  double2 *cx_ = nullptr, *cr_ = nullptr, *cz_ = nullptr, *cp_ = nullptr, *tp_ = nullptr, *cap_ = nullptr;
  double* part_ = nullptr;
  double* rec_ = nullptr;
  double* hrec_ = nullptr;
  cudaEvent_t ev_[2] = {nullptr, nullptr};
};

}  // namespace
}  // namespace bdg

using namespace bdg;

bdg_status bdg_ground_state(const bdg_params* p, double M, const double* V, const double* phi0, double tol,
                            int maxit, double* phi, double* mu, double* resid, int* iters, void* stream) {
  if (!p || !V || !phi0 || !phi || !mu) return fail(nullptr, BDG_ERR_INVALID, "NULL argument");
  if (!(std::fabs(M) < 1.0)) return fail(nullptr, BDG_ERR_INVALID, "magnetization must satisfy |M| < 1");
  if (!(tol > 0) || maxit < 0) return fail(nullptr, BDG_ERR_INVALID, "tol must be > 0 and maxit >= 0");
  cudaStream_t s = (cudaStream_t)stream;
  // the internal plan: mu = 0 so that the FG product of (0, Phi) is H Phi
  bdg_params q = *p;
  q.mu[0] = q.mu[1] = q.mu[2] = 0.0;
  q.prec = BDG_FP64;
  bdg_plan_t plan = nullptr;
  bdg_status st = create_plan(&plan, &q, V, phi0, s, false);
  if (st) return st;
  double res = INFINITY, m[3] = {0, 0, 0};
  int it = 0;
  {
    GroundState gs(plan, M, s);
    st = gs.init(V, phi0);
    if (!st) st = gs.run(tol, maxit, &res, m, &it);
    if (!st) st = gs.download(phi);
  }
  std::string err = st ? plan->err : std::string();
  bdg_plan_destroy(plan);
  if (st) return fail(nullptr, st, err);
  for (int j = 0; j < 3; ++j) mu[j] = m[j];
  if (resid) *resid = res;
  if (iters) *iters = it;
  if (!(res <= tol)) return fail(nullptr, BDG_ERR_NOT_CONVERGED, "ground state did not reach tol within maxit");
  return BDG_OK;
}
