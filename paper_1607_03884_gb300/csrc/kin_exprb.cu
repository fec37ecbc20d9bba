// exprb43 with Krylov phi-function products (kin_exprb_* of the C ABI): the
// fourth-order exponential Rosenbrock method the paper compares with Radau
// IIA (Sec. 2.1, Table of solvers; Sec. 3.1), one state per warp.
//
// Scheme (Hochbruck, Ostermann & Schweitzer), g(u) = F(u) - J_n u,
// D_i = g(U_i) - g(u_n):
//   U2 = u_n + h/2 phi1(h/2 J) F(u_n)
//   U3 = u_n + h phi1(h J) F(u_n) + h phi1(h J) D2
//   u_{n+1} = u_n + h phi1(h J) F(u_n) + h (16 phi3 - 48 phi4)(h J) D2
//             + h (-2 phi3 + 12 phi4)(h J) D3
//   embedded (order 3): 16 phi3 for D2 and -2 phi3 for D3.
// J_n is the analytical Jacobian at u_n (once per accepted point).  Each of
// F(u_n), D2 and D3 spans its own Krylov space (Arnoldi, modified
// Gram-Schmidt, in the inner product of the step's error weights D: on
// D^-1 J D, which keeps the Hessenberg matrix as well scaled as the
// chemistry's time scales; vectors over the warp's lanes as in the Radau
// WARP layout, the basis and the Hessenberg matrix in the warp's global
// slot); its
// dimension grows until Saad's leading error term of every product taken
// from it, h beta (h h_{m+1,m}) c_k |e_m^T phi_{k+1}(h H_m) e1| in the
// step's error weights, is at most kappa, or the space is exhausted.
// phi_1..phi_p(tau H_m) e1 come with exp(tau H_m) from scaling and squaring:
// at A = 2^-s tau H_m with ||A||_1 <= 1/4 by their Taylor series (the powers
// A^j e1 serve all phi_k at once), then s doublings
//   F <- 2 F + F F,  phi_k <- 2^-k (phi_k + F phi_k + sum_{j=1..k} phi_j / (k-j)!)
// with F = E - I, so that the slow modes of a stiff matrix, tiny after the
// scaling, are not rounded against the identity.  These are the blocks of
// squaring the exponential of the augmented matrix [[A, e1, 0], [0, 0, I],
// [0, 0, 0]] without its known rows.  (The paper uses
// a (10,10) Caratheodory-Fejer rational approximant of exp on the negative
// real axis instead; scaling and squaring holds for any spectrum, including
// the positive eigenvalues of igniting states.)  Step size control:
// Hairer-Norsett-Wanner on the embedded difference.
//
// What bounds the kernel is the FP64 unit, and the matrix functions are most
// of its work: a space of 2.3 vectors on average, so F and the phi_k are a few
// entries per lane and the cost is the number of FP64 instructions in a
// doubling.  The squared augmented matrix with its Pade denominator took
// 1150 of them per evaluation and eleven evaluations a step; the blocks take
// 300, and the estimate's evaluation at the accepted dimension also gives the
// step's products (phi_1 at h/2 is the state before the last doubling), so
// seven evaluations remain.  The rates and the Jacobian are a team's
// (kin_team.cuh) with one warp, their tables in shared memory.  Measured (H2
// states, FP64): 309 -> 147 ms by the blocks, 113 ms with the tables.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <vector>

#include "../../include/kin.h"
#include "kin_internal.h"
#include "kin_warp.cuh"

using namespace kin;

namespace {

constexpr int XL = 32;
using XG = Grp<XL>;
constexpr int XWR = XG::WR;
using XV = WVecT<XWR>;
constexpr int XKP = 5;  // phi_1 .. phi_5 at most
// the most species: the entry's documented limit (the vectors hold 63, the
// bath gas at element ns)
constexpr int XSPECIES = 58;
constexpr int XTERMS = 13;  // Taylor terms: (1/4)^14 / 14! < 2^-64

__device__ __constant__ double INVFACT[20] = {
    1.0, 1.0, 1.0 / 2.0, 1.0 / 6.0, 1.0 / 24.0, 1.0 / 120.0, 1.0 / 720.0, 1.0 / 5040.0,
    1.0 / 40320.0, 1.0 / 362880.0, 1.0 / 3628800.0, 1.0 / 39916800.0, 1.0 / 479001600.0,
    1.0 / 6227020800.0, 1.0 / 87178291200.0, 1.0 / 1307674368000.0, 1.0 / 20922789888000.0,
    1.0 / 355687428096000.0, 1.0 / 6402373705728000.0, 1.0 / 121645100408832000.0};

// matrix-function scratch for dimension m: A, two power buffers, two buffers
// of [F | phi_1 .. phi_p]
__host__ __device__ constexpr size_t xmf_doubles(size_t m) { return 5 * m * m + 2 * XKP * m; }

// per-warp workspace in global memory (after the Jacobian slot)
struct XWork {
  double *V;     // basis: vector j at V + j * N, j <= N
  double *H;     // Hessenberg, (N + 1) x N, H[i * N + j]
  double *mf;    // matrix-function scratch of any dimension up to N
  double *half;  // phi_1(tau/2 H) e1
  double *vd;    // N: a vector handed to the matrix-vector product
  double *fast;  // shared-memory matrix-function scratch
  int nfast;     // its size in doubles
};

// A warp's shared memory: the chemistry's buffers of kin_team.cuh for one warp
// (C, g, q, the Jacobian's scratch) and, for small mechanisms, the assembly
// matrix, which is in the global slot otherwise.
constexpr int XSMALL = 16;
__host__ __device__ inline size_t xwarp_bytes(const MechLayout &L) {
  size_t d = 2 * (size_t)team_nv(L.ns) + L.nr + team_js_doubles(L);
  if (L.ns <= XSMALL) d += (size_t)L.ns * team_ld(L.ns);
  return ((sizeof(TeamCtl) + 15) / 16 * 16 + d * sizeof(double) + 15) / 16 * 16;
}

__host__ __device__ inline size_t xslot_doubles(int N) {
  size_t d = 2 * (size_t)N * (N + 1);                               // J, assembly matrix
  d += 2 * (size_t)(N + 1) * N + xmf_doubles(N) + 2 * (size_t)N;    // V, H, mf, half, vd
  return (d + 31) / 32 * 32;
}

__device__ XWork carve_xwork(double *slot, int N) {
  XWork w;
  double *p = slot + 2 * (size_t)N * (N + 1);
  w.V = p;
  p += (size_t)(N + 1) * N;
  w.H = p;
  p += (size_t)(N + 1) * N;
  w.mf = p;
  p += xmf_doubles(N);
  w.half = p;
  p += N;
  w.vd = p;
  w.fast = nullptr;
  w.nfast = 0;
  return w;
}

__device__ __forceinline__ double xdot(int N, const XV &a, const XV &b) {
  double s = 0.0;
#pragma unroll
  for (int r = 0; r < XWR; ++r)
    if (XG::lane() + XL * r < N) s += a.v[r] * b.v[r];
  return XG::sum(s);
}

__device__ __forceinline__ double xwrms(int N, const XV &a, const XV &sc) {
  double s = 0.0;
#pragma unroll
  for (int r = 0; r < XWR; ++r)
    if (XG::lane() + XL * r < N) {
      const double q = a.v[r] / sc.v[r];
      s += q * q;
    }
  return sqrt(XG::sum(s) / N);
}

__device__ __forceinline__ void xload(int N, const double *p, XV &x) {
#pragma unroll
  for (int r = 0; r < XWR; ++r) {
    const int g = XG::lane() + XL * r;
    x.v[r] = g < N ? p[g] : 0.0;
  }
}

__device__ __forceinline__ void xstore(int N, double *p, const XV &x) {
#pragma unroll
  for (int r = 0; r < XWR; ++r) {
    const int g = XG::lane() + XL * r;
    if (g < N) p[g] = x.v[r];
  }
}

// y = J x, J by columns (entry (i, c) at c * ld + i: coalesced), x in memory
__device__ void xmatvec(int N, int ld, const double *J, const double *x, XV &y) {
#pragma unroll
  for (int r = 0; r < XWR; ++r) {
    const int g = XG::lane() + XL * r;
    double s = 0.0;
    if (g < N)
      for (int c = 0; c < N; ++c) s += J[c * ld + g] * x[c];
    y.v[r] = s;
  }
}

// exp(tau H_m) and phi_1 .. phi_p (tau H_m) e1: entry (i, c) of the returned
// m x (m + p) array is F[i][c] = (exp - I)[i][c] for c < m, then
// phi_{c-m+1}[i]; phi_1 at tau/2 in w.half.  nullptr when the norm is not finite.
__device__ __noinline__ const double *xphi(int N, int m, int p, double tau, const XWork &w) {
  const int lane = XG::lane(), cols = m + p, mm = m * m, nz = m * cols;
  double *buf = xmf_doubles(m) <= (size_t)w.nfast ? w.fast : w.mf;
  double *A = buf, *T0 = buf + mm, *T1 = buf + 2 * mm, *Z = buf + 3 * mm, *Zn = Z + m * (m + XKP);
  double nrm = 0.0;
  for (int c = lane; c < m; c += XL) {
    double cs = 0.0;
    for (int i = 0; i <= c + 1 && i < m; ++i) cs += fabs(tau * w.H[i * N + c]);
    nrm = fmax(nrm, cs);
    if (!isfinite(cs)) nrm = INFINITY;
  }
#pragma unroll
  for (int o = XL / 2; o > 0; o >>= 1) nrm = fmax(nrm, __shfl_xor_sync(XG::mask(), nrm, o, XL));
  if (!isfinite(nrm)) return nullptr;
  int sq = 0;
  while (nrm > 0.25 && sq < 1100) {  // finite norms stop well before
    nrm *= 0.5;
    ++sq;
  }
  const double sc = ldexp(1.0, -sq);
  for (int e = lane; e < mm; e += XL) {
    const int i = e / m, c = e - i * m;
    // upper Hessenberg: Arnoldi writes no other entry
    A[e] = i <= c + 1 ? tau * w.H[i * N + c] * sc : 0.0;
    T0[e] = i == c ? 1.0 : 0.0;
  }
  for (int e = lane; e < nz; e += XL) {
    const int i = e / cols, c = e - i * cols;
    Z[e] = (c >= m && i == 0) ? INVFACT[c - m + 1] : 0.0;
  }
  if (sq == 0)
    for (int i = lane; i < m; i += XL) w.half[i] = i == 0 ? 1.0 : 0.0;
  XG::sync();
  double hpow = 1.0;
#pragma unroll 1
  for (int j = 1; j <= XTERMS; ++j) {  // T1 = A T0 = A^j
    for (int e = lane; e < mm; e += XL) {
      const int i = e / m, c = e - i * m;
      double s = 0.0;
      for (int q = i > 0 ? i - 1 : 0; q < m; ++q) s = fma(A[i * m + q], T0[q * m + c], s);
      T1[e] = s;
    }
    XG::sync();
    for (int e = lane; e < nz; e += XL) {
      const int i = e / cols, c = e - i * cols;
      Z[e] = c < m ? fma(T1[i * m + c], INVFACT[j], Z[e])
                   : fma(T1[i * m], INVFACT[j + c - m + 1], Z[e]);
    }
    hpow *= 0.5;
    if (sq == 0)
      for (int i = lane; i < m; i += XL) w.half[i] = fma(T1[i * m] * hpow, INVFACT[j + 1], w.half[i]);
    double *t = T0;
    T0 = T1;
    T1 = t;
    XG::sync();
  }
#pragma unroll 1
  for (int d = 0; d < sq; ++d) {
    if (d == sq - 1)
      for (int i = lane; i < m; i += XL) w.half[i] = Z[i * cols + m];
    for (int e = lane; e < nz; e += XL) {
      const int i = e / cols, c = e - i * cols;
      const double *row = Z + i * cols;
      double s = c < m ? 2.0 * row[c] : row[c];
      for (int q = 0; q < m; ++q) s = fma(row[q], Z[q * cols + c], s);
      if (c >= m) {
        const int k = c - m + 1;
        for (int q = 1; q <= k; ++q) s = fma(row[m + q - 1], INVFACT[k - q], s);
        // 2^-k, exact: by the exponent's own multiplication
        s *= __hiloint2double((1023 - k) << 20, 0);
      }
      Zn[e] = s;
    }
    double *t = Z;
    Z = Zn;
    Zn = t;
    XG::sync();
  }
  return Z;
}

// D beta V_m phi with phi's component i at ph[i * stride]
__device__ void xproduct(int N, int m, double beta, const XWork &w, const double *ph, int stride,
                         const XV &scal, XV &out) {
#pragma unroll
  for (int r = 0; r < XWR; ++r) {
    const int g = XG::lane() + XL * r;
    double s = 0.0;
    if (g < N)
      for (int i = 0; i < m; ++i) s += w.V[i * N + g] * ph[i * stride];
    out.v[r] = scal.v[r] * (beta * s);
  }
}

// The chemistry of one warp: rates as the teams evaluate them, the Jacobian
// assembled by the one warp without atomics.
struct XChem {
  const MechView &m;
  const HotTables &h;
  const TeamBuf<double> &t;
  __device__ __forceinline__ int rates(double P, const XV &y, XV &f) const {
    XG::sync();
    const int rc = team_rhs<>(m, h, t.C(0), t.g(0), t.q(0), P, y, f);
    XG::sync();
    return rc;
  }
  // also the Jacobian, into t.J
  __device__ __noinline__ int jacobian(double P, const XV &y, XV &f) const {
    const TeamMassFrac<double> c{m, h, t};
    XG::sync();
    if (XG::lane() == 0) t.ctl->P = P;
    XG::sync();
    c.jac_prepare(y);
    XG::sync();
    double *J = t.J;
    const int ld = t.ld;
    c.jac_out<1>(0, [J, ld](int i, int k, double v) { J[k * ld + i] = v; });
    XG::sync();
    vec_load(m.ns, t.g(0), f);
    const int rc = t.ctl->ret[0];
    XG::sync();
    return rc;
  }
};

__device__ __forceinline__ TeamBuf<double> xcarve(const MechLayout &L, unsigned char *p,
                                                  double *slot) {
  const int N = L.ns;
  TeamBuf<double> t{};
  t.ld = team_ld(N);
  t.nv = team_nv(N);
  t.wstride = 2 * t.nv + L.nr;
  t.ctl = reinterpret_cast<TeamCtl *>(p);
  t.w0 = reinterpret_cast<double *>(p + (sizeof(TeamCtl) + 15) / 16 * 16);
  t.js = t.w0 + t.wstride;
  t.J = slot;
  t.Jd = N <= XSMALL ? t.js + team_js_doubles(L) : slot + (size_t)N * (N + 1);
  return t;
}

struct XProducts {
  int np, kmax;
  int k[3];
  double c[3];
};

// Arnoldi in the error-weighted inner product (on D^-1 J D from D^-1 v,
// D = diag(scal)) with the stopping rule; returns m (0 for v = 0), -1 when
// a matrix function failed; beta and the matrix functions at the returned
// dimension (xphi's array, kmax + 1 phi functions) out
__device__ int xarnoldi(int N, int ld, const double *J, const XV &v, double h,
                        const XProducts &pr, const XV &scal, double kappa, const XWork &w,
                        double &beta, const double *&Z) {
  const int lane = XG::lane();
  XV q;
#pragma unroll
  for (int r = 0; r < XWR; ++r) q.v[r] = v.v[r] / scal.v[r];  // D^-1 v
  beta = sqrt(xdot(N, q, q));
  if (beta == 0.0) return 0;
#pragma unroll
  for (int r = 0; r < XWR; ++r) q.v[r] = q.v[r] / beta;
  xstore(N, w.V, q);
  XG::sync();
  for (int j = 0; j < N; ++j) {
    XV x;
    xload(N, w.V + (size_t)j * N, x);  // D^-1 J D v_j: the product of J with D v_j
#pragma unroll
    for (int r = 0; r < XWR; ++r) x.v[r] *= scal.v[r];
    xstore(N, w.vd, x);
    XG::sync();
    xmatvec(N, ld, J, w.vd, x);
#pragma unroll
    for (int r = 0; r < XWR; ++r) x.v[r] = x.v[r] / scal.v[r];
    XG::sync();
    const double nw = sqrt(xdot(N, x, x));
    for (int i = 0; i <= j; ++i) {  // modified Gram-Schmidt
      XV vi;
      xload(N, w.V + (size_t)i * N, vi);
      const double hij = xdot(N, vi, x);
#pragma unroll
      for (int r = 0; r < XWR; ++r) x.v[r] -= hij * vi.v[r];
      if (lane == 0) w.H[i * N + j] = hij;
    }
    const double hn = sqrt(xdot(N, x, x));
    if (lane == 0) w.H[(j + 1) * N + j] = hn;
    const int m = j + 1;
    if (hn <= 1e-13 * nw || m == N) {
      XG::sync();
      Z = xphi(N, m, pr.kmax + 1, h, w);
      return Z ? m : -1;
    }
#pragma unroll
    for (int r = 0; r < XWR; ++r) x.v[r] = x.v[r] / hn;
    xstore(N, w.V + (size_t)(j + 1) * N, x);
    XG::sync();
    Z = xphi(N, m, pr.kmax + 1, h, w);
    // a failed matrix function or a non-finite entry gives no estimate: keep growing
    double lead = Z ? 0.0 : NAN;
    if (Z)
      for (int t = 0; t < pr.np; ++t) {
        const double v =
            pr.c[t] * fabs(Z[(m - 1) * (m + pr.kmax + 1) + m + pr.k[t]]);  // phi_{k+1}
        lead = isnan(v) || isnan(lead) ? NAN : fmax(lead, v);
      }
    // v_{m+1} has unit 2-norm in the scaled space: weighted RMS 1/sqrt(N)
    const double est = h * beta * (h * hn) * lead / sqrt((double)N);
    XG::sync();
    if (est <= kappa) return m;
  }
  return -1;  // not reached: the space is exhausted at m = N
}

struct XParams {
  double rtol, atol, dt, kappa;
  int max_steps;
  int64_t n;
  const double *h0;
};

// D = F(U) - F(u) - J (U - u)
__device__ void xremainder(int N, int ld, const double *J, const XV &U, const XV &u,
                           const XV &FU, const XV &Fu, const XWork &w, XV &D) {
  XV d;
#pragma unroll
  for (int r = 0; r < XWR; ++r) d.v[r] = U.v[r] - u.v[r];
  xstore(N, w.vd, d);
  XG::sync();
  XV Jd;
  xmatvec(N, ld, J, w.vd, Jd);
#pragma unroll
  for (int r = 0; r < XWR; ++r) D.v[r] = FU.v[r] - Fu.v[r] - Jd.v[r];
  XG::sync();
}

// one attempt: 0 done (unew, uhat), 1 a stage was not finite, 2 a matrix
// function failed
__device__ int xstep(const XChem &x, double P, const XWork &w,
                     const XV &y, const XV &fy, double h, const XV &scal, double kappa, XV &unew,
                     XV &uhat, int &nf, int &kdim) {
  const int N = x.m.ns, ld = x.t.ld;
  const double *J = x.t.J;
  const XProducts PF = {1, 1, {1, 0, 0}, {1.0, 0.0, 0.0}};
  const XProducts PD2 = {3, 4, {1, 3, 4}, {1.0, 16.0, 48.0}};
  const XProducts PD3 = {2, 4, {3, 4, 0}, {2.0, 12.0, 0.0}};
  nf = 0;
  kdim = 0;
  double beta;
  const double *Z = nullptr;
  XV half, full, U, F, D, q1, q3, q4, r3, r4;
  int mk = xarnoldi(N, ld, J, fy, h, PF, scal, kappa, w, beta, Z);
  if (mk < 0) return 2;
  kdim += mk;
  if (mk == 0) {
#pragma unroll
    for (int r = 0; r < XWR; ++r) half.v[r] = full.v[r] = 0.0;
  } else {
    xproduct(N, mk, beta, w, w.half, 1, scal, half);
    xproduct(N, mk, beta, w, Z + mk, mk + PF.kmax + 1, scal, full);
    XG::sync();
  }
#pragma unroll
  for (int r = 0; r < XWR; ++r) U.v[r] = y.v[r] + 0.5 * h * half.v[r];
  nf++;
  if (x.rates(P, U, F)) return 1;
  xremainder(N, ld, J, U, y, F, fy, w, D);
  mk = xarnoldi(N, ld, J, D, h, PD2, scal, kappa, w, beta, Z);
  if (mk < 0) return 2;
  kdim += mk;
  if (mk == 0) {
#pragma unroll
    for (int r = 0; r < XWR; ++r) q1.v[r] = q3.v[r] = q4.v[r] = 0.0;
  } else {
    const int ld2 = mk + PD2.kmax + 1;
    xproduct(N, mk, beta, w, Z + mk, ld2, scal, q1);
    xproduct(N, mk, beta, w, Z + mk + 2, ld2, scal, q3);
    xproduct(N, mk, beta, w, Z + mk + 3, ld2, scal, q4);
    XG::sync();
  }
#pragma unroll
  for (int r = 0; r < XWR; ++r) U.v[r] = y.v[r] + h * full.v[r] + h * q1.v[r];
  nf++;
  if (x.rates(P, U, F)) return 1;
  xremainder(N, ld, J, U, y, F, fy, w, D);
  mk = xarnoldi(N, ld, J, D, h, PD3, scal, kappa, w, beta, Z);
  if (mk < 0) return 2;
  kdim += mk;
  if (mk == 0) {
#pragma unroll
    for (int r = 0; r < XWR; ++r) r3.v[r] = r4.v[r] = 0.0;
  } else {
    const int ld3 = mk + PD3.kmax + 1;
    xproduct(N, mk, beta, w, Z + mk + 2, ld3, scal, r3);
    xproduct(N, mk, beta, w, Z + mk + 3, ld3, scal, r4);
    XG::sync();
  }
#pragma unroll
  for (int r = 0; r < XWR; ++r) {
    const double base = y.v[r] + h * full.v[r];
    unew.v[r] = base + h * (16.0 * q3.v[r] - 48.0 * q4.v[r]) + h * (-2.0 * r3.v[r] + 12.0 * r4.v[r]);
    uhat.v[r] = base + h * (16.0 * q3.v[r]) + h * (-2.0 * r3.v[r]);
  }
  return 0;
}

struct XCount {
  int nstep, naccpt, nrejct, nfcn, njac, narn, kdim, status;
};

// One state from y (in: [T, Y_0 .. Y_{ns-2}], out: the state at dt or at
// its last accepted point).
__device__ XCount xintegrate(const XChem &ch, double P, const XWork &w,
                             const XParams &p, int64_t idx, XV &y) {
  const int N = ch.m.ns;
  XCount c = {0, 0, 0, 0, 0, 0, 0, 0};
  XV fy, scal, unew, uhat;
  c.nfcn = 1;
  c.njac = 1;
  if (ch.jacobian(P, y, fy)) {
    c.status = 4;
    return c;
  }
#pragma unroll
  for (int r = 0; r < XWR; ++r) scal.v[r] = p.atol + p.rtol * fabs(y.v[r]);
  double h;
  if (p.h0) {
    h = p.h0[idx];
  } else {  // starting step (Hairer-Norsett-Wanner Vol. I, II.4), order 4
    const double d0 = xwrms(N, y, scal), d1 = xwrms(N, fy, scal);
    double h0 = (d0 < 1e-5 || d1 < 1e-5) ? 1e-6 : 0.01 * d0 / d1;
    h0 = fmin(h0, p.dt);
    XV u, fu;
#pragma unroll
    for (int r = 0; r < XWR; ++r) u.v[r] = y.v[r] + h0 * fy.v[r];
    const int rc = ch.rates(P, u, fu);
    c.nfcn++;
    if (rc) {
      h = 0.01 * h0;
    } else {
      XV df;
#pragma unroll
      for (int r = 0; r < XWR; ++r) df.v[r] = fu.v[r] - fy.v[r];
      const double d2 = xwrms(N, df, scal) / h0;
      const double dm = fmax(d1, d2);
      const double h1 = (dm <= 1e-15) ? fmax(1e-6, h0 * 1e-3) : pow(0.01 / dm, 0.25);
      h = fmin(100.0 * h0, h1);
    }
    h = fmin(h, p.dt);
  }
  double x = 0.0, facmax = 5.0;
  bool last = false;
  for (;;) {
    if (c.nstep >= p.max_steps) {
      c.status = 1;
      return c;
    }
    if (0.1 * fabs(h) <= fabs(x) * 1e-16) {
      c.status = 2;
      return c;
    }
    if (x + 1.0001 * h >= p.dt) {
      h = p.dt - x;
      last = true;
    }
    c.nstep++;
#pragma unroll
    for (int r = 0; r < XWR; ++r) scal.v[r] = p.atol + p.rtol * fabs(y.v[r]);
    int nf = 0, kd = 0;
    const int rc = xstep(ch, P, w, y, fy, h, scal, p.kappa, unew, uhat, nf, kd);
    c.nfcn += nf;
    c.narn += 3;
    c.kdim += kd;
    if (rc == 1) {
      c.nrejct++;
      h *= 0.5;
      last = false;
      facmax = 1.0;
      continue;
    }
    XV d, sc;
#pragma unroll
    for (int r = 0; r < XWR; ++r) {
      d.v[r] = unew.v[r] - uhat.v[r];
      sc.v[r] = p.atol + p.rtol * fmax(fabs(y.v[r]), fabs(unew.v[r]));
    }
    // a matrix function that failed, or a non-finite estimate: rejected with
    // the smallest factor
    const double e = rc == 2 ? INFINITY : xwrms(N, d, sc);
    const double err = isfinite(e) ? fmax(e, 1e-10) : INFINITY;
    const double fac = isfinite(err) ? 0.9 * pow(err, -0.25) : 0.0;
    if (err <= 1.0) {
      x = last ? p.dt : x + h;
      y = unew;
      c.naccpt++;
      if (last) return c;
      c.nfcn++;
      c.njac++;
      if (ch.jacobian(P, y, fy)) {
        c.status = 4;
        return c;
      }
      h = h * fmin(facmax, fmax(0.2, fac));
      facmax = 5.0;
    } else {
      c.nrejct++;
      h = h * fmax(0.2, fac);
      facmax = 1.0;
      last = false;
    }
  }
}

struct XArgs {
  MechLayout L;
  const double *tab;
  const int *itab;
  double *Y, *T;
  const double *P;
  int32_t *status, *counters;
  unsigned long long *totals;
  XParams p;
  double *scratch;
  int64_t slots;
  const unsigned char *hot;  // the tables of kin_team.cuh
  int hot_smem;              // copied to shared memory by each block
};

__global__ void __launch_bounds__(256) k_integrate_exprb(XArgs a) {
  extern __shared__ __align__(16) unsigned char xsmem[];
  const MechView m = make_view(a.L, a.tab, a.itab);
  const int N = m.ns, lane = XG::lane(), grp = (int)(threadIdx.x / XL);
  const int64_t n = a.p.n;
  const HotTables h = stage_hot(a.L, a.hot, a.hot_smem != 0, xsmem);
  const size_t hb = a.hot_smem ? hot_offsets(a.L).bytes : 0;
  const int64_t slot = (int64_t)blockIdx.x * (blockDim.x / XL) + grp;  // < slots (launch)
  double *gs = a.scratch + slot * (int64_t)xslot_doubles(N);
  const TeamBuf<double> t = xcarve(a.L, xsmem + hb + grp * xwarp_bytes(a.L), gs);
  const XChem ch{m, h, t};
  XWork w = carve_xwork(gs, N);
  // the Jacobian's scratch is free outside its assembly
  w.fast = t.js;
  w.nfast = (int)team_js_doubles(a.L);
  unsigned long long *queue = a.totals + 9;
  for (;;) {
    unsigned long long q = 0;
    if (lane == 0) q = atomicAdd(queue, 1ull);
    q = XG::bcast(q, 0);
    if (q >= (unsigned long long)n) break;
    const int64_t idx = (int64_t)q;
    const double P = a.P[idx];
    XV y;
#pragma unroll
    for (int r = 0; r < XWR; ++r) {
      const int g = lane + XL * r;
      y.v[r] = (g == 0) ? a.T[idx] : (g < N ? a.Y[(int64_t)(g - 1) * n + idx] : 0.0);
    }
    const XCount c = xintegrate(ch, P, w, a.p, idx, y);
    double sum = 0.0;
#pragma unroll
    for (int r = 0; r < XWR; ++r) {
      const int g = lane + XL * r;
      if (g == 0) a.T[idx] = y.v[r];
      if (g >= 1 && g < N) {
        a.Y[(int64_t)(g - 1) * n + idx] = y.v[r];
        sum += y.v[r];
      }
    }
    sum = XG::sum(sum);
    if (lane == 0) {
      a.Y[(int64_t)(N - 1) * n + idx] = 1.0 - sum;
      if (a.status) a.status[idx] = c.status;
      if (a.counters) {
        const int32_t cc[8] = {c.nstep, c.naccpt, c.nrejct, c.nfcn, c.njac, c.narn, c.kdim,
                               c.status};
        for (int q = 0; q < 8; ++q) a.counters[(int64_t)q * n + idx] = cc[q];
      }
      const unsigned long long c7[7] = {
          (unsigned long long)c.nstep, (unsigned long long)c.naccpt, (unsigned long long)c.nrejct,
          (unsigned long long)c.nfcn,  (unsigned long long)c.njac,   (unsigned long long)c.narn,
          (unsigned long long)c.kdim};
      for (int q = 0; q < 7; ++q) atomicAdd(a.totals + q, c7[q]);
      if (c.status) atomicAdd(a.totals + 7, 1ull);
      atomicMax(a.totals + 8, (unsigned long long)c.nstep);
    }
    XG::sync();
  }
}

// unit entry: phi_1..phi_p (tau H) e1 of one m x m matrix, on one warp
__global__ void k_exprb_phi(const double *H, int m, int p, double tau, double *out,
                            double *scratch, int N) {
  XWork w = carve_xwork(scratch, N);
  for (int e = threadIdx.x; e < m * m; e += XL) w.H[(e / m) * N + e % m] = H[e];
  XG::sync();
  const double *Z = xphi(N, m, p, tau, w);
  for (int e = threadIdx.x; e < m * p; e += XL)
    out[e] = Z ? Z[(e / p) * (m + p) + m + e % p] : NAN;  // out[i * p + k - 1] = phi_k[i]
}

// unit entry: the right-hand side (with and without the Jacobian's assembly)
// and the analytical Jacobian the method uses, one state per warp
__global__ void k_exprb_chem(MechLayout L, const double *tab, const int *itab,
                             const unsigned char *hot, int hot_smem, const double *y,
                             const double *P, int64_t n, double *f, double *f2, double *J,
                             double *scratch, int64_t slots) {
  extern __shared__ __align__(16) unsigned char xsmem[];
  const MechView m = make_view(L, tab, itab);
  const int N = m.ns, lane = XG::lane();
  const HotTables h = stage_hot(L, hot, hot_smem != 0, xsmem);
  const int64_t slot = (int64_t)blockIdx.x;
  if (slot >= slots) return;
  double *gs = scratch + slot * (int64_t)xslot_doubles(N);
  const TeamBuf<double> t = xcarve(L, xsmem + (hot_smem ? hot_offsets(L).bytes : 0), gs);
  const XChem ch{m, h, t};
  for (int64_t i = slot; i < n; i += (int64_t)gridDim.x) {
    XV yy, ff;
#pragma unroll
    for (int r = 0; r < XWR; ++r) {
      const int g = lane + XL * r;
      yy.v[r] = g < N ? y[(int64_t)g * n + i] : 0.0;
      ff.v[r] = 0.0;
    }
    ch.jacobian(P[i], yy, ff);
#pragma unroll
    for (int r = 0; r < XWR; ++r) {
      const int g = lane + XL * r;
      if (g < N) f[(int64_t)g * n + i] = ff.v[r];
    }
    for (int e = lane; e < N * N; e += XL) J[(int64_t)e * n + i] = t.J[(e % N) * t.ld + e / N];
    XG::sync();
    ch.rates(P[i], yy, ff);
#pragma unroll
    for (int r = 0; r < XWR; ++r) {
      const int g = lane + XL * r;
      if (g < N) f2[(int64_t)g * n + i] = ff.v[r];
    }
    XG::sync();
  }
}

// whether the tables are staged, and their bytes; false when not even one
// warp's buffers fit
bool xshape(const MechLayout &L, int &hot_smem, size_t &fixed) {
  const size_t budget = BLOCK_SMEM, hot = hot_offsets(L).bytes, per = xwarp_bytes(L);
  if (per > budget) return false;
  hot_smem = hot + per <= budget;
  fixed = hot_smem ? hot : 0;
  return true;
}

}  // namespace

struct kin_exprb {
  int device = 0;
  MechLayout L;
  double *d_tab = nullptr;
  int *d_itab = nullptr;
  unsigned long long *d_totals = nullptr;
  double *d_scratch = nullptr;
  unsigned char *d_hot = nullptr;
  int64_t slots = 0;
  cudaStream_t last_stream = nullptr;
};

extern "C" void kin_exprb_destroy(kin_exprb *x) {
  if (!x) return;
  cudaFree(x->d_tab);
  cudaFree(x->d_itab);
  cudaFree(x->d_totals);
  cudaFree(x->d_scratch);
  cudaFree(x->d_hot);
  delete x;
}

extern "C" int kin_exprb_create(const kin_mech_desc *desc, kin_exprb **out) {
  if (!desc || !out) return KIN_ERR_INVALID_ARG;
  *out = nullptr;
  MechLayout L;
  std::vector<double> dt;
  std::vector<int> it;
  const int rc = build_tables(desc, L, dt, it);
  if (rc) return rc;
  if (L.ns > XSPECIES) return KIN_ERR_UNSUPPORTED;
  int dev = 0, sms = 0;
  KIN_CUDA_TRY(cudaGetDevice(&dev));
  KIN_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const std::vector<unsigned char> hot = build_hot(L, dt, it);
  kin_exprb *x = new kin_exprb();
  x->device = dev;
  x->L = L;
  x->slots = (int64_t)sms * 16;  // one per resident warp (128 registers: at most 16 per SM)
  const size_t sbytes = (size_t)x->slots * xslot_doubles(L.ns) * sizeof(double);
  if (cudaMalloc(&x->d_tab, sizeof(double) * L.nd) != cudaSuccess ||
      cudaMalloc(&x->d_itab, sizeof(int) * L.ni) != cudaSuccess ||
      cudaMalloc(&x->d_totals, sizeof(unsigned long long) * 16) != cudaSuccess ||
      cudaMalloc(&x->d_hot, hot.size()) != cudaSuccess ||
      cudaMalloc(&x->d_scratch, sbytes) != cudaSuccess) {
    (void)cudaGetLastError();
    kin_exprb_destroy(x);
    return KIN_ERR_NOMEM;
  }
  if (cudaMemcpy(x->d_hot, hot.data(), hot.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(x->d_tab, dt.data(), sizeof(double) * L.nd, cudaMemcpyHostToDevice) !=
          cudaSuccess ||
      cudaMemcpy(x->d_itab, it.data(), sizeof(int) * L.ni, cudaMemcpyHostToDevice) !=
          cudaSuccess ||
      cudaMemset(x->d_totals, 0, sizeof(unsigned long long) * 16) != cudaSuccess) {
    (void)cudaGetLastError();
    kin_exprb_destroy(x);
    return KIN_ERR_CUDA;
  }
  *out = x;
  return KIN_OK;
}

extern "C" int kin_integrate_exprb(kin_exprb *x, double *Y, double *T, const double *P,
                                   int64_t n, double dt, double rtol, double atol, double kappa,
                                   const double *h0, int32_t max_steps, int32_t *status,
                                   int32_t *counters, void *stream) {
  if (!x || n < 0) return KIN_ERR_INVALID_ARG;
  if (n > 0 && (!Y || !T || !P)) return KIN_ERR_INVALID_ARG;
  if (!(dt > 0.0) || !(rtol > 0.0) || !(atol > 0.0) || !std::isfinite(dt) || !(kappa >= 0.0) ||
      !std::isfinite(kappa) || max_steps < 1)
    return KIN_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  x->last_stream = st;
  KIN_CUDA_TRY(cudaMemsetAsync(x->d_totals, 0, sizeof(unsigned long long) * 16, st));
  if (n == 0) return KIN_OK;
  int dev = 0, sms = 0;
  KIN_CUDA_TRY(cudaGetDevice(&dev));
  if (dev != x->device) return KIN_ERR_INVALID_ARG;
  KIN_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  XArgs a;
  a.L = x->L;
  a.tab = x->d_tab;
  a.itab = x->d_itab;
  a.Y = Y;
  a.T = T;
  a.P = P;
  a.status = status;
  a.counters = counters;
  a.totals = x->d_totals;
  a.p.rtol = rtol;
  a.p.atol = atol;
  a.p.dt = dt;
  a.p.kappa = kappa;
  a.p.max_steps = max_steps;
  a.p.n = n;
  a.p.h0 = h0;
  a.scratch = x->d_scratch;
  a.slots = x->slots;
  a.hot = x->d_hot;
  size_t fixed = 0;
  if (!xshape(x->L, a.hot_smem, fixed)) return KIN_ERR_UNSUPPORTED;
  const size_t budget = BLOCK_SMEM, per = xwarp_bytes(x->L);
  auto kern = k_integrate_exprb;
  KIN_CUDA_TRY(open_smem(kern));
  int warps = 0, per_sm = 0;
  for (int wp = 8; wp >= 1; wp >>= 1) {
    const size_t smw = fixed + (size_t)wp * per;
    if (smw > budget) continue;
    int nb = 0;
    KIN_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, 32 * wp, smw));
    if (nb * wp > per_sm * warps) {
      warps = wp;
      per_sm = nb;
    }
  }
  if (warps < 1 || per_sm < 1) return KIN_ERR_UNSUPPORTED;
  const size_t sm = fixed + (size_t)warps * per;
  int64_t grid = (int64_t)sms * per_sm;
  const int64_t need = (n + warps - 1) / warps;
  if (grid > need) grid = need;
  if (grid * warps > x->slots) grid = x->slots / warps;  // one workspace slot per warp
  if (grid < 1) return KIN_ERR_UNSUPPORTED;
  kern<<<(unsigned)grid, 32 * warps, sm, st>>>(a);
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}

extern "C" int kin_exprb_get_stats(kin_exprb *x, int64_t *out) {
  if (!x || !out) return KIN_ERR_INVALID_ARG;
  unsigned long long t[16];
  KIN_CUDA_TRY(cudaStreamSynchronize(x->last_stream));
  KIN_CUDA_TRY(cudaMemcpy(t, x->d_totals, sizeof t, cudaMemcpyDeviceToHost));
  for (int i = 0; i < 9; ++i) out[i] = (int64_t)t[i];
  return out[7] > 0 ? KIN_ERR_STATE_FAILED : KIN_OK;
}

extern "C" int kin_exprb_phi(kin_exprb *x, const double *H, int32_t m, int32_t p, double tau,
                             double *out, void *stream) {
  if (!x || !H || !out || m < 1 || p < 1 || m > x->L.ns || p > XKP || !std::isfinite(tau))
    return KIN_ERR_INVALID_ARG;
  k_exprb_phi<<<1, XL, 0, (cudaStream_t)stream>>>(H, m, p, tau, out, x->d_scratch, x->L.ns);
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}

extern "C" int kin_exprb_chem(kin_exprb *x, const double *y, const double *P, int64_t n,
                              double *f, double *f_rates, double *J, void *stream) {
  if (!x || n < 0 || (n > 0 && (!y || !P || !f || !f_rates || !J))) return KIN_ERR_INVALID_ARG;
  if (n == 0) return KIN_OK;
  int hot_smem = 0;
  size_t fixed = 0;
  if (!xshape(x->L, hot_smem, fixed)) return KIN_ERR_UNSUPPORTED;
  const size_t sm = fixed + xwarp_bytes(x->L);
  KIN_CUDA_TRY(open_smem(k_exprb_chem));
  const int64_t grid = n < x->slots ? n : x->slots;
  k_exprb_chem<<<(unsigned)grid, XL, sm, (cudaStream_t)stream>>>(
      x->L, x->d_tab, x->d_itab, x->d_hot, hot_smem, y, P, n, f, f_rates, J, x->d_scratch,
      x->slots);
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}
