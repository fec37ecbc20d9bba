// Radau IIA on the concentration-based reactor, one state per team of warps,
// with a sparse LU of the Newton matrices: the reformulation the
// paper proposes for large models (Sec. 3.3, "memory traffic"; Sec. 4),
// where a Jacobian in species concentrations is sparse and admits sparse
// factorisation.
//
// State (per unit mass of mixture, constant pressure): T, the volume V and
// the moles n_k of every species but the last, the inert bath gas, whose
// moles close P V = n Ru T.  With C_k = n_k / V and Ctot = P / (Ru T):
//   dn_k/dt = V wdot_k,   dT/dt = -sum_k H_k wdot_k / sum_k C_k Cp_k,
//   dV/dt = V (sum_k wdot_k / Ctot + (dT/dt) / T).
// Two species are coupled in the Jacobian only through a reaction both take
// part in, or a collision efficiency that differs from the bath gas's (which
// must be the default, 1); the T and V rows and columns are full.
//
// The vectors hold the variables in elimination order: the host (kin_conc.cu)
// orders the species by minimum degree and puts T and V last, so the LU needs
// no pivoting and fills only the symbolic pattern.  The matrices are stored
// dense and entries outside the pattern stay zero; the blocked elimination of
// kin_team.cuh (panels of four columns in the given order) skips zero entries
// of a pivot row, which leaves the pattern's entries with the operations of an
// elimination over the pattern's lists, in their order.
// One state per team of three warps as in kin_team.cuh, whose commands, linear
// algebra and tables are shared; this file adds the form's right-hand side and
// Jacobian.  Measured (CH4-like, 4000 states, dt = 1e-5 s, FP32 matrices):
// 276 ms with a warp per state and an elimination over lists of the pattern's
// entries, 152 ms now, the same bits.
// The moles' absolute tolerance is atol / W_k, so that an error in n_k weighs
// as the mass-fraction error W_k dn_k does in the mass-fraction form (T and V
// take atol).
#pragma once
#include "kin_team.cuh"

namespace kin {

struct ConcView {
  int N;           // ns + 1 unknowns
  int posT, posV;  // elements of T and V
  const int *var;  // [N] element -> variable: 0 T, 1 V, 2 + k the moles of species k
  const int *posn; // [ns - 1] species k -> element
  const double *aw;  // [N] factor on atol per element: 1 for T and V, 1 / W_k for n_k
};

template <typename LT>
struct TeamConc {
  static constexpr bool PIVOT = false;
  const MechView &m;
  const HotTables &h;  // its col holds elements, not species
  const TeamBuf<LT> &t;
  const ConcView &cv;

  __device__ __forceinline__ int n() const { return cv.N; }
  __device__ __forceinline__ double atol_w(int g) const { return g < cv.N ? cv.aw[g] : 1.0; }

  // concentrations of species into C (the bath gas's from Ctot); returns the
  // active species' sum
  __device__ __forceinline__ double concentrations(const WVecT<2> &y, double iV, double Ctot,
                                                   double *C) const {
    using G = Grp<32>;
    const int lane = G::lane();
    double sC = 0.0;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int g = lane + 32 * r;
      if (g < cv.N) {
        const int v = cv.var[g];
        if (v >= 2) {
          const double c = y.v[r] * iV;
          C[v - 2] = c;
          sC += c;
        }
      }
    }
    sC = G::sum(sC);
    if (lane == 0) C[m.ns - 1] = Ctot - sC;
    __syncwarp();
    return sC;
  }

  // f by element from fT, fV and the species' rates wd
  __device__ __forceinline__ bool spread(double fT, double fV, double V, const double *wd,
                                         WVecT<2> &f) const {
    const int lane = threadIdx.x & 31;
    bool ok = isfinite(fT) && isfinite(fV);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int g = lane + 32 * r;
      f.v[r] = 0.0;
      if (g < cv.N) {
        const int v = cv.var[g];
        const double val = (v == 0) ? fT : (v == 1) ? fV : V * wd[v - 2];
        f.v[r] = val;
        ok &= isfinite(val);
      }
    }
    return Grp<32>::all(ok);
  }

  // Right-hand side on one warp: y from its g buffer, f into its C buffer.
  __device__ __noinline__ void chem_stage(int wt) const {
    using G = Grp<32>;
    const int lane = G::lane(), ns = m.ns, in = ns - 1;
    double *C = t.C(wt), *g = t.g(wt), *q = t.q(wt);
    WVecT<2> y, f;
    vec_load(n(), g, y);
    __syncwarp();
    const double T = elem<32>(y, cv.posT), V = elem<32>(y, cv.posV);
    const double iV = 1.0 / V, invT = 1.0 / T, logT = log(T);
    const double Ctot = t.ctl->P / (RU * T);
    (void)concentrations(y, iV, Ctot, C);
    double cpl = 0.0, hs[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int k = lane + 32 * r;
      hs[r] = 0.0;
      if (k < ns) {
        const int rg = range_of(m, k, T);
        const double cp = poly_cp(m.cp + (2 * k + rg) * NCP, T);
        g[k] = poly_g(m.gb + (2 * k + rg) * NG, T, logT, invT);
        hs[r] = poly_h(m.h + (2 * k + rg) * NH, T, invT);
        cpl += C[k] * cp;
      }
    }
    const double Cs = G::sum(cpl);  // sum_k C_k cp_k / R
    __syncwarp();
    warp_rates(m, h, C, g, q, T, logT, invT, Ctot);
    __syncwarp();
    double hw = 0.0, ww = 0.0;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int k = lane + 32 * r;
      if (k < in) {
        const double w = net_rate(h, q, k);
        g[k] = w;  // the Gibbs energies are spent
        hw += hs[r] * w;
        ww += w;
      }
    }
    const double Hs = G::sum(hw), Ws = G::sum(ww);
    const double fT = -T * Hs / Cs;
    const double fV = V * (Ws / Ctot + t_mul(fT, invT));
    __syncwarp();
    const bool ok = spread(fT, fV, V, g, f);
    __syncwarp();
    vec_store(n(), C, f);
    if (lane == 0) t.ctl->ret[wt] = ok ? 0 : 4;
  }

  // Leader, before the JAC command (scratch as in TeamMassFrac; ctl.S holds
  // sum_k C_k cp_k / R and ctl.rho the volume)
  __device__ void jac_prepare(const WVecT<2> &y) const {
    using G = Grp<32>;
    const int lane = G::lane(), ns = m.ns, nv = t.nv;
    double *hs = t.js + 4 * nv, *cpk = t.js + 5 * nv;
    const double T = elem<32>(y, cv.posT), V = elem<32>(y, cv.posV);
    const double iV = 1.0 / V, invT = 1.0 / T, logT = log(T);
    const double Ctot = t.ctl->P / (RU * T);
    const double sC = concentrations(y, iV, Ctot, t.C(0));
    double cpl = 0.0, dcpl = 0.0;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int k = lane + 32 * r;
      if (k < ns) {
        const int rg = range_of(m, k, T);
        const double *cc = m.cp + (2 * k + rg) * NCP;
        const double cp = poly_cp(cc, T), C = t.C(0)[k];
        t.g(0)[k] = poly_g(m.gb + (2 * k + rg) * NG, T, logT, invT);
        hs[k] = poly_h(m.h + (2 * k + rg) * NH, T, invT);
        cpk[k] = cp;
        cpl += C * cp;
        dcpl += C * poly_dcp(cc, T);
      }
    }
    const double Cs = G::sum(cpl), dCsT = G::sum(dcpl);
    if (lane == 0) {
      TeamCtl &c = *t.ctl;
      c.T = T;
      c.logT = logT;
      c.invT = invT;
      c.rho = V;
      c.S = Cs;
      c.cpm = sC;
      c.dcpm = dCsT;
      c.ret[0] = c.ret[1] = c.ret[2] = 0;
    }
  }

  // The right-hand side (into warp 0's g buffer) and the Jacobian (into J).
  __device__ __noinline__ void jac(int wt) const {
    using G = Grp<32>;
    const int lane = G::lane(), ns = m.ns, in = ns - 1, N = cv.N, nv = t.nv, nr = m.nr, ld = t.ld;
    TeamCtl &ct = *t.ctl;
    double *B = t.js + nv, *Tc = t.js + 2 * nv, *hs = t.js + 4 * nv, *cpk = t.js + 5 * nv,
           *wd = t.js + 6 * nv;
    double *sig = t.js + 8 * nv, *dq = sig + nr, *D = dq + nr;
    const int nslots = h.off[nr - 1] + rec_nre(h.rec[nr - 1]) + rec_npr(h.rec[nr - 1]);
    const double T = ct.T, logT = ct.logT, invT = ct.invT, V = ct.rho, Cs = ct.S, sC = ct.cpm;
    const double Ctot = ct.P / (RU * T), iV = 1.0 / V, *C = t.C(0), *g = t.g(0);
    double *q = t.q(0);
    for (int e = lane + 32 * wt; e < N * ld; e += TEAM_NT) t.Jd[e] = 0.0;
#pragma unroll 1
    for (int i = lane + 32 * wt; i < nr; i += TEAM_NT) {
      const ReactionJac r = reaction_jac(m, h, C, g, hs, i, T, logT, invT, Ctot);
      q[i] = r.q;
      sig[i] = r.sig;
      dq[i] = r.dqdT_nV;  // at fixed n and V only Ctot (and with it M) moves
      const uint2 rc = h.rec[i];
      const int nre = rec_nre(rc), nsl = nre + rec_npr(rc);
#pragma unroll 1
      for (int s = 0; s < nsl; ++s) {
        const bool re = s < nre;
        const unsigned sl = re ? rc.x : rc.y;
        const int mine = re ? s : s - nre, cnt = re ? nre : nsl - nre;
        double p = re ? r.pkf : r.pkr;
#pragma unroll 1
        for (int x = 0; x < cnt; ++x)
          if (x != mine) p *= C[(sl >> (8 * x)) & 255];
        D[h.off[i] + s] = p;
      }
      if (i < m.nfall) {
        const int e0 = m.eff0[i], ne = meta_neff(m.meta[i]);
#pragma unroll 1
        for (int e = e0; e < e0 + ne; ++e) D[nslots + e] = t_mul(r.u, m.eff[e]);
      }
    }
    named_sync(t.bar, TEAM_NT);
    if (wt == 0) {
      double hw = 0.0, ww = 0.0;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int k = lane + 32 * r;
        if (k < in) {
          const double w = net_rate(h, q, k);
          wd[k] = w;
          hw += hs[k] * w;
          ww += w;
        }
      }
      const double Hs = G::sum(hw), Ws = G::sum(ww);
      const double fT = -T * Hs / Cs;
      const double fV = V * (Ws / Ctot + t_mul(fT, invT));
      __syncwarp();
      WVecT<2> f;
      const bool ok = spread(fT, fV, V, wd, f);
      vec_store(N, t.g(0), f);
      if (lane == 0) {
        ct.Hw = fT;
        ct.CPw = Ws;
        if (!ok) ct.ret[0] = 4;
      }
    } else {
      for (int e = lane + 32 * (wt - 1); e < in; e += 64) {
        const int k = h.rank[e];
        double a = 0.0, b = 0.0, tc = 0.0;
        row_sums(h, sig, dq, k, b, tc);
        row_terms(h, D, k, -1, t.Jd + cv.posn[k] * ld, a);
        B[k] = b;
        Tc[k] = tc;
      }
    }
    named_sync(t.bar, TEAM_NT);
    // species rows' T and V columns; the sums the T and V rows need
    if (wt == 0) {
      double sHB = 0.0, sHT = 0.0, sCW = 0.0, sB = 0.0, sTc = 0.0, sCC = 0.0;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int k = lane + 32 * r;
        if (k < in) {
          double *Jr = t.Jd + cv.posn[k] * ld;
          Jr[cv.posT] = V * Tc[k];
          Jr[cv.posV] = wd[k] - B[k];
          sHB += hs[k] * B[k];
          sHT += hs[k] * Tc[k];
          sCW += cpk[k] * wd[k];
          sB += B[k];
          sTc += Tc[k];
          sCC += cpk[k] * C[k];
        }
      }
      double *o = t.js;  // free: the form has no inert column
      const double v[6] = {G::sum(sHB), G::sum(sHT), G::sum(sCW),
                           G::sum(sB),  G::sum(sTc), G::sum(sCC)};
      if (lane < 6) o[lane] = lane == 0 ? v[0] : lane == 1 ? v[1] : lane == 2 ? v[2]
                              : lane == 3 ? v[3] : lane == 4 ? v[4] : v[5];
    }
    named_sync(t.bar, TEAM_NT);
    const double sHB = t.js[0], sHT = t.js[1], sCW = t.js[2], sB = t.js[3], sTc = t.js[4],
                 sCC = t.js[5];
    const double fT = ct.Hw, Ws = ct.CPw, dCsT = ct.dcpm, cpin = cpk[in];
    bool ok = true;
    for (int c = lane + 32 * wt; c < N; c += TEAM_NT) {
      const int v = cv.var[c];
      double dTH, dCs, dWs;  // d(T Hs), dCs, d(sum wdot) * V along phi_c
      if (v >= 2) {
        double sh = 0.0, sw = 0.0;
#pragma unroll 2
        for (int k = 0; k < in; ++k) {
          const double jk = t.Jd[cv.posn[k] * ld + c];
          sh += hs[k] * jk;
          sw += jk;
        }
        dTH = T * iV * sh;
        dCs = (cpk[v - 2] - cpin) * iV;
        dWs = sw;
      } else if (v == 1) {
        dTH = -T * iV * sHB;
        dCs = (cpin * sC - sCC) * iV;
        dWs = -sB;
      } else {
        dTH = sCW + T * sHT;
        dCs = dCsT - cpin * Ctot * invT;
        dWs = V * sTc;
      }
      const double jt = -(dTH + fT * dCs) / Cs;
      double jv = dWs / Ctot + V * jt * invT;
      if (v == 1) jv += Ws / Ctot + fT * invT;
      if (v == 0) jv += V * (Ws / (Ctot * T) - fT * invT * invT);
      LT *Jc = t.J + (size_t)c * ld;
#pragma unroll 2
      for (int i = 0; i < N; ++i) {
        const double x = i == cv.posT ? jt : i == cv.posV ? jv : t.Jd[i * ld + c];
        ok &= isfinite(x);
        Jc[i] = LT(x);
      }
    }
    if (!G::all(ok) && lane == 0) ct.ret[wt] = 4;
  }
};

}  // namespace kin
