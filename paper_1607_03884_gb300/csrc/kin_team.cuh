// The WARP layout with 32 lanes: one state per team of three warps.
//
// What bounds a large mechanism on this chip is the FP64 unit (an SM
// sub-partition issues one FP64 warp instruction per 64 cycles, independent or
// not) and, next to it, latency: a state's matrices fill 35 to 45 KB of
// shared memory, so four or five states fit an SM, and with one warp each the
// FP64 unit was busy a third of the time (CH4-like, FP32 matrices, 136 M
// cycles per state: 41 % rates, 21 % Jacobian assembly by shared-memory
// atomics, 20 % factorisation, 11 % substitution).  Here three warps work for
// a state:
//   * warp 0 (the leader) runs the step driver of kin_warp.cuh and posts
//     commands in shared memory; warps 1 and 2 wait at the team's named
//     barrier and execute their part of each command;
//   * the three Newton stages' right-hand sides run side by side, a stage per
//     warp, each with its own concentrations and rates;
//   * the Jacobian's reactions are dealt over the warps and its rows gathered
//     per species in a fixed order (no atomics, deterministic);
//   * the real factorisation and substitution run on warp 0, the complex ones
//     on warps 1 and 2, blocked by panels of four columns: the panel's rows in
//     registers, the trailing matrix read and written once per panel;
//   * the rate tables every stage walks (Arrhenius, reaction slots, 2^(j/256),
//     species lists: 35 KB for CH4) are staged in shared memory once per block
//     and serve all its teams.
// Every matrix entry sees the same operations in the same order as in a
// column-by-column elimination, so FP32 matrices factorise to the same bits.
// Measured on CH4-like states (warp per state -> team): 4000 states, dt =
// 1e-4 s, FP32 matrices 579 -> 333 ms, the same bits; dt = 1e-6 s, FP64
// matrices 380 -> 208 ms.  Also tried, FP32: two rows per lane in the trailing
// update, as FP64 has it, 333 -> 340 ms.
#pragma once
#include "kin_warp.cuh"

namespace kin {

constexpr int TEAM_WARPS = 3, TEAM_NT = 32 * TEAM_WARPS;
// Teams per block.  384 threads leave 168 registers each; 672 leave 80, which
// FP32 matrices of up to TEAM_MANY_N unknowns live with: their states are small
// and short of work for three warps, so that four per SM leave the FP64 unit
// idle once a batch has more.  FP32, dt = 1e-6 s, ms with one warp per state
// (16 per SM) / four teams / seven: 13 species, 20000 states 296 / 314 / 297,
// 3000: 51 / 50 / 47; 17 species and 27 reactions, 20000: 315 / 335 / 317, 3000:
// 54 / 53 / 50, 700: 24 / 15 / 15; 24 species and 100 reactions, 20000: 475 / 388
// / 381, 3000: 79 / 63 / 61, 700: 36 / 18 / 19; the concentration form of 13
// species, 10000: 142 / 153 / 143.  Beyond, 40 species: 3000: 130 / 79 / 79; and
// FP64 matrices lose by the spills (24 species, 20000: 631 / 647, 53: 258 / 275).
constexpr int TEAM_MAX = 4, TEAM_MANY = 7, TEAM_MANY_N = 24;
constexpr int TEAM_PANEL = 4;  // columns per factorisation panel

// Rounded products and fused sums, written out where the matrices' bits
// depend on them.
__device__ __forceinline__ float t_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double t_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float t_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double t_fma(double a, double b, double c) { return __fma_rn(a, b, c); }

// s -= l u (complex).  FP32 keeps the rounding of the column-by-column form
// (product, fused difference, subtraction); FP64, whose instructions are the
// cost, takes four fused operations instead of six.
__device__ __forceinline__ void csub(float &sr, float &si, float lr, float li, float ur, float ui) {
  sr -= t_fma(lr, ur, -t_mul(li, ui));
  si -= t_fma(lr, ui, t_mul(li, ur));
}
__device__ __forceinline__ void csub(double &sr, double &si, double lr, double li, double ur,
                                     double ui) {
  sr = t_fma(li, ui, t_fma(-lr, ur, sr));
  si = t_fma(-li, ur, t_fma(-lr, ui, si));
}

// ---------------------------------------------------------------------------
// Tables staged per block
// ---------------------------------------------------------------------------
struct HotTables {
  const double *lnA, *b, *Th, *dnu, *etab;
  const uint2 *rec;  // reactant slots and type | counts; product slots (a byte each)
  const int *net0, *occ0;
  const unsigned short *net;  // species -> reaction << 4 | (nu + 8)
  // species -> reaction << 3 | slot, sorted by round of 32 reactions, slot's
  // position in the reaction (reactants, then products) and reaction
  const unsigned short *occ;
  const unsigned char *rank;  // active species by list length, longest first
  // the Jacobian's sparse rows as lists of terms: a reaction's derivative by
  // the species in a slot (its index: off[reaction] + position among the
  // slots), then by a collision partner (nslots + its efficiency entry)
  const unsigned short *off;   // [nr] first slot index
  const unsigned char *col;    // [nslots + neff] species
  const int *term0;            // [ns] first term of a species' row
  const unsigned short *term;  // index << 1 | (1 for a reactant's row: minus)
};

__host__ __device__ __forceinline__ int rec_type(uint2 r) { return (r.x >> 24) & 3; }
__host__ __device__ __forceinline__ int rec_nre(uint2 r) { return (r.x >> 26) & 3; }
__host__ __device__ __forceinline__ int rec_npr(uint2 r) { return (r.x >> 28) & 3; }
// species in slot s: reactants 0-2, products 3-5
__host__ __device__ __forceinline__ int rec_slot(uint2 r, int s) {
  return s < 3 ? (int)(r.x >> (8 * s)) & 255 : (int)(r.y >> (8 * (s - 3))) & 255;
}

// Where the tables lie in their buffer (byte offsets), which the host fills
// once per mechanism (build_hot) and a block copies to shared memory.
struct HotOffsets {
  size_t d, rec, ints, net, occ, off, term, rank, col, bytes;
};
__host__ __device__ inline HotOffsets hot_offsets(const MechLayout &L) {
  HotOffsets o;
  const size_t nr = L.nr, ns = L.ns, ncsr = L.ni - L.icsr;
  o.d = 0;
  o.rec = sizeof(double) * (4 * nr + EXP_TAB);
  o.ints = o.rec + sizeof(uint2) * nr;
  o.net = o.ints + sizeof(int) * 3 * (ns + 2);
  o.occ = o.net + 2 * ncsr;
  o.off = o.occ + 2 * (size_t)L.nslots;
  o.term = o.off + 2 * nr;
  o.rank = o.term + 2 * (size_t)L.nterms;
  o.col = o.rank + 64;
  o.bytes = (o.col + L.nslots + L.neff + 15) / 16 * 16;
  return o;
}

__device__ __forceinline__ HotTables hot_view(const MechLayout &L, const unsigned char *p) {
  const HotOffsets o = hot_offsets(L);
  const double *d = reinterpret_cast<const double *>(p);
  const int nr = L.nr, *ints = reinterpret_cast<const int *>(p + o.ints);
  HotTables h;
  h.lnA = d;
  h.b = d + nr;
  h.Th = d + 2 * nr;
  h.dnu = d + 3 * nr;
  h.etab = d + 4 * nr;
  h.rec = reinterpret_cast<const uint2 *>(p + o.rec);
  h.net0 = ints;
  h.occ0 = ints + L.ns + 2;
  h.term0 = ints + 2 * (L.ns + 2);
  h.net = reinterpret_cast<const unsigned short *>(p + o.net);
  h.occ = reinterpret_cast<const unsigned short *>(p + o.occ);
  h.off = reinterpret_cast<const unsigned short *>(p + o.off);
  h.term = reinterpret_cast<const unsigned short *>(p + o.term);
  h.rank = p + o.rank;
  h.col = p + o.col;
  return h;
}

// the block's copy in shared memory, or the tables where they are when a
// mechanism's lists leave no room for a team beside them; whole block
__device__ __forceinline__ HotTables stage_hot(const MechLayout &L, const unsigned char *hot,
                                               bool copy, unsigned char *smem) {
  if (!copy) return hot_view(L, hot);
  const uint4 *src = reinterpret_cast<const uint4 *>(hot);
  uint4 *dst = reinterpret_cast<uint4 *>(smem);
  for (size_t e = threadIdx.x; e < hot_offsets(L).bytes / 16; e += blockDim.x) dst[e] = src[e];
  __syncthreads();
  return hot_view(L, smem);
}

// ---------------------------------------------------------------------------
// A team's shared memory
// ---------------------------------------------------------------------------
struct TeamCtl {
  int cmd, ret[TEAM_WARPS], piv[TEAM_PANEL], sing;
  double P, h, T, logT, invT, rho, S, cpm, dcpm, Hw, CPw;
};

template <typename LT>
struct TeamBuf {
  int ld, nv, wstride, bar;
  LT *J;             // global, column by column: entry (i, j) at j * ld + i
  LT *E1;
  cplx_t<LT> *E2;
  double *Jd;        // the FP64 assembly matrix, over E2
  double *w0, *w12;  // warp 0's C, g, q; warp 1's, then warp 2's
  double *js;        // Jacobian scratch, over E1 and warp 1's and 2's buffers
  LT *dr, *dd, *di;  // E2's pivots: Smith's ratio, denominator and its reciprocal
  LT *d1;            // reciprocals of E1's pivots (FP64)
  unsigned char *p1, *p2;  // row sources after all exchanges (p2: bit 7 Smith's case)
  TeamCtl *ctl;
  __host__ __device__ __forceinline__ double *C(int w) const {
    return w ? w12 + (w - 1) * wstride : w0;
  }
  __device__ __forceinline__ double *g(int w) const { return C(w) + nv; }
  __device__ __forceinline__ double *q(int w) const { return C(w) + 2 * nv; }
  // warp w's vectors of a difference Jacobian (team_fd_doubles)
  __host__ __device__ __forceinline__ double *fd(int w) const { return Jd + 3 * w * nv; }
};

__host__ __device__ inline int team_nv(int ns) { return (ns + 2) & ~1; }
__host__ __device__ inline int team_ld(int N) { return N | 1; }
// Three vectors per warp for a state per warp's difference Jacobian, in the
// assembly matrix's area (N x team_ld doubles), which that kernel leaves alone:
// the other areas are its warps' live rate buffers.  They fit from 10 species on.
__host__ __device__ inline size_t team_fd_doubles(int ns) {
  return 3 * TEAM_WARPS * (size_t)team_nv(ns);
}
__host__ __device__ inline bool team_fd_fits(int ns) {
  return team_fd_doubles(ns) <= (size_t)ns * team_ld(ns);
}
// Jacobian scratch in doubles: eight species vectors, two reaction vectors
// and the derivatives by slot and by collision partner
__host__ __device__ inline size_t team_js_doubles(const MechLayout &L) {
  return 8 * (size_t)team_nv(L.ns) + 2 * (size_t)L.nr + L.nslots + L.neff;
}
__host__ __device__ inline size_t team_bytes(const MechLayout &L, int N, size_t lt) {
  const int ns = L.ns, nr = L.nr;
  const size_t mat = (size_t)N * team_ld(N), w = (2 * (size_t)team_nv(ns) + nr) * sizeof(double);
  const size_t e1 = (mat * lt + 7) / 8 * 8;
  size_t mid = e1 + 2 * w;
  const size_t need = team_js_doubles(L) * sizeof(double);
  if (need > mid) mid = need;
  size_t b = (sizeof(TeamCtl) + 15) / 16 * 16 + w + mid;
  if (!warp_e2_global(lt)) b += 2 * mat * lt;
  b += 4 * (size_t)team_nv(N) * lt + 128;
  return (b + 15) / 16 * 16;
}

template <typename LT>
__host__ __device__ inline TeamBuf<LT> carve_team(const MechLayout &L, unsigned char *p, int team, int N,
                                  unsigned char *slot) {
  const int ns = L.ns, nr = L.nr;
  TeamBuf<LT> t;
  t.ld = team_ld(N);
  t.nv = team_nv(ns);
  t.wstride = 2 * t.nv + nr;
  t.bar = 1 + team;
  const size_t mat = (size_t)N * t.ld;
  t.ctl = reinterpret_cast<TeamCtl *>(p);
  p += (sizeof(TeamCtl) + 15) / 16 * 16;
  if (warp_e2_global(sizeof(LT))) {
    t.E2 = reinterpret_cast<cplx_t<LT> *>(slot);
    t.J = reinterpret_cast<LT *>(slot) + 2 * mat;
  } else {
    t.E2 = reinterpret_cast<cplx_t<LT> *>(p);
    p += 2 * mat * sizeof(LT);
    t.J = reinterpret_cast<LT *>(slot);
  }
  t.Jd = reinterpret_cast<double *>(t.E2);
  t.w0 = reinterpret_cast<double *>(p);
  p += t.wstride * sizeof(double);
  const size_t e1 = (mat * sizeof(LT) + 7) / 8 * 8, w2 = 2 * t.wstride * sizeof(double);
  const size_t need = team_js_doubles(L) * sizeof(double);
  t.E1 = reinterpret_cast<LT *>(p);
  t.js = reinterpret_cast<double *>(p);
  t.w12 = reinterpret_cast<double *>(p + e1);
  p += e1 + w2 > need ? e1 + w2 : need;
  t.dr = reinterpret_cast<LT *>(p);
  t.dd = t.dr + team_nv(N);
  t.di = t.dr + 2 * team_nv(N);
  t.d1 = t.dr + 3 * team_nv(N);
  p += 4 * (size_t)team_nv(N) * sizeof(LT);
  t.p1 = p;
  t.p2 = p + 64;
  return t;
}

__device__ __forceinline__ void named_sync(int id, int nt) {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nt) : "memory");
}

// ---------------------------------------------------------------------------
// Rates
// ---------------------------------------------------------------------------
// ln Kc's and the products' sums over a reaction's slots, in slot order
struct SlotSums {
  double fwd, rev, lnKc;
};
__device__ __forceinline__ SlotSums slot_sums(const HotTables &h, const double *C, const double *g,
                                              int i, uint2 r, double lnPf) {
  const int nre = rec_nre(r), npr = rec_npr(r);
  SlotSums o = {1.0, 1.0, t_fma(h.dnu[i], lnPf, -g[r.x & 255])};
  o.fwd = C[r.x & 255];
  o.rev = C[r.y & 255];
  if (nre > 1) {
    const int s = (r.x >> 8) & 255;
    o.lnKc -= g[s];
    o.fwd *= C[s];
  }
  if (nre > 2) {
    const int s = (r.x >> 16) & 255;
    o.lnKc -= g[s];
    o.fwd *= C[s];
  }
  o.lnKc += g[r.y & 255];
  if (npr > 1) {
    const int s = (r.y >> 8) & 255;
    o.lnKc += g[s];
    o.rev *= C[s];
  }
  if (npr > 2) {
    const int s = (r.y >> 16) & 255;
    o.lnKc += g[s];
    o.rev *= C[s];
  }
  return o;
}
// kf prod C' - kr prod C''
__device__ __forceinline__ double net_of(const SlotSums &o, double kf, const double *etab,
                                         double &kr) {
  kr = t_mul(kf, kexp(-o.lnKc, etab));
  return t_fma(kf, o.fwd, -t_mul(kr, o.rev));
}

__device__ __forceinline__ double collider(const MechView &m, const double *C, int i, double Ctot) {
  const int e0 = m.eff0[i], ne = meta_neff(m.meta[i]);
  double M = Ctot;
#pragma unroll 1
  for (int e = 0; e < ne; ++e) M += m.eff[e0 + e] * C[m.effsp[e0 + e]];
  return M;
}

// Net rates of all reactions on one warp: Troe, third-body and elementary
// reactions (the device order) in rounds of their own.
__device__ __forceinline__ void warp_rates(const MechView &m, const HotTables &h, const double *C,
                                           const double *g, double *q, double T, double logT,
                                           double invT, double Ctot) {
  const int lane = threadIdx.x & 31;
  const double lnPf = 2.5003366899611787 - logT;  // ln(Patm / Ru) - ln T
  double kr;
#pragma unroll 1
  for (int part = 0; part < 2; ++part) {
    const int e = part ? m.nfall : m.ntroe;
#pragma unroll 1
    for (int i = (part ? m.ntroe : 0) + lane; i < e; i += 32) {
      const double lnkf = h.lnA[i] + h.b[i] * logT - h.Th[i] * invT;
      const double kf = kexp(lnkf, h.etab);
      const SlotSums o = slot_sums(h, C, g, i, h.rec[i], lnPf);
      const double Rn = net_of(o, kf, h.etab, kr);
      const double M = collider(m, C, i, Ctot);
      double phi = M;
      if (part == 0)
        phi = troe_factor<false>(m.troe + NTROE * meta_troe(m.meta[i]), T, logT, invT, lnkf, 0.0,
                                 M, h.etab).P;
      q[i] = phi * Rn;
    }
  }
#pragma unroll 1
  for (int i = m.nfall + lane; i < m.nr; i += 32) {
    const double kf = kexp(h.lnA[i] + h.b[i] * logT - h.Th[i] * invT, h.etab);
    const SlotSums o = slot_sums(h, C, g, i, h.rec[i], lnPf);
    q[i] = net_of(o, kf, h.etab, kr);
  }
}

// sum over species k's net list of nu q; the small integer nu is built as a
// double in the integer pipe
__device__ __forceinline__ double net_rate(const HotTables &h, const double *q, int k) {
  double w = 0.0;
#pragma unroll 2
  for (int e = h.net0[k]; e < h.net0[k + 1]; ++e) {
    const int code = h.net[e], nu = (code & 15) - 8, a = abs(nu);
    const int hi = (nu < 0 ? 0x80000000 : 0) | (a == 1 ? 0x3ff00000 : a == 2 ? 0x40000000 : 0x40080000);
    w = fma(__hiloint2double(hi, 0), q[code >> 4], w);
  }
  return w;
}

// Mass-fraction right-hand side of one state on one warp (warp_chem's
// formulas, without the Jacobian): 0 or 4 (non-finite).
template <int DUMMY = 0>
__device__ __noinline__ int team_rhs(const MechView &m, const HotTables &h, double *C, double *g,
                                     double *q, double P, const WVecT<2> &y, WVecT<2> &f) {
  using G = Grp<32>;
  const int lane = G::lane(), ns = m.ns, in = ns - 1, N = ns;
  const double T = G::bcast(y.v[0], 0);
  double sY = 0.0, sS = 0.0;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int e = lane + 32 * r;
    if (e >= 1 && e < N) {
      sY += y.v[r];
      sS += y.v[r] * m.invW[e - 1];
    }
  }
  sY = G::sum(sY);
  sS = G::sum(sS);
  const double Yin = 1.0 - sY;
  const double S = sS + Yin * m.invW[in];
  const double rho = P / (RU * T * S);
  const double logT = log(T), invT = 1.0 / T;
  double cpl = 0.0, hs[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int e = lane + 32 * r, k = e - 1;  // species k at element e (the inert at e = ns)
    hs[r] = 0.0;
    if (e >= 1 && e <= ns) {
      const double Yk = (e < N) ? y.v[r] : Yin;
      const int rg = range_of(m, k, T);
      C[k] = rho * Yk * m.invW[k];
      cpl = t_fma(t_mul(Yk, poly_cp(m.cp + (2 * k + rg) * NCP, T)), m.invW[k], cpl);
      hs[r] = poly_h(m.h + (2 * k + rg) * NH, T, invT);
      g[k] = poly_g(m.gb + (2 * k + rg) * NG, T, logT, invT);
    }
  }
  const double cpm = G::sum(cpl);
  __syncwarp();
  warp_rates(m, h, C, g, q, T, logT, invT, rho * S);
  __syncwarp();
  double hw = 0.0;
  bool ok = true;
  const double irho = 1.0 / rho;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int e = lane + 32 * r, k = e - 1;
    if (e >= 1 && e < N) {
      const double w = net_rate(h, q, k);
      f.v[r] = m.W[k] * w * irho;
      ok &= (__double2hiint(f.v[r]) & 0x7ff00000) != 0x7ff00000;
      hw += hs[r] * w;
    }
  }
  hw = G::sum(hw);
  const double fT = -(hw * T) / (rho * cpm);
  if (lane == 0) f.v[0] = fT;
  ok &= isfinite(fT);
  return G::all(ok) ? 0 : 4;
}

__device__ __forceinline__ double flip(double x, int sign) {
  return __hiloint2double(__double2hiint(x) ^ sign, __double2loint(x));
}

// sums over species k's reactions of nu sig and nu dq/dT
__device__ __forceinline__ void row_sums(const HotTables &h, const double *sig, const double *dq,
                                         int k, double &b, double &tc) {
#pragma unroll 2
  for (int o = h.occ0[k]; o < h.occ0[k + 1]; ++o) {
    const int code = h.occ[o], i = code >> 3, neg = (code & 7) < 3 ? 0x80000000 : 0;
    b += flip(sig[i], neg);
    tc += flip(dq[i], neg);
  }
}

// species k's sparse Jacobian row: its terms added to Jr[column], or to a for
// the inert's; the next term's operands are loaded before this one's store
__device__ __forceinline__ void row_terms(const HotTables &h, const double *D, int k, int inert,
                                          double *Jr, double &a) {
  const int e1 = h.term0[k + 1];
  int x = h.term0[k];
  int code = x < e1 ? h.term[x] : 0, col = h.col[code >> 1];
  double d = D[code >> 1];
#pragma unroll 1
  for (; x < e1; ++x) {
    const int c0 = col, neg = code << 31;
    const double v = flip(d, neg);
    code = x + 1 < e1 ? h.term[x + 1] : 0;
    col = h.col[code >> 1];
    d = D[code >> 1];
    if (c0 != inert)
      Jr[c0] += v;
    else
      a += v;
  }
}

// One reaction with what its Jacobian terms need: the net rate, the forward
// and (negated) reverse rate constants with the falloff factor, dq/dM,
// sum_l C_l dq/dC_l, dq/dT at fixed Y, and dq/dT at fixed moles and volume.
struct ReactionJac {
  double q, pkf, pkr, u, sig, dqdT, dqdT_nV;
};
__device__ __forceinline__ ReactionJac reaction_jac(const MechView &m, const HotTables &h,
                                                    const double *C, const double *g,
                                                    const double *hs, int i, double T, double logT,
                                                    double invT, double Ctot) {
  const uint2 rc = h.rec[i];
  const int nre = rec_nre(rc), npr = rec_npr(rc), type = rec_type(rc);
  const double lnkf = h.lnA[i] + h.b[i] * logT - h.Th[i] * invT;
  const double kf = kexp(lnkf, h.etab);
  const double dnu = h.dnu[i], lnPf = 2.5003366899611787 - logT;
  double dH = 0.0, lnKc = t_mul(dnu, lnPf), fwd = 1.0, rev = 1.0;
#pragma unroll 1
  for (int s = 0; s < nre; ++s) {
    const int k = rec_slot(rc, s);
    lnKc -= g[k];
    dH -= hs[k];
    fwd *= C[k];
  }
#pragma unroll 1
  for (int s = 0; s < npr; ++s) {
    const int k = rec_slot(rc, 3 + s);
    lnKc += g[k];
    dH += hs[k];
    rev *= C[k];
  }
  const double kr = t_mul(kf, kexp(-lnKc, h.etab));
  double phi = 1.0, dphi_dT = 0.0, dphi_dM = 0.0, M = Ctot;
  const double dlnkf = h.b[i] * invT + h.Th[i] * invT * invT;
  if (type != 0) {
    M = collider(m, C, i, Ctot);
    if (type == 1) {
      phi = M;
      dphi_dM = 1.0;
    } else {
      const TroeOut t = troe_factor<true>(m.troe + NTROE * meta_troe(m.meta[i]), T, logT, invT,
                                          lnkf, dlnkf, M, h.etab);
      phi = t.P;
      dphi_dT = t.P * t.dlnP_dT;
      dphi_dM = t.P * t.dlnP_dM;
    }
  }
  ReactionJac r;
  const double Rn = t_fma(kf, fwd, -t_mul(kr, rev));
  r.q = phi * Rn;
  const double dlnkr = dlnkf - (dH - dnu) * invT;
  r.u = Rn * dphi_dM;
  r.sig = phi * (nre * kf * fwd - npr * kr * rev) + r.u * (M - Ctot);
  r.dqdT = phi * (kf * dlnkf * fwd - kr * dlnkr * rev) + Rn * dphi_dT -
           (r.sig + r.u * Ctot) * invT;
  r.dqdT_nV = phi * (kf * dlnkf * fwd - kr * dlnkr * rev) + Rn * dphi_dT - r.u * Ctot * invT;
  r.pkf = phi * kf;
  r.pkr = -phi * kr;
  return r;
}

// ---------------------------------------------------------------------------
// Factorisation
// ---------------------------------------------------------------------------
// first row of the largest key >= 0 over rows k .. N-1 (rows lane and lane +
// 32), NaN never; -1 when there is none above zero
__device__ __forceinline__ int arg_pivot(float v0, float v1, int k, int N) {
  const int lane = threadIdx.x & 31;
  const unsigned FULL = 0xffffffffu;
  const unsigned a = (lane >= k && lane < N && v0 == v0) ? __float_as_uint(v0) + 1u : 0u;
  const unsigned b = (lane + 32 >= k && lane + 32 < N && v1 == v1) ? __float_as_uint(v1) + 1u : 0u;
  const unsigned best = __reduce_max_sync(FULL, a > b ? a : b);
  if (best <= 1u) return -1;
  const unsigned m0 = __ballot_sync(FULL, a == best), m1 = __ballot_sync(FULL, b == best);
  return m0 ? __ffs(m0) - 1 : 31 + __ffs(m1);
}
__device__ __forceinline__ int arg_pivot(double v0, double v1, int k, int N) {
  const int lane = threadIdx.x & 31;
  const unsigned FULL = 0xffffffffu;
  const long long b0 = __double_as_longlong(v0), b1 = __double_as_longlong(v1);
  const bool ok0 = lane >= k && lane < N && b0 <= 0x7ff0000000000000ll;
  const bool ok1 = lane + 32 >= k && lane + 32 < N && b1 <= 0x7ff0000000000000ll;
  const unsigned h0 = ok0 ? (unsigned)(b0 >> 32) + 1u : 0u, h1 = ok1 ? (unsigned)(b1 >> 32) + 1u : 0u;
  const unsigned hb = __reduce_max_sync(FULL, h0 > h1 ? h0 : h1);
  if (hb == 0u) return -1;
  const unsigned l0 = h0 == hb ? (unsigned)b0 : 0u, l1 = h1 == hb ? (unsigned)b1 : 0u;
  const unsigned lb = __reduce_max_sync(FULL, l0 > l1 ? l0 : l1);
  if (hb == 1u && lb == 0u) return -1;
  const unsigned m0 = __ballot_sync(FULL, h0 == hb && l0 == lb);
  const unsigned m1 = __ballot_sync(FULL, h1 == hb && l1 == lb);
  return m0 ? __ffs(m0) - 1 : 31 + __ffs(m1);
}

// value of row i of a two-slot register column, on every lane
template <typename X>
__device__ __forceinline__ X row_get(X a, X b, int i) {
  return __shfl_sync(0xffffffffu, i < 32 ? a : b, i & 31);
}
template <typename X>
__device__ __forceinline__ void row_set(X &a, X &b, int i, X v) {
  if ((int)(threadIdx.x & 31) == (i & 31)) (i < 32 ? a : b) = v;
}

// Real LU on one warp, with partial pivoting or (PIVOT false) in the given
// order; returns 0 or k + 1.
template <typename LT, bool PIVOT>
__device__ __noinline__ int team_lu_real(int N, int ld, LT *a, unsigned char *perm, LT *d1) {
  const int lane = threadIdx.x & 31;
  int src0 = lane, src1 = lane + 32;
  for (int kb = 0; kb < N; kb += TEAM_PANEL) {
    const int nb = N - kb < TEAM_PANEL ? N - kb : TEAM_PANEL;
    // the panel's columns not yet eliminated, the next one first
    LT p0[TEAM_PANEL], p1[TEAM_PANEL];
    unsigned pivs = 0;  // the four pivot rows, a byte each
#pragma unroll
    for (int c = 0; c < TEAM_PANEL; ++c) {
      p0[c] = (c < nb && lane >= kb && lane < N) ? a[lane * ld + kb + c] : LT(0);
      p1[c] = (c < nb && lane + 32 >= kb && lane + 32 < N) ? a[(lane + 32) * ld + kb + c] : LT(0);
    }
    __syncwarp();
#pragma unroll 1
    for (int c = 0; c < nb; ++c) {
      const int k = kb + c;
      int p = k;
      if constexpr (PIVOT) {
        p = arg_pivot(fabs(p0[0]), fabs(p1[0]), k, N);
        if (p < 0) return k + 1;
      } else if (!(fabs(row_get(p0[0], p1[0], k)) > LT(0))) {
        return k + 1;
      }
      pivs |= (unsigned)p << (8 * c);
      LT rp[TEAM_PANEL];
#pragma unroll
      for (int d = 0; d < TEAM_PANEL; ++d) {
        rp[d] = row_get(p0[d], p1[d], p);
        if constexpr (PIVOT) {
          const LT vk = row_get(p0[d], p1[d], k);
          row_set(p0[d], p1[d], p, vk);
          row_set(p0[d], p1[d], k, rp[d]);
        }
      }
      if constexpr (PIVOT) {
        const int sk = row_get(src0, src1, k), sp = row_get(src0, src1, p);
        row_set(src0, src1, p, sk);
        row_set(src0, src1, k, sp);
      }
      const LT inv = LT(1) / rp[0];
      if (lane == 0) d1[k] = inv;
      const bool on0 = lane > k && lane < N, on1 = lane + 32 > k && lane + 32 < N;
      if (on0) p0[0] = t_mul(p0[0], inv);
      if (on1) p1[0] = t_mul(p1[0], inv);
      if (lane < c && p != k) {  // the finished columns of the panel
        const LT x = a[k * ld + kb + lane];
        a[k * ld + kb + lane] = a[p * ld + kb + lane];
        a[p * ld + kb + lane] = x;
      }
      if (lane >= kb && lane < N) a[lane * ld + k] = p0[0];
      if (lane + 32 >= kb && lane + 32 < N) a[(lane + 32) * ld + k] = p1[0];
      __syncwarp();
#pragma unroll
      for (int d = 1; d < TEAM_PANEL; ++d) {
        if (rp[d] != LT(0)) {
          if (on0) p0[d] = t_fma(-p0[0], rp[d], p0[d]);
          if (on1) p1[d] = t_fma(-p1[0], rp[d], p1[d]);
        }
      }
#pragma unroll
      for (int d = 1; d < TEAM_PANEL; ++d) {
        p0[d - 1] = p0[d];
        p1[d - 1] = p1[d];
      }
    }
    int piv[TEAM_PANEL];
#pragma unroll
    for (int c = 0; c < TEAM_PANEL; ++c) piv[c] = c < nb ? (int)(pivs >> (8 * c)) & 255 : kb + c;
    const int jt = kb + nb;
    // row exchanges left of the panel; right of it a lane owns a column: its
    // exchanges, its four rows of U, its part of the trailing update
#pragma unroll 1
    for (int j = lane; j < kb; j += 32)
#pragma unroll
      for (int c = 0; c < TEAM_PANEL; ++c)
        if (piv[c] != kb + c) {
          const LT x = a[(kb + c) * ld + j];
          a[(kb + c) * ld + j] = a[piv[c] * ld + j];
          a[piv[c] * ld + j] = x;
        }
#pragma unroll 1
    for (int j = jt + lane; j < N; j += 32) {  // only full panels have columns to the right
      LT u[TEAM_PANEL];
#pragma unroll
      for (int c = 0; c < TEAM_PANEL; ++c) {
        const LT x = a[piv[c] * ld + j];
        if (piv[c] != kb + c) a[piv[c] * ld + j] = a[(kb + c) * ld + j];
        a[(kb + c) * ld + j] = x;
        u[c] = x;
      }
      // later exchanges never touch rows already placed, so u is final here
#pragma unroll
      for (int c = 1; c < TEAM_PANEL; ++c) {
#pragma unroll
        for (int d = 0; d < c; ++d)
          if (u[d] != LT(0)) u[c] = t_fma(-a[(kb + c) * ld + kb + d], u[d], u[c]);
        a[(kb + c) * ld + j] = u[c];
      }
#pragma unroll 2
      for (int i = jt; i < N; ++i) {
        LT v = a[i * ld + j];
        const LT *l = a + i * ld + kb;
#pragma unroll
        for (int c = 0; c < TEAM_PANEL; ++c)
          if (u[c] != LT(0)) v = t_fma(-l[c], u[c], v);
        a[i * ld + j] = v;
      }
    }
    __syncwarp();
  }
  if (lane < N) perm[lane] = (unsigned char)src0;
  if (lane + 32 < N) perm[lane + 32] = (unsigned char)src1;
  return 0;
}

// a / d.  FP32 divides.  FP64, where an IEEE division costs nine instructions
// of the bounding pipe, corrects a times the reciprocal r = 1/d once with the
// exact residual (Markstein, IBM J. Res. Dev. 34, 1990): with r correctly
// rounded, as here, the rounded quotient itself (no difference in 3 10^8 pairs
// of random mantissas and mantissas next to 1 and 2).  A quotient outside the
// normal range is left to the division.
__device__ __forceinline__ float quot(float a, float d, float) { return a / d; }
__device__ __forceinline__ double quot(double a, double d, double r) {
  const double q = a * r;
  const int e = (__double2hiint(q) >> 20) & 0x7ff, f = (__double2hiint(a) >> 20) & 0x7ff;
  if (e < 64 || e > 1980 || f < 64) return a / d;
  return t_fma(t_fma(-q, d, a), r, q);
}
__device__ __forceinline__ float recip(float) { return 0.0f; }  // unused: FP32 divides
__device__ __forceinline__ double recip(double d) { return 1.0 / d; }

// ratio and denominator of Smith's complex division by re + i im (cdiv)
template <typename LT>
__device__ __forceinline__ int smith_div(LT re, LT im, LT &r, LT &den) {
  if (fabs(re) >= fabs(im)) {
    r = im / re;
    den = t_fma(im, r, re);
    return 0;
  }
  r = re / im;
  den = t_fma(re, r, im);
  return 1;
}
template <typename LT>
__device__ __forceinline__ void smith_quot(LT a, LT b, LT r, LT den, LT iden, int mode, LT &re,
                                           LT &im) {
  re = quot(mode ? t_fma(a, r, b) : t_fma(b, r, a), den, iden);
  im = quot(mode ? t_fma(b, r, -a) : t_fma(-a, r, b), den, iden);
}

// Complex LU on warps 1 and 2 of a team: warp 1 factorises the panel, both
// update the rest, a column per lane.
template <typename LT, bool PIVOT>
__device__ __noinline__ int team_lu_cplx(int N, const TeamBuf<LT> &t, int wt) {
  const int lane = threadIdx.x & 31, ld = t.ld, col = lane + 32 * (wt - 1), bar = t.bar + TEAM_MANY;
  cplx_t<LT> *a = t.E2;
  int src0 = lane, src1 = lane + 32;
  unsigned mode0 = 0, mode1 = 0;
  for (int kb = 0; kb < N; kb += TEAM_PANEL) {
    const int nb = N - kb < TEAM_PANEL ? N - kb : TEAM_PANEL;
    if (wt == 1) {
      cplx_t<LT> p0[TEAM_PANEL], p1[TEAM_PANEL];
      const cplx_t<LT> zero = {LT(0), LT(0)};
      int sing = 0;
#pragma unroll
      for (int c = 0; c < TEAM_PANEL; ++c) {
        p0[c] = (c < nb && lane >= kb && lane < N) ? a[lane * ld + kb + c] : zero;
        p1[c] = (c < nb && lane + 32 >= kb && lane + 32 < N) ? a[(lane + 32) * ld + kb + c] : zero;
      }
      if (lane < TEAM_PANEL) t.ctl->piv[lane] = kb + lane;
      __syncwarp();
#pragma unroll 1
      for (int c = 0; c < nb; ++c) {
        const int k = kb + c;
        int p = k;
        if constexpr (PIVOT)
          p = arg_pivot(fabs(p0[0].x) + fabs(p0[0].y), fabs(p1[0].x) + fabs(p1[0].y), k, N);
        else if (!(row_get(fabs(p0[0].x) + fabs(p0[0].y), fabs(p1[0].x) + fabs(p1[0].y), k) > LT(0)))
          p = -1;
        if (p < 0) {
          sing = k + 1;
          break;
        }
        if (lane == 0) t.ctl->piv[c] = p;
        cplx_t<LT> rp[TEAM_PANEL];
#pragma unroll
        for (int d = 0; d < TEAM_PANEL; ++d) {
          rp[d].x = row_get(p0[d].x, p1[d].x, p);
          rp[d].y = row_get(p0[d].y, p1[d].y, p);
          if constexpr (PIVOT) {
            const LT xk = row_get(p0[d].x, p1[d].x, k), yk = row_get(p0[d].y, p1[d].y, k);
            row_set(p0[d].x, p1[d].x, p, xk);
            row_set(p0[d].y, p1[d].y, p, yk);
            row_set(p0[d].x, p1[d].x, k, rp[d].x);
            row_set(p0[d].y, p1[d].y, k, rp[d].y);
          }
        }
        if constexpr (PIVOT) {
          const int sk = row_get(src0, src1, k), sp = row_get(src0, src1, p);
          row_set(src0, src1, p, sk);
          row_set(src0, src1, k, sp);
        }
        LT r, den;
        const unsigned mode = smith_div(rp[0].x, rp[0].y, r, den);
        if (lane == 0) {
          t.dr[k] = r;
          t.dd[k] = den;
        }
        row_set(mode0, mode1, k, mode);
        const bool on0 = lane > k && lane < N, on1 = lane + 32 > k && lane + 32 < N;
        const LT iden = recip(den);
        if (lane == 0) t.di[k] = iden;
        if (on0) smith_quot(p0[0].x, p0[0].y, r, den, iden, (int)mode, p0[0].x, p0[0].y);
        if (on1) smith_quot(p1[0].x, p1[0].y, r, den, iden, (int)mode, p1[0].x, p1[0].y);
        if (lane < c && p != k) {  // the finished columns of the panel
          const cplx_t<LT> x = a[k * ld + kb + lane];
          a[k * ld + kb + lane] = a[p * ld + kb + lane];
          a[p * ld + kb + lane] = x;
        }
        if (lane >= kb && lane < N) a[lane * ld + k] = p0[0];
        if (lane + 32 >= kb && lane + 32 < N) a[(lane + 32) * ld + k] = p1[0];
        __syncwarp();
#pragma unroll
        for (int d = 1; d < TEAM_PANEL; ++d)
          if (rp[d].x != LT(0) || rp[d].y != LT(0)) {
            if (on0) csub(p0[d].x, p0[d].y, p0[0].x, p0[0].y, rp[d].x, rp[d].y);
            if (on1) csub(p1[d].x, p1[d].y, p1[0].x, p1[0].y, rp[d].x, rp[d].y);
          }
#pragma unroll
        for (int d = 1; d < TEAM_PANEL; ++d) {
          p0[d - 1] = p0[d];
          p1[d - 1] = p1[d];
        }
      }
      if (lane == 0) t.ctl->sing = sing;
    }
    named_sync(bar, 64);
    const int sing = t.ctl->sing;
    if (sing) return sing;  // the next command's barrier orders the next write of ctl->sing
    int piv[TEAM_PANEL];
#pragma unroll
    for (int c = 0; c < TEAM_PANEL; ++c) piv[c] = t.ctl->piv[c];
    const int jt = kb + nb;
    // more than 32 columns left: a column per lane of both warps.  Fewer: both
    // warps have the same columns and halve the rows; warp 1 exchanges and
    // forms U there while warp 2 exchanges the finished columns.
    // (FP32 keeps its columns: the second barrier cost more than the rows gave)
    constexpr int UNROLL = sizeof(LT) == 4 ? 1 : 2;
    const bool wide = sizeof(LT) == 4 || N - jt > 32;
    if (wide || wt == 2)
#pragma unroll 1
      for (int j = wide ? col : lane; j < kb; j += wide ? 64 : 32)
#pragma unroll
        for (int c = 0; c < TEAM_PANEL; ++c)
          if (piv[c] != kb + c) {
            const cplx_t<LT> x = a[(kb + c) * ld + j];
            a[(kb + c) * ld + j] = a[piv[c] * ld + j];
            a[piv[c] * ld + j] = x;
          }
    const int j = jt + (wide ? col : lane);
    cplx_t<LT> u[TEAM_PANEL];
    bool nz[TEAM_PANEL];
    if (j < N && (wide || wt == 1)) {  // only full panels have columns to the right
#pragma unroll
      for (int c = 0; c < TEAM_PANEL; ++c) {
        const cplx_t<LT> x = a[piv[c] * ld + j];
        if (piv[c] != kb + c) a[piv[c] * ld + j] = a[(kb + c) * ld + j];
        a[(kb + c) * ld + j] = x;
        u[c] = x;
      }
#pragma unroll
      for (int c = 0; c < TEAM_PANEL; ++c) {
#pragma unroll
        for (int d = 0; d < c; ++d)
          if (nz[d]) {
            const cplx_t<LT> l = a[(kb + c) * ld + kb + d];
            csub(u[c].x, u[c].y, l.x, l.y, u[d].x, u[d].y);
          }
        nz[c] = u[c].x != LT(0) || u[c].y != LT(0);
        if (c) a[(kb + c) * ld + j] = u[c];
      }
    }
    if (!wide) {
      named_sync(bar, 64);
      if (wt == 2 && j < N)
#pragma unroll
        for (int c = 0; c < TEAM_PANEL; ++c) {
          u[c] = a[(kb + c) * ld + j];
          nz[c] = u[c].x != LT(0) || u[c].y != LT(0);
        }
    }
    if (j < N) {
#pragma unroll UNROLL
      for (int i = wide ? jt : jt + wt - 1; i < N; i += wide ? 1 : 2) {
        cplx_t<LT> v = a[i * ld + j];
        const cplx_t<LT> *l = a + i * ld + kb;
#pragma unroll
        for (int c = 0; c < TEAM_PANEL; ++c)
          if (nz[c]) csub(v.x, v.y, l[c].x, l[c].y, u[c].x, u[c].y);
        a[i * ld + j] = v;
      }
    }
    named_sync(bar, 64);
  }
  if (wt == 1) {
    if (lane < N) t.p2[lane] = (unsigned char)(src0 | mode0 << 7);
    if (lane + 32 < N) t.p2[lane + 32] = (unsigned char)(src1 | mode1 << 7);
  }
  return 0;
}

// ---------------------------------------------------------------------------
// Substitutions on one warp, the vector in registers (rows lane, lane + 32)
// ---------------------------------------------------------------------------
template <typename LT>
__device__ __noinline__ void team_solve_real(int N, int ld, const LT *lu, const unsigned char *perm,
                                             const LT *d1, WVecT<2> &x) {
  const int lane = threadIdx.x & 31, i1 = lane + 32;
  const unsigned FULL = 0xffffffffu;
  const int q0 = lane < N ? perm[lane] : 0, q1 = i1 < N ? perm[i1] : 0;
  const LT x0 = LT(x.v[0]), x1 = LT(x.v[1]);
  const LT a0 = __shfl_sync(FULL, x0, q0 & 31), b0 = __shfl_sync(FULL, x1, q0 & 31);
  const LT a1 = __shfl_sync(FULL, x0, q1 & 31), b1 = __shfl_sync(FULL, x1, q1 & 31);
  LT v0 = q0 < 32 ? a0 : b0, v1 = q1 < 32 ? a1 : b1;
  const LT *r0 = lu + lane * ld, *r1 = lu + i1 * ld;
  const int n0 = N < 32 ? N : 32;
#pragma unroll 2
  for (int j = 0; j < n0; ++j) {  // forward, unit lower triangle
    const LT xj = __shfl_sync(FULL, v0, j);
    if (lane > j && lane < N) v0 = t_fma(-r0[j], xj, v0);
    if (i1 < N) v1 = t_fma(-r1[j], xj, v1);
  }
#pragma unroll 2
  for (int j = 32; j < N; ++j) {
    const LT xj = __shfl_sync(FULL, v1, j - 32);
    if (i1 > j && i1 < N) v1 = t_fma(-r1[j], xj, v1);
  }
#pragma unroll 1
  for (int i = N - 1; i >= 32; --i) {  // backward
    const LT xi = quot(__shfl_sync(FULL, v1, i - 32), lu[i * ld + i], d1[i]);
    if (i1 == i) v1 = xi;
    if (i1 < i) v1 = t_fma(-r1[i], xi, v1);
    v0 = t_fma(-r0[i], xi, v0);
  }
#pragma unroll 1
  for (int i = n0 - 1; i >= 0; --i) {
    const LT xi = quot(__shfl_sync(FULL, v0, i), lu[i * ld + i], d1[i]);
    if (lane == i) v0 = xi;
    if (lane < i) v0 = t_fma(-r0[i], xi, v0);
  }
  x.v[0] = lane < N ? double(v0) : 0.0;
  x.v[1] = i1 < N ? double(v1) : 0.0;
}

template <typename LT>
__device__ __noinline__ void team_solve_cplx(int N, const TeamBuf<LT> &t, WVecT<2> &xr,
                                             WVecT<2> &xi) {
  const int lane = threadIdx.x & 31, i1 = lane + 32, ld = t.ld;
  const unsigned FULL = 0xffffffffu;
  const cplx_t<LT> *lu = t.E2;
  const int q0 = lane < N ? t.p2[lane] & 127 : 0, q1 = i1 < N ? t.p2[i1] & 127 : 0;
  LT r0 = LT(xr.v[0]), r1 = LT(xr.v[1]), m0 = LT(xi.v[0]), m1 = LT(xi.v[1]);
  {
    const LT a0 = __shfl_sync(FULL, r0, q0 & 31), b0 = __shfl_sync(FULL, r1, q0 & 31);
    const LT a1 = __shfl_sync(FULL, r0, q1 & 31), b1 = __shfl_sync(FULL, r1, q1 & 31);
    const LT c0 = __shfl_sync(FULL, m0, q0 & 31), d0 = __shfl_sync(FULL, m1, q0 & 31);
    const LT c1 = __shfl_sync(FULL, m0, q1 & 31), d1 = __shfl_sync(FULL, m1, q1 & 31);
    r0 = q0 < 32 ? a0 : b0;
    r1 = q1 < 32 ? a1 : b1;
    m0 = q0 < 32 ? c0 : d0;
    m1 = q1 < 32 ? c1 : d1;
  }
  const cplx_t<LT> *l0 = lu + lane * ld, *l1 = lu + i1 * ld;
  const int n0 = N < 32 ? N : 32;
#pragma unroll 1
  for (int j = 0; j < n0; ++j) {
    const LT a = __shfl_sync(FULL, r0, j), b = __shfl_sync(FULL, m0, j);
    if (lane > j && lane < N) {
      const cplx_t<LT> l = l0[j];
      csub(r0, m0, l.x, l.y, a, b);
    }
    if (i1 < N) {
      const cplx_t<LT> l = l1[j];
      csub(r1, m1, l.x, l.y, a, b);
    }
  }
#pragma unroll 1
  for (int j = 32; j < N; ++j) {
    const LT a = __shfl_sync(FULL, r1, j - 32), b = __shfl_sync(FULL, m1, j - 32);
    if (i1 > j && i1 < N) {
      const cplx_t<LT> l = l1[j];
      csub(r1, m1, l.x, l.y, a, b);
    }
  }
#pragma unroll 1
  for (int i = N - 1; i >= 0; --i) {
    const LT a = i >= 32 ? __shfl_sync(FULL, r1, i - 32) : __shfl_sync(FULL, r0, i);
    const LT b = i >= 32 ? __shfl_sync(FULL, m1, i - 32) : __shfl_sync(FULL, m0, i);
    LT qr, qi;
    smith_quot(a, b, t.dr[i], t.dd[i], t.di[i], t.p2[i] >> 7, qr, qi);
    if (lane == i) {
      r0 = qr;
      m0 = qi;
    }
    if (i1 == i) {
      r1 = qr;
      m1 = qi;
    }
    if (lane < i && lane < N) {
      const cplx_t<LT> l = l0[i];
      csub(r0, m0, l.x, l.y, qr, qi);
    }
    if (i1 < i) {
      const cplx_t<LT> l = l1[i];
      csub(r1, m1, l.x, l.y, qr, qi);
    }
  }
  xr.v[0] = lane < N ? double(r0) : 0.0;
  xr.v[1] = i1 < N ? double(r1) : 0.0;
  xi.v[0] = lane < N ? double(m0) : 0.0;
  xi.v[1] = i1 < N ? double(m1) : 0.0;
}

// ---------------------------------------------------------------------------
// Commands
// ---------------------------------------------------------------------------
enum { TEAM_QUIT = 0, TEAM_CHEM3, TEAM_JAC, TEAM_FACTOR, TEAM_SOLVE };

__device__ __forceinline__ void vec_store(int N, double *p, const WVecT<2> &x) {
  const int lane = threadIdx.x & 31;
  if (lane < N) p[lane] = x.v[0];
  if (lane + 32 < N) p[lane + 32] = x.v[1];
}
__device__ __forceinline__ void vec_load(int N, const double *p, WVecT<2> &x) {
  const int lane = threadIdx.x & 31;
  x.v[0] = lane < N ? p[lane] : 0.0;
  x.v[1] = lane + 32 < N ? p[lane + 32] : 0.0;
}

// The mass-fraction reactor on a team.
template <typename LT>
struct TeamMassFrac {
  static constexpr bool PIVOT = true;
  const MechView &m;
  const HotTables &h;
  const TeamBuf<LT> &t;

  __device__ __forceinline__ int n() const { return m.ns; }
  // factor on atol of element g's error weight
  __device__ __forceinline__ double atol_w(int) const { return 1.0; }

  // warp wt's stage: y from its g buffer, f into its C buffer
  __device__ __forceinline__ void chem_stage(int wt) const {
    WVecT<2> y, f;
    f.v[0] = f.v[1] = 0.0;
    vec_load(n(), t.g(wt), y);
    __syncwarp();
    const int rc = team_rhs<>(m, h, t.C(wt), t.g(wt), t.q(wt), t.ctl->P, y, f);
    __syncwarp();
    vec_store(n(), t.C(wt), f);
    if ((threadIdx.x & 31) == 0) t.ctl->ret[wt] = rc;
  }

  // Leader, before the JAC command: the state's thermodynamics into warp 0's
  // buffers and the scratch, its scalars into ctl.
  __device__ void jac_prepare(const WVecT<2> &y) const {
    using G = Grp<32>;
    const int lane = G::lane(), ns = m.ns, in = ns - 1, N = ns, nv = t.nv;
    double *rW = t.js + 3 * nv, *hs = t.js + 4 * nv, *cpk = t.js + 5 * nv;
    const double T = G::bcast(y.v[0], 0);
    double sY = 0.0, sS = 0.0;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int e = lane + 32 * r;
      if (e >= 1 && e < N) {
        sY += y.v[r];
        sS += y.v[r] * m.invW[e - 1];
      }
    }
    sY = G::sum(sY);
    sS = G::sum(sS);
    const double Yin = 1.0 - sY;
    const double S = sS + Yin * m.invW[in];
    const double rho = t.ctl->P / (RU * T * S);
    const double logT = log(T), invT = 1.0 / T;
    double cpl = 0.0, dcpl = 0.0;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int e = lane + 32 * r, k = e - 1;
      if (e >= 1 && e <= ns) {
        const double Yk = (e < N) ? y.v[r] : Yin;
        const int rg = range_of(m, k, T);
        const double *cc = m.cp + (2 * k + rg) * NCP;
        const double cp = poly_cp(cc, T);
        t.C(0)[k] = rho * Yk * m.invW[k];
        t.g(0)[k] = poly_g(m.gb + (2 * k + rg) * NG, T, logT, invT);
        hs[k] = poly_h(m.h + (2 * k + rg) * NH, T, invT);
        cpk[k] = cp;
        rW[k] = rho * m.invW[k];
        cpl = t_fma(t_mul(Yk, cp), m.invW[k], cpl);
        dcpl = t_fma(t_mul(Yk, poly_dcp(cc, T)), m.invW[k], dcpl);
      }
    }
    const double cpm = G::sum(cpl), dcpm = G::sum(dcpl);
    if (lane == 0) {
      TeamCtl &c = *t.ctl;
      c.T = T;
      c.logT = logT;
      c.invT = invT;
      c.rho = rho;
      c.S = S;
      c.cpm = cpm;
      c.dcpm = dcpm;
      c.ret[0] = c.ret[1] = c.ret[2] = 0;
    }
  }

  // The right-hand side (into warp 0's g buffer) and the Jacobian (into J).
  __device__ __noinline__ void jac(int wt) const {
    LT *J = t.J;
    const int ld = t.ld;
    jac_out<TEAM_WARPS>(wt, [J, ld](int i, int c, double v) { J[(size_t)c * ld + i] = LT(v); });
  }

  // the same on TW warps (one: all phases on one warp, no team barrier), with
  // the Jacobian's entries given to put(i, j, value)
  template <int TW, class Put>
  __device__ __forceinline__ void jac_out(int wt, Put put) const {
    constexpr int NT = 32 * TW;
    using G = Grp<32>;
    const int lane = G::lane(), ns = m.ns, in = ns - 1, N = ns, nv = t.nv, nr = m.nr, ld = t.ld;
    TeamCtl &ct = *t.ctl;
    double *A = t.js, *B = A + nv, *Tc = A + 2 * nv, *rW = A + 3 * nv, *hs = A + 4 * nv,
           *cpk = A + 5 * nv, *wd = A + 6 * nv, *bS = A + 7 * nv;
    double *sig = A + 8 * nv, *dq = sig + nr, *D = dq + nr;
    const int nslots = h.off[nr - 1] + rec_nre(h.rec[nr - 1]) + rec_npr(h.rec[nr - 1]);
    const double T = ct.T, logT = ct.logT, invT = ct.invT, rho = ct.rho, S = ct.S;
    const double Ctot = rho * S, *C = t.C(0), *g = t.g(0);
    double *q = t.q(0);
    for (int e = lane + 32 * wt; e < N * ld; e += NT) t.Jd[e] = 0.0;
    // reactions in rounds of 32, dealt over the warps (the Troe rounds first)
#pragma unroll 1
    for (int i = lane + 32 * wt; i < nr; i += NT) {
      const ReactionJac r = reaction_jac(m, h, C, g, hs, i, T, logT, invT, Ctot);
      q[i] = r.q;
      sig[i] = r.sig;
      dq[i] = r.dqdT;
      // derivatives by the species in each slot: rW times the mass-action product
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
        D[h.off[i] + s] = t_mul(rW[(sl >> (8 * mine)) & 255], p);
      }
      if (i < m.nfall) {
        const int e0 = m.eff0[i], ne = meta_neff(m.meta[i]);
#pragma unroll 1
        for (int e = e0; e < e0 + ne; ++e) {
          const int col = m.effsp[e];
          const double p = t_mul(r.u, m.eff[e]);
          D[nslots + e] = col != in ? t_mul(rW[col], p) : p;
        }
      }
    }
    jac_sync<TW>();
    if (wt == 0) {
      // production rates and f
      WVecT<2> f;
      double hw = 0.0, cpw = 0.0;
      bool ok = true;
      const double irho = 1.0 / rho;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int e = lane + 32 * r, k = e - 1;
        f.v[r] = 0.0;
        if (e >= 1 && e < N) {
          const double w = net_rate(h, q, k);
          wd[k] = w;
          f.v[r] = m.W[k] * w * irho;
          ok &= isfinite(f.v[r]);
          hw += hs[k] * w;
          cpw += cpk[k] * w;
        }
      }
      hw = G::sum(hw);
      cpw = G::sum(cpw);
      const double fT = -(hw * T) / (rho * ct.cpm);
      if (lane == 0) f.v[0] = fT;
      ok &= isfinite(fT);
      ok = G::all(ok);
      __syncwarp();
      vec_store(N, t.g(0), f);
      if (lane == 0) {
        ct.Hw = hw;
        ct.CPw = cpw;
        if (!ok) ct.ret[0] = 4;
      }
    }
    if (TW == 1 || wt != 0) {
      // sparse rows of dwdot/dY, the longest lists on warp 1
      for (int e = lane + (TW == 1 ? 0 : 32 * (wt - 1)); e < in; e += TW == 1 ? 32 : 64) {
        const int k = h.rank[e];
        double *Jr = t.Jd + (1 + k) * ld;
        double a = 0.0, b = 0.0, tc = 0.0;
        row_sums(h, sig, dq, k, b, tc);
        row_terms(h, D, k, in, Jr + 1, a);
        A[k] = a;
        B[k] = b;
        Tc[k] = tc;
      }
    }
    jac_sync<TW>();
    // row coefficients of the dense part, then one pass per column
    const double irho = 1.0 / rho, iS = 1.0 / S, cpm = ct.cpm;
    for (int k = lane + 32 * wt; k < in; k += NT) {
      A[k] *= rW[in];
      B[k] *= iS;
      wd[k] = m.W[k] * wd[k] * irho * irho;
      bS[k] = wd[k] * (rho / S);
    }
    jac_sync<TW>();
    const double HwJ = ct.Hw * RU * T, CPwJ = ct.CPw * RU, rcp = rho * cpm * RU;
    const double hfac = RU * T / rcp, g2 = HwJ / (rcp * rcp);
    bool ok = true;
    for (int c = lane + 32 * wt; c < N; c += NT) {
      double dh = 0.0, drcp, extra = 0.0;
      if (c == 0) {
        const double x = rho * invT;
#pragma unroll 1
        for (int k = 0; k < in; ++k) {
          const double v = Tc[k];
          dh = t_fma(hs[k], v, dh);
          const double w = t_fma(t_mul(m.W[k], irho), v, t_mul(wd[k], x));
          ok &= isfinite(w);
          put(1 + k, c, w);
        }
        drcp = cpm * RU * (-rho * invT) + rho * ct.dcpm * RU;
        extra = -CPwJ / rcp;
      } else {
        const double mj = m.invW[c - 1] - m.invW[in];
        const double *col = t.Jd + ld + c;
#pragma unroll 1
        for (int k = 0; k < in; ++k) {
          const double v = col[(size_t)k * ld] - t_fma(mj, B[k], A[k]);
          dh = t_fma(hs[k], v, dh);
          const double w = t_fma(t_mul(m.W[k], irho), v, t_mul(bS[k], mj));
          ok &= isfinite(w);
          put(1 + k, c, w);
        }
        const double cpin = t_mul(cpk[in], m.invW[in]);
        drcp = t_fma(t_mul(cpm, RU), -rho * mj / S,
                     t_mul(t_mul(rho, t_fma(cpk[c - 1], m.invW[c - 1], -cpin)), RU));
      }
      const double w = t_fma(g2, drcp, t_fma(-hfac, dh, extra));
      ok &= isfinite(w);
      put(0, c, w);
    }
    if (!G::all(ok) && lane == 0) ct.ret[wt] = 4;
  }

  template <int TW>
  __device__ __forceinline__ void jac_sync() const {
    if constexpr (TW == 1)
      __syncwarp();
    else
      named_sync(t.bar, 32 * TW);
  }
};

// E1 = gamma/h - J and E2 = (alpha + i beta)/h - J from J's columns, then the
// factorisations; the results in ctl->ret
template <typename LT, bool PIVOT>
__device__ void team_factor(int N, const TeamBuf<LT> &t, int wt) {
  const int lane = threadIdx.x & 31, ld = t.ld;
  const double h = t.ctl->h;
  const LT fac1 = LT(RC.gam / h), alphn = LT(RC.alp / h), betan = LT(RC.bet / h);
  // six columns' loads in flight per thread (the stores could alias them)
#pragma unroll 1
  for (int j0 = wt; j0 < N; j0 += 6 * TEAM_WARPS) {
    LT v[12];
#pragma unroll
    for (int x = 0; x < 6; ++x) {
      const int j = j0 + TEAM_WARPS * x;
      v[2 * x] = j < N && lane < N ? t.J[(size_t)j * ld + lane] : LT(0);
      v[2 * x + 1] = j < N && lane + 32 < N ? t.J[(size_t)j * ld + lane + 32] : LT(0);
    }
#pragma unroll
    for (int x = 0; x < 12; ++x) {
      const int j = j0 + TEAM_WARPS * (x >> 1), i = lane + 32 * (x & 1);
      if (j >= N || i >= N) continue;
      cplx_t<LT> e;
      e.x = (i == j) ? alphn - v[x] : -v[x];
      e.y = (i == j) ? betan : LT(0);
      t.E1[i * ld + j] = (i == j) ? fac1 - v[x] : -v[x];
      t.E2[i * ld + j] = e;
    }
  }
  named_sync(t.bar, TEAM_NT);
  const int r = wt == 0 ? team_lu_real<LT, PIVOT>(N, ld, t.E1, t.p1, t.d1)
                        : team_lu_cplx<LT, PIVOT>(N, t, wt);
  if (lane == 0) t.ctl->ret[wt] = r;
}

// warp wt's part of a command
template <typename LT, class Form>
__device__ __forceinline__ void team_exec(int cmd, int wt, const Form &f) {
  const TeamBuf<LT> &t = f.t;
  if (cmd == TEAM_CHEM3) {
    f.chem_stage(wt);
  } else if (cmd == TEAM_JAC) {
    f.jac(wt);
  } else if (cmd == TEAM_FACTOR) {
    team_factor<LT, Form::PIVOT>(f.n(), t, wt);
  } else if (cmd == TEAM_SOLVE && wt == 1) {
    WVecT<2> xr, xi;
    vec_load(f.n(), t.C(1), xr);
    vec_load(f.n(), t.g(1), xi);
    __syncwarp();
    team_solve_cplx<LT>(f.n(), t, xr, xi);
    vec_store(f.n(), t.C(1), xr);
    vec_store(f.n(), t.g(1), xi);
  }
}

// The system a team integrates, for the step drivers of kin_warp.cuh (the
// drivers' buffer argument stays unused: the matrices are the team's).
template <typename LT, class Form>
struct TeamSys {
  static constexpr int POINTS = TEAM_WARPS;
  using WV = WVecT<2>;
  const Form &f;
  __device__ __forceinline__ int n() const { return f.n(); }
  __device__ __forceinline__ double atol_w(int g) const { return f.atol_w(g); }
  __device__ __forceinline__ int jat(const WarpBuf<LT> &, int i, int j) const {
    return j * f.t.ld + i;
  }
  // J x: eight columns' loads in flight, widened on the integer pipe
  __device__ __noinline__ void jac_times(const WarpBuf<LT> &, const WV &x, WV &out) const {
    const int lane = threadIdx.x & 31, N = n(), ld = f.t.ld;
    const LT *J = f.t.J;
    double o0 = 0.0, o1 = 0.0;
#pragma unroll 1
    for (int j0 = 0; j0 < N; j0 += 8) {
      LT a[8], b[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int j = j0 + q;
        a[q] = j < N && lane < N ? J[(size_t)j * ld + lane] : LT(0);
        b[q] = j < N && lane + 32 < N ? J[(size_t)j * ld + lane + 32] : LT(0);
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int j = j0 + q;  // eight columns never straddle the two slots
        const double xj = __shfl_sync(0xffffffffu, j0 < 32 ? x.v[0] : x.v[1], j & 31);
        if (j >= N) break;
        o0 = fma(widen(a[q]), xj, o0);
        o1 = fma(widen(b[q]), xj, o1);
      }
    }
    out.v[0] = o0;
    out.v[1] = o1;
  }
  __device__ __forceinline__ static double widen(double v) { return v; }
  // exact: exponent rebiased, mantissa shifted; zeros, subnormals and
  // non-finite values through the conversion unit when there are any
  __device__ __forceinline__ static double widen(float v) {
    const unsigned u = __float_as_uint(v), e = u & 0x7f800000u;
    if (e == 0x7f800000u || (e == 0 && (u << 1) != 0)) return (double)v;
    const unsigned hi = (u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (e ? 0x38000000u : 0u));
    return __hiloint2double((int)hi, (int)(u << 29));
  }
  __device__ __forceinline__ void post(int cmd) const {
    if ((threadIdx.x & 31) == 0) f.t.ctl->cmd = cmd;
    named_sync(f.t.bar, TEAM_NT);
  }
  __device__ __forceinline__ void done() const { named_sync(f.t.bar, TEAM_NT); }
  __device__ __noinline__ int chem(const WarpBuf<LT> &, double, const WV &y, WV &out,
                                   bool wantJ) const {
    const TeamBuf<LT> &t = f.t;
    if (!wantJ) {  // one point: the leader alone
      __syncwarp();
      vec_store(n(), t.g(0), y);
      __syncwarp();
      f.chem_stage(0);
      __syncwarp();
      vec_load(n(), t.C(0), out);
      const int rc = t.ctl->ret[0];
      __syncwarp();
      return rc;
    }
    f.jac_prepare(y);
    post(TEAM_JAC);
    f.jac(0);
    done();
    vec_load(n(), t.g(0), out);
    const int rc = t.ctl->ret[0] | t.ctl->ret[1] | t.ctl->ret[2];
    __syncwarp();
    return rc;
  }
  __device__ __noinline__ int chem3(const WarpBuf<LT> &, double, const WV &y1, const WV &y2,
                                    const WV &y3, WV &f1, WV &f2, WV &f3) const {
    const TeamBuf<LT> &t = f.t;
    vec_store(n(), t.g(0), y1);
    vec_store(n(), t.g(1), y2);
    vec_store(n(), t.g(2), y3);
    post(TEAM_CHEM3);
    f.chem_stage(0);
    done();
    vec_load(n(), t.C(0), f1);
    vec_load(n(), t.C(1), f2);
    vec_load(n(), t.C(2), f3);
    const int rc = t.ctl->ret[0] | t.ctl->ret[1] | t.ctl->ret[2];
    __syncwarp();
    return rc;
  }
  __device__ __forceinline__ int factor(const WarpBuf<LT> &, double h) const {
    const TeamBuf<LT> &t = f.t;
    if ((threadIdx.x & 31) == 0) t.ctl->h = h;
    post(TEAM_FACTOR);
    team_factor<LT, Form::PIVOT>(n(), t, 0);
    done();
    const int rc = t.ctl->ret[0] ? t.ctl->ret[0] : t.ctl->ret[1];
    __syncwarp();
    return rc;
  }
  __device__ __forceinline__ void solve_real(const WarpBuf<LT> &, WV &x) const {
    team_solve_real<LT>(n(), f.t.ld, f.t.E1, f.t.p1, f.t.d1, x);
  }
  __device__ __forceinline__ void solve_both(const WarpBuf<LT> &, WV &x, WV &xr, WV &xi) const {
    const TeamBuf<LT> &t = f.t;
    vec_store(n(), t.C(1), xr);
    vec_store(n(), t.g(1), xi);
    post(TEAM_SOLVE);
    team_solve_real<LT>(n(), t.ld, t.E1, t.p1, t.d1, x);
    done();
    vec_load(n(), t.C(1), xr);
    vec_load(n(), t.g(1), xi);
    __syncwarp();
  }
};

}  // namespace kin
