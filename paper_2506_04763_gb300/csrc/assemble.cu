// assemble.cu — grid set-up (K0) and vertex-centred finite-volume assembly
// (K1: F, exact Jacobian J = F_u and lumped M; K1r: F only).
//
// Compiled with -fmad=false: every product and sum is rounded separately, in
// the order written.  The quantities on which a discrete decision rests — S_e
// (k_r clamps), p_c and p_n = p_w + p_c, the face gradients G, T_w and T_n
// (upwind directions), S_e at x_M and the S hat cap test — are in addition
// written with explicit round-to-nearest intrinsics (__dadd_rn, __dmul_rn, ...),
// so the decisions are taken on exactly the values that order defines.  The
// derivatives stay unfused too: several Jacobian entries are sums of nearly
// cancelling terms (e.g. the NAPL rows where k_rn ~ 0), whose rounding a fused
// multiply-add would change by far more than 1e-12 of the row.
//
// Method (arXiv 2506.04763):
//   Sec. 3.1, Eqs. (dsW),(dpN): dual-mesh control volumes b_i; storage lumped
//     at the vertex; one sub-control-volume face (SCVF) per element edge,
//     flux evaluated at the face midpoint x_M with face size A_f.
//   Sec. 3.2, Eqs. (up_krw),(up_krn): k_r taken from the upstream vertex by
//     the sign of v_alpha . n (v_alpha excludes the capillary-diffusion
//     part); T >= 0 picks the edge's lower vertex a.
//   Sec. 3.3, Eqs. (pdmin),(hSw),(krn_ip),(krw_ip): p_dmin per vertex and the
//     per-sub-control-volume saturation S hat, used in k_rn only.
//   Sec. 2, Eqs. (sW),(pN),(vW),(vN): the water flux splits into k_rw v_w and
//     the capillary-diffusion term, which is not upwinded.
// With p_w as primary pressure, p_n = p_w + p_c at vertices (p_c,i =
// p_dmin,i J(S_e,i)); per face of element e along axis k (edge a->b):
//   T_w = -K_e A_f (G(p_n) - rho_w g_k), T_n = -K_e A_f (G(p_n) - rho_n g_k),
//   T_c = -K_e A_f G(p_c),  G = d/dx_k of the element's Q1 interpolant at x_M,
//   F_w = rho_w (lam_w(S_up) T_w - lam_w(S(x_M)) T_c),
//   F_n = rho_n lam_n(S hat_up) T_n.
//
// K1 runs in two passes, k_asm_faces and k_asm_rows (below).  The first form,
// k_assemble (RF_ASM_VERTEX=1, for comparison), runs one thread per vertex: it
// visits the 2^d elements around its vertex and, in each, the d faces that
// touch it, and accumulates its own block row (27 or 9 2x2 blocks) in shared
// memory.
#include <cstdlib>

#include "rf_common.cuh"
#include "rf_kernels.h"

namespace rf {

struct Phys {
  double rho_w, rho_n, mu_w, mu_n, S_wr, S_nr, lam, den;
  double h[3], g[3];
  double rh[3], rmu_w, rmu_n, rden, nid;   // recip of h, mu_w, mu_n, den; -1 / den
  double Af[3], gw[3], gn[3]; // SCV face sizes, rho_w g, rho_n g per axis
  double gt[3][3];            // w / h by axis and number of 1/4 factors in w
  int scheme;   // SCHEME_* bits (0: the discretisation of Sec. 3)
};

// ---- constitutive laws (Brooks-Corey; J continued linearly outside [0.01, 1])
__device__ __forceinline__ void leverett_pow(double lam, double S, double& J, double& dJ) {
  if (lam == 2.0) {
    double r = __dsqrt_rn(S);
    J = __ddiv_rn(1.0, r);
    dJ = __ddiv_rn(-0.5, __dmul_rn(S, r));
  } else {
    J = pow(S, -1.0 / lam);
    dJ = (-1.0 / lam) * pow(S, -1.0 / lam - 1.0);
  }
}

// J(S_e) (decides nothing by itself but feeds p_c, p_n and T: exact rounding)
__device__ __forceinline__ void leverett(double lam, double Se, double& J, double& dJ) {
  if (Se < 0.01) {
    double j0, d0;
    leverett_pow(lam, 0.01, j0, d0);
    J = __dadd_rn(j0, __dmul_rn(d0, __dsub_rn(Se, 0.01)));
    dJ = d0;
  } else if (Se > 1.0) {
    const double sl = __ddiv_rn(-1.0, lam);
    J = __dadd_rn(1.0, __dmul_rn(sl, __dsub_rn(Se, 1.0)));
    dJ = sl;
  } else {
    leverett_pow(lam, Se, J, dJ);
  }
}

// k_rw, dk_rw/dS_e (k_r use S_e clamped to [0,1], derivative 0 outside)
__device__ __forceinline__ void krw_of(double lam, double Se, double& k, double& dk) {
  double Sc = fmin(fmax(Se, 0.0), 1.0);
  bool inside = Se > 0.0 && Se < 1.0;
  if (lam == 2.0) {
    double s2 = Sc * Sc;
    k = s2 * s2;
    dk = inside ? 4.0 * s2 * Sc : 0.0;
  } else {
    double ew = (2.0 + 3.0 * lam) / lam;
    k = pow(Sc, ew);
    dk = inside ? ew * pow(Sc, ew - 1.0) : 0.0;
  }
}

__device__ __forceinline__ void krn_of(double lam, double Se, double& k, double& dk) {
  double Sc = fmin(fmax(Se, 0.0), 1.0);
  bool inside = Se > 0.0 && Se < 1.0;
  double om = 1.0 - Sc;
  if (lam == 2.0) {
    double s2 = Sc * Sc;
    k = om * om * (1.0 - s2);
    dk = inside ? (-2.0 * om * (1.0 - s2) - 2.0 * Sc * om * om) : 0.0;
  } else {
    double en = (2.0 + lam) / lam, sa = pow(Sc, en);
    k = om * om * (1.0 - sa);
    dk = inside ? (-2.0 * om * (1.0 - sa) - en * om * om * pow(Sc, en - 1.0)) : 0.0;
  }
}

// Per-medium relative permeabilities (Sec. 6, Case 2: each medium has its own
// polynomial k_rw, k_rn).  law < 0 or a row of kind 0: the Brooks-Corey laws
// above.  Kind 1, row {1, a_w, n_w, a_n, b_n, c_n}: k_rw = a_w S^n_w, k_rn =
// a_n (1 - b_n S)^2 (1 - c_n S^2) while both factors are positive and 0 from
// the first of their roots on, S = S_e clamped to [0, 1], derivatives 0
// outside (0, 1).
__device__ __forceinline__ const double* law_row(const double* tab, int law) {
  return (law < 0 || tab[6 * law] == 0.0) ? nullptr : tab + 6 * law;
}

__device__ __forceinline__ void krw_law(double lam, const double* L, double Se, double& k, double& dk) {
  if (!L) { krw_of(lam, Se, k, dk); return; }
  const double aw = L[1];
  const int nw = (int)L[2];
  const double S = fmin(fmax(Se, 0.0), 1.0);
  double p = 1.0;                     // S^(n_w - 1)
  for (int t = 1; t < nw; ++t) p = p * S;
  k = aw * (p * S);
  dk = (Se > 0.0 && Se < 1.0) ? (aw * nw) * p : 0.0;
}

__device__ __forceinline__ void krn_law(double lam, const double* L, double Se, double& k, double& dk) {
  if (!L) { krn_of(lam, Se, k, dk); return; }
  const double an = L[3], bn = L[4], cn = L[5];
  const double S = fmin(fmax(Se, 0.0), 1.0);
  const double r = 1.0 - bn * S, q = 1.0 - cn * (S * S);
  if (r > 0.0 && q > 0.0) {
    k = an * (r * r) * q;
    dk = (Se > 0.0 && Se < 1.0) ? an * (-2.0 * bn * r * q - 2.0 * cn * S * (r * r)) : 0.0;
  } else {
    k = 0.0;
    dk = 0.0;
  }
}

// Eq. (hSw): S_e hat of vertex i inside an element of entry pressure pdc.
__device__ __forceinline__ void shat_of(double lam, double Se, double pdc, double pdmin, double& s, double& ds) {
  if (pdc == pdmin) { s = Se; ds = 1.0; return; }
  double r = __ddiv_rn(pdc, pdmin);
  double rl = (lam == 2.0) ? __dmul_rn(r, r) : pow(r, lam);
  double t = __dmul_rn(rl, Se);
  if (t >= 1.0) { s = 1.0; ds = 0.0; }
  else { s = t; ds = rl; }
}

// ---------------------------------------------------------------- K0
// p_dmin (Eq. pdmin) and lumped pore volume per vertex, parity-split order.
__global__ void k_vertex_setup(Dims d, const double* __restrict__ pd, const double* __restrict__ phi,
                               double vol, double* __restrict__ pdmin, double* __restrict__ phiv) {
  int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= d.nv) return;
  int i, j, k;
  pcoords(d, p, i, j, k);
  const int cx = d.nx - 1, cy = d.ny - 1, cz = d.dim == 3 ? d.nz - 1 : 1;
  const double frac = d.dim == 3 ? 0.125 : 0.25;
  double best = INFINITY, s = 0.0;
  for (int c = 0; c < (1 << d.dim); ++c) {
    int ci = i - (c & 1), cj = j - ((c >> 1) & 1), ck = d.dim == 3 ? k - ((c >> 2) & 1) : 0;
    if (ci < 0 || ci >= cx || cj < 0 || cj >= cy || ck < 0 || ck >= cz) continue;
    int64_t cell = ci + (int64_t)cx * (cj + (int64_t)cy * ck);
    best = fmin(best, pd[cell]);
    s += phi[cell] * vol * frac;
  }
  pdmin[p] = best;
  phiv[p] = s;
}

// natural <-> parity-split permutation of interleaved pairs / bytes
__global__ void k_perm_to_p(Dims d, const double2* __restrict__ nat, double2* __restrict__ out) {
  int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (v >= d.nv) return;
  const uint32_t line = (uint32_t)v / (uint32_t)d.nx;   // nv < 2^31
  const int i = (int)((uint32_t)v - line * (uint32_t)d.nx);
  out[line * d.nx + ((i & 1) ? d.E + (i >> 1) : (i >> 1))] = nat[v];
}

__global__ void k_perm_from_p(Dims d, const double2* __restrict__ pl, double2* __restrict__ nat) {
  int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (v >= d.nv) return;
  const uint32_t line = (uint32_t)v / (uint32_t)d.nx;   // nv < 2^31
  const int i = (int)((uint32_t)v - line * (uint32_t)d.nx);
  nat[v] = pl[line * d.nx + ((i & 1) ? d.E + (i >> 1) : (i >> 1))];
}

__global__ void k_perm_bytes_to_p(Dims d, const uint8_t* __restrict__ nat, uint8_t* __restrict__ out) {
  int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (v >= d.nv) return;
  const uint32_t line = (uint32_t)v / (uint32_t)d.nx;   // nv < 2^31
  const int i = (int)((uint32_t)v - line * (uint32_t)d.nx);
  out[line * d.nx + ((i & 1) ? d.E + (i >> 1) : (i >> 1))] = nat ? nat[v] : 0;
}

__global__ void k_perm_scalar_to_p(Dims d, const double* __restrict__ nat, double* __restrict__ out) {
  int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (v >= d.nv) return;
  const uint32_t line = (uint32_t)v / (uint32_t)d.nx;   // nv < 2^31
  const int i = (int)((uint32_t)v - line * (uint32_t)d.nx);
  out[line * d.nx + ((i & 1) ? d.E + (i >> 1) : (i >> 1))] = nat ? nat[v] : 0.0;
}

// ---------------------------------------------------------------- K1a
// Per-vertex quantities of the state (parity-split order): S_e, p_n = p_w +
// p_c, p_c, dp_c/dS_n, lambda_w, lambda_n and their S_n-derivatives.
__global__ void k_vertex_state(Dims d, Phys ph, const double2* __restrict__ u, const double* __restrict__ pdmin,
                               double* __restrict__ Se, double* __restrict__ pn, double* __restrict__ pc,
                               double* __restrict__ dpc, double* __restrict__ krw, double* __restrict__ dkrw,
                               double* __restrict__ krn, double* __restrict__ dkrn) {
  int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= d.nv) return;
  double2 uv = u[p];
  double se = div_by(__dsub_rn(__dsub_rn(1.0, uv.y), ph.S_wr), ph.den, ph.rden);
  double J, dJ, k, dk;
  leverett(ph.lam, se, J, dJ);
  krw_of(ph.lam, se, k, dk);
  double pdm = pdmin[p];
  double c = __dmul_rn(pdm, J);
  Se[p] = se;
  pc[p] = c;
  dpc[p] = div_by(-(pdm * dJ), ph.den, ph.rden);
  pn[p] = __dadd_rn(uv.x, c);
  // the upwinded water mobility lambda_w = k_rw / mu_w and its S_n-derivative,
  // divided here once per vertex instead of once per face visit
  krw[p] = div_by(k, ph.mu_w, ph.rmu_w);
  dkrw[p] = div_by(div_by(-dk, ph.den, ph.rden), ph.mu_w, ph.rmu_w);
  // lambda_n = k_rn / mu_n where S hat = S_e (the elements of the vertex's
  // lowest entry pressure), and its S_n-derivative
  krn_of(ph.lam, se, k, dk);
  krn[p] = div_by(k, ph.mu_n, ph.rmu_n);
  dkrn[p] = div_by(dk * ph.nid, ph.mu_n, ph.rmu_n);
}

// ---------------------------------------------------------------- K1 / K1r
struct AsmIn {
  const double2* u;
  const double *Se, *pn, *pc, *dpc, *krw, *dkrw, *krn, *dkrn, *pdmin, *phiv;
  const double *K, *pd, *phi;     // per cell (natural cell order)
  double vol;                     // cell volume
  const uint8_t* dir;             // parity-split
  const double* pw_dir;           // parity-split
  const double2* q_in;            // parity-split (may be null)
  const uint8_t* law;             // per cell k_r law (natural cell order), or null
  const double* kr_tab;           // law table, 6 doubles per law
};

template <int DIM, bool WANT_J>
__global__ void __launch_bounds__(128) k_assemble(Dims d, Phys ph, AsmIn in, double2* __restrict__ F,
                                                  double* __restrict__ J, double2* __restrict__ mdiag) {
  extern __shared__ double acc[];  // [nb*4][blockDim]
  constexpr int NC = 1 << DIM, NE = 1 << (DIM - 1), NB = DIM == 3 ? 27 : 9;
  const int tid = threadIdx.x, BS = blockDim.x;
  int64_t p = blockIdx.x * (int64_t)BS + tid;
  const bool live = p < d.nv;
  if (WANT_J) {
#pragma unroll 4
    for (int t = 0; t < NB * 4; ++t) acc[t * BS + tid] = 0.0;
  }
  if (!live) return;
  int i, j, k;
  pcoords(d, p, i, j, k);
  const int cx = d.nx - 1, cy = d.ny - 1, cz = DIM == 3 ? d.nz - 1 : 1;
  double F0 = 0.0, F1 = 0.0;
  if (in.q_in) { double2 q = in.q_in[p]; F0 = q.x; F1 = q.y; }
  const double neg_inv_den = -1.0 / ph.den;
  const bool darcy = (ph.scheme & SCHEME_DARCY_UPWIND) != 0;
  // d G / d q_q = +-w / h_k takes one of DIM magnitudes per axis (w is a
  // product of DIM-1 factors 3/4 or 1/4): divide once per thread.  gtab[k][m]
  // = w / h_k with m = the number of 1/4 factors; IEEE division is correctly
  // rounded and sign-symmetric, so +-gtab equals the per-corner (+-w) / h_k.
  double gtab[DIM][DIM];
#pragma unroll
  for (int kk = 0; kk < DIM; ++kk)
#pragma unroll
    for (int m = 0; m < DIM; ++m) {
      double w = 1.0;
#pragma unroll
      for (int t = 0; t < DIM - 1; ++t) w = w * (t < m ? 0.25 : 0.75);
      gtab[kk][m] = w / ph.h[kk];
    }

#pragma unroll
  for (int c = 0; c < NC; ++c) {
    // element whose corner c (bits: x,y,z offsets) is this vertex
    const int ci = i - (c & 1), cj = j - ((c >> 1) & 1), ck = DIM == 3 ? k - ((c >> 2) & 1) : 0;
    if (ci < 0 || ci >= cx || cj < 0 || cj >= cy || ck < 0 || ck >= cz) continue;
    const int64_t cell = ci + (int64_t)cx * (cj + (int64_t)cy * ck);
    const double Kc = in.K[cell], pdc = in.pd[cell];
    const double* law = in.law ? law_row(in.kr_tab, in.law[cell]) : nullptr;
    int64_t vq[NC];
    double se[NC], pnq[NC], pcq[NC], dpcq[NC], pwq[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      vq[q] = pidx(d, ci + (q & 1), cj + ((q >> 1) & 1), DIM == 3 ? ck + ((q >> 2) & 1) : 0);
      se[q] = in.Se[vq[q]];
      pnq[q] = in.pn[vq[q]];
      pcq[q] = in.pc[vq[q]];
      dpcq[q] = in.dpc[vq[q]];
      pwq[q] = darcy ? in.u[vq[q]].x : 0.0;
    }
#pragma unroll
    for (int kk = 0; kk < DIM; ++kk) {
      // the face of this element along axis kk through this vertex's edge
      int oth[2], no = 0;
#pragma unroll
      for (int m = 0; m < DIM; ++m)
        if (m != kk) oth[no++] = m;
      double Af = 1.0;
#pragma unroll
      for (int t = 0; t < DIM - 1; ++t) Af = __dmul_rn(Af, __dmul_rn(ph.h[oth[t]], 0.5));
      const double KA = __dmul_rn(Kc, Af);
      int o[2] = {0, 0};
#pragma unroll
      for (int t = 0; t < DIM - 1; ++t) o[t] = (c >> oth[t]) & 1;
      const int a = c & ~(1 << kk), b = c | (1 << kk);
      const double sgn = ((c >> kk) & 1) ? 1.0 : -1.0;  // this vertex is b: +flux, a: -flux
      double gpn = 0.0, gpc = 0.0, gpw = 0.0;
#pragma unroll
      for (int e2 = 0; e2 < NE; ++e2) {
        int o2[2] = {e2 & 1, (e2 >> 1) & 1};
        double w = 1.0;
        int a2 = 0;
#pragma unroll
        for (int t = 0; t < DIM - 1; ++t) {
          w = w * (o2[t] == o[t] ? 0.75 : 0.25);
          a2 |= o2[t] << oth[t];
        }
        const int b2 = a2 | (1 << kk);
        gpn = __dadd_rn(gpn, __dmul_rn(w, __dsub_rn(pnq[b2], pnq[a2])));
        gpc = __dadd_rn(gpc, __dmul_rn(w, __dsub_rn(pcq[b2], pcq[a2])));
        if (darcy) gpw = __dadd_rn(gpw, __dmul_rn(w, __dsub_rn(pwq[b2], pwq[a2])));
      }
      gpn = __ddiv_rn(gpn, ph.h[kk]);
      gpc = __ddiv_rn(gpc, ph.h[kk]);
      gpw = __ddiv_rn(gpw, ph.h[kk]);
      double wM[NC], SeM = 0.0;
#pragma unroll
      for (int q = 0; q < NC; ++q) {
        double w = 0.5;
#pragma unroll
        for (int t = 0; t < DIM - 1; ++t) w = w * ((((q >> oth[t]) & 1) == o[t]) ? 0.75 : 0.25);
        wM[q] = w;
        SeM = __dadd_rn(SeM, __dmul_rn(w, se[q]));
      }
      const double Tw = __dmul_rn(-KA, __dsub_rn(gpn, __dmul_rn(ph.rho_w, ph.g[kk])));
      const double Tn = __dmul_rn(-KA, __dsub_rn(gpn, __dmul_rn(ph.rho_n, ph.g[kk])));
      const double Tc = __dmul_rn(-KA, gpc);
      // Darcy-velocity upwinding variant: the whole water flux by the sign of
      // T_pw = -K A_f (G(p_w) - rho_w g_k) (= T_w - T_c in exact arithmetic)
      const double Tpw = __dmul_rn(-KA, __dsub_rn(gpw, __dmul_rn(ph.rho_w, ph.g[kk])));
      const bool wa = darcy ? Tpw >= 0.0 : Tw >= 0.0, na = Tn >= 0.0;
      const int64_t vw = wa ? vq[a] : vq[b];
      const int64_t vn = na ? vq[a] : vq[b];
      double lw_up, dlw_up;   // k_rw / mu_w of the upwind vertex (with this element's law) and its S_n-derivative
      if (!law) {
        lw_up = in.krw[vw];
        dlw_up = in.dkrw[vw];
      } else {
        double k, dk;
        krw_law(ph.lam, law, in.Se[vw], k, dk);
        lw_up = k / ph.mu_w;
        dlw_up = (-dk / ph.den) / ph.mu_w;
      }
      double kM, dkM;
      krw_law(ph.lam, law, SeM, kM, dkM);
      const double lwM = kM / ph.mu_w;
      double sh, dsh, kn, dkn;
      shat_of(ph.lam, in.Se[vn], pdc, in.pdmin[vn], sh, dsh);
      krn_law(ph.lam, law, sh, kn, dkn);
      const double ln_up = kn / ph.mu_n;
      const double Fw = darcy ? ph.rho_w * (lw_up * Tpw) : ph.rho_w * (lw_up * Tw - lwM * Tc);
      const double Fn = ph.rho_n * (ln_up * Tn);
      F0 += sgn * Fw;
      F1 += sgn * Fn;
      if (WANT_J) {
        const double dlwM_dSeM = dkM / ph.mu_w;
        const double dln_up = dkn * dsh * neg_inv_den / ph.mu_n;
        const int qw = wa ? a : b, qn = na ? a : b;
#pragma unroll
        for (int q = 0; q < NC; ++q) {
          int nq = 0;   // number of 1/4 factors of this corner's weight
#pragma unroll
          for (int t = 0; t < DIM - 1; ++t) nq += (((q >> oth[t]) & 1) == o[t]) ? 0 : 1;
          const double gq = ((q >> kk) & 1) ? gtab[kk][nq] : -gtab[kk][nq];
          const double dT = -KA * gq;
          const double dlwM = wM[q] * dlwM_dSeM * neg_inv_den;
          const double d0 = ph.rho_w * lw_up * dT;
          const double d1 = darcy ? ph.rho_w * (q == qw ? dlw_up * Tpw : 0.0)
                                  : ph.rho_w * ((q == qw ? dlw_up * Tw : 0.0) + lw_up * dT * dpcq[q] - dlwM * Tc -
                                                lwM * dT * dpcq[q]);
          const double d2 = ph.rho_n * ln_up * dT;
          const double d3 = ph.rho_n * ((q == qn ? dln_up * Tn : 0.0) + ln_up * dT * dpcq[q]);
          const int dx = (q & 1) - (c & 1), dy = ((q >> 1) & 1) - ((c >> 1) & 1),
                    dz = DIM == 3 ? ((q >> 2) & 1) - ((c >> 2) & 1) : 0;
          const int bi = blk_of(DIM, dx, dy, dz);
          double* r = acc + (bi * 4) * BS + tid;
          r[0] += sgn * d0;
          r[BS] += sgn * d1;
          r[2 * BS] += sgn * d2;
          r[3 * BS] += sgn * d3;
        }
      }
    }
  }
  const bool dirv = in.dir[p] != 0;
  if (dirv) F0 = in.pw_dir[p] - in.u[p].x;
  F[p] = make_double2(F0, F1);
  if (WANT_J) {
    double pv = in.phiv[p];
    if (ph.scheme & SCHEME_SHAT_STORAGE) {
      // S hat storage: d m_n / d S_n = rho_n sum_j Phi_j |b_i^j| d S hat_e / d S_e
      const double frac = DIM == 3 ? 0.125 : 0.25, se = in.Se[p], pdm = in.pdmin[p];
      pv = 0.0;
      for (int c = 0; c < NC; ++c) {
        const int ci = i - (c & 1), cj = j - ((c >> 1) & 1), ck = DIM == 3 ? k - ((c >> 2) & 1) : 0;
        if (ci < 0 || ci >= cx || cj < 0 || cj >= cy || ck < 0 || ck >= cz) continue;
        const int64_t cell = ci + (int64_t)cx * (cj + (int64_t)cy * ck);
        double sh, dsh;
        shat_of(ph.lam, se, in.pd[cell], pdm, sh, dsh);
        pv += in.phi[cell] * in.vol * frac * dsh;
      }
    }
    mdiag[p] = make_double2(dirv ? 0.0 : -ph.rho_w * pv, ph.rho_n * pv);
    const int centre = DIM == 3 ? 13 : 4;
#pragma unroll 3
    for (int bi = 0; bi < NB; ++bi) {
      double e0 = acc[(bi * 4 + 0) * BS + tid], e1 = acc[(bi * 4 + 1) * BS + tid];
      double e2 = acc[(bi * 4 + 2) * BS + tid], e3 = acc[(bi * 4 + 3) * BS + tid];
      if (dirv) { e0 = (bi == centre) ? -1.0 : 0.0; e1 = 0.0; }
      double2* dst = reinterpret_cast<double2*>(J + ((int64_t)bi * d.nv + p) * 4);
      dst[0] = make_double2(e0, e1);
      dst[1] = make_double2(e2, e3);
    }
  }
}

// ---------------------------------------------------------------- K1, faces then rows
// K1 is FP64-pipe-bound on GB300 (0.53 T FMA/s against 6.8 TB/s), so it is
// organised to evaluate nothing twice.  Two passes over slabs of cell planes:
//   k_asm_faces  one thread per element and axis evaluates the element's SCV
//     faces along that axis and leaves, per face, the fluxes F_w, F_n and their
//     derivatives by the 2^d corners' unknowns;
//   k_asm_rows   adds them up per vertex: the water threads write the entries
//     (w, p_w), (w, S_n) and F_w, the NAPL threads (n, p_w), (n, S_n), F_n and
//     M.  Every row is written once, complete (no zero fill, no read-modify-
//     write, no atomics).
// A preconditioned solve amplifies a last-bit difference of its matrix or right-
// hand side by 10^2 or more per iteration, so the values are those of the
// element-by-element assembly to the last bit: each derivative in the vertex
// kernel's operations, and a row's contributions added in the order of the
// elements' colours (parities of their lower corner), within an element along
// x, y, z.  The row pass takes its vertex's neighbours mirrored along the
// axes where the vertex's coordinate is odd: the colour order is then the same
// sequence of offsets for every vertex, and the 27 accumulators stay in
// registers.
// Of a face's derivatives by p_w only d are distinct (the weights of its
// corners: 3/4 or 1/4 per other axis), +- by side; those are stored once.
// Measured on GB300 (F, J and M; then F alone), against one thread per element
// adding its faces' 768 entries into J colour by colour (4,154 FP64 instructions
// per vertex; on small grids 8 dependent chains of about 190 us): 257^3 150.9 ->
// 91.0 ms (52.1 -> 25.2 ms), 65^3 2.79 -> 1.54 ms (1.00 -> 0.47), 17^3 1.57 -> 0.071
// ms (0.60 -> 0.042), 33^2 0.224 -> 0.039 ms.  1,821 FP64-pipe instructions per
// element in the first pass and 806 per vertex in the second, whose pipe is 83%
// and 82% busy (ncu at 97^3); DRAM at 10% and 28% of its peak.  (Summing a row's faces
// before their products with dp_c/dS_n, not to the last bit, took 63.1 ms.)
// numbers per face: F_w, F_n, and with J the distinct dF_w/dp_w and dF_n/dp_w
// and the 2^d dF_w/dS_n and dF_n/dS_n
__host__ __device__ constexpr int nco(int dim, bool want_j) { return want_j ? 2 + 2 * dim + (2 << dim) : 2; }

// A slab: cell planes [c0, c1) along axis ax (z in 3D, y in 2D; y in 3D too
// where z planes are too large for the workspace) in face workspace W, plane c
// in ring slot c % ring (the plane below the slab stays for the slab's first
// vertex plane).  Number m of face f (axis * 2^(d-1) + position) of in-plane
// cell q lies at W[(f * nco + m) * ws + slot * pc + q].  Cells are parity-split
// along x as vertices are.
struct Slab {
  double* W;
  int ws, pc, ring, c0, c1, ax;
};

// a + w x, product and sum rounded separately; a power-of-two weight's product
// is exact, so one fused operation rounds alike
__device__ __forceinline__ double add_term(double a, double w, double x, bool pow2) {
  return pow2 ? __fma_rn(w, x, a) : __dadd_rn(a, __dmul_rn(w, x));
}

// x >= 0 (-0 included) from the bits: comparisons of doubles issue on the FP64
// pipe.  (A NaN flux makes F and J NaN whichever side it takes.)
__device__ __forceinline__ bool not_below(double x) {
  const int hi = __double2hiint(x);
  return hi >= 0 || (((uint32_t)hi << 1) | (uint32_t)__double2loint(x)) == 0u;
}

// -x where neg: the sign bit alone (an addition and a subtraction behind a
// select would both issue on the FP64 pipe)
__device__ __forceinline__ double flip_sign(double x, bool neg) {
  return __hiloint2double(__double2hiint(x) ^ (neg ? (int)0x80000000 : 0), __double2loint(x));
}

template <int DIM, int K, bool WANT_J, bool DARCY>
__device__ __forceinline__ void faces_of_axis(const Dims& d, const Phys& ph, const AsmIn& in, const Slab& sl, int t) {
  constexpr int NC = 1 << DIM, NE = 1 << (DIM - 1), CO = nco(DIM, WANT_J);
  constexpr int O1 = K == 0 ? 1 : 0, O2 = K == 2 ? 1 : 2;   // the other axes, in order
  const int cx = d.nx - 1, cy = d.ny - 1, EC = (cx + 1) / 2;
  const int pl = (int)((uint32_t)t / (uint32_t)sl.pc), q0 = t - pl * sl.pc;
  const int line = (int)((uint32_t)q0 / (uint32_t)cx), pos = q0 - line * cx, plane = sl.c0 + pl;
  const int ci = pos < EC ? 2 * pos : 2 * (pos - EC) + 1;
  const int cj = DIM == 2 || sl.ax == 1 ? plane : line;
  const int ck = DIM == 2 ? 0 : sl.ax == 1 ? line : plane;
  const int64_t cell = ci + (int64_t)cx * (cj + (int64_t)cy * ck);
  const double Kc = in.K[cell], pdc = in.pd[cell];
  const double* law = in.law ? law_row(in.kr_tab, in.law[cell]) : nullptr;
  const double h = ph.h[K], rh = ph.rh[K];
  const double KA = __dmul_rn(Kc, ph.Af[K]);
  int vq[NC];
  double se[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    vq[q] = (int)pidx(d, ci + (q & 1), cj + ((q >> 1) & 1), DIM == 3 ? ck + ((q >> 2) & 1) : 0);
    se[q] = in.Se[vq[q]];
  }
  double dn[NE], dc[NE], dw[NE];
#pragma unroll
  for (int e = 0; e < NE; ++e) {
    const int a = (e & 1) << O1 | (DIM == 3 ? (e >> 1) << O2 : 0), b = a | 1 << K;
    dn[e] = __dsub_rn(in.pn[vq[b]], in.pn[vq[a]]);
    dc[e] = __dsub_rn(in.pc[vq[b]], in.pc[vq[a]]);
    if (DARCY) dw[e] = __dsub_rn(in.u[vq[b]].x, in.u[vq[a]].x);
  }
  const double gw = ph.gw[K], gn = ph.gn[K];
  const int wi = (int)((uint32_t)plane % (uint32_t)sl.ring) * sl.pc + q0;
  double dT[DIM], dpcq[NC];        // K A_f w / h by the number of 1/4 factors
  if (WANT_J) {
#pragma unroll
    for (int m = 0; m < DIM; ++m) dT[m] = KA * ph.gt[K][m];
#pragma unroll
    for (int q = 0; q < NC; ++q) dpcq[q] = in.dpc[vq[q]];
  }
#pragma unroll
  for (int e = 0; e < NE; ++e) {
    const int a = (e & 1) << O1 | (DIM == 3 ? (e >> 1) << O2 : 0), b = a | 1 << K;
    double gpn = 0.0, gpc = 0.0, gpw = 0.0, SeM = 0.0;
#pragma unroll
    for (int e2 = 0; e2 < NE; ++e2) {
      double w = 1.0;
#pragma unroll
      for (int m = 0; m < DIM - 1; ++m) w = w * ((((e ^ e2) >> m) & 1) ? 0.25 : 0.75);
      const bool pow2 = (e ^ e2) == NE - 1;
      gpn = e2 ? add_term(gpn, w, dn[e2], pow2) : __dmul_rn(w, dn[0]);
      gpc = e2 ? add_term(gpc, w, dc[e2], pow2) : __dmul_rn(w, dc[0]);
      if (DARCY) gpw = e2 ? add_term(gpw, w, dw[e2], pow2) : __dmul_rn(w, dw[0]);
    }
    gpn = div_by(gpn, h, rh);
    gpc = div_by(gpc, h, rh);
    if (DARCY) gpw = div_by(gpw, h, rh);
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      double w = 0.5;
      w = w * ((((q >> O1) & 1) == (e & 1)) ? 0.75 : 0.25);
      if (DIM == 3) w = w * ((((q >> O2) & 1) == (e >> 1)) ? 0.75 : 0.25);
      SeM = q ? add_term(SeM, w, se[q], w == (DIM == 3 ? 0.03125 : 0.125)) : __dmul_rn(w, se[0]);
    }
    const double Tw = __dmul_rn(-KA, __dsub_rn(gpn, gw));
    const double Tn = __dmul_rn(-KA, __dsub_rn(gpn, gn));
    const double Tc = __dmul_rn(-KA, gpc);
    const double Tpw = DARCY ? __dmul_rn(-KA, __dsub_rn(gpw, gw)) : 0.0;
    const bool wa = not_below(DARCY ? Tpw : Tw), na = not_below(Tn);
    const int vw = wa ? vq[a] : vq[b], vn = na ? vq[a] : vq[b];   // selects, not indexing
    double lw_up, dlw_up = 0.0;   // k_rw / mu_w of the upwind vertex (with this element's law), its S_n-derivative
    if (!law) {
      lw_up = in.krw[vw];
      if (WANT_J) dlw_up = in.dkrw[vw];
    } else {
      double k, dk;
      krw_law(ph.lam, law, wa ? se[a] : se[b], k, dk);
      lw_up = k / ph.mu_w;
      dlw_up = (-dk / ph.den) / ph.mu_w;
    }
    double kM, dkM;
    if (!law && ph.lam == 2.0 && (uint32_t)__double2hiint(SeM) - 1u < 0x3fefffffu) {   // inside (0, 1): no clamps
      const double s2 = SeM * SeM;
      kM = s2 * s2;
      dkM = 4.0 * s2 * SeM;
    } else {
      krw_law(ph.lam, law, SeM, kM, dkM);
    }
    const double lwM = div_by(kM, ph.mu_w, ph.rmu_w);
    // lambda_n of S hat at the upwind vertex: the vertex's own where S hat = S_e
    double ln_up, dln_up = 0.0;
    const double pdm = in.pdmin[vn];
    if (!law && __double_as_longlong(pdc) == __double_as_longlong(pdm)) {
      ln_up = in.krn[vn];
      if (WANT_J) dln_up = in.dkrn[vn];
    } else {
      double sh, dsh, kn, dkn;
      shat_of(ph.lam, na ? se[a] : se[b], pdc, pdm, sh, dsh);
      krn_law(ph.lam, law, sh, kn, dkn);
      ln_up = kn / ph.mu_n;
      dln_up = dkn * dsh * ph.nid / ph.mu_n;
    }
    double* W = sl.W + (size_t)((K * NE + e) * CO) * sl.ws + wi;
    W[0] = DARCY ? ph.rho_w * (lw_up * Tpw) : ph.rho_w * (lw_up * Tw - lwM * Tc);
    W[(size_t)sl.ws] = ph.rho_n * (ln_up * Tn);
    if (WANT_J) {
      const double dlM = div_by(dkM, ph.mu_w, ph.rmu_w);
      const double rlw = ph.rho_w * lw_up, rln = ph.rho_n * ln_up;
      const double selw = dlw_up * (DARCY ? Tpw : Tw), seln = dln_up * Tn;
      double U[DIM], V[DIM], G[DIM], L[DIM];
#pragma unroll
      for (int m = 0; m < DIM; ++m) {
        W[(size_t)(2 + m) * sl.ws] = rlw * dT[m];
        W[(size_t)(2 + DIM + m) * sl.ws] = rln * dT[m];
        double w = 0.5;
#pragma unroll
        for (int t = 0; t < DIM - 1; ++t) w = w * (t < m ? 0.25 : 0.75);
        U[m] = lw_up * dT[m];
        V[m] = lwM * dT[m];
        L[m] = ln_up * dT[m];
        G[m] = w * dlM * ph.nid * Tc;
      }
      // corner j: bits 0, 1 = differs from the face's position along the other
      // axes, then the side along K; d T / d p(q) is -dT above, +dT below
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        const int side = j >> (DIM - 1), m = (j & 1) + (DIM == 3 ? (j >> 1) & 1 : 0);
        const int q = ((e ^ j) & 1) << O1 | (DIM == 3 ? (((e ^ j) >> 1) & 1) << O2 : 0) | side << K;
        const bool up = (j & (NE - 1)) == 0;       // the face's own edge: its upwind end takes the k_r slope
        double d1, d3;
        if (DARCY) {
          d1 = up && wa == (side == 0) ? selw : 0.0;
        } else {
          const double A = U[m] * dpcq[q], C = V[m] * dpcq[q];
          d1 = side ? -A : A;
          if (up) d1 = (wa == (side == 0) ? selw : 0.0) + d1;
          d1 = d1 - G[m];
          d1 = side ? d1 + C : d1 - C;
        }
        const double B = L[m] * dpcq[q];
        d3 = side ? -B : B;
        if (up) d3 = (na == (side == 0) ? seln : 0.0) + d3;
        W[(size_t)(2 + 2 * DIM + j) * sl.ws] = ph.rho_w * d1;
        W[(size_t)(2 + 2 * DIM + NC + j) * sl.ws] = ph.rho_n * d3;
      }
    }
  }
}

template <int DIM, bool WANT_J, bool DARCY>
__global__ void __launch_bounds__(128) k_asm_faces(const __grid_constant__ Dims d, const __grid_constant__ Phys ph,
                                                   const __grid_constant__ AsmIn in, const __grid_constant__ Slab sl) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (sl.c1 - sl.c0) * sl.pc) return;
  if (blockIdx.y == 0) faces_of_axis<DIM, 0, WANT_J, DARCY>(d, ph, in, sl, t);
  else if (blockIdx.y == 1) faces_of_axis<DIM, 1, WANT_J, DARCY>(d, ph, in, sl, t);
  else if (DIM == 3) faces_of_axis<DIM, DIM - 1, WANT_J, DARCY>(d, ph, in, sl, t);
}

// Vertex planes [v0, v1): 32 vertices per block, one warp their water rows and
// one their NAPL rows (so that the two halves of each 32-byte block are written
// at about the same time; with blocks of two warps an SM holds ten of these
// warps, whose accumulators take 108 registers).  Sources, Dirichlet p_w rows (0
// = p_dir - p_w: J row -e, M row 0) and the mass diagonal are applied here.
// c: the element of colour c, whose corner s = (vertex parity ^ c) the vertex is.
// In mirrored coordinates it extends to +1 along the axes where c's bit is 0
// and to -1 where it is 1.
template <int DIM, bool WANT_J>
__global__ void __launch_bounds__(64) k_asm_rows(const __grid_constant__ Dims d, const __grid_constant__ Phys ph,
                                                 const __grid_constant__ AsmIn in, const __grid_constant__ Slab sl, int v0,
                                                 int v1, double* __restrict__ F, double* __restrict__ J,
                                                 double2* __restrict__ mdiag) {
  constexpr int NC = 1 << DIM, NE = 1 << (DIM - 1), NB = DIM == 3 ? 27 : 9, CO = nco(DIM, WANT_J);
  const int napl = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nline = DIM == 2 ? 1 : sl.ax == 1 ? d.nz : d.ny;    // x-lines per vertex plane
  const int64_t t = (int64_t)blockIdx.x * 32 + lane;
  if (t >= (int64_t)(v1 - v0) * nline * d.nx) return;
  const uint32_t l0 = (uint32_t)t / (uint32_t)d.nx, pl = l0 / (uint32_t)nline;   // nv < 2^31
  const int vpos = (int)((uint32_t)t - l0 * (uint32_t)d.nx), line = (int)(l0 - pl * (uint32_t)nline), vpl = v0 + (int)pl;
  const int i = vpos < d.E ? 2 * vpos : 2 * (vpos - d.E) + 1;
  const int j = DIM == 2 || sl.ax == 1 ? vpl : line, k = DIM == 2 ? 0 : sl.ax == 1 ? line : vpl;
  const int64_t p = ((int64_t)j + (int64_t)d.ny * k) * d.nx + vpos;
  const int cx = d.nx - 1, cy = d.ny - 1, cz = DIM == 3 ? d.nz - 1 : 1, EC = (cx + 1) / 2;
  const int par = (i & 1) | (j & 1) << 1 | (DIM == 3 ? (k & 1) << 2 : 0);
  double a0[NB], a1[NB], f = 0.0;
  if (WANT_J) {
#pragma unroll
    for (int b = 0; b < NB; ++b) { a0[b] = 0.0; a1[b] = 0.0; }
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const int s = par ^ c;
    const int ci = i - (s & 1), cj = j - ((s >> 1) & 1), ck = DIM == 3 ? k - ((s >> 2) & 1) : 0;
    if (ci < 0 || ci >= cx || cj < 0 || cj >= cy || ck < 0 || ck >= cz) continue;
    const int pos = (ci & 1) ? EC + (ci >> 1) : (ci >> 1);
    const int plane = DIM == 2 || sl.ax == 1 ? cj : ck, cl = DIM == 2 ? 0 : sl.ax == 1 ? ck : cj;
    const double* W = sl.W + ((uint32_t)plane % (uint32_t)sl.ring) * (uint32_t)sl.pc + cl * cx + pos;
    double fe = 0.0;
#pragma unroll
    for (int kk = 0; kk < DIM; ++kk) {
      const int o1 = kk == 0 ? 1 : 0, o2 = kk == 2 ? 1 : 2;
      const int e = ((s >> o1) & 1) | (DIM == 3 ? ((s >> o2) & 1) << 1 : 0);
      const double* Wf = W + (size_t)((kk * NE + e) * CO) * sl.ws;
      const int sk = (s >> kk) & 1;              // the vertex is the face's lower (0: row -) or upper (1: row +) end
      const double fv = Wf[(size_t)napl * sl.ws];
      fe = fe + flip_sign(fv, sk == 0);
      if (WANT_J) {
        const double* Wx = Wf + (size_t)(2 + napl * DIM) * sl.ws;
        const double* Wown = Wf + (size_t)(2 + 2 * DIM + napl * NC + sk * NE) * sl.ws;
        const double* Wfar = Wf + (size_t)(2 + 2 * DIM + napl * NC + (1 - sk) * NE) * sl.ws;
        double x[DIM], own[NE], far[NE];
#pragma unroll
        for (int m = 0; m < DIM; ++m) x[m] = Wx[(size_t)m * sl.ws];
#pragma unroll
        for (int r = 0; r < NE; ++r) {
          own[r] = flip_sign(Wown[(size_t)r * sl.ws], sk == 0);
          far[r] = flip_sign(Wfar[(size_t)r * sl.ws], sk == 0);
        }
#pragma unroll
        for (int r = 0; r < NE; ++r) {
          // corner r of the face's other axes: mirrored block offsets of its two sides
          const int D1 = r & 1, D2 = DIM == 3 ? (r >> 1) & 1 : 0, m = D1 + D2;
          const int u1 = D1 ? ((c >> o1) & 1 ? -1 : 1) : 0, u2 = D2 ? ((c >> o2) & 1 ? -1 : 1) : 0;
          const int uk = (c >> kk) & 1 ? -1 : 1;
          const int st1 = o1 == 0 ? 1 : 3, st2 = o2 == 1 ? 3 : 9, stk = kk == 0 ? 1 : kk == 1 ? 3 : 9;
          const int bo = (DIM == 3 ? 13 : 4) + u1 * st1 + (DIM == 3 ? u2 * st2 : 0), bf = bo + uk * stk;
          a0[bo] = a0[bo] - x[m];
          a0[bf] = a0[bf] + x[m];
          a1[bo] = a1[bo] + own[r];
          a1[bf] = a1[bf] + far[r];
        }
      }
    }
    f += fe;
  }
  const bool dirv = in.dir[p] != 0;
  if (WANT_J) {
    constexpr int C = DIM == 3 ? 13 : 4;
    const int fx = i & 1 ? -1 : 1, fy = j & 1 ? -3 : 3, fz = DIM == 3 ? (k & 1 ? -9 : 9) : 0;   // back from the mirror
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int br = C + (b % 3 - 1) * fx + ((b / 3) % 3 - 1) * fy + (DIM == 3 ? (b / 9 - 1) * fz : 0);
      double2 v = make_double2(a0[b], a1[b]);
      if (dirv && !napl) v = make_double2(b == C ? -1.0 : 0.0, 0.0);
      *reinterpret_cast<double2*>(J + ((int64_t)br * d.nv + p) * 4 + 2 * napl) = v;
    }
    if (napl) {
      double pvol = in.phiv[p];
      if (ph.scheme & SCHEME_SHAT_STORAGE) {
        const double frac = DIM == 3 ? 0.125 : 0.25, se = in.Se[p], pdm = in.pdmin[p];
        pvol = 0.0;
        for (int c = 0; c < NC; ++c) {
          const int ci = i - (c & 1), cj = j - ((c >> 1) & 1), ck = DIM == 3 ? k - ((c >> 2) & 1) : 0;
          if (ci < 0 || ci >= cx || cj < 0 || cj >= cy || ck < 0 || ck >= cz) continue;
          const int64_t cell = ci + (int64_t)cx * (cj + (int64_t)cy * ck);
          double sh, dsh;
          shat_of(ph.lam, se, in.pd[cell], pdm, sh, dsh);
          pvol += in.phi[cell] * in.vol * frac * dsh;
        }
      }
      mdiag[p] = make_double2(dirv ? 0.0 : -ph.rho_w * pvol, ph.rho_n * pvol);
    }
  }
  if (in.q_in) f += napl ? in.q_in[p].y : in.q_in[p].x;
  if (dirv && !napl) f = in.pw_dir[p] - in.u[p].x;
  F[2 * p + napl] = f;
}

// ---------------------------------------------------------------- storage (S hat variant)
// sw[p] = sum over the sub-control volumes b_i^j of vertex p of Phi_j |b_i^j|
// S_w(b_i^j), with S_w = S_wr + S hat_e (1 - S_wr - S_nr) (Eq. (hSw)).
__global__ void k_storage_sw(Dims d, Phys ph, const double2* __restrict__ u, const double* __restrict__ pdmin,
                             const double* __restrict__ phi, const double* __restrict__ pd, double vol,
                             double* __restrict__ sw) {
  int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= d.nv) return;
  int i, j, k;
  pcoords(d, p, i, j, k);
  const int cx = d.nx - 1, cy = d.ny - 1, cz = d.dim == 3 ? d.nz - 1 : 1;
  const double frac = d.dim == 3 ? 0.125 : 0.25;
  const double se = __ddiv_rn(__dsub_rn(__dsub_rn(1.0, u[p].y), ph.S_wr), ph.den), pdm = pdmin[p];
  double s = 0.0;
  for (int c = 0; c < (1 << d.dim); ++c) {
    const int ci = i - (c & 1), cj = j - ((c >> 1) & 1), ck = d.dim == 3 ? k - ((c >> 2) & 1) : 0;
    if (ci < 0 || ci >= cx || cj < 0 || cj >= cy || ck < 0 || ck >= cz) continue;
    const int64_t cell = ci + (int64_t)cx * (cj + (int64_t)cy * ck);
    double sh, dsh;
    shat_of(ph.lam, se, pd[cell], pdm, sh, dsh);
    s += phi[cell] * vol * frac * (ph.S_wr + sh * ph.den);
  }
  sw[p] = s;
}

// ---------------------------------------------------------------- launchers
void launch_vertex_setup(const Dims& d, const double* pd, const double* phi, double vol, double* pdmin,
                         double* phiv, void* s) {
  RF_LAUNCH(k_vertex_setup, (int)((d.nv + 255) / 256), 256, 0, s, d, pd, phi, vol, pdmin, phiv);
}

void launch_perm_to_p(const Dims& d, const double* nat, double* out, void* s) {
  RF_LAUNCH(k_perm_to_p, (int)((d.nv + 255) / 256), 256, 0, s, d, (const double2*)nat, (double2*)out);
}
void launch_perm_from_p(const Dims& d, const double* pl, double* nat, void* s) {
  RF_LAUNCH(k_perm_from_p, (int)((d.nv + 255) / 256), 256, 0, s, d, (const double2*)pl, (double2*)nat);
}
void launch_perm_bytes_to_p(const Dims& d, const uint8_t* nat, uint8_t* out, void* s) {
  RF_LAUNCH(k_perm_bytes_to_p, (int)((d.nv + 255) / 256), 256, 0, s, d, nat, out);
}
void launch_perm_scalar_to_p(const Dims& d, const double* nat, double* out, void* s) {
  RF_LAUNCH(k_perm_scalar_to_p, (int)((d.nv + 255) / 256), 256, 0, s, d, nat, out);
}

// Face workspace of one assembly: at most ASM_WS_BYTES (with J; F alone a quarter of
// that, or what it is given), at least two cell planes.  At 257^3 the ring then holds 3
// planes of 151 MB, and a slab of 2 is 10 waves of k_asm_faces.  Slabs go along z, or
// along y where two z planes exceed the limit and y planes are smaller (wide, shallow
// boxes).  With 256 / 128 / 64 MB, J takes 3 / 10 / 23% longer at 65^3 (1.54 ms with 512)
// and 7 / 25 / 35% at 129^3 (11.2 ms), F alone 0 / 4 / 14% and 2 / 7 / 16%.
constexpr size_t ASM_WS_BYTES = (size_t)512 << 20;

struct SlabShape { int ax, planes, ring; int64_t plane; };

static size_t cell_bytes(const Dims& d, bool want_j) {
  return (size_t)(d.dim << (d.dim - 1)) * nco(d.dim, want_j) * sizeof(double);
}

static SlabShape slab_shape(const Dims& d, bool want_j, size_t bytes) {
  const size_t limit = want_j ? ASM_WS_BYTES : ASM_WS_BYTES / 4;
  const int64_t fit = (int64_t)((bytes < limit ? bytes : limit) / cell_bytes(d, want_j));   // cells
  const int64_t zp = (int64_t)(d.nx - 1) * (d.ny - 1), yp = (int64_t)(d.nx - 1) * (d.dim == 3 ? d.nz - 1 : 1);
  SlabShape r;
  r.ax = d.dim == 3 && (2 * zp <= fit || zp <= yp) ? 2 : 1;
  r.plane = r.ax == 2 ? zp : yp;
  r.planes = (r.ax == 2 ? d.nz : d.ny) - 1;
  const int64_t ring = fit / r.plane < 2 ? 2 : fit / r.plane;
  r.ring = (int)(ring < r.planes ? ring : r.planes);
  return r;
}

size_t assemble_workspace(const Dims& d) {
  const SlabShape r = slab_shape(d, true, ASM_WS_BYTES);
  return (size_t)(r.ring * r.plane) * cell_bytes(d, true);
}

template <int DIM, bool WANT_J>
static void slabs_t(const Dims& d, const Phys& ph, const AsmIn& in, const AsmArrays& a, void* s) {
  const SlabShape sh = slab_shape(d, WANT_J, a.faces_bytes);
  const int planes = sh.planes;
  Slab sl;
  sl.ax = sh.ax;
  sl.ring = sh.ring;
  sl.pc = (int)sh.plane;
  sl.ws = (int)(sh.plane * sh.ring);
  sl.W = a.faces;
  // the first slab fills the ring; a later one leaves the plane below it in place
  for (int c0 = 0, v0 = 0; c0 < planes;) {
    const int c1 = c0 == 0 ? sl.ring : (c0 + sl.ring - 1 < planes ? c0 + sl.ring - 1 : planes);
    sl.c0 = c0;
    sl.c1 = c1;
    const int64_t nc = (int64_t)(c1 - c0) * sh.plane;
    const dim3 g((unsigned)((nc + 127) / 128), DIM);
    if (ph.scheme & SCHEME_DARCY_UPWIND) RF_LAUNCH((k_asm_faces<DIM, WANT_J, true>), g, 128, 0, s, d, ph, in, sl);
    else RF_LAUNCH((k_asm_faces<DIM, WANT_J, false>), g, 128, 0, s, d, ph, in, sl);
    const int v1 = c1 == planes ? planes + 1 : c1;
    const int64_t nvert = (int64_t)(v1 - v0) * d.nx * (DIM == 2 ? 1 : sh.ax == 1 ? d.nz : d.ny);
    RF_LAUNCH((k_asm_rows<DIM, WANT_J>), (unsigned)((nvert + 31) / 32), 64, 0, s, d, ph, in, sl, v0, v1, a.F, a.J,
              (double2*)a.mdiag);
    c0 = c1;
    v0 = v1;
  }
}

cudaError_t launch_assemble(const Dims& d, const PhysParams& pp, const AsmArrays& a, bool want_j, void* s) {
  Phys ph;
  ph.rho_w = pp.rho_w; ph.rho_n = pp.rho_n; ph.mu_w = pp.mu_w; ph.mu_n = pp.mu_n;
  ph.S_wr = pp.S_wr; ph.S_nr = pp.S_nr; ph.lam = pp.lambda;
  ph.den = 1.0 - pp.S_wr - pp.S_nr;
  ph.scheme = pp.scheme;
  for (int t = 0; t < 3; ++t) { ph.h[t] = pp.h[t]; ph.g[t] = pp.g[t]; ph.rh[t] = recip(pp.h[t]); }
  ph.rmu_w = recip(pp.mu_w);
  ph.rmu_n = recip(pp.mu_n);
  ph.rden = recip(ph.den);
  ph.nid = -1.0 / ph.den;
  for (int t = 0; t < 3; ++t) {
    ph.Af[t] = 1.0;
    for (int m = 0; m < d.dim; ++m)
      if (m != t) ph.Af[t] *= pp.h[m] * 0.5;
    ph.gw[t] = pp.rho_w * pp.g[t];
    ph.gn[t] = pp.rho_n * pp.g[t];
    for (int m = 0; m < 3; ++m) {
      double w = 1.0;
      for (int q = 0; q < d.dim - 1; ++q) w *= q < m ? 0.25 : 0.75;
      ph.gt[t][m] = w / pp.h[t];
    }
  }
  const int nblk = (int)((d.nv + 255) / 256);
  RF_LAUNCH(k_vertex_state, nblk, 256, 0, s, d, ph, (const double2*)a.u, a.pdmin, a.Se, a.pn, a.pc, a.dpc,
            a.krw, a.dkrw, a.krn, a.dkrn);
  AsmIn in;
  in.u = (const double2*)a.u; in.Se = a.Se; in.pn = a.pn; in.pc = a.pc; in.dpc = a.dpc; in.krw = a.krw;
  in.dkrw = a.dkrw; in.krn = a.krn; in.dkrn = a.dkrn; in.pdmin = a.pdmin; in.phiv = a.phiv; in.K = a.K; in.pd = a.pd; in.phi = a.phi;
  in.vol = a.vol; in.dir = a.dir;
  in.pw_dir = a.pw_dir; in.q_in = (const double2*)a.q_in;
  in.law = a.law; in.kr_tab = a.kr_tab;
  const char* pv = getenv("RF_ASM_VERTEX");   // read per assembly (an alternative kept for comparison)
  const bool per_vertex = pv && atoi(pv) != 0;
  if (!per_vertex) {
    if (d.dim == 3) {
      if (want_j) slabs_t<3, true>(d, ph, in, a, s);
      else slabs_t<3, false>(d, ph, in, a, s);
    } else {
      if (want_j) slabs_t<2, true>(d, ph, in, a, s);
      else slabs_t<2, false>(d, ph, in, a, s);
    }
    return cudaGetLastError();
  }
  const int BS = 128;
  const int grid = (int)((d.nv + BS - 1) / BS);
  const int nb = d.dim == 3 ? 27 : 9;
  size_t smem = want_j ? (size_t)nb * 4 * BS * sizeof(double) : 0;
  if (d.dim == 3) {
    if (want_j) {
      cudaFuncSetAttribute(k_assemble<3, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      RF_LAUNCH((k_assemble<3, true>), grid, BS, smem, s, d, ph, in, (double2*)a.F, a.J, (double2*)a.mdiag);
    } else {
      RF_LAUNCH((k_assemble<3, false>), grid, BS, 0, s, d, ph, in, (double2*)a.F, a.J, (double2*)a.mdiag);
    }
  } else {
    if (want_j) {
      cudaFuncSetAttribute(k_assemble<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      RF_LAUNCH((k_assemble<2, true>), grid, BS, smem, s, d, ph, in, (double2*)a.F, a.J, (double2*)a.mdiag);
    } else {
      RF_LAUNCH((k_assemble<2, false>), grid, BS, 0, s, d, ph, in, (double2*)a.F, a.J, (double2*)a.mdiag);
    }
  }
  return cudaGetLastError();
}

void launch_storage_sw(const Dims& d, const PhysParams& pp, const double* u, const double* pdmin,
                       const double* phi, const double* pd, double vol, double* sw, void* s) {
  Phys ph;
  ph.rho_w = pp.rho_w; ph.rho_n = pp.rho_n; ph.mu_w = pp.mu_w; ph.mu_n = pp.mu_n;
  ph.S_wr = pp.S_wr; ph.S_nr = pp.S_nr; ph.lam = pp.lambda;
  ph.den = 1.0 - pp.S_wr - pp.S_nr;
  ph.scheme = pp.scheme;
  for (int t = 0; t < 3; ++t) { ph.h[t] = pp.h[t]; ph.g[t] = pp.g[t]; ph.rh[t] = recip(pp.h[t]); }
  ph.rmu_w = recip(pp.mu_w);
  ph.rmu_n = recip(pp.mu_n);
  ph.rden = recip(ph.den);
  ph.nid = -1.0 / ph.den;
  for (int t = 0; t < 3; ++t) {
    ph.Af[t] = 1.0;
    for (int m = 0; m < d.dim; ++m)
      if (m != t) ph.Af[t] *= pp.h[m] * 0.5;
    ph.gw[t] = pp.rho_w * pp.g[t];
    ph.gn[t] = pp.rho_n * pp.g[t];
    for (int m = 0; m < 3; ++m) {
      double w = 1.0;
      for (int q = 0; q < d.dim - 1; ++q) w *= q < m ? 0.25 : 0.75;
      ph.gt[t][m] = w / pp.h[t];
    }
  }
  RF_LAUNCH(k_storage_sw, (int)((d.nv + 255) / 256), 256, 0, s, d, ph, (const double2*)u, pdmin, phi, pd, vol, sw);
}

}  // namespace rf
