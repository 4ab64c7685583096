// Exact two-material Riemann solver of the FIVER flux (arXiv 2508.16387,
// Sec. 4.2), FP64 with an optional FP32 start: wave curves of the stiffened
// gas, NASG, Mie-Grueneisen and JWL materials, the Newton iteration on p* and
// the star states. Used by the interface and Riemann kernels of m2c_solver.cu;
// the bulk kernels do not include it.
#pragma once
#include "m2c_physics.cuh"

namespace m2c {

// ---------------------------------------------------------------------------
// Exact two-material Riemann problem (Sec. 4.2, Eq. 1DRiemannProblem with the
// interface conditions of Sec. 3.5.1), FP64. Newton on p* from the PVRS guess,
// stop at the first step with |dp| <= 1e-12 |p|; 50 steps then bisection.
// SG wave curves in closed form; MG shock from the Hugoniot root, MG
// rarefaction by RK4 on equal pressure substeps whose number is fixed once
// per problem (fix_substeps) from a bound of the wave's pressure span.
// ---------------------------------------------------------------------------
// KEPT (template parameter below): the arithmetic of a mixed grid's interface (rcp_kept in
// m2c_physics.cuh says why it is kept), in the same control flow: IEEE roots and quotients,
// two-step reciprocals, the general e and c^2 along the isentrope, the PVRS start. Without
// it, the shorter forms of FP64 grids and Riemann batches. Materials with a finite tension
// cutoff take the kept arithmetic everywhere (has_cutoff): their isentrope can cross the jump
// of c^2 at the cutoff, where last bits and the way the iterates come decide between two
// roots, or whether one is found at all. What it costs: a FIVER launch of
// a late shock-bubble takes 2300 us at 192^3 and 1270 at 131x67x45, against 980 and 312 with
// the shorter forms (3188 and 1733 with the kept arithmetic before the control flow was made
// reconvergent): 35 FP64 instructions instead of 16 in the isentrope's right-hand side, and
// faces without a previous star pressure take 13 Newton iterations from the PVRS estimate.
constexpr double kNewtonTol = 1e-12;
constexpr int kNewtonCap = 50;
constexpr int kBisectCap = 200;
constexpr double kHugTol = 1e-14;
constexpr int kHugCap = 100;
constexpr int kRk4Steps = 64;

// One side of a problem with what its wave curve needs at every pressure.
struct Side {
  double rho, u, p, c, e;
  // SG: p + p_c, its reciprocal, rho c, 2 c/(g - 1), and the shock constants 2/((g + 1) rho),
  // (g - 1)/(g + 1) (p + p_c)
  double pb, ipb, z, cf, A, B;
  // MG: 1/rho, 1/c^2; last Hugoniot root and its slope at pressure hp (NaN: none)
  double iv, ic2, hp, hr, hd;
  int nrk;  // RK4 substeps of this side's MG rarefaction curve in one problem; 0: per evaluation
  // MG: the density the isentrope starts from (rho, or rho/rho0: mg_rhs), the spacing of
  // the problem's fixed RK4 nodes p_K - i dnode (0: none), and the isentrope states after
  // the first mbase and mbase - 1 full substeps, kept between the evaluations of one
  // problem (nearby pressures share their nodes; the iteration may step back over one)
  int mbase;
  // dspan = nrk dnode, the span bound the nodes cover; dreach, how far iterates may use them
  double r0, dnode, idnode, dspan, dreach, rbase, fbase, rprev, fprev;
};

template <bool KEPT>
__device__ inline bool make_side(const EosDev& q, double rho, double u, double p, Side& K) {
  double e = 0.0, c2 = 0.0, iv;
  if constexpr (KEPT) {
    if (!eos_e_c2_kept(q, rho, 1.0 / rho, p, e, c2)) return false;
    K.c = sqrt(c2);
    iv = div_kept(1.0, rho);
  } else {
    iv = rcp_nr(rho);
    if (!eos_e_c2<double, true>(q, rho, iv, p, e, c2)) return false;
    K.c = sqrt_nr(c2);
  }
  K.rho = rho;
  K.u = u;
  K.p = p;
  K.e = e;
  K.nrk = 0;
  K.dnode = K.dspan = K.dreach = 0.0;
  if (q.type == M2C_EOS_SG && KEPT) {
    K.pb = p + q.pc;
    K.z = rho * K.c;
    K.cf = 2.0 * K.c / (q.g - 1.0);
    K.A = 2.0 / ((q.g + 1.0) * rho);
  } else if (q.type == M2C_EOS_SG) {
    K.pb = p + q.pc;
    K.ipb = rcp_nr(K.pb);
    K.z = rho * K.c;
    K.cf = q.two_gm1 * K.c;
    K.A = (1.0 - q.gm) * iv;
    K.B = q.gm * K.pb;
  } else {
    K.iv = iv;
    if constexpr (!KEPT) K.ic2 = rcp_nr(c2);
    K.hp = NAN;
    K.mbase = 0;
    K.r0 = KEPT ? rho : rho * (2.0 * q.inv_2rho0);
    K.rbase = K.rprev = K.r0;
    K.fbase = K.fprev = 0.0;
  }
  return true;
}

// Lowest admissible pressure of a side: p + p_c > 0 (SG, NASG), p > 0 (JWL,
// whose rarefaction is integrated in ln p), the MG tensile cutoff if any.
__device__ inline double eos_plow(const EosDev& q) {
  if (q.type == M2C_EOS_SG || q.type == M2C_EOS_NASG) return -q.pc;
  if (q.type == M2C_EOS_JWL) return 0.0;
  return isfinite(q.eta_min) ? q.pmin : -INFINITY;
}

// An MG material with a finite tension cutoff.
__device__ inline bool has_cutoff(const EosDev& q) { return q.type == M2C_EOS_MG && q.eta_min > -INFINITY; }

// Equal RK4 substeps over a pressure span dp of an MG isentrope: 64 for a span
// of at least 5% of K0 = rho0 c0^2, proportionally fewer (at least one) below.
__device__ inline int mg_substeps(const EosDev& q, double dp) {
  double nsd = ceil(div_nr(kRk4Steps * fabs(dp), q.rk4_span));  // div_nr: the IEEE quotient
  nsd = nsd >= 1.0 ? (nsd > kRk4Steps ? (double)kRk4Steps : nsd) : 1.0;
  return (int)nsd;
}

// JWL rarefactions are integrated in ln p (detonation products expand over
// decades): 256 substeps per unit of ln(p_K/p_lo), at least 8, with p_lo kept
// at or above 1e-6 p_K.
__device__ inline int jwl_substeps(double pK, double p_lo) {
  const double lo = fmax(p_lo, 1e-6 * pK);
  const double nd = ceil(256.0 * log(pK / lo));
  return nd < 8.0 ? 8 : (int)nd;
}

// The substep count of each MG side's rarefaction curve, fixed once per
// problem before the iteration so that the curve is one smooth function of p:
// the count for an upper bound of the pressure drop across the wave,
// p_K - max(p_low, min(p_J, p_ac)), with the acoustic estimate
// p_ac = (Z_R p_L + Z_L p_R - Z_L Z_R (u_R - u_L)) / (Z_L + Z_R), Z = rho c
// (a shock on the other side J keeps p* above p_J; a rarefaction there too
// keeps p* above p_ac, since each rarefaction curve lies below its acoustic
// tangent). Written without contracted multiply-adds.
// Returns p_ac.
__device__ inline double fix_substeps(const EosDev& qL, Side& L, const EosDev& qR, Side& Rs, double plow) {
  const double ZL = __dmul_rn(L.rho, L.c), ZR = __dmul_rn(Rs.rho, Rs.c);
  const double num = __dsub_rn(__dadd_rn(__dmul_rn(ZR, L.p), __dmul_rn(ZL, Rs.p)),
                               __dmul_rn(__dmul_rn(ZL, ZR), __dsub_rn(Rs.u, L.u)));
  const double pac = div_nr(num, __dadd_rn(ZL, ZR));
  const double loL = fmax(plow, fmin(Rs.p, pac)), loR = fmax(plow, fmin(L.p, pac));
  // MG: the count for the span bound and the spacing of the fixed nodes (span / count)
  auto mg_nodes = [](const EosDev& q, Side& K, double lo) {
    const double span = fmax(__dsub_rn(K.p, lo), 0.0);
    K.nrk = mg_substeps(q, span);
    K.dnode = (span > 0.0 && isfinite(span)) ? div_nr(span, (double)K.nrk) : 0.0;
    K.idnode = rcp_nr(K.dnode);
    K.dspan = K.dreach = __dmul_rn((double)K.nrk, K.dnode);
  };
  if (qL.type == M2C_EOS_MG) mg_nodes(qL, L, loL);
  if (qR.type == M2C_EOS_MG) mg_nodes(qR, Rs, loR);
  if (qL.type == M2C_EOS_JWL) L.nrk = jwl_substeps(L.p, loL);
  if (qR.type == M2C_EOS_JWL) Rs.nrk = jwl_substeps(Rs.p, loR);
  return pac;
}

// One side's wave curve at a pressure: f and f', and what the star density
// behind the wave follows from (a: SG rarefaction the power r^((g-1)/(2g)), MG
// shock and rarefaction rho*; b: MG d rho*/dp; NASG and JWL rho* and its slope).
struct Wave {
  double f, df, a, b;
};

// The solver's control flow has one entry and one exit per block (flags instead
// of returns inside loops), so that the lanes of a warp meet again after every
// branch and loop: with returns inside the loops a warp executed 12-15 Newton
// iterations and 90-140 isentrope substeps for an average of 3 and 30 a face
// (late shock-bubble), the lanes taking turns.
template <bool KEPT>
__device__ inline int wave_sg(const EosDev& q, const Side& K, double p, Wave& w) {
  const double pb = p + q.pc, dp = p - K.p;
  if constexpr (KEPT) {
    if (p > K.p) {
      const double B = q.gm * K.pb;
      const double sq = sqrt(K.A / (pb + B));
      w.f = (p - K.p) * sq;
      w.df = sq * (1.0 - 0.5 * (p - K.p) / (pb + B));
    } else {
      const double r = pb / K.pb;
      const double pw = pow(r, q.ex);
      w.f = K.cf * (pw - 1.0);
      w.df = pw / (r * K.rho * K.c);
    }
  } else if (p > K.p) {
    // f = dp sqrt(A/(pb + B)), f' = sqrt(A/(pb + B)) (1 - dp/(2 (pb + B)))
    const double iD = rcp_nr(pb + K.B), sq = sqrt_nr(K.A * iD);
    w.f = dp * sq;
    w.df = sq * fma(-0.5 * dp, iD, 1.0);
  } else {
    // one power serves f, f' (r^{-(g+1)/(2g)} = r^{(g-1)/(2g)} / r) and, after
    // the iteration, the density; r is the IEEE quotient (exactly 1 at p = p_K)
    const double r0 = pb * K.ipb, r = fma(fma(-K.pb, r0, pb), K.ipb, r0);
    const double pw = pow(r, q.ex);
    w.f = K.cf * (pw - 1.0);
    w.df = pw * rcp_nr(r * K.z);
    w.a = pw;
  }
  return pb >= 0.0 && K.pb > 0.0 ? M2C_OK : M2C_ENONPHYS;
}

// Density on the MG Hugoniot through K at pressure p > p_K (safeguarded Newton
// in a closed bracket, stopped at the first step below the tolerance) and
// d rho/dp along it. The start is the root of the problem's previous evaluation
// moved along its slope, else the acoustic density.
template <bool KEPT>
__device__ inline int mg_hugoniot(const EosDev& q, Side& K, double p, double& rho_out, double& drdp) {
  if constexpr (KEPT) {
    double lo = K.rho, hi = q.rmax;
    bool more = hi > lo;
    int st = more ? M2C_OK : M2C_ENONPHYS;
    double rho = K.rho + div_kept(p - K.p, K.c * K.c);
    if (!(rho > lo && rho < hi)) rho = 0.5 * (lo + hi);
    for (int it = 0; more; ++it) {
      const double ir = div_kept(1.0, rho), eta = 1.0 - div_kept(q.rho0, rho);
      double pR = 0.0, dpR = 0.0, eR = 0.0, deR = 0.0;
      mg_ref<double, true>(q, eta, pR, dpR, eR, deR);
      double e = eR + (p - pR) * q.inv_rg;
      double dedr = div_kept((deR - dpR * q.inv_rg) * q.rho0, rho * rho);
      double H = e - K.e - 0.5 * (p + K.p) * (K.iv - ir);
      double dH = dedr - div_kept(0.5 * (p + K.p), rho * rho);
      if (H > 0.0) lo = rho; else hi = rho;
      double rn = rho - div_kept(H, dH);
      if (!(rn >= lo && rn <= hi)) rn = 0.5 * (lo + hi);
      const bool conv = fabs(rn - rho) <= kHugTol * rn;
      rho = rn;
      if (!(eta < q.eta_max)) st = M2C_ENONPHYS;
      else if (!conv && it + 1 == kHugCap) st = M2C_ENOCONV;
      more = st == M2C_OK && !conv;
    }
    const double eta = 1.0 - div_kept(q.rho0, rho);
    if (!st && !(eta < q.eta_max)) st = M2C_ENONPHYS;
    double pR = 0.0, dpR = 0.0, eR = 0.0, deR = 0.0;
    mg_ref<double, true>(q, eta, pR, dpR, eR, deR);
    const double dedr = div_kept((deR - dpR * q.inv_rg) * q.rho0, rho * rho);
    double Hp = q.inv_rg - 0.5 * (K.iv - div_kept(1.0, rho));
    double Hr = dedr - div_kept(0.5 * (p + K.p), rho * rho);
    rho_out = rho;
    drdp = -div_kept(Hp, Hr);
    return st;
  }
  double lo = K.rho, hi = q.rmax;
  bool more = hi > lo;
  int st = more ? M2C_OK : M2C_ENONPHYS;
  double rho = K.hp == K.hp ? fma(K.hd, p - K.hp, K.hr) : fma(p - K.p, K.ic2, K.rho);
  if (!(rho > lo && rho < hi)) rho = 0.5 * (lo + hi);
  const double hp = 0.5 * (p + K.p);
  double dH = 1.0;
  for (int it = 0; more; ++it) {
    const double iv = rcp_nr(rho), eta = fma(-q.rho0, iv, 1.0);
    double pR = 0.0, dpR = 0.0, eR = 0.0, deR = 0.0;
    mg_ref<double>(q, eta, pR, dpR, eR, deR);
    const double H = fma(p - pR, q.inv_rg, eR) - K.e - hp * (K.iv - iv);
    dH = fma(fma(-dpR, q.inv_rg, deR), q.rho0, -hp) * (iv * iv);
    if (H > 0.0) lo = rho; else hi = rho;
    double rn = fma(-H, rcp_nr(dH), rho);
    if (!(rn >= lo && rn <= hi)) rn = 0.5 * (lo + hi);
    const bool conv = fabs(rn - rho) <= kHugTol * rn;
    rho = rn;
    if (!(eta < q.eta_max)) st = M2C_ENONPHYS;
    else if (!conv && it + 1 == kHugCap) st = M2C_ENOCONV;
    more = st == M2C_OK && !conv;
  }
  // along the Hugoniot d rho/dp = -H_p/H_rho, the slope H_rho from the last iterate
  const double Hp = q.inv_rg - 0.5 * (K.iv - rcp_nr(rho));
  rho_out = rho;
  drdp = -Hp * rcp_nr(dH);
  K.hp = p;
  K.hr = rho;
  K.hd = drdp;
  return st;
}

// Right-hand side of the MG isentrope in r = rho/rho0. With d = r - 1 and q = r - s d
// (1 - s eta = q/r) the sound speed of the compression branch is
//   rho^2 c^2 = K0 rho0 A,  A = n r^2/q^3 + g,  n = r + (s - G0) d,  g = (G0/K0) p,
// and the tension branch has the same form with q = r (s = 0). dr/dp = 1/(rho0 c^2) =
// (r y)^2/K0 and df/dp = 1/(rho c) = y/(K0 rho0)^(1/2) with y = A^(-1/2) =
// q^2 (q (n r^2 + g q^3))^(-1/2): 16 FP64 instructions with one root and no
// division (35 through the general e and c^2); the constant factors sit in the
// substep lengths, and r is of order 1 whatever the units of the density (in rho itself the
// root's argument is of order rho^4, which left its range below 4e-10). ok is cleared
// outside the EOS domain (rho <= 0, eta >= 1/s, c^2 not positive and finite). Materials with
// a finite tension cutoff do not come here (has_cutoff).
__device__ inline void mg_rhs(const EosDev& q, double g, double r, double& kr, double& y, bool& ok) {
  const double d = r - 1.0;
  const bool comp = gt0(d);
  double qq = fma(comp ? -q.s : 0.0, d, r);
  const double n = fma(comp ? q.sG : -q.G0, d, r);
  const double C = qq * fma(n, r * r, g * (qq * qq * qq)), q2 = qq * qq;
  ok = ok && gt0(r) && gt0(qq) && gt0(C) && hi_of(C) < 0x7ff00000u;
  y = q2 * rsqrt_nr(C);
  const double ry = r * y;
  kr = ry * ry;
}

// The same in the kept arithmetic: d rho/dp = 1/c^2 and df/dp = 1/(rho c) from one
// reciprocal square root of the general c^2 and the reciprocal of rho.
__device__ inline void mg_rhs_kept(const EosDev& q, double p, double rho, double& drho, double& dfv, bool& ok) {
  double e, c2 = 1.0;
  const double ir = rcp_kept(rho);
  ok = mg_e_c2_kept(q, rho, ir, p, e, c2) && ok;
  const double y = rsqrt_kept(c2);
  drho = y * y;
  dfv = y * ir;
}
// (h6: hs / 6, rounded)
__device__ inline void mg_rk4_substep_kept(const EosDev& q, double pi, double hs, double h6, double& rho, double& fv,
                                           bool& ok) {
  double k1r, k1f, k2r, k2f, k3r, k3f, k4r, k4f;
  mg_rhs_kept(q, pi, rho, k1r, k1f, ok);
  mg_rhs_kept(q, pi + 0.5 * hs, rho + 0.5 * hs * k1r, k2r, k2f, ok);
  mg_rhs_kept(q, pi + 0.5 * hs, rho + 0.5 * hs * k2r, k3r, k3f, ok);
  mg_rhs_kept(q, pi + hs, rho + hs * k3r, k4r, k4f, ok);
  rho = rho + h6 * (k1r + 2.0 * k2r + 2.0 * k3r + k4r);
  fv = fv + h6 * (k1f + 2.0 * k2f + 2.0 * k3f + k4f);
}

// One classical RK4 substep of the MG isentrope (r, f) from pressure pi by hs.
__device__ inline void mg_rk4_substep(const EosDev& q, double pi, double hs, double& r, double& fv, bool& ok) {
  const double g0 = q.gk * pi, gh = q.gk * hs, gm = fma(0.5, gh, g0);
  const double hr = hs * q.kap2, h2 = 0.5 * hr;
  double k1, k2, k3, k4, y1, y2, y3, y4;
  mg_rhs(q, g0, r, k1, y1, ok);
  mg_rhs(q, gm, fma(h2, k1, r), k2, y2, ok);
  mg_rhs(q, gm, fma(h2, k2, r), k3, y3, ok);
  mg_rhs(q, g0 + gh, fma(hr, k3, r), k4, y4, ok);
  r = fma(hr * (1.0 / 6.0), fma(2.0, k2 + k3, k1 + k4), r);
  fv = fma(hs * (q.kap * (1.0 / 6.0)), fma(2.0, y2 + y3, y1 + y4), fv);
}

// MG wave curve. Rarefaction: the isentrope integrated by classical RK4 in p;
// inside a problem's span bound on the fixed nodes p_K - i dnode (full substeps
// down to the last node above p, resumed from a node reached by an earlier
// evaluation of the problem, then one partial substep to p): the curve is
// continuous and smooth in p. Beyond the bound, and for a wave evaluated alone, equal
// substeps over p_K - p. An iterate less than a node spacing beyond the bound may take all
// nodes and the partial substep too (dreach: the nodes serve the next iterate; half the
// time of a batch of water against air), but no solution does: an isentrope into strong
// tension is not convex, its root can lie beyond the acoustic bound, and there the nodes
// carried on were 1e-8 off the equal substeps. All are one loop, so that the lanes of a
// warp take their substeps together. The node arithmetic is written without
// contracted multiply-adds, so that it takes the same nodes as the oracle.
template <bool KEPT>
__device__ inline int wave_mg(const EosDev& q, Side& K, double p, Wave& w) {
  int st = M2C_OK;
  if (p == K.p) {
    w.f = 0.0;
    w.df = KEPT ? 1.0 / (K.rho * K.c) : K.iv * rcp_nr(K.c);
    w.a = K.rho;
    w.b = KEPT ? 1.0 / (K.c * K.c) : K.ic2;
  } else if (p > K.p && KEPT) {
    double rho, drdp;
    st = mg_hugoniot<KEPT>(q, K, p, rho, drdp);
    double dv = K.iv - div_kept(1.0, rho);
    double fv = sqrt((p - K.p) * dv);
    w.f = fv;
    w.df = div_kept(dv + div_kept((p - K.p) * drdp, rho * rho), 2.0 * fv);
    w.a = rho;
    w.b = drdp;
  } else if (p > K.p) {
    double rho, drdp;
    st = mg_hugoniot<KEPT>(q, K, p, rho, drdp);
    const double ir = rcp_nr(rho), dv = K.iv - ir, dp = p - K.p;
    const double fv = sqrt_nr(dp * dv);
    w.f = fv;
    w.df = fma(dp * drdp, ir * ir, dv) * rcp_nr(2.0 * fv);
    w.a = rho;
    w.b = drdp;
  } else {
    const double dp = __dsub_rn(K.p, p);
    const bool within = K.nrk > 1 && K.dnode > 0.0 && dp < K.dreach;
    // (the isentrope's density: kept rho, else rho/rho0)
    double rho = K.r0, fv = 0.0, gap = 0.0, last = dp;
    int i = 0, m = 0;
    if (within) {
      if constexpr (KEPT) {
        m = (int)floor(div_kept(dp, K.dnode));
      } else {
        const double m0 = dp * K.idnode;
        m = (int)floor(fma(fma(-K.dnode, m0, dp), K.idnode, m0));  // the IEEE quotient dp/dnode
      }
      m = min(m, dp < K.dspan ? K.nrk - 1 : K.nrk);
      if (K.mbase <= m) {
        i = K.mbase;
        rho = K.rbase;
        fv = K.fbase;
      } else if (K.mbase == m + 1) {
        i = m;
        rho = K.rprev;
        fv = K.fprev;
      }
      gap = K.dnode;
    } else {
      // the problem's count (beyond its span bound), else one chosen for this span; a
      // count of one is a single substep, the partial one below
      const int ns = K.nrk > 0 ? K.nrk : mg_substeps(q, dp);
      if (ns > 1) {
        m = ns;
        gap = KEPT ? (K.p - p) / ns : div_nr(dp, (double)ns);
        last = 0.0;
      }
    }
    bool ok = true;
    if (i < m) {
      double rp = rho, fp = fv;
      const double h6 = KEPT ? -gap / 6.0 : 0.0;
      for (; i < m; ++i) {
        rp = rho;
        fp = fv;
        if constexpr (KEPT) {
          const double pi = within ? __dsub_rn(K.p, __dmul_rn((double)i, gap)) : fma((double)i, -gap, K.p);
          mg_rk4_substep_kept(q, pi, -gap, h6, rho, fv, ok);
        } else {
          mg_rk4_substep(q, __dsub_rn(K.p, __dmul_rn((double)i, gap)), -gap, rho, fv, ok);
        }
      }
      if (within) {
        K.mbase = m;
        K.rbase = rho;
        K.fbase = fv;
        K.rprev = rp;
        K.fprev = fp;
      }
    }
    const double pm = __dmul_rn((double)m, gap);
    if (within) last = __dsub_rn(dp, pm);
    if constexpr (KEPT) {
      if (last > 0.0) mg_rk4_substep_kept(q, __dsub_rn(K.p, pm), -last, -last / 6.0, rho, fv, ok);
      double e, c2 = 1.0;
      ok = mg_e_c2_kept(q, rho, 1.0 / rho, p, e, c2) && ok;
      w.f = fv;
      w.df = 1.0 / (rho * sqrt(c2));
      w.a = rho;
      w.b = 1.0 / c2;
    } else {
      if (last > 0.0) mg_rk4_substep(q, __dsub_rn(K.p, pm), -last, rho, fv, ok);
      double k, y;
      mg_rhs(q, q.gk * p, rho, k, y, ok);
      w.f = fv;
      w.df = y * q.kap;
      w.a = rho * q.rho0;
      w.b = k * q.kap2 * q.rho0;
    }
    if (!ok) st = M2C_ENONPHYS;
  }
  return st;
}

// NASG wave curves in P = p + p_c and the covolume-reduced specific volume
// w = 1/rho - b. Shock: the Hugoniot energy equation is linear in w,
// w = w_K (gm r + 1)/(r + gm), r = P/P_K, gm = (g - 1)/(g + 1), so
// f = (p - p_K) sqrt(A/(P + gm P_K)) with A = 2 w_K/(g + 1). Rarefaction: the
// isentrope P w^g = const gives rho c = sqrt(g P / w) and
// f = 2 c_K (1 - b rho_K)/(g - 1) (r^((g-1)/(2g)) - 1).
static __device__ __noinline__ int wave_nasg(const EosDev& q, const Side& K, double p, Wave& wv) {
  double &f = wv.f, &df = wv.df, &rs = wv.a, &drs = wv.b;
  const double g = q.g, b = q.b, P = p + q.pc, PK = K.p + q.pc, wK = 1.0 / K.rho - b;
  if (!(P >= 0.0) || !(PK > 0.0) || !(wK > 0.0)) return M2C_ENONPHYS;
  const double r = P / PK;
  if (p > K.p) {
    const double gm = (g - 1.0) / (g + 1.0), A = 2.0 * wK / (g + 1.0), D = P + gm * PK;
    const double sq = sqrt(A / D);
    f = (p - K.p) * sq;
    df = sq * (1.0 - 0.5 * (p - K.p) / D);
    const double w = wK * (gm * r + 1.0) / (r + gm);
    rs = 1.0 / (b + w);
    drs = rs * rs * wK * (1.0 - gm * gm) / ((r + gm) * (r + gm) * PK);
  } else {
    f = 2.0 * K.c * (1.0 - b * K.rho) / (g - 1.0) * (pow(r, (g - 1.0) / (2.0 * g)) - 1.0);
    const double w = wK * pow(r, -1.0 / g);
    df = sqrt(w / (g * P));
    rs = 1.0 / (b + w);
    drs = rs * rs * w / (g * P);
  }
  return M2C_OK;
}

// JWL Hugoniot through K at p > p_K: the root rho > rho_K of
// H(rho) = e(rho, p) - e_K - (p + p_K)(1/rho_K - 1/rho)/2, bracketed from
// [rho_K, rho_K (w + 2)/w] (doubling the upper end until H < 0), then Newton
// kept inside the bracket with the tolerance and stopping rule of the MG root;
// d rho/dp by implicit differentiation. de/drho|_p = -(f'(rho) + w e)/(w rho).
__device__ inline int jwl_hugoniot(const EosDev& q, const Side& K, double p, double& rho_out, double& drdp) {
  const double w = q.om;
  double lo = K.rho, hi = K.rho * (w + 2.0) / w;
  bool bracketed = false;
  for (int k = 0; k < 60 && !bracketed; ++k) {
    double f, df;
    jwl_f<double>(q, hi, 1.0 / hi, f, df);
    const double e = (p - f) / (w * hi);
    if (e - K.e - 0.5 * (p + K.p) * (1.0 / K.rho - 1.0 / hi) < 0.0) bracketed = true;
    else { lo = hi; hi = 2.0 * hi; }
  }
  if (!bracketed) return M2C_ENOCONV;
  double rho = K.rho + (p - K.p) / (K.c * K.c);
  if (!(rho > lo && rho < hi)) rho = 0.5 * (lo + hi);
  bool done = false;
  for (int it = 0; it < kHugCap; ++it) {
    double f, df;
    jwl_f<double>(q, rho, 1.0 / rho, f, df);
    const double e = (p - f) / (w * rho);
    const double dedr = -(df + w * e) / (w * rho);
    const double H = e - K.e - 0.5 * (p + K.p) * (1.0 / K.rho - 1.0 / rho);
    const double dH = dedr - 0.5 * (p + K.p) / (rho * rho);
    if (H > 0.0) lo = rho; else hi = rho;
    double rn = rho - H / dH;
    if (!(rn >= lo && rn <= hi)) rn = 0.5 * (lo + hi);
    const bool conv = fabs(rn - rho) <= kHugTol * rn;
    rho = rn;
    if (conv) { done = true; break; }
  }
  if (!done) return M2C_ENOCONV;
  double f, df;
  jwl_f<double>(q, rho, 1.0 / rho, f, df);
  const double e = (p - f) / (w * rho);
  const double Hp = 1.0 / (w * rho) - 0.5 * (1.0 / K.rho - 1.0 / rho);
  const double Hr = -(df + w * e) / (w * rho) - 0.5 * (p + K.p) / (rho * rho);
  rho_out = rho;
  drdp = -Hp / Hr;
  return M2C_OK;
}

// JWL wave curve: shock f = sqrt((p - p_K)(1/rho_K - 1/rho_H(p))); rarefaction:
// the isentrope d rho/dp = 1/c^2, df/dp = 1/(rho c) integrated by classical RK4
// in s = ln p on equal substeps (fixed per problem, fix_substeps; else for
// this span); it needs p > 0.
static __device__ __noinline__ int wave_jwl(const EosDev& q, const Side& K, double p, Wave& wv) {
  double &f = wv.f, &df = wv.df, &rs = wv.a, &drs = wv.b;
  if (p == K.p) {
    f = 0.0;
    df = 1.0 / (K.rho * K.c);
    rs = K.rho;
    drs = 1.0 / (K.c * K.c);
    return M2C_OK;
  }
  if (p > K.p) {
    double rho, drdp;
    const int st = jwl_hugoniot(q, K, p, rho, drdp);
    if (st) return st;
    const double dv = 1.0 / K.rho - 1.0 / rho;
    const double fv = sqrt((p - K.p) * dv);
    f = fv;
    df = (dv + (p - K.p) * drdp / (rho * rho)) / (2.0 * fv);
    rs = rho;
    drs = drdp;
    return M2C_OK;
  }
  if (!(p > 0.0) || !(K.p > 0.0)) return M2C_ENONPHYS;
  const double span = log(p / K.p);
  int ns = K.nrk;
  if (ns <= 0) {
    const double nd = ceil(256.0 * fabs(span));
    ns = nd < 8.0 ? 8 : (int)nd;
  }
  const double hs = span / ns, s0 = log(K.p);
  double rho = K.rho, fv = 0.0;
  // d(rho, f)/ds at (s, rho): (p / c^2, p / (rho c)) with p = exp(s)
  auto rhs = [&](double si, double r, double& kr, double& kf) {
    const double pp = exp(si);
    double e, c2;
    if (!eos_e_c2<double, true>(q, r, 1.0 / r, pp, e, c2)) return false;
    kr = pp / c2;
    kf = pp / (r * sqrt(c2));
    return true;
  };
  for (int i = 0; i < ns; ++i) {
    const double si = s0 + i * hs;
    double k1r, k1f, k2r, k2f, k3r, k3f, k4r, k4f;
    if (!rhs(si, rho, k1r, k1f) || !rhs(si + 0.5 * hs, rho + 0.5 * hs * k1r, k2r, k2f) ||
        !rhs(si + 0.5 * hs, rho + 0.5 * hs * k2r, k3r, k3f) || !rhs(si + hs, rho + hs * k3r, k4r, k4f))
      return M2C_ENONPHYS;
    rho = rho + hs / 6.0 * (k1r + 2.0 * k2r + 2.0 * k3r + k4r);
    fv = fv + hs / 6.0 * (k1f + 2.0 * k2f + 2.0 * k3f + k4f);
  }
  double e, c2;
  if (!eos_e_c2<double, true>(q, rho, 1.0 / rho, p, e, c2)) return M2C_ENONPHYS;
  f = fv;
  df = 1.0 / (rho * sqrt(c2));
  rs = rho;
  drs = 1.0 / c2;
  return M2C_OK;
}

// A side's wave curve at p; out of line, one copy for both sides.
template <bool KEPT>
static __device__ __noinline__ int wave(const EosDev& q, Side& K, double p, Wave& w) {
  if (q.type == M2C_EOS_SG) return wave_sg<KEPT>(q, K, p, w);
  if (q.type == M2C_EOS_MG) return wave_mg<KEPT>(q, K, p, w);
  if (q.type == M2C_EOS_NASG) return wave_nasg(q, K, p, w);
  return wave_jwl(q, K, p, w);
}

// Density behind the wave w evaluated at p, and its slope d rho*/dp.
template <bool KEPT>
__device__ inline void star_density(const EosDev& q, const Side& K, double p, const Wave& w, double& rs, double& drs) {
  if (q.type != M2C_EOS_SG) {
    rs = w.a;
    drs = w.b;
  } else if (KEPT) {
    const double gm = q.gm, pb = p + q.pc, r = pb / K.pb;
    if (p > K.p) {
      rs = K.rho * (r + gm) / (gm * r + 1.0);
      drs = K.rho * (1.0 - gm * gm) / ((gm * r + 1.0) * (gm * r + 1.0) * K.pb);
    } else {
      rs = K.rho * pow(r, q.inv_g);
      drs = rs / (q.g * pb);
    }
  } else if (p > K.p) {
    const double r = (p + q.pc) * K.ipb, id = rcp_nr(fma(q.gm, r, 1.0));
    rs = K.rho * (r + q.gm) * id;
    drs = K.rho * fma(-q.gm, q.gm, 1.0) * (id * id) * K.ipb;
  } else {
    // r^(1/g) = r/(r^((g-1)/(2g)))^2, r the IEEE quotient as in wave_sg: at p = p_K the
    // density is the side's own to the bit (a contact stays one)
    const double pb = p + q.pc, r0 = pb * K.ipb, r = fma(fma(-K.pb, r0, pb), K.ipb, r0);
    rs = K.rho * r * rcp_nr(w.a * w.a);
    drs = rs * q.inv_g * rcp_nr(pb);
  }
}

// F(p) = f_L + f_R + (u_R - u_L) of the bisection and the vacuum test.
template <bool KEPT>
static __device__ __noinline__ int riemann_F(const EosDev& qL, Side& L, const EosDev& qR, Side& Rs, double p, double& F) {
  Wave wL, wR;
  int st = wave<KEPT>(qL, L, p, wL);
  if (!st) st = wave<KEPT>(qR, Rs, p, wR);
  if (!st) F = wL.f + wR.f + (Rs.u - L.u);
  return st;
}

// Whether the MG isentrope of a side was evaluated at p on nodes beyond its span bound.
__device__ inline bool on_nodes_beyond(const Side& K, double p) {
  const double dp = __dsub_rn(K.p, p);
  return K.nrk > 1 && dp >= K.dspan && dp < K.dreach;
}

struct RiemannOut {
  double p, u, rhoL, rhoR;
};

// A problem whose Newton iteration ran out of steps: the vacuum test, then
// bisection for p* (iters counts its steps too). Then, and for a converged
// problem with a slope that is not finite, the star state from an evaluation at p.
template <bool KEPT>
static __device__ __noinline__ int riemann_finish(const EosDev& qL, Side& L, const EosDev& qR, Side& Rs, double plow,
                                                  bool vacuum_test, bool conv, double p, RiemannOut& out, int& iters) {
  int st;
  double F;
  if (!conv) {
    ++iters;
    if (vacuum_test) {
      st = riemann_F<KEPT>(qL, L, qR, Rs, plow, F);
      if (st) return st;
      if (F >= 0.0) return M2C_EVACUUM;
    }
    double a = plow, b = fmax(L.p, Rs.p);
    if (!isfinite(a)) {
      a = fmin(L.p, Rs.p);
      for (int k = 0; k < kBisectCap; ++k) {
        st = riemann_F<KEPT>(qL, L, qR, Rs, a, F);
        if (st) return st;
        if (F < 0.0) break;
        a = a - 2.0 * fabs(a) - 1.0;
      }
    }
    for (int k = 0; k < kBisectCap; ++k) {
      st = riemann_F<KEPT>(qL, L, qR, Rs, b, F);
      if (st) return st;
      if (F > 0.0) break;
      b = 2.0 * b + fabs(b) + 1.0;
    }
    bool ok = false;
    for (int k = 0; k < kBisectCap; ++k) {
      double m = 0.5 * (a + b);
      st = riemann_F<KEPT>(qL, L, qR, Rs, m, F);
      if (st) return st;
      if (F < 0.0) a = m; else b = m;
      ++iters;
      if (b - a <= 1e-14 * fmax(fabs(a), fabs(b))) { ok = true; break; }
    }
    if (!ok) return M2C_ENOCONV;
    p = 0.5 * (a + b);
  }
  Wave wL, wR;
  double d;
  st = wave<KEPT>(qL, L, p, wL);
  if (!st) st = wave<KEPT>(qR, Rs, p, wR);
  if (st) return st;
  out.p = p;
  out.u = 0.5 * (L.u + Rs.u) + 0.5 * (wR.f - wL.f);
  star_density<KEPT>(qL, L, p, wL, out.rhoL, d);
  star_density<KEPT>(qR, Rs, p, wR, out.rhoR, d);
  return M2C_OK;
}

// One side in the FP32 start below: a stiffened gas, or an MG material taken as one
// with the exponent n = 4 s - 1 of its isentrope near the reference state and the
// side's sound speed.
struct GuessSide {
  float rho, p, c, n, pb;
};
__device__ inline GuessSide guess_side(const EosDev& q, const Side& K) {
  const float rho = d2f(K.rho), c = d2f(K.c);
  const bool sg = q.type == M2C_EOS_SG;
  const float n = sg ? d2f(q.g) : fmaf(4.0f, d2f(q.s), -1.0f);
  return {rho, d2f(K.p), c, n, sg ? d2f(K.pb) : __fdividef(rho * c * c, n)};
}
__device__ inline void guess_wave(const GuessSide& K, float p, float& f, float& df) {
  const float dp = p - K.p, m = __fdividef(K.n - 1.0f, K.n + 1.0f);
  if (dp > 0.0f) {
    const float id = __fdividef(1.0f, fmaf(1.0f + m, K.pb, dp)), sq = sqrtf((1.0f - m) * __fdividef(id, K.rho));
    f = dp * sq;
    df = sq * fmaf(-0.5f * dp, id, 1.0f);
  } else {
    const float r = fmaxf(1.0f + __fdividef(dp, K.pb), 1e-6f);
    const float w = __powf(r, __fdividef(0.5f * (K.n - 1.0f), K.n));
    f = __fdividef(2.0f * K.c, K.n - 1.0f) * (w - 1.0f);
    df = __fdividef(w, r * K.rho * K.c);
  }
}

// Start of the Newton iteration of a face without a previous star pressure: p* to
// a few per cent from eight FP32 Newton steps on closed-form curves, from the
// acoustic pressure p_ac. NaN where that fails. The PVRS estimate is far off p*
// when the sides' impedances differ (water against air) and takes 13
// iterations, three of them over the whole isentrope; one such face held up its
// launch (1.51 against 0.59 ms in the late shock-bubble, 131x67x45, before mixed grids
// went back to the kept arithmetic; FP64 grids take it).
static __device__ __noinline__ double start_guess(const EosDev& qL, const Side& L, const EosDev& qR, const Side& Rs,
                                                  double plow, double pac) {
  if ((qL.type != M2C_EOS_SG && qL.type != M2C_EOS_MG) || (qR.type != M2C_EOS_SG && qR.type != M2C_EOS_MG)) return NAN;
  const GuessSide gl = guess_side(qL, L), gr = guess_side(qR, Rs);
  const float du = d2f(Rs.u - L.u), low = d2f(fmax(plow, -1e30));
  float p = fmaxf(d2f(pac), fmaf(1e-3f, fminf(gl.p, gr.p) - low, low));
  for (int k = 0; k < 8; ++k) {
    float fl, dl, fr, dr;
    guess_wave(gl, p, fl, dl);
    guess_wave(gr, p, fr, dr);
    const float pn = p - __fdividef(fl + fr + du, dl + dr);
    p = pn > low ? pn : fmaf(0.5f, p - low, low);
  }
  return p > low && p < INFINITY ? f2d(p) : (double)NAN;
}

// Solves the 1D problem between (rho, u, p) states; returns a status and the
// Newton/bisection iteration count. p_start: a start of the Newton iteration
// (the FIVER kernel passes the same face's star pressure of its previous
// solve); NaN, or a value not above the lowest admissible pressure, takes the
// PVRS estimate, or, with `guess`, start_guess() where the PVRS estimate and the
// acoustic pressure differ by more than 5 %. The root and the stopping rule do
// not depend on the start. resolution: of a pressure, in units of rho c^2 (used where a
// shock is too weak to resolve): the last bit of 64, which is what a curve resolves; on
// mixed grids the binary32 unit 2^-24 of the strains that their pressures come from.
template <bool KEPT>
static __device__ __noinline__ int riemann_solve(const EosDev& qL, double rl, double ul, double pl, const EosDev& qR, double rr,
                                    double ur, double pr, RiemannOut& out, int& iters,
                                    double p_start = NAN, bool guess = false, double resolution = 0x1p-52) {
  Side L, Rs;
  iters = 0;
  if (!make_side<KEPT>(qL, rl, ul, pl, L) || !make_side<KEPT>(qR, rr, ur, pr, Rs)) return M2C_ENONPHYS;
  const double plow = fmax(eos_plow(qL), eos_plow(qR));
  const double pac = fix_substeps(qL, L, qR, Rs, plow);
  int st = M2C_OK;
  // vacuum test (F(p_low) >= 0); both wave curves increase with p and vanish at
  // their side's pressure, so F(p_low) <= u_R - u_L and the test is only made
  // when u_R - u_L >= 0; no vacuum test with a JWL side (its rarefaction needs
  // p > 0). F increases with p, so a root above p_low found by the Newton
  // iteration implies F(p_low) < 0: the test is made only when the iteration
  // does not converge (before the bisection), which spares each converged
  // problem an evaluation of its curves down to p_low
  const bool vacuum_test = isfinite(plow) && Rs.u - L.u >= 0.0 && qL.type != M2C_EOS_JWL && qR.type != M2C_EOS_JWL;
  double p = 0.5 * (L.p + Rs.p) - 0.125 * (Rs.u - L.u) * (L.rho + Rs.rho) * (L.c + Rs.c);
  const bool warm = p_start > plow && p_start < INFINITY;
  if (warm) {
    p = p_start;
  } else if (!KEPT && guess && !(fabs(p - pac) <= 0.05 * fabs(pac))) {
    const double pg = start_guess(qL, L, qR, Rs, plow, pac);
    if (pg > plow) p = pg;
  }
  if (!(p > plow)) {
    double gap = fmin(L.p, Rs.p) - plow;
    if (!(gap > 0.0)) gap = fmax(L.p, Rs.p) - plow;
    p = plow + 1e-3 * gap;
  }
  if constexpr (!KEPT) {
    L.dreach = L.dspan + L.dnode;
    Rs.dreach = Rs.dspan + Rs.dnode;
  }
  // the solution follows from the last evaluation to first order in its step (at
  // most the tolerance: the error is of the order of its square) instead of from
  // one more evaluation
  Wave wL{}, wR{};
  double p_last = p;
  bool conv = false, more = true;
  int it = 0, counted = 0;
  while (more) {
    ++it;
    st = wave<KEPT>(qL, L, p, wL);
    const int sr = wave<KEPT>(qR, Rs, p, wR);
    if (!st) st = sr;
    const double F = wL.f + wR.f + (Rs.u - L.u), dF = wL.df + wR.df;
    double pn = p - (KEPT ? F / dF : div_nr(F, dF));
    if (isinf(dF)) {
      // an iterate a few units above a side's pressure: its shock is too weak to resolve, and
      // the slope of its curve infinite. The step F/F' = 0 says nothing then: the step with
      // that side's acoustic curve tells whether p is the root (a face at rest that starts
      // from its own pressure; to the tolerance, or to the resolution times rho c^2) or only a
      // start next to a side's pressure
      const bool iL = isinf(wL.df), iR = isinf(wR.df);
      const double dL = iL ? 1.0 / (L.rho * L.c) : wL.df, dR = iR ? 1.0 / (Rs.rho * Rs.c) : wR.df;
      const double fL = iL ? (p - L.p) * dL : wL.f, fR = iR ? (p - Rs.p) * dR : wR.f;
      const double pa = p - (fL + fR + (Rs.u - L.u)) / (dL + dR);
      const double res = resolution * fmax(iL ? L.rho * L.c * L.c : 0.0, iR ? Rs.rho * Rs.c * Rs.c : 0.0);
      if (!(fabs(pa - p) <= fmax(kNewtonTol * fabs(pa), res))) pn = pa;
    }
    if (!(pn > plow)) pn = 0.5 * (p + plow);
    conv = !st && fabs(pn - p) <= kNewtonTol * fabs(pn);
    if constexpr (!KEPT) {
      // a root found on nodes beyond a side's bound: on with the equal substeps (a step or
      // two within 1e-8 of p, which the count leaves out: the oracle takes them from the start)
      if (conv && (on_nodes_beyond(L, p) || on_nodes_beyond(Rs, p))) {
        L.dreach = L.dspan;
        Rs.dreach = Rs.dspan;
        conv = false;
        counted = it;
      }
    }
    p_last = p;
    p = pn;
    more = !st && !conv && it < kNewtonCap;
  }
  L.dreach = L.dspan;
  Rs.dreach = Rs.dspan;
  if (st) return st;
  if (conv && isfinite(wL.df) && isfinite(wR.df)) {
    double rL, dL, rR, dR;
    star_density<KEPT>(qL, L, p_last, wL, rL, dL);
    star_density<KEPT>(qR, Rs, p_last, wR, rR, dR);
    if (isfinite(dL) && isfinite(dR)) {
      const double d = p - p_last;
      out.p = p;
      out.u = 0.5 * (L.u + Rs.u) + 0.5 * (wR.f - wL.f) + 0.5 * (wR.df - wL.df) * d;
      out.rhoL = rL + dL * d;
      out.rhoR = rR + dR * d;
      iters = counted ? counted : it;
      return M2C_OK;
    }
  }
  return riemann_finish<KEPT>(qL, L, qR, Rs, plow, vacuum_test, conv, p, out, iters = it);
}

// ---------------------------------------------------------------------------
// Mixed-precision exact Riemann solve: Newton on p* first runs on FP32 wave
// curves (the same PVRS start and curves, with FP32 tolerances; weak waves of
// a stiff MG material, |p - p_K| <= 1e-5 rho_K c_K^2, take the acoustic
// curve, which is all an FP32 start can resolve there), then one FP64 Newton
// step from the FP32 root on the FP64 wave curves (two if the first moves p by
// more than 1e-9 |p|) gives p*; u* and the star densities follow from the last
// FP64 evaluation to first order in the step. An FP32 failure, a vacuum
// signal, a slope that is not finite, or a step larger than 1e-5 |p| leaves
// the problem to the FP64 iteration above.
// ---------------------------------------------------------------------------
struct SideF {
  float rho, u, p, c, e;
};

__device__ inline bool make_side_f(const EosP<float>& q, float rho, float u, float p, SideF& K) {
  if (!(rho > 0.0f)) return false;
  float e, c2;
  if (!eos_e_c2<float>(q, rho, 1.0f / rho, p, e, c2)) return false;
  K.rho = rho;
  K.u = u;
  K.p = p;
  K.c = sqrtf(c2);
  K.e = e;
  return true;
}

__device__ inline float eos_plow_f(const EosP<float>& q) {
  if (q.type == M2C_EOS_SG) return -q.pc;
  return isfinite(q.eta_min) ? q.pmin : -INFINITY;
}

__device__ inline bool wave_sg_f(const EosP<float>& q, const SideF& K, float p, float& f, float& df) {
  const float g = q.g, pb = p + q.pc, pbK = K.p + q.pc, dp = p - K.p;
  if (!(pb >= 0.0f) || !(pbK > 0.0f)) return false;
  if (p > K.p) {
    const float A = 2.0f / ((g + 1.0f) * K.rho);
    const float B = (g - 1.0f) / (g + 1.0f) * pbK;
    const float sq = sqrtf(A / (pb + B));
    f = dp * sq;
    df = sq * (1.0f - 0.5f * dp / (pb + B));
  } else {
    // (pb/pbK)^a - 1 as expm1(a log1p(dp/pbK)): no cancellation for weak waves
    const float x = dp / pbK;
    const float qm1 = expm1f((g - 1.0f) / (2.0f * g) * log1pf(x));
    f = 2.0f * K.c / (g - 1.0f) * qm1;
    df = (1.0f + qm1) / ((1.0f + x) * K.rho * K.c);
  }
  return true;
}

__device__ inline bool mg_hugoniot_f(const EosP<float>& q, const SideF& K, float p, float& rho_out, float& drdp) {
  float lo = K.rho, hi = q.rho0 * q.s / (q.s - 1.0f);
  if (!(hi > lo)) return false;
  float rho = K.rho + (p - K.p) / (K.c * K.c);
  if (!(rho > lo && rho < hi)) rho = 0.5f * (lo + hi);
  for (int it = 0; it < 40; ++it) {
    const float eta = 1.0f - q.rho0 / rho;
    if (!(eta < q.eta_max)) return false;
    float pR, dpR, eR, deR;
    mg_ref<float>(q, eta, pR, dpR, eR, deR);
    const float e = eR + (p - pR) * q.inv_rg;
    const float ir2 = 1.0f / (rho * rho);
    const float dedr = (deR - dpR * q.inv_rg) * q.rho0 * ir2;
    const float H = e - K.e - 0.5f * (p + K.p) * (1.0f / K.rho - 1.0f / rho);
    const float dH = dedr - 0.5f * (p + K.p) * ir2;
    if (H > 0.0f) lo = rho; else hi = rho;
    float rn = rho - H / dH;
    if (!(rn >= lo && rn <= hi)) rn = 0.5f * (lo + hi);
    const bool conv = fabsf(rn - rho) <= 1e-6f * rn;
    rho = rn;
    if (conv) {
      const float ir = 1.0f / rho;
      mg_ref<float>(q, 1.0f - q.rho0 * ir, pR, dpR, eR, deR);
      const float dedn = (deR - dpR * q.inv_rg) * q.rho0 * ir * ir;
      const float Hp = q.inv_rg - 0.5f * (1.0f / K.rho - ir);
      const float Hr = dedn - 0.5f * (p + K.p) * ir * ir;
      rho_out = rho;
      drdp = -Hp / Hr;
      return true;
    }
  }
  return false;
}

__device__ inline bool mg_rhs_f(const EosP<float>& q, float p, float rho, float& drho, float& dfv) {
  float e, c2;
  if (!eos_e_c2<float>(q, rho, 1.0f / rho, p, e, c2)) return false;
  drho = 1.0f / c2;
  dfv = 1.0f / (rho * sqrtf(c2));
  return true;
}

__device__ inline bool wave_mg_f(const EosP<float>& q, const SideF& K, float p, float& f, float& df) {
  const float dp = p - K.p, z = K.rho * K.c;
  if (fabsf(dp) <= 1e-5f * z * K.c) {  // acoustic start for rounding-level waves
    f = dp / z;
    df = 1.0f / z;
    return true;
  }
  if (p > K.p) {
    float rho, drdp;
    if (!mg_hugoniot_f(q, K, p, rho, drdp)) return false;
    const float dv = 1.0f / K.rho - 1.0f / rho;
    const float fv = sqrtf(dp * dv);
    if (!(fv > 0.0f)) return false;
    f = fv;
    df = (dv + dp * drdp / (rho * rho)) / (2.0f * fv);
    return true;
  }
  float nsd = ceilf((float)kRk4Steps * fabsf(dp) / q.rk4_span);
  nsd = nsd >= 1.0f ? (nsd > (float)kRk4Steps ? (float)kRk4Steps : nsd) : 1.0f;
  const int ns = (int)nsd;
  const float hs = dp / (float)ns;
  float rho = K.rho, fv = 0.0f;
  for (int i = 0; i < ns; ++i) {
    const float pi = K.p + (float)i * hs;
    float k1r, k1f, k2r, k2f, k3r, k3f, k4r, k4f;
    if (!mg_rhs_f(q, pi, rho, k1r, k1f) || !mg_rhs_f(q, pi + 0.5f * hs, rho + 0.5f * hs * k1r, k2r, k2f) ||
        !mg_rhs_f(q, pi + 0.5f * hs, rho + 0.5f * hs * k2r, k3r, k3f) ||
        !mg_rhs_f(q, pi + hs, rho + hs * k3r, k4r, k4f))
      return false;
    rho = rho + hs / 6.0f * (k1r + 2.0f * k2r + 2.0f * k3r + k4r);
    fv = fv + hs / 6.0f * (k1f + 2.0f * k2f + 2.0f * k3f + k4f);
  }
  float e, c2;
  if (!eos_e_c2<float>(q, rho, 1.0f / rho, p, e, c2)) return false;
  f = fv;
  df = 1.0f / (rho * sqrtf(c2));
  return true;
}

// F(p) = f_L + f_R + (u_R - u_L) and its slope on the FP32 curves; false if a
// curve is undefined at p or F is not finite (the caller checks the slope).
__device__ inline bool riemann_F_f(const EosP<float>& qL, const SideF& L, const EosP<float>& qR, const SideF& Rs,
                                   float p, float& F, float& dF) {
  float fL, dfL, fR, dfR;
  const bool okL = qL.type == M2C_EOS_SG ? wave_sg_f(qL, L, p, fL, dfL) : wave_mg_f(qL, L, p, fL, dfL);
  if (!okL) return false;
  const bool okR = qR.type == M2C_EOS_SG ? wave_sg_f(qR, Rs, p, fR, dfR) : wave_mg_f(qR, Rs, p, fR, dfR);
  if (!okR) return false;
  F = fL + fR + (Rs.u - L.u);
  dF = dfL + dfR;
  return isfinite(F);
}

// FP32 Newton on p* from the PVRS guess; false if it fails, ends within 1e-4
// of the lowest admissible pressure (where a vacuum would take it) or does not
// reach |dp| <= 1e-5 |p| in 30 steps.
static __device__ __noinline__ bool riemann_newton_f(const EosP<float>& qL, float rl, float ul, float pl, const EosP<float>& qR,
                                        float rr, float ur, float pr, float& p_out, int& iters,
                                        float p_start) {
  // FP32 wave curves exist for the stiffened gas and Mie-Grueneisen only
  if ((qL.type != M2C_EOS_SG && qL.type != M2C_EOS_MG) || (qR.type != M2C_EOS_SG && qR.type != M2C_EOS_MG))
    return false;
  SideF L, Rs;
  if (!make_side_f(qL, rl, ul, pl, L) || !make_side_f(qR, rr, ur, pr, Rs)) return false;
  const float plow = fmaxf(eos_plow_f(qL), eos_plow_f(qR));
  float F, dF;
  // no vacuum test here (as in the FP64 solve, a root above p_low rules a vacuum
  // out): with a vacuum the iterates only approach p_low, so a "root" within
  // 1e-4 of p_low is rejected and the problem left to the FP64 solve
  float p = 0.5f * (L.p + Rs.p) - 0.125f * (Rs.u - L.u) * (L.rho + Rs.rho) * (L.c + Rs.c);
  if (p_start > plow && p_start < INFINITY) p = p_start;
  if (!(p > plow)) {
    float gap = fminf(L.p, Rs.p) - plow;
    if (!(gap > 0.0f)) gap = fmaxf(L.p, Rs.p) - plow;
    p = plow + 1e-3f * gap;
  }
  for (int it = 1; it <= 30; ++it) {
    if (!riemann_F_f(qL, L, qR, Rs, p, F, dF) || !(dF > 0.0f)) return false;
    float pn = p - F / dF;
    if (!(pn > plow)) pn = 0.5f * (p + plow);
    const bool small = fabsf(pn - p) <= 1e-5f * fabsf(pn);
    p = pn;
    if (small) {
      if (isfinite(plow) && !(p - plow > 1e-4f * fabsf(p))) return false;
      p_out = p;
      iters = it;
      return true;
    }
  }
  return false;
}

template <bool KEPT>
static __device__ __noinline__ int riemann_solve_mixed(const EosP<float>& qLf, const EosDev& qL, double rl, double ul, double pl,
                                          const EosP<float>& qRf, const EosDev& qR, double rr, double ur, double pr,
                                          RiemannOut& out, int& iters,
                                          double p_start = NAN, double resolution = 0x1p-52) {
  float p32;
  int it32 = 0;
  Side L, Rs;
  if (riemann_newton_f(qLf, d2f(rl), d2f(ul), d2f(pl), qRf, d2f(rr), d2f(ur), d2f(pr), p32, it32, (float)p_start) &&
      make_side<KEPT>(qL, rl, ul, pl, L) && make_side<KEPT>(qR, rr, ur, pr, Rs)) {
    const double plow = fmax(eos_plow(qL), eos_plow(qR));
    fix_substeps(qL, L, qR, Rs, plow);
    double p = f2d(p32);
    for (int k = 0; k < 2; ++k) {
      Wave wL, wR;
      double rL, dL, rR, dR;
      if (!(p > plow) || wave<KEPT>(qL, L, p, wL) || wave<KEPT>(qR, Rs, p, wR)) break;
      star_density<KEPT>(qL, L, p, wL, rL, dL);
      star_density<KEPT>(qR, Rs, p, wR, rR, dR);
      const double F = wL.f + wR.f + (Rs.u - L.u), dF = wL.df + wR.df;
      const double dp = -F / dF;
      // a slope that is not finite (a wave of rounding-level strength on a
      // shock curve) leaves the problem to the FP64 iteration
      if (!(isfinite(dF) && dF > 0.0 && isfinite(dL) && isfinite(dR) && fabs(dp) <= 1e-5 * fabs(p) &&
            p + dp > plow))
        break;
      if (k == 1 || fabs(dp) <= 1e-9 * fabs(p)) {
        out.p = p + dp;
        out.u = 0.5 * (L.u + Rs.u) + 0.5 * (wR.f - wL.f) + 0.5 * (wR.df - wL.df) * dp;
        out.rhoL = rL + dL * dp;
        out.rhoR = rR + dR * dp;
        iters = it32 + 1 + k;
        return M2C_OK;
      }
      p += dp;
    }
  }
  return riemann_solve<KEPT>(qL, rl, ul, pl, qR, rr, ur, pr, out, iters, p_start, false, resolution);
}

}  // namespace m2c
