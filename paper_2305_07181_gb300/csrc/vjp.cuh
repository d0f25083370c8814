// Reverse mode (vector-Jacobian product) of the entropy-split residual with
// EC SATs and matrix interface dissipation: grad = (d dudt / d u)^T cot.
//
// The residual of element k at node m is
//   r_m = sum_i (M_i f_i)_m - 1/(beta+1) sum_i A~_i(u_m) (D_i w)_m + sat_m,
// with f_i, w pointwise in u and sat_m = -G(u_km, u_vn)/H_km for the facet
// node pair (k, m) ~ (v, n) (and +G/H_vn on the other side).  Its transpose:
//   gbar_i   = -1/(beta+1) A~_i(u_m) cot_m          (A~_i symmetric, Sec. 2.4)
//   fbar_i   = M_i^T cot,   wbar = sum_i D_i^T gbar_i           (per element)
//   grad_m   = sum_i (df_i/du)^T fbar_i + (dw/du)^T wbar
//              - 1/(beta+1) d/du [cot_m . sum_i A~_i(u) g_i]|_(g_i = (D_i w)_m)
//              + facet part (dG/du)^T (-cot_km/H_km + cot_vn/H_vn).
// The pointwise derivatives are exact: the facet terms by a hand-written
// reverse sweep at the values, the volume's pointwise part with closed-form
// products and one dual direction (dual.cuh; see split_vjp_kernel).  The
// contractions apply the forward operators: D_i^T y = E_i (y/H) - H D_i (y/H)
// (Def. 1), on the tensor cores as the residual's (tc64.cuh).  Float64
// throughout.
// Included by vjp.cu, the reverse mode's own translation unit with its own
// copy of the constant-memory operator tables.
#pragma once

namespace esplit {

__device__ __forceinline__ double sgn0(double x) { return x > 0.0 ? 1.0 : (x < 0.0 ? -1.0 : 0.0); }

// exp_avg (Eq. (47)) and its partial derivatives at the values:
// E = (ar - br)/(r (a - b)) or ar ia g(eps), eps = (b - a) ia, with the series
// g and g' in fixed point (terms 0 to 6; the rest in float32) as exp_avg_pair
struct ExpAvgD {
  double E, Ea, Eb, Ear, Ebr, Eia;
};
__device__ __forceinline__ void exp_avg_d(double a, double b, double ar, double br, double r, double ia,
                                          const double* coef, const long long* s62, const float* tail, int ok,
                                          ExpAvgD& o) {
  const double df = b - a, eps = df * ia;
  if (!fm::abs_below(eps, 0x3FA999999999999AULL)) {  // 0.05
    const double id = rcp64(a - b), q = id / r;
    o.E = (ar - br) * q;
    o.Ear = q;
    o.Ebr = -q;
    o.Ea = -o.E * id;
    o.Eb = -o.Ea;
    o.Eia = 0.0;
    return;
  }
  double sv, dv;
  if (ok) {
    const long long x = im::small_to_fixed(eps);
    const float xf = __int2float_rn((int)(x >> 32)) * 0x1p-34f;
    float t = tail[5], td = 0.0f;
#pragma unroll
    for (int k = 4; k >= 0; --k) {
      td = td * xf + t;
      t = t * xf + tail[k];
    }
    long long s = (long long)__float2int_rn(t * 0x1p30f) << 32, d = (long long)__float2int_rn(td * 0x1p28f) << 34;
#pragma unroll
    for (int k = 6; k >= 0; --k) {
      d = im::horner62(d, x, s);
      s = im::horner62(s, x, s62[k]);
    }
    sv = im::unit62_to_double(s);
    // g'(0) = (r - 1)/2 < 0 and stays negative below the switch
    dv = -im::unit62_to_double(-d);
  } else {
    sv = coef[ExpAvgCfg<double>::NTERMS - 1];
    dv = 0.0;
#pragma unroll
    for (int k = ExpAvgCfg<double>::NTERMS - 2; k >= 0; --k) {
      dv = dv * eps + sv;
      sv = sv * eps + coef[k];
    }
  }
  o.Ear = ia * sv;
  o.Ebr = 0.0;
  o.E = ar * o.Ear;
  const double w = ar * ia * dv;
  o.Eb = w * ia;
  o.Ea = -o.Eb;
  o.Eia = ar * sv + w * df;
}

// The pair's averages, the derivatives of its exponential averages, and the
// reciprocals the reverse sweep multiplies by instead of dividing
template <int D>
struct PairRev {
  PairAvg<double, D> a;
  ExpAvgD e1, e2;  // E1 (of p), E2 (of q)
  double iA1, iE1, iE2, iz;
};

template <int D, typename C>
__device__ __forceinline__ void pair_rev_prep(const ZNode<double, D>& k, const ZNode<double, D>& v, const C& c,
                                              PairRev<D>& p) {
  exp_avg_d(k.p, v.p, k.P2, v.P2, c.r2, k.ip, c.ser2, c.s2, c.t2, c.im_ok, p.e1);
  exp_avg_d(k.q, v.q, k.P1, v.P1, c.r1, k.iq, c.ser1, c.s1, c.t1, c.im_ok, p.e2);
  p.a.A1 = 0.5 * (k.P1 + v.P1);
  p.a.E1 = p.e1.E;
  p.a.A2 = 0.5 * (k.P2 + v.P2);
  p.a.E2 = p.e2.E;
  p.a.z1a = 0.5 * (k.q + v.q);
  p.a.pa = 0.5 * (k.p + v.p);
  p.a.ke = 0.0;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    p.a.qV[i] = 0.5 * (k.q * k.V[i] + v.q * v.V[i]);
    p.a.Va[i] = 0.5 * (k.V[i] + v.V[i]);
    p.a.ke += 0.5 * k.V[i] * v.V[i];
  }
  p.iA1 = rcp64(p.a.A1);
  p.iE1 = rcp64(p.a.E1);
  p.iE2 = rcp64(p.a.E2);
  p.iz = rcp64(p.a.z1a);
}

// Adjoints of the nodal quantities of both sides (ZNode fields) for
//   s = gb . [sum_i nu_i F*_i(k, v) + (|nu|/2) X^|L|S^X^T dw]   (dw held fixed),
// the reverse sweep of pair_avg, sy_flux_dir and the dissipation's hat state
// and columns in plain float64.  With r_k the columns of X^ and l_k =
// |lambda_k| S_k, the dissipation part is (|nu|/2) sum_k l_k (r_k.gb)(r_k.dw):
// column adjoints (|nu|/2) l_k ((r_k.dw) gb + (r_k.gb) dw), weight adjoints
// (|nu|/2) (r_k.gb)(r_k.dw).
template <int D, typename C>
__device__ __forceinline__ void pair_reverse(const ZNode<double, D>& k, const ZNode<double, D>& v,
                                             const PairRev<D>& pr, const C& c, const double* nu, int dissipation, double b, const double* n,
                                             const double* gb, const double* dw, ZNode<double, D>& kb,
                                             ZNode<double, D>& vb) {
  constexpr int NC = D + 2;
  const PairAvg<double, D>& a = pr.a;
  const double iden = pr.iA1 * pr.iE1;  // 1/(A1 E1)
  double A1b = 0.0, E1b = 0.0, A2b = 0.0, E2b = 0.0, z1ab = 0.0, pab = 0.0, keb = 0.0;
  double qVb[D], Vab[D];
#pragma unroll
  for (int i = 0; i < D; ++i) qVb[i] = Vab[i] = 0.0;
  // ---- two-point flux: s_f = mn C + pa (gb_m . nu)
  {
    double mq = 0.0;
#pragma unroll
    for (int i = 0; i < D; ++i) mq += nu[i] * a.qV[i];
    const double mn = mq * iden;
    const double h = c.gam_gm1 * a.A2 * a.E2 + a.ke;
    double Cc = gb[0] + gb[NC - 1] * h, gmn = 0.0;
#pragma unroll
    for (int j = 0; j < D; ++j) {
      Cc += gb[1 + j] * a.Va[j];
      gmn += gb[1 + j] * nu[j];
    }
    const double mnb = Cc, hb = mn * gb[NC - 1];
#pragma unroll
    for (int j = 0; j < D; ++j) Vab[j] += mn * gb[1 + j];
    pab += gmn;
    const double mqb = mnb * iden, idenb = mnb * mq;
#pragma unroll
    for (int i = 0; i < D; ++i) qVb[i] += mqb * nu[i];
    A1b -= idenb * iden * pr.iA1;
    E1b -= idenb * iden * pr.iE1;
    A2b += hb * c.gam_gm1 * a.E2;
    E2b += hb * c.gam_gm1 * a.A2;
    keb += hb;
  }
  // ---- dissipation's averages part
  if (dissipation) {
    const double iz = pr.iz, rho_h = a.z1a * iden, irho = a.A1 * a.E1 * iz;
    double Vh[D], vh2 = 0.0, vn = 0.0;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      Vh[i] = a.qV[i] * iz;
      vh2 += Vh[i] * Vh[i];
      vn += Vh[i] * n[i];
    }
    const double p_h = a.pa;
    const double ip_h = rcp64(p_h);
    const double theta = rho_h * iden * ip_h;
    const double eta = iz * pr.iE2 * pr.iE1;
    const double a2 = c.gam * p_h * irho, ah = a2 * rsqrt64(a2);
    const double Hh = ah * ah * c.inv_gm1 + 0.5 * vh2;
    double Vhb[D];
#pragma unroll
    for (int i = 0; i < D; ++i) Vhb[i] = 0.0;
    double vnb = 0.0, ahb = 0.0, Hhb = 0.0, vh2b = 0.0, thetab = 0.0, etab = 0.0;
    const double hb2 = 0.5 * b;
#pragma unroll
    for (int kk = 0; kk < NC; ++kk) {
      double col[NC];
      double l;
      const bool ac = (kk == 0 || kk == NC - 1);
      const double sg = (kk == 0) ? -1.0 : 1.0;
      if (ac) {
        col[0] = 1.0;
#pragma unroll
        for (int i = 0; i < D; ++i) col[1 + i] = Vh[i] + sg * ah * n[i];
        col[NC - 1] = Hh + sg * ah * vn;
        l = fabs(vn + sg * ah) * c.s_ac * theta;
      } else if (kk == 1) {
        col[0] = 1.0;
#pragma unroll
        for (int i = 0; i < D; ++i) col[1 + i] = Vh[i];
        col[NC - 1] = 0.5 * vh2;
        l = fabs(vn) * c.s_en * theta;
      } else {
#pragma unroll
        for (int r = 0; r < NC; ++r) col[r] = 0.0;
        if (kk == 2) {
          col[1] = n[1];
          col[2] = -n[0];
          col[NC - 1] = Vh[0] * n[1] - Vh[1] * n[0];
        } else {
          col[1] = -n[D - 1];
          col[3] = n[0];
          col[NC - 1] = Vh[D - 1] * n[0] - Vh[0] * n[D - 1];
        }
        l = fabs(vn) * eta;
      }
      double al = 0.0, be = 0.0;
#pragma unroll
      for (int r = 0; r < NC; ++r) {
        al += col[r] * gb[r];
        be += col[r] * dw[r];
      }
      const double lb = hb2 * al * be;
      double cb[NC];
#pragma unroll
      for (int r = 0; r < NC; ++r) cb[r] = hb2 * l * (be * gb[r] + al * dw[r]);
      if (ac) {
        double cn = 0.0;
#pragma unroll
        for (int i = 0; i < D; ++i) {
          Vhb[i] += cb[1 + i];
          cn += cb[1 + i] * n[i];
        }
        ahb += sg * cn + sg * cb[NC - 1] * vn;
        Hhb += cb[NC - 1];
        vnb += sg * cb[NC - 1] * ah;
        const double t = vn + sg * ah;
        const double w = lb * c.s_ac;
        vnb += w * sgn0(t) * theta;
        ahb += w * sgn0(t) * sg * theta;
        thetab += w * fabs(t);
      } else if (kk == 1) {
#pragma unroll
        for (int i = 0; i < D; ++i) Vhb[i] += cb[1 + i];
        vh2b += 0.5 * cb[NC - 1];
        vnb += lb * sgn0(vn) * c.s_en * theta;
        thetab += lb * fabs(vn) * c.s_en;
      } else {
        if (kk == 2) {
          Vhb[0] += cb[NC - 1] * n[1];
          Vhb[1] -= cb[NC - 1] * n[0];
        } else {
          Vhb[D - 1] += cb[NC - 1] * n[0];
          Vhb[0] -= cb[NC - 1] * n[D - 1];
        }
        vnb += lb * sgn0(vn) * eta;
        etab += lb * fabs(vn);
      }
    }
    // hat state back to the averages
    ahb += Hhb * 2.0 * ah * c.inv_gm1;
    vh2b += 0.5 * Hhb;
#pragma unroll
    for (int i = 0; i < D; ++i) Vhb[i] += 2.0 * vh2b * Vh[i] + vnb * n[i];
    const double ah2 = 0.5 * ahb * ah, et = etab * eta, th = thetab * theta;
    const double p_hb = (ah2 - th) * ip_h;
    const double rho_hb = (th - ah2) * irho;
    const double rr = th + rho_hb * rho_h;
    z1ab -= et * iz;
    E2b -= et * pr.iE2;
    E1b -= (et + rr) * pr.iE1;
    A1b -= rr * pr.iA1;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      qVb[i] += Vhb[i] * iz;
      z1ab -= Vhb[i] * Vh[i] * iz;
    }
    z1ab += rho_hb * iden;
    pab += p_hb;
  }
  // ---- pair averages back to the nodal quantities
  kb.q = kb.p = kb.P1 = kb.P2 = kb.v2 = kb.iq = kb.ip = 0.0;
  vb.q = vb.p = vb.P1 = vb.P2 = vb.v2 = vb.iq = vb.ip = 0.0;
#pragma unroll
  for (int i = 0; i < D; ++i) kb.V[i] = vb.V[i] = 0.0;
  kb.P1 += 0.5 * A1b;
  vb.P1 += 0.5 * A1b;
  kb.P2 += 0.5 * A2b;
  vb.P2 += 0.5 * A2b;
  kb.q += 0.5 * z1ab;
  vb.q += 0.5 * z1ab;
  kb.p += 0.5 * pab;
  vb.p += 0.5 * pab;
  kb.v2 -= 0.25 * keb;
  vb.v2 -= 0.25 * keb;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    const double vab = Vab[i] + 2.0 * keb * a.Va[i];
    kb.V[i] += 0.5 * vab + 0.5 * qVb[i] * k.q;
    vb.V[i] += 0.5 * vab + 0.5 * qVb[i] * v.q;
    kb.q += 0.5 * qVb[i] * k.V[i];
    vb.q += 0.5 * qVb[i] * v.V[i];
  }
  kb.p += E1b * pr.e1.Ea;
  vb.p += E1b * pr.e1.Eb;
  kb.P2 += E1b * pr.e1.Ear;
  vb.P2 += E1b * pr.e1.Ebr;
  kb.ip += E1b * pr.e1.Eia;
  kb.q += E2b * pr.e2.Ea;
  vb.q += E2b * pr.e2.Eb;
  kb.P1 += E2b * pr.e2.Ear;
  vb.P1 += E2b * pr.e2.Ebr;
  kb.iq += E2b * pr.e2.Eia;
}

// Reverse of the nodal chain u -> (q, V, p, P1, P2, v2, 1/q, 1/p) at the
// values (ZNode adjoints zb -> state adjoint ub):
//   V = m/rho, v2 = |V|^2, p = (gam-1)(e - rho v2/2), q = rho^a_q p^b_q,
//   P1 = q^r1, P2 = p^r2.
template <int D, typename C>
__device__ __forceinline__ void node_chain_rev(const Node<double, D>& n, const ZNode<double, D>& z,
                                               const ZNode<double, D>& zb, const C& c, double iq, double ip,
                                               double* ub) {
  constexpr int NC = D + 2;
  const double qb = zb.q + zb.P1 * c.r1 * z.P1 * iq - zb.iq * iq * iq;
  const double pb = zb.p + zb.P2 * c.r2 * z.P2 * ip - zb.ip * ip * ip + qb * n.q * c.b_q * ip;
  double rhob = qb * n.q * c.a_q * n.ir - 0.5 * c.gm1 * n.v2 * pb;
  const double v2b = zb.v2 - 0.5 * c.gm1 * n.rho * pb;
  ub[NC - 1] = c.gm1 * pb;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    const double Vb = zb.V[j] + 2.0 * v2b * n.V[j];
    ub[1 + j] = Vb * n.ir;
    rhob -= Vb * n.V[j] * n.ir;
  }
  ub[0] = rhob;
}

// facet pairs: each thread writes the facet part of grad at its two slots.
// A reverse sweep at the values: the pair computation (averages, two-point
// flux, dissipation; pair_reverse), then each side's nodal chain
// (node_chain_rev); no dual numbers.
template <int D>
__global__ void __launch_bounds__(64) face_vjp_kernel(const double* __restrict__ u, const double* __restrict__ cot,
                                                      const int2* __restrict__ fp, int n_pairs,
                                                      const double* __restrict__ nu,
                                                      const double* __restrict__ ihd,
                                                      const double* __restrict__ nscale,
                                                      double* __restrict__ gsat, Phys<double> c, int dissipation) {
  constexpr int NC = D + 2;
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n_pairs) return;
  const int NP = c_ref.n_p, NS = c_ref.n_slot;
  int2 pr = __ldg(&fp[t]);
  int k = pr.x / NS, s = pr.x - k * NS;
  int v = pr.y / NS, s2 = pr.y - v * NS;
  int m = c_ref.slot_node[s], n = c_ref.slot_node[s2];
  double uk[NC], uv[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    uk[q] = __ldg(&u[((size_t)k * NC + q) * NP + m]);
    uv[q] = __ldg(&u[((size_t)v * NC + q) * NP + n]);
  }
  Node<double, D> nk, nv;
  node_from_u<double, D>(uk, c, nk);
  node_from_u<double, D>(uv, c, nv);
  ZNode<double, D> zk, zv;
  znode<double, D>(nk, c, zk);
  znode<double, D>(nv, c, zv);
  // 1/q and 1/p of each side by a reciprocal of its own: as products of one
  // reciprocal 1/(q p) they carry up to three more roundings into every term of
  // the nodal chains (relative error of the gradient with dissipation, 3,200
  // triangles p 1 / 1,296 tetrahedra p 1: 2.71e-15 / 2.46e-15 instead of 2.93e-15 /
  // 2.64e-15; by divisions 2.75e-15 / 2.45e-15)
  const double iqk = rcp64(nk.q), ipk = rcp64(nk.p), iqv = rcp64(nv.q), ipv = rcp64(nv.p);
  const JvpPrep<double> jk = jvp_prep_from<double, D>(nk, c, iqk, nk.rho * ipk);
  const JvpPrep<double> jv = jvp_prep_from<double, D>(nv, c, iqv, nv.rho * ipv);
  zk.iq = iqk;
  zk.ip = ipk;
  double nud[D], nh[D];
  const double* ns = nscale + (size_t)pr.x * (D + 1);  // |nu|, nu/|nu| of slot (k, s)
  const double b = __ldg(&ns[0]);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    nud[i] = __ldg(&nu[((size_t)k * NS + s) * D + i]);
    nh[i] = __ldg(&ns[1 + i]);
  }
  const double ihk = __ldg(&ihd[(size_t)k * NP + m]), ihv = __ldg(&ihd[(size_t)v * NP + n]);
  double gb[NC], dw[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    gb[q] = -__ldg(&cot[((size_t)k * NC + q) * NP + m]) * ihk + __ldg(&cot[((size_t)v * NC + q) * NP + n]) * ihv;
    dw[q] = nk.W[q] - nv.W[q];
  }
  // d[gb . G(u_k, u_v)]: the pair computation reversed at the values, then
  // each side's nodal chain; with dissipation also (M gb) . (dw_k - dw_v),
  // M = X^|L|S^X^T symmetric, through the symmetric dW/du of each side
  ZNode<double, D> kb, vb;
  PairRev<D> pv;
  pair_rev_prep<D>(zk, zv, c, pv);
  pair_reverse<D>(zk, zv, pv, c, nud, dissipation, b, nh, gb, dw, kb, vb);
  double gk[NC], gv[NC];
  node_chain_rev<D>(nk, zk, kb, c, iqk, ipk, gk);
  node_chain_rev<D>(nv, zv, vb, c, iqv, ipv, gv);
  if (dissipation) {
    PairSums<D> ps;
    ps.dn = 2.0 * pv.a.A1 * pv.a.E1;
    ps.idn = 0.5 * pv.iA1 * pv.iE1;
    ps.E1 = pv.a.E1;
    ps.E2 = pv.a.E2;
    ps.Sq = 2.0 * pv.a.z1a;
    ps.Sp = 2.0 * pv.a.pa;
#pragma unroll
    for (int i = 0; i < D; ++i) ps.SqV[i] = 2.0 * pv.a.qV[i];
    double Mgb[NC], wk[NC], wv[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) Mgb[q] = 0.0;
    diss_add2<D>(ps, c, nh, gb, 0.5 * b, Mgb);  // (|nu|/2) M gb
    dW_dU_apply<double, D>(nk, jk, c, Mgb, wk);
    dW_dU_apply<double, D>(nv, jv, c, Mgb, wv);
#pragma unroll
    for (int cc = 0; cc < NC; ++cc) {
      gk[cc] += wk[cc];
      gv[cc] -= wv[cc];
    }
  }
#pragma unroll
  for (int cc = 0; cc < NC; ++cc) {
    gsat[((size_t)k * NC + cc) * NS + s] = gk[cc];
    gsat[((size_t)v * NC + cc) * NS + s2] = gv[cc];
  }
}

// Volume part of the reverse.  The transposed operators follow from the
// forward ones: D_i = H^-1 Q_i and Q_i + Q_i^T = E_i (diagonal, nu_i at the
// facet nodes) give D_i^T y = E_i (y/H) - H D_i (y/H), so
//   M_i^T cot = [E_i (cot/H) + beta H D_i (cot/H)] / (beta+1),
//   wbar = sum_i D_i^T gbar_i = sum_i E_i (gbar_i/H) - H sum_i D_i (gbar_i/H):
// both contractions are forward ones, on the tensor cores as in the split
// volume kernel (tc64.cuh), with 2 n_c columns (w, cot/H) and then n_c
// summed ones; 7-node triangles keep float64 loops.  On the float64 pipe the
// pointwise part is left.
template <int D, int NP, int EB, int TH = round32(EB * NP)>
struct VjpCfg {
  static constexpr bool TENSOR = tensor_path(D, NP);
  static constexpr int NC = D + 2;
  static constexpr int THREADS = TH;
  using S1 = tc::Shape<D, NP, EB, 0, 2 * NC, TH>;
  using S2 = tc::Shape<D, NP, EB, NC, 0, TH>;
  static constexpr size_t mx(size_t a, size_t b) { return a > b ? a : b; }
  static constexpr size_t DIG = mx(S1::DIG_BYTES, S2::DIG_BYTES), RES = mx(S1::RES_BYTES, S2::RES_BYTES);
  static constexpr size_t EXB = mx(S1::EX_BYTES, S2::EX_BYTES);
  static constexpr size_t SMEM = TENSOR ? DIG + RES + EXB + EB * sizeof(int) : (size_t)EB * D * NC * NP * 8;
  static constexpr int BY_SMEM = (int)(233472 / (SMEM + 1024));
  static constexpr int BY_REGS = (NP > 32 ? 384 : 512) / THREADS;
  static constexpr int BLOCKS = EB * NP <= 32 || EB == 1 ? 2 : BY_SMEM < BY_REGS ? BY_SMEM : BY_REGS;
};

template <int D, int NP, int EB, int TH = round32(EB * NP)>
__global__ void __launch_bounds__(TH, VjpCfg<D, NP, EB, TH>::BLOCKS) split_vjp_kernel(
    const double* __restrict__ u, const double* __restrict__ cot, const double* __restrict__ ops,
    const uint4* __restrict__ opsP, const short* __restrict__ opsE, const double* __restrict__ J,
    const double* __restrict__ ihd, const double* __restrict__ nu, const double* __restrict__ gsat, int n_e,
    double* __restrict__ grad, Phys<double> c) {
  constexpr int NC = D + 2;
  using Cfg = VjpCfg<D, NP, EB, TH>;
  using S1 = typename Cfg::S1;
  using S2 = typename Cfg::S2;
  constexpr int THREADS = Cfg::THREADS;
  extern __shared__ __align__(16) unsigned char vjp_smem[];
  const int NS = c_ref.n_slot;
  const int el = threadIdx.x / NP;
  const int m = threadIdx.x - el * NP;
  const int e = blockIdx.x * EB + el;
  const bool slot = el < EB, active = slot && e < n_e;
  const int ms = slot ? m : 0, els = slot ? el : 0;
  Node<double, D> nd;
  double vv[NC], x1[2 * NC], ih = 0.0, Hm = 0.0;
#pragma unroll
  for (int q = 0; q < NC; ++q) vv[q] = 0.0;
#pragma unroll
  for (int q = 0; q < 2 * NC; ++q) x1[q] = 0.0;
  if (active) {
    if constexpr (Cfg::TENSOR) {
      constexpr unsigned OPB = D * NP * tc::pairs_for(NP) * sizeof(uint4);
      if (m == 0) tc::prefetch_l2(opsP + (size_t)e * (OPB / sizeof(uint4)), OPB);
    }
    double uu[NC];
    ih = __ldg(&ihd[(size_t)e * NP + m]);
    Hm = c_ref.H[m] * __ldg(&J[(size_t)e * NP + m]);
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      uu[q] = __ldg(&u[((size_t)e * NC + q) * NP + m]);
      vv[q] = __ldg(&cot[((size_t)e * NC + q) * NP + m]);
    }
    node_from_u<double, D>(uu, c, nd);
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      x1[q] = nd.W[q];
      x1[NC + q] = vv[q] * ih;
    }
  }
  __half* dig = reinterpret_cast<__half*>(vjp_smem);
  double* resb = reinterpret_cast<double*>(vjp_smem + Cfg::DIG);
  int* ex = reinterpret_cast<int*>(vjp_smem + Cfg::DIG + Cfg::RES);
  int* elems = reinterpret_cast<int*>(vjp_smem + Cfg::DIG + Cfg::RES + Cfg::EXB);
  double* sx = reinterpret_cast<double*>(vjp_smem);  // float64 loops: [EB][columns][NP]
  const double* op = ops + (size_t)(active ? e : 0) * (D * NP * NP);
  double g[D][NC], t[D][NC];  // D_i w, D_i (cot/H)
  if constexpr (Cfg::TENSOR) {
    if (m == 0 && slot) elems[el] = active ? e : -1;
    tc::digitize<S1, NP, EB, THREADS>(x1, slot, el, m, ex, dig);
    __syncthreads();
    tc::contract<S1, D, NP, EB, 0, 2 * NC, THREADS>(dig, ex, elems, opsP, opsE, resb);
    __syncthreads();
    const double* rs = S1::results(dig, resb, els) + ms;
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int q = 0; q < NC; ++q) {
        g[i][q] = rs[(i * 2 * NC + q) * S1::NPO];
        t[i][q] = rs[(i * 2 * NC + NC + q) * S1::NPO];
      }
    __syncthreads();
  } else {
    if (active) {
#pragma unroll
      for (int q = 0; q < 2 * NC; ++q) sx[(el * 2 * NC + q) * NP + m] = x1[q];
    }
    __syncthreads();
    if (active) {
#pragma unroll
      for (int i = 0; i < D; ++i) {
#pragma unroll
        for (int q = 0; q < NC; ++q) g[i][q] = t[i][q] = 0.0;
#pragma unroll
        for (int n = 0; n < NP; ++n) {
          const double dt = __ldg(&op[(i * NP + n) * NP + m]);  // D_i[m][n]
#pragma unroll
          for (int q = 0; q < NC; ++q) {
            g[i][q] += dt * sx[(el * 2 * NC + q) * NP + n];
            t[i][q] += dt * sx[(el * 2 * NC + NC + q) * NP + n];
          }
        }
      }
    }
    __syncthreads();
  }
  double x2[S2::COLS];  // gbar_i / H
#pragma unroll
  for (int q = 0; q < S2::COLS; ++q) x2[q] = 0.0;
  JvpPrep<double> jp;
  if (active) {
    jp = jvp_prep<double, D>(nd, c);
    const double sc = -c.inv_bp1 * ih;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      double a[NC];
      dflux_dw<double, D>(nd, jp, c, i, vv, a);
#pragma unroll
      for (int q = 0; q < NC; ++q) x2[i * NC + q] = sc * a[q];
    }
  }
  double wb[NC];  // sum_i D_i (gbar_i / H)
  if constexpr (Cfg::TENSOR) {
    tc::digitize<S2, NP, EB, THREADS>(x2, slot, el, m, ex, dig);
    __syncthreads();
    tc::contract<S2, D, NP, EB, NC, 0, THREADS>(dig, ex, elems, opsP, opsE, resb);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NC; ++q) wb[q] = S2::results(dig, resb, els)[q * S2::NPO + ms];
  } else {
    if (active) {
#pragma unroll
      for (int q = 0; q < S2::COLS; ++q) sx[(el * S2::COLS + q) * NP + m] = x2[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NC; ++q) wb[q] = 0.0;
    if (active) {
#pragma unroll
      for (int i = 0; i < D; ++i)
#pragma unroll
        for (int n = 0; n < NP; ++n) {
          const double dt = __ldg(&op[(i * NP + n) * NP + m]);
#pragma unroll
          for (int q = 0; q < NC; ++q) wb[q] += dt * sx[(el * S2::COLS + i * NC + q) * NP + n];
        }
    }
  }
  if (!active) return;
  // fbar_i = M_i^T cot and wbar
  const int sl = c_ref.node_slot[m];
  double nv[D];
#pragma unroll
  for (int i = 0; i < D; ++i) nv[i] = sl >= 0 ? __ldg(&nu[((size_t)e * NS + sl) * D + i]) : 0.0;
  const double kH = c.beta * c.inv_bp1 * Hm;
  double z[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    double s = 0.0;
    const double ci = c.inv_bp1 * x1[NC + q];
#pragma unroll
    for (int i = 0; i < D; ++i) {
      s += nv[i] * x2[i * NC + q];
      t[i][q] = nv[i] * ci + kH * t[i][q];
    }
    z[q] = s - Hm * wb[q];
  }
  // pointwise part.  With A~_i = dF_i/dW symmetric and dW/du the symmetric
  // Hessian of the entropy,
  //   (dF_i/du)^T fb_i = (dW/du) A~_i fb_i,   (dw/du)^T wb = (dW/du) wb,
  // and, F_i being the W-gradient of its flux potential (Sec. 2.4), the
  // derivative of A~_i(W) g along W is symmetric in its three arguments, so the
  // u-gradient of cot_m . A~_i(u) g_i is (dW/du) applied to the derivative of
  // A~_i g_i along W in the single direction cot_m (a one-direction dual
  // number, the state moved by (dU/dW) cot_m):
  //   grad_m = (dW/du) [sum_i A~_i fb_i + wb - 1/(beta+1) sum_i d_cot(A~_i g_i)].
  {
    double a[NC];
    dflux_dw_sum<double, D>(nd, jp, c, 1.0, t, a);
#pragma unroll
    for (int q = 0; q < NC; ++q) z[q] += a[q];
  }
  {
    using T1 = Dual<1>;
    double du[NC];
    dU_dW_apply<double, D>(nd, jp, c, vv, du);
    // the nodal quantities A~_i depends on, with their tangent along du in
    // closed form (no logarithm, exponential or division on the duals):
    //   drho = du_0, dV = (du_m - V drho)/rho, dv2 = 2 V.dV, de = du_E,
    //   dp = (gam-1)(de - (drho v2 + rho dv2)/2), dq = q (a_q drho/rho + b_q dp/p)
    // and those of jvp_prep: d(1/q) = -dq/q^2, dtheta = (dp - theta drho)/rho, ...
    Node<T1, D> n1;
    JvpPrep<T1> j1;
    {
      const double drho = du[0], ip = jp.itheta * jp.ir;
      double hv2 = 0.0;  // V.dV
      n1.rho = T1(nd.rho);
      n1.rho.d[0] = drho;
#pragma unroll
      for (int j = 0; j < D; ++j) {
        const double dVj = (du[1 + j] - nd.V[j] * drho) * nd.ir;
        n1.V[j] = T1(nd.V[j]);
        n1.V[j].d[0] = dVj;
        hv2 += nd.V[j] * dVj;
      }
      const double de = du[NC - 1];
      const double dp = c.gm1 * (de - (0.5 * drho * nd.v2 + nd.rho * hv2));
      n1.v2 = T1(nd.v2);
      n1.v2.d[0] = 2.0 * hv2;
      const double lq = c.a_q * drho * nd.ir + c.b_q * dp * ip;  // dq/q
      const double dth = (dp - jp.theta * drho) * nd.ir;
      j1.iq = T1(jp.iq);
      j1.iq.d[0] = -jp.iq * lq;
      j1.theta = T1(jp.theta);
      j1.theta.d[0] = dth;
      j1.itheta = T1(jp.itheta);
      j1.itheta.d[0] = -jp.itheta * jp.itheta * dth;
      j1.w0q = T1(jp.w0q);
      j1.w0q.d[0] = c.w1c * dth - hv2;
      j1.rq = T1(jp.rq);
      j1.rq.d[0] = c.inv_apb * drho;
      j1.ep = T1(jp.ep);
      j1.ep.d[0] = de + dp;
    }
    T1 dF[NC];
    dflux_dw_sum<T1, D>(n1, j1, c, -c.inv_bp1, g, dF);
#pragma unroll
    for (int q = 0; q < NC; ++q) z[q] += dF[q].d[0];
  }
  double gr[NC];
  dW_dU_apply<double, D>(nd, jp, c, z, gr);
#pragma unroll
  for (int cc = 0; cc < NC; ++cc) {
    if (sl >= 0) gr[cc] += __ldg(&gsat[((size_t)e * NC + cc) * NS + sl]);
    grad[((size_t)e * NC + cc) * NP + m] = gr[cc];
  }
}

template <int D, int NP, int EB, int TH>
static int split_vjp_launch(esplit_ctx* c, const double* u, const double* cot, double* grad, const Phys<double>& ph,
                             cudaStream_t s) {
  using Cfg = VjpCfg<D, NP, EB, TH>;
  auto* kern = split_vjp_kernel<D, NP, EB, TH>;
  if (opt_in_smem(c, kern, Cfg::SMEM, true)) return -1;
  kern<<<(c->n_e + EB - 1) / EB, TH, Cfg::SMEM, s>>>(u, cot, c->b.ops64, c->b.opsP, c->b.opsE, c->b.J, c->b.ihd,
                                                     c->b.nu, c->b.sat, c->n_e, grad, ph);
  return 0;
}

template <int D, int NP>
static int vjp_np(esplit_ctx* c, const double* u, const double* cot, double* grad, cudaStream_t s) {
  const Phys<double> ph = make_phys<double>(c->prm.gam, c->prm.beta, c->prm.R, c->prm.mu, c->prm.Pr);
  {
    const int bs = spread_block(c->n_pairs, 64);
    int nb = (c->n_pairs + bs - 1) / bs;
    ProfScope ps(c, PG_FACE, s);
    face_vjp_kernel<D><<<nb, bs, 0, s>>>(u, cot, c->b.face_pairs, c->n_pairs, c->b.nu, c->b.ihd, c->b.nscale,
                                         c->b.sat, ph, c->prm.dissipation);
    c->launches++;
  }
  {
    // blocks that fill their warps, as the split volume kernel's (12-node
    // tetrahedra, 24,576 elements: ten per block 360 us, five 306)
    constexpr int EB = NP == 7 ? 18 : NP == 12 ? (D == 3 ? 5 : 10) : NP == 18 || NP == 27 ? 7 : NP == 25 ? 5 : 2;
    constexpr int EBS = NP < 32 ? 32 / NP : 1, TASKS = EBS * ((NP + 7) / 8), MIN = round32(EBS * NP);
    constexpr int BY_TASKS = 32 * (TASKS < 4 ? TASKS : 4);
    constexpr int THS = VjpCfg<D, NP, EB>::TENSOR && BY_TASKS > MIN ? BY_TASKS : MIN;
    ProfScope ps(c, PG_SPLIT, s);
    // small meshes: short blocks, as for the split volume kernel
    const int rc = (c->n_e + EBS - 1) / EBS <= SMALL_BLOCKS
                       ? split_vjp_launch<D, NP, EBS, THS>(c, u, cot, grad, ph, s)
                       : split_vjp_launch<D, NP, EB, round32(EB * NP)>(c, u, cot, grad, ph, s);
    if (rc) return rc;
    c->launches++;
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_residual_vjp(esplit_ctx* c, const double* u, const double* cot, double* grad, cudaStream_t s) {
  if (c->dim == 2) {
    switch (c->n_p) {
      case 7: return vjp_np<2, 7>(c, u, cot, grad, s);
      case 12: return vjp_np<2, 12>(c, u, cot, grad, s);
      case 18: return vjp_np<2, 18>(c, u, cot, grad, s);
      case 27: return vjp_np<2, 27>(c, u, cot, grad, s);
    }
  } else if (c->dim == 3) {
    switch (c->n_p) {
      case 12: return vjp_np<3, 12>(c, u, cot, grad, s);
      case 25: return vjp_np<3, 25>(c, u, cot, grad, s);
      case 58: return vjp_np<3, 58>(c, u, cot, grad, s);
      case 78: return vjp_np<3, 78>(c, u, cot, grad, s);
    }
  }
  return -2;
}

}  // namespace esplit
