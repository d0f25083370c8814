// Pointwise physics of the entropy-split scheme, device side, templated on the
// arithmetic type T (double for the FP64 path, float for the FP32-bulk path)
// and the dimension D (n_c = D + 2 components).
//
// Paper: Worku & Zingg, entropy-split multidimensional SBP (Secs. 2-4).
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>

#include "dual.cuh"
#include "fmath.cuh"
#include "imath.cuh"

namespace esplit {

// Constants derived from (gam, beta) on the host, Sec. 2.4 / Eq. (16):
// alpha = -gam - beta (gam - 1).
template <typename T>
struct Phys {
  T gam, alpha, beta;
  T gm1, inv_gm1;      // gam - 1, 1/(gam - 1)
  T a_q, b_q;          // q = rho^a_q p^b_q = (rho/p)(p rho^-gam)^(1/(alpha+gam)), Eq. (41)
  T w1c;               // -alpha/(gam-1): W_1 = q (w1c p/rho - |V|^2/2), Eq. (25)
  T inv_w1c;           // -(gam-1)/alpha
  T inv_apb;           // 1/(a_q + b_q) = (alpha+gam)/(1-gam)
  T r1, r2;            // -gam/alpha and (1-gam)/alpha: the powers of z_1 and z_nc
                       // appearing in Eq. (48) (arithmetic and exponential means)
  T inv_bp1;           // 1/(beta+1)
  T gam_gm1;           // gam/(gam-1)
  T gm1_gam;           // (gam-1)/gam
  T ir_a, ir_b;        // (gam+1)/(2 gam), (gam-1)/(2 gam), times gam/(gam-1)
  T s_ac, s_en;        // S^ entries: 1/(2 gam), (gam-1)(gam+alpha)/(gam alpha), Eq. (76)
  T mu, kappa, R;      // viscosity, conductivity mu gam R/((gam-1) Pr), gas constant
  T iR, k_T;           // 1/R, (gam-1)/(alpha R)
  // Taylor coefficients of g(eps) = ((1+eps)^r - 1)/(r eps) for r = r1, r2
  // (c_0 = 1, c_k = c_(k-1) (r - k)/(k + 1)), used by exp_avg
  T ser1[16], ser2[16];
  // a_q, b_q, r1, r2 in units of 2^-60 for the fixed-point logarithms
  // (imath.cuh); im_ok: all below 8 in size
  long long a60, b60, r160, r260;
  int im_ok;
  // ser1, ser2: c_0 .. c_6 in units of 2^-62, c_7 .. c_12 in float32 (exp_avg_pair)
  long long s1[7], s2[7];
  float t1[6], t2[6];
};

template <typename T>
__host__ inline Phys<T> make_phys(double gam, double beta, double R, double mu, double Pr) {
  Phys<T> c;
  double alpha = -gam - beta * (gam - 1.0);
  c.gam = (T)gam;
  c.alpha = (T)alpha;
  c.beta = (T)beta;
  c.gm1 = (T)(gam - 1.0);
  c.inv_gm1 = (T)(1.0 / (gam - 1.0));
  c.a_q = (T)(alpha / (alpha + gam));
  c.b_q = (T)((1.0 - alpha - gam) / (alpha + gam));
  c.w1c = (T)(-alpha / (gam - 1.0));
  c.inv_w1c = (T)(-(gam - 1.0) / alpha);
  c.inv_apb = (T)((alpha + gam) / (1.0 - gam));
  c.r1 = (T)(-gam / alpha);
  c.r2 = (T)((1.0 - gam) / alpha);
  c.inv_bp1 = (T)(1.0 / (beta + 1.0));
  c.gam_gm1 = (T)(gam / (gam - 1.0));
  c.gm1_gam = (T)((gam - 1.0) / gam);
  c.ir_a = (T)(gam / (gam - 1.0) * ((gam + 1.0) / (2.0 * gam)));
  c.ir_b = (T)(gam / (gam - 1.0) * ((gam - 1.0) / (2.0 * gam)));
  c.s_ac = (T)(1.0 / (2.0 * gam));
  c.s_en = (T)((gam - 1.0) * (gam + alpha) / (gam * alpha));
  c.mu = (T)mu;
  c.kappa = (T)(mu * gam * R / ((gam - 1.0) * Pr));
  c.R = (T)R;
  c.iR = (T)(1.0 / R);
  c.k_T = (T)((gam - 1.0) / (alpha * R));
  double r1 = -gam / alpha, r2 = (1.0 - gam) / alpha;
  const double pw[4] = {alpha / (alpha + gam), (1.0 - alpha - gam) / (alpha + gam), r1, r2};
  c.im_ok = 1;
  for (int k = 0; k < 4; ++k)
    if (!(fabs(pw[k]) < 8.0)) c.im_ok = 0;
  const double sc = c.im_ok ? 1152921504606846976.0 : 0.0;  // 2^60
  c.a60 = (long long)(pw[0] * sc);
  c.b60 = (long long)(pw[1] * sc);
  c.r160 = (long long)(pw[2] * sc);
  c.r260 = (long long)(pw[3] * sc);
  if (!(r1 > 0.0 && r1 < 1.0 && r2 > 0.0 && r2 < 1.0)) c.im_ok = 0;
  double a1 = 1.0, a2 = 1.0;
  for (int k = 0; k < 16; ++k) {
    if (k > 0) {
      a1 *= (r1 - k) / (k + 1);
      a2 *= (r2 - k) / (k + 1);
    }
    c.ser1[k] = (T)a1;
    c.ser2[k] = (T)a2;
    if (k < 7) {  // |c_k| <= 1 for exponents in (0, 1); exp_avg_pair is not used otherwise
      const double u62 = 4611686018427387904.0;
      c.s1[k] = fabs(a1) <= 1.0 ? (long long)(a1 * u62) : 0;
      c.s2[k] = fabs(a2) <= 1.0 ? (long long)(a2 * u62) : 0;
    } else if (k < 13) {
      c.t1[k - 7] = (float)a1;
      c.t2[k - 7] = (float)a2;
    }
  }
  return c;
}

__device__ __forceinline__ double t_log(double x) { return fm::log(x); }
__device__ __forceinline__ float t_log(float x) { return logf(x); }
__device__ __forceinline__ double t_exp(double x) { return fm::exp(x); }
__device__ __forceinline__ float t_exp(float x) { return expf(x); }
__device__ __forceinline__ double t_sqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float t_sqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double t_abs(double x) { return fabs(x); }
__device__ __forceinline__ float t_abs(float x) { return fabsf(x); }
__device__ __forceinline__ double t_expm1(double x) { return fm::expm1(x); }
__device__ __forceinline__ float t_expm1(float x) { return expm1f(x); }
__device__ __forceinline__ double t_log1p(double x) { return fm::log1p(x); }
__device__ __forceinline__ float t_log1p(float x) { return log1pf(x); }
__device__ __forceinline__ bool t_isfinite(double x) { return ::isfinite(x); }
__device__ __forceinline__ bool t_isfinite(float x) { return ::isfinite(x); }
// x > 0 (NaN: false) and x finite, from the bit pattern: integer operations
// instead of float64 compares (which take the float64 pipe)
__device__ __forceinline__ bool t_positive(double x) {
  return (unsigned long long)__double_as_longlong(x) - 1ULL < 0x7FF0000000000000ULL;
}
__device__ __forceinline__ bool t_positive(float x) { return (unsigned)__float_as_uint(x) - 1u < 0x7F800000u; }
__device__ __forceinline__ bool t_finite_bits(double x) {
  return ((unsigned long long)__double_as_longlong(x) & 0x7FF0000000000000ULL) != 0x7FF0000000000000ULL;
}
__device__ __forceinline__ bool t_finite_bits(float x) { return (__float_as_uint(x) & 0x7F800000u) != 0x7F800000u; }
template <int N>
__device__ __forceinline__ bool t_positive(const Dual<N>& x) {
  return t_positive(x.v);
}
template <int N>
__device__ __forceinline__ bool t_finite_bits(const Dual<N>& x) {
  return t_finite_bits(x.v);
}

// 1/d by the cubic iteration y0 (1 + e + e^2), e = 1 - d y0 (Chebyshev's
// method), from the hardware's 20-bit estimate: three float64 FMAs, where the
// division takes about nine float64 instructions.  The error before the last
// rounding is e^3 < 2^-57 relative.  Subnormal d gives a NaN where the
// division gives a huge value: such states are not physical (t_positive
// passes them, the logarithms then fail) or columns of no weight.
__device__ __forceinline__ double rcp64(double d) {
  double y0;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y0) : "d"(d));
  const double e = fma(-d, y0, 1.0);
  return fma(y0, fma(e, e, e), y0);
}
// 1/sqrt(x) by the cubic iteration r0 (1 + e/2 + 3 e^2/8), e = 1 - x r0^2,
// from the hardware's 19-bit estimate.  Error at most 1.7 2^-53 relative: the
// last rounding, half the rounding of x r0, and the next term 5/16 e^3.
__device__ __forceinline__ double rsqrt64(double x) {
  double r0;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r0) : "d"(x));
  const double e = fma(-(x * r0), r0, 1.0);
  return fma(r0 * e, fma(e, 0.375, 0.5), r0);
}

template <typename T>
__device__ __forceinline__ T t_rcp(const T& d) {
  if constexpr (std::is_same<T, double>::value)
    return rcp64(d);
  else
    return T(1) / d;
}

// Nodal state: primitives, q = z_1 of Eq. (45) (= -W_nc), Harten entropy
// variables W of Eq. (25).
template <typename T, int D>
struct Node {
  T rho, V[D], p, e, q, v2;
  T lnq, lnp;  // log q, log p (reused by the parameter-vector powers)
  T ir;        // 1/rho
  T W[D + 2];
};

// log p, log q and q = rho^a_q p^b_q: in fixed point (imath.cuh) inside its
// domain, which holds every ordinary state; the float64 functions otherwise.
__device__ __forceinline__ void node_logs(double rho, double p, const Phys<double>& c, double& lnp, double& lnq,
                                          double& q) {
  long long lr, lp, la, lb;
  if (c.im_ok && im::log_fixed(rho, lr) && im::log_fixed(p, lp) && im::mul_q60(lr, c.a60, la) &&
      im::mul_q60(lp, c.b60, lb)) {
    lnp = im::to_double(lp);
    lnq = im::to_double(la + lb);
    q = im::exp_fixed(la + lb);
  } else {
    lnp = t_log(p);
    lnq = c.a_q * t_log(rho) + c.b_q * lnp;
    q = t_exp(lnq);
  }
}

// log x to an absolute 2^-59 near 1, in fixed point; the float64 function elsewhere
__device__ __forceinline__ double log_abs(double x) {
  long long L;
  return im::log_fixed62(x, L) ? im::to_double<62>(L) : t_log(x);
}

// exp(r l) for a power r (r60: in units of 2^-60) and a logarithm l
__device__ __forceinline__ double pow_from_log(double l, double r, long long r60, const Phys<double>& c) {
  long long L, X;
  if (c.im_ok && im::from_double(l, L) && im::mul_q60(L, r60, X)) return im::exp_fixed(X);
  return t_exp(r * l);
}

// Returns false for a non-physical state (rho <= 0, p <= 0 or NaN).
template <typename T, int D, typename C>
__device__ __forceinline__ bool node_from_u(const T* u, const C& c, Node<T, D>& n) {
  n.rho = u[0];
  T ir = t_rcp(n.rho);
  n.ir = ir;
  n.v2 = T(0);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    n.V[i] = u[1 + i] * ir;
    n.v2 += n.V[i] * n.V[i];
  }
  n.e = u[D + 1];
  n.p = c.gm1 * (n.e - T(0.5) * n.rho * n.v2);
  bool ok = t_positive(n.rho) && t_positive(n.p) && t_finite_bits(n.e);
  if constexpr (std::is_same<T, double>::value) {
    node_logs(n.rho, n.p, c, n.lnp, n.lnq, n.q);
  } else {
    n.lnp = t_log(n.p);
    n.lnq = c.a_q * t_log(n.rho) + c.b_q * n.lnp;
    n.q = t_exp(n.lnq);
  }
  n.W[0] = n.q * (c.w1c * n.p * ir - T(0.5) * n.v2);
#pragma unroll
  for (int i = 0; i < D; ++i) n.W[1 + i] = n.q * n.V[i];
  n.W[D + 1] = -n.q;
  return ok;
}

// dF^{I(i)} = A~_i v (Eq. (19)): the change of F_i(U(W)) for a change v of
// the entropy variables, by the chain rule through (q, V, theta = p/rho, rho):
//   q = -W_nc, V = W_(1..d)/q, W_1/q = w1c theta - |V|^2/2,
//   q = rho^(a_q + b_q) theta^b_q.
// reciprocals shared by the d directions of dflux_dw
template <typename T>
struct JvpPrep {
  T iq, ir, theta, itheta;
  T w0q, rq, ep;  // w1c theta - |V|^2/2, rho/(a_q + b_q), e + p (shared by the directions)
};

// from 1/q and rho/p
template <typename T, int D, typename C>
__device__ __forceinline__ JvpPrep<T> jvp_prep_from(const Node<T, D>& n, const C& c, const T& iq, const T& itheta) {
  JvpPrep<T> j;
  j.iq = iq;
  j.ir = n.ir;
  j.theta = n.p * j.ir;
  j.itheta = itheta;
  j.w0q = c.w1c * j.theta - T(0.5) * n.v2;
  j.rq = n.rho * c.inv_apb;
  j.ep = n.e + n.p;
  return j;
}

// one division for 1/q and rho/p: y = 1/(q p), 1/q = p y, 1/p = q y
template <typename T, int D, typename C>
__device__ __forceinline__ JvpPrep<T> jvp_prep(const Node<T, D>& n, const C& c) {
  const T y = t_rcp(n.q * n.p);
  return jvp_prep_from<T, D>(n, c, n.p * y, n.rho * (n.q * y));
}

template <typename T, int D, typename C>
__device__ __forceinline__ void dflux_dw(const Node<T, D>& n, const JvpPrep<T>& jp, const C& c, int i,
                                         const T* v, T* dF) {
  T iq = jp.iq;
  T dq = -v[D + 1];
  T dV[D];
  T vdv = T(0);
#pragma unroll
  for (int j = 0; j < D; ++j) {
    dV[j] = (v[1 + j] - dq * n.V[j]) * iq;
    vdv += n.V[j] * dV[j];
  }
  T theta = jp.theta;
  T dtheta = c.inv_w1c * ((v[0] - dq * jp.w0q) * iq + vdv);
  T drho = jp.rq * (dq * iq - c.b_q * dtheta * jp.itheta);
  T dp = drho * theta + n.rho * dtheta;
  T dm = drho * n.V[i] + n.rho * dV[i];
  dF[0] = dm;
  T rvi = n.rho * n.V[i];
#pragma unroll
  for (int j = 0; j < D; ++j) dF[1 + j] = dm * n.V[j] + rvi * dV[j] + (j == i ? dp : T(0));
  T de = dp * c.inv_gm1 + T(0.5) * drho * n.v2 + n.rho * vdv;
  dF[D + 1] = (de + dp) * n.V[i] + jp.ep * dV[i];
}

// Euler fluxes of all directions, F[i (D+2) + q] = F^{I(i)}_q of Eq. (5), with
// the momenta taken from the state itself (no rho V product) and the symmetric
// momentum fluxes m_i V_j = m_j V_i formed once: 6 float64 operations in 2D
// and 13 in 3D instead of 10 and 21.
template <int D>
__device__ __forceinline__ void euler_fluxes(const Node<double, D>& n, const double* u, double* F) {
  constexpr int NC = D + 2;
  const double ep = n.e + n.p;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    F[i * NC] = u[1 + i];
    F[i * NC + 1 + i] = u[1 + i] * n.V[i] + n.p;
#pragma unroll
    for (int j = i + 1; j < D; ++j) F[i * NC + 1 + j] = F[j * NC + 1 + i] = u[1 + i] * n.V[j];
    F[i * NC + NC - 1] = ep * n.V[i];
  }
}

// out = s sum_i A~_i g_i (Eq. (19)), g_i = D_i w: dflux_dw summed over the
// directions before the products with the node's state, so that only the
// temperature and pressure changes are formed per direction:
//   Q = -sum_i V_i dq_i,  div = sum_i dV_i[i],  adv_j = sum_i V_i dV_i[j],
//   T = sum_i V_i dtheta_i,  A = sum_i V_i drho_i,
//   out_0 = A + rho div,  out_j = out_0 V_j + rho adv_j + dp_j,
//   out_E = gam/(gam-1) sum_i V_i dp_i + (|V|^2/2) A + rho V.adv + (e + p) div,
//   dtheta_i = (g_i0 + V.g_im + g_iE (W_1/q + |V|^2)) / (w1c q).
// 48 float64 operations in 2D and 72 in 3D; dflux_dw direction by direction
// takes 72 and 139.  s is carried by the reciprocal 1/q of the linear terms.
template <typename T, int D, typename C>
__device__ __forceinline__ void dflux_dw_sum(const Node<T, D>& n, const JvpPrep<T>& jp, const C& c, double s,
                                             const double (&g)[D][D + 2], T* out) {
  constexpr int NC = D + 2;
  const T iq = s * jp.iq, k = c.inv_w1c * iq, we = jp.w0q + n.v2, c1 = c.b_q * jp.itheta;
  const T rt = jp.rq * jp.theta, cp = n.rho - rt * c1, cq = rt * iq;
  T Q, TT, P, dp[D], S[D];
  double tr = 0.0;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    T t = g[i][0] + g[i][NC - 1] * we;
#pragma unroll
    for (int j = 0; j < D; ++j) t = t + n.V[j] * g[i][1 + j];
    t = t * k;
    dp[i] = cp * t - cq * g[i][NC - 1];  // drho theta + rho dtheta, dq = -g_E
    if (i == 0) {
      Q = n.V[0] * g[0][NC - 1];
      TT = n.V[0] * t;
      P = n.V[0] * dp[0];
      tr = g[0][1];
    } else {
      Q = Q + n.V[i] * g[i][NC - 1];
      TT = TT + n.V[i] * t;
      P = P + n.V[i] * dp[i];
      tr += g[i][1 + i];
    }
#pragma unroll
    for (int j = 0; j < D; ++j) S[j] = i == 0 ? n.V[0] * g[0][1 + j] : S[j] + n.V[i] * g[i][1 + j];
  }
  const T div = iq * (Q + tr);  // Q here is sum_i V_i g_iE = -sum_i V_i dq_i
  const T A = jp.rq * (-(iq * Q) - c1 * TT);
  const T M = A + n.rho * div;
  const T riq = n.rho * iq;
  T va;
  out[0] = M;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    const T ra = riq * (S[j] + n.V[j] * Q);  // rho adv_j
    va = j == 0 ? n.V[0] * ra : va + n.V[j] * ra;
    out[1 + j] = M * n.V[j] + (ra + dp[j]);
  }
  out[NC - 1] = c.gam_gm1 * P + (0.5 * n.v2 * A + (va + jp.ep * div));
}

// (dW/dU) z: the change of the entropy variables (Eq. (25)) for a change z of
// the conservative variables, by the chain rule through (rho, V, p, q):
//   dV = (dm - V drho)/rho, dp = (gam-1)(dE - V.dm + |V|^2 drho/2),
//   dq/q = a_q drho/rho + b_q dp/p, d(p/rho) = (dp - (p/rho) drho)/rho,
//   dW = [dq (w1c p/rho - |V|^2/2) + q (w1c d(p/rho) - V.dV), dq V + q dV, -dq].
// dW/dU is the Hessian of the entropy, symmetric.
template <typename T, int D, typename C>
__device__ __forceinline__ void dW_dU_apply(const Node<T, D>& n, const JvpPrep<T>& jp, const C& c, const T* z,
                                            T* out) {
  const T drho = z[0];
  T dV[D], vdm = T(0);
#pragma unroll
  for (int j = 0; j < D; ++j) {
    vdm += n.V[j] * z[1 + j];
    dV[j] = (z[1 + j] - n.V[j] * drho) * jp.ir;
  }
  const T dp = c.gm1 * (z[D + 1] - vdm + T(0.5) * n.v2 * drho);
  const T ip = jp.itheta * jp.ir;  // 1/p
  const T dq = n.q * (c.a_q * drho * jp.ir + c.b_q * dp * ip);
  const T dth = (dp - jp.theta * drho) * jp.ir;
  T vdv = T(0);
#pragma unroll
  for (int j = 0; j < D; ++j) vdv += n.V[j] * dV[j];
  out[0] = dq * jp.w0q + n.q * (c.w1c * dth - vdv);
#pragma unroll
  for (int j = 0; j < D; ++j) out[1 + j] = dq * n.V[j] + n.q * dV[j];
  out[D + 1] = -dq;
}

// (dU/dW) v: the change of the conservative variables for a change v of the
// entropy variables (the inverse map of Eq. (25), the chain rule dflux_dw
// starts with): dq = -v_nc, dV = (v_m - dq V)/q,
// d(p/rho) = ((v_1 - dq W_1/q)/q + V.dV)/w1c, drho from q = rho^(a_q+b_q) (p/rho)^b_q,
// dU = [drho, drho V + rho dV, dp/(gam-1) + drho |V|^2/2 + rho V.dV].
template <typename T, int D, typename C>
__device__ __forceinline__ void dU_dW_apply(const Node<T, D>& n, const JvpPrep<T>& jp, const C& c, const T* v,
                                            T* out) {
  const T dq = -v[D + 1];
  T dV[D], vdv = T(0);
#pragma unroll
  for (int j = 0; j < D; ++j) {
    dV[j] = (v[1 + j] - dq * n.V[j]) * jp.iq;
    vdv += n.V[j] * dV[j];
  }
  const T dth = c.inv_w1c * ((v[0] - dq * jp.w0q) * jp.iq + vdv);
  const T drho = jp.rq * (dq * jp.iq - c.b_q * dth * jp.itheta);
  const T dp = drho * jp.theta + n.rho * dth;
  out[0] = drho;
#pragma unroll
  for (int j = 0; j < D; ++j) out[1 + j] = drho * n.V[j] + n.rho * dV[j];
  out[D + 1] = dp * c.inv_gm1 + T(0.5) * drho * n.v2 + n.rho * vdv;
}

// Powers of the parameter vector used by the two-point flux and the
// dissipation: P1 = z_1^r1 = q^r1, P2 = z_nc^r2 = p^r2.
template <typename T, int D, typename C>
__device__ __forceinline__ void z_powers(const Node<T, D>& n, const C& c, T& P1, T& P2) {
  if constexpr (std::is_same<T, double>::value) {
    P1 = pow_from_log(n.lnq, c.r1, c.r160, c);
    P2 = pow_from_log(n.lnp, c.r2, c.r260, c);
  } else {
    P1 = t_exp(c.r1 * n.lnq);
    P2 = t_exp(c.r2 * n.lnp);
  }
}

// Exponential average of Eq. (47), {u^(r-1)}_e = (a^r - b^r)/(r (a - b)),
// given ar = a^r and br = b^r.  For |b/a - 1| >= EPS_SWITCH the quotient is
// used directly; below it the equivalent form a^(r-1) g(eps),
// g(eps) = ((1+eps)^r - 1)/(r eps) = sum_k c_k eps^k with c_0 = 1,
// c_k = c_(k-1) (r - k)/(k + 1), summed to NTERMS terms.  For gam > 1 and
// beta > 0 both exponents lie in (0, 1), so |c_k| <= 1 and the terms that
// float64's 13 drop weigh at most 0.05^13/0.95 = 0.12 ulp of g at
// |eps| = 0.05 (0.005 ulp for gam = 1.4, beta = 2.5: r = 7/12 and 1/6).
template <typename T>
struct ExpAvgCfg;
template <>
struct ExpAvgCfg<double> {
  static constexpr double EPS_SWITCH = 0.05;
  static constexpr int NTERMS = 13;
};
template <>
struct ExpAvgCfg<float> {
  static constexpr float EPS_SWITCH = 0.25f;
  static constexpr int NTERMS = 14;
};

template <typename T, typename S>
__device__ __forceinline__ T exp_avg(T a, T b, T ar, T br, S r, T ia, const S* coef) {
  T eps = (b - a) * ia;
  if (t_abs(eps) >= ExpAvgCfg<T>::EPS_SWITCH) {
    return (ar - br) / (r * (a - b));
  }
  T sum = coef[ExpAvgCfg<T>::NTERMS - 1];
#pragma unroll
  for (int k = ExpAvgCfg<T>::NTERMS - 2; k >= 0; --k) sum = sum * eps + coef[k];  // Horner
  return ar * ia * sum;
}

// Everything the two-point flux needs at one node.
template <typename T, int D>
struct ZNode {
  T q, V[D], p, P1, P2, v2;
  T iq, ip;  // 1/q, 1/p (used by the exponential averages)
};

template <typename T, int D, typename C>
__device__ __forceinline__ void znode(const Node<T, D>& n, const C& c, ZNode<T, D>& z) {
  z.q = n.q;
  z.p = n.p;
  z.v2 = n.v2;
#pragma unroll
  for (int i = 0; i < D; ++i) z.V[i] = n.V[i];
  z_powers<T, D>(n, c, z.P1, z.P2);
  z.iq = T(0);
  z.ip = T(0);
}

// the reciprocals the exponential averages of a pair need (side k only)
template <typename T, int D>
__device__ __forceinline__ void znode_recips(ZNode<T, D>& z) {
  z.iq = t_rcp(z.q);
  z.ip = t_rcp(z.p);
}

// Pair averages shared by the Sjogreen-Yee flux (Eq. (48)) and the
// intermediate state of the dissipation (Eqs. (73)-(78)).
template <typename T, int D>
struct PairAvg {
  T A1;       // {z_1^(-gam/alpha)}            arithmetic
  T E1;       // {z_nc^((1-gam-alpha)/alpha)}_e exponential
  T A2;       // {z_nc^(-(gam-1)/alpha)}       arithmetic
  T E2;       // {z_1^(-(gam+alpha)/alpha)}_e  exponential
  T z1a;      // {z_1}
  T qV[D];    // {z_1 z_(i+1)}
  T Va[D];    // {V}
  T pa;       // {p}
  T ke;       // sum {V_j}^2 - 1/2 {sum V_j^2}
};

template <typename T, int D, typename C>
__device__ __forceinline__ void pair_avg(const ZNode<T, D>& k, const ZNode<T, D>& v, const C& c,
                                         PairAvg<T, D>& a) {
  a.A1 = T(0.5) * (k.P1 + v.P1);
  a.E1 = exp_avg(k.p, v.p, k.P2, v.P2, c.r2, k.ip, c.ser2);
  a.A2 = T(0.5) * (k.P2 + v.P2);
  a.E2 = exp_avg(k.q, v.q, k.P1, v.P1, c.r1, k.iq, c.ser1);
  a.z1a = T(0.5) * (k.q + v.q);
  a.ke = T(0);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    a.qV[i] = T(0.5) * (k.q * k.V[i] + v.q * v.V[i]);
    a.Va[i] = T(0.5) * (k.V[i] + v.V[i]);
    a.ke += a.Va[i] * a.Va[i];
  }
  a.ke -= T(0.25) * (k.v2 + v.v2);
  a.pa = T(0.5) * (k.p + v.p);
}

// sum_i nu_i F*_i(U_k, U_v) (Eq. (48)) for a direction vector nu.
template <typename T, int D, typename C>
__device__ __forceinline__ void sy_flux_dir(const PairAvg<T, D>& a, const C& c, const T* nu, T* F) {
  T inv_den = t_rcp(a.A1 * a.E1);
  T mn = T(0);
#pragma unroll
  for (int i = 0; i < D; ++i) mn += nu[i] * a.qV[i];
  mn *= inv_den;
  F[0] = mn;
#pragma unroll
  for (int j = 0; j < D; ++j) F[1 + j] = mn * a.Va[j] + nu[j] * a.pa;
  F[D + 1] = mn * (c.gam_gm1 * a.A2 * a.E2 + a.ke);
}

// Exponential average of Eq. (47) as exp_avg, float64, the series in fixed
// point: Horner's rule on 64-bit integers for c_0 .. c_6 and in float32 for
// c_7 .. c_12 (below 2^-30 of the sum), ~110 integer instructions instead of
// 12 float64 ones (which cost ~900 clocks of the pipe).
__device__ __forceinline__ double exp_avg_pair(double a, double b, double ar, double br, double r, double ia,
                                               const double* coef, const long long* s62, const float* tail, int ok) {
  const double eps = (b - a) * ia;
  if (!fm::abs_below(eps, 0x3FA999999999999AULL)) return (ar - br) / (r * (a - b));  // 0.05
  if (!ok) {
    double sum = coef[ExpAvgCfg<double>::NTERMS - 1];
#pragma unroll
    for (int k = ExpAvgCfg<double>::NTERMS - 2; k >= 0; --k) sum = sum * eps + coef[k];
    return ar * ia * sum;
  }
  const long long x = im::small_to_fixed(eps);
  const float xf = __int2float_rn((int)(x >> 32)) * 0x1p-34f;
  float t = tail[5];
#pragma unroll
  for (int k = 4; k >= 0; --k) t = t * xf + tail[k];
  long long s = (long long)__float2int_rn(t * 0x1p30f) << 32;
#pragma unroll
  for (int k = 6; k >= 0; --k) s = im::horner62(s, x, s62[k]);
  const double sum = im::unit62_to_double(s);
  return ar * ia * sum;
}

// Two-point quantities of a node pair in float64, as sums instead of means
// (twice PairAvg's fields, the halves cancel in the flux and its doubled
// result): the Sjogreen-Yee flux and the dissipation of Eqs. (48) and (69)
// with the fewest float64 operations.
//   dn = {P1}' E1 (= 2 A1 E1), idn = 1/dn, h2 = 2 [gam/(gam-1) A2 E2 + ke],
//   ke = sum {V_j}^2 - {sum V_j^2}/2 = V_k . V_v / 2.
template <int D>
struct PairSums {
  double dn, idn, E1, E2, Sq, Sp, SqV[D], SV[D], h2;
};

// qVk, qVv: q V of the two sides
template <int D, typename C>
__device__ __forceinline__ void pair_sums(const ZNode<double, D>& k, const ZNode<double, D>& v, const double* qVk,
                                          const double* qVv, const C& c, PairSums<D>& a) {
  a.E1 = exp_avg_pair(k.p, v.p, k.P2, v.P2, c.r2, k.ip, c.ser2, c.s2, c.t2, c.im_ok);
  a.E2 = exp_avg_pair(k.q, v.q, k.P1, v.P1, c.r1, k.iq, c.ser1, c.s1, c.t1, c.im_ok);
  a.dn = (k.P1 + v.P1) * a.E1;
  a.idn = rcp64(a.dn);
  a.Sq = k.q + v.q;
  a.Sp = k.p + v.p;
  a.h2 = c.gam_gm1 * (k.P2 + v.P2) * a.E2;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    a.SqV[i] = qVk[i] + qVv[i];
    a.SV[i] = k.V[i] + v.V[i];
    a.h2 += k.V[i] * v.V[i];
  }
}

// 2 sum_i nu_i F*_i(U_k, U_v) (Eq. (48)) for a direction vector nu
template <int D>
__device__ __forceinline__ void sy_flux2(const PairSums<D>& a, const double* nu, double* G2) {
  double mn = 0.0;
#pragma unroll
  for (int i = 0; i < D; ++i) mn = i == 0 ? nu[0] * a.SqV[0] : mn + nu[i] * a.SqV[i];
  mn *= a.idn;
  G2[0] = mn + mn;
#pragma unroll
  for (int j = 0; j < D; ++j) G2[1 + j] = mn * a.SV[j] + nu[j] * a.Sp;
  G2[D + 1] = mn * a.h2;
}

// out += b X^ |Lambda_n| S^ X^T dw (Eq. (69), unit normal n) at the
// intermediate state: the terms of diss_apply with the two acoustic columns
// taken together,
//   y0 = (c_0 . dw) l_0, y-+ = (base -+ s) l-+,  base = dw_0 + V.dw_m + H dw_E,
//   s = a (n.dw_m + vn dw_E),
//   out = [y- + y+ + y0, V out_0 + a (y+ - y-) n, H (y- + y+) + vn a (y+ - y-) + |V|^2/2 y0]
// plus the printed tangential columns.  theta/(2 gam) = idn / a^2 and
// 1/(z1 E1 E2), 1/z1 come from one reciprocal, a and 1/a from one rsqrt.
template <int D, typename C>
__device__ __forceinline__ void diss_add2(const PairSums<D>& p, const C& c, const double* n, const double* dw,
                                          double b, double* out) {
  constexpr int NC = D + 2;
  const double E12 = p.E1 * p.E2, y = rcp64(p.Sq * E12);
  const double iSq = E12 * y, eta = 2.0 * y;
  double V[D], vn = 0.0, h = 0.0, ndm = 0.0, base = dw[0];
#pragma unroll
  for (int i = 0; i < D; ++i) {
    V[i] = p.SqV[i] * iSq;
    vn = i == 0 ? V[0] * n[0] : vn + V[i] * n[i];
    h = i == 0 ? V[0] * V[0] : h + V[i] * V[i];
    ndm = i == 0 ? n[0] * dw[1] : ndm + n[i] * dw[1 + i];
    base += V[i] * dw[1 + i];
  }
  h *= 0.5;
  const double x = (0.5 * c.gam) * p.Sp * p.dn * iSq;  // a^2 = gam p^ / rho^
  const double ia = rsqrt64(x), ah = x * ia;
  const double kac = b * p.idn * (ia * ia);            // b theta / (2 gam)
  const double Hh = x * c.inv_gm1 + h, e = dw[NC - 1];
  const double s = ah * (ndm + vn * e);
  const double avn = fabs(vn);
  const double y0 = (base + h * e) * (avn * (2.0 * c.gam * c.s_en) * kac);
  base += Hh * e;
  const double ym = (base - s) * (fabs(vn - ah) * kac), yp = (base + s) * (fabs(vn + ah) * kac);
  const double sp = ym + yp, sd = ah * (yp - ym), o0 = sp + y0;
  out[0] += o0;
  double oE = Hh * sp + (h * y0 + vn * sd);
#pragma unroll
  for (int i = 0; i < D; ++i) out[1 + i] += V[i] * o0 + sd * n[i];
  if constexpr (D >= 2) {  // (0, n2, -n1, 0, V1 n2 - V2 n1)
    const double l = avn * eta * b;
    const double c2 = V[0] * n[1] - V[1] * n[0];
    const double t = (n[1] * dw[1] - n[0] * dw[2] + c2 * e) * l;
    out[1] += n[1] * t;
    out[2] -= n[0] * t;
    oE += c2 * t;
    if constexpr (D == 3) {  // (0, -n3, 0, n1, V3 n1 - V1 n3)
      const double c3 = V[2] * n[0] - V[0] * n[2];
      const double t3 = (n[0] * dw[3] - n[2] * dw[1] + c3 * e) * l;
      out[1] -= n[2] * t3;
      out[3] += n[0] * t3;
      oE += c3 * t3;
    }
  }
  out[NC - 1] += oE;
}

// X^ |Lambda_n| S^ X^T dw of Eq. (69) at the intermediate state (Eqs.
// (73)-(80)); n is a unit normal.  3D eigenvectors as printed, 2D by
// deleting the fourth row and column.
template <typename T, int D, typename C>
__device__ __forceinline__ void diss_apply(const PairAvg<T, D>& a, const C& c, const T* n, const T* dw,
                                           T* out) {
  // the reciprocals of z1a, A1 E1 and p_h, and eta, from one division:
  // D0 = 1/(z1a A1 E1 E2 p_h)
  const T ae = a.A1 * a.E1;
  T p_h = a.pa;
  const T D0 = T(1) / (a.z1a * ae * a.E2 * p_h);
  const T iz = ae * a.E2 * p_h * D0;        // 1/z1a
  const T iae = a.z1a * a.E2 * p_h * D0;    // 1/(A1 E1)
  const T ip_h = a.z1a * ae * a.E2 * D0;    // 1/p_h
  T rho_h = a.z1a * iae;
  T Vh[D];
  T vh2 = T(0), vn = T(0);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    Vh[i] = a.qV[i] * iz;
    vh2 += Vh[i] * Vh[i];
    vn += Vh[i] * n[i];
  }
  T theta = rho_h * iae * ip_h;             // rho_h / (p_h A1 E1)
  T eta = a.A1 * p_h * D0;                  // 1/(z1a E2 E1)
  T ah = t_sqrt(c.gam * p_h * ae * iz);     // sqrt(gam p_h / rho_h)
  T Hh = ah * ah * c.inv_gm1 + T(0.5) * vh2;
  constexpr int NC = D + 2;
  // columns of X^
  T X[NC][NC];  // X[row][col]
  X[0][0] = T(1);
  X[0][1] = T(1);
  X[0][NC - 1] = T(1);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    X[1 + i][0] = Vh[i] - ah * n[i];
    X[1 + i][1] = Vh[i];
    X[1 + i][NC - 1] = Vh[i] + ah * n[i];
  }
  X[NC - 1][0] = Hh - ah * vn;
  X[NC - 1][1] = T(0.5) * vh2;
  X[NC - 1][NC - 1] = Hh + ah * vn;
  if constexpr (D == 1) {
    // no shear modes: the acoustic and entropy columns only
  } else if constexpr (D == 2) {
    X[0][2] = T(0);
    X[1][2] = n[1];
    X[2][2] = -n[0];
    X[3][2] = Vh[0] * n[1] - Vh[1] * n[0];
  } else {
    X[0][2] = T(0);
    X[1][2] = n[1];
    X[2][2] = -n[0];
    X[3][2] = T(0);
    X[4][2] = Vh[0] * n[1] - Vh[1] * n[0];
    X[0][3] = T(0);
    X[1][3] = -n[2];
    X[2][3] = T(0);
    X[3][3] = n[0];
    X[4][3] = Vh[2] * n[0] - Vh[0] * n[2];
  }
  T s_ac = c.s_ac * theta;
  T lam_s[NC];
  lam_s[0] = t_abs(vn - ah) * s_ac;
  lam_s[1] = t_abs(vn) * c.s_en * theta;
#pragma unroll
  for (int k = 2; k < NC - 1; ++k) lam_s[k] = t_abs(vn) * eta;
  lam_s[NC - 1] = t_abs(vn + ah) * s_ac;
  T y[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    T s = T(0);
#pragma unroll
    for (int r = 0; r < NC; ++r) s += X[r][k] * dw[r];
    y[k] = s * lam_s[k];
  }
#pragma unroll
  for (int r = 0; r < NC; ++r) {
    T s = T(0);
#pragma unroll
    for (int k = 0; k < NC; ++k) s += X[r][k] * y[k];
    out[r] = s;
  }
}

// ---------------------------------------------------------------------------
// Comparator of Sec. 6: the Ismail-Roe entropy-conservative flux (Ismail &
// Roe, J. Comput. Phys. 228, 2009; not printed in the paper), for the
// standard entropy.  With z = sqrt(rho/p) [1, V, p]:
//   rho^ = {z_1} {z_nc}_log,  V^ = {z_1 V}/{z_1},  p1^ = {z_nc}/{z_1},
//   p2^ = (gam+1)/(2 gam) {z_nc}_log/{z_1}_log + (gam-1)/(2 gam) {z_nc}/{z_1},
//   H^ = gam p2^/((gam-1) rho^) + |V^|^2/2,
//   n . F = [m, m V^ + p1^ n, m H^],  m = rho^ V^ . n.
// Logarithmic mean from the nodal logs: (a - b)/(log a - log b), or, for
// u = ((a-b)/(a+b))^2 < 1e-2, (a+b)/2 / (1 + u/3 + u^2/5 + ... + u^8/17)
// (the next term is below 1e-18).
// ---------------------------------------------------------------------------
template <typename T, int D>
struct IRNode {
  T z1, zn, l1, ln;  // sqrt(rho/p), sqrt(rho p) and their logs
  T b;               // rho/p (float64 nodes)
  T V[D];
};

template <typename T, int D>
__device__ __forceinline__ void ir_node(const Node<T, D>& n, IRNode<T, D>& z) {
  T lr;
  if constexpr (std::is_same<T, double>::value) {
    // sqrt(rho/p): quotient and root from the iterated reciprocals, each with
    // one correction step (as accurate as the division and the square root;
    // an error here enters every pair of the node)
    const double ip = rcp64(n.p), b0 = n.rho * ip, b = fma(fma(-b0, n.p, n.rho), ip, b0);
    const double r = rsqrt64(b), s0 = b * r;
    z.b = b;
    z.z1 = fma(fma(-s0, s0, b), 0.5 * r, s0);
    z.zn = n.p * z.z1;
    lr = log_abs(n.rho);
  } else {
    z.z1 = t_sqrt(n.rho / n.p);
    z.zn = n.p * z.z1;
    lr = t_log(n.rho);
  }
  T lp = n.lnp;
  if constexpr (std::is_same<T, double>::value) lp = log_abs(n.p);
  z.l1 = T(0.5) * (lr - lp);
  z.ln = T(0.5) * (lr + lp);
#pragma unroll
  for (int i = 0; i < D; ++i) z.V[i] = n.V[i];
}

template <typename T>
__device__ __forceinline__ T log_mean(T a, T b, T la, T lb) {
  T s = a + b;
  T f = (a - b) / s;
  T u = f * f;
  if (u < T(1e-2)) {
    T q = T(1.0 / 17.0);
    q = q * u + T(1.0 / 15.0);
    q = q * u + T(1.0 / 13.0);
    q = q * u + T(1.0 / 11.0);
    q = q * u + T(1.0 / 9.0);
    q = q * u + T(1.0 / 7.0);
    q = q * u + T(1.0 / 5.0);
    q = q * u + T(1.0 / 3.0);
    q = q * u + T(1.0);
    return T(0.5) * s / q;
  }
  return (a - b) / (la - lb);
}

// Pair averages of the Ismail-Roe flux (shared with its dissipation)
template <typename T, int D>
struct IRAvg {
  T rh, p1, p2, vv;  // rho^, p1^, p2^, |V^|^2
  T irh, hq;         // 1/rho^ and gam/(gam-1) p2^/rho^ (float64; p2 is not formed)
  T Vh[D];
};

// Pair averages in float64: {.}_log of z_nc and 1/{.}_log of z_1 from the
// arithmetic means, log mean = {.}/q(u), u = ((a - b)/(a + b))^2, and from the
// nodal logarithms above the switch; three reciprocals by iteration instead of
// five divisions.  Volume kernel, 8,192 triangles p 2: 170 -> 95 us.
template <int D, typename C>
__device__ __forceinline__ void ir_avg(const IRNode<double, D>& k, const IRNode<double, D>& v, const C& c,
                                       IRAvg<double, D>& a) {
  const double s1 = k.z1 + v.z1, sn = k.zn + v.zn, a1 = 0.5 * s1, an = 0.5 * sn;
  const double ia1 = rcp64(a1), isn = rcp64(sn);
  const double d1 = k.z1 - v.z1, dn = k.zn - v.zn, f1 = 0.5 * (d1 * ia1), fn = dn * isn;
  const double u1 = f1 * f1, un = fn * fn;
  constexpr unsigned long long SWITCH = 0x3F847AE147AE147BULL;  // 1e-2
  double q1, Ln;  // {z_1}/{z_1}_log, {z_nc}_log
  if (fm::abs_below(u1, SWITCH))
    q1 = im::atanhc(im::small_to_fixed(u1));
  else
    q1 = a1 * (k.l1 - v.l1) / d1;
  if (fm::abs_below(un, SWITCH))
    Ln = an * im::inv_atanhc(im::small_to_fixed(un));
  else
    Ln = dn / (k.ln - v.ln);
  a.vv = 0.0;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    a.Vh[i] = 0.5 * (k.z1 * k.V[i] + v.z1 * v.V[i]) * ia1;
    a.vv += a.Vh[i] * a.Vh[i];
  }
  a.rh = a1 * Ln;
  a.irh = ia1 * rcp64(Ln);
  a.p1 = an * ia1;
  // p2^/rho^ = (gam+1)/(2 gam) / ({z_1}_log {z_1}) + (gam-1)/(2 gam) p1^/rho^;
  // 1/{z_1}^2 corrected to its last bit (the enthalpy is the largest term)
  const double x = ia1 * ia1, e1 = fma(-a1, ia1, 1.0), i2 = fma(x, e1 + e1, x);
  a.hq = fma(c.ir_a, q1 * i2, c.ir_b * (a.p1 * a.irh));
}

template <typename T, int D, typename C>
__device__ __forceinline__ void ir_avg_t(const IRNode<T, D>& k, const IRNode<T, D>& v, const C& c, IRAvg<T, D>& a) {
  if constexpr (std::is_same<T, double>::value) {
    ir_avg<D>(k, v, c, a);
    return;
  }
  T a1 = T(0.5) * (k.z1 + v.z1), an = T(0.5) * (k.zn + v.zn);
  T L1 = log_mean<T>(k.z1, v.z1, k.l1, v.l1), Ln = log_mean<T>(k.zn, v.zn, k.ln, v.ln);
  T ia1 = t_rcp(a1);
  a.vv = T(0);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    a.Vh[i] = T(0.5) * (k.z1 * k.V[i] + v.z1 * v.V[i]) * ia1;
    a.vv += a.Vh[i] * a.Vh[i];
  }
  a.rh = a1 * Ln;
  a.p1 = an * ia1;
  a.p2 = (c.gam + T(1)) / (T(2) * c.gam) * (Ln / L1) + (c.gam - T(1)) / (T(2) * c.gam) * a.p1;
}

template <typename T, int D, typename C>
__device__ __forceinline__ void ir_flux_dir(const IRAvg<T, D>& a, const C& c, const T* nu, T* F) {
  T vn = T(0);
#pragma unroll
  for (int i = 0; i < D; ++i) vn += a.Vh[i] * nu[i];
  T Hh;
  if constexpr (std::is_same<T, double>::value)
    Hh = a.hq + 0.5 * a.vv;
  else
    Hh = c.gam * c.inv_gm1 * a.p2 / a.rh + T(0.5) * a.vv;
  T m = a.rh * vn;
  F[0] = m;
#pragma unroll
  for (int j = 0; j < D; ++j) F[1 + j] = m * a.Vh[j] + a.p1 * nu[j];
  F[D + 1] = m * Hh;
}

// Standard entropy variables w = [(gam - s)/(gam-1) - rho|V|^2/(2p), rho V/p,
// -rho/p], s = log p - gam log rho, from the nodal state and its IR node.
template <typename T, int D, typename C>
__device__ __forceinline__ void std_entropy_vars(const Node<T, D>& n, const IRNode<T, D>& z, const C& c, T* w) {
  T b;
  if constexpr (std::is_same<T, double>::value)
    b = z.b;
  else
    b = n.rho / n.p;
  const T lr = z.l1 + z.ln, lp = z.ln - z.l1;  // log rho, log p
  w[0] = (c.gam - (lp - c.gam * lr)) * c.inv_gm1 - T(0.5) * b * n.v2;
#pragma unroll
  for (int i = 0; i < D; ++i) w[1 + i] = b * n.V[i];
  w[D + 1] = -b;
}

// Standard entropy variables of a node (log rho formed here; the comparator's
// viscous terms, whose nodes carry no parameter-vector logs).
template <typename C, int D>
__device__ __forceinline__ void std_entropy_vars_node(const Node<double, D>& n, const C& c, double* w) {
  const double ip = rcp64(n.p), b0 = n.rho * ip, b = fma(fma(-b0, n.p, n.rho), ip, b0);
  const double s = log_abs(n.p) - c.gam * log_abs(n.rho);
  w[0] = (c.gam - s) * c.inv_gm1 - 0.5 * b * n.v2;
#pragma unroll
  for (int i = 0; i < D; ++i) w[1 + i] = b * n.V[i];
  w[D + 1] = -b;
}

// Matrix dissipation of the comparator (not printed in the paper; the form of
// Eq. (69) carried over to the standard entropy), applied to dw = jump of the
// standard entropy variables, n a unit normal:
//   out = sum_k |lambda_k| T_k r_k (r_k . dw) + |V^.n| p^ B^T (I - n n^T) B dw
// at rho^, V^, p^ = p1^; r_k the acoustic and entropy columns of Eq. (80),
// T = rho^/(2 gam), (gam-1) rho^/gam, rho^/(2 gam); B dw = dw_m + V^ dw_E.
template <typename T, int D, typename C>
__device__ __forceinline__ void ir_diss_apply(const IRAvg<T, D>& a, const C& c, const T* n, const T* dw, T* out) {
  constexpr int NC = D + 2;
  T ah, a2;
  if constexpr (std::is_same<T, double>::value) {
    a2 = c.gam * a.p1 * a.irh;
    ah = a2 * rsqrt64(a2);
  } else {
    ah = t_sqrt(c.gam * a.p1 / a.rh);
    a2 = ah * ah;
  }
  T Hh = a2 * c.inv_gm1 + T(0.5) * a.vv;
  T vn = T(0);
#pragma unroll
  for (int i = 0; i < D; ++i) vn += a.Vh[i] * n[i];
  // r . dw for the three columns
  T vdm = T(0), ndm = T(0);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    vdm += a.Vh[i] * dw[1 + i];
    ndm += n[i] * dw[1 + i];
  }
  const T e = dw[NC - 1];
  const T base = dw[0] + vdm;
  T ym = (base - ah * ndm + (Hh - ah * vn) * e) * (t_abs(vn - ah) * a.rh * c.s_ac);
  T y0 = (base + T(0.5) * a.vv * e) * (t_abs(vn) * a.rh * c.gm1_gam);
  T yp = (base + ah * ndm + (Hh + ah * vn) * e) * (t_abs(vn + ah) * a.rh * c.s_ac);
  out[0] = ym + y0 + yp;
  // shear part
  T y[D], yn = T(0);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    y[i] = dw[1 + i] + a.Vh[i] * e;
    yn += n[i] * y[i];
  }
  const T sh = t_abs(vn) * a.p1;
  T vpy = T(0);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    const T py = sh * (y[i] - n[i] * yn);
    out[1 + i] = ym * (a.Vh[i] - ah * n[i]) + y0 * a.Vh[i] + yp * (a.Vh[i] + ah * n[i]) + py;
    vpy += a.Vh[i] * py;
  }
  out[NC - 1] = ym * (Hh - ah * vn) + y0 * (T(0.5) * a.vv) + yp * (Hh + ah * vn) + vpy;
}

}  // namespace esplit
