// rslb_device.cuh -- device building blocks of the R-SLB step (sm_103a).
//
// Landau matching and the f^eq expansion coefficients, templated on the working precision.  Used by the Sod and Bjorken kernels.
#pragma once

#include <cfloat>
#include <cstdint>
#include <cuda_runtime.h>

namespace rslb {

constexpr int kMaxM = 13;    // N_Omega <= 12
constexpr int kAeqNodes = 32;  // Gauss-Legendre nodes for the a_{l,m} integrals

template <typename T> struct Prec;
template <> struct Prec<float> {
  static __device__ __forceinline__ float tiny() { return FLT_MIN; }
  static __device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
};
template <> struct Prec<double> {
  static __device__ __forceinline__ double tiny() { return DBL_MIN; }
  static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
};

__device__ __forceinline__ float dev_exp(float x) { return expf(x); }
__device__ __forceinline__ double dev_exp(double x) { return exp(x); }
__device__ __forceinline__ float dev_expm1(float x) { return expm1f(x); }
__device__ __forceinline__ double dev_expm1(double x) { return expm1(x); }

// ---------------------------------------------------------------------------
// Landau frame of the 1-D stress tensor (Sec. II E, Eqs. E_landau, u_landau),
// in FP64, from the five direct sums
//   Np = sum f(1+xi), Nm = sum f(1-xi), Ap = sum f p (1+xi)^2,
//   Am = sum f p (1-xi)^2, D = sum f p (1-xi^2).
// With a = sqrt(Ap), b = sqrt(Am) the discriminant of Eq. E_landau is
// (T^tt+T^zz)^2 - 4(T^tz)^2 = Ap*Am, so
//   E = (D + a b)/2,  beta = (a - b)/(a + b),  gamma = (a + b)/(2 sqrt(ab)),
//   n = gamma (N^t - beta N^z) = (b Np + a Nm)/(2 sqrt(ab)),
// which is algebraically identical to the printed formulas and has no
// cancellation as |beta| -> 1 when f >= 0.
// ---------------------------------------------------------------------------
struct LandauOut {
  double n, E, T, beta, gamma, u;  // u = gamma |beta|
  double ub;                       // gamma beta (signed)
  bool ok;
};

// 1/x and 1/sqrt(x) in FP64 from the 20-bit hardware seeds and one step of
// Householder's third-order iteration (e = 1 - x y or 1 - x y^2; the residual
// is of order e^3 < 2^-57, so the result is within about an ulp).  GB300 issues
// ~2 FP64 lane operations per SM and cycle, so these 3 and 5 operations
// replace the ~10-20 of the IEEE division and square root.  x must be a
// positive normal number; other inputs give inf or NaN, which the callers'
// range checks reject.
__device__ __forceinline__ double rcp64(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double rsqrt64(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x * y, y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

__device__ __forceinline__ LandauOut landau_factored(double Np, double Nm, double Ap,
                                                     double Am, double D) {
  LandauOut o;
  const double a = Ap * rsqrt64(Ap), b = Am * rsqrt64(Am);  // square roots
  const double ab = a * b, apb = a + b, amb = a - b;
  const double h = 0.5 * rsqrt64(ab);  // 1/(2 sqrt(ab))
  o.E = fma(0.5, ab, 0.5 * D);
  o.beta = amb * rcp64(apb);
  o.gamma = apb * h;
  o.ub = amb * h;
  o.u = fabs(o.ub);
  o.n = fma(b, Np, a * Nm) * h;
  o.T = o.E * rcp64(3.0 * o.n);
  // Ap, Am, E, n positive, normal and finite and |gamma beta| < gamma, tested on the
  // bit patterns (an FP64 comparison costs as much as a product)
  auto good = [](double x) {
    return (unsigned)__double2hiint(x) - 0x00100000u < 0x7FE00000u;
  };
  o.ok = good(Ap) && good(Am) && good(o.E) && good(o.n) && good(o.gamma) &&
         __double_as_longlong(o.u) < __double_as_longlong(o.gamma);
  return o;
}

// ---------------------------------------------------------------------------
// f^eq expansion coefficients (Sec. III D, Eq. aeq_aux).  With u0 = cosh A,
// u = sinh A and the exact substitution u0 - u c = e^{-s}, s = A t:
//   a_{l,m} = n (l+1)(l+2)/(8 pi) (A/u) int_{-1}^{1} dt e^{2s}
//             (1 - theta e^{s})^l P_m(c(s)),
//   c(s) = (2 sinh^2(A/2) - expm1(-s))/u   (c = t when u = 0).
// The integrand is a short sum of exponentials; kAeqNodes Gauss-Legendre
// nodes give round-off accuracy for |beta| up to ~0.95.  This helper adds the
// contribution of one node to J3_m = int e^{2s} P_m, J4_m = int e^{3s} P_m,
// so that a_{0,m} = n (A/u) J3_m/(4 pi) and
// a_{1,m} = 3 n (A/u) (J3_m - theta J4_m)/(4 pi).
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void aeq_node(T t, T wt, T A, T sh2, T uinv, bool at_rest, int nm,
                                         T* J3, T* J4) {
  const T s = A * t;
  const T c = at_rest ? t : (sh2 - dev_expm1(-s)) * uinv;
  const T e1 = dev_exp(s);
  const T e2 = e1 * e1;
  const T w3 = wt * e2, w4 = w3 * e1;
  T p0 = T(1), p1 = c;
  J3[0] += w3;
  J4[0] += w4;
#pragma unroll
  for (int m = 1; m < kMaxM; ++m) {
    if (m < nm) {
      J3[m] += w3 * p1;
      J4[m] += w4 * p1;
      const T p2 = (T(2 * m + 1) * c * p1 - T(m) * p0) * T(1.0 / (m + 1));
      p0 = p1;
      p1 = p2;
    }
  }
}

// ---------------------------------------------------------------------------
// The same integrals by recurrence over m (stage kernels).  With z = 1/|beta|,
//   X3_m = (A/u) J3_m = int P_m(c) (u0 - u c)^{-3} dc,   X4_m likewise with -4,
// are the second and third derivatives of the Legendre function Q_m(z) up to
// a factor, i.e. the minimal solutions of
//   (m+2) D_{m-1} = (2m+1) z D_m - (m-1) D_{m+1},
//   (m+3) E_{m-1} = (2m+1) z E_m - (m-2) E_{m+1}
// (associated Legendre recurrence), so the downward recurrence from a large
// order (Miller's algorithm) is stable.  Writing D_m = beta^m S_m delta_m with
// S_{m-1} = S_{m+1} (m-1)/(m+2) leaves
//   delta_{m-1} = alpha_m delta_m - beta^2 delta_{m+1}
// (two operations per order), regular at beta = 0, and the same form for E; the
// norms are X3_0 = 2 u0 and X4_0 = 2 u0^2 + 2 u^2/3.  The starting order
// follows from the decay rate rho = (1 + sqrt(1 - beta^2))/|beta| of D_{m+1}/D_m;
// all m <= 12 agree with the integrals to 2e-15 (FP64; 9e-16 for m <= 5) and 2e-6 (FP32;
// 1e-6) of X_0, as a replay in numpy against 40 digits shows.
// ~20 orders of 4 operations replace 32 (16) nodes with an exp, an expm1 and
// 13 Legendre orders each.
// ---------------------------------------------------------------------------
constexpr int kAeqSteps = 128;  // largest starting order
struct AeqTab {
  double aD[kAeqSteps + 2], aE[kAeqSteps + 2];  // alpha_m of the two recurrences
  double sD[kMaxM + 1], sE[kMaxM + 1];          // S_m
  float aDf[kAeqSteps + 2], aEf[kAeqSteps + 2], sDf[kMaxM + 1], sEf[kMaxM + 1];
};
constexpr AeqTab make_aeq_tab() {
  AeqTab t{};
  double SD[kAeqSteps + 3] = {}, SE[kAeqSteps + 3] = {};
  SD[0] = SD[1] = SD[2] = 1.0;
  SE[0] = SE[1] = SE[2] = SE[3] = 1.0;
  for (int m = 2; m <= kAeqSteps + 1; ++m) SD[m + 1] = SD[m - 1] * (m + 2) / (m - 1);
  for (int m = 3; m <= kAeqSteps + 1; ++m) SE[m + 1] = SE[m - 1] * (m + 3) / (m - 2);
  for (int m = 2; m <= kAeqSteps + 1; ++m) t.aD[m] = (2.0 * m + 1) / (m + 2) * (SD[m] / SD[m - 1]);
  for (int m = 3; m <= kAeqSteps + 1; ++m) t.aE[m] = (2.0 * m + 1) / (m + 3) * (SE[m] / SE[m - 1]);
  for (int m = 0; m <= kMaxM; ++m) {
    t.sD[m] = SD[m];
    t.sE[m] = SE[m];
    t.sDf[m] = float(SD[m]);
    t.sEf[m] = float(SE[m]);
  }
  for (int m = 0; m <= kAeqSteps + 1; ++m) {
    t.aDf[m] = float(t.aD[m]);
    t.aEf[m] = float(t.aE[m]);
  }
  return t;
}
static __constant__ AeqTab c_aeq = make_aeq_tab();

template <typename T>
__device__ __forceinline__ T aeq_alpha(bool e, int m);
template <>
__device__ __forceinline__ float aeq_alpha<float>(bool e, int m) {
  return e ? c_aeq.aEf[m] : c_aeq.aDf[m];
}
template <>
__device__ __forceinline__ double aeq_alpha<double>(bool e, int m) {
  return e ? c_aeq.aE[m] : c_aeq.aD[m];
}
template <typename T>
__device__ __forceinline__ T aeq_scale(bool e, int m);
template <>
__device__ __forceinline__ float aeq_scale<float>(bool e, int m) {
  return e ? c_aeq.sEf[m] : c_aeq.sDf[m];
}
template <>
__device__ __forceinline__ double aeq_scale<double>(bool e, int m) {
  return e ? c_aeq.sE[m] : c_aeq.sD[m];
}

// Starting order for truncation nm (>= 4 here) at u = gamma |beta|, and the
// starting ratio delta_{M+1}/delta_M ~ 1/(1 + 1/gamma).  The truncation error
// falls by rho^-2 per order: 17/ln(rho) orders for FP64, 8/ln(rho) for FP32.
// Past kAeqSteps (FP32: 96, so that the growth of at most 2 per order stays
// in range) the caller uses the quadrature.
template <typename T>
__device__ __forceinline__ int aeq_start(float u, float gamma, int nm4, float* r) {
  *r = gamma / (gamma + 1.f);
  const float l2 = fmaxf(-__log2f(fmaxf(u / (gamma + 1.f), 1e-30f)), 1e-6f);  // log2(rho)
  const float need = (sizeof(T) == 8 ? 24.53f : 11.55f) / l2;
  const int M = nm4 + (int)fminf(need, 4096.f);
  return M;
}
template <typename T>
__host__ __device__ constexpr int aeq_max_start() { return sizeof(T) == 8 ? kAeqSteps : 96; }

// delta_m for 2 <= m < nm4 (nm4 = max(nm, 4)), and delta_1 for the D chain,
// handed to put(m, delta).  All lanes of the warp loop from the largest
// starting order Mw among them, so that alpha is read uniformly, but each starts
// at its own M: a cell's result does not depend on its neighbours.
template <typename T, typename Put>
__device__ __forceinline__ void aeq_chain(bool e_chain, T b2, T r, int M, int Mw, int nm4, Put put) {
  T d1 = r, d0 = T(1);  // delta_{m+1}, delta_m
  for (int m = Mw; m >= nm4; --m) {
    const T dn = fma(-b2, d1, aeq_alpha<T>(e_chain, m) * d0);
    const bool on = m <= M;
    d1 = on ? d0 : d1;
    d0 = on ? dn : d0;
  }
#pragma unroll
  for (int m = kMaxM - 1; m >= 3; --m)
    if (m < nm4) {
      put(m, d0);
      const T dn = fma(-b2, d1, aeq_alpha<T>(e_chain, m) * d0);
      d1 = d0;
      d0 = dn;
    }
  put(2, d0);
  if (!e_chain) put(1, fma(-b2, d1, aeq_alpha<T>(false, 2) * d0));
}

// Both chains side by side: delta_m in D[m], eps_m in E[m] for m < min(nm4, MAXM).
template <typename T, int MAXM>
__device__ __forceinline__ void aeq_chains(T b2, T r, int M, int Mw, int nm4, T* D, T* E) {
  T d1 = r, d0 = T(1), e1 = r, e0 = T(1);
  for (int m = Mw; m >= nm4; --m) {
    const T dn = fma(-b2, d1, aeq_alpha<T>(false, m) * d0);
    const T en = fma(-b2, e1, aeq_alpha<T>(true, m) * e0);
    const bool on = m <= M;
    d1 = on ? d0 : d1;
    d0 = on ? dn : d0;
    e1 = on ? e0 : e1;
    e0 = on ? en : e0;
  }
#pragma unroll
  for (int m = MAXM - 1; m >= 3; --m)
    if (m < nm4) {
      D[m] = d0;
      E[m] = e0;
      const T dn = fma(-b2, d1, aeq_alpha<T>(false, m) * d0);
      const T en = fma(-b2, e1, aeq_alpha<T>(true, m) * e0);
      d1 = d0;
      d0 = dn;
      e1 = e0;
      e0 = en;
    }
  D[2] = d0;
  E[2] = e0;
  D[1] = fma(-b2, d1, aeq_alpha<T>(false, 2) * d0);
}

__device__ __forceinline__ double fast_inv(double x) { return rcp64(x); }
__device__ __forceinline__ float fast_inv(float x) {  // 1 ulp
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// The integrals X3_m, X4_m of one cell by the 32-node rule, for |beta| so close
// to 1 that the recurrence would need more than its table (u beyond ~7 (FP64)
// or ~11 (FP32)): the truncated f^eq is strongly negative there, so no flow
// the method can follow reaches this; kept for the stray cell that does.
template <typename T>
__device__ __noinline__ void aeq_far(const double* __restrict__ gl_t,
                                     const double* __restrict__ gl_w, T u, T sh2, int nm, T* X) {
  T J3[kMaxM], J4[kMaxM];
  for (int m = 0; m < kMaxM; ++m) { J3[m] = T(0); J4[m] = T(0); }
  const T A = asinh(u), uinv = T(1) / u;
  for (int i = 0; i < kAeqNodes; ++i)
    aeq_node<T>(T(gl_t[i]), T(gl_w[i]), A, sh2, uinv, false, nm, J3, J4);
  for (int m = 0; m < nm; ++m) {
    X[m] = J3[m] * (A * uinv);
    X[kMaxM + m] = J4[m] * (A * uinv);
  }
}

// What the coefficients of one cell need of its Landau frame (n = 0: none).
template <typename T>
struct AeqCell {
  T n, T_, gamma, ub;  // ub = gamma beta
};

// c_{k,m} = (m + 1/2) q^m [p3_m + L1_k (p3_m - p4_m)] of one cell (c_{k,m} as in
// aeq_node's comment): after this D[m], E[m] (m < nm <= MAXM) hold the chains
// relative to their norms, so that p3_m = A3 S_m D[m], p4_m = A4 S_m E[m].
// mask holds the lanes that call this together.
template <typename T>
struct AeqScalars {
  T A3, A4, q;
};
template <typename T, int MAXM>
__device__ __forceinline__ AeqScalars<T> aeq_cell(const AeqCell<T>& c, int nm, unsigned mask,
                                                  const double* __restrict__ gl_t,
                                                  const double* __restrict__ gl_w, T* D, T* E) {
  static_assert(MAXM >= 4, "the chains end at order 3");
  const int nm4 = max(nm, 4);
  const T u = fabs(c.ub);
  float r;
  const int M = aeq_start<T>(float(u), float(c.gamma), nm4, &r);
  const bool far = M > aeq_max_start<T>();
  const int Mc = min(M, aeq_max_start<T>()), Mw = __reduce_max_sync(mask, Mc);
  AeqScalars<T> o;
  o.q = c.ub * fast_inv(c.gamma);  // beta
  const T b2 = far ? T(0) : o.q * o.q;
#pragma unroll
  for (int m = 0; m < MAXM; ++m) { D[m] = T(0); E[m] = T(0); }
  aeq_chains<T, MAXM>(b2, T(r), Mc, Mw, nm4, D, E);
  // relative to the norms X3_0 = 2 u0 and X4_0 = (2/3) u0^2 (3 + beta^2), so the
  // isotropic part of f^eq carries the roundings of A3 and A4 only
  const T rD = fast_inv(D[1]), rE = fast_inv(fma(T(0.25), b2, T(0.75)) * E[2]);
  o.A3 = T(0.5) * c.n * c.gamma;
  o.A4 = o.A3 * (c.T_ * c.gamma) * fma(T(1.0 / 3.0), b2, T(1));
  D[0] = D[1] = T(1);
  E[1] = E[2] * rE;
  E[0] = T(1);
#pragma unroll
  for (int m = 2; m < MAXM; ++m) {
    D[m] *= rD;
    E[m] *= rE;
  }
  if (far) {
    T X[2 * kMaxM];
    aeq_far<T>(gl_t, gl_w, u, u * u / (c.gamma + T(1)), nm, X);
#pragma unroll
    for (int m = 0; m < MAXM; ++m)
      if (m < nm) {
        D[m] = X[m] / aeq_scale<T>(false, m);
        E[m] = X[kMaxM + m] / aeq_scale<T>(true, m);
      }
    o.A3 = T(0.25) * c.n;
    o.A4 = T(0.25) * c.n * c.T_;
    o.q = c.ub < T(0) ? T(-1) : T(1);
  }
  return o;
}

}  // namespace rslb
