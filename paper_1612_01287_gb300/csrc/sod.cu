// sod.cu -- fused RK-stage kernel of the R-SLB Sod shock tube (sm_103a).
//
// One CTA owns a tile of B consecutive cells (128, 64, 32 or 16 for FP32, 16, 8,
// 4 or 2 for FP64) and all V velocities.  A stage (Eq. rk3) is one launch:
//   1. the tile plus a 4-cell halo on each side is staged in shared memory
//      with 16-byte cp.async copies (velocity-major rows; boundary tiles map
//      out-of-domain cells through the boundary condition);
//   2. moments: the five sums of the factored Landau form, from three sums per
//      radial node.  A thread owns one cell and a slice of the rows (blocks of
//      four rows, Kahan-compensated in FP32); the slices of a cell meet by
//      shuffles and in shared memory (double-floats in FP32);
//   3. per cell: Landau matching in FP64 (Sec. II E), the relaxation time, and
//      the f^eq expansion coefficients (Sec. III D) by a downward recurrence
//      over the Legendre order;
//   4. per (velocity, cell): the WENO5 flux difference (Sec. III F) along the
//      row, written in terms of first and second differences of f so
//      that a sliding window shares them between neighbouring faces; f^eq
//      from the per-cell coefficients; Anderson-Witting relaxation
//      (Eq. L_Sod); the RK combination.  Rows are visited negative-xi first so
//      that the upwind direction is uniform within a warp; with few
//      velocities each row is split into segments of B/2 .. B/8 cells so that
//      enough threads have work;
//   5. vectorised, coalesced store of the tile interior (with the f_n term of
//      stages 2 and 3).
// Shared-memory rows have a pitch whose 16-byte count is odd, so the 16-byte
// accesses of eight consecutive rows fall in distinct bank groups.
//
// What bounds it: FP64, the FP64 pipe of the SM (~2 lane operations per cycle):
// ~61 pipe slots per cell and velocity here (moments 4.5, faces 30, differences
// 7, f^eq 6, update 7, the rest halo and idle lanes), 99 with five moment sums,
// IEEE divisions, FP64 maxima and predicated-off orders.  65536 x 600: 4.23 ms
// per stage (7.34 before); 256 x 60 on 2-cell tiles: 18 us (79 on 16-cell
// tiles with the quadrature for a_{l,m}).  FP32: latency.  With few velocities
// that of the per-cell phases (V = 24: FP64 pipe 15%, FMA 12%, most warps at a
// barrier while the cells' FP64 runs), else of the sweep, whose code also has to
// fit the instruction cache (V = 60: FMA pipe 18%, issue slots 31%).
#include <algorithm>
#include <type_traits>

#include "rslb_device.cuh"
#include "sod.cuh"

namespace rslb {

constexpr int kMaxQL = 8;
constexpr int kHalo = 4;

template <typename T> struct V16;
template <> struct V16<float> {
  using type = float4;
  static constexpr int n = 4;
};
template <> struct V16<double> {
  using type = double2;
  static constexpr int n = 2;
};

template <typename T>
__host__ __device__ constexpr int tile_pitch(int W) {
  // smallest P >= W with P a multiple of the 16-byte vector and P/vector odd
  constexpr int n = V16<T>::n;
  int p = (W + n - 1) / n;
  if (p % 2 == 0) ++p;
  return p * n;
}

template <typename T>
__host__ __device__ inline int coef_pitch(int nm) {
  constexpr int n = V16<T>::n;
  return (nm + n - 1) / n * n;
}

// Shared-memory carve-up of one CTA (all offsets 16-byte aligned).  np partial
// slots of the moment sums follow the fixed part; with np = 0 the groups add
// into msum one after another.
template <typename T>
struct SodSmem {
  size_t tile, outb, msum, cell, coef, gco, part, total;
  __host__ __device__ SodSmem(int V, int B, int QL, int nm, bool seg, int np) {
    auto al = [](size_t x) { return (x + 15) & ~size_t(15); };
    const int P = tile_pitch<T>(B + 2 * kHalo);
    tile = 0;
    outb = al(sizeof(T) * (size_t)V * P);
    msum = outb + (seg ? al(sizeof(T) * (size_t)V * B) : 0);
    cell = msum + al(sizeof(double) * 5 * B);
    coef = cell + al(sizeof(double) * 8 * B);
    gco = coef + al(sizeof(T) * (size_t)QL * B * coef_pitch<T>(nm));
    part = gco + al(sizeof(T) * 2 * B);
    total = part + al(sizeof(double) * 5 * (size_t)np * B);
  }
};

__device__ __forceinline__ void report_error(int* err, int code, int cell) {
  if (atomicCAS(err, 0, code) == 0) err[1] = cell;
}

__device__ __forceinline__ float fast_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_all;\n" ::);
}

template <typename T>
__device__ __forceinline__ T load_cell(const T* __restrict__ fin, const SodGeom& g,
                                       const SodTables<T>& tb, int v, int s) {
  if (s >= 0 && s < g.Z) return fin[(size_t)v * g.ldz + s];
  if (g.bc == kBcPeriodic) {
    int sp = s % g.Z;
    if (sp < 0) sp += g.Z;
    return fin[(size_t)v * g.ldz + sp];
  }
  if (g.bc == kBcOutflow) return fin[(size_t)v * g.ldz + (s < 0 ? 0 : g.Z - 1)];
  return s < 0 ? tb.ghostL[v] : tb.ghostR[v];
}

// One thread's share of the moments of one cell.  With a = sum f (1+xi)^2,
// b = sum f (1-xi)^2 and d = sum f (1-xi^2) over the polar nodes of one radial
// node p, all with non-negative weights,
//   N+- = sum_k ({a, b}_k + d_k)/2,  A+- = sum_k p_k {a, b}_k,  D = sum_k p_k d_k
// ((1 +- xi)^2 + (1 - xi^2) = 2 (1 +- xi)): three products per velocity instead
// of five, the rest once per radial node (flush).
template <typename T> struct Moments;
template <> struct Moments<double> {
  double S[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  double a = 0.0, b = 0.0, d = 0.0;
  __device__ __forceinline__ void row(double f, const double* w) {
    const double2 w01 = __ldg(reinterpret_cast<const double2*>(w));
    a = fma(f, w01.x, a);
    b = fma(f, w01.y, b);
    d = fma(f, __ldg(w + 2), d);
  }
  __device__ __forceinline__ void block() {}
  __device__ __forceinline__ void flush(const double* pk) {
    const double p = pk[0];
    S[0] = fma(0.5, a + d, S[0]);
    S[1] = fma(0.5, b + d, S[1]);
    S[2] = fma(p, a, S[2]);
    S[3] = fma(p, b, S[3]);
    S[4] = fma(p, d, S[4]);
    a = b = d = 0.0;
  }
  __device__ __forceinline__ void merge_xor(int off, unsigned mask) {
#pragma unroll
    for (int q = 0; q < 5; ++q) S[q] += __shfl_xor_sync(mask, S[q], off);
  }
  __device__ __forceinline__ void put(double* slot, int B, bool add) const {
#pragma unroll
    for (int q = 0; q < 5; ++q) slot[q * B] = add ? slot[q * B] + S[q] : S[q];
  }
  static __device__ __forceinline__ double total(const double* slot, int B5, int n) {
    double s = slot[0];
    for (int i = 1; i < n; ++i) s += slot[(size_t)i * B5];
    return s;
  }
};
// FP32: blocks of four rows, Kahan-compensated across blocks; the radial sums
// and the groups are added as double-floats (error-free TwoSum and products).
template <> struct Moments<float> {
  float H[5] = {0.f, 0.f, 0.f, 0.f, 0.f}, L[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
  float s[3] = {0.f, 0.f, 0.f}, c[3] = {0.f, 0.f, 0.f}, k[3] = {0.f, 0.f, 0.f};
  static __device__ __forceinline__ void two_sum(float& h, float& l, float x) {
    const float t = h + x, bp = t - h;
    l += (h - (t - bp)) + (x - bp);
    h = t;
  }
  __device__ __forceinline__ void row(float f, const float* w) {
    const float4 w4 = __ldg(reinterpret_cast<const float4*>(w));
    k[0] = fmaf(f, w4.x, k[0]);
    k[1] = fmaf(f, w4.y, k[1]);
    k[2] = fmaf(f, w4.z, k[2]);
  }
  __device__ __forceinline__ void block() {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const float y = k[q] - c[q];
      const float t = s[q] + y;
      c[q] = (t - s[q]) - y;
      s[q] = t;
      k[q] = 0.f;
    }
  }
  __device__ __forceinline__ void flush(const float* pk) {
    block();
    const float ph = pk[0], pl = pk[1];
    two_sum(H[0], L[0], 0.5f * s[0]);
    two_sum(H[0], L[0], 0.5f * s[2]);
    L[0] -= 0.5f * (c[0] + c[2]);
    two_sum(H[1], L[1], 0.5f * s[1]);
    two_sum(H[1], L[1], 0.5f * s[2]);
    L[1] -= 0.5f * (c[1] + c[2]);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const float x = ph * s[q];
      two_sum(H[2 + q], L[2 + q], x);
      L[2 + q] += fmaf(ph, s[q], -x) + (pl * s[q] - ph * c[q]);
      s[q] = c[q] = 0.f;
    }
  }
  __device__ __forceinline__ void merge_xor(int off, unsigned mask) {
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const float h = __shfl_xor_sync(mask, H[q], off), l = __shfl_xor_sync(mask, L[q], off);
      two_sum(H[q], L[q], h);
      L[q] += l;
    }
  }
  __device__ __forceinline__ void put(double* slot, int B, bool add) const {
    float2* f = reinterpret_cast<float2*>(slot);
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      float2 v = make_float2(H[q], L[q]);
      if (add) {
        v = f[q * B];
        two_sum(v.x, v.y, H[q]);
        v.y += L[q];
      }
      f[q * B] = v;
    }
  }
  static __device__ __forceinline__ double total(const double* slot, int B5, int n) {
    const float2* f = reinterpret_cast<const float2*>(slot);
    float2 v = f[0];
    for (int i = 1; i < n; ++i) {
      const float2 x = f[(size_t)i * B5];
      two_sum(v.x, v.y, x.x);
      v.y += x.y;
    }
    return (double)v.x + (double)v.y;
  }
};

// ---------------------------------------------------------------------------
// WENO5 face correction in difference form.
// For the upwind-ordered values (a, b, c, d, e) of Sec. III F with first
// differences D0 = b-a, D1 = c-b, D2 = d-c, D3 = e-d and second differences
// S1 = a-2b+c, S2 = b-2c+d, S3 = c-2d+e (K_q = 13/3 S_q^2):
//   4 sigma_1 = K_1 + (3 D1 - D0)^2, 4 sigma_2 = K_2 + (D1 + D2)^2,
//   4 sigma_3 = K_3 + (D3 - 3 D2)^2,
//   F^q = c + g_q/6 with g_1 = 5 D1 - 2 D0, g_2 = D1 + 2 D2, g_3 = 4 D2 - D3,
// so F = c + (omega . g)/6 (the common factor 4 of the indicators cancels in the
// weights).  With omega_q ~ delta_q / sigma_q^2 multiplied
// through by prod_p (sigma_p/sigma_max)^2, the limiting rules (i)-(iii) of
// the paper all reduce to "correction = 0" when every product vanishes (the
// g_q of the vanishing stencils are exactly zero there), and rule (iii) is
// the natural limit of the formula.  The products are taken in the ratio
// 1/3 : 2 : 1 of delta_q.  Returns (omega . g) (without the 1/6).  26 FP64
// operations per face; the scaling and the zero test are integer work on the
// high words, which the FP64 pipe (the FP64 kernel's limit) does not see.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void weno_scale(float& s1, float& s2, float& s3) {
  // the power of two at or below the maximum, from the exponent bits; a zero
  // or subnormal maximum gives the largest such power, which keeps zero
  // indicators zero and brings subnormal ones into range
  const float smax = fmaxf(s1, fmaxf(s2, s3));
  const float inv = __int_as_float(0x7F000000 - (__float_as_int(smax) & 0x7F800000));
  s1 *= inv;
  s2 *= inv;
  s3 *= inv;
}
__device__ __forceinline__ void weno_scale(double& s1, double& s2, double& s3) {
  // the same by subtracting the exponent of the maximum from the high words
  // (the indicators are >= 0, so their high words order like integers).  Words that
  // would fall below zero, zero indicators and subnormal ones become subnormal:
  // their squares are 0.
  const int h1 = __double2hiint(s1), h2 = __double2hiint(s2), h3 = __double2hiint(s3);
  const int sh = (max(h1, max(h2, h3)) & 0x7FF00000) - 0x3FF00000;
  auto shift = [&](int h) { return h < 0x00100000 ? 0 : max(h - sh, 0); };
  s1 = __hiloint2double(shift(h1), __double2loint(s1));
  s2 = __hiloint2double(shift(h2), __double2loint(s2));
  s3 = __hiloint2double(shift(h3), __double2loint(s3));
}
// num/den, 0 where den is below the smallest normal number (the reciprocals
// flush subnormal inputs, and a vanishing denominator means a vanishing correction)
__device__ __forceinline__ float weno_quotient(float num, float den) {
  return den > Prec<float>::tiny() ? num * fast_rcp(den) : 0.f;
}
__device__ __forceinline__ double weno_quotient(double num, double den) {
  return __double2hiint(den) >= 0x00100000 ? num * rcp64(den) : 0.0;
}

template <typename T>
__device__ __forceinline__ T weno_corr(T D0, T D1, T D2, T D3, T K1, T K2, T K3) {
  const T e1 = fma(T(3), D1, -D0), e2 = D1 + D2, e3 = fma(T(-3), D2, D3);
  T s1 = fma(e1, e1, K1), s2 = fma(e2, e2, K2), s3 = fma(e3, e3, K3);
  weno_scale(s1, s2, s3);
  const T t1 = s1 * s1, t2 = s2 * s2, t3 = s3 * s3;
  const T p13 = t1 * t3, n3 = t1 * t2;
  const T n2 = p13 + p13, n1 = t2 * t3 * T(1.0 / 3.0);
  const T den = (n3 + n2) + n1;
  // g_1 = 2 e1 - D1, g_2 = e2 + D2, g_3 = D2 - e3
  const T num = fma(n1, fma(T(2), e1, -D1), fma(n2, e2 + D2, n3 * (D2 - e3)));
  return weno_quotient(num, den);
}

// 16-byte chunk of a shared-memory row as scalars.
template <typename T>
__device__ __forceinline__ void ld_chunk(const T* p, T* out) {
  using VT = typename V16<T>::type;
  const VT v = *reinterpret_cast<const VT*>(p);
  if constexpr (V16<T>::n == 4) {
    out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w;
  } else {
    out[0] = v.x; out[1] = v.y;
  }
}
template <typename T>
__device__ __forceinline__ void st_chunk(T* p, const T* in) {
  using VT = typename V16<T>::type;
  VT v;
  if constexpr (V16<T>::n == 4) {
    v.x = in[0]; v.y = in[1]; v.z = in[2]; v.w = in[3];
  } else {
    v.x = in[0]; v.y = in[1];
  }
  *reinterpret_cast<VT*>(p) = v;
}

// ---------------------------------------------------------------------------
// Phase 4: sweep one row segment [i0, i0+SL) (local cells; tile element
// e = cell + kHalo) in chunks of VN cells with a sliding window of f over
// cells [i-4, i+VN+4) of the current chunk start i, and of the differences of
// J = xi f (rounded products, as the oracle takes them: the noise that the
// weights amplify then follows the oracle's more closely).  POS: xi > 0.
// Positive: face s+1/2 uses J_{s-2..s+2} with centre J_s:
//   (D0..D3) = Delta_{s-2..s+1}, (K1, K2, K3) = K_{s-1}, K_s, K_{s+1}.
// Negative: the mirror (J_{s+3}, ..., J_{s-1}) with centre J_{s+1}:
//   (D0..D3) = -Delta_{s+2}, -Delta_{s+1}, -Delta_s, -Delta_{s-1},
//   (K1, K2, K3) = K_{s+2}, K_{s+1}, K_s; weno_corr is odd in its differences,
//   so C is minus the value for the un-negated ones.
// (Delta_s = J_{s+1} - J_s, K_s = 13/3 (J_{s-1} - 2 J_s + J_{s+1})^2.)
// The flux difference of cell i is
//   POS: Delta_{i-1} + (C_{i+1/2} - C_{i-1/2})/6,
//   NEG: Delta_i     + (C_{i+1/2} - C_{i-1/2})/6,
// and c1 = dt/dz; gco holds (gamma, gamma beta) dt/tau; wpr (FP32) holds the row's
// weights of the first NO orders, NO >= MP.
// ---------------------------------------------------------------------------
template <typename T, bool POS, int SL, int NO>
__device__ __forceinline__ void sweep_segment(const T* row, T* orow, int i0, T xi, T c1,
                                              const T* wpr, const T* __restrict__ wp,
                                              int wstride, int MP, const T* __restrict__ ck,
                                              const T* __restrict__ gco) {
  constexpr int VN = V16<T>::n;
  constexpr int NW = VN + 2 * kHalo;  // window cells [i-4, i+VN+4)
  const T sixth = T(1) / T(6);
  const T k13 = T(13) / T(3);
  T R[NW];  // f at cells i-4+c
  T Dw[NW - 1], Kw[NW - 1];
  auto diffs = [&](int c0) {
#pragma unroll
    for (int c = 0; c < NW - 1; ++c)
      if (c >= c0) Dw[c] = Prec<T>::mul(xi, R[c + 1]) - Prec<T>::mul(xi, R[c]);
#pragma unroll
    for (int c = 1; c < NW - 1; ++c)
      if (c >= c0) {
        const T s2 = Dw[c] - Dw[c - 1];
        Kw[c] = (k13 * s2) * s2;
      }
  };
  auto face = [&](int wc) {  // the face right of window cell wc
    if constexpr (POS)
      return weno_corr<T>(Dw[wc - 2], Dw[wc - 1], Dw[wc], Dw[wc + 1], Kw[wc - 1], Kw[wc],
                          Kw[wc + 1]);
    else
      return weno_corr<T>(Dw[wc + 2], Dw[wc + 1], Dw[wc], Dw[wc - 1], Kw[wc + 2], Kw[wc + 1],
                          Kw[wc]);
  };
#pragma unroll
  for (int c = 0; c < NW; c += VN) ld_chunk<T>(row + i0 + c, R + c);
  Kw[0] = T(0);
  diffs(0);
  T Cl = face(kHalo - 1);
  // FP32: four chunks of straight-line code.  A whole row of them (two directions of
  // up to 64 cells) streams through the instruction cache: 65536 x 120, N_Omega = 5
  // 238 us per step against 334, 4000 x 8 33 against 45.
  constexpr int kUnroll = sizeof(T) == 4 ? 4 : SL / VN;
#pragma unroll kUnroll
  for (int t = 0; t < SL / VN; ++t) {
    const int i = i0 + t * VN;
    T out[VN];
#pragma unroll
    for (int c = 0; c < VN; ++c) {
      const int wc = kHalo + c;  // window index of cell i + c
      const T Cr = face(wc);
      const T dF = POS ? fma(Cr - Cl, sixth, Dw[wc - 1]) : fma(Cl - Cr, sixth, Dw[wc]);
      Cl = Cr;
      const T* cc = ck + (size_t)(i + c) * MP;
      // f^eq: a real loop over the orders in FP64 (an instruction that is
      // predicated off still takes its slot on the FP64 pipe; coefficients past
      // nm are zero, so any row of the weight table serves them), weights in
      // registers in FP32.
      T feq = T(0);
      if constexpr (sizeof(T) == 8) {
#pragma unroll 1
        for (int m0 = 0; m0 < MP; m0 += VN) {
          T cv[VN];
          ld_chunk<T>(cc + m0, cv);
#pragma unroll
          for (int q = 0; q < VN; ++q)
            feq = fma(cv[q], __ldg(wp + min(m0 + q, kMaxM - 1) * wstride), feq);
        }
      } else {
#pragma unroll
        for (int m0 = 0; m0 < NO; m0 += VN)
          if (m0 < MP) {
            T cv[VN];
            ld_chunk<T>(cc + m0, cv);
#pragma unroll
            for (int q = 0; q < VN; ++q) feq = fma(cv[q], wpr[m0 + q], feq);
          }
      }
      const T f = R[kHalo + c];
      const T rate = fma(-xi, gco[2 * (i + c) + 1], gco[2 * (i + c)]);
      out[c] = fma(-rate, f - feq, fma(-c1, dF, f));
    }
    if (t + 1 < SL / VN) {
      // slide the window by one chunk: load the chunk at cells i+VN+4 ..
#pragma unroll
      for (int c = 0; c < NW - VN; ++c) R[c] = R[c + VN];
#pragma unroll
      for (int c = 0; c < NW - 1 - VN; ++c) {
        Dw[c] = Dw[c + VN];
        Kw[c] = Kw[c + VN];
      }
      ld_chunk<T>(row + i + NW, R + NW - VN);  // tile element of cell i+VN+4 is i + NW
      diffs(NW - 1 - VN);
    }
    st_chunk<T>(orow + kHalo + i, out);
  }
}

template <typename T, int B, int NT>
__device__ __forceinline__ void sod_tile(const T* __restrict__ fin, const T* __restrict__ fn,
                                         T* fout, int stage, int* err, const SodGeom& g,
                                         const SodTables<T>& tb, const int* __restrict__ rowv,
                                         int nneg, int nseg, int np, int s0) {
  constexpr int VN = V16<T>::n;
  constexpr int W = B + 2 * kHalo;
  constexpr int P = tile_pitch<T>(W);
  constexpr int CH = B / VN;  // 16-byte chunks of interior cells
  constexpr bool kF64 = sizeof(T) == 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int V = g.V;
  const SodSmem<T> lay(V, B, g.QL, g.nm, nseg > 1, np);
  T* tile = reinterpret_cast<T*>(smem_raw + lay.tile);
  T* outb = (nseg > 1) ? reinterpret_cast<T*>(smem_raw + lay.outb) : nullptr;
  double* msum = reinterpret_cast<double*>(smem_raw + lay.msum);
  T* cellT = reinterpret_cast<T*>(smem_raw + lay.cell);
  T* coef = reinterpret_cast<T*>(smem_raw + lay.coef);
  T* gco = reinterpret_cast<T*>(smem_raw + lay.gco);
  double* part = np ? reinterpret_cast<double*>(smem_raw + lay.part) : msum;
  const int MP = coef_pitch<T>(g.nm);

  const int tid = threadIdx.x;
  const int lane = tid & 31;

  // ---- 1. stage tile + halo ----
  const bool interior = (s0 - kHalo >= 0) && (s0 + B + kHalo <= g.Z);
  if (interior) {
    constexpr int CPR = W / VN;  // chunks per row
    for (int idx = tid; idx < V * CPR; idx += NT) {
      const int v = idx / CPR, c = idx - v * CPR;
      cp_async16(tile + v * P + c * VN, fin + (size_t)v * g.ldz + (s0 - kHalo) + c * VN);
    }
    cp_async_wait_all();
  } else {
    for (int idx = tid; idx < V * W; idx += NT) {
      const int v = idx / W, e = idx - v * W;
      tile[v * P + e] = load_cell<T>(fin, g, tb, v, s0 - kHalo + e);
    }
  }
  __syncthreads();

  const bool collide = g.tau_mode != kTauNone;
  if (collide) {
    // ---- 2. moments: thread (cell c, row group gr); the group's rows are a
    // contiguous slice, so it meets at most two or three radial nodes ----
    {
      constexpr int G = NT / B;                    // row groups
      constexpr int WB = B < 32 ? B : 32;          // lanes per group in a warp
      constexpr int NS = NT / (B < 32 ? 32 : B);   // slots: groups after the in-warp merge
      const int c = tid % B, gr = tid / B;
      const bool work = gr < G;  // whole warps (B >= 32: NT - G B is a multiple of 32)
      if (work) {
        Moments<T> m;
        const int v1 = (int)((long long)V * (gr + 1) / G);
        int v = (int)((long long)V * gr / G);
        const T* col = tile + kHalo + c;
        while (v < v1) {
          const int k = v / g.Qx, ve = min(v1, (k + 1) * g.Qx);
          for (; v + 4 <= ve; v += 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) m.row(col[(v + u) * P], tb.m3 + 4 * (v + u));
            m.block();
          }
          for (; v < ve; ++v) m.row(col[v * P], tb.m3 + 4 * v);
          m.flush(tb.pk + 2 * k);
        }
#pragma unroll
        for (int off = WB; off < 32; off *= 2) m.merge_xor(off, 0xffffffffu);
        // slot sl of cell c; slots beyond np are added in later rounds
        const int sl = B < 32 ? tid / 32 : gr;
        const bool owner = B >= 32 || lane < B;
        if (np >= NS) {
          if (owner) m.put(part + (size_t)sl * 5 * B + c, B, false);
        } else {
          const int n = np ? np : 1;
          for (int r = 0; r * n < NS; ++r) {
            if (owner && sl / n == r) m.put(part + (size_t)(sl % n) * 5 * B + c, B, r > 0);
            __syncwarp();
            asm volatile("barrier.sync 1, %0;" ::"n"(NS * (B < 32 ? 32 : B)) : "memory");
          }
        }
      }
      __syncthreads();
      const int n = np >= NS ? NS : (np ? np : 1);
      for (int e = tid; e < 5 * B; e += NT) {
        // np = 0 shares msum: each element is read and written by one thread
        const double t = Moments<T>::total(part + e, 5 * B, n);
        msum[e] = t;
      }
    }
    __syncthreads();

    // ---- 3. Landau matching (FP64), relaxation time and f^eq coefficients.
    // FP32: one thread per cell does all.  FP64: two lanes per cell of warp 0
    // run the two recurrences side by side (an FP64 instruction costs a
    // sub-partition ~64 cycles however many lanes are active), and the
    // coefficients follow by (cell, m) over the CTA ----
    constexpr bool kCanSplit = kF64 && 2 * B <= 32;
    const bool split = kCanSplit && g.QL >= 2;
    const int nt3 = split ? 2 * B : B;
    if (tid < nt3) {
      const int c = tid % B;
      const bool second = tid >= B;  // the E chain's lane when split
      const int wl = min(32, nt3 - (tid & ~31));
      const unsigned mask = wl == 32 ? 0xffffffffu : ((1u << wl) - 1u);
      LandauOut Lo = landau_factored(msum[c], msum[B + c], msum[2 * B + c], msum[3 * B + c],
                                     msum[4 * B + c]);
      T g0 = T(0), g1 = T(0);
      if (!Lo.ok) {
        if (!second && s0 + c < g.Z) report_error(err, 6, s0 + c);
        Lo.n = 0.0; Lo.T = 1.0; Lo.beta = 0.0; Lo.gamma = 1.0; Lo.u = Lo.ub = 0.0;
      } else if (g.tau_mode == kTauEtas) {
        const double lam = Lo.n * g.lambda_ref * rcp64(Lo.T * Lo.T * Lo.T);
        const double r = g.dt * Lo.T * rcp64(g.tau_AW0 * fma(-0.25, log(lam), 1.0));
        g0 = T(Lo.gamma * r);
        g1 = T(Lo.ub * r);
      } else {
        const T r = T(g.dt_tau);
        g0 = T(Lo.gamma) * r;
        g1 = T(Lo.ub) * r;
      }
      if (!second) {
        gco[2 * c] = g0;
        gco[2 * c + 1] = g1;
      }
      const int nm = g.nm;
      if (split) {
        // slot k = 0 of the cell's coefficients holds delta_m, slot 1 eps_m; the
        // scalars A3, A4 (with the factor T) carry the norms of the chains
        const int nm4 = max(nm, 4);
        float r;
        const int M = aeq_start<T>(float(Lo.u), float(Lo.gamma), nm4, &r);
        const bool far = M > aeq_max_start<T>();
        const int Mc = min(M, aeq_max_start<T>()), Mw = __reduce_max_sync(mask, Mc);
        const T beta = T(Lo.beta), gam = T(Lo.gamma), b2 = far ? T(0) : beta * beta;
        const T n4 = T(0.25 * Lo.n);
        T* dst = coef + ((size_t)(second ? B : 0) + c) * MP;
        T d2 = T(0), d1 = T(0);
        aeq_chain<T>(second, b2, T(r), Mc, Mw, nm4, [&](int m, T x) {
          if (m < nm && m >= 2) dst[m] = x;
          if (m == 2) d2 = x;
          if (m == 1) d1 = x;
        });
        if (!second) {
          dst[0] = d1;
          if (nm > 1) dst[1] = d1;
          cellT[c] = n4 * (gam + gam) * T(rcp64(double(d1)));
        } else {
          dst[0] = fma(T(0.25), b2, T(0.75)) * d2;
          if (nm > 1) dst[1] = d2;
          cellT[B + c] = n4 * T(Lo.T) * (T(8.0 / 3.0) * gam * gam) * T(rcp64(double(d2)));
          cellT[2 * B + c] = beta;
        }
        if (far) {
          T X[2 * kMaxM];
          aeq_far<T>(tb.gl_t, tb.gl_w, T(Lo.u), T(Lo.u * Lo.u / (Lo.gamma + 1.0)), nm, X);
          // as delta_m, eps_m that give X3_m, X4_m with A = n/4 (T), sign^m in beta
          for (int m = 0; m < nm; ++m)
            dst[m] = X[second ? kMaxM + m : m] / aeq_scale<T>(second, m);
          cellT[second ? B + c : c] = second ? n4 * T(Lo.T) : n4;
          if (second) cellT[2 * B + c] = Lo.beta < 0.0 ? T(-1) : T(1);
        }
      } else {
        T D[kMaxM], E[kMaxM];
        const AeqCell<T> cell{T(Lo.n), T(Lo.T), T(Lo.gamma), T(Lo.ub)};
        const AeqScalars<T> o = aeq_cell<T, kMaxM>(cell, nm, mask, tb.gl_t, tb.gl_w, D, E);
        T bm = T(1);
#pragma unroll
        for (int m = 0; m < kMaxM; ++m) {
          if (m < nm) {
            const T um = T(m + 0.5) * bm;
            const T p3 = um * (o.A3 * (aeq_scale<T>(false, m) * D[m]));
            const T pd = p3 - um * (o.A4 * (aeq_scale<T>(true, m) * E[m]));
            for (int k = 0; k < g.QL; ++k)
              coef[((size_t)k * B + c) * MP + m] = fma(tb.L1k[k], pd, p3);
            bm *= o.q;
          }
        }
        for (int m = nm; m < MP; ++m)
          for (int k = 0; k < g.QL; ++k) coef[((size_t)k * B + c) * MP + m] = T(0);
      }
    }
    if (split) {
      __syncthreads();
      for (int e = tid; e < B * MP; e += NT) {
        const int c = e / MP, m = e - c * MP;
        T p3 = T(0), pd = T(0);
        if (m < g.nm) {
          const T q = cellT[2 * B + c];
          T um = T(m + 0.5);
          for (int i = 0; i < m; ++i) um *= q;
          p3 = um * (cellT[c] * (aeq_scale<T>(false, m) * coef[(size_t)c * MP + m]));
          pd = p3 - um * (cellT[B + c] * (aeq_scale<T>(true, m) * coef[((size_t)B + c) * MP + m]));
        }
        for (int k = 0; k < g.QL; ++k) coef[((size_t)k * B + c) * MP + m] = fma(tb.L1k[k], pd, p3);
      }
    }
    __syncthreads();
  } else {
    for (int i = tid; i < 2 * B; i += NT) gco[i] = T(0);
    for (int i = tid; i < g.QL * B * MP; i += NT) coef[i] = T(0);
    __syncthreads();
  }

  // ---- 4. WENO5 + relaxation + RK update, row sweeps ----
  const T c1 = T(g.inv_dz * g.dt);
  const int SLr = B / nseg;
  // unsegmented rows: the negative ones padded to whole warps, so that no warp
  // runs both directions
  const int pad = nseg == 1 ? (32 - nneg % 32) % 32 : 0;
  auto rows = [&](auto order) {
    constexpr int NO = decltype(order)::value;  // orders held in registers (FP32)
    for (int u = tid; u < V * nseg + pad; u += NT) {
      if (u >= nneg && u < nneg + pad) continue;
      const int up = u >= nneg ? u - pad : u;
      const int ir = up % V, seg = up / V;
      const int v = rowv[ir];
      const bool pos = ir >= nneg;
      const T xi = tb.xi[v];
      const int k = tb.kidx[v];
      const T* wp = tb.wp + v;
      T wpr[NO];
      if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int m = 0; m < NO; ++m) wpr[m] = (m < g.nm) ? wp[m * V] : T(0);
      }
      const T* row = tile + v * P;
      T* orow = (nseg > 1) ? (outb + v * B - kHalo) : (tile + v * P);
      const T* ck = coef + (size_t)k * B * MP;
      const int i0 = seg * SLr;
      // the segment length is one of B, B/2, B/4, B/8 (>= one 16-byte chunk)
      if (SLr == B) {
        if (pos) sweep_segment<T, true, B, NO>(row, orow, i0, xi, c1, wpr, wp, V, MP, ck, gco);
        else sweep_segment<T, false, B, NO>(row, orow, i0, xi, c1, wpr, wp, V, MP, ck, gco);
      } else if constexpr (B / 2 >= VN) {
       if (SLr == B / 2) {
        if (pos) sweep_segment<T, true, B / 2, NO>(row, orow, i0, xi, c1, wpr, wp, V, MP, ck, gco);
        else sweep_segment<T, false, B / 2, NO>(row, orow, i0, xi, c1, wpr, wp, V, MP, ck, gco);
       } else if constexpr (B / 4 >= VN) {
        if (SLr == B / 4) {
          if (pos) sweep_segment<T, true, B / 4, NO>(row, orow, i0, xi, c1, wpr, wp, V, MP, ck, gco);
          else sweep_segment<T, false, B / 4, NO>(row, orow, i0, xi, c1, wpr, wp, V, MP, ck, gco);
        } else if constexpr (B / 8 >= VN) {
          if (pos) sweep_segment<T, true, B / 8, NO>(row, orow, i0, xi, c1, wpr, wp, V, MP, ck, gco);
          else sweep_segment<T, false, B / 8, NO>(row, orow, i0, xi, c1, wpr, wp, V, MP, ck, gco);
        }
       }
      }
    }
  };
  // the code of low truncations carries no orders past eight
  if (kF64 || MP <= 8) rows(std::integral_constant<int, 8>());
  else if constexpr (!kF64) rows(std::integral_constant<int, 16>());
  __syncthreads();

  // ---- 5. coalesced store of the interior ----
  const T a = (stage == 1) ? T(0.75) : T(1.0 / 3.0);
  const T b = (stage == 1) ? T(0.25) : T(2.0 / 3.0);
  const T* res = (nseg > 1) ? outb : tile + kHalo;
  const int rp = (nseg > 1) ? B : P;
  if (s0 + B <= g.Z) {
    for (int idx = tid; idx < V * CH; idx += NT) {
      const int v = idx / CH, c = idx - v * CH;
      const size_t o = (size_t)v * g.ldz + s0 + c * VN;
      T r[VN];
      ld_chunk<T>(res + v * rp + c * VN, r);
      if (stage != 0) {
        T fo[VN];
        ld_chunk<T>(fn + o, fo);
#pragma unroll
        for (int q = 0; q < VN; ++q) r[q] = a * fo[q] + b * r[q];
      }
      st_chunk<T>(fout + o, r);
    }
  } else {
    for (int idx = tid; idx < V * B; idx += NT) {
      const int v = idx / B, i = idx - v * B;
      const int s = s0 + i;
      if (s < g.Z) {
        const size_t o = (size_t)v * g.ldz + s;
        T r = res[v * rp + i];
        if (stage != 0) r = a * fn[o] + b * r;
        fout[o] = r;
      }
    }
  }
}

template <typename T, int B, int NT>
__global__ void __launch_bounds__(NT, 2)
sod_stage_kernel(const T* __restrict__ fin, const T* __restrict__ fn, T* fout, int stage,
                 int* err, SodGeom g, SodTables<T> tb, const int* __restrict__ rowv, int nneg,
                 int nseg, int np) {
  sod_tile<T, B, NT>(fin, fn, fout, stage, err, g, tb, rowv, nneg, nseg, np, blockIdx.x * B);
}

template <typename T, int B, int NT>
__global__ void __launch_bounds__(NT, 2)
sod_batch_kernel(const SodRunDesc<T>* __restrict__ runs, const SodTask* __restrict__ tasks,
                 int ntasks, const long long* __restrict__ step, int step_off, int stage,
                 int* err, int nseg, int np) {
  const long long n = *step + step_off;
  for (int t = blockIdx.x; t < ntasks; t += gridDim.x) {
    const SodTask tk = tasks[t];
    const SodRunDesc<T> R = runs[tk.run];
    if (n >= R.nsteps) break;  // tasks are ordered by decreasing step count
    const T* fin = stage == 0 ? R.F0 : (stage == 1 ? R.F1 : R.F2);
    T* fout = stage == 0 ? R.F1 : (stage == 1 ? R.F2 : R.F0);
    sod_tile<T, B, NT>(fin, R.F0, fout, stage, err, R.g, R.tb, R.rowv, R.nneg, nseg, np, tk.s0);
    __syncthreads();
  }
}

constexpr int kNT = 320;           // threads of the scalar kernels
constexpr int kMaxSmem = 232448;   // opt-in shared memory per CTA

static int pick_nseg(int V, int B, int VN) {
  int nseg = 1;
  while (nseg < 8 && B / (2 * nseg) >= VN && V * 2 * nseg <= kNT) nseg *= 2;
  return nseg;
}

// Shared memory of a tile without the partial slots of the moment sums; what
// the kernels accept is decided by this size.
template <typename T>
static size_t smem_base(int V, int B, int QL, int nm) {
  return SodSmem<T>(V, B, QL, nm, pick_nseg(V, B, V16<T>::n) > 1, 0).total;
}

// Partial slots: one per row group of the CTA where they fit beside the tile
// without costing the second CTA of an SM, fewer (added in rounds) otherwise.
template <typename T>
static int pick_np(int V, int B, int QL, int nm) {
  const size_t base = smem_base<T>(V, B, QL, nm), half = kMaxSmem / 2 - 2048;
  const size_t room = (base <= half ? half : (size_t)kMaxSmem) - std::min<size_t>(base, kMaxSmem);
  const size_t full = kNT / (B < 32 ? 32 : B);
  return (int)std::min(full, room / (sizeof(double) * 5 * B));
}

template <typename T>
static size_t smem_for(int V, int B, int QL, int nm) {
  return SodSmem<T>(V, B, QL, nm, pick_nseg(V, B, V16<T>::n) > 1, pick_np<T>(V, B, QL, nm)).total;
}

// Opt every stage kernel into the large dynamic shared-memory carve-out
// (done once at set-up, outside any stream capture).
cudaError_t sod_set_attributes() {
  const void* fns[] = {(const void*)sod_stage_kernel<float, 128, 320>,
                       (const void*)sod_stage_kernel<float, 64, 320>,
                       (const void*)sod_stage_kernel<float, 32, 320>,
                       (const void*)sod_stage_kernel<float, 16, 320>,
                       (const void*)sod_stage_kernel<double, 16, 320>,
                       (const void*)sod_stage_kernel<double, 8, 320>,
                       (const void*)sod_stage_kernel<double, 4, 320>,
                       (const void*)sod_stage_kernel<double, 2, 320>,
                       (const void*)sod_batch_kernel<float, 128, 320>,
                       (const void*)sod_batch_kernel<float, 64, 320>,
                       (const void*)sod_batch_kernel<float, 32, 320>,
                       (const void*)sod_batch_kernel<float, 16, 320>,
                       (const void*)sod_batch_kernel<double, 16, 320>,
                       (const void*)sod_batch_kernel<double, 8, 320>};
  for (const void* f : fns) {
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
    if (e != cudaSuccess) return e;
  }
  cudaError_t e = sod32_set_attributes();
  if (e != cudaSuccess) return e;
  return sod32p_set_attributes();
}

SodLaunch sod_pick_launch(bool fp64, int V, int QL, int nm, int max_smem, int Z, int nsm) {
  SodLaunch L{0, 0};
  if (QL > kMaxQL || V < 1 || nm < 1 || nm > kMaxM) return L;
  const size_t half = (size_t)max_smem / 2 - 2048;
  if (!fp64) {
    // packed FP32x2 kernel: whole rows per thread, so it needs enough rows to
    // fill a CTA, N_Omega <= 7, and two CTAs per SM at least.  65536 cells, us per
    // step, packed / best scalar tile: V = 150 244 / 274, V = 300 388 / 425, V = 600
    // 715 / 758
    if (V >= 128 && nm <= 8 && sod32_smem_bytes(V, QL) <= half) return {kSod32Cells, 0};
    // few velocities: wide tiles share each tile's fixed costs among more
    // cells and give the row segments more cells (65536 cells, us per step with
    // 128-, 64- and 32-cell tiles: V = 24 91, 124, 184; V = 60 144, 162, 220; few
    // cells run faster on narrower tiles: 4000 x 24 40, 32, 29)
    if (V < 48 && smem_base<float>(V, 128, QL, nm) <= half) return {128, 0};
    if (V < 128 && smem_base<float>(V, 64, QL, nm) <= half) return {64, 0};
    if (smem_base<float>(V, 32, QL, nm) <= half) return {32, 0};
    if (smem_base<float>(V, 16, QL, nm) <= half) return {16, 0};
    if (smem_base<float>(V, 16, QL, nm) <= (size_t)max_smem) return {16, 0};
  } else {
    if (smem_base<double>(V, 16, QL, nm) <= half) L.B = 16;
    else if (smem_base<double>(V, 8, QL, nm) <= (size_t)max_smem) L.B = 8;
    // The FP64 pipe of an SM (~2 lane operations per cycle) sets the time of a
    // tile: about 49 operations per cell and velocity and 42 per row for the
    // halo, so a tube with few tiles runs faster on narrower ones until every
    // SM has one.  17000 lane operations stand for the phases that wait on
    // latency (two CTAs per SM overlap them).
    if (L.B && nsm > 0) {
      double best = 0.0;
      for (int B = L.B, first = 1; B >= 2; B /= 2, first = 0) {
        const long long tiles = (Z + B - 1) / B;
        const double t = (double)((tiles + nsm - 1) / nsm) * V * (49.0 * B + 42.0) +
                         17000.0 * (double)((tiles + 2 * nsm - 1) / (2 * nsm));
        if (first || t < best) {
          best = t;
          L.B = B;
        }
      }
    }
  }
  return L;
}

template <typename T, int B>
static cudaError_t launch_b(const SodGeom& g, const SodTables<T>& tb, const int* rowv, int nneg,
                            const T* fin, const T* fn, T* fout, int stage, int* err,
                            cudaStream_t st) {
  const int nseg = pick_nseg(g.V, B, V16<T>::n);
  const int np = pick_np<T>(g.V, B, g.QL, g.nm);
  const size_t smem = smem_for<T>(g.V, B, g.QL, g.nm);
  const int grid = (g.Z + B - 1) / B;
  sod_stage_kernel<T, B, kNT><<<grid, kNT, smem, st>>>(fin, fn, fout, stage, err, g, tb, rowv,
                                                       nneg, nseg, np);
  return cudaGetLastError();
}

template <typename T>
cudaError_t sod_stage_launch(const SodLaunch& L, const SodGeom& g, const SodTables<T>& tb,
                             const int* rowv, int nneg, const T* fin, const T* fn, T* fout,
                             int stage, int* err, cudaStream_t st) {
  if constexpr (sizeof(T) == 4) {
    if (L.B == kSod32Cells && L.form == 1)
      return sod32p_stage_launch(g, tb, rowv, nneg, fin, fn, fout, stage, err, L.nsm, st);
    if (L.B == kSod32Cells) return sod32_stage_launch(g, tb, rowv, nneg, fin, fn, fout, stage, err, st);
  }
  switch (L.B) {
    case 128:
      if constexpr (sizeof(T) == 4) return launch_b<T, 128>(g, tb, rowv, nneg, fin, fn, fout, stage, err, st);
      break;
    case 64:
      if constexpr (sizeof(T) == 4) return launch_b<T, 64>(g, tb, rowv, nneg, fin, fn, fout, stage, err, st);
      break;
    case 32:
      if constexpr (sizeof(T) == 4) return launch_b<T, 32>(g, tb, rowv, nneg, fin, fn, fout, stage, err, st);
      break;
    case 16: return launch_b<T, 16>(g, tb, rowv, nneg, fin, fn, fout, stage, err, st);
    case 8:
      if constexpr (sizeof(T) == 8) return launch_b<T, 8>(g, tb, rowv, nneg, fin, fn, fout, stage, err, st);
      break;
    case 4:
      if constexpr (sizeof(T) == 8) return launch_b<T, 4>(g, tb, rowv, nneg, fin, fn, fout, stage, err, st);
      break;
    case 2:
      if constexpr (sizeof(T) == 8) return launch_b<T, 2>(g, tb, rowv, nneg, fin, fn, fout, stage, err, st);
      break;
    default: break;
  }
  return cudaErrorInvalidValue;
}

template cudaError_t sod_stage_launch<float>(const SodLaunch&, const SodGeom&,
                                             const SodTables<float>&, const int*, int,
                                             const float*, const float*, float*, int, int*,
                                             cudaStream_t);
template cudaError_t sod_stage_launch<double>(const SodLaunch&, const SodGeom&,
                                              const SodTables<double>&, const int*, int,
                                              const double*, const double*, double*, int, int*,
                                              cudaStream_t);

size_t sod_stage_smem_bytes(bool fp64, int B, int V, int QL, int nm) {
  if (!fp64) {
    if (B == kSod32Cells) return sod32_smem_bytes(V, QL);
    if (B == 128 || B == 64 || B == 32 || B == 16) return smem_for<float>(V, B, QL, nm);
  } else {
    if (B == 16 || B == 8) return smem_for<double>(V, B, QL, nm);
  }
  return 0;
}

cudaError_t sod32_batch_launch(size_t smem, int grid, const SodRunDesc<float>* runs,
                               const SodTask* tasks, int ntasks, const long long* step, int step_off,
                               int stage, int* err, const void* maps, cudaStream_t st);

const void* sod32_batch_function(size_t smem);

int sod_batch_resident(bool fp64, int B, size_t smem) {
  const void* f = nullptr;
  int nt = kNT;
  if (fp64) {
    if (B == 16) f = (const void*)sod_batch_kernel<double, 16, kNT>;
    if (B == 8) f = (const void*)sod_batch_kernel<double, 8, kNT>;
  } else {
    if (B == 128) f = (const void*)sod_batch_kernel<float, 128, kNT>;
    if (B == 64) f = (const void*)sod_batch_kernel<float, 64, kNT>;
    if (B == 32) f = (const void*)sod_batch_kernel<float, 32, kNT>;
    if (B == 16) f = (const void*)sod_batch_kernel<float, 16, kNT>;
    if (B == kSod32Cells) {
      f = sod32_batch_function(smem);
      nt = kSod32Threads;
    }
  }
  int n = 0;
  if (!f || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f, nt, smem) != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  return std::max(n, 1);
}

// Batched stages: all runs of a class share V (so nseg and the tile width).
template <typename T, int B>
static cudaError_t batch_b(size_t smem, int grid, const SodRunDesc<T>* runs, const SodTask* tasks,
                           int ntasks, const long long* step, int step_off, int stage, int* err, int V, int QL,
                           int nm, cudaStream_t st) {
  sod_batch_kernel<T, B, kNT><<<grid, kNT, smem, st>>>(runs, tasks, ntasks, step, step_off, stage, err,
                                                       pick_nseg(V, B, V16<T>::n),
                                                       pick_np<T>(V, B, QL, nm));
  return cudaGetLastError();
}

template <typename T>
cudaError_t sod_batch_stage_launch(int B, size_t smem, int grid, const SodRunDesc<T>* runs,
                                   const SodTask* tasks, int ntasks, const long long* step,
                                   int step_off, int stage, int* err, int V, int QL, int nm, cudaStream_t st,
                                   const void* maps) {
  if (ntasks == 0) return cudaSuccess;
  if constexpr (sizeof(T) == 4) {
    switch (B) {
      case kSod32Cells:
        return sod32_batch_launch(smem, grid, runs, tasks, ntasks, step, step_off, stage, err, maps,
                                  st);
      case 128: return batch_b<T, 128>(smem, grid, runs, tasks, ntasks, step, step_off, stage, err, V, QL, nm, st);
      case 64: return batch_b<T, 64>(smem, grid, runs, tasks, ntasks, step, step_off, stage, err, V, QL, nm, st);
      case 32: return batch_b<T, 32>(smem, grid, runs, tasks, ntasks, step, step_off, stage, err, V, QL, nm, st);
      case 16: return batch_b<T, 16>(smem, grid, runs, tasks, ntasks, step, step_off, stage, err, V, QL, nm, st);
      default: break;
    }
  } else {
    switch (B) {
      case 16: return batch_b<T, 16>(smem, grid, runs, tasks, ntasks, step, step_off, stage, err, V, QL, nm, st);
      case 8: return batch_b<T, 8>(smem, grid, runs, tasks, ntasks, step, step_off, stage, err, V, QL, nm, st);
      default: break;
    }
  }
  return cudaErrorInvalidValue;
}

template cudaError_t sod_batch_stage_launch<float>(int, size_t, int, const SodRunDesc<float>*,
                                                   const SodTask*, int, const long long*, int, int,
                                                   int*, int, int, int, cudaStream_t, const void*);
template cudaError_t sod_batch_stage_launch<double>(int, size_t, int, const SodRunDesc<double>*,
                                                    const SodTask*, int, const long long*, int, int,
                                                    int*, int, int, int, cudaStream_t, const void*);

// ---------------------------------------------------------------------------
// Initialisation: per-cell FP64 coefficients, then populations.
// ---------------------------------------------------------------------------
__global__ void sod_init_coef_kernel(SodGeom g, SodTablesF64 tb, const double* __restrict__ n,
                                     const double* __restrict__ Tt,
                                     const double* __restrict__ beta, double* coef, int* err) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.Z) return;
  const double nn = n[s], TT = Tt[s], bb = beta[s];
  double* cs = coef + (size_t)s * kMaxQL * kMaxM;
  if (!(nn > 0.0) || !(TT > 0.0) || !(fabs(bb) < 1.0)) {
    report_error(err, 6, s);
    for (int i = 0; i < kMaxQL * kMaxM; ++i) cs[i] = 0.0;
    return;
  }
  const double gam = 1.0 / sqrt((1.0 - bb) * (1.0 + bb));
  const double u = gam * fabs(bb);
  const double A = asinh(u);
  const double sh = sinh(0.5 * A);
  const double sh2 = 2.0 * sh * sh;
  const double uinv = u > 0.0 ? 1.0 / u : 0.0;
  double J3[kMaxM], J4[kMaxM];
#pragma unroll
  for (int m = 0; m < kMaxM; ++m) { J3[m] = 0.0; J4[m] = 0.0; }
  for (int i = 0; i < kAeqNodes; ++i)
    aeq_node<double>(tb.gl_t[i], tb.gl_w[i], A, sh2, uinv, !(u > 0.0), g.nm, J3, J4);
  const double r = u > 0.0 ? A / u : 1.0;
  double sm = nn * r * 0.25;
  const double sgn = bb < 0.0 ? -1.0 : 1.0;
#pragma unroll
  for (int m = 0; m < kMaxM; ++m) {
    if (m < g.nm) {
      const double h = sm * 0.5 * (2 * m + 1);
      const double d = J3[m] - TT * J4[m];
      for (int k = 0; k < g.QL; ++k) cs[k * kMaxM + m] = h * (J3[m] + tb.L1k[k] * d);
      sm *= sgn;
    }
  }
}

template <typename T>
__global__ void sod_init_pop_kernel(SodGeom g, SodTablesF64 tb, const double* __restrict__ coef,
                                    T* f) {
  const size_t total = (size_t)g.V * g.Z;
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
       idx += (size_t)gridDim.x * blockDim.x) {
    const int v = (int)(idx / g.Z), s = (int)(idx - (size_t)v * g.Z);
    const int k = tb.kidx[v];
    const double* c = coef + (size_t)s * kMaxQL * kMaxM + k * kMaxM;
    double acc = 0.0;
    for (int m = 0; m < g.nm; ++m) acc += c[m] * tb.wp[m * g.V + v];
    f[(size_t)v * g.ldz + s] = T(acc);
  }
}

template <typename T>
cudaError_t sod_init_launch(const SodGeom& g, const SodTablesF64& tb, const double* n,
                            const double* Tt, const double* beta, double* coef_scratch, T* f,
                            int* err, cudaStream_t st) {
  sod_init_coef_kernel<<<(g.Z + 127) / 128, 128, 0, st>>>(g, tb, n, Tt, beta, coef_scratch, err);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  sod_init_pop_kernel<T><<<1024, 256, 0, st>>>(g, tb, coef_scratch, f);
  return cudaGetLastError();
}

template cudaError_t sod_init_launch<float>(const SodGeom&, const SodTablesF64&, const double*,
                                            const double*, const double*, double*, float*, int*,
                                            cudaStream_t);
template cudaError_t sod_init_launch<double>(const SodGeom&, const SodTablesF64&, const double*,
                                             const double*, const double*, double*, double*,
                                             int*, cudaStream_t);

}  // namespace rslb
