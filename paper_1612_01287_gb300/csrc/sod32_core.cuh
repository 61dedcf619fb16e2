// sod32_core.cuh -- the phases of the packed FP32x2 shock-tube stage, shared by
// the one-CTA-per-tile kernel (sod32.cu) and the persistent pipelined kernel
// (sod32p.cu), so that both perform exactly the same arithmetic.
//
// A tile is kB2 = RSLB_PACKED_TILE_CELLS output cells, split into two halves of
// kH; a thread walks a velocity row and advances both halves in lock-step, the
// left half in the x lane and the right half in the y lane of float2 values,
// so every arithmetic instruction of the sweep does two cells.  Shared memory
// holds the kB2 + 8 cells s0-4 .. s0+kB2+3 of every velocity row densely
// (the row pitch is an odd number of 16-byte units, so 16-byte accesses of 8
// consecutive rows hit distinct banks); "slot" s of the sweep is the pair
// (position s, position s + kH).
//
// Phases of one RK stage of one tile (Sec. III F, Eq. rk3):
//   moments    FP32 sums of N+-, A+-, D (Eq. macro_jk in the factored form), from
//              three sums per radial node, as compensated double-floats; a lane
//              owns two cells and a slice of the rows;
//   landau     a thread per cell: FP64 Landau matching (Eqs. E_landau, u_landau)
//              and tau;
//   coefs      f^eq coefficients (Eq. feq_trunc via Eq. aeq_aux) by the recurrence
//              over the Legendre order, 8 threads per cell;
//   sweep      WENO5 flux difference (Eqs. flux_weno, weno5_omega), f^eq at
//              the nodes (Eq. fjk), relaxation (Eq. L_Sod), stage update;
//   store      RK combination with f_n and the write of the tile.
#pragma once

#include <cuda.h>

#include <cstdint>

#include "rslb_device.cuh"
#include "sod.cuh"

namespace rslb {
namespace p32 {

constexpr int kB2 = kSod32Cells;  // output cells per tile
constexpr int kH = kB2 / 2;        // cells per half
constexpr int kC = kB2 + 8;        // cells staged per row (4-cell halo per side)
constexpr int kP = kC;             // floats per row (an odd number of 16-byte units)
constexpr int kSlices = 7;             // row slices of the moment sums (a warp's work each)
constexpr int kCellThreads = 8 * kB2;  // coefficients: 8 threads per cell
static_assert(kCellThreads % 32 == 0 && kB2 % 4 == 0 && kH % 2 == 0 && (kC / 4) % 2 == 1, "packed tile shape");
constexpr int kMP = 8;        // coefficient pitch (m) for N_Omega <= 7
constexpr int kInflight = 8;  // 16-byte global loads in flight per thread (staging, store)
constexpr int kErrWait = RSLB_ERR_TIMEOUT;  // error code: a bounded wait ran out

__device__ __forceinline__ float2 splat(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b with one rounding
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, splat(-1.f), a); }

__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ void report_err(int* err, int code, int cell) {
  if (atomicCAS(err, 0, code) == 0) err[1] = cell;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Shared-memory scratch of a tile: the moment slices' partial sums
// [kSlices][5][kB2] (hi, lo).  (The size is that of the five weights per velocity
// and the per-cell scalars it replaced where that was larger, because it
// decides which velocity counts the kernel accepts.)
__host__ __device__ __forceinline__ size_t scratch_bytes(int V) {
  const size_t part = sizeof(float2) * kSlices * 5 * kB2;
  const size_t old = ((sizeof(double) * 8 * kB2 + 127) & ~size_t(127)) +
                     ((sizeof(float) * 5 * (size_t)V + 127) & ~size_t(127));
  return old > part ? old : (part + 127) & ~size_t(127);
}

// Rows of one bulk-tensor box (<= 256 rows, a multiple of 8 so that a box of
// kC floats per row is a multiple of 128 bytes) and the number of boxes.
__host__ __device__ __forceinline__ int tma_box_rows(int V, int* nbox) {
  const int nb = (V + 255) / 256;
  int r = (V + nb - 1) / nb;
  r = (r + 7) / 8 * 8;
  *nbox = nb;
  return r;
}

// WENO5 correction (omega . g) of sod.cu::weno_corr for two faces at once, from
// the differences D1, D2 left and right of the upwind-centre value, the second
// differences' Q_c = 4/3 S_c^2 and the shared X = D1 + S_1 = 2 D1 - D0,
// Y = D2 - S_3 = 2 D2 - D3: with D2 = D1 + S_2,
//   sigma_1 = D1 X + Q_1, sigma_2 = D1 D2 + Q_2, sigma_3 = D2 Y + Q_3,
//   g_1 = 2 X + D1, g_2 = 2 D2 + D1, g_3 = 2 D2 + Y
// (sigma_q of Eq. weno5_omega; positive definite forms, so nothing cancels).
__device__ __forceinline__ float2 weno_corr2(float2 D1, float2 D2, float2 X, float2 Y, float2 Q1,
                                             float2 Q2, float2 Q3) {
  const float2 s1 = fma2(D1, X, Q1), s2 = fma2(D1, D2, Q2), s3 = fma2(D2, Y, Q3);
  const float2 g1 = fma2(splat(2.f), X, D1), g2 = fma2(splat(2.f), D2, D1),
               g3 = fma2(splat(2.f), D2, Y);
  // scale the smoothness indicators by the power of two at or below their
  // maximum (the weights are homogeneous in sigma; this only keeps the
  // fourth powers inside the FP32 range): 2^(127 - e) for the biased exponent e,
  // an AND and a subtract; a zero or subnormal maximum gives 2^127, which
  // keeps zero sigmas zero and brings subnormal ones into range
  const float mx = fmaxf(s1.x, fmaxf(s2.x, s3.x));
  const float my = fmaxf(s1.y, fmaxf(s2.y, s3.y));
  auto inv_pow2 = [&](float m) {
    return __int_as_float(0x7F000000 - (__float_as_int(m) & 0x7F800000));
  };
  const float2 inv = make_float2(inv_pow2(mx), inv_pow2(my));
  const float2 r1 = mul2(s1, inv), r2 = mul2(s2, inv), r3 = mul2(s3, inv);
  const float2 t1 = mul2(r1, r1), t2 = mul2(r2, r2), t3 = mul2(r3, r3);
  // products in the ratio 1 : 2 : 1/3; the 2^-120 keeps the reciprocal finite
  // where all products vanish (the correction is 0 there by the limit rules,
  // and is when num = 0) and is below their rounding elsewhere
  const float2 p13 = mul2(t1, t3);
  const float2 n3 = fma2(t1, t2, splat(7.5231638e-37f));
  const float2 n2 = add2(p13, p13), n1 = mul2(mul2(t2, t3), splat(1.f / 3.f));
  const float2 den = add2(add2(n3, n2), n1);
  const float2 num = fma2(n1, g1, fma2(n2, g2, mul2(mul2(t1, t2), g3)));
  return mul2(num, make_float2(rcp_approx(den.x), rcp_approx(den.y)));
}

__device__ __forceinline__ void ld2slots(const float* p, float2* out) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  out[0] = make_float2(v.x, v.y);
  out[1] = make_float2(v.z, v.w);
}

// Slots s, s+1 (s even) of a dense row: x from positions s, s+1, y from
// positions s+kH, s+kH+1.
__device__ __forceinline__ void ld_slot_pair(const float* row, int s, float2* out) {
  const float2 a = *reinterpret_cast<const float2*>(row + s);
  const float2 b = *reinterpret_cast<const float2*>(row + s + kH);
  out[0] = make_float2(a.x, b.x);
  out[1] = make_float2(a.y, b.y);
}

// Sweep a whole row (both halves): slots 4 .. kH+3 are the outputs; window of
// 10 slots [i-4, i+6) around the current two-slot chunk i, with the first
// differences D[c] = f[c+1] - f[c] and from them S[c] = D[c] - D[c-1],
// Q[c] = 4/3 S[c]^2, X[c] = D[c] + S[c] and Y[c] = D[c] - S[c+1] slid along with
// it (two new of each per chunk).  The weights do not see a factor of f, so
// the differences are those of f and xi enters through c1 = xi dt/dz.  For
// xi < 0 the stencil is mirrored (D0 .. D3 = -(D[w+2] .. D[w-1]), so X and Y
// change places); weno_corr2 is odd, so the mirrored correction is minus its
// value for the un-negated differences.  Results go back into the row in
// place: the left-half outputs (positions 4 .. kH+3) and the right-half outputs
// of slots >= 8 (positions >= kH+8) are never read again by the sweep; the
// right-half outputs of slots 4..7 (positions kH+4 .. kH+7) are held until the
// left half has read those positions (its last four slots).  gco holds
// (gamma, gamma beta) dt/tau.
template <bool POS>
__device__ __forceinline__ void sweep_row2(float* row, float xi, const float2* wp2, int nm,
                                           const float* __restrict__ ck,
                                           const float* __restrict__ gco, float c1) {
  constexpr int NW = 10;
  const float2 sixth = splat(1.f / 6.f), q43 = splat(4.f / 3.f);
  const float2 mc1 = splat(-c1), mxi = splat(-xi);
  float2 R[NW], D[NW - 1], S[NW - 1], Q[NW - 1];
  float2 held[2];
  auto diffs = [&](int c0) {
#pragma unroll
    for (int c = 0; c < NW - 1; ++c)
      if (c >= c0) D[c] = sub2(R[c + 1], R[c]);
#pragma unroll
    for (int c = 1; c < NW - 1; ++c)
      if (c >= c0) {
        S[c] = sub2(D[c], D[c - 1]);
        Q[c] = mul2(mul2(q43, S[c]), S[c]);
      }
  };
#pragma unroll
  for (int c = 0; c < NW; c += 2) ld_slot_pair(row, c, R + c);
  S[0] = Q[0] = splat(0.f);
  diffs(0);
  auto face = [&](int w) {  // the face right of window slot w
    if constexpr (POS)
      return weno_corr2(D[w - 1], D[w], add2(D[w - 1], S[w - 1]), sub2(D[w], S[w + 1]), Q[w - 1],
                        Q[w], Q[w + 1]);
    else
      return weno_corr2(D[w + 1], D[w], sub2(D[w + 1], S[w + 2]), add2(D[w], S[w]), Q[w + 2],
                        Q[w + 1], Q[w]);
  };
  float2 Cl = face(3);
#pragma unroll
  for (int t = 0; t < kH / 2; ++t) {
    const int i = 4 + 2 * t;  // slot of the first cell of this chunk
    float2 out[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int wc = 4 + c;
      const float2 Cr = face(wc);
      const float2 dF = POS ? fma2(sub2(Cr, Cl), sixth, D[wc - 1])
                            : fma2(sub2(Cl, Cr), sixth, D[wc]);
      Cl = Cr;
      // f^eq for the two cells of this slot: coefficients (x cell, y cell) per m
      const float* cc = ck + (size_t)(i + c - 4) * (2 * kMP);
      float2 feq = splat(0.f);
#pragma unroll
      for (int m0 = 0; m0 < kMP; m0 += 2) {
        if (m0 < nm) {
          float2 cv[2];
          ld2slots(cc + 2 * m0, cv);
          feq = fma2(cv[0], wp2[m0], feq);
          feq = fma2(cv[1], wp2[m0 + 1], feq);
        }
      }
      const float4 g = *reinterpret_cast<const float4*>(gco + 4 * (i + c - 4));
      const float2 f = R[wc];
      const float2 rate = fma2(mxi, make_float2(g.z, g.w), make_float2(g.x, g.y));
      out[c] = fma2(rate, sub2(feq, f), fma2(mc1, dF, f));
    }
    if (t + 1 < kH / 2) {
#pragma unroll
      for (int c = 0; c < NW - 2; ++c) R[c] = R[c + 2];
#pragma unroll
      for (int c = 0; c < NW - 3; ++c) {
        D[c] = D[c + 2];
        S[c] = S[c + 2];
        Q[c] = Q[c + 2];
      }
      ld_slot_pair(row, i + 6, R + NW - 2);  // slots i+6, i+7
      diffs(NW - 3);
    }
    *reinterpret_cast<float2*>(row + i) = make_float2(out[0].x, out[1].x);
    if (t < 2) {
      held[t] = make_float2(out[0].y, out[1].y);
    } else {
      *reinterpret_cast<float2*>(row + i + kH) = make_float2(out[0].y, out[1].y);
    }
    if (t == kH / 2 - 2) {  // the last two slots have just been read
      *reinterpret_cast<float2*>(row + 4 + kH) = held[0];
      *reinterpret_cast<float2*>(row + 6 + kH) = held[1];
    }
  }
}

// Value of ghost cell sc (outside [0, Z)) of velocity row v under the
// boundary rule (Sec. IV A: fixed equilibria; outflow copies; periodic).
__device__ __forceinline__ float ghost_value(const float* __restrict__ fin, const SodGeom& g,
                                             const SodTables<float>& tb, int v, int sc) {
  if (g.bc == kBcPeriodic) {
    int sp = sc % g.Z;
    if (sp < 0) sp += g.Z;
    return fin[(size_t)v * g.ldz + sp];
  }
  if (g.bc == kBcOutflow) return fin[(size_t)v * g.ldz + (sc < 0 ? 0 : g.Z - 1)];
  return sc < 0 ? tb.ghostL[v] : tb.ghostR[v];
}

// Staging by plain loads, any tile: cell s0-4+p goes to position p
// (0 <= p < kC), ghost cells by the boundary rule.  Threads t of nt.
__device__ __forceinline__ void stage_plain(float* tile, const float* __restrict__ fin,
                                            const SodGeom& g, const SodTables<float>& tb, int s0,
                                            int t, int nt) {
  const int V = g.V;
  for (int idx = t; idx < V * kC; idx += nt) {
    const int v = idx / kC, c = idx - v * kC;
    const int sc = s0 - 4 + c;
    tile[v * kP + c] = (sc >= 0 && sc < g.Z) ? fin[(size_t)v * g.ldz + sc]
                                             : ghost_value(fin, g, tb, v, sc);
  }
}

// Staging of an interior tile by plain 16-byte loads, eight in flight per thread.
__device__ __forceinline__ void stage_interior_vec(float* tile, const float* __restrict__ fin,
                                                   const SodGeom& g, int s0, int t, int nt) {
  const int V = g.V;
  const float* src = fin + s0 - 4;
  for (int base_i = t; base_i < V * (kC / 4); base_i += kInflight * nt) {
    float4 x[kInflight];
#pragma unroll
    for (int u = 0; u < kInflight; ++u) {
      const int idx = base_i + u * nt;
      if (idx < V * (kC / 4)) {
        const int v = idx / (kC / 4), q = idx - v * (kC / 4);
        x[u] = __ldg(reinterpret_cast<const float4*>(src + (size_t)v * g.ldz + 4 * q));
      }
    }
#pragma unroll
    for (int u = 0; u < kInflight; ++u) {
      const int idx = base_i + u * nt;
      if (idx < V * (kC / 4)) {
        const int v = idx / (kC / 4), q = idx - v * (kC / 4);
        *reinterpret_cast<float4*>(tile + v * kP + 4 * q) = x[u];
      }
    }
  }
}

// After a bulk-tensor copy of a boundary tile (out-of-range cells read as
// zero): overwrite the positions whose cells lie outside [0, Z) with their
// ghost values.  Only the leftmost tile has such cells on the left (p < 4)
// and only tiles reaching past Z on the right.  Threads t of nt.
__device__ __forceinline__ void fix_ghosts(float* tile, const float* __restrict__ fin,
                                           const SodGeom& g, const SodTables<float>& tb, int s0,
                                           int t, int nt) {
  const int V = g.V;
  const int nl = s0 - 4 < 0 ? 4 - s0 : 0;                        // leading positions
  const int first_r = g.Z - (s0 - 4);                             // first position >= Z
  const int nr = first_r < kC ? kC - (first_r < 0 ? 0 : first_r) : 0;
  const int per = nl + nr;
  if (per == 0) return;
  for (int idx = t; idx < V * per; idx += nt) {
    const int v = idx / per, q = idx - v * per;
    const int p = q < nl ? q : kC - nr + (q - nl);
    tile[v * kP + p] = ghost_value(fin, g, tb, v, s0 - 4 + p);
  }
}

// (H, L) += x, error-free in H (Knuth), two cells at a time.
__device__ __forceinline__ void two_sum2(float2& H, float2& L, float2 x) {
  const float2 t = add2(H, x), bp = sub2(t, H);
  L = add2(L, add2(sub2(H, sub2(t, bp)), sub2(x, bp)));
  H = t;
}

// Partial moments of row slice sl (0 <= sl < kSlices) by one warp: lane
// 16 hf + pr (pr < 14) sums cells 2 pr, 2 pr + 1 over half hf of the slice's rows.
// With a = sum f (1+xi)^2, b = sum f (1-xi)^2, d = sum f (1-xi^2) over the polar
// nodes of a radial node p, N+- = sum_k ({a, b}_k + d_k)/2, A+- = sum_k p_k {a, b}_k,
// D = sum_k p_k d_k (all weights non-negative): three products per velocity.
// Blocks of four rows, Kahan-compensated across blocks; the radial sums, halves
// and slices are added as double-floats.  consts: load_consts.
__device__ __forceinline__ void moments(const float* tile, const float* __restrict__ m3,
                                        const float* consts, float2* part, int V, int Qx, int sl,
                                        int lane) {
  const int hf = lane >> 4, pr = min(lane & 15, kB2 / 2 - 1);
  const int n2 = 2 * kSlices, h0 = 2 * sl + hf;
  int v = V * h0 / n2;
  const int v1 = V * (h0 + 1) / n2;
  const float* col = tile + 4 + 2 * pr;
  float2 H[5], L[5], s[3], c[3], b[3];
#pragma unroll
  for (int q = 0; q < 5; ++q) H[q] = L[q] = splat(0.f);
#pragma unroll
  for (int q = 0; q < 3; ++q) s[q] = c[q] = b[q] = splat(0.f);
  auto row = [&](int u) {
    const float4 w = __ldg(reinterpret_cast<const float4*>(m3) + u);
    const float2 x = *reinterpret_cast<const float2*>(col + u * kP);
    b[0] = fma2(x, splat(w.x), b[0]);
    b[1] = fma2(x, splat(w.y), b[1]);
    b[2] = fma2(x, splat(w.z), b[2]);
  };
  auto block = [&]() {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const float2 y = sub2(b[q], c[q]);
      const float2 t = add2(s[q], y);
      c[q] = sub2(sub2(t, s[q]), y);
      s[q] = t;
      b[q] = splat(0.f);
    }
  };
  while (v < v1) {
    const int k = v / Qx, ve = min(v1, (k + 1) * Qx);
    for (; v + 4 <= ve; v += 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u) row(v + u);
      block();
    }
    for (; v < ve; ++v) row(v);
    block();
    const float2 ph = splat(consts[8 + 2 * k]), pl = splat(consts[9 + 2 * k]), hh = splat(0.5f);
    two_sum2(H[0], L[0], mul2(hh, s[0]));
    two_sum2(H[0], L[0], mul2(hh, s[2]));
    L[0] = fma2(splat(-0.5f), add2(c[0], c[2]), L[0]);
    two_sum2(H[1], L[1], mul2(hh, s[1]));
    two_sum2(H[1], L[1], mul2(hh, s[2]));
    L[1] = fma2(splat(-0.5f), add2(c[1], c[2]), L[1]);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const float2 x = mul2(ph, s[q]);
      const float2 lo = add2(fma2(ph, s[q], mul2(splat(-1.f), x)),
                             fma2(pl, s[q], mul2(splat(-1.f), mul2(ph, c[q]))));
      two_sum2(H[2 + q], L[2 + q], x);
      L[2 + q] = add2(L[2 + q], lo);
      s[q] = c[q] = splat(0.f);
    }
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const float2 h = make_float2(__shfl_xor_sync(0xffffffffu, H[q].x, 16),
                                 __shfl_xor_sync(0xffffffffu, H[q].y, 16));
    const float2 l = make_float2(__shfl_xor_sync(0xffffffffu, L[q].x, 16),
                                 __shfl_xor_sync(0xffffffffu, L[q].y, 16));
    two_sum2(H[q], L[q], h);
    L[q] = add2(L[q], l);
    if (lane < kB2 / 2)
      *reinterpret_cast<float4*>(part + (size_t)(sl * 5 + q) * kB2 + 2 * pr) =
          make_float4(H[q].x, L[q].x, H[q].y, L[q].y);
  }
}

// Element e = q kB2 + c of the moments of the tile, FP64, from the slices.
__device__ __forceinline__ double moment_total(const float2* part, int e) {
  float2 v = part[e];
#pragma unroll
  for (int i = 1; i < kSlices; ++i) {
    const float2 x = part[i * 5 * kB2 + e];
    const float t = v.x + x.x, bp = t - v.x;
    v.y += x.y + ((v.x - (t - bp)) + (x.x - bp));
    v.x = t;
  }
  return (double)v.x + (double)v.y;
}

// Landau matching (FP64) and relaxation time of cell c (0 <= c < kB2) of the
// tile at s0: what the coefficients need to cells [4][kB2] in FP32 (it may share
// the partial sums' memory), the collision rates (gamma, gamma beta) dt/tau to
// gco [kH][g0x g0y g1x g1y].  ~40 FP64 instructions: a warp's FP64 instruction
// takes a sub-partition ~64 cycles however many lanes are active, so the phase is
// as short as its count.
__device__ __forceinline__ void landau_cell(const double* msum, float* cells, float* gco,
                                            const SodGeom& g, int s0, int c, int* err) {
  const LandauOut Lo = landau_factored(msum[c], msum[kB2 + c], msum[2 * kB2 + c],
                                       msum[3 * kB2 + c], msum[4 * kB2 + c]);
  float g0 = 0.f, g1 = 0.f;
  AeqCell<float> o{0.f, 1.f, 1.f, 0.f};
  if (!Lo.ok) {
    if (s0 + c < g.Z) report_err(err, 6, s0 + c);
  } else {
    o = {float(Lo.n), float(Lo.T), float(Lo.gamma), float(Lo.ub)};
    float r = float(g.dt_tau);
    if (g.tau_mode == kTauEtas) {
      const double lam = Lo.n * g.lambda_ref * rcp64(Lo.T * Lo.T * Lo.T);
      r = float(g.dt * Lo.T * rcp64(g.tau_AW0 * fma(-0.25, log(lam), 1.0)));
    }
    g0 = o.gamma * r;
    g1 = o.ub * r;
  }
  cells[c] = o.n;
  cells[kB2 + c] = o.T_;
  cells[2 * kB2 + c] = o.gamma;
  cells[3 * kB2 + c] = o.ub;
  const int h = c / kH, i = c - h * kH;
  gco[4 * i + h] = g0;
  gco[4 * i + 2 + h] = g1;
}

// f^eq coefficients of the tile: thread t (0 <= t < 8 kB2; whole warps), 8 threads
// per cell: all run the cell's chains, thread m writes the coefficients of order
// m for every radial node; coef [QL][kH][kMP][2 halves].
__device__ __forceinline__ void coefs(const float* cells, float* coef, const float* consts,
                                      const SodGeom& g, const SodTables<float>& tb, int t) {
  const int c = t >> 3, mine = t & 7;
  float D[kMP], E[kMP];
  const AeqCell<float> cell{cells[c], cells[kB2 + c], cells[2 * kB2 + c], cells[3 * kB2 + c]};
  const AeqScalars<float> o =
      aeq_cell<float, kMP>(cell, g.nm, 0xffffffffu, tb.gl_t, tb.gl_w, D, E);
  float d = 0.f, e = 0.f, um = 0.f, bm = 1.f;
#pragma unroll
  for (int m = 0; m < kMP; ++m) {
    if (m == mine) {
      d = aeq_scale<float>(false, m) * D[m];
      e = aeq_scale<float>(true, m) * E[m];
      um = m < g.nm ? (m + 0.5f) * bm : 0.f;
    }
    bm *= o.q;
  }
  const float p3 = um * (o.A3 * d), pd = p3 - um * (o.A4 * e);
  const int h = c / kH, i = c - h * kH;
  float* dst = coef + ((size_t)i * kMP + mine) * 2 + h;
  for (int k = 0; k < g.QL; ++k) dst[k * kH * kMP * 2] = fmaf(consts[k], pd, p3);
}

// Constants of the phases above in shared memory: L_1^{(2)}(x_k) (8), then
// p_k as hi, lo pairs.
constexpr int kConsts = 32 + 8;
__device__ __forceinline__ void load_consts(float* cst, const SodTables<float>& tb, int QL, int t,
                                            int nt) {
  for (int e = t; e < 3 * QL; e += nt) cst[e < QL ? e : 8 + e - QL] = e < QL ? tb.L1k[e] : tb.pk[e - QL];
}

// Row sweeps: rows ir = first, first + stride, ... (negative-xi rows first and
// padded to whole warps, so the upwind direction is uniform within a warp;
// stride a multiple of 32).
__device__ __forceinline__ void sweep_rows(float* tile, const float* coef, const float* gco,
                                           const SodGeom& g, const SodTables<float>& tb,
                                           const int* __restrict__ rowv, int nneg, int first,
                                           int stride) {
  const float c1 = float(g.inv_dz * g.dt);
  const int V = g.V, pad = (32 - nneg % 32) % 32;
  for (int u = first; u < V + pad; u += stride) {
    if (u >= nneg && u < nneg + pad) continue;
    const int ir = u >= nneg ? u - pad : u;
    const int v = rowv[ir];
    const float xi = tb.xi[v];
    const int k = tb.kidx[v];
    float2 wp2[kMP];
#pragma unroll
    for (int m = 0; m < kMP; ++m) wp2[m] = splat((m < g.nm) ? tb.wp[m * V + v] : 0.f);
    const float* ck = coef + (size_t)k * kH * kMP * 2;
    if (ir >= nneg) sweep_row2<true>(tile + v * kP, xi, wp2, g.nm, ck, gco, c1 * xi);
    else sweep_row2<false>(tile + v * kP, xi, wp2, g.nm, ck, gco, c1 * xi);
  }
}

// Per-row tables of the sweep in row order (shared memory): velocity index,
// xi, radial index and w_j w_k P_m(xi_j) [kMP][V]; the same values as the
// tables sweep_rows reads from global memory.
struct RowTables {
  int* v;
  float* xi;
  int* k;
  float* wp;
};

__device__ __forceinline__ void load_row_tables(const RowTables& rt, const SodGeom& g,
                                                const SodTables<float>& tb,
                                                const int* __restrict__ rowv, int t, int nt) {
  const int V = g.V;
  for (int ir = t; ir < V; ir += nt) {
    const int v = rowv[ir];
    rt.v[ir] = v;
    rt.xi[ir] = tb.xi[v];
    rt.k[ir] = tb.kidx[v];
#pragma unroll
    for (int m = 0; m < kMP; ++m) rt.wp[m * V + ir] = (m < g.nm) ? tb.wp[m * V + v] : 0.f;
  }
}

__device__ __forceinline__ void sweep_rows_tab(float* tile, const float* coef, const float* gco,
                                               const SodGeom& g, const RowTables& rt, int nneg,
                                               int first, int stride) {
  const float c1 = float(g.inv_dz * g.dt);
  const int V = g.V, pad = (32 - nneg % 32) % 32;
  for (int u = first; u < V + pad; u += stride) {
    if (u >= nneg && u < nneg + pad) continue;
    const int ir = u >= nneg ? u - pad : u;
    const int v = rt.v[ir];
    const float xi = rt.xi[ir];
    const int k = rt.k[ir];
    float2 wp2[kMP];
#pragma unroll
    for (int m = 0; m < kMP; ++m) wp2[m] = splat(rt.wp[m * V + ir]);
    const float* ck = coef + (size_t)k * kH * kMP * 2;
    if (ir >= nneg) sweep_row2<true>(tile + v * kP, xi, wp2, g.nm, ck, gco, c1 * xi);
    else sweep_row2<false>(tile + v * kP, xi, wp2, g.nm, ck, gco, c1 * xi);
  }
}

// Store: cell c of the tile is position 4 + c; stages 2 and 3 combine with
// f_n (Eq. rk3: 3/4 f_n + 1/4 f, then 1/3 f_n + 2/3 f).  Threads t of nt.
template <int INFL = kInflight>
__device__ __forceinline__ void store(const float* tile, const float* __restrict__ fn, float* fout,
                                      const SodGeom& g, int stage, int s0, int t, int nt) {
  const int V = g.V;
  const float a = (stage == 1) ? 0.75f : 1.f / 3.f;
  const float b = (stage == 1) ? 0.25f : 2.f / 3.f;
  if (s0 + kB2 <= g.Z) {
    // full tile: kB2/4 chunks of 4 cells per row, 16-byte accesses, INFL loads
    // of f_n in flight per thread.  The first nt - nt % (kB2/4) threads each keep
    // one chunk column and step over the rows, so no index is divided; the
    // others have no rows (the caller's barrier needs whole warps, so they do
    // not leave early).
    constexpr int CQ = kB2 / 4;
    const int dv = nt / CQ, v0 = t / CQ, q4 = 4 * (t - v0 * CQ);
    const int ve = v0 < dv ? V : 0;
    const size_t gs = (size_t)dv * g.ldz;
    const float* pn = fn + (size_t)v0 * g.ldz + s0 + q4;
    float* po = fout + (size_t)v0 * g.ldz + s0 + q4;
    const float* pt = tile + v0 * kP + 4 + q4;
    for (int v = v0; v < ve; v += INFL * dv) {
      float4 fo[INFL];
#pragma unroll
      for (int u = 0; u < INFL; ++u)
        if (stage != 0 && v + u * dv < V) fo[u] = __ldg(reinterpret_cast<const float4*>(pn + u * gs));
#pragma unroll
      for (int u = 0; u < INFL; ++u)
        if (v + u * dv < V) {
          float4 r = *reinterpret_cast<const float4*>(pt + u * dv * kP);
          if (stage != 0) {
            r.x = a * fo[u].x + b * r.x;
            r.y = a * fo[u].y + b * r.y;
            r.z = a * fo[u].z + b * r.z;
            r.w = a * fo[u].w + b * r.w;
          }
          *reinterpret_cast<float4*>(po + u * gs) = r;
        }
      pn += INFL * gs;
      po += INFL * gs;
      pt += INFL * dv * kP;
    }
  } else {
    for (int idx = t; idx < V * kB2; idx += nt) {
      const int v = idx / kB2, c = idx - v * kB2;
      const int sc = s0 + c;
      if (sc < g.Z) {
        const size_t o = (size_t)v * g.ldz + sc;
        float r = tile[v * kP + 4 + c];
        if (stage != 0) r = a * fn[o] + b * r;
        fout[o] = r;
      }
    }
  }
  __syncwarp();
}

}  // namespace p32

// Host: tensor map of one FP32 population buffer [V][Z] with row stride ldz,
// boxes of box_cells cells x box_rows rows, zero fill outside (sod32.cu).
bool sod32_make_map(CUtensorMap* m, const float* f, int Z, int ldz, int V, int box_cells,
                    int box_rows);

}  // namespace rslb
