// moments.cu -- output moments of the shock-tube populations (sm_103a).
//
// Per cell: the first and second moments (Eq. macro_jk), Landau matching
// (Sec. II E, Eqs. E_landau-pi_val) in FP64 and the 14 fields of rslb.h.
// The factored Landau form needs five sums, each with a non-negative weight:
//   N+- = sum f (1 +- xi),  A+- = sum f p (1 +- xi)^2,  D = sum f p (1 - xi^2);
// the conserved currents follow exactly:
//   N^t = (N+ + N-)/2,  N^z = (N+ - N-)/2,  T^tz = (A+ - A-)/4,
//   T^tt = (A+ + A-)/4 + D/2,  T^zz = (A+ + A-)/4 - D/2.
//
// With a, b, d the sums over one radial node p of f (1+xi)^2, f (1-xi)^2 and
// f (1-xi^2), N+- = sum_k ({a, b} + d)/2, A+- = sum_k p {a, b}, D = sum_k p d: three
// products per velocity, the rest once per radial node.
//
// Layout: a block covers kMomCells32 (FP32) or kMomCells64 (FP64) cells; each of
// its warps reads one of kMomChunks velocity chunks, so every load is a
// coalesced piece of a row of the [V][ldz] population array.  The chunk
// partials meet in shared memory and one thread per cell finishes the cell in
// FP64.
//
// FP32 populations: the FP64 weight w is split as w_hi + w_lo (two FP32
// numbers, host-made table); f w_hi is formed exactly as a product plus its
// fma remainder, and the sum is kept as a double-float: the hi parts are
// added with an error-free TwoSum (Knuth), the remainders, f w_lo and the
// TwoSum errors in a plain FP32 sum of the low part.  Two neighbouring cells
// share a thread in packed FP32x2 arithmetic.  GB300's FP64 pipe is a small
// fraction of its FP32 rate, so FP64 is used only for the per-cell finish.
// What bounds it: the latency of its loads.  65536 x 600: 87 us cold, DRAM 23% of
// peak, FMA pipe 22%, issue slots 31%, warps waiting on a load for 16 of the ~20
// cycles between their instructions at 26 warps per SM (118 us with five sums in
// four chunks of 64 threads and chunk sums in FP64).
// FP64 populations: plain FP64 products and sums, one cell per thread.
#include "rslb_device.cuh"
#include "sod.cuh"

namespace rslb {

namespace {

constexpr int kMomChunks = 8;                 // velocity chunks per block, a warp each
constexpr int kMomThreads = 32 * kMomChunks;
constexpr int kMomRows = 5;                   // rows whose loads are in flight together

__device__ __forceinline__ float2 mom_add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
// a - b with one rounding
__device__ __forceinline__ float2 mom_sub2(float2 a, float2 b) {
  return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
}

// (H, L) += x * (wh + wl) for two cells; H + L is a double-float.
__device__ __forceinline__ void mom_acc2(float2& H, float2& L, float2 x, float wh, float wl) {
  const float2 WH = make_float2(wh, wh), WL = make_float2(wl, wl);
  const float2 ph = __fmul2_rn(x, WH);
  float2 pl = __ffma2_rn(x, WH, make_float2(-ph.x, -ph.y));  // exact: x wh = ph + pl
  pl = __ffma2_rn(x, WL, pl);
  const float2 s = mom_add2(H, ph);  // TwoSum(H, ph) = s + e exactly
  const float2 bp = mom_sub2(s, H);
  const float2 e = mom_add2(mom_sub2(H, mom_sub2(s, bp)), mom_sub2(ph, bp));
  H = s;
  L = mom_add2(L, mom_add2(e, pl));
}

__device__ __forceinline__ void mom_two_sum2(float2& H, float2& L, float2 x) {
  const float2 s = mom_add2(H, x), bp = mom_sub2(s, H);
  L = mom_add2(L, mom_add2(mom_sub2(H, mom_sub2(s, bp)), mom_sub2(x, bp)));
  H = s;
}

// Per-cell finish: Landau matching and the 14 output fields (rslb.h order).
__device__ __forceinline__ void mom_finish(const double* S, int s, int Z, double* out, int* err) {
  const double Np = S[0], Nm = S[1], Ap = S[2], Am = S[3], D = S[4];
  const LandauOut L = landau_factored(Np, Nm, Ap, Am, D);
  if (!L.ok && atomicCAS(err, 0, 6) == 0) err[1] = s;
  const double Nt = 0.5 * (Np + Nm), Nz = 0.5 * (Np - Nm);
  const double tr = 0.25 * (Ap + Am);
  const size_t z = (size_t)Z;
  const double P = L.E * (1.0 / 3.0);
  out[0 * z + s] = L.n;
  out[1 * z + s] = L.E;
  out[2 * z + s] = P;
  out[3 * z + s] = L.T;
  out[4 * z + s] = L.beta;
  out[5 * z + s] = L.gamma;
  out[6 * z + s] = L.n * rcp64(L.T * L.T * L.T);
  out[7 * z + s] = -4.0 * L.T * (Nz - L.n * L.ub);
  out[8 * z + s] = 2.0 * P - D;
  out[9 * z + s] = Nt;
  out[10 * z + s] = Nz;
  out[11 * z + s] = tr + 0.5 * D;
  out[12 * z + s] = 0.25 * (Ap - Am);
  out[13 * z + s] = tr - 0.5 * D;
}

// FP32 populations.  w: per velocity two float4 = {hi of a, b, d, 0} {lo ..., 0},
// then per radial node {p hi, p lo}.
constexpr int kMomCells32 = 64;  // 32 lanes x 2 cells

__global__ void __launch_bounds__(kMomThreads, 4)
sod_moments32_kernel(int Z, int ldz, int V, int Qx, const float4* __restrict__ w,
                     const float* __restrict__ f, double* out, int* err) {
  // [chunk][sum][cell] (hi, lo); a lane's two cells are accessed as one float4
  __shared__ __align__(16) float2 part[kMomChunks][5][kMomCells32];
  const int chunk = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c0 = blockIdx.x * kMomCells32 + 2 * lane;  // first cell of the pair
  const bool active = c0 < ldz;                        // ldz is even: the pair fits
  const float* pk = reinterpret_cast<const float*>(w + 2 * V);
  int v = (chunk * V) / kMomChunks;
  const int ve = ((chunk + 1) * V) / kMomChunks;
  float2 H[3], L[3];
  // the sums over radial nodes live in the lane's own slots of `part`, which are
  // touched once per radial node: 64 registers, four blocks per SM
  float4* slot = reinterpret_cast<float4*>(&part[chunk][0][2 * lane]);
  constexpr int kSlot = kMomCells32 / 2;  // float4s between the sums of a slot
#pragma unroll
  for (int q = 0; q < 5; ++q) slot[q * kSlot] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int q = 0; q < 3; ++q) H[q] = L[q] = make_float2(0.f, 0.f);
  const float* fp = f + c0;
  auto load = [&](int u) {
    return active ? __ldg(reinterpret_cast<const float2*>(fp + (size_t)u * ldz))
                  : make_float2(0.f, 0.f);
  };
  auto row = [&](int u, float2 x) {
    const float4 h = __ldg(w + 2 * u), l = __ldg(w + 2 * u + 1);
    mom_acc2(H[0], L[0], x, h.x, l.x);
    mom_acc2(H[1], L[1], x, h.y, l.y);
    mom_acc2(H[2], L[2], x, h.z, l.z);
  };
  while (v < ve) {
    const int k = v / Qx, vk = min(ve, (k + 1) * Qx);
    for (; v + kMomRows <= vk; v += kMomRows) {
      float2 x[kMomRows];
#pragma unroll
      for (int u = 0; u < kMomRows; ++u) x[u] = load(v + u);
#pragma unroll
      for (int u = 0; u < kMomRows; ++u) row(v + u, x[u]);
    }
    for (; v < vk; ++v) row(v, load(v));
    const float ph = __ldg(pk + 2 * k), pl = __ldg(pk + 2 * k + 1);
    const float2 P = make_float2(ph, ph), PL = make_float2(pl, pl), h2 = make_float2(0.5f, 0.5f);
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const float4 t4 = slot[q * kSlot];
      float2 HH = make_float2(t4.x, t4.z), LL = make_float2(t4.y, t4.w);
      if (q < 2) {  // N+-
        mom_two_sum2(HH, LL, __fmul2_rn(h2, H[q]));
        mom_two_sum2(HH, LL, __fmul2_rn(h2, H[2]));
        LL = __ffma2_rn(h2, mom_add2(L[q], L[2]), LL);
      } else {  // A+-, D
        const float2 t = __fmul2_rn(P, H[q - 2]);
        float2 lo = __ffma2_rn(P, H[q - 2], make_float2(-t.x, -t.y));
        lo = __ffma2_rn(PL, H[q - 2], __ffma2_rn(P, L[q - 2], lo));
        mom_two_sum2(HH, LL, t);
        LL = mom_add2(LL, lo);
      }
      slot[q * kSlot] = make_float4(HH.x, LL.x, HH.y, LL.y);
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) H[q] = L[q] = make_float2(0.f, 0.f);
  }
  __syncthreads();
  // chunk sums as double-floats: thread (q, cell), then the cell's finish
  for (int e = threadIdx.x; e < 5 * kMomCells32; e += kMomThreads) {
    const int q = e / kMomCells32, c = e - q * kMomCells32;
    float2 t = part[0][q][c];
#pragma unroll
    for (int k = 1; k < kMomChunks; ++k) {
      const float2 x = part[k][q][c];
      const float s = t.x + x.x, bp = s - t.x;
      t.y += x.y + ((t.x - (s - bp)) + (x.x - bp));
      t.x = s;
    }
    part[0][q][c] = t;
  }
  __syncthreads();
  const int cl = threadIdx.x, s = blockIdx.x * kMomCells32 + cl;
  if (cl >= kMomCells32 || s >= Z) return;
  double S[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) S[q] = (double)part[0][q][cl].x + (double)part[0][q][cl].y;
  mom_finish(S, s, Z, out, err);
}

// FP64 populations.  w: per velocity two double2 = {a b} {d 0}, then p per radial node.
constexpr int kMomCells64 = 32;

__global__ void __launch_bounds__(kMomThreads)
sod_moments64_kernel(int Z, int ldz, int V, int Qx, const double2* __restrict__ w,
                     const double* __restrict__ f, double* out, int* err) {
  __shared__ double part[kMomChunks][5][kMomCells64];
  const int chunk = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int s0 = blockIdx.x * kMomCells64 + lane;
  const bool active = s0 < ldz;
  const double* pk = reinterpret_cast<const double*>(w + 2 * V);
  int v = (chunk * V) / kMomChunks;
  const int ve = ((chunk + 1) * V) / kMomChunks;
  double S[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  const double* fp = f + s0;
  while (v < ve) {
    const int k = v / Qx, vk = min(ve, (k + 1) * Qx);
    double a = 0.0, b = 0.0, d = 0.0;
    for (; v + 4 <= vk; v += 4) {
      double x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = active ? __ldg(fp + (size_t)(v + u) * ldz) : 0.0;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const double2 ab = __ldg(w + 2 * (v + u)), dd = __ldg(w + 2 * (v + u) + 1);
        a = fma(x[u], ab.x, a);
        b = fma(x[u], ab.y, b);
        d = fma(x[u], dd.x, d);
      }
    }
    for (; v < vk; ++v) {
      const double x = active ? __ldg(fp + (size_t)v * ldz) : 0.0;
      const double2 ab = __ldg(w + 2 * v), dd = __ldg(w + 2 * v + 1);
      a = fma(x, ab.x, a);
      b = fma(x, ab.y, b);
      d = fma(x, dd.x, d);
    }
    const double p = __ldg(pk + k);
    S[0] = fma(0.5, a + d, S[0]);
    S[1] = fma(0.5, b + d, S[1]);
    S[2] = fma(p, a, S[2]);
    S[3] = fma(p, b, S[3]);
    S[4] = fma(p, d, S[4]);
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) part[chunk][q][lane] = S[q];
  __syncthreads();
  if (threadIdx.x < 5 * kMomCells64) {
    const int q = threadIdx.x / kMomCells64, c = threadIdx.x - q * kMomCells64;
    double t = part[0][q][c];
#pragma unroll
    for (int k = 1; k < kMomChunks; ++k) t += part[k][q][c];
    part[0][q][c] = t;
  }
  __syncthreads();
  const int s = blockIdx.x * kMomCells64 + threadIdx.x;
  if (threadIdx.x >= kMomCells64 || s >= Z) return;
  double T[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) T[q] = part[0][q][threadIdx.x];
  mom_finish(T, s, Z, out, err);
}

}  // namespace

size_t sod_moment_weights(bool fp64, int V, int Qx, const double* xi, const double* p, void* out) {
  const int QL = V / Qx;
  const size_t bytes = fp64 ? sizeof(double) * (4 * (size_t)V + QL) : sizeof(float) * (8 * (size_t)V + 2 * QL);
  if (!out) return bytes;
  for (int v = 0; v < V; ++v) {
    const double x = xi[v];
    const double wq[4] = {(1.0 + x) * (1.0 + x), (1.0 - x) * (1.0 - x), (1.0 - x) * (1.0 + x), 0.0};
    for (int q = 0; q < 4; ++q) {
      if (fp64) {
        static_cast<double*>(out)[4 * (size_t)v + q] = wq[q];
      } else {
        float* o = static_cast<float*>(out) + 8 * (size_t)v;
        o[q] = (float)wq[q];
        o[4 + q] = (float)(wq[q] - (double)o[q]);
      }
    }
  }
  for (int k = 0; k < QL; ++k) {
    const double pv = p[(size_t)k * Qx];
    if (fp64) {
      static_cast<double*>(out)[4 * (size_t)V + k] = pv;
    } else {
      float* o = static_cast<float*>(out) + 8 * (size_t)V + 2 * k;
      o[0] = (float)pv;
      o[1] = (float)(pv - (double)o[0]);
    }
  }
  return bytes;
}

template <>
cudaError_t sod_moments_launch<float>(const SodGeom& g, const void* w, const float* f,
                                      double* out, int* err, cudaStream_t st) {
  if (g.Z <= 0) return cudaSuccess;
  sod_moments32_kernel<<<(g.Z + kMomCells32 - 1) / kMomCells32, kMomThreads, 0, st>>>(
      g.Z, g.ldz, g.V, g.Qx, static_cast<const float4*>(w), f, out, err);
  return cudaGetLastError();
}

template <>
cudaError_t sod_moments_launch<double>(const SodGeom& g, const void* w, const double* f,
                                       double* out, int* err, cudaStream_t st) {
  if (g.Z <= 0) return cudaSuccess;
  sod_moments64_kernel<<<(g.Z + kMomCells64 - 1) / kMomCells64, kMomThreads, 0, st>>>(
      g.Z, g.ldz, g.V, g.Qx, static_cast<const double2*>(w), f, out, err);
  return cudaGetLastError();
}

}  // namespace rslb
