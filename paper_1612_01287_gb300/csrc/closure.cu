// closure.cu -- learned closure of a low-order velocity set (an addition to
// the paper's method): a per-cell MLP, trained on data the method generates
// with a high-order velocity set, corrects the low-order populations after
// every RK3 step.
//
//  * restriction R: high-order populations -> low-order ones, per radial
//    node, through the Legendre moments m < Q_lo (exact for m <= 2, so the
//    moments of Eq. macro_jk are preserved);
//  * features of cell s, over n_s = sum_v f_{v,s}: the low-order populations
//    of cell s, f_{s+1} - f_s and f_s - f_{s-1}; then log10(tau);
//  * MLP D -> H -> H -> O with SiLU after the hidden layers, BF16 weights
//    (FP32 master copy for Adam), FP32 biases and accumulation, behind a
//    fixed input/output normalisation fitted to the training data;
//  * correction delta = n_s * out_sd * y, minus its component along the collision
//    invariants (1, p, p xi) in the quadrature-weighted sense, so the cell's
//    N^t, T^tt and T^tz are unchanged; the result is scaled down where it
//    would take more than half of a positive population (a positivity
//    limiter that keeps the conservation).
//
// The network's kernels use four threads per sample (64 samples per CTA; training
// 128), each with a quarter of every layer's outputs in packed FP32x2
// accumulators; activations pass between layers through shared memory, and a
// warp's lanes share the weights they read (broadcasts).  What bounds them are
// the shared-memory broadcasts and latency (application: shared memory 56% of its
// rate, issue slots 45%, FMA pipe 21%, 16 warps per SM; training: 64 CTAs of 16
// warps for a minibatch of 8192, issue slots 51% on their SMs); one thread per
// sample (64 scalar accumulators) left the chip with one warp per scheduler.
// 65536 cells, 73-64-64-24: 78 us per application (163 with one thread per sample);
// a minibatch of 8192 with its update: 76 us (240).  Networks of 16 or 32 hidden
// units and few inputs leave four threads little to do between barriers, so many
// samples of these go by one thread each, in warps that share nothing (Team).
//
// Training: forward and backward of the CTA's samples, then the CTA reduces the
// weight gradients over its samples into a per-CTA partial (a thread holds a
// tile of 4 rows x 3 columns of a layer's gradient); a second kernel sums the
// partials in a fixed order (deterministic) and applies Adam.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <initializer_list>
#include <type_traits>
#include <vector>

#include "mod_range.h"
#include "swap_steps.h"
#include "../../include/rslb.h"
#include "host_common.h"

namespace rslb {
namespace {

constexpr int kMaxD = 128;
constexpr int kMaxO = 32;
constexpr int kNarrowD = 32;                  // one thread per sample: inputs at most
constexpr int kNarrowV = (kNarrowD - 1) / 3;  // and populations of a cell
constexpr int kSmemLimit = 232448 - 2048;  // dynamic; the rest holds the static arrays
constexpr float kLimitTheta = 0.5f;  // positivity limiter of the correction

struct MlpShape {
  int D, H, O;
  int oW1, ob1, oW2, ob2, oW3, ob3, P;
};

MlpShape make_shape(int D, int H, int O) {
  MlpShape s;
  s.D = D;
  s.H = H;
  s.O = O;
  s.oW1 = 0;
  s.ob1 = H * D;
  s.oW2 = s.ob1 + H;
  s.ob2 = s.oW2 + H * H;
  s.oW3 = s.ob2 + H;
  s.ob3 = s.oW3 + O * H;
  s.P = s.ob3 + O;
  return s;
}

constexpr int kNS = 64;    // samples per CTA
constexpr int kParts = 4;  // threads per sample

__host__ __device__ inline int o_pad(const MlpShape& s) { return (s.O + 7) & ~7; }

// Shared-memory weight block (BF16 values widened to FP32): W1T [D][H], W2T [H][H]
// (input-major), W3T [H][OP] (OP = O rounded up to 8, zero columns), b1 [H],
// b2 [H], b3 [OP], then the fixed normalisation mu [D], inv_sd [D], out_sd [OP]
// (the network sees (x - mu) * inv_sd, its output is scaled by out_sd).
struct NetSmem {
  int W1T, W2T, W3T, b1, b2, b3, mu, isd, osd, end;
  __host__ __device__ NetSmem(const MlpShape& s) {
    const int OP = o_pad(s);
    W1T = 0;
    W2T = W1T + s.D * s.H;
    W3T = W2T + s.H * s.H;
    b1 = W3T + s.H * OP;
    b2 = b1 + s.H;
    b3 = b2 + s.H;
    mu = b3 + OP;
    isd = mu + s.D;
    osd = isd + s.D;
    end = (osd + OP + 3) & ~3;
  }
};

__device__ inline void load_weights(const MlpShape& s, const NetSmem& L,
                                    const __nv_bfloat16* __restrict__ wb,
                                    const float* __restrict__ theta,
                                    const float* __restrict__ nrm, float* sw) {
  const int OP = o_pad(s), t = threadIdx.x, nt = blockDim.x;
  // consecutive threads write consecutive shared words; the strided reads of the
  // few KB of weights hit L1
  for (int e = t; e < s.H * s.D; e += nt) {
    const int d = e / s.H, h = e - d * s.H;
    sw[L.W1T + e] = __bfloat162float(wb[s.oW1 + h * s.D + d]);
  }
  for (int e = t; e < s.H * s.H; e += nt) {
    const int i = e / s.H, h = e - i * s.H;
    sw[L.W2T + e] = __bfloat162float(wb[s.oW2 + h * s.H + i]);
  }
  for (int e = t; e < OP * s.H; e += nt) {
    const int i = e / OP, o = e - i * OP;
    sw[L.W3T + e] = o < s.O ? __bfloat162float(wb[s.oW3 + o * s.H + i]) : 0.f;
  }
  for (int e = t; e < s.H; e += nt) {
    sw[L.b1 + e] = theta[s.ob1 + e];
    sw[L.b2 + e] = theta[s.ob2 + e];
  }
  for (int e = t; e < OP; e += nt) {
    sw[L.b3 + e] = e < s.O ? theta[s.ob3 + e] : 0.f;
    sw[L.osd + e] = e < s.O ? nrm[2 * s.D + e] : 1.f;
  }
  for (int e = t; e < 2 * s.D; e += nt) sw[L.mu + e] = nrm[e];
}

__device__ __forceinline__ float silu_f(float a, float* ds) {
  const float sg = 1.f / (1.f + __expf(-a));
  *ds = sg * (1.f + a * (1.f - sg));
  return a * sg;
}

// acc += W^T x for N consecutive outputs (pairs in packed FP32x2): x is the
// sample's input row, w the first of its N columns of the input-major weights.
template <int N>
__device__ __forceinline__ void dense(float2 (&acc)[N / 2], const float* x, int nin,
                                      const float* w, int ldw) {
#pragma unroll 4
  for (int i = 0; i < nin; ++i) {
    const float2 xi = make_float2(x[i], x[i]);
    if constexpr (N % 4 == 0) {
#pragma unroll
      for (int q = 0; q < N / 4; ++q) {
        const float4 v = *reinterpret_cast<const float4*>(w + i * ldw + 4 * q);
        acc[2 * q] = __ffma2_rn(xi, make_float2(v.x, v.y), acc[2 * q]);
        acc[2 * q + 1] = __ffma2_rn(xi, make_float2(v.z, v.w), acc[2 * q + 1]);
      }
    } else {
#pragma unroll
      for (int q = 0; q < N / 2; ++q)
        acc[q] = __ffma2_rn(xi, *reinterpret_cast<const float2*>(w + i * ldw + 2 * q), acc[q]);
    }
  }
}

// One hidden layer: this thread's share (1 / PARTS) of the outputs of its sample;
// with ds, silu' goes there.
template <int H, int PARTS>
__device__ __forceinline__ void hidden(const float* x, int nin, const float* w, const float* b,
                                       int part, float* out, float* ds) {
  constexpr int N = H / PARTS;
  float2 acc[N / 2];
#pragma unroll
  for (int q = 0; q < N / 2; ++q) acc[q] = *reinterpret_cast<const float2*>(b + part * N + 2 * q);
  dense<N>(acc, x, nin, w + part * N, H);
#pragma unroll
  for (int q = 0; q < N; ++q) {
    float d;
    out[part * N + q] = silu_f((q & 1) ? acc[q / 2].y : acc[q / 2].x, &d);
    if (ds) ds[part * N + q] = d;
  }
}

// The output layer: put(o, y) for this thread's share of the OP outputs.
template <int PARTS, typename Put>
__device__ __forceinline__ void outputs(const float* x, int nin, const float* w, const float* b,
                                        int OP, int O, int part, Put put) {
  auto run = [&](auto Nc) {
    constexpr int N = decltype(Nc)::value;
    float2 acc[N / 2];
#pragma unroll
    for (int q = 0; q < N / 2; ++q) acc[q] = *reinterpret_cast<const float2*>(b + part * N + 2 * q);
    dense<N>(acc, x, nin, w + part * N, OP);
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (part * N + q < O) put(part * N + q, (q & 1) ? acc[q / 2].y : acc[q / 2].x);
  };
  switch (OP) {
    case 8: run(std::integral_constant<int, 8 / PARTS>()); break;
    case 16: run(std::integral_constant<int, 16 / PARTS>()); break;
    case 24: run(std::integral_constant<int, 24 / PARTS>()); break;
    default: run(std::integral_constant<int, 32 / PARTS>()); break;
  }
}

// ---------------------------------------------------------------------------
// Training: forward + backward of NS (128, 64 or 32) samples per CTA of 4 NS threads,
// per-CTA partial gradient
// ---------------------------------------------------------------------------
// Sample row in shared memory (pitch odd): [x (D) | h1 (H) | ga1 (H) | h2 (H) |
// ga2 (H) | gy (O)].

// Gradient tile of one layer: rows r0 .. r0 + NR - 1 (activations at column ca of
// the sample rows) x columns lane, lane + 32, ... < ncol (at column cb), and the
// bias gradient (the plain sum of the rows) of those rows.
template <int NR>
__device__ __forceinline__ void grad_tile(const float* act, int pitch, int cnt, int ca, int cb,
                                          int ncol, int r0, int nrow, int lane, float* out,
                                          float* outb) {
  for (int c0 = 0; c0 < ncol; c0 += 96) {
    float acc[NR][3], sum[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      sum[r] = 0.f;
#pragma unroll
      for (int j = 0; j < 3; ++j) acc[r][j] = 0.f;
    }
    // lanes past the last column read column 0 and write nothing
    int cj[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) cj[j] = cb + (c0 + lane + 32 * j < ncol ? c0 + lane + 32 * j : 0);
#pragma unroll 4
    for (int n = 0; n < cnt; ++n) {
      const float* row = act + n * pitch;
      float bv[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) bv[j] = c0 + 32 * j < ncol ? row[cj[j]] : 0.f;
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const float av = row[ca + min(r0 + r, nrow - 1)];
        sum[r] += av;
#pragma unroll
        for (int j = 0; j < 3; ++j)
          if (c0 + 32 * j < ncol) acc[r][j] = fmaf(av, bv[j], acc[r][j]);
      }
    }
#pragma unroll
    for (int r = 0; r < NR; ++r)
      if (r0 + r < nrow) {
#pragma unroll
        for (int j = 0; j < 3; ++j)
          if (c0 + lane + 32 * j < ncol) out[(size_t)(r0 + r) * ncol + c0 + lane + 32 * j] = acc[r][j];
        if (c0 == 0 && lane == 0) outb[r0 + r] = sum[r];
      }
  }
}

// This thread's quarter of the gradient with respect to a layer's inputs, times
// silu': sum over the layer's n outputs (in order) of their gradients g times
// the input-major weights' row of the input.
template <int H, int NMAX>
__device__ __forceinline__ void back_layer(const float* g, int n, const float* wT, int ldw,
                                           int part, float* ds) {
  constexpr int N = H / kParts;
  float gr[NMAX];
#pragma unroll
  for (int h = 0; h < NMAX; ++h) gr[h] = h < n ? g[h] : 0.f;
#pragma unroll 4
  for (int q = 0; q < N; ++q) {
    const float4* w = reinterpret_cast<const float4*>(wT + (part * N + q) * ldw);
    float acc = 0.f;
#pragma unroll
    for (int h = 0; h < NMAX; h += 4)
      if (h < n) {  // zero weights and gradients past n add nothing
        const float4 v = w[h / 4];
        acc = fmaf(v.x, gr[h], acc);
        acc = fmaf(v.y, gr[h + 1], acc);
        acc = fmaf(v.z, gr[h + 2], acc);
        acc = fmaf(v.w, gr[h + 3], acc);
      }
    ds[part * N + q] *= acc;
  }
}

template <int H>
__global__ void __launch_bounds__(512, H == 64 ? 1 : 2)
mlp_train_kernel(MlpShape s, const float* __restrict__ theta, const __nv_bfloat16* __restrict__ wb,
                 const float* __restrict__ nrm, const float* __restrict__ X,
                 const float* __restrict__ T, const int* __restrict__ perm, int n0, int nb,
                 float inv_norm, int pitch, float* part_out, double* lossp) {
  extern __shared__ __align__(16) float smem_f[];
  const NetSmem L(s);
  float* sw = smem_f;
  float* act = sw + L.end;
  __shared__ double red[512 / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int NS = blockDim.x / kParts;
  const int smp = tid % NS, part = tid / NS;
  const int base = blockIdx.x * NS;
  const int cnt = min(NS, nb - base);
  load_weights(s, L, wb, theta, nrm, sw);
  __syncthreads();
  // stage the normalised inputs of the CTA's samples, a warp per row (coalesced)
  for (int r = warp; r < NS; r += nw) {
    int src = 0;
    if (r < cnt) src = perm ? perm[n0 + base + r] : n0 + base + r;
    for (int c = lane; c < s.D; c += 32)
      act[r * pitch + c] =
          r < cnt ? (X[(size_t)src * s.D + c] - sw[L.mu + c]) * sw[L.isd + c] : 0.f;
  }
  __syncthreads();
  float* row = act + smp * pitch;
  float* rh1 = row + s.D;
  float* rg1 = rh1 + H;
  float* rh2 = rg1 + H;
  float* rg2 = rh2 + H;
  float* rgy = rg2 + H;
  // silu'(a1) and silu'(a2) go to the ga1 and ga2 columns, overwritten below
  hidden<H, kParts>(row, s.D, sw + L.W1T, sw + L.b1, part, rh1, rg1);
  __syncthreads();
  hidden<H, kParts>(rh1, H, sw + L.W2T, sw + L.b2, part, rh2, rg2);
  __syncthreads();
  double sq = 0.0;
  {
    const int n = n0 + base + smp;
    const int src = smp < cnt ? (perm ? perm[n] : n) : 0;
    const float* t = T + (size_t)src * s.O;
    outputs<kParts>(rh2, H, sw + L.W3T, sw + L.b3, o_pad(s), s.O, part, [&](int o, float y) {
      const float r = smp < cnt ? y - t[o] / sw[L.osd + o] : 0.f;
      sq += (double)r * r;
      rgy[o] = 2.f * r * inv_norm;
    });
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
  if (lane == 0) red[warp] = sq;
  __syncthreads();
  // layer 3: gh2 = W3^T gy, ga2 = gh2 * silu'(a2); layer 2 likewise
  back_layer<H, kMaxO>(rgy, s.O, sw + L.W3T, o_pad(s), part, rg2);
  __syncthreads();
  back_layer<H, H>(rg2, H, sw + L.W2T, H, part, rg1);
  __syncthreads();
  // weight gradients summed over the CTA's samples in their order; the tiles of the
  // three layers are dealt to the warps as one list, so that a narrow network's
  // few tiles run side by side (16-unit layers: one pass instead of three)
  float* out = part_out + (size_t)blockIdx.x * s.P;
  const int nt1 = H / 4, nt3 = (s.O + 1) / 2;
  for (int j = warp; j < 2 * nt1 + nt3; j += nw) {
    if (j < nt1)
      grad_tile<4>(act, pitch, cnt, s.D + H, 0, s.D, 4 * j, H, lane, out + s.oW1, out + s.ob1);
    else if (j < 2 * nt1)
      grad_tile<4>(act, pitch, cnt, s.D + 3 * H, s.D, H, 4 * (j - nt1), H, lane, out + s.oW2,
                   out + s.ob2);
    else
      grad_tile<2>(act, pitch, cnt, s.D + 4 * H, s.D + 2 * H, H, 2 * (j - 2 * nt1), s.O, lane,
                   out + s.oW3, out + s.ob3);
  }
  if (tid == 0) {
    double t = 0.0;
    for (int i = 0; i < nw; ++i) t += red[i];
    lossp[blockIdx.x] = t;
  }
}

// Sum of the CTAs' partial gradients in their order (deterministic) and, with
// adam, the parameter update; the last CTA sums the losses.
struct AdamStep {
  float* theta;
  float* m;
  float* v;
  __nv_bfloat16* wb;
  float lr, c1, c2;
};

// A CTA takes 32 parameters: its warps bring rounds of kRedRows partials into shared
// memory, many loads in flight, and one warp adds them in order.  A thread per
// parameter that loaded 16 partials at a time, and one that added all losses,
// waited on each load: 7813 partials (10^6 samples) of a 1-16-16-1 network 775 us,
// 64 of a 73-64-64-24 network 5 us.
constexpr int kRedThreads = 256, kRedRows = 128;

__global__ void __launch_bounds__(kRedThreads)
mlp_reduce_kernel(const float* __restrict__ part, int nblk, int P, float* grad,
                  const double* __restrict__ lossp, double loss_scale, double* loss_acc,
                  AdamStep ad) {
  constexpr int kWarps = kRedThreads / 32, kLoads = kRedRows / kWarps;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (blockIdx.x == gridDim.x - 1) {
    __shared__ double red[kRedThreads];
    double t = 0.0;
    for (int b = tid; b < nblk; b += kRedThreads) t += lossp[b];
    red[tid] = t;
    __syncthreads();
    for (int o = kRedThreads / 2; o >= 1; o >>= 1) {
      if (tid < o) red[tid] += red[tid + o];
      __syncthreads();
    }
    if (tid == 0) *loss_acc += red[0] * loss_scale;
    return;
  }
  __shared__ float buf[2][kRedRows][32];
  const int e = blockIdx.x * 32 + lane;
  float g = 0.f;
  for (int b0 = 0, k = 0; b0 < nblk; b0 += kRedRows, k ^= 1) {
    const int n = min(kRedRows, nblk - b0);
    float x[kLoads];
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const int b = warp + kWarps * u;
      x[u] = b < n && e < P ? part[(size_t)(b0 + b) * P + e] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < kLoads; ++u) buf[k][warp + kWarps * u][lane] = x[u];
    // one barrier a round: warp 0 reads buffer k while the others fill k ^ 1, and
    // reaches the next barrier before anyone writes k again
    __syncthreads();
    if (warp == 0) {
#pragma unroll 8
      for (int b = 0; b < n; ++b) g += buf[k][b][lane];
    }
  }
  if (warp != 0 || e >= P) return;
  grad[e] = g;
  if (ad.theta) {
    const float mm = 0.9f * ad.m[e] + 0.1f * g;
    const float vv = 0.999f * ad.v[e] + 0.001f * g * g;
    ad.m[e] = mm;
    ad.v[e] = vv;
    const float th = ad.theta[e] - ad.lr * (mm * ad.c1) / (sqrtf(vv * ad.c2) + 1e-8f);
    ad.theta[e] = th;
    ad.wb[e] = __float2bfloat16_rn(th);
  }
}

__global__ void mlp_round_kernel(const float* __restrict__ theta, int P, __nv_bfloat16* wb) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < P) wb[e] = __float2bfloat16_rn(theta[e]);
}

// Sample row of the inference kernels (pitch odd): [x, then h2 (max(D, H)) | h1, then
// the outputs (max(H, O))].
__host__ __device__ inline int infer_h1(const MlpShape& s) { return s.D > s.H ? s.D : s.H; }
__host__ __device__ inline int infer_pitch(const MlpShape& s) {
  return (infer_h1(s) + (s.H > s.O ? s.H : s.O)) | 1;
}
__host__ __device__ inline size_t infer_smem(const MlpShape& s, int rows) {
  return sizeof(float) * ((size_t)NetSmem(s).end + (size_t)rows * infer_pitch(s));
}

// The samples that go through the layers together: with one thread per sample a
// warp's, which meets no barrier of the CTA, else the CTA's.
template <int PARTS>
struct Team {
  static constexpr int kThreads = PARTS == 1 ? 128 : kNS * PARTS;  // of a CTA
  static constexpr int kRows = kThreads / PARTS;                   // samples of a CTA
  static constexpr int kSize = PARTS == 1 ? 32 : kNS;              // samples of a team
  static constexpr int kWork = kSize * PARTS;                      // threads of a team
  static __device__ __forceinline__ void sync() {
    if constexpr (PARTS == 1) __syncwarp();
    else __syncthreads();
  }
};

// Forward of the team's staged samples.
template <int H, int PARTS, typename Put>
__device__ __forceinline__ void forward_rows(const MlpShape& s, const NetSmem& L, const float* sw,
                                             float* row, int part, Put put) {
  float* r1 = row + infer_h1(s);
  hidden<H, PARTS>(row, s.D, sw + L.W1T, sw + L.b1, part, r1, nullptr);
  Team<PARTS>::sync();
  hidden<H, PARTS>(r1, H, sw + L.W2T, sw + L.b2, part, row, nullptr);
  Team<PARTS>::sync();
  outputs<PARTS>(row, H, sw + L.W3T, sw + L.b3, o_pad(s), s.O, part, put);
  Team<PARTS>::sync();
}

// Inference on given inputs.
template <int H, int PARTS>
__global__ void __launch_bounds__(Team<PARTS>::kThreads)
mlp_infer_kernel(MlpShape s, const float* __restrict__ theta, const __nv_bfloat16* __restrict__ wb,
                 const float* __restrict__ nrm, const float* __restrict__ X, int n, float* Y) {
  using T = Team<PARTS>;
  extern __shared__ __align__(16) float smem_f[];
  const NetSmem L(s);
  float* sw = smem_f;
  const int pitch = infer_pitch(s);
  const int smp = threadIdx.x % T::kRows, row0 = smp / T::kSize * T::kSize;
  const int tid = threadIdx.x % T::kWork;
  float* act = sw + L.end + row0 * pitch;  // the team's rows
  load_weights(s, L, wb, theta, nrm, sw);
  __syncthreads();
  // element e of the team's inputs (outputs) is column e mod D (O) of row e / D (O)
  auto walk = [&](int cnt, int cols, auto f) {
    const int dr = T::kWork / cols, dc = T::kWork - dr * cols;
    int r = tid / cols, c = tid - r * cols;
    for (int e = tid; e < cnt * cols; e += T::kWork) {
      f(e, r, c);
      r += dr;
      c += dc;
      if (c >= cols) {
        c -= cols;
        ++r;
      }
    }
  };
  for (int base = blockIdx.x * T::kRows + row0; base < n; base += gridDim.x * T::kRows) {
    const int cnt = min(T::kSize, n - base);
    const float* x = X + (size_t)base * s.D;
    walk(cnt, s.D, [&](int e, int r, int c) {
      act[r * pitch + c] = (x[e] - sw[L.mu + c]) * sw[L.isd + c];
    });
    T::sync();
    float* row = act + (smp - row0) * pitch;
    const int oy = infer_h1(s);
    forward_rows<H, PARTS>(s, L, sw, row, threadIdx.x / T::kRows,
                           [&](int o, float y) { row[oy + o] = y * sw[L.osd + o]; });
    float* y = Y + (size_t)base * s.O;
    walk(cnt, s.O, [&](int e, int r, int c) { y[e] = act[r * pitch + oy + c]; });
    T::sync();
  }
}

// ---------------------------------------------------------------------------
// Closure kernels (FP32 populations, layout [v][ldz])
// ---------------------------------------------------------------------------
struct ClosureConsts {
  float phi[kMaxO][3];  // (1, p_k, p_k xi_j)
  float w[kMaxO];       // w_j w_k
  float ginv[9];        // (Phi^T W Phi)^{-1}
};

__device__ __forceinline__ void project_add(const ClosureConsts& cc, int V, const float* delta,
                                            float* out) {
  float b0 = 0.f, b1 = 0.f, b2 = 0.f;
  for (int v = 0; v < V; ++v) {
    b0 = fmaf(delta[v], cc.phi[v][0], b0);
    b1 = fmaf(delta[v], cc.phi[v][1], b1);
    b2 = fmaf(delta[v], cc.phi[v][2], b2);
  }
  const float c0 = cc.ginv[0] * b0 + cc.ginv[1] * b1 + cc.ginv[2] * b2;
  const float c1 = cc.ginv[3] * b0 + cc.ginv[4] * b1 + cc.ginv[5] * b2;
  const float c2 = cc.ginv[6] * b0 + cc.ginv[7] * b1 + cc.ginv[8] * b2;
  for (int v = 0; v < V; ++v)
    out[v] = delta[v] - cc.w[v] * (c0 * cc.phi[v][0] + c1 * cc.phi[v][1] + c2 * cc.phi[v][2]);
}

// f_out = f_in + projected correction; PARTS threads per cell.
template <int H, int PARTS>
__global__ void __launch_bounds__(Team<PARTS>::kThreads)
closure_apply_kernel(MlpShape s, const float* __restrict__ theta,
                     const __nv_bfloat16* __restrict__ wb, const float* __restrict__ nrm,
                     const float* __restrict__ fin, float* fout, int Z, int ldz, float logtau,
                     ClosureConsts cc) {
  using T = Team<PARTS>;
  extern __shared__ __align__(16) float smem_f[];
  __shared__ float lim[PARTS][T::kRows];
  constexpr int kMaxV4 = PARTS == 1 ? kNarrowV : kMaxO / PARTS;
  const NetSmem L(s);
  float* sw = smem_f;
  float* act = sw + L.end;
  const int pitch = infer_pitch(s);
  const int V = s.O, part = threadIdx.x / T::kRows, smp = threadIdx.x % T::kRows;
  const int row0 = smp / T::kSize * T::kSize;
  load_weights(s, L, wb, theta, nrm, sw);
  __syncthreads();
  const float* mu = sw + L.mu;
  const float* isd = sw + L.isd;
  for (int base = blockIdx.x * T::kRows + row0; base < Z; base += gridDim.x * T::kRows) {
    const int cell = base + smp - row0, c = min(cell, Z - 1);
    const bool live = cell < Z;
    const int cl = c > 0 ? c - 1 : 0, cr = c < Z - 1 ? c + 1 : Z - 1;
    float* row = act + smp * pitch;
    // this thread's populations v = part + 4 j and their neighbours, all loads at
    // once; kept for the limiter and the update
    float fc[kMaxV4], fr[kMaxV4], fl[kMaxV4], np = 0.f;
#pragma unroll
    for (int j = 0; j < kMaxV4; ++j) {
      const int v = part + PARTS * j;
      const float* f = fin + (size_t)v * ldz;
      fc[j] = v < V ? f[c] : 0.f;
      fr[j] = v < V ? f[cr] : 0.f;
      fl[j] = v < V ? f[cl] : 0.f;
    }
#pragma unroll
    for (int j = 0; j < kMaxV4; ++j) np += fc[j];
    lim[part][smp] = np;
    T::sync();
    float n = lim[0][smp];
    if constexpr (PARTS == 4) n = (lim[0][smp] + lim[1][smp]) + (lim[2][smp] + lim[3][smp]);
    const float inv_n = 1.f / n;
    // features: f_s, f_{s+1} - f_s, f_s - f_{s-1} (over n_s), log10 tau
#pragma unroll
    for (int j = 0; j < kMaxV4; ++j) {
      const int v = part + PARTS * j;
      if (v < V) {
        row[v] = (fc[j] * inv_n - mu[v]) * isd[v];
        row[V + v] = ((fr[j] - fc[j]) * inv_n - mu[V + v]) * isd[V + v];
        row[2 * V + v] = ((fc[j] - fl[j]) * inv_n - mu[2 * V + v]) * isd[2 * V + v];
      }
    }
    if (part == 0) row[3 * V] = (logtau - mu[3 * V]) * isd[3 * V];
    T::sync();
    float* dl = row + infer_h1(s);
    forward_rows<H, PARTS>(s, L, sw, row, part,
                    [&](int o, float y) { dl[o] = n * sw[L.osd + o] * y; });
    // the correction without its component along the collision invariants
    const float* delta = dl;
    float b0 = 0.f, b1 = 0.f, b2 = 0.f;
    for (int v = 0; v < V; ++v) {
      b0 = fmaf(delta[v], cc.phi[v][0], b0);
      b1 = fmaf(delta[v], cc.phi[v][1], b1);
      b2 = fmaf(delta[v], cc.phi[v][2], b2);
    }
    const float c0 = cc.ginv[0] * b0 + cc.ginv[1] * b1 + cc.ginv[2] * b2;
    const float c1 = cc.ginv[3] * b0 + cc.ginv[4] * b1 + cc.ginv[5] * b2;
    const float c2 = cc.ginv[6] * b0 + cc.ginv[7] * b1 + cc.ginv[8] * b2;
    auto corr = [&](int v) {
      return delta[v] -
             cc.w[v] * (c0 * cc.phi[v][0] + c1 * cc.phi[v][1] + c2 * cc.phi[v][2]);
    };
    // positivity limiter: scale the (conserving) correction so that no
    // positive population loses more than kLimitTheta of itself
    float alpha = 1.f;
#pragma unroll
    for (int j = 0; j < kMaxV4; ++j) {
      const int v = part + PARTS * j;
      if (v < V) {
        fr[j] = corr(v);
        if (fc[j] > 0.f && fr[j] < 0.f) alpha = fminf(alpha, kLimitTheta * fc[j] / -fr[j]);
      }
    }
    lim[part][smp] = alpha;
    T::sync();
#pragma unroll
    for (int q = 0; q < PARTS; ++q) alpha = fminf(alpha, lim[q][smp]);
#pragma unroll
    for (int j = 0; j < kMaxV4; ++j) {
      const int v = part + PARTS * j;
      if (live && v < V) fout[(size_t)v * ldz + c] = fc[j] + alpha * fr[j];
    }
    T::sync();
  }
}

// Restriction, thread per cell: f_lo[k*Ql + i] = sum_j R[i][j] f_hi[k*Qh + j].
__global__ void restrict_kernel(const float* __restrict__ fh, int ldh, int Qh,
                                float* fl, int ldl, int Ql, int QL, const float* __restrict__ Rm,
                                int Z) {
  extern __shared__ float Rs[];
  for (int e = threadIdx.x; e < Ql * Qh; e += blockDim.x) Rs[e] = Rm[e];
  __syncthreads();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= Z) return;
  for (int k = 0; k < QL; ++k) {
    float acc[kMaxO];
    for (int i = 0; i < Ql; ++i) acc[i] = 0.f;
    for (int j = 0; j < Qh; ++j) {
      const float f = fh[(size_t)(k * Qh + j) * ldh + c];
      for (int i = 0; i < Ql; ++i) acc[i] = fmaf(Rs[i * Qh + j], f, acc[i]);
    }
    for (int i = 0; i < Ql; ++i) fl[(size_t)(k * Ql + i) * ldl + c] = acc[i];
  }
}

// Features of the low-order state (rows of X) and n_s: f_s, f_{s+1} - f_s,
// f_s - f_{s-1}, all over n_s, then log10 tau.
__global__ void features_kernel(const float* __restrict__ f, int Z, int ldz, int V, float logtau,
                                float* X, float* ns) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= Z) return;
  const int cl = c > 0 ? c - 1 : 0, cr = c < Z - 1 ? c + 1 : Z - 1;
  float n = 0.f;
  for (int v = 0; v < V; ++v) n += f[(size_t)v * ldz + c];
  ns[c] = n;
  const float inv = 1.f / n;
  float* row = X + (size_t)c * (3 * V + 1);
  for (int v = 0; v < V; ++v) {
    const float fc = f[(size_t)v * ldz + c];
    row[v] = fc * inv;
    row[V + v] = (f[(size_t)v * ldz + cr] - fc) * inv;
    row[2 * V + v] = (fc - f[(size_t)v * ldz + cl]) * inv;
  }
  row[3 * V] = logtau;
}

// Targets: T[s] = P(f_ref[s] - f_pred[s]) / n_s.
__global__ void target_kernel(const float* __restrict__ fref, const float* __restrict__ fpred,
                              const float* __restrict__ ns, int Z, int ldz, int V,
                              ClosureConsts cc, float* T) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= Z) return;
  float d[kMaxO], p[kMaxO];
  for (int v = 0; v < V; ++v) d[v] = fref[(size_t)v * ldz + c] - fpred[(size_t)v * ldz + c];
  project_add(cc, V, d, p);
  const float inv = 1.f / ns[c];
  for (int v = 0; v < V; ++v) T[(size_t)c * V + v] = p[v] * inv;
}

// ---------------------------------------------------------------------------
// host helpers
// ---------------------------------------------------------------------------
// Column statistics for the normalisation, one CTA per column (fixed-order
// tree reductions in FP64, two passes for the variance): columns of X give
// mu and 1/sd, columns of T give the root-mean-square (1 for constant or
// zero columns).
__global__ void fit_norm_kernel(const float* __restrict__ X, const float* __restrict__ T, int n,
                                int D, int O, float* nrm) {
  __shared__ double red[256];
  const int col = blockIdx.x, tid = threadIdx.x;
  const bool is_x = col < D;
  const float* src = is_x ? X + col : T + (col - D);
  const int stride = is_x ? D : O;
  auto reduce = [&](double v) {
    red[tid] = v;
    __syncthreads();
    for (int o = 128; o >= 1; o >>= 1) {
      if (tid < o) red[tid] += red[tid + o];
      __syncthreads();
    }
    const double r = red[0];
    __syncthreads();
    return r;
  };
  double a = 0.0;
  for (int r = tid; r < n; r += 256) a += (double)src[(size_t)r * stride];
  const double mean = reduce(a) / n;
  double b = 0.0;
  for (int r = tid; r < n; r += 256) {
    const double x = (double)src[(size_t)r * stride];
    const double d = is_x ? x - mean : x;
    b += d * d;
  }
  const double sd = sqrt(reduce(b) / n);
  if (tid == 0) {
    if (is_x) {
      nrm[col] = (float)mean;
      nrm[D + col] = sd > 0.0 ? (float)(1.0 / sd) : 1.f;
    } else {
      nrm[2 * D + (col - D)] = sd > 0.0 ? (float)sd : 1.f;
    }
  }
}

uint64_t splitmix(uint64_t& x) {
  uint64_t z = (x += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

double unit_normal(uint64_t& st) {
  const double u1 = ((splitmix(st) >> 11) + 0.5) * (1.0 / 9007199254740992.0);
  const double u2 = ((splitmix(st) >> 11) + 0.5) * (1.0 / 9007199254740992.0);
  return std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2);
}

int closure_consts(int Q, int QL, ClosureConsts* cc) {
  const int V = Q * QL;
  if (V > kMaxO) return RSLB_ERR_UNSUPPORTED;
  std::vector<double> xi(Q), w(Q), xk(QL), wk(QL);
  gauss_legendre_host(Q, xi.data(), w.data());
  gauss_laguerre2_host(QL, xk.data(), wk.data());
  double G[9] = {0};
  std::memset(cc, 0, sizeof(*cc));
  for (int k = 0; k < QL; ++k)
    for (int j = 0; j < Q; ++j) {
      const int v = k * Q + j;
      const double ph[3] = {1.0, xk[k], xk[k] * xi[j]};
      const double wv = w[j] * wk[k];
      for (int a = 0; a < 3; ++a) {
        cc->phi[v][a] = (float)ph[a];
        for (int b = 0; b < 3; ++b) G[3 * a + b] += ph[a] * wv * ph[b];
      }
      cc->w[v] = (float)wv;
    }
  // 3x3 inverse by cofactors
  const double det = G[0] * (G[4] * G[8] - G[5] * G[7]) - G[1] * (G[3] * G[8] - G[5] * G[6]) +
                     G[2] * (G[3] * G[7] - G[4] * G[6]);
  if (!(std::fabs(det) > 0.0)) return RSLB_ERR_ARG;
  const double inv[9] = {(G[4] * G[8] - G[5] * G[7]) / det, (G[2] * G[7] - G[1] * G[8]) / det,
                         (G[1] * G[5] - G[2] * G[4]) / det, (G[5] * G[6] - G[3] * G[8]) / det,
                         (G[0] * G[8] - G[2] * G[6]) / det, (G[2] * G[3] - G[0] * G[5]) / det,
                         (G[3] * G[7] - G[4] * G[6]) / det, (G[1] * G[6] - G[0] * G[7]) / det,
                         (G[0] * G[4] - G[1] * G[3]) / det};
  for (int i = 0; i < 9; ++i) cc->ginv[i] = (float)inv[i];
  return RSLB_OK;
}

}  // namespace
}  // namespace rslb

using namespace rslb;

struct rslb_mlp {
  MlpShape s;
  cudaStream_t stream;
  float* norm;  // mu [D] | inv_sd [D] | out_sd [O]
  float* theta;
  __nv_bfloat16* wb;
  float* grad;
  float* m;
  float* v;
  float* part;
  double* lossp;
  double* loss_acc;
  int* perm;
  int part_blocks;
  int infer_places[2], apply_places[2];  // CTAs the GPU holds, [0]: four threads per
                                         // sample, [1]: one
  int perm_n;
  long long adam_t;
};

namespace {

int mlp_pitch(const MlpShape& s) {
  int p = s.D + 4 * s.H + s.O;
  return (p % 2) ? p : p + 1;
}

size_t train_smem(const MlpShape& s, int ns) {
  return sizeof(float) * ((size_t)NetSmem(s).end + (size_t)ns * mlp_pitch(s));
}

// Samples per CTA of the training kernel (0: the network does not fit).
int train_ns(const MlpShape& s) {
  for (int ns = 128; ns >= 32; ns /= 2)
    if (train_smem(s, ns) <= (size_t)kSmemLimit) return ns;
  return 0;
}

template <typename F>
cudaError_t dispatch_h(int H, F f) {
  switch (H) {
    case 16: return f(std::integral_constant<int, 16>());
    case 32: return f(std::integral_constant<int, 32>());
    case 64: return f(std::integral_constant<int, 64>());
    default: return cudaErrorInvalidValue;
  }
}

void mlp_free(rslb_mlp* m) {
  if (!m) return;
  void* p[] = {m->theta, m->wb, m->grad, m->m, m->v, m->part, m->lossp, m->loss_acc, m->perm,
               m->norm};
  for (void* x : p)
    if (x) cudaFree(x);
  delete m;
}

// One thread per sample of a network with few inputs, from `many` samples on; four
// otherwise.  f(H, PARTS).
template <typename F>
cudaError_t dispatch_team(const MlpShape& s, int n, int many, F f) {
  return dispatch_h(s.H, [&](auto Hc) {
    if constexpr (decltype(Hc)::value <= 32)
      if (s.D <= kNarrowD && n >= many) return f(Hc, std::integral_constant<int, 1>());
    return f(Hc, std::integral_constant<int, kParts>());
  });
}

// Where one thread per sample overtakes four (us, one / four threads).  Inference: 16
// units 9.0 / 8.6 at 30000 samples of 1-16-16-1, 10.6 / 10.6 at 60000 and 11.0 / 13.0
// at 100000, 15.1 / 15.1 and 18.7 / 20.8 at the last two of 31-16-16-10; 32 units
// 49.1 / 47.6 at 300000 of 2-32-32-1 and 119 / 140 at 10^6, 74.8 / 76.6 and 228 /
// 244 of 31-32-32-10.  Closure steps: 4 populations, 16 units 46.2 / 48.3 at 30000
// cells and 62.6 / 68.2 at 65536; 10 populations, 32 units 56.7 / 54.5 and 75.0 /
// 81.1.
constexpr int kApplyMany = 49152;
int infer_many(const MlpShape& s) { return s.H == 16 ? kApplyMany : 327680; }

// CTAs of a kernel that the GPU holds at once.  The inference kernels' CTAs load the
// weights once and walk groups of samples, so there are as many as this (registers
// and threads count, not the shared memory alone: a second, partial wave of
// long-lived CTAs doubles the time).
cudaError_t places_of(const void* kernel, int threads, size_t smem, int* places) {
  int dev = 0, nsm = 0, per = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem);
  *places = std::max(per, 1) * std::max(nsm, 1);
  return e;
}

template <int H, int PARTS>
cudaError_t prepare_team(rslb_mlp* m, int i) {
  using T = Team<PARTS>;
  const void* infer = (const void*)mlp_infer_kernel<H, PARTS>;
  const void* apply = (const void*)closure_apply_kernel<H, PARTS>;
  const size_t smem = infer_smem(m->s, T::kRows);
  cudaError_t e = cudaSuccess;
  for (const void* f : {infer, apply})
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
  if (e == cudaSuccess) e = places_of(infer, T::kThreads, smem, &m->infer_places[i]);
  if (e == cudaSuccess) e = places_of(apply, T::kThreads, smem, &m->apply_places[i]);
  return e;
}

// Opts the network's kernels into large shared memory and counts their places.
cudaError_t prepare_kernels(rslb_mlp* m) {
  return dispatch_h(m->s.H, [&](auto Hc) {
    constexpr int H = decltype(Hc)::value;
    cudaError_t e =
        cudaFuncSetAttribute((const void*)mlp_train_kernel<H>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    if (e == cudaSuccess) e = prepare_team<H, kParts>(m, 0);
    if constexpr (H <= 32)
      if (e == cudaSuccess && m->s.D <= kNarrowD) e = prepare_team<H, 1>(m, 1);
    return e;
  });
}

// Gradient of the mean-squared loss over samples [n0, n0 + nb) of the
// (permuted) data into m->grad; adds loss * loss_scale to m->loss_acc; with adam,
// the update follows in the same kernel as the sum of the partials.
cudaError_t mlp_batch_grad(rslb_mlp* m, const float* X, const float* T, const int* perm, int n0,
                           int nb, double loss_scale, const AdamStep& adam) {
  const MlpShape& s = m->s;
  const int ns = train_ns(s);
  const int nblk = (nb + ns - 1) / ns;
  if (nblk > m->part_blocks) {
    if (m->part) cudaFree(m->part);
    if (m->lossp) cudaFree(m->lossp);
    m->part = nullptr;
    m->lossp = nullptr;
    if (cudaMalloc((void**)&m->part, sizeof(float) * (size_t)nblk * s.P) != cudaSuccess ||
        cudaMalloc((void**)&m->lossp, sizeof(double) * nblk) != cudaSuccess)
      return cudaErrorMemoryAllocation;
    m->part_blocks = nblk;
  }
  const float inv_norm = 1.f / ((float)nb * (float)s.O);
  cudaError_t e = dispatch_h(s.H, [&](auto Hc) {
    constexpr int H = decltype(Hc)::value;
    mlp_train_kernel<H><<<nblk, ns * kParts, train_smem(s, ns), m->stream>>>(
        s, m->theta, m->wb, m->norm, X, T, perm, n0, nb, inv_norm, mlp_pitch(s), m->part,
        m->lossp);
    return cudaGetLastError();
  });
  if (e != cudaSuccess) return e;
  mlp_reduce_kernel<<<(s.P + 31) / 32 + 1, kRedThreads, 0, m->stream>>>(
      m->part, nblk, s.P, m->grad, m->lossp, loss_scale, m->loss_acc, adam);
  return cudaGetLastError();
}

}  // namespace

extern "C" int rslb_mlp_create(rslb_mlp** out, int n_in, int n_hidden, int n_out,
                               unsigned long long seed, void* stream) {
  clear_error();
  if (!out) return set_error(RSLB_ERR_ARG, "rslb_mlp_create: NULL output");
  *out = nullptr;
  if (n_in < 1 || n_in > kMaxD || n_out < 1 || n_out > kMaxO ||
      (n_hidden != 16 && n_hidden != 32 && n_hidden != 64))
    return set_error(RSLB_ERR_ARG,
                     "rslb_mlp_create: need 1 <= n_in <= %d, n_hidden in {16, 32, 64}, "
                     "1 <= n_out <= %d",
                     kMaxD, kMaxO);
  rslb_mlp* m = new rslb_mlp();
  std::memset(m, 0, sizeof(*m));
  m->s = make_shape(n_in, n_hidden, n_out);
  m->stream = (cudaStream_t)stream;
  const int P = m->s.P;
  if (train_ns(m->s) == 0) {
    delete m;
    return set_error(RSLB_ERR_UNSUPPORTED, "rslb_mlp_create: network too large for a CTA");
  }
  // initial parameters: weights N(0, 1/fan_in) (output layer scaled by 0.1),
  // biases zero
  std::vector<float> th(P, 0.f);
  uint64_t st = seed ^ 0x243F6A8885A308D3ull;
  const MlpShape& s = m->s;
  for (int e = 0; e < s.H * s.D; ++e) th[s.oW1 + e] = (float)(unit_normal(st) / std::sqrt(s.D));
  for (int e = 0; e < s.H * s.H; ++e) th[s.oW2 + e] = (float)(unit_normal(st) / std::sqrt(s.H));
  for (int e = 0; e < s.O * s.H; ++e)
    th[s.oW3 + e] = (float)(0.1 * unit_normal(st) / std::sqrt(s.H));
  bool ok = cudaMalloc((void**)&m->theta, sizeof(float) * P) == cudaSuccess &&
            cudaMalloc((void**)&m->wb, sizeof(__nv_bfloat16) * P) == cudaSuccess &&
            cudaMalloc((void**)&m->grad, sizeof(float) * P) == cudaSuccess &&
            cudaMalloc((void**)&m->m, sizeof(float) * P) == cudaSuccess &&
            cudaMalloc((void**)&m->v, sizeof(float) * P) == cudaSuccess &&
            cudaMalloc((void**)&m->loss_acc, sizeof(double)) == cudaSuccess &&
            cudaMalloc((void**)&m->norm, sizeof(float) * (2 * s.D + s.O)) == cudaSuccess;
  if (!ok) {
    mlp_free(m);
    return set_error(RSLB_ERR_ALLOC, "rslb_mlp_create: cudaMalloc failed");
  }
  std::vector<float> nrm(2 * s.D + s.O, 1.f);
  for (int d = 0; d < s.D; ++d) nrm[d] = 0.f;  // mu = 0, inv_sd = 1, out_sd = 1
  cudaError_t e = prepare_kernels(m);
  if (e == cudaSuccess)
    e = cudaMemcpy(m->norm, nrm.data(), sizeof(float) * nrm.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(m->theta, th.data(), sizeof(float) * P, cudaMemcpyHostToDevice, m->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(m->m, 0, sizeof(float) * P, m->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(m->v, 0, sizeof(float) * P, m->stream);
  if (e == cudaSuccess) {
    mlp_round_kernel<<<(P + 255) / 256, 256, 0, m->stream>>>(m->theta, P, m->wb);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  if (e != cudaSuccess) {
    mlp_free(m);
    return cuda_error(e, "rslb_mlp_create");
  }
  *out = m;
  return RSLB_OK;
}

extern "C" int rslb_mlp_num_params(const rslb_mlp* m) { return m ? m->s.P : 0; }

extern "C" int rslb_mlp_get_params(rslb_mlp* m, float* theta) {
  clear_error();
  if (!m || !theta) return set_error(RSLB_ERR_ARG, "rslb_mlp_get_params: NULL argument");
  cudaError_t e = cudaMemcpyAsync(theta, m->theta, sizeof(float) * m->s.P, cudaMemcpyDeviceToHost,
                                  m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  return e == cudaSuccess ? RSLB_OK : cuda_error(e, "rslb_mlp_get_params");
}

extern "C" int rslb_mlp_set_params(rslb_mlp* m, const float* theta) {
  clear_error();
  if (!m || !theta) return set_error(RSLB_ERR_ARG, "rslb_mlp_set_params: NULL argument");
  const int P = m->s.P;
  cudaError_t e =
      cudaMemcpyAsync(m->theta, theta, sizeof(float) * P, cudaMemcpyHostToDevice, m->stream);
  if (e == cudaSuccess) {
    mlp_round_kernel<<<(P + 255) / 256, 256, 0, m->stream>>>(m->theta, P, m->wb);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(m->m, 0, sizeof(float) * P, m->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(m->v, 0, sizeof(float) * P, m->stream);
  m->adam_t = 0;
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  return e == cudaSuccess ? RSLB_OK : cuda_error(e, "rslb_mlp_set_params");
}

extern "C" int rslb_mlp_set_normalization(rslb_mlp* m, const float* mu, const float* inv_sd,
                                          const float* out_sd) {
  clear_error();
  if (!m || !mu || !inv_sd || !out_sd)
    return set_error(RSLB_ERR_ARG, "rslb_mlp_set_normalization: NULL argument");
  const MlpShape& s = m->s;
  std::vector<float> h(2 * s.D + s.O);
  std::memcpy(h.data(), mu, sizeof(float) * s.D);
  std::memcpy(h.data() + s.D, inv_sd, sizeof(float) * s.D);
  std::memcpy(h.data() + 2 * s.D, out_sd, sizeof(float) * s.O);
  cudaError_t e = cudaMemcpyAsync(m->norm, h.data(), sizeof(float) * h.size(),
                                  cudaMemcpyHostToDevice, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  return e == cudaSuccess ? RSLB_OK : cuda_error(e, "rslb_mlp_set_normalization");
}

extern "C" int rslb_mlp_get_normalization(rslb_mlp* m, float* mu, float* inv_sd, float* out_sd) {
  clear_error();
  if (!m || !mu || !inv_sd || !out_sd)
    return set_error(RSLB_ERR_ARG, "rslb_mlp_get_normalization: NULL argument");
  const MlpShape& s = m->s;
  std::vector<float> h(2 * s.D + s.O);
  cudaError_t e = cudaMemcpyAsync(h.data(), m->norm, sizeof(float) * h.size(),
                                  cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  if (e != cudaSuccess) return cuda_error(e, "rslb_mlp_get_normalization");
  std::memcpy(mu, h.data(), sizeof(float) * s.D);
  std::memcpy(inv_sd, h.data() + s.D, sizeof(float) * s.D);
  std::memcpy(out_sd, h.data() + 2 * s.D, sizeof(float) * s.O);
  return RSLB_OK;
}

extern "C" int rslb_mlp_fit_normalization(rslb_mlp* m, const float* X, const float* T, int n) {
  clear_error();
  if (!m || !X || !T || n < 1)
    return set_error(RSLB_ERR_ARG, "rslb_mlp_fit_normalization: bad arguments");
  const MlpShape& s = m->s;
  fit_norm_kernel<<<s.D + s.O, 256, 0, m->stream>>>(X, T, n, s.D, s.O, m->norm);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  return e == cudaSuccess ? RSLB_OK : cuda_error(e, "rslb_mlp_fit_normalization");
}

extern "C" int rslb_mlp_forward(rslb_mlp* m, const float* X, int n, float* Y) {
  clear_error();
  if (!m || !X || !Y || n < 0) return set_error(RSLB_ERR_ARG, "rslb_mlp_forward: bad arguments");
  if (n == 0) return RSLB_OK;
  const MlpShape& s = m->s;
  cudaError_t e = dispatch_team(s, n, infer_many(s), [&](auto Hc, auto Pc) {
    constexpr int H = decltype(Hc)::value, PARTS = decltype(Pc)::value;
    using T = Team<PARTS>;
    const int grid = std::min((n + T::kRows - 1) / T::kRows, m->infer_places[PARTS == 1]);
    mlp_infer_kernel<H, PARTS><<<grid, T::kThreads, infer_smem(s, T::kRows), m->stream>>>(
        s, m->theta, m->wb, m->norm, X, n, Y);
    return cudaGetLastError();
  });
  return e == cudaSuccess ? RSLB_OK : cuda_error(e, "rslb_mlp_forward");
}

extern "C" int rslb_mlp_loss_grad(rslb_mlp* m, const float* X, const float* T, int n,
                                  double* loss, float* grad) {
  clear_error();
  if (!m || !X || !T || n < 1) return set_error(RSLB_ERR_ARG, "rslb_mlp_loss_grad: bad arguments");
  cudaError_t e = cudaMemsetAsync(m->loss_acc, 0, sizeof(double), m->stream);
  if (e == cudaSuccess)
    e = mlp_batch_grad(m, X, T, nullptr, 0, n, 1.0 / ((double)n * m->s.O), AdamStep{});
  double L = 0.0;
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(&L, m->loss_acc, sizeof(double), cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess && grad)
    e = cudaMemcpyAsync(grad, m->grad, sizeof(float) * m->s.P, cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  if (e != cudaSuccess) return cuda_error(e, "rslb_mlp_loss_grad");
  if (loss) *loss = L;
  return RSLB_OK;
}

extern "C" int rslb_mlp_train(rslb_mlp* m, const float* X, const float* T, int n, int epochs,
                              int batch, double lr, unsigned long long seed, double* epoch_loss) {
  clear_error();
  if (!m || !X || !T || n < 1 || epochs < 0 || batch < 1 || !(lr > 0.0))
    return set_error(RSLB_ERR_ARG, "rslb_mlp_train: bad arguments");
  if (n > m->perm_n) {
    if (m->perm) cudaFree(m->perm);
    m->perm = nullptr;
    if (cudaMalloc((void**)&m->perm, sizeof(int) * (size_t)n) != cudaSuccess)
      return set_error(RSLB_ERR_ALLOC, "rslb_mlp_train: cudaMalloc failed");
    m->perm_n = n;
  }
  std::vector<int> perm(n);
  uint64_t st = seed ^ 0x13198A2E03707344ull;
  cudaError_t e = cudaSuccess;
  for (int ep = 0; ep < epochs && e == cudaSuccess; ++ep) {
    for (int i = 0; i < n; ++i) perm[i] = i;
    for (int i = n - 1; i > 0; --i)
      std::swap(perm[i], perm[mod_range(splitmix(st), (uint32_t)i + 1)]);
    e = cudaMemcpyAsync(m->perm, perm.data(), sizeof(int) * (size_t)n, cudaMemcpyHostToDevice,
                        m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->loss_acc, 0, sizeof(double), m->stream);
    for (int n0 = 0; n0 < n && e == cudaSuccess; n0 += batch) {
      const int nb = std::min(batch, n - n0);
      m->adam_t += 1;
      const double c1 = 1.0 / (1.0 - std::pow(0.9, (double)m->adam_t));
      const double c2 = 1.0 / (1.0 - std::pow(0.999, (double)m->adam_t));
      e = mlp_batch_grad(m, X, T, m->perm, n0, nb, 1.0 / ((double)n * m->s.O),
                         AdamStep{m->theta, m->m, m->v, m->wb, (float)lr, (float)c1, (float)c2});
    }
    if (e == cudaSuccess && epoch_loss) {
      // the stream-ordered copy lands before the host buffer is read at the sync below
      e = cudaMemcpyAsync(epoch_loss + ep, m->loss_acc, sizeof(double), cudaMemcpyDeviceToHost,
                          m->stream);
      if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    }
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  return e == cudaSuccess ? RSLB_OK : cuda_error(e, "rslb_mlp_train");
}

extern "C" void rslb_mlp_destroy(rslb_mlp* m) {
  if (!m) return;
  cudaStreamSynchronize(m->stream);
  mlp_free(m);
}

// ---------------------------------------------------------------------------
// closure entry points
// ---------------------------------------------------------------------------
namespace {

int check_pair(rslb_handle* hi, rslb_handle* lo, SodView* vh, SodView* vl, const char* what) {
  if (sod_view(hi, vh) || sod_view(lo, vl)) return set_error(RSLB_ERR_ARG, "%s: NULL handle", what);
  if (vh->fp64 || vl->fp64) return set_error(RSLB_ERR_UNSUPPORTED, "%s: needs RSLB_F32 handles", what);
  if (vh->Z != vl->Z || vh->Q_L != vl->Q_L || vh->Q_xi < vl->Q_xi || vl->V > kMaxO)
    return set_error(RSLB_ERR_ARG,
                     "%s: handles need equal Z and Q_L, Q_xi(hi) >= Q_xi(lo), Q_L*Q_xi(lo) <= %d",
                     what, kMaxO);
  return RSLB_OK;
}

// R[i][j] = w_i sum_{m < Ql} (2m+1)/2 P_m(xi^lo_i) P_m(xi^hi_j), FP64 -> FP32.
cudaError_t upload_restriction(int Qh, int Ql, float** dev, cudaStream_t st) {
  std::vector<double> xh(Qh), wh(Qh), xl(Ql), wl(Ql);
  gauss_legendre_host(Qh, xh.data(), wh.data());
  gauss_legendre_host(Ql, xl.data(), wl.data());
  std::vector<float> R((size_t)Ql * Qh);
  for (int i = 0; i < Ql; ++i)
    for (int j = 0; j < Qh; ++j) {
      double acc = 0.0;
      for (int mm = 0; mm < Ql; ++mm)
        acc += 0.5 * (2.0 * mm + 1.0) * legendre_p(mm, xl[i]) * legendre_p(mm, xh[j]);
      R[(size_t)i * Qh + j] = (float)(wl[i] * acc);
    }
  cudaError_t e = cudaMalloc((void**)dev, sizeof(float) * R.size());
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(*dev, R.data(), sizeof(float) * R.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return e;
}

cudaError_t launch_restrict(const SodView& vh, const SodView& vl, const float* R, float* dst,
                            cudaStream_t st) {
  const int T = 128;
  restrict_kernel<<<(vh.Z + T - 1) / T, T, sizeof(float) * vl.Q_xi * vh.Q_xi, st>>>(
      (const float*)vh.F0, vh.ldz, vh.Q_xi, dst, vl.ldz, vl.Q_xi, vl.Q_L, R, vh.Z);
  return cudaGetLastError();
}

}  // namespace

extern "C" int rslb_restrict(rslb_handle* hi, rslb_handle* lo) {
  clear_error();
  SodView vh, vl;
  int rc = check_pair(hi, lo, &vh, &vl, "rslb_restrict");
  if (rc) return rc;
  float* R = nullptr;
  cudaError_t e = cudaStreamSynchronize(vh.stream);
  if (e == cudaSuccess) e = upload_restriction(vh.Q_xi, vl.Q_xi, &R, vl.stream);
  if (e == cudaSuccess) e = launch_restrict(vh, vl, R, (float*)vl.F0, vl.stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(vl.stream);
  if (R) cudaFree(R);
  return e == cudaSuccess ? RSLB_OK : cuda_error(e, "rslb_restrict");
}

extern "C" int rslb_closure_sample(rslb_handle* hi, rslb_handle* lo, double tau, float* X,
                                   float* T) {
  clear_error();
  SodView vh, vl;
  int rc = check_pair(hi, lo, &vh, &vl, "rslb_closure_sample");
  if (rc) return rc;
  if (!X || !T || !(tau > 0.0)) return set_error(RSLB_ERR_ARG, "rslb_closure_sample: bad arguments");
  ClosureConsts cc;
  rc = closure_consts(vl.Q_xi, vl.Q_L, &cc);
  if (rc) return set_error(rc, "rslb_closure_sample: low-order set too large");
  float *R = nullptr, *ns = nullptr, *ref = nullptr;
  cudaStream_t st = vl.stream;
  cudaError_t e = cudaStreamSynchronize(vh.stream);
  if (e == cudaSuccess) e = upload_restriction(vh.Q_xi, vl.Q_xi, &R, st);
  if (e == cudaSuccess) e = cudaMalloc((void**)&ns, sizeof(float) * vl.Z);
  if (e == cudaSuccess) e = cudaMalloc((void**)&ref, sizeof(float) * (size_t)vl.V * vl.ldz);
  const int TB = 128, G = (vl.Z + TB - 1) / TB;
  if (e == cudaSuccess) e = launch_restrict(vh, vl, R, (float*)vl.F0, st);
  if (e == cudaSuccess) {
    features_kernel<<<G, TB, 0, st>>>((const float*)vl.F0, vl.Z, vl.ldz, vl.V,
                                      (float)std::log10(tau), X, ns);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess && (rc = rslb_step(lo, 1)) != RSLB_OK) e = cudaErrorUnknown;
  if (e == cudaSuccess && (rc = rslb_step(hi, 1)) != RSLB_OK) e = cudaErrorUnknown;
  if (e == cudaSuccess) e = cudaStreamSynchronize(vh.stream);
  if (e == cudaSuccess) e = launch_restrict(vh, vl, R, ref, st);
  if (e == cudaSuccess) {
    target_kernel<<<G, TB, 0, st>>>(ref, (const float*)vl.F0, ns, vl.Z, vl.ldz, vl.V, cc, T);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (R) cudaFree(R);
  if (ns) cudaFree(ns);
  if (ref) cudaFree(ref);
  if (rc) return rc;
  return e == cudaSuccess ? RSLB_OK : cuda_error(e, "rslb_closure_sample");
}

extern "C" int rslb_closure_step(rslb_handle* lo, rslb_mlp* m, double tau, int nsteps) {
  clear_error();
  SodView vl;
  if (sod_view(lo, &vl) || !m || nsteps < 0 || !(tau > 0.0))
    return set_error(RSLB_ERR_ARG, "rslb_closure_step: bad arguments");
  if (vl.fp64) return set_error(RSLB_ERR_UNSUPPORTED, "rslb_closure_step: needs an RSLB_F32 handle");
  if (m->s.O != vl.V || m->s.D != 3 * vl.V + 1)
    return set_error(RSLB_ERR_ARG, "rslb_closure_step: network shape (%d -> %d) does not match "
                     "3V+1 -> V for V = %d", m->s.D, m->s.O, vl.V);
  ClosureConsts cc;
  int rc = closure_consts(vl.Q_xi, vl.Q_L, &cc);
  if (rc) return set_error(rc, "rslb_closure_step: low-order set too large");
  const MlpShape& s = m->s;
  const float lt = (float)std::log10(tau);
  // the correction reads its neighbours, so it writes the other buffer, which
  // then holds the state: the two change roles every step
  float* F[2] = {(float*)vl.F0, (float*)vl.F1};
  const cudaError_t e = swap_steps(
      nsteps, cudaSuccess,
      [&](int cur) {
        const cudaError_t es = sod_step_in(lo, cur);
        if (es != cudaSuccess) return es;
        return dispatch_team(s, vl.Z, kApplyMany, [&](auto Hc, auto Pc) {
          constexpr int H = decltype(Hc)::value, PARTS = decltype(Pc)::value;
          using T = Team<PARTS>;
          const int grid =
              std::min((vl.Z + T::kRows - 1) / T::kRows, m->apply_places[PARTS == 1]);
          closure_apply_kernel<H, PARTS><<<grid, T::kThreads, infer_smem(s, T::kRows), vl.stream>>>(
              s, m->theta, m->wb, m->norm, F[cur], F[cur ^ 1], vl.Z, vl.ldz, lt, cc);
          return cudaGetLastError();
        });
      },
      [&]() {
        return cudaMemcpyAsync(vl.F0, vl.F1, sizeof(float) * (size_t)vl.V * vl.ldz,
                               cudaMemcpyDeviceToDevice, vl.stream);
      });
  if (e != cudaSuccess) return cuda_error(e, "rslb_closure_step");
  return RSLB_OK;
}
