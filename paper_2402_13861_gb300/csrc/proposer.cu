// Cell-subdivision proposer.  The paper keeps or culls cells by range analysis alone (Algorithm 1);
// this addition scores (cell, iso-value) pairs with a small MLP trained on labels the method itself
// produces (dense evaluation plus the marching-cubes crossing test of Sec. IV-D), so that confident
// pairs skip the affine bound, and range analysis stays the fallback and decides the rest.
//
// Model: 8 -> 64 -> 64 -> 64 -> 1, ReLU hidden layers, sigmoid output, binary cross-entropy.
// Numerics: BF16 weights, BF16 inputs and activations (round to nearest even after every layer),
// FP32 accumulation; FP32 master weights, gradients and Adam moments.  The model costs 17.5 kFLOP
// per pair against 203 MFLOP for one affine bound of the 256-wide 5-layer INR, so it runs on CUDA
// cores, weights staged once per block as FP32 (exact).  k_prop_forward and k_prop_grad work on tiles of
// samples, activations [neuron][sample] in shared memory, with register tiles of samples x neurons (every
// output one multiply-add chain over the inputs); k_prop_gate, whose pairs come from bit masks, runs one thread
// per cell with its activation rows in padded shared memory (row stride 65 floats, so the 32 rows a warp
// touches fall in 32 different banks).
//
// Kernels: k_prop_forward (logits of given feature rows), k_prop_grad (forward + backward of the
// mean BCE, per-block gradient sums in registers, one atomic add per parameter per block),
// k_prop_adam (one Adam step over the flat parameter vector, refreshes the BF16 copy),
// k_prop_gate (extraction: builds the features of every (cell, iso) pair in the cell's mask, drops
// confident negatives, keeps confident positives, flags the rest for bounding), k_prop_merge
// (applies the bound of the flagged cells).
#include "internal.cuh"
#include "sgemm.cuh"

#include <algorithm>
#include <cmath>
#include <vector>

struct isx_proposer_s {
  int device = 0;
  float* params = nullptr;          // FP32 master weights, packed (isx.h)
  __nv_bfloat16* pb = nullptr;      // BF16 copy used by every forward and backward
  float* m = nullptr;               // Adam first moment
  float* v = nullptr;               // Adam second moment
  float* grad = nullptr;            // gradient accumulator of one step
  float* loss = nullptr;            // device scratch for the loss of one step
  float mu[8], inv_sd[8];
  int64_t t = 0;                    // Adam step count
};

namespace isx {
namespace {

constexpr int kF = 8, kH = 64;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + kH * kF, OFF_W2 = OFF_B1 + kH, OFF_B2 = OFF_W2 + kH * kH,
              OFF_W3 = OFF_B2 + kH, OFF_B3 = OFF_W3 + kH * kH, OFF_W4 = OFF_B3 + kH, OFF_B4 = OFF_W4 + kH,
              kNParam = OFF_B4 + 1;
static_assert(kNParam == ISX_PROPOSER_NPARAM, "packed parameter layout");
static_assert(OFF_W2 % 4 == 0 && OFF_W3 % 4 == 0 && OFF_W4 % 4 == 0, "float4 weight rows");
constexpr int kNParamPad = (kNParam + 3) & ~3;
constexpr int kTB = 128;          // threads per block (k_prop_gate: cells per tile)
constexpr int kRow = kH + 1;      // padded activation row

struct Norm {
  float mu[kF], inv_sd[kF];
};

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

__device__ __forceinline__ void stage_weights(float* sw, const __nv_bfloat16* pb) {
  for (int k = threadIdx.x; k < kNParamPad; k += blockDim.x) sw[k] = k < kNParam ? __bfloat162float(pb[k]) : 0.f;
}

// out_row[o] = bf16(relu(b[o] + sum_i W[o][i] in[i])), o < 64; W row-major [64][IN] in shared memory.
template <int IN>
__device__ __forceinline__ void dense_relu(const float* W, const float* b, const float (&in)[IN], float* out_row) {
#pragma unroll 1
  for (int o = 0; o < kH; ++o) {
    const float4* w4 = reinterpret_cast<const float4*>(W + o * IN);
    float acc = b[o];
#pragma unroll
    for (int i = 0; i < IN / 4; ++i) {
      const float4 w = w4[i];
      acc = fmaf(w.x, in[4 * i], acc);
      acc = fmaf(w.y, in[4 * i + 1], acc);
      acc = fmaf(w.z, in[4 * i + 2], acc);
      acc = fmaf(w.w, in[4 * i + 3], acc);
    }
    out_row[o] = bf16r(fmaxf(acc, 0.f));
  }
}

template <int N>
__device__ __forceinline__ void load_row(const float* row, float (&v)[N]) {
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] = row[i];
}

__device__ __forceinline__ void normalise(const Norm& nm, float (&x)[kF]) {
#pragma unroll
  for (int d = 0; d < kF; ++d) x[d] = bf16r((x[d] - nm.mu[d]) * nm.inv_sd[d]);
}

// Logit of one normalised sample; r1, r2, r3 receive the three hidden activation rows (r3 may
// alias r1 when the caller does not keep them).
__device__ __forceinline__ float forward_sample(const float* sw, const float (&x)[kF], float* r1, float* r2,
                                                float* r3) {
  dense_relu<kF>(sw + OFF_W1, sw + OFF_B1, x, r1);
  float h[kH];
  load_row(r1, h);
  dense_relu<kH>(sw + OFF_W2, sw + OFF_B2, h, r2);
  load_row(r2, h);
  dense_relu<kH>(sw + OFF_W3, sw + OFF_B3, h, r3);
  load_row(r3, h);
  float z = sw[OFF_B4];
#pragma unroll
  for (int i = 0; i < kH; ++i) z = fmaf(sw[OFF_W4 + i], h[i], z);
  return z;
}

// ---- tiles of samples -------------------------------------------------------------------------------
// Shared memory of a block: the transposed hidden weights Wt[i][o] (pitch kWP, so that staging them costs
// four-way bank conflicts, not 32-way), the biases and W4, and activations [neuron][sample].
constexpr int kWP = kH + 4;
constexpr int kWtFloats = (kF + 2 * kH) * kWP + 4 * kH + 4;   // W1t, W2t, W3t; b1, b2, b3, W4, b4

static_assert(OFF_B1 % 8 == 0 && OFF_W2 % 8 == 0 && OFF_B2 % 8 == 0 && OFF_W3 % 8 == 0 && OFF_B3 % 8 == 0 &&
                  OFF_B4 % 8 == 0 && OFF_B4 == kNParam - 1, "16-byte groups of parameters");
// Also W2 and W3 as they are ([o][i], one after the other) into w23 when given.  16-byte loads, four in flight.
__device__ __forceinline__ void stage_transposed(float* wt, float* w23, const __nv_bfloat16* pb) {
  float* vec = wt + (kF + 2 * kH) * kWP;
  const uint4* src = reinterpret_cast<const uint4*>(pb);
  for (int g0 = threadIdx.x; g0 < OFF_B4 / 8; g0 += 4 * blockDim.x) {
    uint4 u[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (g0 + q * (int)blockDim.x < OFF_B4 / 8) u[q] = src[g0 + q * blockDim.x];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = 8 * (g0 + q * (int)blockDim.x);
      if (k >= OFF_B4) break;
      float v[8];
      const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u[q]);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 f = __bfloat1622float2(h[e]);
        v[2 * e] = f.x;
        v[2 * e + 1] = f.y;
      }
      // the group's eight values: inputs i .. i + 7 of output o, or eight entries of a vector
      float* d = nullptr;
      int step = kWP;
      if (k < OFF_B1) {
        d = wt + k / kF;
      } else if (k >= OFF_W2 && k < OFF_B2) {
        d = wt + (kF + (k - OFF_W2) % kH) * kWP + (k - OFF_W2) / kH;
      } else if (k >= OFF_W3 && k < OFF_B3) {
        d = wt + (kF + kH + (k - OFF_W3) % kH) * kWP + (k - OFF_W3) / kH;
      } else {
        d = vec + (k < OFF_W2 ? k - OFF_B1 : (k < OFF_W3 ? kH + k - OFF_B2 : 2 * kH + k - OFF_B3));
        step = 1;
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) d[e * step] = v[e];
      if (w23 && step > 1 && k >= OFF_W2) {
        float* c = w23 + (k < OFF_B2 ? k - OFF_W2 : kH * kH + k - OFF_W3);
#pragma unroll
        for (int e = 0; e < 8; e += 4) *reinterpret_cast<float4*>(c + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
      }
    }
  }
  if (threadIdx.x == 0) vec[4 * kH] = __bfloat162float(pb[OFF_B4]);
}

// acc[s][j]: output pair j of this thread's outputs for sample s; samples sp(s), outputs op(j), op(j) + 1.
// NS samples in groups of 4 at s0, s0 + SS, ...; NO outputs in groups of 4 at o0, o0 + OS, ...
template <int NS, int NO>
struct PropTile {
  uint64_t acc[NS][NO / 2];
  __device__ __forceinline__ void bias(const float* b, int o0, int os) {
#pragma unroll
    for (int j = 0; j < NO / 2; ++j) {
      const int o = o0 + (j >> 1) * os + 2 * (j & 1);
      const uint64_t v = b ? sgemm::pack2(b[o], b[o + 1]) : 0ull;
#pragma unroll
      for (int s = 0; s < NS; ++s) acc[s][j] = v;
    }
  }
  // acc += sum_i X[i][sample] W[i][output], i ascending
  template <int IN>
  __device__ __forceinline__ void contract(const float* W, int wp, const float* X, int xp, int s0, int ss, int o0, int os) {
#pragma unroll 4
    for (int i = 0; i < IN; ++i) {
      uint64_t x[NS];
#pragma unroll
      for (int g = 0; g < NS / 4; ++g) {
        const float4 v = *reinterpret_cast<const float4*>(X + i * xp + s0 + g * ss);
        x[4 * g] = sgemm::pack2(v.x, v.x);
        x[4 * g + 1] = sgemm::pack2(v.y, v.y);
        x[4 * g + 2] = sgemm::pack2(v.z, v.z);
        x[4 * g + 3] = sgemm::pack2(v.w, v.w);
      }
#pragma unroll
      for (int g = 0; g < NO / 4; ++g) {
        const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(W + i * wp + o0 + g * os);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
          acc[s][2 * g] = sgemm::fma2(x[s], w.x, acc[s][2 * g]);
          acc[s][2 * g + 1] = sgemm::fma2(x[s], w.y, acc[s][2 * g + 1]);
        }
      }
    }
  }
  __device__ __forceinline__ float get(int s, int o) const {
    const float2 v = sgemm::unpack2(acc[s][o >> 1]);
    return (o & 1) ? v.y : v.x;
  }
  // Y[output][sample] = f(value, output, sample index s)
  template <class F>
  __device__ __forceinline__ void store(float* Y, int yp, int s0, int ss, int o0, int os, F f) const {
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      float* d = Y + (o0 + (o >> 2) * os + (o & 3)) * yp;
#pragma unroll
      for (int g = 0; g < NS / 4; ++g)
        *reinterpret_cast<float4*>(d + s0 + g * ss) =
            make_float4(f(get(4 * g, o), d, s0 + g * ss), f(get(4 * g + 1, o), d, s0 + g * ss + 1),
                        f(get(4 * g + 2, o), d, s0 + g * ss + 2), f(get(4 * g + 3, o), d, s0 + g * ss + 3));
    }
  }
};
__device__ __forceinline__ float act_bf16(float v, const float*, int) { return bf16r(fmaxf(v, 0.f)); }

// Logits: 128-sample tiles, an 8 x 8 register tile per thread, activations written back in place.  Bound by the
// shared-memory return bandwidth (16 values read per 64 multiply-adds): 2 M samples 0.74 ms, 48 TFLOP/s (1.48 ms with one
// thread per sample).
constexpr int kFwdS = 128, kFwdP = kFwdS + 4;
constexpr size_t kFwdSmem = (size_t)(kWtFloats + kH * kFwdP) * sizeof(float);
__global__ void __launch_bounds__(kTB) k_prop_forward(const __nv_bfloat16* pb, Norm nm, const float* feat, int64_t n,
                                                      float* logit) {
  extern __shared__ __align__(16) float sm[];
  float* wt = sm;
  const float* vec = wt + (kF + 2 * kH) * kWP;
  float* A = sm + kWtFloats;                             // [kH][kFwdP]
  stage_transposed(wt, nullptr, pb);
  const int t = threadIdx.x, s0 = 4 * (t & 15), o0 = 4 * (t >> 4);
  for (int64_t base = (int64_t)blockIdx.x * kFwdS; base < n; base += (int64_t)gridDim.x * kFwdS) {
    float x[kF];
#pragma unroll
    for (int d = 0; d < kF; ++d) x[d] = base + t < n ? feat[(base + t) * kF + d] : nm.mu[d];
    normalise(nm, x);
    __syncthreads();                                     // weights staged; the tile before is read
#pragma unroll
    for (int d = 0; d < kF; ++d) A[d * kFwdP + t] = x[d];
    __syncthreads();
    PropTile<8, 8> tile;
    tile.bias(vec, o0, 32);
    tile.contract<kF>(wt, kWP, A, kFwdP, s0, 64, o0, 32);
    __syncthreads();
    tile.store(A, kFwdP, s0, 64, o0, 32, act_bf16);
    __syncthreads();
#pragma unroll 1
    for (int l = 1; l < 3; ++l) {
      tile.bias(vec + l * kH, o0, 32);
      tile.contract<kH>(wt + (kF + (l - 1) * kH) * kWP, kWP, A, kFwdP, s0, 64, o0, 32);
      __syncthreads();
      tile.store(A, kFwdP, s0, 64, o0, 32, act_bf16);
      __syncthreads();
    }
    float z = vec[4 * kH];
#pragma unroll 16
    for (int i = 0; i < kH; ++i) z = fmaf(vec[3 * kH + i], A[i * kFwdP + t], z);
    if (base + t < n) logit[base + t] = z;
  }
}

// Forward and backward of the mean BCE over n samples: grad += dL/dtheta, loss += L.  Tiles of 64 samples, 256
// threads with 4 x 4 register tiles: a training batch of 8192 gives 128 blocks.  Parameter gradients stay in
// registers over a block's tiles.  8192 samples: 30 us a call, the two clears included (one thread per sample
// in 64 blocks of 128 threads: 96 us); 2 M samples 3.27 ms (8.4 ms).
constexpr int kGS = 64, kGP = kGS + 4, kGT = 256;
constexpr size_t kGradSmemFloats = kWtFloats + 2 * kH * kH + kF * kGP + 5 * kH * kGP + kGS + 32;

// dW[o][i] += sum_s dZ[o][s] A[i][s] for o = og + 16 r, i = ig + 16 c, and db[o] (threads with ig = 0).  The tile's
// samples are summed by themselves first: one sum over all of a block's samples would take as many roundings as it has
// samples (2^20 equal ones: up to 1.0e-4 of an entry, instead of 4e-6).
__device__ __forceinline__ void grad_layer(const float* dZ, const float* A, int og, int ig, float (&dw)[4][4], float (&db)[4]) {
  float tw[4][4] = {}, tb[4] = {};
#pragma unroll 4
  for (int s = 0; s < kGS; s += 4) {
    float4 z[4], a[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      z[r] = *reinterpret_cast<const float4*>(dZ + (og + 16 * r) * kGP + s);
      a[r] = *reinterpret_cast<const float4*>(A + (ig + 16 * r) * kGP + s);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
#pragma unroll
      for (int c = 0; c < 4; ++c)
        tw[r][c] = fmaf(z[r].w, a[c].w, fmaf(z[r].z, a[c].z, fmaf(z[r].y, a[c].y, fmaf(z[r].x, a[c].x, tw[r][c]))));
      if (ig == 0) tb[r] = (((tb[r] + z[r].x) + z[r].y) + z[r].z) + z[r].w;
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
#pragma unroll
    for (int c = 0; c < 4; ++c) dw[r][c] += tw[r][c];
    db[r] += tb[r];
  }
}

__global__ void __launch_bounds__(kGT) k_prop_grad(const __nv_bfloat16* pb, Norm nm, const float* feat,
                                                   const float* label, int64_t n, float inv_n, float* grad,
                                                   float* loss) {
  extern __shared__ __align__(16) float sm[];
  float* wt = sm;
  const float* vec = wt + (kF + 2 * kH) * kWP;
  float* W2 = sm + kWtFloats;                            // [o][i]
  float* W3 = W2 + kH * kH;
  float* A0 = W3 + kH * kH;
  float* A1 = A0 + kF * kGP;
  float* A2 = A1 + kH * kGP;
  float* A3 = A2 + kH * kGP;
  float* Za = A3 + kH * kGP;
  float* Zb = Za + kH * kGP;
  float* dz4 = Zb + kH * kGP;
  float* red = dz4 + kGS;
  stage_transposed(wt, W2, pb);
  const int t = threadIdx.x, s0 = 4 * (t & 15), o0 = 4 * (t >> 4), og = t >> 4, ig = t & 15;
  float dw3[4][4] = {}, dw2[4][4] = {}, db3[4] = {}, db2[4] = {}, dw1[2] = {}, db1 = 0.f, dw4 = 0.f, db4 = 0.f, lsum = 0.f;
  for (int64_t base = (int64_t)blockIdx.x * kGS; base < n; base += (int64_t)gridDim.x * kGS) {
    // ---- forward ----
    __syncthreads();                                     // weights staged; the tile before is read
    if (t < kGS) {
      const bool valid = base + t < n;
      float x[kF];
#pragma unroll
      for (int d = 0; d < kF; ++d) x[d] = valid ? feat[(base + t) * kF + d] : nm.mu[d];
      normalise(nm, x);
#pragma unroll
      for (int d = 0; d < kF; ++d) A0[d * kGP + t] = x[d];
    }
    __syncthreads();
    PropTile<4, 4> tile;
    tile.bias(vec, o0, 0);
    tile.contract<kF>(wt, kWP, A0, kGP, s0, 0, o0, 0);
    tile.store(A1, kGP, s0, 0, o0, 0, act_bf16);
    __syncthreads();
    tile.bias(vec + kH, o0, 0);
    tile.contract<kH>(wt + kF * kWP, kWP, A1, kGP, s0, 0, o0, 0);
    tile.store(A2, kGP, s0, 0, o0, 0, act_bf16);
    __syncthreads();
    tile.bias(vec + 2 * kH, o0, 0);
    tile.contract<kH>(wt + (kF + kH) * kWP, kWP, A2, kGP, s0, 0, o0, 0);
    tile.store(A3, kGP, s0, 0, o0, 0, act_bf16);
    __syncthreads();
    if (t < kGS) {
      float z = vec[4 * kH];
#pragma unroll 16
      for (int i = 0; i < kH; ++i) z = fmaf(vec[3 * kH + i], A3[i * kGP + t], z);
      const bool valid = base + t < n;
      const float y = valid ? label[base + t] : 0.f;
      const float p = 1.f / (1.f + expf(-z));
      if (valid) lsum += fmaxf(z, 0.f) - z * y + log1pf(expf(-fabsf(z)));
      dz4[t] = valid ? (p - y) * inv_n : 0.f;
    }
    __syncthreads();
    // ---- dZ3 = (dz W4) masked by A3 > 0; dW4, db4 (threads < 64: one input each) ----
    for (int k = t; k < kH * kGS; k += kGT) {
      const int i = k / kGS, q = k % kGS;
      Za[i * kGP + q] = A3[i * kGP + q] > 0.f ? dz4[q] * vec[3 * kH + i] : 0.f;
    }
    if (t < kH) {
      float tw = 0.f, tb = 0.f;
#pragma unroll 8
      for (int q = 0; q < kGS; ++q) {
        tw = fmaf(dz4[q], A3[t * kGP + q], tw);
        tb += dz4[q];
      }
      dw4 += tw;
      db4 += tb;
    }
    __syncthreads();
    // ---- dW3, db3; dZ2 = (W3^T dZ3) masked by A2 > 0 ----
    grad_layer(Za, A2, og, ig, dw3, db3);
    tile.bias(nullptr, o0, 0);
    tile.contract<kH>(W3, kH, Za, kGP, s0, 0, o0, 0);
    tile.store(Zb, kGP, s0, 0, o0, 0, [&](float v, const float* d, int q) { return (A2 + (d - Zb))[q] > 0.f ? v : 0.f; });
    __syncthreads();
    // ---- dW2, db2; dZ1 = (W2^T dZ2) masked by A1 > 0 ----
    grad_layer(Zb, A1, og, ig, dw2, db2);
    tile.bias(nullptr, o0, 0);
    tile.contract<kH>(W2, kH, Zb, kGP, s0, 0, o0, 0);
    tile.store(Za, kGP, s0, 0, o0, 0, [&](float v, const float* d, int q) { return (A1 + (d - Za))[q] > 0.f ? v : 0.f; });
    __syncthreads();
    // ---- dW1, db1: output t / 4, inputs 2 (t % 4), + 1 ----
    {
      const float* z = Za + (t >> 2) * kGP;
      const float* a = A0 + 2 * (t & 3) * kGP;
      float tw[2] = {}, tb = 0.f;
#pragma unroll 8
      for (int q = 0; q < kGS; ++q) {
        tw[0] = fmaf(z[q], a[q], tw[0]);
        tw[1] = fmaf(z[q], a[kGP + q], tw[1]);
        tb += z[q];
      }
      dw1[0] += tw[0];
      dw1[1] += tw[1];
      db1 += tb;
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int o = og + 16 * r;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      atomicAdd(&grad[OFF_W3 + o * kH + ig + 16 * c], dw3[r][c]);
      atomicAdd(&grad[OFF_W2 + o * kH + ig + 16 * c], dw2[r][c]);
    }
    if (ig == 0) {
      atomicAdd(&grad[OFF_B3 + o], db3[r]);
      atomicAdd(&grad[OFF_B2 + o], db2[r]);
    }
  }
  atomicAdd(&grad[OFF_W1 + (t >> 2) * kF + 2 * (t & 3)], dw1[0]);
  atomicAdd(&grad[OFF_W1 + (t >> 2) * kF + 2 * (t & 3) + 1], dw1[1]);
  if ((t & 3) == 0) atomicAdd(&grad[OFF_B1 + (t >> 2)], db1);
  if (t < kH) atomicAdd(&grad[OFF_W4 + t], dw4);
  if (t == 0) atomicAdd(&grad[OFF_B4], db4);
  // ---- loss: block sum, one atomic ----
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
  if ((t & 31) == 0) red[t >> 5] = lsum;
  __syncthreads();
  if (t == 0) {
    float sacc = 0.f;
    for (int w = 0; w < kGT / 32; ++w) sacc += red[w];
    atomicAdd(loss, sacc * inv_n);
  }
}

__global__ void k_prop_adam(float* params, __nv_bfloat16* pb, float* m, float* v, float* grad, float lr, float b1,
                            float b2, float eps, float bc1, float bc2) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= kNParam) return;
  const float gk = grad[k];
  const float mk = b1 * m[k] + (1.f - b1) * gk;
  const float vk = b2 * v[k] + (1.f - b2) * gk * gk;
  m[k] = mk;
  v[k] = vk;
  const float p = params[k] - lr * (mk / bc1) / (sqrtf(vk / bc2) + eps);
  params[k] = p;
  pb[k] = __float2bfloat16_rn(p);
  grad[k] = 0.f;
}

__global__ void k_to_bf16(const float* src, __nv_bfloat16* dst, int n) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) dst[k] = __float2bfloat16_rn(src[k]);
}

// Extraction gate: for every cell (packed code at `level`) and every iso q in its mask, the logit of
// the pair's features against the thresholds.  keep[i] = bits with logit >= z_hi (kept without a
// bound); need[i] = 1 if some bit lies strictly between the thresholds (the cell is bounded).
__global__ void __launch_bounds__(kTB) k_prop_gate(const __nv_bfloat16* pb, Norm nm, const uint32_t* codes,
                                                   const uint32_t* masks, const float* anc_c, const float* anc_s,
                                                   const uint8_t* anc_gap, int64_t n, int level, IsoSet iso,
                                                   float z_lo, float z_hi, uint32_t* keep, uint8_t* need) {
  extern __shared__ float sm[];
  float* sw = sm;
  float* rows = sm + kNParamPad;
  stage_weights(sw, pb);
  __syncthreads();
  float* rx = rows + threadIdx.x * kRow;
  float* ry = rows + (kTB + threadIdx.x) * kRow;
  const float h = ldexpf(1.0f, -level);
  for (int64_t i = (int64_t)blockIdx.x * kTB + threadIdx.x; i < n; i += (int64_t)gridDim.x * kTB) {
    const uint32_t code = codes[i];
    uint32_t m = masks[i];
    const float cx = -1.0f + (2.0f * float(code & 1023u) + 1.0f) * h;
    const float cy = -1.0f + (2.0f * float((code >> 10) & 1023u) + 1.0f) * h;
    const float cz = -1.0f + (2.0f * float((code >> 20) & 1023u) + 1.0f) * h;
    const float ac = anc_c[i], as = anc_s[i], gap = (float)anc_gap[i];
    uint32_t kbits = 0;
    bool unsure = false;
    while (m) {
      const int q = __ffs(m) - 1;
      m &= m - 1;
      const float c = iso.c[q];
      float x[kF] = {cx, cy, cz, -(float)level, c, ac - c, as, gap};
      normalise(nm, x);
      const float z = forward_sample(sw, x, rx, ry, rx);
      if (z >= z_hi) kbits |= 1u << q;
      else if (z > z_lo) unsure = true;
      // NaN logits (never expected) fall through to "unsure": the cell is bounded
      else if (!(z <= z_lo)) unsure = true;
    }
    keep[i] = kbits;
    need[i] = unsure ? 1 : 0;
  }
}

}  // namespace

namespace {
// Range-analysis decision of the flagged cells (idx[j], j < nb): their mask becomes
// mask & (cull test of Algorithm 1 on their bound), and that bound becomes the ancestor bound of
// their children (gap 0).
__global__ void k_prop_merge(const uint32_t* idx, int64_t nb, const uint32_t* masks, const float* c_sub,
                             const float* s_sub, IsoSet iso, int mode, float k, int inflate, uint32_t* keep,
                             float* anc_c, float* anc_s, uint8_t* anc_gap) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nb) return;
  const uint32_t i = idx[j];
  const float c = c_sub[j], s = s_sub[j];
  float lo, hi;
  if (sound_readout(mode)) {
    lo = inflate ? __fsub_rd(c, s) : c - s;
    hi = inflate ? __fadd_ru(c, s) : c + s;
  } else {
    lo = c - k * s;
    hi = c + k * s;
  }
  uint32_t bits = 0;
  for (int q = 0; q < iso.n; ++q)
    if (lo <= iso.c[q] && iso.c[q] <= hi) bits |= 1u << q;
  if (!(lo <= hi)) bits = 0xffffffffu;
  keep[i] = masks[i] & bits;
  anc_c[i] = c;
  anc_s[i] = s;
  anc_gap[i] = 0;
}

__global__ void k_gather_codes(const uint32_t* codes, const uint32_t* idx, int64_t nb, uint32_t* out) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j < nb) out[j] = codes[idx[j]];
}

Norm norm_of(isx_proposer p) {
  Norm nm;
  for (int d = 0; d < kF; ++d) {
    nm.mu[d] = p->mu[d];
    nm.inv_sd[d] = p->inv_sd[d];
  }
  return nm;
}

int grid_for(int64_t n, int dev, int tile = kTB, int per_sm = 4) {
  int sms = 148;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t tiles = (n + tile - 1) / tile;
  return (int)std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)per_sm * sms));
}

size_t fwd_smem() { return (size_t)(kNParamPad + 2 * kTB * kRow) * sizeof(float); }

isx_status set_smem(const void* fn, size_t bytes) {
  ISX_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  return ISX_OK;
}

isx_status check_prop(isx_proposer p) {
  if (!p || !p->params) {
    set_error("null proposer handle");
    return ISX_ERR_ARG;
  }
  return ISX_OK;
}

}  // namespace

isx_status proposer_gate(isx_proposer p, const uint32_t* codes, const uint32_t* masks, const float* anc_c,
                         const float* anc_s, const uint8_t* anc_gap, int64_t n, int level, const IsoSet& iso,
                         float z_lo, float z_hi, uint32_t* keep, uint8_t* need, cudaStream_t st) {
  if (n == 0) return ISX_OK;
  ISX_TRY(set_smem((const void*)k_prop_gate, fwd_smem()));
  {
    prof::Scope _ps(K_PROP_GATE, st, 2.0 * 8768 * (double)n, 0);
    k_prop_gate<<<grid_for(n, p->device), kTB, fwd_smem(), st>>>(p->pb, norm_of(p), codes, masks, anc_c, anc_s,
                                                                  anc_gap, n, level, iso, z_lo, z_hi, keep, need);
  }
  ISX_LAUNCH_CHECK("k_prop_gate");
  return ISX_OK;
}

isx_status proposer_merge(const uint32_t* idx, int64_t nb, const uint32_t* masks, const float* c_sub,
                          const float* s_sub, const IsoSet& iso, isx_bound_mode mode, float k, int inflate,
                          uint32_t* keep, float* anc_c, float* anc_s, uint8_t* anc_gap, cudaStream_t st) {
  if (nb == 0) return ISX_OK;
  {
    prof::Scope _ps(K_PROP_MERGE, st, 0, 0);
    k_prop_merge<<<(unsigned)((nb + 255) / 256), 256, 0, st>>>(idx, nb, masks, c_sub, s_sub, iso, (int)mode, k,
                                                               inflate, keep, anc_c, anc_s, anc_gap);
  }
  ISX_LAUNCH_CHECK("k_prop_merge");
  return ISX_OK;
}

isx_status gather_codes(const uint32_t* codes, const uint32_t* idx, int64_t nb, uint32_t* out, cudaStream_t st) {
  if (nb == 0) return ISX_OK;
  {
    prof::Scope _ps(K_PROP_MERGE, st, 0, 0);
    k_gather_codes<<<(unsigned)((nb + 255) / 256), 256, 0, st>>>(codes, idx, nb, out);
  }
  ISX_LAUNCH_CHECK("k_gather_codes");
  return ISX_OK;
}

}  // namespace isx

using namespace isx;

extern "C" {

isx_status isx_proposer_create(const float* params, const float* feat_mean, const float* feat_std,
                               isx_proposer* out) {
  if (!params || !feat_mean || !feat_std || !out) {
    set_error("null proposer argument");
    return ISX_ERR_ARG;
  }
  *out = nullptr;
  for (int d = 0; d < kF; ++d)
    if (!(feat_std[d] > 0.f) || !std::isfinite(feat_mean[d])) {
      set_error("feature standard deviations must be positive and means finite");
      return ISX_ERR_ARG;
    }
  isx_proposer p = new isx_proposer_s();
  ISX_CUDA(cudaGetDevice(&p->device));
  for (int d = 0; d < kF; ++d) {
    p->mu[d] = feat_mean[d];
    p->inv_sd[d] = 1.0f / feat_std[d];
  }
  auto fail = [&](cudaError_t e, const char* what) {
    isx_proposer_destroy(p);
    return cuda_fail(e, what, __FILE__, __LINE__);
  };
  cudaError_t e;
  const size_t fb = kNParam * sizeof(float);
  if ((e = cudaMalloc(&p->params, fb)) != cudaSuccess) return fail(e, "proposer params");
  if ((e = cudaMalloc(&p->pb, kNParam * 2)) != cudaSuccess) return fail(e, "proposer bf16");
  if ((e = cudaMalloc(&p->m, fb)) != cudaSuccess || (e = cudaMalloc(&p->v, fb)) != cudaSuccess ||
      (e = cudaMalloc(&p->grad, fb)) != cudaSuccess || (e = cudaMalloc(&p->loss, 16)) != cudaSuccess)
    return fail(e, "proposer optimiser state");
  if ((e = cudaMemcpy(p->params, params, fb, cudaMemcpyHostToDevice)) != cudaSuccess ||
      (e = cudaMemset(p->m, 0, fb)) != cudaSuccess || (e = cudaMemset(p->v, 0, fb)) != cudaSuccess ||
      (e = cudaMemset(p->grad, 0, fb)) != cudaSuccess)
    return fail(e, "proposer upload");
  k_to_bf16<<<(kNParam + 255) / 256, 256>>>(p->params, p->pb, kNParam);
  if ((e = cudaGetLastError()) != cudaSuccess || (e = cudaDeviceSynchronize()) != cudaSuccess)
    return fail(e, "proposer bf16 copy");
  *out = p;
  return ISX_OK;
}

isx_status isx_proposer_destroy(isx_proposer p) {
  if (!p) return ISX_OK;
  int prev = -1;
  cudaGetDevice(&prev);
  cudaSetDevice(p->device);
  for (void* q : {(void*)p->params, (void*)p->pb, (void*)p->m, (void*)p->v, (void*)p->grad, (void*)p->loss})
    if (q) cudaFree(q);
  if (prev >= 0) cudaSetDevice(prev);
  delete p;
  return ISX_OK;
}

isx_status isx_proposer_get_params(isx_proposer p, float* out) {
  ISX_TRY(check_prop(p));
  if (!out) {
    set_error("null output");
    return ISX_ERR_ARG;
  }
  ISX_CUDA(cudaMemcpy(out, p->params, kNParam * sizeof(float), cudaMemcpyDeviceToHost));
  return ISX_OK;
}

isx_status isx_proposer_predict(isx_proposer p, const float* d_feat, int64_t n, float* d_logit, void* stream) {
  ISX_TRY(check_prop(p));
  if (n < 0 || (n > 0 && (!d_feat || !d_logit))) {
    set_error("bad size or null pointer");
    return ISX_ERR_ARG;
  }
  if (n == 0) return ISX_OK;
  cudaStream_t st = (cudaStream_t)stream;
  ISX_TRY(set_smem((const void*)k_prop_forward, kFwdSmem));
  {
    prof::Scope _ps(K_PROP_FWD, st, 2.0 * 8768 * (double)n, 0);
    k_prop_forward<<<grid_for(n, p->device, kFwdS, 3), kTB, kFwdSmem, st>>>(p->pb, norm_of(p), d_feat, n, d_logit);
  }
  ISX_LAUNCH_CHECK("k_prop_forward");
  return ISX_OK;
}

isx_status isx_proposer_grad(isx_proposer p, const float* d_feat, const float* d_label, int64_t n, float* d_grad,
                             float* d_loss, void* stream) {
  ISX_TRY(check_prop(p));
  if (n <= 0 || !d_feat || !d_label || !d_grad || !d_loss) {
    set_error("bad size or null pointer");
    return ISX_ERR_ARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  const size_t smem = kGradSmemFloats * sizeof(float);
  ISX_TRY(set_smem((const void*)k_prop_grad, smem));
  ISX_CUDA(cudaMemsetAsync(d_grad, 0, kNParam * sizeof(float), st));
  ISX_CUDA(cudaMemsetAsync(d_loss, 0, sizeof(float), st));
  {
    prof::Scope _ps(K_PROP_GRAD, st, 3.0 * 2.0 * 8768 * (double)n, 0);
    k_prop_grad<<<grid_for(n, p->device, kGS, 1), kGT, smem, st>>>(p->pb, norm_of(p), d_feat, d_label, n, 1.0f / (float)n,
                                                                   d_grad, d_loss);
  }
  ISX_LAUNCH_CHECK("k_prop_grad");
  return ISX_OK;
}

isx_status isx_proposer_train_step(isx_proposer p, const float* d_feat, const float* d_label, int64_t n, float lr,
                                   float* d_loss, void* stream) {
  ISX_TRY(check_prop(p));
  if (n <= 0 || !d_feat || !d_label || !(lr > 0.f)) {
    set_error("bad size, learning rate or null pointer");
    return ISX_ERR_ARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  ISX_TRY(isx_proposer_grad(p, d_feat, d_label, n, p->grad, d_loss ? d_loss : p->loss, stream));
  p->t += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float bc1 = 1.f - (float)std::pow((double)b1, (double)p->t);
  const float bc2 = 1.f - (float)std::pow((double)b2, (double)p->t);
  {
    prof::Scope _ps(K_PROP_ADAM, st, 0, 0);
    k_prop_adam<<<(kNParam + 255) / 256, 256, 0, st>>>(p->params, p->pb, p->m, p->v, p->grad, lr, b1, b2, 1e-8f,
                                                       bc1, bc2);
  }
  ISX_LAUNCH_CHECK("k_prop_adam");
  return ISX_OK;
}

}  // extern "C"
