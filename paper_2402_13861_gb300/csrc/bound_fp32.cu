// Float32 bound path: affine / probabilistic-affine forms propagated layer by layer through a ReLU
// MLP (Sec. III-B and IV-C), one kernel per step, cells processed in chunks.
//
// Per cell the form of the pre-activation z_j of hidden layer j is a centre c (w floats) and the rows X of
// its noise symbols in float32, the cells' rows one after another (offsets from a scan of the per-cell
// counts):
//   z_1:  c = W_0 x_c + b_0, X = diag(h) W_0^T                      (input box, Eq. 3 / Eq. 8)
//   ReLU: alpha, beta, gamma per neuron from (c, r) or (mu, sigma)  (Eq. 4 / Eq. 9, Table VII)
//   L_j:  c' = W_j (alpha c + beta) + b_j,
//         X' = [X diag(alpha) W_j^T ; gamma_n W_j[:, n] for every n with gamma_n != 0]   (Eq. 3 / Eq. 8)
//   out:  y_i = X diag(alpha) w_out (+ gamma_m w_out,m for the last ReLU's symbols),
//         r = sum |y_i| (Eq. 2) or sigma^2 = sum y_i^2 (Eq. 7), RA-UA: sigma^2 / 3 (Sec. IV-A).
// A symbol whose coefficient gamma_n is exactly 0 has an all-zero row in every later layer and is never
// created.  Bound by the FP32 FMA rate of the row GEMM: 20003 random cells of levels 5-9 of the fitted
// 3 -> 256 x 5 -> 1 network take 16.1 ms (43 TFLOP/s in the GEMM), where carrying all 1027 rows of every
// cell took 142.6 ms; with every symbol alive (ELU, 3 -> 128 x 4 -> 1, 5003 boxes) 2.3 ms against 4.0 ms.
// A cell's result depends neither on the chunking nor on the launch shapes.
//
// Rounding-error inflation (SOUND, inflate != 0).  The library carries, per neuron, a slack
// delta >= |true z - carried form| and widens the ReLU interval by it; the linearisation error,
// alpha * delta and the rounding of the new centre all go into the neuron's new symbol, so after
// every ReLU the carried form is exact again.  Float32 rounding of each step is bounded by
// standard error analysis: a K-term dot product errs by at most gamma_K sum |a_k b_k| with
// gamma_K = K u / (1 - K u), u = 2^-24; products alpha_k W_nk rounded once more add u.
#include "internal.cuh"

#include <string>
#include "linearise.cuh"
#include "cell_box.cuh"
#include "rows.cuh"
#include "sgemm.cuh"

#include <algorithm>
#include <cooperative_groups.h>
#include <cmath>

namespace isx {
namespace {

constexpr float kU = 5.9604645e-08f;        // 2^-24, float32 unit roundoff
constexpr float kSafe = 1.0000010f;         // (1 + 16 u): slack for evaluating error formulas, and for the output layer's
                                            // sums, which take at most 13 roundings of a term
constexpr float kInvSqrt3 = 0.57735026918962576f;

__host__ __device__ __forceinline__ float gamma_k(int k) { return (k * kU) / (1.0f - k * kU); }

// Linearisation of activation j for one (cell, neuron): pre-activation centre c, radius / sigma rad, slack dl.
__device__ __forceinline__ Lin linearise(int mode, int act, int inflate, float c, float rad, float dl) {
  return mode == ISX_BOUND_CLT ? act_clt(act, c, rad) : relu_sound(c, rad, inflate ? dl : 0.0f, inflate != 0);
}

// Threads per cell and cells per block of the per-(cell, neuron) kernels: blocks of up to 256 threads.
struct CellBlock {
  int tpc, cpb;
  explicit CellBlock(int w) : tpc(std::min(w, 256)), cpb(std::max(1, 256 / std::min(w, 256))) {}
  unsigned blocks(int nc) const { return (unsigned)((nc + cpb - 1) / cpb); }
  unsigned threads() const { return (unsigned)(tpc * cpb); }
};

// The roundings of every sum over symbols, spelled out: a cell's result must not depend on the kernel that formed it.
// One compensated step of a sum of x^2 (sq) or |x|, the slack, and the radius of the three input rows.
__device__ __forceinline__ void add_term(float& s, float& comp, float x, bool sq) {
  const float y = sq ? fmaf(x, x, -comp) : __fsub_rn(fabsf(x), comp), t = __fadd_rn(s, y);
  comp = __fsub_rn(__fsub_rn(t, s), y);
  s = t;
}
__device__ __forceinline__ float slack(float kappa, float g, int w, float e) {
  return __fmul_rn(fmaf(kappa, g, __fmul_rn(gamma_k(w + 2), e)), kSafe);
}
__device__ __forceinline__ float input_radius(int mode, float x0, float x1, float x2) {
  if (mode == ISX_BOUND_CLT) return sqrtf(fmaf(x2, x2, fmaf(x0, x0, __fmul_rn(x1, x1))));
  return __fadd_rn(__fadd_rn(fabsf(x0), fabsf(x1)), fabsf(x2));
}

// z_1 = W_0 x + b_0 over the box and activation 1: the 3 input rows with their row -> cell map, the
// post-activation centre, alpha, gamma (and, inflate, radius and slack), the cell's row counts (3 now,
// 3 + #(gamma != 0) after the next layer) and the offset of its rows (rs = 3, or 4 with padding, apart).
__global__ void __launch_bounds__(256) k_input_layer(CellSource src, int64_t first, int nc, int tpc, int rs,
                                                     const float* __restrict__ W0, const float* __restrict__ b0, int w,
                                                     int mode, int act, int inflate, float* C, float* X, int* rowcell,
                                                     float* RAD, float* ALPHA, float* GAMMA, int64_t* off, int* cnt,
                                                     int* cnt_next) {
  __shared__ int made[16];
  const int sub = threadIdx.x / tpc, t = threadIdx.x - sub * tpc;
  const int cell = blockIdx.x * (blockDim.x / tpc) + sub;
  if (threadIdx.x < 16) made[threadIdx.x] = 0;
  __syncthreads();
  if (cell < nc) {
    float xc[3], h[3];
    cell_box(src, first + cell, inflate, xc, h);
    if (mode == ISX_BOUND_CLT)
      for (int d = 0; d < 3; ++d) h[d] *= kInvSqrt3;   // uniform on [-h, h] has std h / sqrt 3
    float* Xc = X + (size_t)cell * rs * w;
    int m = 0;
    for (int n = t; n < w; n += tpc) {
      float w0 = W0[3 * n], w1 = W0[3 * n + 1], w2 = W0[3 * n + 2];
      float c = fmaf(w2, xc[2], fmaf(w1, xc[1], fmaf(w0, xc[0], b0[n])));
      float x0 = h[0] * w0, x1 = h[1] * w1, x2 = h[2] * w2;
      Xc[n] = x0;
      Xc[w + n] = x1;
      Xc[2 * w + n] = x2;
      const float rad = input_radius(mode, x0, x1, x2);
      float dl = 0.0f;
      if (inflate) {
        float e = fabsf(w0 * xc[0]) + fabsf(w1 * xc[1]) + fabsf(w2 * xc[2]) + fabsf(b0[n]);
        dl = (5.0f * kU * e + 3.0f * kU * rad) * kSafe;
      }
      const Lin L = linearise(mode, act, inflate, c, rad, dl);
      const size_t i = (size_t)cell * w + n;
      C[i] = L.center;
      ALPHA[i] = L.alpha;
      GAMMA[i] = L.gamma;
      if (inflate) RAD[i] = rad;
      m += L.gamma != 0.0f;
    }
    if (t < rs) rowcell[rs * cell + t] = t < 3 ? cell : -1;
    if (m) atomicAdd(&made[sub], m);
  }
  __syncthreads();
  if (cell < nc && t == 0) {
    off[cell] = rs * (int64_t)cell;
    cnt[cell] = 3;
    cnt_next[cell] = 3 + made[sub];
  }
}

// Centre of the next layer, Y = W a + b, and (inflate) the slack of the next pre-activation:
// kappa * sum_k |W_nk| (alpha_k r_k + gamma_k) + gamma_{K+1} (sum_k |W_nk a_k| + |b_n|).
// One thread per neuron, blockIdx.y a slice of them; bound by the latency of the weight loads, so up to 32 are in flight.
__global__ void __launch_bounds__(256) k_center_gemv(int w, const float* __restrict__ Wt, const float* __restrict__ bias,
                                                     const float* __restrict__ C, const float* ALPHA, const float* RAD,
                                                     const float* GAMMA, float* Y, float* DELTA, int inflate, float kappa) {
  extern __shared__ float sh[];
  float* a = sh;             // a-form centre
  float* ra = sh + w;        // a-form radius
  const size_t c0 = (size_t)blockIdx.x * w;
  for (int k = threadIdx.x; k < w; k += blockDim.x) {
    a[k] = C[c0 + k];
    ra[k] = inflate ? fmaf(ALPHA[c0 + k], RAD[c0 + k], GAMMA[c0 + k]) : 0.0f;
  }
  __syncthreads();
  for (int n = blockIdx.y * blockDim.x + threadIdx.x; n < w; n += gridDim.y * blockDim.x) {
    float acc = bias[n], e = fabsf(acc), g = 0.0f;
    float x[16], y[16];                            // w is a multiple of 16
    auto load = [&](float (&v)[16], int k0) {
      if (k0 < w)
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q] = Wt[(size_t)(k0 + q) * w + n];
    };
    auto add = [&](const float (&v)[16], int k0) {
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        acc = fmaf(v[q], a[k0 + q], acc);
        if (inflate) {
          e = fmaf(fabsf(v[q]), fabsf(a[k0 + q]), e);
          g = fmaf(fabsf(v[q]), ra[k0 + q], g);
        }
      }
    };
    load(x, 0);
    for (int k0 = 0; k0 < w; k0 += 32) {
      load(y, k0 + 16);
      add(x, k0);
      if (k0 + 16 >= w) break;
      load(x, k0 + 32);
      add(y, k0 + 16);
    }
    Y[c0 + n] = acc;
    if (inflate) DELTA[c0 + n] = slack(kappa, g, w, e);
  }
}

// Y[row] = X[row] diag(alpha_cell) W^T for R rows of all cells, or Y[row] = X[row] W^T + b (the centres):
// persistent CTAs over tiles of P rows, staged k-major in shared memory (sgemm.cuh).  Every output is one
// multiply-add chain over k whatever the launch shape, so all shapes give bit-identical results and the
// autotuner may pick any of them.  R comes from device memory (d_R) where the host does not know it.
//
// alpha scales the rows while they are staged (kRows) or, for the ELU, the weights (kWeights), which then are
// rounded once per cell and not once per row and cell: the ELU's second moments cancel at small sigma and turn
// a different rounding of the rows into up to 5e-3 of the spread.  A cell's rows start at multiples of four there
// (kPad), so that the four neighbouring rows of a thread share their scaled weights.
enum Scale { kCentres, kRows, kWeights };
constexpr int kPad = 4;
struct GemmArgs {
  const float* X;
  float* Y;
  const float* Wt;
  const float* alpha;                  // [cell][w] (but for the centres)
  const float* bias;                   // centres
  const int* rowcell;                  // cell of every row (-1: padding), first rows of the cells in X and in Y
  const int64_t* off_in;
  const int64_t* off_out;
  const int64_t* d_R;                  // null: R
  int64_t R;
};
template <int TN, Scale SC>
__global__ void __launch_bounds__(256, 2) k_gemm_fp32(GemmArgs g, sgemm::Shape sh, int w) {
  extern __shared__ __align__(16) float sm[];
  const int P = sh.P, KB = sh.KB, spl = w / KB;
  float* A = sm;                                   // [w][P]
  int64_t* dst = reinterpret_cast<int64_t*>(sm + (size_t)w * P + (size_t)sgemm::kStages * KB * w);   // [P] row in Y, -1: none
  int* rcell = reinterpret_cast<int*>(dst + P);                                                       // [P] cell
  const int64_t R = g.d_R ? *g.d_R : g.R;
  const int64_t ntiles = (R + P - 1) / P;
  if (blockIdx.x >= ntiles) return;
  const int64_t mine = (ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x;
  sgemm::Stream ws{sm + (size_t)w * P, w, KB, mine * spl};
  int sk = 0;                                      // K block of the stage to load next
  auto load_next = [&] {
    ws.load(g.Wt + (size_t)sk * KB * w);
    sk = sk + 1 == spl ? 0 : sk + 1;
  };
  for (int s = 0; s < sgemm::kStages - 1; ++s) load_next();
  const int t = threadIdx.x, T = blockDim.x;
  const int PG = P / sgemm::kTM, pg = t % PG, ng = t / PG;
  const bool own = ng < w / TN;
  int slot = 0;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t r0 = tile * P;
    for (int p = t; p < P; p += T) {
      int c = 0;
      int64_t d = -1;
      if (r0 + p < R) {
        c = SC == kCentres ? 0 : g.rowcell[r0 + p];
        d = SC == kCentres ? r0 + p : SC == kWeights && c < 0 ? -1 : g.off_out[c] + (r0 + p - g.off_in[c]);
      }
      dst[p] = d;
      rcell[p] = c;
    }
    // the next tile's rows are asked into L2 while this one is computed
    const int64_t nt = tile + gridDim.x;
    if (t == 0 && nt < ntiles)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(g.X + (size_t)nt * P * w),
                   "r"((uint32_t)(min((int64_t)P, R - nt * P) * w * 4))
                   : "memory");
    __syncthreads();
    constexpr int NF = 4;                          // 16-byte loads of a thread in flight
    const int nq = (w / 4) * P;
    for (int q0 = t; q0 < nq; q0 += NF * T) {
      float4 v[NF], al[NF];
#pragma unroll
      for (int i = 0; i < NF; ++i) {
        const int q = q0 + i * T, p = q % P, k = 4 * (q / P);
        v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (q < nq && r0 + p < R) {
          v[i] = *reinterpret_cast<const float4*>(g.X + (size_t)(r0 + p) * w + k);
          if (SC == kRows) al[i] = *reinterpret_cast<const float4*>(g.alpha + (size_t)rcell[p] * w + k);
        } else {
          al[i] = v[i];
        }
      }
#pragma unroll
      for (int i = 0; i < NF; ++i) {
        const int q = q0 + i * T, p = q % P, k = 4 * (q / P);
        if (q >= nq) break;
        if (SC == kRows) {
          v[i].x *= al[i].x; v[i].y *= al[i].y; v[i].z *= al[i].z; v[i].w *= al[i].w;
        }
        float* d = A + (size_t)k * P + p;
        d[0] = v[i].x; d[P] = v[i].y; d[2 * P] = v[i].z; d[3 * P] = v[i].w;
      }
    }
    sgemm::Tile<TN> acc;
    if (own)
#pragma unroll
      for (int c = 0; c < TN / 2; ++c) {
        const int n = sgemm::Tile<TN>::neuron(c, ng, w);
        const uint64_t z = SC != kCentres ? 0ull : sgemm::pack2(g.bias[n], g.bias[n + 1]);
#pragma unroll
        for (int i = 0; i < sgemm::kTM; ++i) acc.acc[i][c] = z;
      }
    const float *al0 = nullptr, *al1 = nullptr;    // the scales of the thread's two groups of four rows
    if (SC == kWeights && own) {
      al0 = g.alpha + (size_t)rcell[4 * pg] * w;
      al1 = g.alpha + (size_t)rcell[(P >> 1) + 4 * pg] * w;
    }
    for (int kb = 0; kb < spl; ++kb) {
      sgemm::cp_wait<sgemm::kStages - 2>();
      __syncthreads();                             // the stage has landed, the one before it is free, A is written
      load_next();
      if (own) {
        const float *a = A + (size_t)kb * KB * P, *wk = ws.Ws + (size_t)slot * KB * w;
        if (SC == kWeights)
          acc.stage_scaled(a, wk, P, w, KB, pg, ng, al0 + kb * KB, al1 + kb * KB);
        else
          acc.stage(a, wk, P, w, KB, pg, ng);
      }
      slot = slot == sgemm::kStages - 1 ? 0 : slot + 1;
    }
    if (own)
#pragma unroll
      for (int i = 0; i < sgemm::kTM; ++i) {
        const int64_t row = dst[sgemm::Tile<TN>::row(i, pg, P)];
        if (row >= 0)
#pragma unroll
          for (int c = 0; c < TN / 2; c += 2) {
            const float2 u = sgemm::unpack2(acc.acc[i][c]), v = sgemm::unpack2(acc.acc[i][c + 1]);
            *reinterpret_cast<float4*>(g.Y + (size_t)row * w + sgemm::Tile<TN>::neuron(c, ng, w)) =
                make_float4(u.x, u.y, v.x, v.y);
          }
      }
    __syncthreads();                               // every thread is done with A and dst
  }
}

// Tile shapes of the float32 GEMM the autotuner chooses from: TN neurons per thread, about `elems`
// staged row elements per CTA (P = elems / w rows) and up to `stage` weights per stage.
struct GemmShape {
  int tn, elems, stage;
  const char* name;
};
constexpr GemmShape kGemmShapes[] = {{8, 16384, 4096, "8x8, 256 threads"}, {8, 8192, 2048, "8x8, 128 threads"},
                                     {8, 4096, 2048, "8x8, 64 threads"}, {4, 8192, 4096, "8x4, 256 threads"},
                                     {4, 4096, 8192, "8x4, 128 threads"}};
constexpr int kGemmVariants = sizeof(kGemmShapes) / sizeof(kGemmShapes[0]);

template <Scale SC>
isx_status launch_gemm(int v, const GemmArgs& g, int w, int sms, cudaStream_t st) {
  const GemmShape& gs = kGemmShapes[v];
  const int KB = 32 * w <= gs.stage && w % 32 == 0 ? 32 : (16 * w <= gs.stage ? 16 : (8 * w <= gs.stage ? 8 : 4));
  const sgemm::Shape sh{gs.tn, std::max(8, gs.elems / w / 8 * 8), KB};
  const size_t smem = sh.smem(w) + (size_t)sh.P * (sizeof(int64_t) + sizeof(int));
  const int threads = (sh.threads(w) + 31) / 32 * 32;
  const auto kernel = sh.tn == 8 ? k_gemm_fp32<8, SC> : k_gemm_fp32<4, SC>;
  ISX_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
  int per_sm = 1;
  ISX_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem));
  const int64_t ntiles = (g.R + sh.P - 1) / sh.P;  // d_R: g.R is an upper bound
  kernel<<<(unsigned)std::min<int64_t>(ntiles, (int64_t)sms * std::max(1, per_sm)), threads, smem, st>>>(g, sh, w);
  ISX_LAUNCH_CHECK("k_gemm_fp32");
  return ISX_OK;
}

// Rows of the symbols created by the last activation, gamma_n W[:, n] for every neuron with gamma_n != 0,
// after the cell's carried rows, and the row -> cell map of all of its rows.  WPC gridDim.y warps per cell share
// the neurons in units of eight.  Bound by the writes with many cells, by each warp's chain of loads with few.
template <int WPC>
__global__ void __launch_bounds__(256) k_fresh_rows(int nc, int w, const float* __restrict__ GAMMA,
                                                    const float* __restrict__ Wt, const int* cnt_in, const int* cnt_out,
                                                    const int64_t* off_out, float* Xout, int* rowcell, int pad) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int u = blockIdx.y * WPC + warp % WPC, warps = WPC * gridDim.y;
  const int cell = blockIdx.x * (8 / WPC) + warp / WPC;
  if (cell >= nc) return;
  const int64_t o0 = off_out[cell];
  const int co = cnt_out[cell];
  for (int r = u * 32 + lane; r < ((co + pad) & ~pad); r += 32 * warps) rowcell[o0 + r] = r < co ? cell : -1;
  // lane i: the alive neurons of the 32-group i (w <= 512), how many rows come before them, and how many there are
  const float* ga = GAMMA + (size_t)cell * w;
  float gm[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) gm[i] = 32 * i + lane < w ? ga[32 * i + lane] : 0.0f;
  unsigned mask = 0;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const unsigned b = __ballot_sync(0xffffffffu, gm[i] != 0.0f);
    if (lane == i) mask = b;
  }
  int before = __popc(mask);
#pragma unroll
  for (int o = 1; o < 16; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, before, o);
    if (lane >= o) before += v;
  }
  before -= __popc(mask);
  float* Y = Xout + (size_t)(o0 + cnt_in[cell]) * w;
  for (int q = u; q < w / 8; q += warps) {
    const unsigned all = __shfl_sync(0xffffffffu, mask, q >> 2);
    int row = __shfl_sync(0xffffffffu, before, q >> 2) + __popc(all & ((1u << (8 * (q & 3))) - 1u));
    const float gq = ga[8 * q + (lane & 7)];
    for (unsigned b = (all >> (8 * (q & 3))) & 0xffu; b; b &= b - 1, ++row) {
      const int l = __ffs(b) - 1;
      const float g = __shfl_sync(0xffffffffu, gq, l);
      const float4* src = reinterpret_cast<const float4*>(Wt + (size_t)(8 * q + l) * w);
      float4* d = reinterpret_cast<float4*>(Y + (size_t)row * w);
      for (int n = lane; n < w / 4; n += 32) {
        const float4 x = src[n];
        d[n] = make_float4(g * x.x, g * x.y, g * x.z, g * x.w);
      }
    }
  }
}

struct ReduceArgs {
  const float* X;
  const int64_t* off;
  const int* cnt;
  int nc, w, mode, act, inflate;
  float* C;
  float* RAD;
  const float* DELTA;
  float* ALPHA;
  float* GAMMA;
};

// One neuron's reduction over its cell's S rows (compensated, in row order), r = sum |x| (sound) or sigma =
// sqrt(sum x^2), and activation j + 1: post-activation centre in place, alpha, gamma (and, inflate, the radius).
// 16 rows are summed while the loads of the next 16 are in flight.  Returns whether the symbol is alive.
__device__ __forceinline__ int reduce_neuron(const ReduceArgs& g, int cell, int n, int S) {
  const bool sq = g.mode == ISX_BOUND_CLT;
  const float* Xc = g.X + (size_t)g.off[cell] * g.w + n;
  float s = 0.0f, comp = 0.0f, x[16], y[16];
  int r = 0;
  if (S >= 16) {
#pragma unroll
    for (int q = 0; q < 16; ++q) x[q] = Xc[(size_t)q * g.w];
    for (; r + 32 <= S; r += 16) {
#pragma unroll
      for (int q = 0; q < 16; ++q) y[q] = Xc[(size_t)(r + 16 + q) * g.w];
#pragma unroll
      for (int q = 0; q < 16; ++q) add_term(s, comp, x[q], sq);
#pragma unroll
      for (int q = 0; q < 16; ++q) x[q] = y[q];
    }
    r += 16;
  }
  // the last S - r < 16 rows, loaded before the 16 ahead of them are summed
#pragma unroll
  for (int q = 0; q < 16; ++q) y[q] = r + q < S ? Xc[(size_t)(r + q) * g.w] : 0.0f;
  if (S >= 16)
#pragma unroll
    for (int q = 0; q < 16; ++q) add_term(s, comp, x[q], sq);
#pragma unroll
  for (int q = 0; q < 16; ++q)
    if (r + q < S) add_term(s, comp, y[q], sq);
  const float rad = sq ? sqrtf(s) : s;
  const size_t i = (size_t)cell * g.w + n;
  const Lin L = linearise(g.mode, g.act, g.inflate, g.C[i], rad, g.inflate ? g.DELTA[i] : 0.0f);
  g.C[i] = L.center;
  g.ALPHA[i] = L.alpha;
  g.GAMMA[i] = L.gamma;
  if (g.inflate) g.RAD[i] = rad;
  return L.gamma != 0.0f;
}

// The reduction of whole cells, tpc threads each, and the next layer's row count, cnt + #(gamma != 0).
__global__ void __launch_bounds__(256) k_reduce_act(ReduceArgs g, int tpc, int* cnt_next) {
  __shared__ int made[16];
  const int sub = threadIdx.x / tpc, t = threadIdx.x - sub * tpc;
  const int cell = blockIdx.x * (blockDim.x / tpc) + sub;
  if (threadIdx.x < 16) made[threadIdx.x] = 0;
  __syncthreads();
  int S = 0;
  if (cell < g.nc) {
    S = g.cnt[cell];
    int m = 0;
    for (int n = t; n < g.w; n += tpc) m += reduce_neuron(g, cell, n, S);
    if (m) atomicAdd(&made[sub], m);
  }
  __syncthreads();
  if (cnt_next && cell < g.nc && t == 0) cnt_next[cell] = S + made[sub];
}

// The same for few cells, each with a cluster of blocks of 64 neurons, which count into the first one's shared
// memory: a column's chain of loads bounds it, and one block per cell would leave most SMs idle.
__global__ void __launch_bounds__(64) k_reduce_few(ReduceArgs g, int* cnt_next) {
  __shared__ int made;
  const auto cluster = cooperative_groups::this_cluster();
  const unsigned slice = cluster.block_rank();
  const int cell = blockIdx.x / cluster.num_blocks(), n = slice * 64 + threadIdx.x;
  if (threadIdx.x == 0) made = 0;
  cluster.sync();
  const int S = g.cnt[cell];
  const int alive = __syncthreads_count(n < g.w && reduce_neuron(g, cell, n, S));
  if (threadIdx.x == 0) atomicAdd(cluster.map_shared_rank(&made, 0), alive);
  cluster.sync();
  if (cnt_next && slice == 0 && threadIdx.x == 0) cnt_next[cell] = S + made;
}

// Output layer w -> 1 and the read-off.  Row r's term goes to partial sum r % 8 (compensated, r ascending),
// held by WPC warps per cell: all eight by one warp or one per warp, four rows' 16-byte loads in flight.  With
// WPC = 32 and 64 (few cells) a cluster of four or eight blocks shares the rows (one SM alone reads about 60 GB/s of them) and
// their products pass to the eight sums through the first block's shared memory.  The cell's result does not
// depend on WPC.
constexpr int kOutRows = 1024;                     // rows between two of those hand-overs
template <int WPC>
__global__ void __launch_bounds__(256)
    k_output(const float* __restrict__ X, const int64_t* off, const int* cnt, int nc, int w, const float* C,
             const float* ALPHA, const float* GAMMA, const float* RAD, const float* __restrict__ wout, float bout,
             int mode, int inflate, float* center, float* spread, int64_t first) {
  extern __shared__ __align__(16) float s_aw[];    // [cells of the block][w]: alpha o w_out; WPC > 8: [kOutRows] products
  __shared__ float red[8];
  constexpr int BPC = WPC > 8 ? WPC / 8 : 1, CPB = WPC > 8 ? 1 : 8 / WPC;   // blocks per cell, cells per block
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = warp / WPC;
  const int u = (blockIdx.x % BPC) * 8 + warp % WPC;                     // the warp's place among the cell's
  const int cell = blockIdx.x / BPC * CPB + sub;
  for (int i = threadIdx.x; i < CPB * w; i += blockDim.x) {
    const int c = blockIdx.x / BPC * CPB + i / w;
    s_aw[i] = c < nc ? ALPHA[(size_t)c * w + i % w] * wout[i % w] : 0.0f;
  }
  __syncthreads();
  const bool sq = (mode != ISX_BOUND_SOUND);
  float rows = 0.0f;                               // the rows' sum over the eight partials
  if (cell < nc) {
    const float* aw = s_aw + sub * w;
    const float* Xc = X + (size_t)off[cell] * w;
    const int S = cnt[cell];
    constexpr int NS = WPC == 1 ? 8 : 1;           // partial sums of this warp
    float s[NS] = {}, comp[NS] = {};
    // the products of rows r0 + q step, q < 4 (the last row's in place of rows past the end)
    auto four = [&](int r0, int step, float (&y)[4]) {
#pragma unroll
      for (int q = 0; q < 4; ++q) y[q] = 0.0f;
      for (int n = 4 * lane; n < w; n += 128) {
        const float4 a = *reinterpret_cast<const float4*>(aw + n);
        float4 x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = *reinterpret_cast<const float4*>(Xc + (size_t)min(r0 + q * step, S - 1) * w + n);
#pragma unroll
        for (int q = 0; q < 4; ++q) y[q] = fmaf(x[q].w, a.w, fmaf(x[q].z, a.z, fmaf(x[q].y, a.y, fmaf(x[q].x, a.x, y[q]))));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < 4; ++q) y[q] += __shfl_xor_sync(0xffffffffu, y[q], o);
    };
    // rows r0 + q WPC into the partials h + q (WPC = 1) or into the warp's own
    auto add_four = [&](int r0, int h) {
      float y[4];
      four(r0, WPC, y);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (r0 + q * WPC < S) {
          const int k = WPC == 1 ? h + q : 0;
          add_term(s[k], comp[k], y[q], sq);
        }
    };
    if constexpr (WPC == 1) {
      for (int r0 = 0; r0 < S; r0 += 8) {
        add_four(r0, 0);
        if (r0 + 4 < S) add_four(r0 + 4, 4);
      }
    } else if constexpr (WPC == 8) {
      for (int r0 = u; r0 < S; r0 += 4 * WPC) add_four(r0, 0);
    } else {
      const auto cluster = cooperative_groups::this_cluster();
      float* prod = cluster.map_shared_rank(s_aw + w, 0);
      for (int base = 0; base < S; base += kOutRows) {
        const int end = min(S - base, kOutRows);
        cluster.sync();                            // the products before are summed (at first: every block runs)
        for (int r = 4 * u; r < end; r += 4 * WPC) {
          float y[4];
          four(base + r, 1, y);
          if (lane < 4 && r + lane < end) prod[r + lane] = lane == 0 ? y[0] : lane == 1 ? y[1] : lane == 2 ? y[2] : y[3];
        }
        cluster.sync();
        if (u == 0 && lane < 8)
          for (int r = lane; r < end; r += 8) add_term(s[0], comp[0], prod[r], sq);
      }
    }
    if (WPC == 1) {
#pragma unroll
      for (int q = 0; q < NS; ++q) rows += s[q];
    } else if (WPC == 8 ? lane == 0 : u == 0 && lane < 8) {
      red[WPC == 8 ? warp : lane] = s[0];
    }
  }
  if (WPC > 1) {
    __syncthreads();
    if (u == 0)
      for (int k = 0; k < 8; ++k) rows += red[k];
  }
  if (u > 0 || cell >= nc) return;
  // symbols of the last activation, y_m = gamma_m w_m, and the centre
  // sum |y| or y^2, w . c, and the two error sums (inflate): a lane's terms in groups of four, so that none of the sums
  // takes more than 13 roundings of a term (sixteen one after the other took 23 at w = 512)
  float v[4] = {0.f, 0.f, 0.f, 0.f};
  for (int m0 = 0; m0 < w; m0 += 128) {
    float g[4] = {0.f, 0.f, 0.f, 0.f};
    for (int m = m0 + lane; m < min(w, m0 + 128); m += 32) {
      const size_t i = (size_t)cell * w + m;
      const float y = GAMMA[i] * wout[m];
      g[0] = sq ? fmaf(y, y, g[0]) : g[0] + fabsf(y);
      g[1] = fmaf(wout[m], C[i], g[1]);
      if (inflate) {
        g[2] = fmaf(fabsf(wout[m]), fabsf(C[i]), g[2]);
        g[3] = fmaf(fabsf(wout[m]), fmaf(ALPHA[i], RAD[i], GAMMA[i]), g[3]);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] += g[q];
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
  if (lane == 0) {
    const float tot = rows + v[0], x0 = v[1] + bout;
    float sp;
    if (mode == ISX_BOUND_SOUND) {
      sp = tot;
      if (inflate) {
        float ge = gamma_k(w + 1) + kU;
        sp = __fadd_ru(__fmul_ru(sp, kSafe), (ge * v[3] + gamma_k(w + 2) * (v[2] + fabsf(bout))) * 1.01f);
      }
    } else if (mode == ISX_BOUND_CLT) {
      sp = sqrtf(tot);
    } else {
      sp = sqrtf(tot / 3.0f);
    }
    center[first + cell] = x0;
    spread[first + cell] = sp;
  }
}

// ---- small networks: the whole propagation of a cell in one block ----------------------------------------
// Widths up to 64: a cell's rows fit in shared memory, and what the path above spends is launches (seven per
// layer and call) and passes over memory, not multiply-adds.  Every sum is taken in the order of the kernels
// above, so the results are the same bit for bit.  Bound by latency (a cell's chain of layers): four warps per
// cell and several blocks per SM, or sixteen warps where there are several layers of rows to carry (64 x 6, every
// symbol alive: 229 -> 178 us for one cell).  3 -> 64 x 2 -> 1, levels 4-6, with the row path before it: 1 cell
// 54 -> 31 us, 608 cells 72 -> 37, 8192 cells 139 -> 120; FP32 extraction of that network to level 6, 895 -> 690.
constexpr int kSmallT = 512;                       // threads at most
struct SmallNet {
  const float* W0;
  const float* b0;
  const float* Wt[ISX_MAX_LAYERS];     // hidden layers 1 .. H - 1
  const float* b[ISX_MAX_LAYERS];
  const float* wout;
  float bout;
  int w, H, act;
};
__host__ __device__ __forceinline__ int small_rows(int w, int H) { return 3 + w * (H - 1); }
size_t small_smem(int w, int H) { return ((size_t)small_rows(w, H) + 7) * w * sizeof(float); }

__global__ void __launch_bounds__(kSmallT) k_bound_small(CellSource src, int64_t n, SmallNet net, int mode, int inflate,
                                                         float* center, float* spread) {
  extern __shared__ __align__(16) float sm[];
  __shared__ float part[8];
  const int w = net.w, H = net.H, t = threadIdx.x, T = blockDim.x, lane = t & 31, warp = t >> 5, warps = T >> 5;
  float* X = sm;                                   // [rows][w]
  float* a = X + (size_t)small_rows(w, H) * w;     // centre, alpha, gamma, radius, slack of the current layer
  float* al = a + w;
  float* ga = al + w;
  float* ra = ga + w;                              // inflate: radius of the post-activation form
  float* rad = ra + w;
  float* de = rad + w;
  float* aw = de + w;
  const float kappa = 3.0f * kU + gamma_k(w);
  const bool elu = net.act == ISX_ACT_ELU;
  for (int64_t cell = blockIdx.x; cell < n; cell += gridDim.x) {
    float xc[3], h[3];
    cell_box(src, cell, inflate, xc, h);
    if (mode == ISX_BOUND_CLT)
      for (int d = 0; d < 3; ++d) h[d] *= kInvSqrt3;
    auto activate = [&](int k, float c, float r, float dl) {
      const Lin L = linearise(mode, net.act, inflate, c, r, dl);
      a[k] = L.center;
      al[k] = L.alpha;
      ga[k] = L.gamma;
      rad[k] = r;
      if (inflate) ra[k] = fmaf(L.alpha, r, L.gamma);
    };
    __syncthreads();                               // the cell before is done
    if (t < w) {
      const float w0 = net.W0[3 * t], w1 = net.W0[3 * t + 1], w2 = net.W0[3 * t + 2], bb = net.b0[t];
      const float c = fmaf(w2, xc[2], fmaf(w1, xc[1], fmaf(w0, xc[0], bb)));
      const float x0 = h[0] * w0, x1 = h[1] * w1, x2 = h[2] * w2;
      X[t] = x0;
      X[w + t] = x1;
      X[2 * w + t] = x2;
      const float r = input_radius(mode, x0, x1, x2);
      float dl = 0.0f;
      if (inflate) {
        const float e = fabsf(w0 * xc[0]) + fabsf(w1 * xc[1]) + fabsf(w2 * xc[2]) + fabsf(bb);
        dl = (5.0f * kU * e + 3.0f * kU * r) * kSafe;
      }
      activate(t, c, r, dl);
    }
    int S = 3;
    for (int j = 1; j < H; ++j) {
      const float* __restrict__ Wt = net.Wt[j];
      __syncthreads();
      // centre (and slack) of the next layer: one neuron per thread of the last two warps
      float cn = 0.0f;
      const int nn = t - (T - 64);
      if (nn >= 0 && nn < w) {
        cn = net.b[j][nn];
        float e = fabsf(cn), g = 0.0f;
        for (int k = 0; k < w; ++k) {
          const float wk = Wt[k * w + nn];
          cn = fmaf(wk, a[k], cn);
          if (inflate) {
            e = fmaf(fabsf(wk), fabsf(a[k]), e);
            g = fmaf(fabsf(wk), ra[k], g);
          }
        }
        if (inflate) de[nn] = slack(kappa, g, w, e);
      }
      // carried rows, four per warp and turn, in place: (x alpha) W^T
      for (int r0 = 4 * warp; r0 < S; r0 += 4 * warps) {
        const int nr = min(4, S - r0);
        if (!elu)
          for (int q = 0; q < nr; ++q)
            for (int k = lane; k < w; k += 32) X[(r0 + q) * w + k] *= al[k];
        __syncwarp();
        float y[4][2] = {};
        for (int k = 0; k < w; ++k) {
          float wv[2];
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            wv[c] = lane + 32 * c < w ? Wt[k * w + lane + 32 * c] : 0.0f;
            if (elu) wv[c] = __fmul_rn(wv[c], al[k]);   // scaled weights, as in the row path
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float x = X[min(r0 + q, S - 1) * w + k];
#pragma unroll
            for (int c = 0; c < 2; ++c) y[q][c] = fmaf(x, wv[c], y[q][c]);
          }
        }
        __syncwarp();
        for (int q = 0; q < nr; ++q)
#pragma unroll
          for (int c = 0; c < 2; ++c)
            if (lane + 32 * c < w) X[(r0 + q) * w + lane + 32 * c] = y[q][c];
      }
      // new rows gamma_n W[:, n], in increasing n
      int made = 0;
      for (int g0 = 0; g0 < w; g0 += 32) {
        const float gm = g0 + lane < w ? ga[g0 + lane] : 0.0f;
        for (unsigned b = __ballot_sync(0xffffffffu, gm != 0.0f); b; b &= b - 1, ++made) {
          if (made % warps != warp) continue;
          const int l = __ffs(b) - 1;
          const float g = __shfl_sync(0xffffffffu, gm, l);
          for (int m = lane; m < w; m += 32) X[(S + made) * w + m] = g * Wt[(g0 + l) * w + m];
        }
      }
      S += made;
      __syncthreads();
      if (nn >= 0 && nn < w) {
        float s = 0.0f, comp = 0.0f;
        for (int r = 0; r < S; ++r) add_term(s, comp, X[r * w + nn], mode == ISX_BOUND_CLT);
        activate(nn, cn, (mode == ISX_BOUND_CLT) ? sqrtf(s) : s, inflate ? de[nn] : 0.0f);
      }
    }
    __syncthreads();
    // output layer: the terms of rows r to partial sum r % 8, as in k_output
    if (t < w) aw[t] = al[t] * net.wout[t];
    __syncthreads();
    const bool sq = (mode != ISX_BOUND_SOUND);
    for (int u = warp; u < 8; u += warps) {
      float s = 0.0f, comp = 0.0f;
      for (int r = u; r < S; r += 8) {
        float y = 0.0f;
        if (4 * lane < w) {
          const float4 v = *reinterpret_cast<const float4*>(aw + 4 * lane), x = *reinterpret_cast<const float4*>(X + r * w + 4 * lane);
          y = fmaf(x.w, v.w, fmaf(x.z, v.z, fmaf(x.y, v.y, fmaf(x.x, v.x, y))));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
        add_term(s, comp, y, sq);
      }
      if (lane == 0) part[u] = s;
    }
    __syncthreads();
    if (warp == 0) {
      float rows = 0.0f;
      for (int k = 0; k < 8; ++k) rows += part[k];
      float v[4] = {0.f, 0.f, 0.f, 0.f};
      for (int m = lane; m < w; m += 32) {
        const float wo = net.wout[m], y = ga[m] * wo;
        v[0] = sq ? fmaf(y, y, v[0]) : v[0] + fabsf(y);
        v[1] = fmaf(wo, a[m], v[1]);
        if (inflate) {
          v[2] = fmaf(fabsf(wo), fabsf(a[m]), v[2]);
          v[3] = fmaf(fabsf(wo), fmaf(al[m], rad[m], ga[m]), v[3]);
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
      if (lane == 0) {
        const float tot = rows + v[0];
        float sp;
        if (mode == ISX_BOUND_SOUND) {
          sp = tot;
          if (inflate) {
            float ge = gamma_k(w + 1) + kU;
            sp = __fadd_ru(__fmul_ru(sp, kSafe), (ge * v[3] + gamma_k(w + 2) * (v[2] + fabsf(net.bout))) * 1.01f);
          }
        } else if (mode == ISX_BOUND_CLT) {
          sp = sqrtf(tot);
        } else {
          sp = sqrtf(tot / 3.0f);
        }
        center[cell] = v[1] + net.bout;
        spread[cell] = sp;
      }
    }
  }
}

}  // namespace

isx_status bound_fp32(isx_inr inr, const CellSource& src, int64_t n, isx_bound_mode mode,
                      int inflate, float* d_center, float* d_spread, cudaStream_t st) {
  if (n <= 0) return ISX_OK;
  const int w = inr->w, H = inr->H;
  if (mode != ISX_BOUND_SOUND) inflate = 0;
  // Small networks in one launch: with up to two hidden layers to 8192 cells (32768 cells: 392 us against 364 at
  // 64 x 2, 234 against 189 at 32 x 2), deeper ones to 64 neurons per SM (16 x 8, 200 cells: 75 us against 274;
  // 64 x 6 with every symbol alive, 152 cells: 178 against 321; beyond that the row path's tuned tiles, whose
  // products use a weight more than four times, take over).
  if (w <= 64 && small_smem(w, H) <= 100 * 1024 && (H <= 2 ? n <= 8192 : n * w <= 64 * (int64_t)inr->sms)) {
    SmallNet net{};
    net.W0 = inr->W[0];
    net.b0 = inr->b[0];
    for (int j = 1; j < H; ++j) {
      net.Wt[j] = inr->Wt[j];
      net.b[j] = inr->b[j];
    }
    net.wout = inr->W[H];
    net.bout = inr->hb[H][0];
    net.w = w;
    net.H = H;
    net.act = inr->act;
    const size_t smem = small_smem(w, H);
    if (smem > 48 * 1024)
      ISX_CUDA(cudaFuncSetAttribute(k_bound_small, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024));
    {
      prof::Scope _ps(K_BOUND_SMALL, st, 2.0 * n * w * (double)w * 4.0 * (H - 1), 0);
      k_bound_small<<<(unsigned)std::min<int64_t>(n, 16 * (int64_t)inr->sms), H <= 2 ? 128 : kSmallT, smem, st>>>(src, n, net, (int)mode, inflate,
                                                                                                 d_center, d_spread);
    }
    ISX_LAUNCH_CHECK("k_bound_small");
    return ISX_OK;
  }
  const bool elu = inr->act == ISX_ACT_ELU;
  const int pad = elu ? kPad - 1 : 0, rs = elu ? kPad : 3;   // row alignment - 1, rows kept for the input's three
  const int Smax = rs + w * (H - 1);
  // Even chunks of as many cells as the two row buffers hold with every symbol alive, so that the host needs no row
  // count and a call only enqueues.  (Chunks of as many cells as the rows that exist allow need one count per layer
  // on the host, which waits for the stream: 20003 cells of the 3 -> 256 x 5 -> 1 network 15.7 ms against 16.1, but 30000
  // of 3 -> 128 x 4 -> 1 with inflation 12.4 against 8.9, for the chunks that it starts over.)  The last layer's rows
  // go to one buffer, fewer to the other.  They take at most 12 GB (with 6 GB those 20003 cells take 17.0 ms), or 6
  // for good on a device that does not have them.
  const int64_t Sprev = H > 1 ? Smax - w : 0;
  const size_t per_cell = (size_t)(Smax + Sprev) * w * sizeof(float);
  auto& ws = inr->ws;
  const Slot xs[2] = {WS_X0, WS_X1}, rc[2] = {WS_R_RC0, WS_R_RC1}, ns[2] = {WS_R_CNT0, WS_R_CNT1},
             os[2] = {WS_R_OFF0, WS_R_OFF1};
  int64_t chunk = 0;
  auto reserve = [&]() -> isx_status {
    const int64_t fit = std::min<int64_t>((int64_t)1 << 16, std::max<int64_t>(1, inr->fp32_row_bytes / (int64_t)per_cell));
    const int64_t chunks = (n + fit - 1) / fit;
    const int64_t cap = std::min(n, fit);          // not the chunk, so that a shorter list never needs more
    chunk = (n + chunks - 1) / chunks;
    for (int i = 0; i < 2; ++i) {
      const size_t rows = (size_t)cap * ((i == 0) == (H % 2 == 1) ? Smax : Sprev);   // layer j's go to buffer (j - 1) % 2
      ISX_TRY(ws[xs[i]].ensure(rows * w * sizeof(float), "rows"));
      ISX_TRY(ws[rc[i]].ensure(rows * sizeof(int), "row cells"));
    }
    for (Slot s : {WS_C, WS_R_A, WS_RAD, WS_ALPHA, WS_GAMMA, WS_DELTA})
      ISX_TRY(ws[s].ensure((size_t)cap * w * sizeof(float), "per-neuron"));
    for (Slot s : {WS_R_CNT0, WS_R_CNT1}) ISX_TRY(ws[s].ensure((size_t)cap * sizeof(int), "row counts"));
    for (Slot s : {WS_R_OFF0, WS_R_OFF1}) ISX_TRY(ws[s].ensure((size_t)cap * sizeof(int64_t), "row offsets"));
    return ws[WS_R_TOT].ensure(rows::scan_bytes(cap), "row total and scan block sums");
  };
  isx_status reserved = reserve();
  if (reserved == ISX_ERR_NOMEM && inr->fp32_row_bytes > kFp32RowBytesLess) {
    for (int i = 0; i < 2; ++i) {
      ws[xs[i]].release();
      ws[rc[i]].release();
    }
    inr->fp32_row_bytes = kFp32RowBytesLess;
    reserved = reserve();
  }
  ISX_TRY(reserved);
  int64_t* d_tot = ws[WS_R_TOT].as<int64_t>();
  float* RAD = ws[WS_RAD].as<float>();
  float* AL = ws[WS_ALPHA].as<float>();
  float* GA = ws[WS_GAMMA].as<float>();
  float* DE = ws[WS_DELTA].as<float>();
  const int sms = inr->sms;
  const CellBlock cb(w);
  for (int64_t first = 0; first < n; first += chunk) {
    const int nc = (int)std::min<int64_t>(chunk, n - first);
    float* C = ws[WS_C].as<float>();
    float* C2 = ws[WS_R_A].as<float>();
    // few cells: a whole block per cell in the kernels that walk over a cell's rows (up to 8 cells per SM, or 64 where
    // a cell may have 256 KB of them: a chunk of 3334 cells of the 3 -> 256 x 5 -> 1 network 3.14 -> 2.80 ms, but 5000
    // cells of 80 x 1 40 -> 54 us and of 16 x 5 202 -> 237); up to one
    // cell per SM they are spread over several blocks per cell, since one SM alone is bound by
    // its loads' latency (every symbol alive, 400 x 5: 1 cell 672 -> 350 us, 152 cells 3918 -> 3601; 256 x 5, 600
    // cells: 775 us either way)
    const bool wide = nc < ((int64_t)w * w * (H - 1) >= 65536 ? 64 : 8) * sms;
    const bool few = nc <= sms;
    int cur = 0;
    int64_t R = rs * (int64_t)nc;                  // rows of z_j: an upper bound, but for the input's
    {
      prof::Scope _ps(K_INPUT, st, 0, 0);
      k_input_layer<<<cb.blocks(nc), cb.threads(), 0, st>>>(
          src, first, nc, cb.tpc, rs, inr->W[0], inr->b[0], w, (int)mode, inr->act, inflate, C, ws[xs[0]].as<float>(),
          ws[rc[0]].as<int>(), RAD, AL, GA, ws[os[0]].as<int64_t>(), ws[ns[0]].as<int>(), ws[ns[1]].as<int>());
    }
    ISX_LAUNCH_CHECK("k_input_layer");
    for (int j = 1; j <= H - 1; ++j) {
      const int nxt = cur ^ 1;
      int* cnt_in = ws[ns[cur]].as<int>();
      int* cnt_out = ws[ns[nxt]].as<int>();
      int64_t* off_in = ws[os[cur]].as<int64_t>();
      int64_t* off_out = ws[os[nxt]].as<int64_t>();
      float* Xa = ws[xs[cur]].as<float>();
      float* Xb = ws[xs[nxt]].as<float>();
      // d_tot[j & 1]: rows of z_{j+1}; the other one still holds those of z_j
      {
        prof::Scope _ps(K_SCAN, st, 0, 0);
        ISX_TRY(rows::scan_counts(cnt_out, nc, d_tot, j & 1, off_out, st, pad));
      }
      // the tile shape comes from the autotuner (timed once per width and row-count bucket)
      {
        GemmArgs g{};
        g.X = Xa;
        g.Y = Xb;
        g.Wt = inr->Wt[j];
        g.alpha = AL;
        g.rowcell = ws[rc[cur]].as<int>();
        g.off_in = off_in;
        g.off_out = off_out;
        g.d_R = j == 1 ? nullptr : d_tot + ((j - 1) & 1);
        g.R = R;
        int64_t bucket = 1;
        while (bucket < std::min<int64_t>(R, 1 << 16)) bucket <<= 1;
        const std::string key = std::string(elu ? "gemm_fp32 elu w=" : "gemm_fp32 w=") + std::to_string(w) + " rows<=" + std::to_string(bucket);
        auto run = [&](int v) { return elu ? launch_gemm<kWeights>(v, g, w, sms, st) : launch_gemm<kRows>(v, g, w, sms, st); };
        int v = 0;
        ISX_TRY(tune::pick(key, kGemmVariants, [&](int i) { return kGemmShapes[i].name; }, run, st, &v));
        // the work that is counted: the input rows alone, since only the device knows how many there are from layer 2 on
        const double rows_known = g.d_R ? 3.0 * nc : (double)R;
        prof::Scope _ps(K_GEMM_FP32, st, 2.0 * rows_known * w * w, 8.0 * rows_known * w);
        ISX_TRY(run(v));
      }
      {
        prof::Scope _ps(K_FRESH, st, 0, 0);
        if (wide)
          k_fresh_rows<8><<<dim3(nc, few ? (w + 63) / 64 : 1), 256, 0, st>>>(nc, w, GA, inr->Wt[j], cnt_in, cnt_out, off_out,
                                                                             Xb, ws[rc[nxt]].as<int>(), pad);
        else
          k_fresh_rows<1><<<(nc + 7) / 8, 256, 0, st>>>(nc, w, GA, inr->Wt[j], cnt_in, cnt_out, off_out, Xb,
                                                        ws[rc[nxt]].as<int>(), pad);
      }
      ISX_LAUNCH_CHECK("k_fresh_rows");
      {
        prof::Scope _ps(K_GEMV, st, 2.0 * nc * w * w, 0);
        if (inflate || few) {
          k_center_gemv<<<dim3(nc, few ? (w + 63) / 64 : 1), few ? 64 : std::min(w, 256), 2 * w * sizeof(float), st>>>(
              w, inr->Wt[j], inr->b[j], C, AL, RAD, GA, C2, DE, inflate, 3.0f * kU + gamma_k(w));
          ISX_LAUNCH_CHECK("k_center_gemv");
        } else {
          GemmArgs g{};
          g.X = C;
          g.Y = C2;
          g.Wt = inr->Wt[j];
          g.bias = inr->b[j];
          g.R = nc;
          ISX_TRY(launch_gemm<kCentres>((int64_t)nc * w < (int64_t)sms * 8192 ? 4 : 0, g, w, sms, st));
        }
        std::swap(C, C2);
      }
      {
        prof::Scope _ps(K_REDUCE, st, 0, 0);
        const ReduceArgs g{Xb, off_out, cnt_out, nc, w, (int)mode, inr->act, inflate, C, RAD, DE, AL, GA};
        int* next = j < H - 1 ? cnt_in : nullptr;
        if (few)
          ISX_TRY(launch_clusters(k_reduce_few, (unsigned)(w + 63) / 64, nc, 64, 0, st, g, next));
        else
          k_reduce_act<<<cb.blocks(nc), cb.threads(), 0, st>>>(g, cb.tpc, next);
      }
      ISX_LAUNCH_CHECK("k_reduce_act");
      cur = nxt;
      R = (int64_t)nc * (rs + (int64_t)w * j);
    }
    const int L = inr->n_layers - 1;
    {
      prof::Scope _ps(K_OUTPUT, st, 0, 0);
      const float* X = ws[xs[cur]].as<float>();
      const int64_t* off = ws[os[cur]].as<int64_t>();
      const int* cnt = ws[ns[cur]].as<int>();
      if (few && H > 1)                              // one hidden layer leaves a cell three rows
        ISX_TRY(launch_clusters(8 * nc <= 2 * sms ? k_output<64> : k_output<32>, 8 * nc <= 2 * sms ? 8 : 4, nc, 256,
                                (w + kOutRows) * sizeof(float), st, X, off, cnt, nc, w, (const float*)C, (const float*)AL,
                                (const float*)GA, (const float*)RAD, (const float*)inr->W[L], inr->hb[L][0], (int)mode,
                                inflate, d_center, d_spread, first));
      else if (wide)
        k_output<8><<<nc, 256, w * sizeof(float), st>>>(X, off, cnt, nc, w, C, AL, GA, RAD, inr->W[L], inr->hb[L][0],
                                                        (int)mode, inflate, d_center, d_spread, first);
      else
        k_output<1><<<(nc + 7) / 8, 256, 8 * w * sizeof(float), st>>>(X, off, cnt, nc, w, C, AL, GA, RAD, inr->W[L],
                                                                      inr->hb[L][0], (int)mode, inflate, d_center,
                                                                      d_spread, first);
    }
    ISX_LAUNCH_CHECK("k_output");
  }
  return ISX_OK;
}

}  // namespace isx
