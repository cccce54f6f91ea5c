// RA-Fixed bounds (the reduced range-analysis baseline of Sec. V-A.4 and App. A): sound affine
// arithmetic that keeps only the three input symbols and condenses every other coefficient of a
// neuron into one non-negative radius private to that neuron.
//
// Per cell and neuron the carried form is  c + a_1 eps_1 + a_2 eps_2 + a_3 eps_3 + r eta_n:
//   input box:  c = W_0 x_c + b_0,  a_d = h_d W_0[:, d],  r = 0
//   linear:     c' = W c + b,  a_d' = W a_d,  r' = |W| r               (Eq. 3 on the kept symbols)
//   ReLU:       Chebyshev line on [c - s, c + s], s = |a_1| + |a_2| + |a_3| + r   (Eq. 4)
//               c' = alpha c + beta,  a_d' = alpha a_d,  r' = alpha r + gamma
//   output:     [y_c - s_y, y_c + s_y],  s_y = sum_d |w . a_d| + |w| . r   (Eq. 2)
//
// One fused kernel runs the whole network for a tile of cells with the cells' forms resident in
// shared memory: [quantity][neuron][cell] for the quantities c, a_1..3, r.  A layer is a dense
// contraction of the rows c, a_d with W and of r with |W|, computed in float32 by register tiles: a
// thread owns 8 neurons of CPT = 4 (or 2) cells and accumulates all quantities of those pairs over k, so
// the ReLU is applied in registers and written back in place after a block barrier.  Bound by FP32 FMA
// issue and the shared-memory return bandwidth: two neighbouring cells share a 64-bit accumulator
// (fma.rn.f32x2, the same results as two fmaf) and 28 values read feed 160 multiply-adds; W^T streams
// through the cp.async ring of sgemm.cuh.  131075 cells of the 3 -> 256 x 5 -> 1 network: 6.38 ms, 54 TFLOP/s
// (8.05 ms with 4 x 4 tiles that read 36 values per 80 multiply-adds, the weights from global memory).
//
// Rounding-error inflation (inflate != 0): every float32 rounding is charged to r, which is a
// private symbol of its neuron, so the carried form stays a sound enclosure.  A K-term dot product
// errs by at most gamma_K sum |a_k b_k| (gamma_K = K u / (1 - K u), u = 2^-24).  Those sums are
// bounded by ||W_n||_1 M, M the largest magnitude m = |c| + sum_d |a_d| + r over the cell's neurons
// (kept per cell in shared memory, rounded up).
#include "internal.cuh"

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "cell_box.cuh"
#include "linearise.cuh"
#include "sgemm.cuh"

namespace isx {
namespace {

constexpr int ra_threads(int cpt) { return 512 / cpt; }   // threads at most, for cpt cells per thread
constexpr int kRaCols = 8;                // neurons of one thread's register tile
constexpr float kRaU = 5.9604645e-08f;    // 2^-24

__host__ __device__ __forceinline__ float ra_gamma(int k) { return (k * kRaU) / (1.0f - k * kRaU); }

struct RaLayers {
  const float* Wt[ISX_MAX_LAYERS];        // hidden layers 1 .. H-1: W^T, [w_in][w_out]
  const float* b[ISX_MAX_LAYERS];
};

// Quantities per (cell, neuron): 0 = c, 1..3 = a_d, 4 = r.
constexpr int kRaQ = 5;

// Sound ReLU on the reduced form of one (cell, neuron); v = {c, a_1, a_2, a_3, r}.  Returns the
// magnitude |c| + sum_d |a_d| + r of the result, rounded up (inflation only).
template <bool INFL>
__device__ __forceinline__ float ra_relu(float* v) {
  if (INFL) {
    const float sa = __fadd_ru(__fadd_ru(fabsf(v[1]), fabsf(v[2])), fabsf(v[3]));
    const float s = __fadd_ru(sa, v[4]);
    Lin L = relu_sound(v[0], s, 0.0f, true);
    v[0] = L.center;
    v[1] *= L.alpha;
    v[2] *= L.alpha;
    v[3] *= L.alpha;
    // r' = alpha r + gamma, plus the rounding of the three products alpha a_d
    float r = __fadd_ru(__fmul_ru(L.alpha, v[4]), L.gamma);
    v[4] = __fadd_ru(r, __fmul_ru(2.0f * kRaU, __fmul_ru(L.alpha, sa)));
    return __fadd_ru(__fadd_ru(__fadd_ru(fabsf(v[0]), fabsf(v[1])), __fadd_ru(fabsf(v[2]), fabsf(v[3]))), v[4]);
  } else {
    const float s = fabsf(v[1]) + fabsf(v[2]) + fabsf(v[3]) + v[4];
    Lin L = relu_sound(v[0], s, 0.0f, false);
    v[0] = L.center;
    v[1] *= L.alpha;
    v[2] *= L.alpha;
    v[3] *= L.alpha;
    v[4] = fmaf(L.alpha, v[4], L.gamma);
    return 0.0f;
  }
}

// Shared memory of a CTA, in floats: the forms [Q][w][cells], the weight ring, the largest magnitudes [2][cells].
// The output layer's sums [Q + 1][cells] go over the ring, which at w = 16 is smaller than they are (256 cells per
// CTA: 1536 floats over 768), so the region is sized for both.
__host__ __device__ __forceinline__ size_t ra_ring(int cells, int KB, int w) {
  const size_t ring = (size_t)sgemm::kStages * KB * w, sums = (size_t)(kRaQ + 1) * cells;
  return ring > sums ? ring : sums;
}
size_t ra_smem(int cells, int KB, int w) {
  return ((size_t)kRaQ * cells * w + ra_ring(cells, KB, w)) * sizeof(float) + 2 * (size_t)cells * sizeof(unsigned);
}

template <bool INFL, int CPT>
__global__ void __launch_bounds__(ra_threads(CPT), 2)
k_bound_rafixed(CellSource src, int64_t first, int64_t n, int cells, int KB, int w, int H, const float* __restrict__ W0,
                const float* __restrict__ b0, RaLayers layers, const float* __restrict__ wout, float bout,
                float* __restrict__ center, float* __restrict__ spread) {
  constexpr int Q = kRaQ;
  constexpr int TN = kRaCols;
  extern __shared__ float4 ra_smem4[];
  float* S = reinterpret_cast<float*>(ra_smem4);   // [Q][w][cells]
  const int t = threadIdx.x;
  const int pgs = cells / CPT, pg = t % pgs, ng = t / pgs;
  const bool active = ng < w / TN;
  const int64_t cta_first = first + (int64_t)blockIdx.x * cells;
  auto at = [&](int q, int cell, int col) -> float& { return S[((size_t)q * w + col) * cells + cell]; };
  // the thread's neuron pair j (of TN / 2): neurons col(j), col(j) + 1
  auto col_of = [&](int j) { return (j >> 1) * (w >> 1) + 4 * ng + 2 * (j & 1); };
  const int spl = w / KB;
  sgemm::Stream ws{S + (size_t)Q * cells * w, w, KB, (int64_t)(H - 1) * spl};
  // per-cell largest magnitude, double-buffered across layers (non-negative floats order as ints)
  unsigned* Mx = reinterpret_cast<unsigned*>(S + (size_t)Q * cells * w + ra_ring(cells, KB, w));
  int sl = 1, sk = 0;                              // layer and K block of the stage to load next
  auto load_next = [&] {
    ws.load(layers.Wt[min(sl, H - 1)] + (size_t)sk * KB * w);
    if (++sk == spl) {
      sk = 0;
      ++sl;
    }
  };
  for (int s = 0; s < sgemm::kStages - 1; ++s) load_next();
  if (INFL) {
    for (int i = t; i < 2 * cells; i += blockDim.x) Mx[i] = 0u;
    __syncthreads();
  }

  // the thread's cells of (quantity, neuron), one 8- or 16-byte store
  auto put = [&](int col, const float (*v)[Q]) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      float* d = &at(q, pg * CPT, col);
      if constexpr (CPT == 4) *reinterpret_cast<float4*>(d) = make_float4(v[0][q], v[1][q], v[2][q], v[3][q]);
      else *reinterpret_cast<float2*>(d) = make_float2(v[0][q], v[1][q]);
    }
  };

  // ---- input layer (3 -> w) and first ReLU, written into shared memory ----
  if (active) {
    float xc[CPT][3], h[CPT][3];
#pragma unroll
    for (int i = 0; i < CPT; ++i) {
      int64_t gi = cta_first + pg * CPT + i;
      if (gi >= first + n) gi = first + n - 1;     // ragged tile: recompute the last cell, never stored
      cell_box(src, gi, INFL ? 1 : 0, xc[i], h[i]);
    }
#pragma unroll 1
    for (int j = 0; j < TN; ++j) {
      const int col = col_of(j >> 1) + (j & 1);
      const float w0 = W0[3 * col], w1 = W0[3 * col + 1], w2 = W0[3 * col + 2], bb = b0[col];
      float v[CPT][Q];
#pragma unroll
      for (int i = 0; i < CPT; ++i) {
        v[i][0] = fmaf(w2, xc[i][2], fmaf(w1, xc[i][1], fmaf(w0, xc[i][0], bb)));
        v[i][1] = h[i][0] * w0;
        v[i][2] = h[i][1] * w1;
        v[i][3] = h[i][2] * w2;
        v[i][4] = 0.0f;
        if (INFL) {
          // three fused multiply-adds and three products, each rounded once
          const float e = fabsf(w0 * xc[i][0]) + fabsf(w1 * xc[i][1]) + fabsf(w2 * xc[i][2]) + fabsf(bb);
          const float sa = fabsf(v[i][1]) + fabsf(v[i][2]) + fabsf(v[i][3]);
          v[i][4] = (5.0f * kRaU * e + 3.0f * kRaU * sa) * 1.01f;
        }
        const float mag = ra_relu<INFL>(v[i]);
        if (INFL) atomicMax(&Mx[pg * CPT + i], __float_as_uint(mag));
      }
      put(col, v);
    }
  }

  // ---- hidden layers 1 .. H-1: contraction with W (rows c, a_d) and |W| (row r), then ReLU ----
  int slot = 0;
  for (int l = 1; l < H; ++l) {
    const float* __restrict__ bias = layers.b[l];
    uint64_t acc[Q][CPT / 2][TN];                  // pairs of neighbouring cells
    float wabs[TN];                                // ||W_n||_1 of the thread's neurons (inflation)
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
      for (int i = 0; i < CPT / 2; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[q][i][j] = 0ull;
#pragma unroll
    for (int j = 0; j < TN; ++j) wabs[j] = 0.0f;
    const unsigned* Mprev = Mx + ((l - 1) & 1) * cells;
    unsigned* Mnext = Mx + (l & 1) * cells;
    for (int kb = 0; kb < spl; ++kb) {
      sgemm::cp_wait<sgemm::kStages - 2>();
      __syncthreads();                             // the stage has landed, the one before it is free, S is written
      load_next();
      if (INFL && kb == 0)
        for (int i = t; i < cells; i += blockDim.x) Mnext[i] = 0u;   // its last reader was layer l - 1
      if (active) {
        const float* xr = S + (size_t)kb * KB * cells + CPT * pg;
        const float* wr = ws.Ws + (size_t)slot * KB * w + 4 * ng;
        for (int k0 = 0; k0 < KB; k0 += 4) {
          float pair01[TN], pair23[TN];
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const int k = k0 + kk;
            const float4 wl = *reinterpret_cast<const float4*>(wr + k * w);
            const float4 wh = *reinterpret_cast<const float4*>(wr + k * w + (w >> 1));
            const float wv[TN] = {wl.x, wl.y, wl.z, wl.w, wh.x, wh.y, wh.z, wh.w};
            if (INFL) {
              // ||W_n||_1 in groups of four k: (|w_0| + |w_1|) + (|w_2| + |w_3|)
#pragma unroll
              for (int j = 0; j < TN; ++j) {
                float& u = kk < 2 ? pair01[j] : pair23[j];
                u = (kk & 1) ? u + fabsf(wv[j]) : fabsf(wv[j]);
                if (kk == 3) wabs[j] += pair01[j] + pair23[j];
              }
            }
            uint64_t x[Q][CPT / 2];
#pragma unroll
            for (int q = 0; q < Q; ++q) {
              const float* xq = xr + ((size_t)q * w + k) * cells;
              if constexpr (CPT == 4) {
                const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(xq);
                x[q][0] = u.x;
                x[q][1] = u.y;
              } else {
                x[q][0] = *reinterpret_cast<const uint64_t*>(xq);
              }
            }
#pragma unroll
            for (int j = 0; j < TN; ++j) {
              const uint64_t ww = sgemm::pack2(wv[j], wv[j]), wa = sgemm::pack2(fabsf(wv[j]), fabsf(wv[j]));
#pragma unroll
              for (int q = 0; q < Q; ++q) {
#pragma unroll
                for (int i = 0; i < CPT / 2; ++i) acc[q][i][j] = sgemm::fma2(x[q][i], q >= 4 ? wa : ww, acc[q][i][j]);
              }
            }
          }
        }
      }
      slot = slot == sgemm::kStages - 1 ? 0 : slot + 1;
    }
    __syncthreads();                               // every thread is done reading layer l-1
    if (active) {
      const float gk = ra_gamma(w + 8);
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int col = col_of(j >> 1) + (j & 1);
        const float bb = bias[col];
        float v[CPT][Q];
#pragma unroll
        for (int i = 0; i < CPT; ++i) {
          const int cell = pg * CPT + i;
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            const float2 a = sgemm::unpack2(acc[q][i >> 1][j]);
            v[i][q] = (i & 1) ? a.y : a.x;
          }
          v[i][0] += bb;
          if (INFL) {
            // E = ||W_n||_1 M + |b_n| >= sum_k |W_nk| (|c_k| + sum_d |a_dk| + r_k) + |b_n| bounds
            // every row's dot-product error by gamma_K E; four rows (c, a_1..3) are charged, and r'
            // (a sum of non-negative terms) is scaled up by its own relative error
            const float one = 1.0f + 2.0f * gk;
            const float E = __fmul_ru(__fadd_ru(__fmul_ru(wabs[j], __uint_as_float(Mprev[cell])), fabsf(bb)), one);
            v[i][4] = __fadd_ru(__fmul_ru(v[i][4], one), __fmul_ru(4.0f * gk, E));
            v[i][4] = __fadd_ru(v[i][4], __fmul_ru(kRaU, fabsf(v[i][0])));      // the bias addition
          }
          const float mag = ra_relu<INFL>(v[i]);
          if (INFL) atomicMax(&Mnext[cell], __float_as_uint(mag));
        }
        put(col, v);
      }
    }
  }
  __syncthreads();

  // ---- output layer (w -> 1) and the read-off: one thread per (quantity, cell), then one per cell.  Each sum is 32
  //      partial sums over the neurons l, l + 32, ..., added as a 32-lane butterfly adds them ----
  constexpr int YQ = INFL ? Q + 1 : Q;             // quantity Q: ||w_out||_1
  float* Y = ws.Ws;                                // [YQ][cells], the weight stages are done (ra_ring holds both)
  for (int u = t; u < YQ * cells; u += blockDim.x) {
    const int q = u / cells, cell = u - q * cells;
    const bool ones = q == Q;                      // a sum of |wout| alone: fmaf(|wout|, 1, y)
    const float* x = S + (ones ? 0 : (size_t)q * w * cells) + cell;
    float y[32];
#pragma unroll
    for (int l = 0; l < 32; ++l) y[l] = 0.0f;
    // N neurons from c0 on with every load in flight: w is a multiple of 16, so none of them needs a test (with a test
    // per neuron the loads went one after the other, 75 ns each: a CTA's output layer took 35 us at w = 512)
    auto add = [&](int c0, auto N) {
      float wo[N], xv[N];
#pragma unroll
      for (int l = 0; l < N; ++l) {
        wo[l] = wout[c0 + l];
        xv[l] = x[(size_t)(c0 + l) * cells];
      }
#pragma unroll
      for (int l = 0; l < N; ++l) y[l] = fmaf(q >= 4 ? fabsf(wo[l]) : wo[l], ones ? 1.0f : xv[l], y[l]);
    };
    int c0 = 0;
    for (; c0 + 32 <= w; c0 += 32) add(c0, std::integral_constant<int, 32>{});
    if (c0 < w) add(c0, std::integral_constant<int, 16>{});
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int l = 0; l < o; ++l) y[l] += y[l + o];
    Y[u] = y[0];
  }
  __syncthreads();
  const unsigned* Mlast = Mx + ((H - 1) & 1) * cells;
  for (int cell = t; cell < cells; cell += blockDim.x) {
    const int64_t gi = cta_first + cell;
    if (gi >= first + n) break;
    float y[YQ];
#pragma unroll
    for (int q = 0; q < YQ; ++q) y[q] = Y[q * cells + cell];
    const float c = y[0] + bout;
    float s;
    if (INFL) {
      const float gk = ra_gamma(w + 8);
      const float one = 1.0f + 2.0f * gk;
      const float sa = __fadd_ru(__fadd_ru(fabsf(y[1]), fabsf(y[2])), fabsf(y[3]));
      const float E = __fmul_ru(__fadd_ru(__fmul_ru(y[YQ - 1], __uint_as_float(Mlast[cell])), fabsf(bout)), one);
      s = __fadd_ru(__fadd_ru(sa, __fmul_ru(y[4], one)), __fmul_ru(4.0f * gk, E));
      s = __fadd_ru(s, __fmul_ru(kRaU, fabsf(c)));
    } else {
      s = fabsf(y[1]) + fabsf(y[2]) + fabsf(y[3]) + y[4];
    }
    center[gi] = c;
    spread[gi] = s;
  }
}

}  // namespace

bool rafixed_supported(isx_inr inr) { return inr->w % 16 == 0 && inr->w / kRaCols <= ra_threads(4); }

isx_status bound_rafixed(isx_inr inr, const CellSource& src, int64_t n, int inflate, float* d_center,
                         float* d_spread, cudaStream_t st) {
  if (n <= 0) return ISX_OK;
  const int w = inr->w, H = inr->H;
  if (!rafixed_supported(inr)) {
    set_error("RA-Fixed bounds need a hidden width that is a multiple of 16 and at most 1024");
    return ISX_ERR_UNSUPPORTED;
  }
  RaLayers lay{};
  for (int l = 1; l < H; ++l) {
    lay.Wt[l] = inr->Wt[l];
    lay.b[l] = inr->b[l];
  }
  const int L = inr->n_layers - 1;
  // Cells per CTA: 128 threads' worth of four cells each (eight warps on the SM's two CTAs keep the multiply-adds
  // fed); with fewer than that for every SM one CTA each, of at least 64 threads (they share the weight stream).  Two
  // smaller ones may put two warps on the same sub-partition of the SM: 4300 cells of w = 144 in 182 us, not 125.
  const int sms = inr->sms;
  // At small widths the input and output layers weigh more and twice the warps with two cells each hide more of their
  // latency (w = 64, two hidden layers, 5000 cells: 41 us against 45, 39000 cells 72 against 77).  So do they while one
  // CTA of 128 threads per SM takes all cells, where a CTA's own chain is the time (w = 512, eight layers, up to 608
  // cells: 480 us against 609; w = 256, five: 137 against 185 up to 1216 cells; beyond, four: 2400 cells of w = 512 in
  // 970 us against 1071).
  const int few_cells = 2 * (128 * kRaCols / w);
  const bool few = few_cells > 0 && n <= (int64_t)sms * few_cells;
  const int cpt = w <= 64 || few ? 2 : 4;
  const int most = ra_threads(cpt) / (w / kRaCols) * cpt;
  const int64_t even = (n + sms - 1) / sms;
  const int cells = few ? few_cells
                        : (int)std::min<int64_t>(most, std::max<int64_t>((most / 2 + 3) / 4 * 4, (even + 3) / 4 * 4) / cpt * cpt);
  const int KB = 16 * w <= 2048 ? 16 : (8 * w <= 2048 ? 8 : 4);
  const int threads = (w / kRaCols * (cells / cpt) + 31) / 32 * 32;
  const size_t smem = ra_smem(cells, KB, w);
  // the grid's x dimension is bounded; long lists run in slices
  const int64_t max_ctas = 1 << 30;
  const double flops = 2.0 * 5.0 * w * (double)w * (H - 1) + 2.0 * 3.0 * 4.0 * w + 2.0 * 5.0 * w;
  for (int64_t off = 0; off < n; off += max_ctas * cells) {
    const int64_t m = std::min<int64_t>(n - off, max_ctas * cells);
    const unsigned grid = (unsigned)((m + cells - 1) / cells);
    prof::Scope _ps(K_BOUND_RAFIXED, st, flops * (double)m, 8.0 * (double)m + 4.0 * w * w * (H - 1) * grid);
    const auto kernel = inflate ? (cpt == 4 ? k_bound_rafixed<true, 4> : k_bound_rafixed<true, 2>)
                                : (cpt == 4 ? k_bound_rafixed<false, 4> : k_bound_rafixed<false, 2>);
    ISX_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
    kernel<<<grid, threads, smem, st>>>(src, off, m, cells, KB, w, H, inr->W[0], inr->b[0], lay, inr->W[L], inr->hb[L][0],
                                        d_center, d_spread);
    ISX_LAUNCH_CHECK("k_bound_rafixed");
  }
  return ISX_OK;
}

}  // namespace isx
