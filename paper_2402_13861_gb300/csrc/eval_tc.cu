// MLP evaluation at points on the tensor cores (the corner queries of Sec. IV-D and the dense
// baseline of Sec. V-A), with FP32-class accuracy from BF16 operands.
//
// Every operand is split into two BF16 terms, x = x_hi + x_lo with x_hi = bf16(x) and
// x_lo = bf16(x - x_hi) (|x_lo| <= 2^-9 |x|, x_hi + x_lo within 2^-17 |x| of x), and a product is
// taken as a_hi b_hi + a_hi b_lo + a_lo b_hi; the dropped a_lo b_lo term is below 2^-18 |a b|.
// Three tcgen05.mma (kind::f16, BF16 x BF16 -> FP32 in TMEM) per K step, so the tensor cores do 3x
// the algorithmic work, against 1/28 of their BF16 rate for FP32 FMAs on the CUDA cores.
//
// Layout: one persistent CTA per 128-point tile at a time; point p of the tile = TMEM lane p.  Bound by the
// tensor cores (three products), so everything else is kept off their path:
//  - a producer warp streams W_l through a ring of 16 KB stages (128 weight rows x one 64-wide K chunk, high
//    or low term) by TMA, ahead of the MMAs and across layers and tiles;
//  - an MMA warp starts a K chunk as soon as its 64 activations per point are in shared memory (one mbarrier
//    per chunk), into one of two accumulators;
//  - four groups of four epilogue warps (two at w = 128) read the accumulator of the layer before, each group a
//    quarter of every chunk's columns: bias, activation (ReLU, ELU or sine), split into A_hi, A_lo (K-major,
//    128-byte swizzle), chunk by chunk, so the next layer's MMAs begin after a quarter of the work;
//  - layer 0 (3 -> w, FP32 CUDA cores) of the next tile runs before the output layer of this one, whose
//    contraction with w_out (FP32, one chain over the neurons per point, handed from group to group) so
//    overlaps the next tile's first MMAs.
// With one 128-thread warpgroup that issued, waited and drained in turn 2.1 M points of 3 -> 256 x 5 -> 1 took
// 3.62 ms; this form takes 2.42 ms: of 11.2 k cycles per layer the MMAs take 6.1 k, 3.3 k go by waiting for
// weights (the 80 KB of the ring, all that fits, cover too little of the load latency) and 1.8 k until the
// first chunk of the next layer's operand is ready.  Every wait is bounded (2 s): on timeout the kernel
// records ISX_ERR_TIMEOUT, lets copies land, frees TMEM and returns.
#include "internal.cuh"
#include "tc_ptx.cuh"
#include "linearise.cuh"

#include <algorithm>
#include <cstring>

namespace isx {
namespace {

using namespace tc;

constexpr int kT = 128;                        // points per tile
constexpr uint64_t kEvWaitNs = 2000000000ull;

struct EvArgs {
  const float* xyz;
  const uint32_t* ids;
  int R;
  int64_t n;
  float* out;
  int H;                                       // activation layers; hidden GEMMs are layers 1 .. H-1
  const float* W0;                             // [w][3]
  const float* b[ISX_MAX_LAYERS];              // biases of layers 0 .. H-1
  const float* wout;                           // [w]
  float bout;
  int act;                             // isx_activation of the hidden layers
  int ns;                              // weight stages
  int* status;
};
struct EvMaps {
  CUtensorMap hi[ISX_MAX_LAYERS];              // W_l high parts, box {64, 128}
  CUtensorMap lo[ISX_MAX_LAYERS];              // W_l low parts, box {64, 128}
};

template <int W>
struct EvSmem {
  static constexpr int KC = W / 64;
  static constexpr int NH = W / 128;                      // 128-neuron halves of a layer's outputs
  static constexpr int G = W / 64;                        // epilogue groups (of four warps)
  static constexpr int NS = W == 256 ? 5 : 2;             // weight stages at most; w = 128 runs two CTAs per SM
  static constexpr int kThreads = 32 * (4 * G + 2);
  static constexpr size_t kA = (size_t)kT * W * 2;        // one activation term
  static constexpr size_t kS = 128 * 128;                 // one weight stage
  static constexpr int kBars = 2 * NS + KC + 2 + 2 * (G - 1);   // stage full / empty, chunk ready, accumulator done,
                                                                // sums handed over
  static constexpr size_t bytes(int H, int ns) {
    return 1024 + 2 * kA + ns * kS + (size_t)(3 * W + (size_t)H * W + W + 2 * (G - 1) * kT) * 4 + kBars * 8 + 16;
  }
  // stages that fit: five up to H = 10 at w = 256, four at the most layers
  static constexpr int stages(int H) { return bytes(H, NS) <= kMaxSmem ? NS : NS - 1; }
};
static_assert(EvSmem<256>::stages(10) == 5 && EvSmem<256>::stages(11) == 4 && EvSmem<256>::bytes(12, 4) <= kMaxSmem &&
              EvSmem<128>::bytes(12, 2) <= kMaxSmem);

__device__ __forceinline__ uint32_t aoff(int row, int k) {  // byte offset of (row, k..k+7), k % 8 == 0
  return (uint32_t)((k >> 6) * kT * 128 + row * 128 + ((((k & 63) >> 3) ^ (row & 7)) << 4));
}

__device__ __forceinline__ bool ewait(uint64_t* b, uint32_t parity, volatile int* abort, int* status) {
  if (mbar_try(b, parity)) return true;
  const uint64_t t0 = global_ns();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try(b, parity)) return true;
    if ((it & 3) == 0) {
      if (*abort) return false;
      if (global_ns() - t0 > kEvWaitNs) {
        *abort = 1;
        atomicExch(status, (int)ISX_ERR_TIMEOUT);
        return false;
      }
    }
  }
}

// v (after the activation) split into two BF16 terms, 8 consecutive columns, stored at A_hi / A_lo.
__device__ __forceinline__ void store_split8(uint8_t* Ahi, uint8_t* Alo, int row, int k, const float* v) {
  uint32_t ph[4], pl[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float a = v[2 * i], b = v[2 * i + 1];
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    const float2 hf = __bfloat1622float2(h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(a - hf.x, b - hf.y);
    ph[i] = *reinterpret_cast<const uint32_t*>(&h);
    pl[i] = *reinterpret_cast<const uint32_t*>(&l);
  }
  const uint32_t o = aoff(row, k);
  *reinterpret_cast<uint4*>(Ahi + o) = make_uint4(ph[0], ph[1], ph[2], ph[3]);
  *reinterpret_cast<uint4*>(Alo + o) = make_uint4(pl[0], pl[1], pl[2], pl[3]);
}

template <int W>
__global__ void __launch_bounds__(EvSmem<W>::kThreads, W == 256 ? 1 : 2)
k_eval_tc(const __grid_constant__ EvArgs args, const __grid_constant__ EvMaps maps) {
  using S = EvSmem<W>;
  constexpr int KC = S::KC, NH = S::NH, G = S::G;
  const int NS = args.ns;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* Ahi = base;
  uint8_t* Alo = Ahi + S::kA;
  uint8_t* Wst = Alo + S::kA;
  float* sW0 = reinterpret_cast<float*>(Wst + NS * S::kS);
  float* sb = sW0 + 3 * W;                     // [H][W]: biases of layers 0 .. H-1
  float* swo = sb + (size_t)args.H * W;
  float* sy = swo + W;                         // [2][G - 1][kT] the output layer's running sums, by tile parity
  uint64_t* wfull = reinterpret_cast<uint64_t*>(sy + 2 * (G - 1) * kT);
  uint64_t* wempty = wfull + NS;
  uint64_t* aready = wempty + NS;              // [KC] chunk c of the next layer's operand is in shared memory
  uint64_t* dfull = aready + KC;               // [2] accumulator complete (and A free)
  uint64_t* yready = dfull + 2;                // [2][G - 1]
  uint32_t* tslot = reinterpret_cast<uint32_t*>(yready + 2 * (G - 1));
  volatile int* abort = reinterpret_cast<volatile int*>(tslot + 1);
  const int t = threadIdx.x, warp = __shfl_sync(0xffffffffu, t >> 5, 0), lane = t & 31;
  const int H = args.H;
  const int64_t ntiles = (args.n + kT - 1) / kT;
  const int64_t tile0 = blockIdx.x;

  if (t == 0) {
    for (int i = 0; i < NS; ++i) {
      mbar_init(&wfull[i], 1);
      mbar_init(&wempty[i], 1);
    }
    for (int i = 0; i < KC; ++i) mbar_init(&aready[i], 4 * G);
    for (int i = 0; i < 2; ++i) mbar_init(&dfull[i], 1);
    for (int i = 0; i < 2 * (G - 1); ++i) mbar_init(&yready[i], 4);
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tslot)), "n"(2 * W)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  for (int i = t; i < 3 * W; i += S::kThreads) sW0[i] = args.W0[i];
  for (int l = 0; l < H; ++l)
    for (int i = t; i < W; i += S::kThreads) sb[l * W + i] = args.b[l][i];
  for (int i = t; i < W; i += S::kThreads) swo[i] = args.wout[i];
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tslot, 0);

  if (warp == 4 * G) {
    // ---- producer: per layer and K chunk, the high terms of every 128-row half, then the low terms ----
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int64_t tile = tile0; tile < ntiles && ok; tile += gridDim.x)
        for (int l = 1; l <= H - 1 && ok; ++l)
          for (int c = 0; c < KC && ok; ++c)
            for (int q = 0; q < 2 * NH; ++q, ++it) {
              const int sidx = it % NS;
              if (!ewait(&wempty[sidx], ((it / NS) & 1) ^ 1, abort, args.status)) { ok = false; break; }
              mbar_expect_tx(&wfull[sidx], (uint32_t)S::kS);
              tma_load_2d(Wst + sidx * S::kS, q < NH ? &maps.hi[l] : &maps.lo[l], &wfull[sidx], c * 64, (q % NH) * 128);
            }
    }
  } else if (warp == 4 * G + 1) {
    // ---- MMA issuer: D = A_hi W_hi^T + A_lo W_hi^T + A_hi W_lo^T, K chunk by chunk, in 128-neuron halves ----
    const uint32_t id = idesc(128), lead = elect_one();
    uint32_t sidx = 0, sph = 0, ly = 0;        // weight stage and its phase; layers so far
    bool ok = true;
    for (int64_t tile = tile0; tile < ntiles && ok; tile += gridDim.x)
      for (int l = 1; l <= H - 1 && ok; ++l, ++ly) {
        const uint32_t d = tmem + (ly & 1) * W;
        for (int c = 0; c < KC && ok; ++c) {
          ok = __all_sync(0xffffffffu, ewait(&aready[c], ly & 1, abort, args.status));
          if (!ok) break;
          tc_fence_after();
          const uint32_t ah = sdesc_lo(su32(Ahi) + c * kT * 128), al = sdesc_lo(su32(Alo) + c * kT * 128);
#pragma unroll
          for (int q = 0; q < 2 * NH; ++q) {
            ok = __all_sync(0xffffffffu, ewait(&wfull[sidx], sph, abort, args.status));
            if (!ok) break;
            tc_fence_after();
            const uint32_t w0 = sdesc_lo(su32(Wst) + sidx * (uint32_t)S::kS), dh = d + (q % NH) * 128;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
              mma_bf16_lead(dh, ah + 2 * kk, w0 + 2 * kk, id, (q >= NH || c > 0 || kk > 0) ? 1u : 0u, lead);
              if (q < NH) mma_bf16_lead(dh, al + 2 * kk, w0 + 2 * kk, id, 1u, lead);
            }
            mma_commit_lead(&wempty[sidx], lead);
            if (++sidx == (uint32_t)NS) {
              sidx = 0;
              sph ^= 1;
            }
          }
        }
        if (ok) mma_commit_lead(&dfull[ly & 1], lead);
      }
  } else {
    // ---- activations: point p = TMEM lane, group g ----
    const int g = warp >> 2, p = 32 * (warp & 3) + lane;
    const uint32_t lane_off = (uint32_t)(32 * (warp & 3)) << 16;
    constexpr int CW = 64 / G;                 // columns of a chunk per group (16 or 32)
    // chunk c of the next operand is complete for this warp
    auto ready = [&](int c) {
      fence_async_shared();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&aready[c]);
    };
    // coordinates of this thread's point of a tile (loaded a tile ahead)
    auto load_x = [&](int64_t tile, float* x) {
      const int64_t i = tile * kT + p;
      x[0] = x[1] = x[2] = 0.f;
      if (i < args.n) {
        if (args.ids) {
          const uint32_t idv = args.ids[i], n1 = (uint32_t)args.R + 1u;
          const uint32_t ix = idv % n1, iy = (idv / n1) % n1, iz = idv / (n1 * n1);
          const float inv = 2.0f / (float)args.R;
          x[0] = -1.0f + inv * (float)ix;
          x[1] = -1.0f + inv * (float)iy;
          x[2] = -1.0f + inv * (float)iz;
        } else {
          x[0] = args.xyz[3 * i];
          x[1] = args.xyz[3 * i + 1];
          x[2] = args.xyz[3 * i + 2];
        }
      }
    };
    auto layer0 = [&](const float* x) {
#pragma unroll 1
      for (int c = 0; c < KC; ++c) {
#pragma unroll
        for (int k = 0; k < CW; k += 8) {
          const int k0 = 64 * c + CW * g + k;
          float v[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const int nn = k0 + e;
            const float z = fmaf(sW0[3 * nn + 2], x[2], fmaf(sW0[3 * nn + 1], x[1], fmaf(sW0[3 * nn], x[0], sb[nn])));
            v[e] = act_fwd(args.act, z);
          }
          store_split8(Ahi, Alo, p, k0, v);
        }
        ready(c);
      }
    };
    uint32_t ly = 0, tt = 0;
    bool ok = true;
    float x[3];
    if (tile0 < ntiles) {
      load_x(tile0, x);
      layer0(x);
    }
    for (int64_t tile = tile0; tile < ntiles && ok; tile += gridDim.x, ++tt) {
      load_x(tile + gridDim.x, x);
      for (int l = 1; l <= H - 1; ++l, ++ly) {
        const bool got = ewait(&dfull[ly & 1], (ly >> 1) & 1, abort, args.status);
        if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
        tc_fence_after();
        const float* bl = sb + (size_t)l * W;
        const uint32_t trow = tmem + (ly & 1) * W + lane_off;
        if (l < H - 1) {
#pragma unroll 1
          for (int c = 0; c < KC; ++c) {
            const int k0 = 64 * c + CW * g;
            float v[CW];
            if constexpr (CW == 16) tmem_ld16(trow + k0, v);
            else tmem_ld32(trow + k0, v);
#pragma unroll
            for (int e = 0; e < CW; ++e) v[e] = act_fwd(args.act, v[e] + bl[k0 + e]);
#pragma unroll
            for (int u = 0; u < CW / 8; ++u) store_split8(Ahi, Alo, p, k0 + 8 * u, v + 8 * u);
            ready(c);
          }
        } else {
          // the operand buffers are free: layer 0 of the next tile first, then this tile's output layer,
          // one chain over the neurons, 64 of them per group
          if (tile + gridDim.x < ntiles) layer0(x);
          float y = 0.f;
#pragma unroll 1
          for (int hf = 0; hf < 2; ++hf) {
            const int k0 = 64 * g + 32 * hf;
            float v[32];
            tmem_ld32(trow + k0, v);
#pragma unroll
            for (int e = 0; e < 32; ++e) v[e] = act_fwd(args.act, v[e] + bl[k0 + e]);
            if (hf == 0 && g > 0) {
              const int q = (tt & 1) * (G - 1) + g - 1;
              const bool up = ewait(&yready[q], (tt >> 1) & 1, abort, args.status);
              if (!__all_sync(0xffffffffu, up)) ok = false;
              y = sy[q * kT + p];
            }
#pragma unroll
            for (int e = 0; e < 32; ++e) y = fmaf(swo[k0 + e], v[e], y);
          }
          if (!ok) break;
          if (g < G - 1) {
            const int q = (tt & 1) * (G - 1) + g;
            sy[q * kT + p] = y;
            __syncwarp();
            if (lane == 0) mbar_arrive(&yready[q]);
          } else {
            const int64_t i = tile * kT + p;
            if (i < args.n) args.out[i] = y + args.bout;
          }
        }
      }
    }
  }
  // ---- teardown: let in-flight copies land, free TMEM ----
  tc_fence_before();
  __syncthreads();
  if (*abort)
    for (int i = 0; i < 1000; ++i) __nanosleep(1000);
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(2 * W) : "memory");
  }
}

template <int W>
isx_status launch_eval(isx_inr inr, EvArgs a, const EvMaps& maps, int64_t ntiles, cudaStream_t st) {
  const int ns = EvSmem<W>::stages(inr->H);
  a.ns = ns;
  const size_t smem = EvSmem<W>::bytes(inr->H, ns);
  ISX_CUDA(cudaFuncSetAttribute(k_eval_tc<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
  int per_sm = 1;
  const int sms = inr->sms;
  ISX_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_eval_tc<W>, EvSmem<W>::kThreads, smem));
  // TMEM: two accumulators of W columns per CTA out of 512
  per_sm = std::max(1, std::min(per_sm, 512 / (2 * W)));
  const int grid = (int)std::min<int64_t>(ntiles, (int64_t)sms * per_sm);
  k_eval_tc<W><<<grid, EvSmem<W>::kThreads, smem, st>>>(a, maps);
  ISX_LAUNCH_CHECK("k_eval_tc");
  return ISX_OK;
}

}  // namespace

bool eval_tc_supported(isx_inr inr) { return (inr->w == 128 || inr->w == 256) && inr->H >= 2 && inr->H <= 12; }

isx_status eval_points_tc(isx_inr inr, const float* xyz, const uint32_t* lattice_ids, int R, int64_t n, float* out,
                          cudaStream_t st) {
  if (!eval_tc_supported(inr)) {
    set_error("tensor-core evaluation supports hidden widths 128 and 256 with 2..12 activation layers");
    return ISX_ERR_UNSUPPORTED;
  }
  if (n <= 0) return ISX_OK;
  const int w = inr->w, H = inr->H;
  EvArgs a{};
  a.xyz = xyz;
  a.ids = lattice_ids;
  a.R = R;
  a.n = n;
  a.out = out;
  a.H = H;
  a.W0 = inr->W[0];
  for (int l = 0; l < H; ++l) a.b[l] = inr->b[l];
  a.wout = inr->W[H];
  a.bout = inr->hb[H][0];
  a.act = inr->act;
  auto& ws = inr->ws;
  ISX_TRY(ws[WS_TC_STATUS].ensure(64, "tc status"));
  a.status = ws[WS_TC_STATUS].as<int>();
  EvMaps maps;
  std::memset(&maps, 0, sizeof(maps));
  for (int l = 1; l <= H - 1; ++l) {
    ISX_TRY(tensor_map_bf16(&maps.hi[l], inr->W_bf16[l], w, w, 64, 128));
    ISX_TRY(tensor_map_bf16(&maps.lo[l], inr->Wlo_bf16[l], w, w, 64, 128));
  }
  ISX_CUDA(cudaMemsetAsync(a.status, 0, sizeof(int), st));
  const int64_t ntiles = (n + kT - 1) / kT;
  {
    // algorithmic work: 2 (4 w + (H-1) w^2) FLOP per point
    prof::Scope ps(K_EVAL_TC, st, 2.0 * n * (4.0 * w + (H - 1.0) * w * w), 0);
    if (w == 256) {
      ISX_TRY(launch_eval<256>(inr, a, maps, ntiles, st));
    } else {
      ISX_TRY(launch_eval<128>(inr, a, maps, ntiles, st));
    }
  }
  int status = 0;
  ISX_CUDA(cudaMemcpyAsync(&status, a.status, sizeof(int), cudaMemcpyDeviceToHost, st));
  ISX_CUDA(cudaStreamSynchronize(st));
  if (status != 0) {
    set_error("tensor-core evaluation kernel gave up waiting (bounded wait expired)");
    return (isx_status)status;
  }
  return ISX_OK;
}

}  // namespace isx
