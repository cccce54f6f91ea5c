// Centre, input rows and activation of one layer of the row-batched tensor-core bound path in one kernel: the
// two-term products c' = W a + b, I'_d = (I_d diag(alpha)) W^T (Eq. 3 / 8) and, in the epilogue of the same
// tile, the reduction of z_{j+1} and its linearisation (Eq. 2 / 7, 4 / 9) from the column sums that the row GEMM
// and k_rows_new left, so that centre and input rows (4 w floats per cell) never go through memory.
#include "rows.cuh"

#include <algorithm>
#include <cstring>

#include "linearise.cuh"

namespace isx {
namespace rows {
namespace {

using namespace tc;

constexpr int kLC = 32;                         // cells of a tile (4 A rows each)
constexpr int kLE = 16;                         // epilogue warps: four per TMEM lane group, 8 cells each
constexpr int kLT = 64 + 32 * kLE;              // threads: producer, MMA, epilogue
constexpr int kLQ = 128;                        // queue entries of an epilogue warp (2 cells x 2 neurons x 32 lanes)
enum { LB_FULL, LB_EMPTY = LB_FULL + 2, LB_TFULL = LB_EMPTY + 2, LB_TEMPTY = LB_TFULL + 2, LB_COUNT = LB_TEMPTY + 2 };

struct LayerMaps {
  CUtensorMap ahi, alo;                         // split operand terms [4 nc][W] bf16, box {64, 128}
  CUtensorMap whi[2], wlo[2];                   // W_j terms, rows 2 m + h of W_j as row m of map h (W >= 256)
};

template <int W>
struct LayerSmem {
  static constexpr int KC = W / 64;
  static constexpr int NHALF = W > 256 ? 2 : 1; // W = 512: a CTA computes 256 of the output neurons
  static constexpr int NH = W >= 256 ? 2 : 1;   // 128-row MMA halves of the CTA's output neurons
  static constexpr int WR = W < 128 ? W : 128;  // weight rows of a half (W = 64: the MMA's other 64 rows are zero)
  static constexpr size_t kA = 128 * 128;       // one 64-wide K chunk of 128 rows
  static constexpr size_t kStage = (2 + 2 * NH) * kA;
  static constexpr size_t kQueue = (size_t)kLE * kLQ * 3 * sizeof(float);
  static constexpr size_t bytes() { return 1024 + 2 * kStage + kQueue + LB_COUNT * 8 + 16; }
};

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float v[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// N = 1 or 2 consecutive floats
template <int N>
__device__ __forceinline__ void ldn(const float* p, float v[N]) {
  if constexpr (N == 2) {
    const float2 x = *reinterpret_cast<const float2*>(p);
    v[0] = x.x;
    v[1] = x.y;
  } else {
    v[0] = *p;
  }
}
template <int N>
__device__ __forceinline__ void stn(float* p, const float v[N]) {
  if constexpr (N == 2) *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
  else *p = v[0];
}
// x as two bf16 terms, x_hi = bf16(x), x_lo = bf16(x - x_hi)
template <int N>
__device__ __forceinline__ void st_split(__nv_bfloat16* hi, __nv_bfloat16* lo, const float v[N]) {
  if constexpr (N == 2) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v[0], v[1]);
    const float2 f = __bfloat1622float2(h);
    *reinterpret_cast<__nv_bfloat162*>(hi) = h;
    *reinterpret_cast<__nv_bfloat162*>(lo) = __floats2bfloat162_rn(v[0] - f.x, v[1] - f.y);
  } else {
    const __nv_bfloat16 h = __float2bfloat16_rn(v[0]);
    *hi = h;
    *lo = __float2bfloat16_rn(v[0] - __bfloat162float(h));
  }
}

// D = W_j [a; alpha I]^T, transposed: TMEM lane m of half h holds neuron 2 m + h (of the CTA's 256; W <= 128: neuron
// m), column 4 c + q quantity q (0: a, 1-3: alpha I_d) of cell c of the tile.  An epilogue thread therefore
// has the centre and the three input-row entries of its two neurons of a cell in its own registers, and a
// warp's loads and stores of per-cell vectors are contiguous.
//  - warp 0 streams A_hi, A_lo, W_hi, W_lo K chunks by TMA into a two-stage ring; warp 1 issues the MMAs (three
//    products per accumulator: hi hi, lo hi, hi lo) into one of two TMEM accumulators;
//  - warps 2-17 drain the other accumulator, two cells at a time: column sums of the cell's symbol rows
//    (new rows, then the 64-row blocks of the row GEMM, compensated) plus the input rows, the linearisation, and
//    the next layer's operands.  UP with ReLU: most neurons lie on one side of the kink and need no erfc /
//    exp, so the others are queued in shared memory and evaluated 32 at a time.
// Bound by HBM: per cell 4 w bf16 pairs read and written, alpha, gamma and 2-3 column-sum vectors (12 w floats).
// LAST: no next layer; the centre and the input rows go to memory for the output layer.
template <int W, bool LAST>
__global__ void __launch_bounds__(kLT, 1) k_rows_layer(const __grid_constant__ RowsLayerArgs args,
                                                       const __grid_constant__ LayerMaps maps) {
  using S = LayerSmem<W>;
  constexpr int KC = S::KC, NHALF = S::NHALF, NH = S::NH;
  constexpr uint32_t kCols = 2 * NH * 128;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  float* queue = reinterpret_cast<float*>(base + 2 * S::kStage);
  uint64_t* bar = reinterpret_cast<uint64_t*>(base + 2 * S::kStage + S::kQueue);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + LB_COUNT);
  volatile int* abort = reinterpret_cast<volatile int*>(tslot + 1);
  const int t = threadIdx.x, warp = __shfl_sync(0xffffffffu, t >> 5, 0), lane = t & 31;
  const int64_t ntiles = (args.nc + kLC - 1) / kLC;
  const int hq = blockIdx.x % NHALF;
  const int64_t t0 = blockIdx.x / NHALF, TS = gridDim.x / NHALF;
  auto stage = [&](int s) { return base + (size_t)s * S::kStage; };

  if (S::WR < 128) {
    // W = 64: rows 64 .. 127 of the weight chunks are never loaded
    for (int s = 0; s < 2; ++s)
      for (int i = t; i < 2 * (128 - S::WR) * 8; i += kLT) {
        const int term = i / ((128 - S::WR) * 8), k = i % ((128 - S::WR) * 8);
        reinterpret_cast<uint4*>(stage(s) + (2 + term) * S::kA + S::WR * 128)[k] = make_uint4(0, 0, 0, 0);
      }
    fence_async_shared();
  }
  if (t == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bar[LB_FULL + i], 1);
      mbar_init(&bar[LB_EMPTY + i], 1);
      mbar_init(&bar[LB_TFULL + i], 1);
      mbar_init(&bar[LB_TEMPTY + i], kLE);
    }
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tslot)), "n"(kCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tslot, 0);

  if (warp == 0) {
    // ---- producer ----
    if (lane == 0) {
      uint32_t it = 0;
      for (int64_t tile = t0; tile < ntiles; tile += TS) {
        for (int c = 0; c < KC; ++c, ++it) {
          const int sidx = it & 1;
          if (!rwait(&bar[LB_EMPTY + sidx], ((it >> 1) & 1) ^ 1, abort, args.status)) break;
          uint8_t* sp = stage(sidx);
          uint64_t* full = &bar[LB_FULL + sidx];
          mbar_expect_tx(full, (uint32_t)(2 * S::kA + 2 * NH * S::WR * 128));
          tma_load_2d(sp, &maps.ahi, full, c * 64, (int)(tile * 4 * kLC));
          tma_load_2d(sp + S::kA, &maps.alo, full, c * 64, (int)(tile * 4 * kLC));
          for (int h = 0; h < NH; ++h) {
            tma_load_2d(sp + (2 + h) * S::kA, &maps.whi[h], full, c * 64, hq * 128);
            tma_load_2d(sp + (2 + NH + h) * S::kA, &maps.wlo[h], full, c * 64, hq * 128);
          }
        }
        if (*abort) break;
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer: the whole warp walks the loop, one lane issues ----
    const uint32_t id = idesc(4 * kLC), lead = elect_one();
    uint32_t it = 0, tt = 0;
    for (int64_t tile = t0; tile < ntiles; tile += TS, ++tt) {
      const uint32_t b = tt & 1;
      if (!__all_sync(0xffffffffu, rwait(&bar[LB_TEMPTY + b], ((tt >> 1) & 1) ^ 1, abort, args.status))) break;
      tc_fence_after();
      const uint32_t dt = tmem + b * NH * 128;
      bool ok = true;
      for (int c = 0; c < KC; ++c, ++it) {
        const uint32_t sidx = it & 1;
        ok = __all_sync(0xffffffffu, rwait(&bar[LB_FULL + sidx], (it >> 1) & 1, abort, args.status));
        if (!ok) break;
        tc_fence_after();
        constexpr uint32_t kD = (uint32_t)(S::kA >> 4);      // one operand chunk, in descriptor units
        const uint32_t ah = sdesc_lo(su32(base) + sidx * (uint32_t)S::kStage), al = ah + kD, w0 = al + kD;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
          for (int h = 0; h < NH; ++h) {
            const uint32_t wh = w0 + h * kD + 2 * kk, wl = wh + NH * kD;
            mma_bf16_lead(dt + h * 128, wh, ah + 2 * kk, id, (c > 0 || kk > 0) ? 1u : 0u, lead);
            mma_bf16_lead(dt + h * 128, wh, al + 2 * kk, id, 1u, lead);
            mma_bf16_lead(dt + h * 128, wl, ah + 2 * kk, id, 1u, lead);
          }
        mma_commit_lead(&bar[LB_EMPTY + sidx], lead);
      }
      if (!ok) break;
      mma_commit_lead(&bar[LB_TFULL + b], lead);
    }
  } else {
    // ---- epilogue: TMEM lane group warp % 4, cells 8 g .. 8 g + 7 of a tile ----
    const int g = (warp - 2) >> 2;
    const int m = 32 * (warp & 3) + lane;
    const bool own = m < S::WR;
    const int n0 = hq * 256 + NH * m;                       // first of this thread's NH neurons
    const uint32_t lane_off = (uint32_t)(32 * (warp & 3)) << 16;
    float* qs = queue + (size_t)(warp - 2) * kLQ * 3;       // [3][kLQ]: mu, sigma in; alpha, beta, gamma out
    const bool sq = args.sq != 0;
    const bool kink = sq && args.act == ISX_ACT_RELU;
    float bias[NH];
#pragma unroll
    for (int h = 0; h < NH; ++h) bias[h] = own ? args.bias[n0 + h] : 0.0f;
    // lanes 0-7 hold the symbol rows of the warp's eight cells: slot of the first 64-row block's column
    // sums, and how many blocks
    auto load_meta = [&](int64_t tile, int64_t& slot, int& nblk) {
      slot = 0;
      nblk = 0;
      const int64_t cell = tile * kLC + 8 * g + lane;
      if (lane < 8 && tile < ntiles && cell < args.nc) {
        const int rows = args.cnt_in[cell];
        if (rows > 0) {
          const int64_t o = args.off_in[cell], b0 = o / kPT;
          slot = rows_part_slot(cell, b0);
          nblk = (int)((o + rows - 1) / kPT - b0) + 1;
        }
      }
    };
    struct Sums {                                           // of two cells
      float pn[2][NH], p0[2][NH], p1[2][NH];
    };
    int64_t slot_cur, slot_nxt;
    int nblk_cur, nblk_nxt;
    load_meta(t0, slot_cur, nblk_cur);
    uint32_t tt = 0;
    for (int64_t tile = t0; tile < ntiles; tile += TS, ++tt) {
      const uint32_t b = tt & 1;
      const int64_t cell0 = tile * kLC + 8 * g;
      load_meta(tile + TS, slot_nxt, nblk_nxt);
      auto load_sums = [&](int c2, Sums& s) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int64_t cell = cell0 + 2 * c2 + c;
          const int64_t slot = __shfl_sync(0xffffffffu, slot_cur, 2 * c2 + c);
          const int nb = __shfl_sync(0xffffffffu, nblk_cur, 2 * c2 + c);
#pragma unroll
          for (int h = 0; h < NH; ++h) s.pn[c][h] = s.p0[c][h] = s.p1[c][h] = 0.0f;
          if (own && cell < args.nc) {
            ldn<NH>(args.pnew + (size_t)cell * W + n0, s.pn[c]);
            if (nb > 0) ldn<NH>(args.part + (size_t)slot * W + n0, s.p0[c]);
            if (nb > 1) ldn<NH>(args.part + (size_t)(slot + 1) * W + n0, s.p1[c]);
          }
        }
      };
      Sums cur, nxt;
      load_sums(0, cur);
      const bool got = rwait(&bar[LB_TFULL + b], (tt >> 1) & 1, abort, args.status);
      if (!__all_sync(0xffffffffu, got)) break;
      tc_fence_after();
      const uint32_t trow = tmem + b * NH * 128 + lane_off + 32 * g;
#pragma unroll 1
      for (int c2 = 0; c2 < 4; ++c2) {
        float v[NH][8];
#pragma unroll
        for (int h = 0; h < NH; ++h) tmem_ld8(trow + h * 128 + 8 * c2, v[h]);
        if (c2 < 3) load_sums(c2 + 1, nxt);
        tmem_wait_ld();
        if (c2 == 3) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&bar[LB_TEMPTY + b]);
        }
        // centre and radius / sigma of the two cells
        float rad[2][NH];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int nb = __shfl_sync(0xffffffffu, nblk_cur, 2 * c2 + c);
          const int64_t slot = __shfl_sync(0xffffffffu, slot_cur, 2 * c2 + c);
          float s[NH], e[NH], sI[NH];
          auto add = [&](int h, float x) {
            const float y = x - e[h], u = s[h] + y;
            e[h] = (u - s[h]) - y;
            s[h] = u;
          };
#pragma unroll
          for (int h = 0; h < NH; ++h) {
            v[h][4 * c] += bias[h];
            s[h] = e[h] = sI[h] = 0.0f;
#pragma unroll
            for (int d = 1; d < 4; ++d) sI[h] += sq ? v[h][4 * c + d] * v[h][4 * c + d] : fabsf(v[h][4 * c + d]);
            add(h, cur.pn[c][h]);
            if (nb > 0) add(h, cur.p0[c][h]);
            if (nb > 1) add(h, cur.p1[c][h]);
          }
          if (own)
            for (int k = 2; k < nb; ++k) {
              float q[NH];
              ldn<NH>(args.part + (size_t)(slot + k) * W + n0, q);
#pragma unroll
              for (int h = 0; h < NH; ++h) add(h, q[h]);
            }
#pragma unroll
          for (int h = 0; h < NH; ++h) {
            const float tot = s[h] + sI[h];
            rad[c][h] = sq ? sqrtf(tot) : tot;
          }
        }
        // linearisation
        Lin L[2][NH];
        if (kink) {
          int pos[2][NH], nq = 0;
#pragma unroll
          for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int h = 0; h < NH; ++h) {
              const bool need = own && relu_clt_mixed(v[h][4 * c], rad[c][h]);
              const unsigned bm = __ballot_sync(0xffffffffu, need);
              pos[c][h] = need ? nq + __popc(bm & ((1u << lane) - 1u)) : -1;
              nq += __popc(bm);
              if (need) {
                qs[pos[c][h]] = v[h][4 * c];
                qs[kLQ + pos[c][h]] = rad[c][h];
              }
            }
          __syncwarp();
          for (int i = lane; i < nq; i += 32) {
            const Lin r = relu_clt(qs[i], qs[kLQ + i]);
            qs[i] = r.alpha;
            qs[kLQ + i] = r.beta;
            qs[2 * kLQ + i] = r.gamma;
          }
          __syncwarp();
#pragma unroll
          for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int h = 0; h < NH; ++h) {
              const float mu = v[h][4 * c];
              L[c][h].alpha = mu > 0.0f ? 1.0f : (mu == 0.0f ? 0.5f : 0.0f);
              L[c][h].beta = L[c][h].gamma = 0.0f;
              if (pos[c][h] >= 0) {
                L[c][h].alpha = qs[pos[c][h]];
                L[c][h].beta = qs[kLQ + pos[c][h]];
                L[c][h].gamma = qs[2 * kLQ + pos[c][h]];
              }
              L[c][h].center = fmaf(L[c][h].alpha, mu, L[c][h].beta);
            }
          __syncwarp();                                     // the queue is read before its next use
        } else {
#pragma unroll
          for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int h = 0; h < NH; ++h)
              L[c][h] = sq ? act_clt(args.act, v[h][4 * c], rad[c][h])
                           : relu_sound(v[h][4 * c], rad[c][h], 0.0f, false);
        }
        // the next layer's operands
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int64_t cell = cell0 + 2 * c2 + c;
          const bool valid = own && cell < args.nc;
          const size_t o = (size_t)cell * W + n0;
          float al[NH], ga[NH], ce[NH];
          int made = 0;
#pragma unroll
          for (int h = 0; h < NH; ++h) {
            al[h] = L[c][h].alpha;
            ga[h] = L[c][h].gamma;
            ce[h] = L[c][h].center;
            made += __popc(__ballot_sync(0xffffffffu, valid && ga[h] != 0.0f));
          }
          if (valid) {
            stn<NH>(args.AL + o, al);
            stn<NH>(args.GA + o, ga);
            if constexpr (LAST) {
              stn<NH>(args.A + o, ce);
#pragma unroll
              for (int d = 0; d < 3; ++d) {
                float x[NH];
#pragma unroll
                for (int h = 0; h < NH; ++h) x[h] = v[h][4 * c + 1 + d];
                stn<NH>(args.I + ((size_t)cell * 3 + d) * W + n0, x);
              }
            } else {
              const size_t q0 = (size_t)cell * 4 * W + n0;
              st_split<NH>(args.AH + q0, args.ALO + q0, ce);
#pragma unroll
              for (int d = 0; d < 3; ++d) {
                float x[NH];
#pragma unroll
                for (int h = 0; h < NH; ++h) x[h] = al[h] * v[h][4 * c + 1 + d];
                st_split<NH>(args.AH + q0 + (size_t)(d + 1) * W, args.ALO + q0 + (size_t)(d + 1) * W, x);
              }
            }
          }
          if (!LAST && lane == 0 && cell < args.nc && made > 0) atomicAdd(args.cnt_next + cell, made);
        }
        cur = nxt;
      }
      slot_cur = slot_nxt;
      nblk_cur = nblk_nxt;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (*abort)
    for (int i = 0; i < 1000; ++i) __nanosleep(1000);
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kCols) : "memory");
  }
}

template <int W, bool LAST>
isx_status launch_w(isx_inr inr, const RowsLayerArgs& a, const LayerMaps& maps, cudaStream_t st) {
  using S = LayerSmem<W>;
  const size_t smem = S::bytes();
  ISX_CUDA(cudaFuncSetAttribute(k_rows_layer<W, LAST>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int sms = inr->sms;
  const int64_t ntiles = (a.nc + kLC - 1) / kLC;
  int grid = (int)std::min<int64_t>(ntiles * S::NHALF, sms);
  grid -= grid % S::NHALF;
  k_rows_layer<W, LAST><<<grid, kLT, smem, st>>>(a, maps);
  ISX_LAUNCH_CHECK("k_rows_layer");
  return ISX_OK;
}

}  // namespace

isx_status launch_rows_layer(isx_inr inr, int layer, const RowsLayerArgs& a, const __nv_bfloat16* AHin,
                             const __nv_bfloat16* ALOin, cudaStream_t st) {
  const int w = inr->w;
  LayerMaps maps;
  std::memset(&maps, 0, sizeof(maps));
  ISX_TRY(tensor_map_bf16(&maps.ahi, AHin, w, 4 * (uint64_t)a.nc, 64, 128));
  ISX_TRY(tensor_map_bf16(&maps.alo, ALOin, w, 4 * (uint64_t)a.nc, 64, 128));
  const int nh = w >= 256 ? 2 : 1;
  for (int h = 0; h < nh; ++h) {
    // every nh-th row of W_j, from row h
    ISX_TRY(tensor_map_bf16(&maps.whi[h], inr->W_bf16[layer] + (size_t)h * w, w, w / nh, 64, std::min(w, 128), nh * w));
    ISX_TRY(tensor_map_bf16(&maps.wlo[h], inr->Wlo_bf16[layer] + (size_t)h * w, w, w / nh, 64, std::min(w, 128), nh * w));
  }
  const bool last = a.AH == nullptr;
  if (w == 512) return last ? launch_w<512, true>(inr, a, maps, st) : launch_w<512, false>(inr, a, maps, st);
  if (w == 256) return last ? launch_w<256, true>(inr, a, maps, st) : launch_w<256, false>(inr, a, maps, st);
  if (w == 128) return last ? launch_w<128, true>(inr, a, maps, st) : launch_w<128, false>(inr, a, maps, st);
  return last ? launch_w<64, true>(inr, a, maps, st) : launch_w<64, false>(inr, a, maps, st);
}

}  // namespace rows
}  // namespace isx
