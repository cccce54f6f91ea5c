// Float32 matrix tile on the CUDA cores, shared by the point evaluation (mesh.cu) and the float32
// bound path (bound_fp32.cu): Y[p][n] = sum_k A[p][k] W[n][k] for the P rows (points) a CTA holds and
// all w neurons, every output one fused multiply-add chain over k = 0 .. w - 1 in that order.
//
// What bounds it: the FP32 FMA rate (128 lanes / SM).  So everything else is kept off the issue slots:
//  - the row operand of the whole K extent sits in shared memory k-major, A[k][P], and a thread owns
//    an 8-row x TN-neuron register tile, so 8 + TN values loaded (16-byte loads, conflict-free or
//    broadcast) feed 8 TN multiply-adds;
//  - two adjacent neurons share one 64-bit accumulator (fma.rn.f32x2: two IEEE fused multiply-adds
//    per instruction, the same results bit for bit as two fmaf);
//  - W^T streams through three shared-memory stages of KB rows with cp.async, one block barrier per
//    stage; the stream runs on across layers.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace isx {
namespace sgemm {

constexpr int kTM = 8;                 // rows of a thread's tile: 4 of each half of the CTA's P rows
constexpr int kStages = 3;

__device__ __forceinline__ uint64_t pack2(float x, float y) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ void cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Launch shape of one tile kernel: TN neurons per thread, P rows per CTA (a multiple of 8), KB rows of
// W^T per stage (a divisor of w).  Threads: one per (8 rows, TN neurons); thread t < threads() owns
// row group t % (P / 8) and neuron group t / (P / 8).
struct Shape {
  int tn, P, KB;
  __host__ __device__ int threads(int w) const { return (w / tn) * (P / kTM); }
  __host__ __device__ size_t smem(int w) const { return ((size_t)w * P + (size_t)kStages * KB * w) * sizeof(float); }
};

// The W^T stream of a CTA: stages of KB rows, taken from one or several w x w matrices in turn.
struct Stream {
  float* Ws;                           // [kStages][KB * w]
  int w, KB;
  int64_t left;                        // stages still to load
  int slot = 0;                        // ring slot of the next one
  // loads the next stage of the stream from `src` (its KB rows) and commits a group, also when none is left
  __device__ __forceinline__ void load(const float* src) {
    if (left > 0) {
      float* dst = Ws + (size_t)slot * KB * w;
      for (int i = threadIdx.x * 4; i < KB * w; i += blockDim.x * 4) cp16(dst + i, src + i);
    }
    cp_commit();
    --left;
    slot = slot == kStages - 1 ? 0 : slot + 1;
  }
};

// acc[i][c]: row i of the thread's 8, neuron pair c of its TN / 2.  Row i < 4 is row 4 pg + i of the
// CTA, row i >= 4 is P / 2 + 4 pg + i - 4; pair c covers neurons neuron(c), neuron(c) + 1.
template <int TN>
struct Tile {
  uint64_t acc[kTM][TN / 2];
  __device__ __forceinline__ static int neuron(int c, int ng, int w) { return (c >> 1) * (w / (TN / 4)) + 4 * ng + 2 * (c & 1); }
  __device__ __forceinline__ static int row(int i, int pg, int P) { return (i >> 2) * (P >> 1) + 4 * pg + (i & 3); }

  // KB steps of k: A the stage's first row of the k-major operand, Ws the stage
  __device__ __forceinline__ void stage(const float* A, const float* Ws, int P, int w, int KB, int pg, int ng) {
    const float* a0 = A + 4 * pg;
    const float* a1 = a0 + (P >> 1);
    const float* bp = Ws + 4 * ng;
    const int cs = w / (TN / 4);
#pragma unroll 8
    for (int k = 0; k < KB; ++k) {
      const float4 x = *reinterpret_cast<const float4*>(a0 + k * P), y = *reinterpret_cast<const float4*>(a1 + k * P);
      const float av[kTM] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
      ulonglong2 b[TN / 4];
#pragma unroll
      for (int c = 0; c < TN / 4; ++c) b[c] = *reinterpret_cast<const ulonglong2*>(bp + k * w + c * cs);
#pragma unroll
      for (int i = 0; i < kTM; ++i) {
        const uint64_t aa = pack2(av[i], av[i]);
#pragma unroll
        for (int c = 0; c < TN / 4; ++c) {
          acc[i][2 * c] = fma2(aa, b[c].x, acc[i][2 * c]);
          acc[i][2 * c + 1] = fma2(aa, b[c].y, acc[i][2 * c + 1]);
        }
      }
    }
  }

  // The same with the weights of k times u[k] (rows i < 4) or v[k] (rows i >= 4), rounded before the
  // multiply-add: a quarter more instructions.  KB is a multiple of 4.
  __device__ __forceinline__ void stage_scaled(const float* A, const float* Ws, int P, int w, int KB, int pg, int ng,
                                               const float* __restrict__ u, const float* __restrict__ v) {
    const float* a0 = A + 4 * pg;
    const float* a1 = a0 + (P >> 1);
    const float* bp = Ws + 4 * ng;
    const int cs = w / (TN / 4);
#pragma unroll 2
    for (int k0 = 0; k0 < KB; k0 += 4) {
      const float4 u4 = *reinterpret_cast<const float4*>(u + k0), v4 = *reinterpret_cast<const float4*>(v + k0);
      const float uk[4] = {u4.x, u4.y, u4.z, u4.w}, vk[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const int k = k0 + kk;
        const float4 x = *reinterpret_cast<const float4*>(a0 + k * P), y = *reinterpret_cast<const float4*>(a1 + k * P);
        const float av[kTM] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
        const uint64_t uu = pack2(uk[kk], uk[kk]), vv = pack2(vk[kk], vk[kk]);
#pragma unroll
        for (int c = 0; c < TN / 4; ++c) {
          const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(bp + k * w + c * cs);
          const uint64_t b0[2] = {mul2(uu, b.x), mul2(uu, b.y)}, b1[2] = {mul2(vv, b.x), mul2(vv, b.y)};
#pragma unroll
          for (int i = 0; i < kTM; ++i) {
            const uint64_t aa = pack2(av[i], av[i]);
#pragma unroll
            for (int q = 0; q < 2; ++q) acc[i][2 * c + q] = fma2(aa, i < 4 ? b0[q] : b1[q], acc[i][2 * c + q]);
          }
        }
      }
    }
  }
};

}  // namespace sgemm
}  // namespace isx
