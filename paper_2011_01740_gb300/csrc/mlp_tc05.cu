// mlp_tc05.cu -- ensemble forward on the 5th-generation tensor cores
// (tcgen05): accumulators in tensor memory, operands in shared memory.  Serves
// the screening forward and the per-member outputs.
//
// One CTA per SM serves one ensemble member: it stages that member's three
// 128 x 128 BF16 weight matrices in shared memory once, then walks its share of
// the 128-point tiles with four independent warpgroups, each with a tile, a
// 128-column accumulator and an mbarrier of its own.  Per tile:
//   layer 1 (2 -> 128)  FP32 FMAs, thread = point, GELU, BF16 into the
//                       warpgroup's activation tile (layout in tc05.cuh);
//   layers 2..4         one thread issues 8 tcgen05.mma (M = N = 128, K = 16,
//                       BF16 x BF16 -> FP32 in TMEM), commits to the mbarrier;
//                       the four warps read their 32 TMEM lanes (tcgen05.ld
//                       32x32b), add the bias, apply GELU and write the next
//                       activation tile;
//   layer 5 (128 -> 2)  folded into the layer-4 epilogue as FP32 dot products.
// The erf-GELU bounds the kernel: 512 per point and member, about 16 times the
// cycles of the tensor products.  One warpgroup per SM left the issue slots
// idle 47 % of the time, in the waits for its products and in the latencies of
// the erf chains; four fill each other's waits (224 KB of tiles, all 512 TMEM
// columns): 2048 x 2048 points, 4 members, with features, steepness and gate
// 13.55 ms -> 9.08 ms, the same bits.
// The per-member outputs [members][n][2] are reduced to mean / spread /
// period-1 probability by a second, elementwise kernel.
//
// Waits on the mbarrier are bounded; a wait that expires sets the error word
// (the outputs are then invalid), and the warpgroup runs on through waits that
// are bounded as well and waits once more before the TMEM is freed.
#include <cuda_bf16.h>

#include <cstdint>

#include "mlp.cuh"
#include "tc05.cuh"

namespace ens {
namespace mlp {

namespace {

using namespace tc05;
constexpr int kGroups = 4;                     // warpgroups, one tile each
constexpr int kTcThreads = kGroups * 128;
constexpr uint32_t kTcCols = kGroups * 128;
// shared memory map
constexpr size_t kSW = 0;                      // W2, W3, W4 (3 x 32 KB)
constexpr size_t kSA = kSW + 3 * kMatBytes;    // activation tiles (4 x 32 KB)
constexpr size_t kSF = kSA + kGroups * kMatBytes;   // fp32 W1[128][2], b2..b4[3][128]
constexpr size_t kSBar = kSF + (256 + 384) * sizeof(float);   // mbarriers, TMEM slot
constexpr size_t kTcSmem = kSBar + kGroups * 8 + 16;
static_assert(kTcSmem <= 232448, "shared memory of one CTA");
static_assert(oW5 % 8 == 0 && ob1 % 2 == 0, "vector loads of W5 and b1");

}  // namespace

struct TcArgs {
  int64_t n;
  int members;
  const float* x;            // [n][2]
  const float* master;       // [members][kP]
  const __nv_bfloat16* wbf;  // [members][kPS]
  float* out;                // [members][n][2]
  unsigned* error;           // set to 1 if a wait expired
};

// barrier of one warpgroup's 128 threads
__device__ __forceinline__ void group_sync(int g) { asm volatile("bar.sync %0, 128;" ::"r"(g + 1) : "memory"); }

// grid = (CTAs per member, members)
__global__ void __launch_bounds__(kTcThreads, 1) mlp_forward_tc05_kernel(TcArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, g = tid >> 7, row = tid & 127;
  const int m = blockIdx.y;
  const int64_t tiles = (a.n + kTile - 1) / kTile;
  float* sW1 = reinterpret_cast<float*>(smem + kSF);   // [128][2]
  float* sB = sW1 + 256;                               // b2..b4
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kSBar);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + kSBar + kGroups * 8);
  const uint32_t bar_a = smem_u32(bars + g);

  // stage this member's parameters
  const float* P = a.master + (int64_t)m * kP;
  const __nv_bfloat16* Pb = a.wbf + (int64_t)m * kPS;
  if (tid < 256) sW1[tid] = __bfloat162float(Pb[oW1 + tid]);
  if (tid < 384) sB[tid] = P[ob2 + (tid >> 7) * (ob3 - ob2) + (tid & 127)];
  stage3_tiles<kTcThreads>(smem + kSW, Pb + oW2, Pb + oW3, Pb + oW4);
  if (tid < kGroups) {
    bar_init(smem_u32(bars + tid));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc<kTcCols>(tslot);
  fence_to_mma();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = *tslot;
  const uint32_t acc = tmem + (uint32_t)(g * 128);
  const uint32_t lane0 = (uint32_t)((warp & 3) * 32) << 16;
  unsigned char* tile = smem + kSA + g * kMatBytes;
  const uint32_t sA = smem_u32(tile), sW = smem_u32(smem + kSW);
  const float2* b1 = reinterpret_cast<const float2*>(P + ob1);
  const uint32_t* w5 = reinterpret_cast<const uint32_t*>(Pb + oW5);   // BF16 pairs, rows 64 words apart
  const float b50 = P[ob5], b51 = P[ob5 + 1];
  uint32_t parity = 0;
  bool ok = true;

  // tile t goes to CTA t mod gridDim.x first: few tiles spread over the SMs
  for (int64_t t = blockIdx.x + (int64_t)g * gridDim.x; t < tiles; t += (int64_t)kGroups * gridDim.x) {
    const int64_t p = t * kTile + row;
    const bool live = p < a.n;
    const float x0 = live ? a.x[2 * p] : 0.f, x1 = live ? a.x[2 * p + 1] : 0.f;
    // layer 1: thread = point, 16 chunks of 8 features
#pragma unroll 1
    for (int kc = 0; kc < 16; ++kc) {
      float h[8];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 w = *reinterpret_cast<const float4*>(sW1 + 2 * (kc * 8 + 2 * j));
        const float2 b = b1[kc * 4 + j];
        h[2 * j] = fmaf(w.y, x1, fmaf(w.x, x0, b.x));
        h[2 * j + 1] = fmaf(w.w, x1, fmaf(w.z, x0, b.y));
        gelu2(h[2 * j], h[2 * j + 1]);
      }
      store_bf16x8(tile, row, kc * 8, h);
    }
    float o0 = b50, o1 = b51;
#pragma unroll 1
    for (int l = 0; l < 3; ++l) {
      fence_to_mma();
      group_sync(g);
      fence_after_sync();
      if (row == 0) {
        mma_128<false, false>(acc, sA, sW + l * (uint32_t)kMatBytes);
        mma_commit(bar_a);
      }
      ok &= bar_wait(bar_a, parity);
      parity ^= 1u;
      fence_after_sync();
      const float* bl = sB + l * 128;
#pragma unroll 1
      for (int c = 0; c < 4; ++c) {
        float v[32];
        tmem_ld32(acc + lane0 + (uint32_t)(c * 32), v);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float4 b = *reinterpret_cast<const float4*>(bl + c * 32 + 4 * q);
          bias_gelu2(v[4 * q], v[4 * q + 1], b.x, b.y);
          bias_gelu2(v[4 * q + 2], v[4 * q + 3], b.z, b.w);
        }
        if (l < 2) {
#pragma unroll
          for (int q = 0; q < 4; ++q) store_bf16x8(tile, row, c * 32 + q * 8, v + q * 8);
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint4 u0 = *reinterpret_cast<const uint4*>(w5 + c * 16 + q * 4);
            const uint4 u1 = *reinterpret_cast<const uint4*>(w5 + 64 + c * 16 + q * 4);
            const uint32_t w0[4] = {u0.x, u0.y, u0.z, u0.w}, w1[4] = {u1.x, u1.y, u1.z, u1.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              // round to BF16 like the activations of the hidden layers
              const uint32_t hh = pack_bf16x2(v[q * 8 + 2 * j], v[q * 8 + 2 * j + 1]);
              o0 = fmaf(bf16_lo(hh), bf16_lo(w0[j]), o0);
              o1 = fmaf(bf16_lo(hh), bf16_lo(w1[j]), o1);
              o0 = fmaf(bf16_hi(hh), bf16_hi(w0[j]), o0);
              o1 = fmaf(bf16_hi(hh), bf16_hi(w1[j]), o1);
            }
          }
        }
      }
    }
    if (live) {
      a.out[((int64_t)m * a.n + p) * 2] = o0;
      a.out[((int64_t)m * a.n + p) * 2 + 1] = o1;
    }
  }
  if (!ok) {
    bar_wait(bar_a, parity ^ 1u);   // the last product issued
    atomicOr(a.error, 1u);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  fence_after_sync();
  if (warp == 0) tmem_dealloc<kTcCols>(tmem);
}

// mean / population spread of output 0 and mean sigmoid of output 1 over members
__global__ void mlp_reduce_members_kernel(int64_t n, int members, const float* out, float* mean, float* stdv,
                                          float* p1) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float s = 0.f, p = 0.f;
    for (int m = 0; m < members; ++m) {
      s += out[((int64_t)m * n + i) * 2];
      p += 1.0f / (1.0f + __expf(-out[((int64_t)m * n + i) * 2 + 1]));
    }
    const float mu = s / members;
    float s2 = 0.f;
    for (int m = 0; m < members; ++m) {
      const float d = out[((int64_t)m * n + i) * 2] - mu;
      s2 += d * d;
    }
    mean[i] = mu;
    stdv[i] = sqrtf(s2 / members);
    p1[i] = p / members;
  }
}

cudaError_t launch_forward_tc05(int64_t n, int members, const float* x, const float* master, const __nv_bfloat16* wbf,
                                float* out, unsigned* error, int sms, cudaStream_t s) {
  // once per process (thread-safe static initialisation)
  static const cudaError_t attr = cudaFuncSetAttribute(mlp_forward_tc05_kernel,
                                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmem);
  if (attr != cudaSuccess) return attr;
  if (n == 0) return cudaSuccess;
  TcArgs a{};
  a.n = n;
  a.members = members;
  a.x = x;
  a.master = master;
  a.wbf = wbf;
  a.out = out;
  a.error = error;
  const int64_t tiles = (n + kTile - 1) / kTile;
  const int64_t per = sms / members > 1 ? sms / members : 1;   // one CTA per SM in all
  mlp_forward_tc05_kernel<<<dim3((unsigned)(tiles < per ? tiles : per), members), kTcThreads, kTcSmem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_screen_tc05(int64_t n, int members, const float* x, const float* master, const __nv_bfloat16* wbf,
                               float* out, unsigned* error, float* mean, float* stdv, float* p1, int sms,
                               cudaStream_t s) {
  cudaError_t e = launch_forward_tc05(n, members, x, master, wbf, out, error, sms, s);
  if (e != cudaSuccess || n == 0) return e;
  int64_t blocks = (n + 255) / 256;
  blocks = blocks > 8192 ? 8192 : blocks;
  mlp_reduce_members_kernel<<<(unsigned)blocks, 256, 0, s>>>(n, members, out, mean, stdv, p1);
  return cudaGetLastError();
}

}  // namespace mlp
}  // namespace ens
