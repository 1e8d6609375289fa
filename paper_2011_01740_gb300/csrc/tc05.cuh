// tc05.cuh -- 5th-generation tensor-core (tcgen05) building blocks shared by
// the surrogate-network kernels: the no-swizzle shared-memory operand layout
// and its descriptors, the BF16 MMA with FP32 accumulation in tensor memory,
// the commit to an mbarrier, a bounded mbarrier wait, tensor-memory loads and
// stores.
//
// Operand layout: a 128 x 128 BF16 matrix X as 8-row x 16-byte core matrices,
// core (r/8, c/8) at byte ((r/8) * 16 + c/8) * 128.  One tile in this layout
// serves as an operand in either direction, so no product needs a transposed
// copy:
//   K-major   rows r are the M (or N) index, columns c the K index: cores
//             128 B apart along K (leading byte offset), 2048 B along M / N
//             (stride byte offset); a K = 16 step advances 256 B;
//   MN-major  columns c are the M (or N) index, rows r the K index (the
//             product takes X^T): 8-element groups of M / N 128 B apart (stride
//             byte offset), 8-row groups of K 2048 B (leading byte offset); a
//             K = 16 step advances 4096 B.
#pragma once

#include <cuda_bf16.h>

#include <cstdint>

#include "mlp.cuh"

namespace ens {
namespace mlp {
namespace tc05 {

constexpr size_t kMatBytes = (size_t)H * H * sizeof(__nv_bfloat16);  // 32 KB
constexpr uint32_t kWaitLimit = 1u << 20;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// byte offset of element (r, k) of a 128 x 128 BF16 operand in core-matrix layout
__device__ __forceinline__ uint32_t core_off(int r, int k) {
  return (uint32_t)(((r >> 3) * 16 + (k >> 3)) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

// shared-memory matrix descriptor: start >> 4, leading and stride byte
// offsets, descriptor version 1 (bit 46), no swizzle
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)(lbo >> 4) << 16;
  d |= (uint64_t)(sbo >> 4) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// instruction descriptor, kind::f16: D = F32, A = B = BF16, N = 128 (bits
// 17-22 = N >> 3), M = 128 (bits 24-28 = M >> 4); A, B MN-major: bits 15, 16
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
constexpr uint32_t kAmn = 1u << 15, kBmn = 1u << 16;

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

// D (TMEM) = A B^T over K = 128, eight K = 16 steps, with the tiles at sa and
// sb read K-major or, where the flag is set, MN-major; added onto D when acc.
// One thread issues.
template <bool A_MN, bool B_MN>
__device__ __forceinline__ void mma_128(uint32_t d_tmem, uint32_t sa, uint32_t sb, bool acc = false) {
  constexpr uint32_t idesc = kIdesc | (A_MN ? kAmn : 0u) | (B_MN ? kBmn : 0u);
#pragma unroll
  for (int k = 0; k < 8; ++k)
    mma_bf16(d_tmem, A_MN ? make_desc(sa + k * 4096, 2048, 128) : make_desc(sa + k * 256, 128, 2048),
             B_MN ? make_desc(sb + k * 4096, 2048, 128) : make_desc(sb + k * 256, 128, 2048), idesc, acc || k > 0 ? 1u : 0u);
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// bounded wait for the mbarrier phase `parity`; returns false on expiry
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity) {
  for (uint32_t it = 0; it < kWaitLimit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

// the transposing counterpart for stores to memory: the warp's 32 lanes x 32
// columns as four m16n8-style fragments per 16 lanes (16x256b): v[16 h + 4 j +
// 2 u + e] is row 16 h + 8 u + lane / 4, column 8 j + 2 (lane % 4) + e, so a quad
// of lanes holds 32 contiguous bytes of a row
__device__ __forceinline__ void tmem_ld_frag32(uint32_t taddr, float* v) {
  uint32_t r[32];
#pragma unroll
  for (int h = 0; h < 2; ++h)
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[16 * h + 0]), "=r"(r[16 * h + 1]), "=r"(r[16 * h + 2]), "=r"(r[16 * h + 3]), "=r"(r[16 * h + 4]),
          "=r"(r[16 * h + 5]), "=r"(r[16 * h + 6]), "=r"(r[16 * h + 7]), "=r"(r[16 * h + 8]), "=r"(r[16 * h + 9]),
          "=r"(r[16 * h + 10]), "=r"(r[16 * h + 11]), "=r"(r[16 * h + 12]), "=r"(r[16 * h + 13]),
          "=r"(r[16 * h + 14]), "=r"(r[16 * h + 15])
        : "r"(taddr + ((uint32_t)(16 * h) << 16)));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

// this thread's 32 values into 32 columns of its TMEM lane, complete on return
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const float* v) {
  uint32_t r[32];
#pragma unroll
  for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(v[j]);
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
      "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
      "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const float* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr),
      "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
      "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7]))
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// TMEM allocation of COLS columns by the calling warp, its address in *slot
template <uint32_t COLS>
__device__ __forceinline__ void tmem_alloc(uint32_t* slot) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(COLS));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
template <uint32_t COLS>
__device__ __forceinline__ void tmem_dealloc(uint32_t tmem) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(COLS));
}

__device__ __forceinline__ void bar_init(uint32_t bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
}

// eight floats as BF16 into the 16 bytes of row r, columns k .. k + 7 of a tile
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 h2 = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h2);
}
__device__ __forceinline__ void store_bf16x8(unsigned char* base, int r, int k, const float* v) {
  *reinterpret_cast<uint4*>(base + core_off(r, k)) =
      make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]), pack_bf16x2(v[6], v[7]));
}

// the two BF16 halves of a word as floats
__device__ __forceinline__ float bf16_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }

// Stage three row-major 128 x 128 BF16 matrices M_i[r][c] as tiles at
// dst + i * kMatBytes with T threads.  Thread index bits: 0-2 the row within a
// core matrix, 3-6 the 16-byte chunk of the row, 7 and up the row group; a
// phase of 8 threads then writes one whole 128-byte core matrix (no bank
// conflict) and a warp reads 8 rows x 64 contiguous bytes.  All loads of a
// thread are issued before its stores.
template <int T>
__device__ __forceinline__ void stage3_tiles(unsigned char* dst, const __nv_bfloat16* M0, const __nv_bfloat16* M1,
                                             const __nv_bfloat16* M2) {
  constexpr int kIt = H * (H / 8) / T;
  const __nv_bfloat16* Ms[3] = {M0, M1, M2};
  uint4 v[3][kIt];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
#pragma unroll
    for (int it = 0; it < kIt; ++it) {
      const int idx = it * T + (int)threadIdx.x;
      const int n = (idx >> 7) * 8 + (idx & 7), kc = (idx >> 3) & 15;
      v[i][it] = *reinterpret_cast<const uint4*>(Ms[i] + n * H + kc * 8);
    }
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
#pragma unroll
    for (int it = 0; it < kIt; ++it) {
      const int idx = it * T + (int)threadIdx.x;
      const int n = (idx >> 7) * 8 + (idx & 7), kc = (idx >> 3) & 15;
      *reinterpret_cast<uint4*>(dst + i * kMatBytes + core_off(n, kc * 8)) = v[i][it];
    }
  }
}

__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// make shared-memory writes of the generic proxy visible to the tensor cores
// and order them against the thread barrier that follows
__device__ __forceinline__ void fence_to_mma() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

}  // namespace tc05
}  // namespace mlp
}  // namespace ens
