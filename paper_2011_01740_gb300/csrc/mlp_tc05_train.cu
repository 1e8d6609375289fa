// mlp_tc05_train.cu -- loss and gradient of one training batch of the surrogate
// network on the 5th-generation tensor cores (tcgen05): one kernel runs the
// forward and the input gradients of a tile, a second the weight gradients.
//
// The batch is cut into up to 8 slices of a.rows samples (the partial gradients
// that Adam sums in order) and each slice into 128-sample tiles.
//
// mlp_step_tc05_kernel: grid = (CTAs, members); a CTA walks every gridDim.x-th
// tile for its member.  512 threads: warp w owns samples (TMEM lanes) 32 (w % 4)
// .. + 31 and columns 32 (w / 4) .. + 31 of every epilogue, so a thread handles
// one sample and 32 features.  Between the samples and the operands of the
// weight gradients everything stays on the SM: W_2..W_4 and the running
// activation / gradient tiles in shared memory (BF16, layout in tc05.cuh),
// gelu'(z_1..z_3) in FP32 in TMEM beside the accumulator, gelu'(z_4) in
// registers.  The products, each 128 x 128 x 128:
//   forward       Z_l[s][out] = H_{l-1}[s][in] W_l[out][in]      l = 2..4
//   input grad.   G[s][in] = DZ_l[s][out] W_l[out][in]           l = 4..2
// Both read W_l as staged, K-major or MN-major.  Every tile goes to memory as
// it lies (32 KB bulk copies) for the second kernel, with the FP32 dz_l and
// gelu(z_4) that the biases and the 2-wide layers need unrounded: those in
// blocks of 32 samples, four features of a sample together and the threads of
// a warp in a row, so that both the stores here and the column sums there are
// contiguous (as rows of 128 floats each store took 32 lines: 79 us for 64
// tiles and four members against 58).
//
// mlp_wgrad_tc05_kernel: grid = (members, 4, slices); y = 0..2: layers 2..4,
//   dW_l[out][in] = sum_s DZ_l[s][out] H_{l-1}[s][in],
// a slice's tiles bulk-loaded and multiplied MN-major x MN-major, accumulating in
// TMEM, while other warps sum the bias gradient; y = 3: layers 1 and 5 in FP32.
// The FP32 sums run in sample order, one thread per feature and half; their
// blocks stream through rings in shared memory (33 us with plain loads, 23 so,
// near the memory rate: 134 MB of tiles and blocks).
// BF16 operands and FP32 accumulation as in the mma.sync kernels of mlp.cu.
//
// What bounds it: 512 erf-GELUs with derivative per sample and member, about
// 11 us of issue per tile, and for a batch of few tiles one tile's chain of six
// products and epilogues.  Batch 8,192, 4 members: 58 us here, 23 us for the
// weight gradients and 6 us for Adam, against 250 us for the gather, forward,
// transposition, backward and weight-gradient kernels this replaces, which
// passed z, gelu' and dz through memory in FP32; 1,000 samples: loss, gradient
// and predictions 187 -> 100 us.  All sums keep their order, so the gradients and
// the trained weights are the same bits.
//
// A wait that expires sets the error word; the CTA runs on through bounded
// waits (its results are invalid), waits for the last products and copies and
// frees its tensor memory.
#include <cuda_bf16.h>

#include <cstdint>

#include "mlp.cuh"
#include "tc05.cuh"

namespace ens {
namespace mlp {

namespace {

using namespace tc05;
constexpr int kT = 512;

__host__ __device__ constexpr int64_t w_of(int l) { return l == 2 ? oW2 : l == 3 ? oW3 : oW4; }
__host__ __device__ constexpr int64_t b_of(int l) { return l == 1 ? ob1 : l == 2 ? ob2 : l == 3 ? ob3 : ob4; }
static_assert(kP % 2 == 0 && ob1 % 2 == 0 && ob2 % 2 == 0 && ob3 % 2 == 0 && ob4 % 2 == 0 && oW2 % 2 == 0 &&
                  oW3 % 2 == 0 && oW4 % 2 == 0,
              "8-byte bias loads and gradient stores");
static_assert(kPS % 8 == 0 && oW1 % 8 == 0 && oW2 % 8 == 0 && oW3 % 8 == 0 && oW4 % 8 == 0 && oW5 % 8 == 0,
              "16-byte weight loads");

// step kernel, shared memory: W_2..W_4, a ring of four tiles (h_1, h_2, h_3, dz_4,
// dz_3, dz_2 of one tile after the other), barrier and TMEM slot
constexpr size_t kRing = 3 * kMatBytes, kBar = 7 * kMatBytes;
constexpr size_t kStepSmem = kBar + 32;
// TMEM columns: the accumulator, then gelu'(z_l) of layers 1..3
constexpr uint32_t kAcc = 0, kCols = 512;
__device__ __forceinline__ constexpr uint32_t gelu_cols(int l) { return (uint32_t)(128 * l); }
// weight-gradient kernel: rings of kDepth blocks of 32 samples for each group of
// 128 threads.  Layers 2..4: two slots of (h, dz) tiles before two rings; layers
// 1 and 5: four rings, the pairs (x or dout) of their samples, reduction scratch.
// Barriers and the TMEM slot last.
constexpr int kDepth = 3;
constexpr size_t kBlockBytes = (size_t)kBlock * sizeof(float), kRingBytes = kDepth * kBlockBytes;
constexpr size_t kPairs = 4 * kRingBytes, kPart = kPairs + 4 * kDepth * 256;
constexpr size_t kGBar = 4 * kMatBytes + 2 * kRingBytes;
constexpr size_t kGradSmemTc = kGBar + (5 + 4 * kDepth) * 8 + 16;
static_assert(kPart + 2 * 768 * sizeof(float) <= kGBar && kBlockBytes % 16 == 0, "weight-gradient layout");
static_assert(kStepSmem <= 232448 && kGradSmemTc <= 232448, "shared memory of one CTA");

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// tile in shared memory -> memory (one thread); the group is committed
__device__ __forceinline__ void bulk_store_tile(void* dst, uint32_t src) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src),
               "r"((uint32_t)kMatBytes)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// memory -> shared memory, counted on the mbarrier (one thread)
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
      "r"(bytes), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void expect_bytes(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// a thread's 32 features (columns c0 ..) of one sample into its block: four
// features together, [8][4 column groups][32 samples][4], the eight planes 516
// floats apart so that the column sums read 32 different banks
__device__ __forceinline__ void store_block(float* block, int c0, int lane, const float* v) {
#pragma unroll
  for (int q = 0; q < 8; ++q)
    reinterpret_cast<float4*>(block)[q * (kBlock / 32) + c0 + lane] =
        make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
}

// samples of a tile: its first one and the end of its slice
__device__ __forceinline__ void tile_range(const TrainTcArgs& a, int64_t t, int64_t& p0, int64_t& end) {
  const int64_t per = (a.rows + kTile - 1) / kTile, slice = t / per;
  p0 = slice * a.rows + (t - slice * per) * kTile;
  end = (slice + 1) * a.rows < a.n ? (slice + 1) * a.rows : a.n;
}

}  // namespace

__global__ void __launch_bounds__(kT, 1) mlp_step_tc05_kernel(TrainTcArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int s = (warp & 3) * 32 + lane, c0 = (warp >> 2) * 32;   // sample (TMEM lane), first column
  const int m = blockIdx.y;
  const uint32_t bar = smem_u32(smem + kBar);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + kBar + 8);
  float* red = reinterpret_cast<float*>(smem + kBar + 16);   // loss sums of warps 0..3
  const float* P = a.master + (int64_t)m * kP;
  const __nv_bfloat16* Pb = a.wbf + (int64_t)m * kPS;

  stage3_tiles<kT>(smem, Pb + w_of(2), Pb + w_of(3), Pb + w_of(4));
  if (tid == 0) {
    bar_init(bar);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc<kCols>(tslot);
  fence_to_mma();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = *tslot;
  const uint32_t mine = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0;   // this thread's lane and columns
  const uint32_t sW = smem_u32(smem), kM = (uint32_t)kMatBytes;
  uint32_t parity = 0, stage = 0;
  bool ok = true;
  float loss = 0.f;
  const float inv_n = 1.0f / (float)a.n;

  // A stage: every thread has written its part of ring tile stage % 4; one
  // thread issues the tile's product with W_l (FWD: K-major, else MN-major)
  // and its copy to memory.  The ring tile written next was stored three
  // stages ago: its copy has been read out once at most two groups are left.
  auto issue = [&](int l, bool fwd, __nv_bfloat16* copy) {
    fence_to_mma();
    if (tid == 0) asm volatile("cp.async.bulk.wait_group.read 2;" ::: "memory");
    __syncthreads();
    fence_after_sync();
    if (tid == 0) {
      const uint32_t src = sW + (uint32_t)kRing + (stage & 3) * kM, w = sW + (uint32_t)(l - 2) * kM;
      if (fwd) mma_128<false, false>(tmem + kAcc, src, w);
      else mma_128<false, true>(tmem + kAcc, src, w);
      mma_commit(bar);
      bulk_store_tile(copy, src);
    }
    ++stage;
  };
  auto wait = [&] {
    ok &= bar_wait(bar, parity);
    parity ^= 1u;
    fence_after_sync();
  };
  auto ring = [&] { return smem + kRing + (stage & 3) * kMatBytes; };

  for (int64_t t = blockIdx.x; t < a.tiles; t += gridDim.x) {
    int64_t p0, end;
    tile_range(a, t, p0, end);
    if (p0 >= end) continue;   // block-uniform
    const int64_t p = p0 + s;
    const bool live = p < end;
    const int64_t src = live ? (a.perm ? (int64_t)a.perm[p] : p) : 0;
    const float x0 = live ? a.x[2 * src] : 0.f, x1 = live ? a.x[2 * src + 1] : 0.f;
    __nv_bfloat16* copy = a.tile + ((int64_t)m * a.tiles + t) * 6 * H * H;   // h_1, h_2, h_3, dz_4, dz_3, dz_2
    // this warp's blocks of dz_1..dz_4 and gelu(z_4)
    float* blocks = a.block + (((int64_t)m * a.tiles + t) * 5 * 4 + (warp & 3)) * kBlock;
    float v[32], g[32];
    // layer 1 in FP32, eight features at a time; h of samples past the end is 0
    {
      const uint4* w1 = reinterpret_cast<const uint4*>(Pb + oW1 + 2 * c0);
      const float2* b1 = reinterpret_cast<const float2*>(P + ob1 + c0);
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        float h[8], gq[8];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const uint4 w = w1[2 * q + u];
          const float2 ba = b1[4 * q + 2 * u], bb = b1[4 * q + 2 * u + 1];
          const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
          const float b[4] = {ba.x, ba.y, bb.x, bb.y};
#pragma unroll
          for (int j = 0; j < 4; j += 2) {
            const int c = 4 * u + j;
            gelu_and_grad2(df::f2(fmaf(bf16_hi(ww[j]), x1, fmaf(bf16_lo(ww[j]), x0, b[j])),
                                  fmaf(bf16_hi(ww[j + 1]), x1, fmaf(bf16_lo(ww[j + 1]), x0, b[j + 1]))),
                           h[c], h[c + 1], gq[c], gq[c + 1]);
            if (!live) h[c] = h[c + 1] = 0.f;
          }
        }
        store_bf16x8(ring(), s, c0 + 8 * q, h);
        tmem_st8(mine + gelu_cols(1) + 8 * q, gq);
      }
    }
    // layers 2..4
#pragma unroll 1
    for (int l = 2; l <= 4; ++l) {
      issue(l, true, copy + (l - 2) * H * H);
      float2 b[16];   // the bias, loaded while the product runs
#pragma unroll
      for (int j = 0; j < 16; ++j) b[j] = reinterpret_cast<const float2*>(P + b_of(l) + c0)[j];
      wait();
      tmem_ld32(mine + kAcc, v);
#pragma unroll
      for (int j = 0; j < 16; ++j)
        gelu_and_grad2(df::add_f(df::f2(v[2 * j], v[2 * j + 1]), df::f2(b[j].x, b[j].y)), v[2 * j], v[2 * j + 1],
                       g[2 * j], g[2 * j + 1]);
      if (l < 4) {
        if (!live) {
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = 0.f;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) store_bf16x8(ring(), s, c0 + 8 * q, v + 8 * q);
        tmem_st32(mine + gelu_cols(l), g);
      }
    }
    store_block(blocks + 4 * 4 * kBlock, c0, lane, v);
    // v = gelu(z_4), g = gelu'(z_4).  Layer 5: the outputs read the BF16-rounded
    // activations.  Each half of the features is one running sum, begun by its
    // first column group and continued by the second; the partial sums pass
    // through the ring tile that dz_4 takes next
    const uint4* w5 = reinterpret_cast<const uint4*>(Pb + oW5 + c0);   // rows 16 words of 16 bytes apart
    float2* so = reinterpret_cast<float2*>(ring());   // [2][2][128]: after the half's first group, its second
    const int half = warp >> 3;
    const bool second = (warp >> 2) & 1;
    float o0 = half ? 0.f : P[ob5], o1 = half ? 0.f : P[ob5 + 1];
#pragma unroll 1
    for (int turn = 0; turn < 2; ++turn) {
      if (second == (turn == 1)) {
        if (second) {
          const float2 q = so[half * 128 + s];
          o0 = q.x;
          o1 = q.y;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint4 ua = w5[q], ub = w5[16 + q];
          const uint32_t wa[4] = {ua.x, ua.y, ua.z, ua.w}, wb[4] = {ub.x, ub.y, ub.z, ub.w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint32_t hh = pack_bf16x2(v[8 * q + 2 * j], v[8 * q + 2 * j + 1]);
            o0 = fmaf(bf16_hi(hh), bf16_hi(wa[j]), fmaf(bf16_lo(hh), bf16_lo(wa[j]), o0));
            o1 = fmaf(bf16_hi(hh), bf16_hi(wb[j]), fmaf(bf16_lo(hh), bf16_lo(wb[j]), o1));
          }
        }
        so[(turn * 2 + half) * 128 + s] = make_float2(o0, o1);
      }
      __syncthreads();
    }
    float d0 = 0.f, d1 = 0.f;
    {
      const float2 qa = so[256 + s], qb = so[384 + s];
      o0 = qa.x + qb.x;
      o1 = qa.y + qb.y;
      if (live) {
        const float y0 = a.y[2 * src], y1 = a.y[2 * src + 1];
        d0 = 2.0f * (o0 - y0) * inv_n;
        d1 = (1.0f / (1.0f + __expf(-o1)) - y1) * inv_n;
        if (c0 == 0) {
          loss += (o0 - y0) * (o0 - y0) + fmaxf(o1, 0.f) - o1 * y1 + log1pf(__expf(-fabsf(o1)));
          reinterpret_cast<float2*>(a.dout)[(int64_t)m * pair_rows(a.n) + p] = make_float2(d0, d1);
          if (m == 0) reinterpret_cast<float2*>(a.xb)[p] = make_float2(x0, x1);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint4 ua = w5[q], ub = w5[16 + q];
      const uint32_t wa[4] = {ua.x, ua.y, ua.z, ua.w}, wb[4] = {ub.x, ub.y, ub.z, ub.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {   // dz_4, 0 for samples past the end
        const int c = 8 * q + 2 * j;
        v[c] = live ? fmaf(d0, bf16_lo(wa[j]), d1 * bf16_lo(wb[j])) * g[c] : 0.f;
        v[c + 1] = live ? fmaf(d0, bf16_hi(wa[j]), d1 * bf16_hi(wb[j])) * g[c + 1] : 0.f;
      }
    }
    __syncthreads();   // the partial outputs have been read
    // input gradients of layers 4..2
#pragma unroll 1
    for (int l = 4; l >= 2; --l) {
#pragma unroll
      for (int q = 0; q < 4; ++q) store_bf16x8(ring(), s, c0 + 8 * q, v + 8 * q);
      issue(l, false, copy + (7 - l) * H * H);
      store_block(blocks + (l - 1) * 4 * kBlock, c0, lane, v);
      tmem_ld32(mine + gelu_cols(l - 1), g);
      wait();
      tmem_ld32(mine + kAcc, v);
#pragma unroll
      for (int j = 0; j < 32; ++j) v[j] = live ? v[j] * g[j] : 0.f;   // dz_{l-1}
    }
    store_block(blocks, c0, lane, v);
  }
  if (tid == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  loss = warp_sum(loss);
  if (warp < 4 && lane == 0) red[warp] = loss;
  if (!ok) {
    bar_wait(bar, parity ^ 1u);   // the last product issued
    atomicOr(a.error, 1u);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  fence_after_sync();
  if (tid == 0) atomicAdd(&a.loss[m], (red[0] + red[1]) + (red[2] + red[3]));
  if (warp == 0) tmem_dealloc<kCols>(tmem);
}

namespace {

// A group of 128 threads (thread = feature f) walks the 32-sample blocks
// quarter(0), quarter(1), .. of one array over a slice's rows [lo, hi), in
// order: use(d, row in the block, pairs of the block's rows).  Blocks arrive through a ring of
// kDepth; pairs (may be null) are the slice's [rows][2] x or dout.  After a wait that
// expired a thread waits no more, and the one that copies starts no copy on that
// barrier again and ends with a wait for those under way.
template <class Quarter, class Use>
__device__ __forceinline__ bool walk_blocks(int grp, const float* src, const float* pairs, int64_t lo, int64_t hi,
                                            unsigned char* ring, unsigned char* pair_ring, uint32_t bars,
                                            Quarter quarter, Use use) {
  const int f = threadIdx.x & 127;
  const int at = ((f & 31) >> 2) * (kBlock / 8) + (f >> 5) * 128 + (f & 3);
  const uint32_t ring_a = smem_u32(ring), pair_a = smem_u32(pair_ring);
  bool ok = true;
  int64_t lost = 0;   // the block whose wait expired
  auto load = [&](int64_t k) {
    const int64_t g = quarter(k);
    if (f != 0 || 32 * g >= hi) return;
    const uint32_t slot = (uint32_t)(k % kDepth), bar = bars + 8 * slot;
    // pairs of the block's rows, an even number of them (16-byte copies)
    const uint32_t pb = pairs ? (uint32_t)((hi - 32 * g < 32 ? hi - 32 * g + 1 : 32) & ~1LL) * 8 : 0u;
    expect_bytes(bar, (uint32_t)kBlockBytes + pb);
    bulk_load(ring_a + slot * (uint32_t)kBlockBytes, src + ((g >> 2) * 5 * 4 + (g & 3)) * kBlock,
              (uint32_t)kBlockBytes, bar);
    if (pairs) bulk_load(pair_a + slot * 256, pairs + 64 * g, pb, bar);
  };
  auto arrived = [&](int64_t k) { return bar_wait(bars + 8 * (uint32_t)(k % kDepth), (uint32_t)((k / kDepth) & 1)); };
#pragma unroll
  for (int k = 0; k < kDepth; ++k) load(k);
  for (int64_t k = 0; 32 * quarter(k) < hi; ++k) {
    const int64_t row = 32 * quarter(k);
    const uint32_t slot = (uint32_t)(k % kDepth);
    if (ok && !arrived(k)) {
      ok = false;
      lost = k;
    }
    const float* d = reinterpret_cast<const float*>(ring + slot * kBlockBytes) + at;
    const float2* q = reinterpret_cast<const float2*>(pair_ring + slot * 256);
    if (row >= lo && row + 32 <= hi) {
#pragma unroll
      for (int i = 0; i < 32; ++i) use(d[4 * i], q + i);
    } else {
      for (int i = 0; i < 32; ++i)
        if (row + i >= lo && row + i < hi) use(d[4 * i], q + i);
    }
    asm volatile("bar.sync %0, 128;" ::"r"(grp + 1) : "memory");   // the slot has been read
    if (ok) load(k + kDepth);
  }
  if (!ok && f == 0)
    for (int64_t k = lost; k < lost + kDepth && 32 * quarter(k) < hi; ++k) arrived(k);
  return ok;
}

}  // namespace

__global__ void __launch_bounds__(kT, 1) mlp_wgrad_tc05_kernel(TrainTcArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, grp = tid >> 7, f = tid & 127;
  const int m = blockIdx.x;
  float* G = a.grad + ((int64_t)blockIdx.z * a.members + m) * kP;
  const int64_t r0 = (int64_t)blockIdx.z * a.rows < a.n ? (int64_t)blockIdx.z * a.rows : a.n;
  const int64_t r1 = r0 + a.rows < a.n ? r0 + a.rows : a.n;   // r0 = r1: a slice past the end, zeros
  const int64_t live = r1 - r0, per = (a.rows + kTile - 1) / kTile;
  const int64_t tile0 = (int64_t)m * a.tiles + blockIdx.z * per;   // the slice's first tile
  const float* blocks = a.block + tile0 * 5 * 4 * kBlock;          // its blocks: dz_1..dz_4, gelu(z_4)
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kGBar);      // full[2], free[2], done, rings[4][kDepth]
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 5 + 4 * kDepth);
  const uint32_t ring_bars = smem_u32(bars + 5 + kDepth * grp);
  const bool narrow = blockIdx.y == 3;
  if (tid == 0) {
    for (int k = 0; k < 5 + 4 * kDepth; ++k) bar_init(smem_u32(bars + k));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (!narrow && warp == 0) tmem_alloc<128>(tslot);
  fence_to_mma();
  __syncthreads();
  fence_after_sync();
  if (narrow) {
    // layers 1 and 5: thread = (layer, half of the slice's samples, feature),
    // running sums in sample order
    //   layer 1: dW1[f][i] = sum dz_1[f] x[i], db1[f] = sum dz_1[f];
    //   layer 5: dW5[j][f] = sum dout[j] gelu(z_4[f]), db5[j] = sum dout[j]
    const bool first = grp < 2;
    const int64_t mid = live / 2, lo = (grp & 1) ? mid : 0, hi = (grp & 1) ? live : mid;
    const float* pairs = first ? a.xb + 2 * r0 : a.dout + 2 * ((int64_t)m * pair_rows(a.n) + r0);
    float s0 = 0.f, s1 = 0.f, sb = 0.f;
    const bool ok = walk_blocks(
        grp, blocks + (first ? 0 : 4) * 4 * kBlock, pairs, lo, hi, smem + grp * kRingBytes,
        smem + kPairs + grp * kDepth * 256, ring_bars, [&](int64_t k) { return lo / 32 + k; },
        [&](float d, const float2* p) {
          const float2 q = *p;
          s0 = fmaf(d, q.x, s0);
          s1 = fmaf(d, q.y, s1);
          sb += first ? d : (f ? q.y : q.x);
        });
    if (!ok) atomicOr(a.error, 1u);
    float* part = reinterpret_cast<float*>(smem + kPart) + (first ? 0 : 768);
    float* mine = part + 3 * ((grp & 1) * H + f);
    mine[0] = s0;
    mine[1] = s1;
    mine[2] = sb;
    __syncthreads();
    if ((grp & 1) == 0) {
      const float* other = mine + 3 * H;
      const float w0 = mine[0] + other[0], w1 = mine[1] + other[1], bb = mine[2] + other[2];
      if (first) {
        G[oW1 + 2 * f] = w0;
        G[oW1 + 2 * f + 1] = w1;
        G[ob1 + f] = bb;
      } else {
        G[oW5 + f] = w0;
        G[oW5 + H + f] = w1;
        if (f < 2) G[ob5 + f] = bb;
      }
    }
    return;
  }
  const int l = blockIdx.y + 2;
  const uint32_t tmem = *tslot;
  const int chunks = (int)((live + kTile - 1) / kTile);
  bool ok = true;
  float bsum = 0.f;
  if (warp == 8) {
    // one thread loads the slice's (h_{l-1}, dz_l) tiles two ahead and multiplies
    if (lane == 0 && chunks > 0) {
      const uint32_t base = smem_u32(smem), kM = (uint32_t)kMatBytes;
      const uint32_t full = smem_u32(bars), freed = smem_u32(bars + 2);
      const __nv_bfloat16* src = a.tile + tile0 * 6 * H * H;
      auto load = [&](int c) {
        const uint32_t slot = base + (uint32_t)(c & 1) * 2 * kM, bar = full + (c & 1) * 8;
        expect_bytes(bar, 2 * kM);
        bulk_load(slot, src + ((int64_t)c * 6 + (l - 2)) * H * H, kM, bar);
        bulk_load(slot + kM, src + ((int64_t)c * 6 + (7 - l)) * H * H, kM, bar);
      };
      auto arrived = [&](int c) { return bar_wait(full + (c & 1) * 8, (uint32_t)(c >> 1) & 1); };
      load(0);
      if (chunks > 1) load(1);
      for (int c = 0; c < chunks && ok; ++c) {
        const uint32_t slot = base + (uint32_t)(c & 1) * 2 * kM;
        ok = arrived(c);
        if (ok) {
          mma_128<true, true>(tmem, slot + kM, slot, c > 0);
          mma_commit(c + 1 < chunks ? freed + (c & 1) * 8 : smem_u32(bars + 4));
          if (c + 2 < chunks) {
            ok = bar_wait(freed + (c & 1) * 8, (uint32_t)(c >> 1) & 1);
            if (ok) load(c + 2);
          }
        }
        if (!ok) {   // the others wait for the products issued so far, this thread for the copies under way
          mma_commit(smem_u32(bars + 4));
          arrived(c);
          if (c + 1 < chunks) arrived(c + 1);
          atomicOr(a.error, 1u);
        }
      }
    }
  } else if (grp < 2) {
    // bias gradient: group 0 takes the first 64 samples of every tile, group 1
    // the others, each one running sum in sample order
    ok = walk_blocks(
        grp, blocks + (l - 1) * 4 * kBlock, nullptr, 0, live, smem + 4 * kMatBytes + grp * kRingBytes, smem, ring_bars,
        [&](int64_t k) { return (k >> 1) * 4 + 2 * grp + (k & 1); }, [&](float d, const float2*) { bsum += d; });
    if (!ok) atomicOr(a.error, 1u);
  }
  // the last product; the limit of the wait grows with the slice
  bool done = chunks == 0;
  for (int c = 0; c < chunks && !done; ++c) done = bar_wait(smem_u32(bars + 4), 0);
  if (!done && tid == 0) atomicOr(a.error, 1u);
  fence_after_sync();
  __syncthreads();   // the slots are free: bias halves meet there
  float* red = reinterpret_cast<float*>(smem);
  if (tid < 256) red[tid] = bsum;
  __syncthreads();
  if (tid < H) G[b_of(l) + tid] = red[tid] + red[tid + H];
  // dW_l: rows 32 (warp % 4) + .., columns 32 (warp / 4) + ..; a quad of lanes
  // writes one 32-byte sector
  {
    const int c0 = (warp >> 2) * 32;
    float v[32];
    tmem_ld_frag32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0, v);
    float* Wg = G + w_of(l) + (int64_t)((warp & 3) * 32 + (lane >> 2)) * H + c0 + 2 * (lane & 3);
#pragma unroll
    for (int h = 0; h < 4; ++h)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int k = 16 * (h >> 1) + 4 * j + 2 * (h & 1);
        *reinterpret_cast<float2*>(Wg + 8 * h * H + 8 * j) =
            chunks > 0 ? make_float2(v[k], v[k + 1]) : make_float2(0.f, 0.f);
      }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  fence_after_sync();
  if (warp == 0) tmem_dealloc<128>(tmem);
}

// tiles of a batch of n samples in slices of rows
int64_t step_tiles(int64_t rows, int splits) { return (int64_t)splits * ((rows + kTile - 1) / kTile); }

cudaError_t launch_step_tc05(const TrainTcArgs& a, int splits, int sms, cudaStream_t s) {
  // once per process (thread-safe static initialisation)
  static const cudaError_t attr = [] {
    cudaError_t e = cudaFuncSetAttribute(mlp_step_tc05_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kStepSmem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(mlp_wgrad_tc05_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGradSmemTc);
    return e;
  }();
  if (attr != cudaSuccess) return attr;
  if (a.n <= 0 || a.members < 1 || a.members > kMaxMembers || splits < 1 || splits > kMaxSplits || a.rows < 1 ||
      a.rows * splits < a.n || a.tiles != step_tiles(a.rows, splits))
    return cudaErrorInvalidValue;
  // one CTA per SM in all; no more CTAs than full rounds of tiles need
  const int64_t per = sms / a.members > 1 ? sms / a.members : 1;
  const int64_t rounds = (a.tiles + per - 1) / per;
  mlp_step_tc05_kernel<<<dim3((unsigned)((a.tiles + rounds - 1) / rounds), a.members), kT, kStepSmem, s>>>(a);
  mlp_wgrad_tc05_kernel<<<dim3(a.members, 4, splits), kT, kGradSmemTc, s>>>(a);
  return cudaGetLastError();
}

}  // namespace mlp
}  // namespace ens
