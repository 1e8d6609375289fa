// controller.cuh -- error norm, step factor and system claiming of the adaptive
// kernels (rkck45.cu, rkck45_teams.cu).
#pragma once

#include "common.cuh"
#include "fcmp.cuh"
#include "fifth_root_fx.cuh"
#include "fp64ops.cuh"
#include "rcp_fx.cuh"

namespace ens {

// right-hand-side evaluations of one trial besides k1
constexpr uint32_t pair_rhs(int PAIR) { return PAIR == kDormandPrince ? 6u : 5u; }

// E = max_c |err_c| / (atol + rtol max(|y_c|, |y5_c|)), >= 0, or NaN (sign
// clear) when a trial blew up.  rcp_fx (integer pipe) is within half an ulp
// plus 2^-57 of 1/sc for the normal sc below 2^1022 of a solve; a zero,
// subnormal, infinite or NaN sc gives NaN, and a NaN stays the maximum.
// (1 / sc and the ratio on their own: err_weight, err_ratio)
__device__ __forceinline__ double err_weight(double y, double y5, double rtol, double atol) {
  return rcp_fx(fma(rtol, nnmax(absd(y), absd(y5)), atol));
}
template <class Ops = FusedOps>
__device__ __forceinline__ double err_ratio(double err, double weight) { return absd(Ops::mul(absd(err), weight)); }
template <int D, class Ops = FusedOps>
__device__ __forceinline__ double err_norm(const double* y, const double* y5, const double* err,
                                           double rtol, double atol) {
  double E = 0.0;
#pragma unroll
  for (int c = 0; c < D; ++c) {
    E = nnmax(E, err_ratio<Ops>(err[c], err_weight(y[c], y5[c], rtol, atol)));
  }
  return E;
}
// accept iff E <= 1 (false for NaN)
__device__ __forceinline__ bool accept(double E) { return nnbits(E) <= nnbits(1.0); }

// fac = clamp(0.9 E^(-1/5), 0.2, 5).  0.9 E^(-1/5) leaves [0.2, 5] for
// E > 4.5^5 = 1845.3 and E < 0.18^5 = 1.9e-4, so E is clamped to [1e-4, 2000]
// first (same result, and keeps the float seed of inv_fifth_root_fx in range).
// E >= 0 or NaN as err_norm returns it.
template <class Ops = FusedOps>
__device__ __forceinline__ double step_factor(double E) {
  if (nnbits(E) > nnbits(__longlong_as_double(0x7ff0000000000000LL))) return 0.2;  // NaN
  const double Ec = nnmin(nnmax(E, 1e-4), 2000.0);
  const double fac = Ops::mul(0.9, inv_fifth_root_fx(Ec));
  return nnmin(nnmax(fac, 0.2), 5.0);
}

// Claim the next system of a persistent lane (or, in plain mode, the own system
// of lane `me` of the block's `lanes`).  Returns -1 when no work is left.
__device__ __forceinline__ int64_t claim(const AdaptArgs& a, bool first, int lanes, int me) {
  if (!a.persistent) {
    if (!first) return -1;
    const int64_t i = blockIdx.x * (int64_t)lanes + me;
    return i < a.n ? i : -1;
  }
  const unsigned long long k = atomicAdd(&a.scratch->next, 1ULL);
  if (k >= (unsigned long long)a.n) return -1;
  return a.order ? (int64_t)a.order[k] : (int64_t)k;
}

// First claim of a lane in a persistent, longest-first launch with one block
// per SM, deterministic and aware of the sub-partitions: warp w of a block
// runs on sub-partition w mod 4, and a warp that shares its sub-partition
// gets about half of that sub-partition's FP64 pipe (W warps hold systems; helper
// warps after them use none of it).  The lanes of warps that
// own their sub-partition take the first ranks of the claim order (the
// longest systems), the others the next ones; later claims continue from rank
// gridDim.x * lanes in order (claim_next_after_ranked).  The claim order
// never changes what a system computes.
__device__ __forceinline__ int64_t claim_first_by_subpartition(const AdaptArgs& a, int W, int w) {
  const int lane = (int)(threadIdx.x & 31);
  int u_total = 0, u_before = 0;
  for (int x = 0; x < W; ++x) {
    const bool own = ((W - (x & 3) + 3) >> 2) == 1;  // the only warp of block x's sub-partition
    u_total += own;
    u_before += own && x < w;
  }
  const bool own = ((W - (w & 3) + 3) >> 2) == 1;
  const int64_t U = (int64_t)gridDim.x * u_total * 32;
  const int64_t rank = own ? ((int64_t)blockIdx.x * u_total + u_before) * 32 + lane
                           : U + ((int64_t)blockIdx.x * (W - u_total) + (w - u_before)) * 32 + lane;
  return rank < a.n ? (int64_t)a.order[rank] : -1;
}
__device__ __forceinline__ int64_t claim_next_after_ranked(const AdaptArgs& a, int lanes) {
  const unsigned long long k = (unsigned long long)gridDim.x * lanes + atomicAdd(&a.scratch->next, 1ULL);
  return k < (unsigned long long)a.n ? (int64_t)a.order[k] : -1;
}

}  // namespace ens
