// fp64ops.cuh -- FP64 products and sums issued as fused multiply-adds.
//
// The FP64 pipe takes a DFMA of a warp every 64 cycles whatever the number of
// warps, but with two or more warps on a sub-partition a DMUL or DADD holds it
// for 76 (dependent chains of each, 32 lanes, GB300).  So products and sums of
// the adaptive trial are written as a b + (-0) and a 1 + b, which round to the
// same bits: a b + (-0) is exact before its one rounding, and adding -0 keeps
// the sign of a zero product; a 1 is exact.  The constants are read from
// constant memory, where the compiler cannot fold them back into a DMUL or DADD.
#pragma once

#include <cuda_runtime.h>

namespace ens {

static __constant__ double kOneOpaque = 1.0;
static __constant__ double kNegZeroOpaque = -0.0;

__device__ __forceinline__ double fmul(double a, double b) { return __fma_rn(a, b, kNegZeroOpaque); }
__device__ __forceinline__ double fadd(double a, double b) { return __fma_rn(a, kOneOpaque, b); }
__device__ __forceinline__ double fsub(double a, double b) { return __fma_rn(a, kOneOpaque, -b); }

// The products and sums a system's trials take: fused ones in the kernels above, where
// they were measured.
struct FusedOps {
  static __device__ __forceinline__ double mul(double a, double b) { return fmul(a, b); }
  static __device__ __forceinline__ double add(double a, double b) { return fadd(a, b); }
  static __device__ __forceinline__ double sub(double a, double b) { return fsub(a, b); }
};
struct PlainOps {
  static __device__ __forceinline__ double mul(double a, double b) { return a * b; }
  static __device__ __forceinline__ double add(double a, double b) { return a + b; }
  static __device__ __forceinline__ double sub(double a, double b) { return a - b; }
};

}  // namespace ens
