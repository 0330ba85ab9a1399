// Device helpers shared by the CUDA translation units.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

namespace prd {

// Weideman expansion coefficients of the Faddeeva function (host-computed at
// prd_create, uploaded to constant memory of each translation unit that
// evaluates W): a_k, k = 1..N, and the scale L.
struct WeidemanConst {
  double a64[36];
  double L64;
};

template <typename T> struct Cx { T re, im; };

inline int ceil_div(long long a, long long b) { return (int)((a + b - 1) / b); }

}  // namespace prd
