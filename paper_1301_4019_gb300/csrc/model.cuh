// model.cuh -- the 1-D linear-Gaussian state-space model's noise and constants, shared by the
// kernels that propagate and weight its particles.
#pragma once

#include <cmath>
#include <cstdint>

#include "common.cuh"

namespace rsk {
namespace {

// One standard normal per particle by Box-Muller from the Philox words 0 and 1 of counter
// (i, 0, step, filter * 8 + 5): u1 = 1 - U_0 in (0, 1], u2 = U_1 in [0, 1).
__device__ __forceinline__ float normal_draw(const Keys& keys, int64_t i) {
  const uint4 r = draw(keys, static_cast<uint32_t>(i), 0u);
  const float u1 = 1.0f - __fmul_rn(__uint2float_rn(r.x >> 8), 0x1p-24f);
  const float u2 = __fmul_rn(__uint2float_rn(r.y >> 8), 0x1p-24f);
  return sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
}

// The stationary standard deviation sigma_x / sqrt(1 - phi^2) and 1 / (2 sigma_y^2).
struct LgssmConsts {
  float sigma_0, inv_2vy;
};
inline LgssmConsts lgssm_consts(float phi, float sigma_x, float sigma_y) {
  const double s0 = static_cast<double>(sigma_x) / std::sqrt(1.0 - static_cast<double>(phi) * phi);
  return LgssmConsts{static_cast<float>(s0),
                     static_cast<float>(0.5 / (static_cast<double>(sigma_y) * sigma_y))};
}

}  // namespace
}  // namespace rsk
