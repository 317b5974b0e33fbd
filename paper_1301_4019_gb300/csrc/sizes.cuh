// sizes.cuh -- the sizes of the scan's units of work. No CUDA header is needed to compile it.
#pragma once

namespace rsk {

constexpr int kPer = 8;          // consecutive particles per lane of a warp
constexpr int kSeg = 32 * kPer;  // particles of a segment: one warp's, lane l holding the offsets
                                 // kPer l .. kPer l + kPer - 1

}  // namespace rsk
