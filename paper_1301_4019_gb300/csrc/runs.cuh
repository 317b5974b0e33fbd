// runs.cuh -- Code 11 by a warp: from the cumulative counts of a segment's particles to the runs of
// positions that they own, and the counts at the end of a sequence. Warp-level integer work on
// sequences of up to 2^31 - 1 particles and positions: what may pass 2^31 is a difference, an
// unsigned number or a 64-bit address. Needs the warp intrinsics only.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "sizes.cuh"

namespace rsk {
namespace {

constexpr int kRunWin = 32 * kPer;   // positions a warp reads back at a time
constexpr int kRunSpan = 2 * kRunWin;  // positions of a warp's window

// Valid particles of the segment at `base` of a sequence ending at N: offsets 0 .. count - 1 (zero
// or negative past the end).
__device__ __forceinline__ int seg_count(int64_t base, int64_t N) {
  const int64_t c = N - base;
  return c < kSeg ? static_cast<int>(c) : kSeg;
}

// Index b0 + k of a lane's first particle (past the sequence's end it may pass 2^31 - 1 and wrap:
// lanes without valid particles only).
__device__ __forceinline__ int32_t at_i32(int32_t b0, int k) {
  return static_cast<int32_t>(static_cast<uint32_t>(b0) + static_cast<uint32_t>(k));
}

// The count after a lane's particles, O those of its kPer particles, of which cnt (or all, for cnt
// >= kPer) are valid: n where the last of the sequence is among them or before them. tail: the
// segment holds the sequence's last particle, or lies past it.
__device__ __forceinline__ int32_t last_count(const int32_t (&O)[kPer], int cnt, bool tail,
                                              int32_t n) {
  return cnt >= kPer && !(tail && cnt == kPer) ? O[kPer - 1] : n;
}
// In a tail segment: the sequence's last particle gets the count n, the positions past it repeat
// the count before them (prev: the count before the lane's particles).
__device__ __forceinline__ void end_counts(int32_t (&O)[kPer], int32_t prev, int cnt, int32_t n) {
  int32_t p = prev;
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    O[q] = q >= cnt ? p : q + 1 == cnt ? n : O[q];
    p = O[q];
  }
}

// Counts of a warp's segment in non-decreasing order between those of its two ends: a count below
// one before it is raised to it, and none exceeds the last lane's last count. For accumulators
// whose scaling does not preserve order: two-float products rise and fall by up to 2^-46 relative
// across a step of the high word, so that W_i < W_j can give r_i > r_j and, with an integer between
// them, a count one lower. Nearly always the test finds nothing to do.
__device__ __forceinline__ void order_counts(int32_t (&O)[kPer], int32_t& prev) {
  bool down = false;
  int32_t p = prev;
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    down |= O[q] < p;
    p = O[q];
  }
  if (!__any_sync(0xffffffffu, down)) return;
  const int lane = threadIdx.x & 31;
  const int32_t P0 = __shfl_sync(0xffffffffu, prev, 0);
  const int32_t P1 = max(P0, __shfl_sync(0xffffffffu, O[kPer - 1], 31));
#pragma unroll
  for (int q = 1; q < kPer; ++q) O[q] = max(O[q], O[q - 1]);
  int32_t m = O[kPer - 1];
#pragma unroll
  for (int dd = 1; dd < 32; dd <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, m, dd);
    if (lane >= dd) m = max(m, y);
  }
  const int32_t before = __shfl_up_sync(0xffffffffu, m, 1);
  prev = lane == 0 ? P0 : min(max(before, P0), P1);
#pragma unroll
  for (int q = 0; q < kPer; ++q) O[q] = min(max(O[q], prev), P1);
}

// Eight consecutive values to a 32-byte aligned address (one whole sector).
__device__ __forceinline__ void st_global_v8(int32_t* p, const int32_t (&v)[kPer]) {
#ifdef __CUDACC__
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
#else
  for (int k = 0; k < kPer; ++k) p[k] = v[k];
#endif
}

// Code 11 for the particles of one warp: out[j] = the index of the particle whose run
// [O_{i-1}, O_i) holds j, for every j of the warp's range [P0, P1) (P0 = the count before the
// warp's first particle, P1 = after its last). Lane l holds the non-decreasing counts Oe[q] of
// its kPer particles i0 + q and `prev`, the count before them. Returns the bits of this lane's
// particles that have a run (bit q: particle i0 + q).
//
// The range is written through the warp's shared window of kRunSpan positions (nearly always
// one: a segment's kSeg particles have about kSeg offspring): -1 everywhere, then the first
// position of each run receives its particle's index; the window is read back, eight consecutive
// positions per lane, and filled by a running maximum (in-lane; then the last head before the
// lane, found by ballot; or the last value of the part before, which every lane takes into
// account: a run can cover a whole part). Windows start at 32-byte boundaries of `out`, so a
// lane's eight positions are one 256-bit store; the two groups of eight that the range's ends
// cut are written back and stored by sixteen lanes. A short rest beyond the first 256 positions
// (half of the segments have one, mostly under 32 positions) is read two positions per lane.
// The first position P0 always starts a run, so the carry of the first part can be -1.
//
// The counts are non-decreasing from P0 to P1 over the warp (monotone functions of the cumulative
// weights for binary32 and binary64 sums, order_counts for two-float sums, checked counts from a
// caller), so every head lies in [P0, P1) and one window holds them all when P1 - base <= kRunSpan;
// longer ranges test every head.
// Same result as writing out[j] = i for j in [O_{i-1}, O_i) particle by particle, without its
// divergent loops.
__device__ __forceinline__ uint32_t warp_runs(const int32_t (&Oe)[kPer], int32_t prev, int32_t i0,
                                              int32_t* __restrict__ out, int32_t* win) {
  static_assert(kPer == 8 && kRunWin == 256, "a lane's positions are one 32-byte sector");
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  const int32_t P0 = __shfl_sync(0xffffffffu, prev, 0);
  const int32_t P1 = __shfl_sync(0xffffffffu, Oe[kPer - 1], 31);
  if (P1 <= P0) return 0u;  // no position (warp-uniform)
  const uint32_t shift = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(out) >> 2) & 7u;
  int4* const w4 = reinterpret_cast<int4*>(win);
  uint32_t bits = 0;
  int32_t carry = -1;
  // the last head at or before this lane's last position of a part (top: its in-lane maximum)
  auto before_lane = [&](int32_t top) {
    const unsigned heads = __ballot_sync(0xffffffffu, top >= 0);
    const unsigned earlier = heads & below;
    const int32_t m = __shfl_sync(0xffffffffu, top, 31 - __clz(earlier | 1u));
    const int32_t em = earlier ? m : carry;
    const int32_t last = __shfl_sync(0xffffffffu, top, 31 - __clz(heads | 1u));
    carry = heads ? last : carry;
    return em;
  };
  // (a lane's position j0 may pass 2^31 - 1 and wrap to one far below P0, which is never stored; the
  // ends are compared as P0 - 8 and P1 - 8, which cannot wrap)
  auto part8 = [&](int h, int32_t base) {  // 256 positions
    const int4 u0 = w4[64 * h + 2 * lane], u1 = w4[64 * h + 2 * lane + 1];
    int32_t v[kPer] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
#pragma unroll
    for (int k = 1; k < kPer; ++k) v[k] = max(v[k], v[k - 1]);
    const int32_t em = before_lane(v[kPer - 1]);
#pragma unroll
    for (int k = 0; k < kPer; ++k) v[k] = max(v[k], em);
    const int32_t j0 = at_i32(base, kRunWin * h + kPer * lane);
    if (j0 >= P0 && j0 <= P1 - kPer) {
      st_global_v8(out + j0, v);
    } else if (j0 > P0 - kPer && j0 < P1) {  // cut by an end of the range
      w4[64 * h + 2 * lane] = make_int4(v[0], v[1], v[2], v[3]);
      w4[64 * h + 2 * lane + 1] = make_int4(v[4], v[5], v[6], v[7]);
    }
  };
  // (the first window begins at -7 or after; `len` positions from there to P1, below 2^31 + 7)
  for (int32_t base = at_i32(static_cast<int32_t>((static_cast<uint32_t>(P0) + shift) & ~7u),
                             -static_cast<int>(shift));;
       base += kRunSpan) {  // warp-uniform
    const uint32_t len = static_cast<uint32_t>(P1) - static_cast<uint32_t>(base);
    const int4 none = make_int4(-1, -1, -1, -1);
    __syncwarp();
    w4[lane] = none;
    w4[32 + lane] = none;
    if (len > kRunWin) {
      w4[64 + lane] = none;
      w4[96 + lane] = none;
    }
    __syncwarp();
    int32_t p = prev;
    if (len <= kRunSpan && base <= P0) {
      int32_t* const wb = win - base;
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        if (Oe[q] > p) {
          bits |= 1u << q;
          wb[p] = i0 + q;
        }
        p = Oe[q];
      }
    } else {
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        if (Oe[q] > p) {
          bits |= 1u << q;
          const uint32_t pos = static_cast<uint32_t>(p) - static_cast<uint32_t>(base);
          if (pos < static_cast<uint32_t>(kRunSpan)) win[pos] = i0 + q;
        }
        p = Oe[q];
      }
    }
    __syncwarp();
    part8(0, base);
    // the group that the range's end cuts
    int32_t cut = len < kRunSpan ? static_cast<int32_t>(len & ~7u) : kRunSpan;
    if (len > kRunWin + 64) {
      part8(1, base);
    } else if (len > kRunWin) {  // a short rest: two positions per lane
      const int2 u = reinterpret_cast<const int2*>(win + kRunWin)[lane];
      const int32_t top = max(u.x, u.y);
      const int32_t em = before_lane(top);
      const uint32_t k = kRunWin + 2 * lane;
      const int32_t j0 = at_i32(base, kRunWin + 2 * lane);
      if (k < len) out[j0] = max(u.x, em);
      if (k + 1 < len) out[j0 + 1] = max(top, em);
      cut = kRunSpan;  // (nothing left to store)
    }
    __syncwarp();
    // the groups that the ends cut: the window's first (where it starts before P0), by the first
    // eight lanes, and the one that holds P1, by the next eight
    const int idx = lane < kPer ? lane : cut + lane - kPer;
    if (lane < 2 * kPer && static_cast<uint32_t>(idx) < len && idx < kRunSpan &&
        at_i32(base, idx) >= P0 && (lane >= kPer ? (len & 7u) != 0 : base < P0))
      out[base + idx] = win[idx];
    if (len <= kRunSpan) break;
  }
  return bits;
}

}  // namespace
}  // namespace rsk
