// Code 11 of one segment (csrc/runs.cuh) on the host.
#include <cuda_runtime.h>

#include "runs.cuh"
#include "values.cuh"

using namespace rsk;

// Counts floor(W c + u) of two-float cumulative weights W by the library's operations (c and u:
// high and low words).
extern "C" void two_float_counts(const float* W, int n, const float* c, const float* u, int32_t* O) {
  for (int i = 0; i < n; ++i)
    O[i] = static_cast<int32_t>(floor_to_i64(vplus_u(
        vscale(make_float2(W[2 * i], W[2 * i + 1]), make_float2(c[0], c[1])), make_float2(u[0], u[1]))));
}

// The 256 particles from b0 on of a sequence of n, counts O and the count `before`; positions
// [first, first + len) of the output are kept in `out` (guards around them belong to the caller),
// the output's base being `shift` elements off a 32-byte boundary. bits: 32 bytes. Returns 0, or 1
// for a write outside the warp's window. two_float: the counts of two-float sums.
extern "C" int segment_runs(int two_float, const int32_t* O, int32_t before, int32_t b0, int32_t n, int64_t first,
                            int32_t* out, int shift, uint8_t* bits) {
  constexpr int kGuard = 4096;
  alignas(32) static int32_t mem[kRunSpan + 2 * kGuard];
  for (int32_t& x : mem) x = -77;
  int32_t* const win = mem + kGuard;
  // (the address of position 0: `out` is 32-byte aligned where first + shift is a multiple of 8)
  int32_t* const base = reinterpret_cast<int32_t*>(reinterpret_cast<uintptr_t>(out) - 4 * first);
  if (((reinterpret_cast<uintptr_t>(base) >> 2) & 7u) != static_cast<uintptr_t>(shift)) return 2;
  host_warp::run([&](int lane) {
    const bool tail = n - b0 <= kSeg;
    const int cnt = seg_count(b0, n) - kPer * lane;
    const int32_t i0 = at_i32(b0, kPer * lane);
    int32_t o[kPer];
    for (int q = 0; q < kPer; ++q) o[q] = O[kPer * lane + q];
    int32_t prev = __shfl_up_sync(0xffffffffu, last_count(o, cnt, tail, n), 1);
    if (lane == 0) prev = cnt > 0 ? before : n;
    if (tail) end_counts(o, prev, cnt, n);
    if (two_float) order_counts(o, prev);
    bits[lane] = static_cast<uint8_t>(warp_runs(o, prev, i0, base, win));
  });
  for (int k = 0; k < kGuard; ++k)
    if (mem[k] != -77 || mem[kGuard + kRunSpan + k] != -77) return 1;
  return 0;
}
