// permute.cuh -- one slot of the parallel Permute of Code 10 (Appendix C), shared by the
// single-filter and batched kernels. The claims d (Prepermute: d[j] = lowest i with a[i] = j,
// or the sentinel n) must be complete before any thread runs this.
#pragma once

#include <cstdint>

#include "common.cuh"

namespace rsk {
namespace {

// Second procedure of Code 10 fused with its gather c^i = a^{d^i}, for index i of a vector
// of n ancestors (local indices):
//  - a claimed slot i (d_i < n) keeps its own particle: c_i = a[d_i] = i;
//  - a particle whose claim failed (d[a_i] != i) walks x = i, d[x], d[d[x]], ... to the
//    first unclaimed slot x and writes c_x = a_i there.
// The walks start at indices absent from d and d is injective on claimed slots, so the
// walks are disjoint and end at distinct unclaimed slots (the termination argument of
// Appendix C): they only read d, and every slot of c is written exactly once, in any order.
// kCoherent: a and d were written earlier in the same kernel launch (by other CTAs), so they
// are read through L2 only.
template <bool kCoherent>
__device__ __forceinline__ int32_t ld_i32(const int32_t* p) {
  if constexpr (kCoherent) return __ldcg(p); else return *p;
}
template <bool kCoherent = false>
__device__ __forceinline__ void permute_one(const int32_t* __restrict__ a,
                                            const int32_t* __restrict__ d, int64_t n,
                                            int32_t* __restrict__ c, int64_t i, int* err) {
  const int32_t sentinel = static_cast<int32_t>(n);
  const int32_t ai = ld_i32<kCoherent>(a + i);
  if (ai < 0 || ai >= n) {
    flag_error(err, RS_ERR_ARG);
    return;
  }
  if (ld_i32<kCoherent>(d + i) != sentinel) c[i] = static_cast<int32_t>(i);
  if (ld_i32<kCoherent>(d + ai) != static_cast<int32_t>(i)) {
    int64_t x = i;
    int64_t steps = 0;
    for (;;) {
      const int32_t dx = ld_i32<kCoherent>(d + x);
      if (dx == sentinel) break;
      if (dx < 0 || dx > sentinel || ++steps > n) {  // only a corrupted d can get here
        flag_error(err, RS_ERR_ARG);
        return;
      }
      x = dx;
    }
    c[x] = ai;
  }
}

// Claims of Code 10 read from the Prepermute vector d (d[x] = the lowest position whose
// ancestor is x, or the sentinel n).
struct ClaimsOf {
  const int32_t* __restrict__ d;
  __device__ __forceinline__ int32_t operator()(int32_t x) const { return d[x]; }
};

// Walks of Code 10 for a whole warp, K walkers per lane, queued: walker q stands at slot
// x[q] with dx[q] = claim(x[q]) already loaded (claim: the Prepermute claim of a slot, the
// sentinel n for an unclaimed one) and ends at the first unclaimed slot, where c receives
// val[q]. A walker whose claim ends at its own slot (dx = the sentinel) is done at once; the
// others take their first step and are collected, by ballot, into the warp's shared list
// `pend` (32 K entries), which the lanes then work off one walk each to its end (lane l takes
// entries l, l + 32, ...), so every lane runs only walks that go on. The walks start at
// distinct failed claims and are disjoint (see permute_one): c is the same as walking each
// one alone. Called by all 32 lanes (lanes without walkers pass act = false).
template <int K, typename Claim>
__device__ __forceinline__ void walk_queue(const Claim& claim, int32_t sentinel,
                                           int32_t* __restrict__ c, const int32_t (&x)[K],
                                           const int32_t (&dx)[K], const int32_t (&val)[K],
                                           const bool (&act)[K], int64_t n, int2* pend,
                                           int* err) {
  const uint32_t us = static_cast<uint32_t>(sentinel);
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  bool bad = false;
  int total = 0;
#pragma unroll
  for (int q = 0; q < K; ++q) {
    bool go = false;
    if (act[q]) {
      const uint32_t v = static_cast<uint32_t>(dx[q]);
      if (v == us) c[x[q]] = val[q];  // its own slot is unclaimed: the walk ends there
      else if (v > us) bad = true;    // (only a corrupted claim vector)
      else go = true;
    }
    const unsigned m = __ballot_sync(0xffffffffu, go);
    if (go) pend[total + __popc(m & below)] = make_int2(dx[q], val[q]);  // one step taken
    total += __popc(m);
  }
  __syncwarp();
  for (int e = lane; e < total; e += 32) {
    const int2 w = pend[e];
    int32_t xs = w.x;
    for (int64_t steps = 0;; ++steps) {
      const uint32_t v = static_cast<uint32_t>(claim(xs));
      if (v == us) {
        c[xs] = w.y;
        break;
      }
      if (v > us || steps > n) {  // only a corrupted claim vector can get here
        bad = true;
        break;
      }
      xs = static_cast<int32_t>(v);
    }
  }
  __syncwarp();
  if (bad) flag_error(err, RS_ERR_ARG);
}

// Four consecutive slots i0 .. i0 + 3 of the Permute of n ancestors a with claims d (any
// ancestry; the general form of permute_one): 128-bit slot loads where the addresses allow, the
// four claim checks d[a_i] issued together, and the walks of failed claims run together
// (walk_queue). Called by all 32 lanes of a warp; slots at n or beyond do nothing. Same reads
// and writes per slot as permute_one, so c is the same.
__device__ __forceinline__ void permute4_slots(const int32_t* __restrict__ a,
                                               const int32_t* __restrict__ d, int64_t n,
                                               int32_t* __restrict__ c, int64_t i0, int2* pend,
                                               int* err) {
  const int32_t sentinel = static_cast<int32_t>(n);
  int32_t A[4], D[4];
  const bool vec = i0 + 3 < n && ((reinterpret_cast<uintptr_t>(a + i0) |
                                   reinterpret_cast<uintptr_t>(d + i0)) & 15u) == 0;
  if (vec) {
    const int4 va = *reinterpret_cast<const int4*>(a + i0);
    const int4 vd = *reinterpret_cast<const int4*>(d + i0);
    A[0] = va.x; A[1] = va.y; A[2] = va.z; A[3] = va.w;
    D[0] = vd.x; D[1] = vd.y; D[2] = vd.z; D[3] = vd.w;
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      A[q] = i0 + q < n ? a[i0 + q] : 0;
      D[q] = i0 + q < n ? d[i0 + q] : sentinel;
    }
  }
  bool ok[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    ok[q] = i0 + q < n;
    if (ok[q] && (A[q] < 0 || A[q] >= n)) {
      flag_error(err, RS_ERR_ARG);
      ok[q] = false;
    }
  }
  int32_t claim[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) claim[q] = ok[q] ? d[A[q]] : static_cast<int32_t>(i0 + q);
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (ok[q] && D[q] != sentinel) c[i0 + q] = static_cast<int32_t>(i0 + q);
  bool fail[4];
  int32_t x[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    fail[q] = ok[q] && claim[q] != static_cast<int32_t>(i0 + q);
    x[q] = static_cast<int32_t>(i0 + q);
  }
  walk_queue<4>(ClaimsOf{d}, sentinel, c, x, D, A, fail, n, pend, err);
}

// Permute of a non-decreasing ancestry from a and the claimed bits of its emission (cl: bit
// i % 8 of cl[i / 8] set when particle i has offspring). For such an ancestry the claims of
// Prepermute are d_j = the first position of the run of j for every claimed j, so Code 10's
// walks can be followed from their ends instead of their starts:
//  - a claimed slot x keeps its particle: c_x = x;
//  - an unclaimed slot x that is not the first of its run (a_{x-1} = a_x) is a failed claim
//    whose walk ends at once, at x: c_x = a_x;
//  - an unclaimed slot x that is the first of its run was reached from z = a_x (d_z = x);
//    while z is itself the first of its run (z = 0 or a_{z-1} != a_z) it was reached from
//    a_z in turn, and the first z that is not is the walk's start: c_x = a_z.
// d is injective on the claimed slots and the walks end (Appendix C), so each backward chain
// is one walk reversed and c is Code 10's exactly; the claims are never stored.
//
// The chain of one unclaimed run head whose ancestor is z < n, to its start: returns the value
// that the head receives, or sets bad (only a corrupted a can do that).
__device__ __forceinline__ int32_t sorted_chain(const int32_t* __restrict__ a, int32_t z,
                                                int32_t n, bool& bad) {
  for (int32_t left = n;; --left) {
    const int32_t* const p = a + z;
    const int32_t y = *p;
    const int32_t before = z > 0 ? p[-1] : -1;
    if (static_cast<uint32_t>(y) >= static_cast<uint32_t>(n) || left == 0) {
      bad = true;
      return 0;
    }
    if (before == y) return y;  // not the first of its run
    z = y;
  }
}

// One slot i of it (n ancestors, local indices).
__device__ __forceinline__ void permute_sorted_one(const int32_t* __restrict__ a,
                                                   const uint8_t* __restrict__ cl, int64_t n,
                                                   int32_t* __restrict__ c, int64_t i, int* err) {
  const int32_t ai = a[i];
  if (ai < 0 || ai >= n) {
    flag_error(err, RS_ERR_ARG);
    return;
  }
  bool bad = false;
  int32_t v;
  if ((cl[i >> 3] >> (i & 7)) & 1) v = static_cast<int32_t>(i);
  else if (i > 0 && a[i - 1] == ai) v = ai;
  else v = sorted_chain(a, ai, static_cast<int32_t>(n), bad);
  if (bad) flag_error(err, RS_ERR_ARG);
  else c[i] = v;
}

// K consecutive slots i0 .. i0 + K - 1 of it per lane (lane l's follow lane l - 1's), called by
// all 32 lanes of a warp; slots at n or beyond do nothing. The chains that go on past their
// first step are queued per warp in slot order (pend: 32 K entries) and run one per lane; the
// warp's results are gathered in cw (32 K entries, 16-byte aligned) and stored 128 bits at a time
// where the addresses allow. A warp with all its slots below n and all its ancestors in range
// (every warp but the last of a sequence) takes no tests per slot.
template <int K>
__device__ __forceinline__ void permute_sorted_slots(const int32_t* __restrict__ a,
                                                     const uint8_t* __restrict__ cl, int64_t n64,
                                                     int32_t* __restrict__ c, int64_t i064,
                                                     int32_t* cw, int2* pend, int* err) {
  static_assert(K == 1 || K == 4, "one or four slots per thread");
  const int lane = threadIdx.x & 31;
  // (n < 2^31; slots past n only need to compare as such: i0 < n + 2^12 < 2^32)
  const uint32_t n = static_cast<uint32_t>(n64), i0 = static_cast<uint32_t>(i064);
  const bool full = i0 + K <= n;
  uint32_t A[K];
  if (K == 4 && full && (reinterpret_cast<uintptr_t>(a + i0) & 15u) == 0) {
    const uint4 va = *reinterpret_cast<const uint4*>(a + i0);
    A[0] = va.x; A[1] = va.y; A[2] = va.z; A[3] = va.w;
  } else {
#pragma unroll
    for (int q = 0; q < K; ++q) A[q] = i0 + q < n ? static_cast<uint32_t>(a[i0 + q]) : 0u;
  }
  uint32_t bits = 0u;
  if (i0 < n) {
    const int sh = static_cast<int>(i0 & 7u);
    bits = static_cast<uint32_t>(cl[i0 >> 3]) >> sh;
    if (K == 4 && sh > 4 && i0 + (8 - sh) < n)  // (the slots reach into the next byte)
      bits |= static_cast<uint32_t>(cl[(i0 >> 3) + 1]) << (8 - sh);
  }
  // a_{i0-1}: the previous lane's last slot, loaded by lane 0 only
  uint32_t prev = __shfl_up_sync(0xffffffffu, A[K - 1], 1);
  if (lane == 0) prev = (i0 > 0 && i0 - 1 < n) ? static_cast<uint32_t>(a[i0 - 1]) : ~0u;
  // this lane's unclaimed run heads (bit q: slot i0 + q), and every other slot's result
  uint32_t top = A[0], go = 0u;
  int32_t R[K];
#pragma unroll
  for (int q = 0; q < K; ++q) {
    if (q > 0) top = max(top, A[q]);
    const bool claimed = (bits >> q) & 1u;
    go |= static_cast<uint32_t>(!claimed && A[q] != (q > 0 ? A[q > 0 ? q - 1 : 0] : prev)) << q;
    R[q] = static_cast<int32_t>(claimed ? i0 + q : A[q]);
  }
  bool bad = false;
  if (!full || top >= n) {  // the sequence's end, or an ancestor out of range: slot by slot
    go = 0u;
#pragma unroll
    for (int q = 0; q < K; ++q) {
      if (i0 + q >= n) continue;
      if (A[q] >= n) bad = true;
      else if (!((bits >> q) & 1u) && A[q] != (q > 0 ? A[q > 0 ? q - 1 : 0] : prev)) go |= 1u << q;
    }
  }
  // places in the queue: the heads of the lanes below (counts 0 .. 4, a ballot per bit of them)
  const uint32_t cnt = __popc(go), below = (1u << lane) - 1u;
  const uint32_t b0 = __ballot_sync(0xffffffffu, cnt & 1u);
  int at = __popc(b0 & below), total = __popc(b0);
  if (K == 4) {
    const uint32_t b1 = __ballot_sync(0xffffffffu, cnt & 2u);
    const uint32_t b2 = __ballot_sync(0xffffffffu, cnt & 4u);
    at += 2 * __popc(b1 & below) + 4 * __popc(b2 & below);
    total += 2 * __popc(b1) + 4 * __popc(b2);
  }
#pragma unroll
  for (int q = 0; q < K; ++q)
    if ((go >> q) & 1u) pend[at++] = make_int2(K * lane + q, static_cast<int32_t>(A[q]));
  if (K == 4) {
    reinterpret_cast<int4*>(cw)[lane] = make_int4(R[0], R[K > 1 ? 1 : 0], R[K > 2 ? 2 : 0], R[K - 1]);
  } else {
    cw[lane] = R[0];
  }
  __syncwarp();
  for (int e = lane; e < total; e += 32) {
    const int2 w = pend[e];
    bool cbad = false;
    const int32_t v = sorted_chain(a, w.y, static_cast<int32_t>(n), cbad);
    if (cbad) bad = true;
    else cw[w.x] = v;
  }
  __syncwarp();
  if (K == 4 && full && (reinterpret_cast<uintptr_t>(c + i0) & 15u) == 0) {
    *reinterpret_cast<int4*>(c + i0) = reinterpret_cast<const int4*>(cw)[lane];
  } else {
#pragma unroll
    for (int q = 0; q < K; ++q)
      if (i0 + q < n) c[i0 + q] = cw[K * lane + q];
  }
  if (bad) flag_error(err, RS_ERR_ARG);
}

}  // namespace
}  // namespace rsk
