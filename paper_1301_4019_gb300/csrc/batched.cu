// batched.cu -- many independent filters of uneven sizes resampled in a handful of launches
// (F filters in CSR layout: filter f holds the particles offsets[f] .. offsets[f+1]-1).
//
// The paper resamples one filter per call; resampling thousands of small filters one call at a
// time is launch-bound, and giving each filter to one CTA serialises its passes and leaves the
// largest (or, for Metropolis, the highest-B) filters as a long tail. Here the work units are
// the tiles and the particles of all filters together:
//   plan    : tiles per filter (kTile particles, starting at the filter's first particle) and
//             their prefix over filters; per-filter maxima reset            (1 CTA)
//   max     : per tile, maximum log-weight, combined per filter by an atomic max of keys
//   sums    : per tile, the tile scan total                               (tile-parallel)
//   prefix  : per filter, tile prefixes, W^N and N / W^N                  (CTA per filter)
//   emit    : per tile, cumulative offspring + Code-11 scatter + claimed bits, or stored W
//   search  : one thread per particle, its filter found by a binary search of the offsets
//   chains  : binary32 Metropolis from shared memory, chunks of equal work per CTA
//             (batch_chain_kernel); binary64 one thread per particle
//   rejection : a warp per run of particles, its lanes sharing the last ones
//   Permute : a warp per 32 or 128 consecutive slots, its filter looked up once.
// With cooperative launches (the default), max, sums, prefixes and emission run as one
// persistent launch over the segments of all filters (batch_coop_kernel) after the plan, so a
// scan-based scheme is plan + one launch (+ the search for the multinomial) + Permute.
// Every unit runs the same device functions as the single-filter kernels on the same segment
// structure (relative to the filter's first particle), with the filter index in the
// random-number counter: filter f of a batched call equals rs_resample on that filter's slice
// with filter = f, bit for bit.
#include <algorithm>
#include <climits>
#include <mutex>

#include "common.cuh"
#include "grid.cuh"
#include "internal.h"
#include "mcmc.cuh"
#include "permute.cuh"
#include "ragged.cuh"
#include "tile.cuh"
#include "values.cuh"

namespace rsk {
namespace {

// locate_in with the filter of position g looked up; false for positions past the batch's end.
__device__ __forceinline__ bool locate_particle(const int64_t* __restrict__ off, int F,
                                                int64_t max_n, int64_t g, PartLoc& P) {
  const int64_t end = batch_end(off, F, max_n);
  return g < end && locate_in(off, filter_of(off, F, g), end, g, P);
}

// Flags descending offsets (the per-particle schemes, whose kernels look every particle's filter
// up themselves and stay inside it). Not inlined: in line it cost the rejection 10 %.
__device__ __noinline__ void flag_descending(const int64_t* __restrict__ off, int F, int* err) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t f = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; f < F; f += stride)
    if (descends(off, static_cast<int>(f))) flag_error(err, RS_ERR_ARG);
}

// filter_of for one position g, by a whole warp (every lane calls it with the same g): 32
// offsets are compared at a time, so 4096 filters take three dependent loads instead of twelve.
template <typename I>
__device__ __forceinline__ int filter_of_warp(const I* __restrict__ off, int F, I g) {
  const int lane = threadIdx.x & 31;
  int lo = 0, hi = F;  // invariant: off[lo] <= g < off[hi]
  while (hi - lo > 1) {
    const int step = (hi - lo + 31) >> 5;
    const int at = lo + (lane + 1) * step;
    const bool below = at < hi && __ldg(off + at) <= g;
    const int cnt = __popc(__ballot_sync(0xffffffffu, below));
    lo += cnt * step;
    hi = min(hi, lo + step);
  }
  return lo;
}

// The filter of position g >= off[f] from the filter f of an earlier position: a few steps
// past the offsets g has crossed, else filter_of. Same filter as filter_of(off, F, g).
__device__ __forceinline__ int advance_filter(const int64_t* __restrict__ off, int F, int64_t g,
                                              int f) {
  for (int st = 0; st < 8; ++st) {
    if (f + 1 >= F || __ldg(off + f + 1) > g) return f;
    ++f;
  }
  return (f + 1 < F && __ldg(off + f + 1) <= g) ? filter_of(off, F, g) : f;
}

// Tile t of the batch -> its filter (the last f with tile_start[f] <= t).
__device__ __forceinline__ int filter_of_tile(const int32_t* __restrict__ ts, int F, int t) {
  int lo = 0, hi = F;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (__ldg(ts + mid) <= t) lo = mid; else hi = mid;
  }
  return lo;
}

struct Batch {
  const int64_t* off;
  int F;
  int64_t max_n;
  int32_t* tile_start;   // F + 1: first tile of each filter
  int32_t* seg_start;    // F + 2: first segment (of kSeg particles) of each filter, and the
                         // segments of the longest one
  long long* fmax;       // F, keys of the per-filter maxima
  double2* fS;           // F: total (accumulator type)
  double2* fscale;       // F: N / total
  double* fSd;           // F: total in binary64
  double2* s_rec;        // tile totals, indexed by batch tile
  double2* P_rec;        // tile prefixes, filter f at tile_start[f] + f
  const uint8_t* resample;  // F flags (0: the filter keeps its particles), or null = all
  uint8_t* cl;           // claimed bits (filter f's bytes at (off[f] >> 3) + f), or null
  int32_t* limit;        // set by the plan: the batch's end, 0 if its offsets descend
  int* err;
};

// The claimed bits of filter f, whose particles start at lo: its bytes end before those of
// filter f + 1 start, (lo >> 3) + ceil(n / 8) <= ((lo + n) >> 3) + 1.
__device__ __forceinline__ uint8_t* claimed_bits(const Batch& b, int f, int64_t lo) {
  return b.cl ? b.cl + (lo >> 3) + f : nullptr;
}

// Filter f is resampled unless a flag array says otherwise (rs_resample_batched_masked).
__device__ __forceinline__ bool resampled(const uint8_t* flags, int f) {
  return flags == nullptr || __ldg(flags + f) != 0;
}

// Plan: tiles and segments per filter and their exclusive prefixes; per-filter maxima reset;
// offsets checked.
__global__ void __launch_bounds__(1024) batch_plan_kernel(Batch b) {
  pdl_wait();
  __shared__ int3 sh[32];  // (all 32 warps write theirs)
  const int F = b.F;
  const int chunk = (F + blockDim.x - 1) / blockDim.x;
  const int f0 = min(F, static_cast<int>(threadIdx.x) * chunk), f1 = min(F, f0 + chunk);
  const int64_t end = batch_end(b.off, F, b.max_n);
  auto counts = [&](int f) -> int2 {  // (tiles, segments) of filter f
    const int64_t n = filter_size(b.off, f, end);
    if (n < 0) return make_int2(0, 0);
    return make_int2(static_cast<int>((n + kTile - 1) / kTile),
                     static_cast<int>((n + kSeg - 1) / kSeg));
  };
  int2 local = make_int2(0, 0);
  int longest = 0;
  bool rejected = false, down = false;
  for (int f = f0; f < f1; ++f) {
    const int2 c = counts(f);
    local.x += c.x;
    local.y += c.y;
    longest = max(longest, c.y);
    b.fmax[f] = LLONG_MIN;
    rejected |= filter_size(b.off, f, end) < 0;
    down |= descends(b.off, f);
  }
  if (rejected) flag_error(b.err, RS_ERR_ARG);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  longest = __reduce_max_sync(0xffffffffu, longest);
  int2 incl = local;
#pragma unroll
  for (int dd = 1; dd < 32; dd <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, incl.x, dd);
    const int y = __shfl_up_sync(0xffffffffu, incl.y, dd);
    if (lane >= dd) {
      incl.x += x;
      incl.y += y;
    }
  }
  if (lane == 31) sh[warp] = make_int3(incl.x, incl.y, longest);
  down = __syncthreads_or(down);
  // (the sums of the warps before this one; the longest filter of all)
  const int3 w = sh[lane];
  int2 p = make_int2(__reduce_add_sync(0xffffffffu, lane < warp ? w.x : 0) + incl.x - local.x,
                     __reduce_add_sync(0xffffffffu, lane < warp ? w.y : 0) + incl.y - local.y);
  longest = __reduce_max_sync(0xffffffffu, w.z);
  if (down) p = make_int2(0, 0);
  for (int f = f0; f < f1; ++f) {
    b.tile_start[f] = p.x;
    b.seg_start[f] = p.y;
    if (down) continue;
    const int2 c = chunk == 1 ? local : counts(f);
    p.x += c.x;
    p.y += c.y;
  }
  if (f1 == F && f0 < F) {
    b.tile_start[F] = p.x;
    b.seg_start[F] = p.y;
  }
  if (threadIdx.x == 0) {
    b.seg_start[F + 1] = longest;
    *b.limit = down ? 0 : static_cast<int32_t>(end);
  }
}

// Locates batch tile t: its filter f, the filter's bounds and the tile's first particle.
struct TileLoc {
  int f;
  int t;       // tile index inside the filter
  int64_t lo, hi, base;
};
__device__ __forceinline__ bool locate_tile(const Batch& b, int tile, TileLoc& L) {
  if (tile >= __ldg(b.tile_start + b.F)) return false;
  L.f = filter_of_tile(b.tile_start, b.F, tile);
  L.t = tile - __ldg(b.tile_start + L.f);
  L.lo = __ldg(b.off + L.f);
  L.hi = __ldg(b.off + L.f + 1);
  L.base = L.lo + static_cast<int64_t>(L.t) * kTile;
  return true;
}

// Every slot of a tile claimed (cl: the filter's claimed bits, or null).
__device__ __forceinline__ void claim_all(uint8_t* cl, const TileLoc& L) {
  if (!cl) return;
  const int64_t i0 = L.base - L.lo;  // (a multiple of 8)
  const int64_t i1 = min(i0 + kTile, L.hi - L.lo);
  for (int64_t k = (i0 >> 3) + threadIdx.x; k < ((i1 + 7) >> 3); k += kBlock) cl[k] = 0xFFu;
}

template <typename T>
__global__ void __launch_bounds__(kBlock) batch_max_kernel(const T* __restrict__ lw, Batch b) {
  pdl_wait();
  __shared__ long long sh[kWarps];
  TileLoc L;
  if (!locate_tile(b, blockIdx.x, L)) return;
  if (!resampled(b.resample, L.f)) return;  // a filter that keeps its particles: no passes
  const bool vec = (reinterpret_cast<uintptr_t>(lw) & 15u) == 0;
  const int64_t end = min(L.hi, L.base + kTile);
  long long m = max_key(neg_inf<T>());
  bool bad = false;
  for (int64_t i0 = L.base + 4 * static_cast<int64_t>(threadIdx.x); i0 < end; i0 += 4 * kBlock) {
    T x[4];
    load4(lw, i0, L.lo, end, vec, x);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const bool nan = is_nan(x[q]);
      bad |= nan || is_pos_inf(x[q]);
      const long long k = max_key(x[q]);
      if (!nan && k > m) m = k;
    }
  }
  if (bad) flag_error(b.err, RS_ERR_NONFINITE);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long y = __shfl_xor_sync(0xffffffffu, m, o);
    m = y > m ? y : m;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) sh[warp] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long bm = sh[0];
    for (int k = 1; k < kWarps; ++k) bm = sh[k] > bm ? sh[k] : bm;
    // stored as the key of the binary64 value, comparable across both input types
    atomicMax(b.fmax + L.f, max_key(key_to_double(bm, T())));
  }
}

__device__ __forceinline__ double filter_M(const Batch& b, int f) {
  return key_to_double(__ldcg(b.fmax + f), 0.0);
}

template <typename T, typename V>
__global__ void __launch_bounds__(kBlock) batch_sum_kernel(const T* __restrict__ lw, Batch b) {
  pdl_wait();
  __shared__ float2 sh_tab[64];
  TileLoc L;
  if (!locate_tile(b, blockIdx.x, L)) return;
  if (!resampled(b.resample, L.f)) return;
  if (threadIdx.x < 64) sh_tab[threadIdx.x] = kExp2Frac64[threadIdx.x];
  __syncthreads();
  const bool vec = (reinterpret_cast<uintptr_t>(lw) & 15u) == 0;
  const int warp = threadIdx.x >> 5;
  bool bad = false;  // (the max pass flags non-finite input)
  long long ref = kTileMaxRef;
  if constexpr (!Path<T, V>::kTileRef) {
    const double M = filter_M(b, L.f);
    if (M > -DBL_MAX) ref = max_key(static_cast<T>(M));  // (records relative to M)
  }
  seg_record<T, V>(lw, L.lo, L.hi, L.base + kSeg * warp, sh_tab, vec,
                   b.s_rec + kWarps * blockIdx.x + warp, bad, ref);
}

template <typename T, typename V>
__global__ void __launch_bounds__(kBlock) batch_prefix_kernel(Batch b) {
  pdl_wait();
  const int f = blockIdx.x;
  const int64_t lo = b.off[f], hi = b.off[f + 1], n = hi - lo;
  const int t0 = b.tile_start[f], nt = b.tile_start[f + 1] - t0;
  if (nt <= 0 || n <= 0 || !resampled(b.resample, f)) return;
  if (!(filter_M(b, f) > -DBL_MAX)) {
    if (threadIdx.x == 0) {
      b.fSd[f] = 0.0;
      flag_error(b.err, RS_ERR_ZERO_WEIGHT);
    }
    return;
  }
  seg_prefix_compute<T, V>(b.s_rec + kWarps * t0, b.P_rec + kWarps * t0 + f, kWarps * nt, n,
                           static_cast<T>(filter_M(b, f)), reinterpret_cast<V*>(b.fS + f),
                           reinterpret_cast<V*>(b.fscale + f), b.fSd + f);
}

template <typename T, typename V, int SCHEME>
__global__ void __launch_bounds__(kBlock)
batch_emit_kernel(const T* __restrict__ lw, Batch b, Keys base_keys,
                  int32_t* __restrict__ a, int32_t* __restrict__ d, V* __restrict__ W) {
  pdl_wait();
  __shared__ SegSh sh;
  __shared__ float2 sh_tab[64];
  TileLoc L;
  if (!locate_tile(b, blockIdx.x, L)) return;
  const int64_t n = L.hi - L.lo;
  const double M = filter_M(b, L.f);
  const double Sd = __ldcg(b.fSd + L.f);
  // all weights zero (flagged), or a filter that is not resampled: the identity
  if (!resampled(b.resample, L.f) || !(M > -DBL_MAX) || !(Sd > 0.0)) {
    for (int64_t e = L.base + threadIdx.x; e < L.hi && e < L.base + kTile; e += kBlock) {
      a[e] = static_cast<int32_t>(e - L.lo);
      if (d) d[e] = static_cast<int32_t>(e - L.lo);
      if (W) W[e] = vzero(V());
    }
    claim_all(claimed_bits(b, L.f, L.lo), L);
    return;
  }
  const WeightCtx wc = make_ctx<T, V>(M, sh_tab);
  const bool vec = (reinterpret_cast<uintptr_t>(lw) & 15u) == 0;
  const int warp = threadIdx.x >> 5;
  const double2* P = b.P_rec + kWarps * __ldg(b.tile_start + L.f) + L.f;
  const int gl = kWarps * L.t + warp;  // this warp's segment within the filter
  const V Ps = load_v_cg<V>(P + gl), Pn = load_v_cg<V>(P + gl + 1);
  const int64_t base = L.base + kSeg * warp;
  if constexpr (SCHEME == RS_MULTINOMIAL) {
    if (d)  // claims of the search kernel start from the sentinel n
      for (int64_t e = L.base + threadIdx.x; e < L.hi && e < L.base + kTile; e += kBlock)
        d[e] = static_cast<int32_t>(n);
    emit_seg_W<T, V, V>(lw, L.lo, L.hi, base, wc, vec, Ps, Pn, W);
  } else {
    const Keys keys = with_tag(base_keys, static_cast<uint32_t>(L.f), SCHEME);
    const typename Path<T, V>::U u_sys =
        SCHEME == RS_STRATIFIED ? typename Path<T, V>::U() : cta_uniform0<T, V>(keys);
    emit_seg_cumoff<T, V, SCHEME == RS_STRATIFIED>(
        lw, L.lo, L.hi, base, wc, vec, Ps, Pn, load_v_cg<V>(b.fS + L.f),
        load_v_cg<V>(b.fscale + L.f), u_sys, keys, a, sh.win[warp],
        claimed_bits(b, L.f, L.lo));
  }
}

// ---------------------------------------------------------------------------------------
// The max, sum, prefix and emission passes of all filters in one cooperative launch (after the
// plan kernel). The unit of work is the segment, and each warp of the grid owns a contiguous
// range of the segments of all filters together (so filters of any sizes share the grid evenly);
// all passes but the prefixes of very long filters are warp-level work, and a filter's bounds,
// totals and uniform are looked up when a warp comes to a new filter. The phases meet at two
// grid barriers (three for compensated binary32, whose records follow the filter maxima):
//   phase 1  the records of the warp's segments (seg_record: the segment's maximum log-weight
//            and its weights' sum relative to it), last to first, and the filter maxima (an
//            atomic max of keys per warp and filter);
//   phase 2  per filter, one warp or, for a long one, a CTA: the exact sums of its records scaled to
//            its maximum, rounded once to the segment prefixes and W^N;
//   phase 3  the emission of the warp's segments, first to last (those phase 1 read last).
// Every segment goes through the same device functions and rounded prefixes as in the separate
// batched kernels and the single-filter kernels, so filter f still equals rs_resample on its
// slice with filter = f, bit for bit.
// ---------------------------------------------------------------------------------------
//
// The prefixes of one filter by one warp are a chain of steps of 32 records, which sets the length of
// phase 2 where the filters are few and long. So a CTA takes a filter from kFewPrefixSegs segments
// on where there are at most half as many filters as CTAs, from kSomePrefixSegs up to twice as many
// (20 filters of 30000 .. 100000: binary32 32.9 -> 22.7 us, binary64 61.4 -> 47.3; stratified
// binary64 over 256 of 16384 .. 262144: 525 -> 485; from 64 segments 500 of up to 20000 lost 2 of 25
// us), and many filters keep all warps busy.
constexpr int kWarpPrefixSegs = 1024;
constexpr int kSomePrefixSegs = 256;
constexpr int kFewPrefixSegs = 64;
constexpr int kOwnPrefixSegs = 512;

// Position of a warp in the batch: filter f and its bounds, segments [s0, s1) of the batch.
struct SegWalk {
  int f, s0, s1;
  int64_t lo, hi;
};
__device__ __forceinline__ void seg_enter(const Batch& b, int f, SegWalk& w) {
  w.f = f;
  w.s0 = __ldg(b.seg_start + f);
  w.s1 = __ldg(b.seg_start + f + 1);
  w.lo = __ldg(b.off + f);
  w.hi = __ldg(b.off + f + 1);
}

// Prefixes, total and N / total of filter f by one warp (the sums and roundings of
// seg_prefix_compute: exact in fixed point, each prefix rounded once).
template <typename T, typename V>
__device__ __forceinline__ void warp_prefix(const Batch& b, int f, int s0, int nseg, int64_t n,
                                            T M, const float2* tab) {
  const int lane = threadIdx.x & 31;
  double2* const P = b.P_rec + s0 + f;
  u128 carry = 0;
  for (int k0 = 0; k0 < nseg; k0 += 32) {
    const int k = k0 + lane;
    const u128 v = k < nseg ? rec_fixed<T, V>(b.s_rec + s0 + k, M, tab) : static_cast<u128>(0);
    u128 incl = v;
#pragma unroll
    for (int dd = 1; dd < 32; dd <<= 1) {
      const u128 y = shfl_up_u128(incl, dd);
      if (lane >= dd) incl += y;
    }
    if (k < nseg) store_v<V>(P + k, fixed_to(carry + (incl - v), V(), kFixFrac));
    const uint64_t hi = __shfl_sync(0xffffffffu, static_cast<uint64_t>(incl >> 64), 31);
    const uint64_t lo = __shfl_sync(0xffffffffu, static_cast<uint64_t>(incl), 31);
    carry += (static_cast<u128>(hi) << 64) | lo;
  }
  if (lane == 0) {
    const V S = fixed_to(carry, V(), kFixFrac);
    const double Sd = vto_double(S);
    store_v<V>(P + nseg, S);
    store_v<V>(b.fS + f, S);
    store_v<V>(b.fscale + f, vfrom_double(__ddiv_rn(static_cast<double>(n), Sd), V()));
    b.fSd[f] = Sd;
  }
}

// The same sums for one segment `own` of filter f, by the warp that emits it: its prefix Ps, the
// next one Pn, the total S and N / S (every lane gets them); the warp of the filter's first
// segment also stores the totals (for the search kernel).
template <typename T, typename V>
__device__ __forceinline__ void warp_own_prefix(const Batch& b, int f, int s0, int nseg, int own,
                                                int64_t n, T M, const float2* tab, V& Ps, V& Pn,
                                                V& S, V& scale) {
  u128 upto = 0, all = 0, mine = 0;  // (mine: the segment's own sum, in lane own mod 32)
  for (int k = threadIdx.x & 31; k < nseg; k += 32) {
    const u128 v = rec_fixed<T, V>(b.s_rec + s0 + k, M, tab);
    all += v;
    if (k <= own) upto += v;
    if (k == own) mine = v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    upto += shfl_xor_u128(upto, o);
    all += shfl_xor_u128(all, o);
  }
  const uint64_t mh = __shfl_sync(0xffffffffu, static_cast<uint64_t>(mine >> 64), own & 31);
  const uint64_t ml = __shfl_sync(0xffffffffu, static_cast<uint64_t>(mine), own & 31);
  const u128 before = upto - ((static_cast<u128>(mh) << 64) | ml);
  // one rounding for the three: each in a lane of its own
  const int lane = threadIdx.x & 31;
  const V r = fixed_to(lane == 0 ? before : lane == 1 ? upto : all, V(), kFixFrac);
  Ps = vshfl(r, 0);
  Pn = vshfl(r, 1);
  S = vshfl(r, 2);
  const double Sd = vto_double(S);
  scale = vfrom_double(__ddiv_rn(static_cast<double>(n), Sd), V());
  if (own == 0 && lane == 0) {
    store_v<V>(b.fS + f, S);
    store_v<V>(b.fscale + f, scale);
    b.fSd[f] = Sd;
  }
}

template <typename T, typename V, int SCHEME>
__global__ void __launch_bounds__(kBlock, 3)
batch_coop_kernel(const T* __restrict__ lw, Batch b, Keys base_keys, int32_t* __restrict__ a,
                  int32_t* __restrict__ d, V* __restrict__ W, GridBar* bar) {
  __shared__ SegSh sh;
  __shared__ float2 sh_tab[64];
  unsigned int target = 0;
  const int U = __ldcg(b.seg_start + b.F);  // segments of the batch
  const int warps = static_cast<int>(gridDim.x) * kWarps;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gw = static_cast<int>(blockIdx.x) * kWarps + warp;
  const int u0 = static_cast<int>(static_cast<int64_t>(gw) * U / warps);
  const int u1 = static_cast<int>(static_cast<int64_t>(gw + 1) * U / warps);
  const bool vec = (reinterpret_cast<uintptr_t>(lw) & 15u) == 0;
  if (threadIdx.x < 64) sh_tab[threadIdx.x] = kExp2Frac64[threadIdx.x];
  __syncthreads();

  // ---- phase 1: segment records -> filter maxima (compensated binary32: the maxima only) ----
  const int f_last = u1 > u0 ? filter_of_warp(b.seg_start, b.F, u1 - 1) : 0;
  auto records = [&](bool with_max) {
    SegWalk w;
    bool bad = false, on = false;
    long long fm = LLONG_MIN;  // the running maximum of the current filter's segments
    long long ref = kTileMaxRef;
    for (int u = u1 - 1; u >= u0; --u) {
      if (u == u1 - 1 || u < w.s0) {
        if (u < u1 - 1) {
          if (with_max && on && lane == 0) atomicMax(b.fmax + w.f, max_key(key_to_double(fm, T())));
          int f = w.f - 1;
          while (__ldg(b.seg_start + f) > u) --f;  // (empty filters)
          seg_enter(b, f, w);
        } else {
          seg_enter(b, f_last, w);
        }
        on = resampled(b.resample, w.f);
        fm = max_key(neg_inf<T>());
        if (!with_max) {
          const double M = filter_M(b, w.f);
          ref = M > -DBL_MAX ? max_key(static_cast<T>(M)) : kTileMaxRef;
        }
      }
      if (!on) continue;  // a filter that keeps its particles: no passes
      const int64_t base = w.lo + static_cast<int64_t>(u - w.s0) * kSeg;
      long long k;
      if (Path<T, V>::kTileRef || !with_max) {
        k = seg_record<T, V>(lw, w.lo, w.hi, base, sh_tab, vec, b.s_rec + u, bad, ref,
                             L2Hint::kEvictLast);
      } else {
        T x[kPer];
        load_per(lw, base + kPer * static_cast<int64_t>(lane), w.lo, w.hi, vec, x,
                 L2Hint::kEvictLast);
        k = max_key(neg_inf<T>());
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
          const bool nan = is_nan(x[q]);
          bad |= nan || is_pos_inf(x[q]);
          const long long kq = max_key(x[q]);
          if (!nan && kq > k) k = kq;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const long long y = __shfl_xor_sync(0xffffffffu, k, o);
          k = y > k ? y : k;
        }
      }
      fm = k > fm ? k : fm;
    }
    // (stored as the key of the binary64 value, comparable across both input types)
    if (with_max && on && lane == 0) atomicMax(b.fmax + w.f, max_key(key_to_double(fm, T())));
    if (with_max && bad) flag_error(b.err, RS_ERR_NONFINITE);
  };
  records(true);
  grid_barrier(bar, target, b.err);
  if constexpr (!Path<T, V>::kTileRef) {
    records(false);
    grid_barrier(bar, target, b.err);
  }

  // ---- phase 2: per filter, the exact prefixes of its segments and its total -----------------
  // Small batches (a segment per warp at most, no filter above kOwnPrefixSegs segments) skip it and
  // its barrier: every warp sums its filter's records itself (without Permute, 78 filters of up to
  // 23655: 18.6 -> 16.2 us, 64 of up to 65536: 24.7 -> 19.9, with 64 segments as the most before).
  const bool own_prefix = U <= warps && __ldcg(b.seg_start + b.F + 1) <= kOwnPrefixSegs;
  const int G = static_cast<int>(gridDim.x);
  const int cta_segs = 2 * b.F <= G   ? kFewPrefixSegs
                       : b.F <= 2 * G ? kSomePrefixSegs
                                      : kWarpPrefixSegs;
  for (int pass = 0; pass < 2 && !own_prefix; ++pass) {  // (by warps; then the longer filters by CTAs)
    for (int f = pass == 0 ? gw : static_cast<int>(blockIdx.x); f < b.F;
         f += pass == 0 ? warps : static_cast<int>(gridDim.x)) {
      const int s0 = __ldg(b.seg_start + f), nseg = __ldg(b.seg_start + f + 1) - s0;
      if (nseg == 0 || (nseg >= cta_segs) != (pass == 1) || !resampled(b.resample, f)) continue;
      const double M = filter_M(b, f);
      if (!(M > -DBL_MAX)) {
        if (pass == 0 ? lane == 0 : threadIdx.x == 0) {
          b.fSd[f] = 0.0;
          flag_error(b.err, RS_ERR_ZERO_WEIGHT);
        }
        continue;
      }
      const int64_t n = __ldg(b.off + f + 1) - __ldg(b.off + f);
      if (pass == 0)
        warp_prefix<T, V>(b, f, s0, nseg, n, static_cast<T>(M), sh_tab);  // (exact: M is a log-weight)
      else
        seg_prefix_compute<T, V>(b.s_rec + s0, b.P_rec + s0 + f, nseg, n, static_cast<T>(M),
                                 reinterpret_cast<V*>(b.fS + f),
                                 reinterpret_cast<V*>(b.fscale + f), b.fSd + f);
    }
  }
  if (!own_prefix) grid_barrier(bar, target, b.err);

  // ---- phase 3: emission ---------------------------------------------------------------------
  SegWalk w;
  bool live = false;
  WeightCtx wc;
  V S = vzero(V()), scale = vzero(V()), Ps = vzero(V()), Pn = vzero(V());
  typename Path<T, V>::U u_sys = typename Path<T, V>::U();
  for (int u = u0; u < u1; ++u) {
    if (u == u0 || u >= w.s1) {
      int f = u == u0 ? filter_of_warp(b.seg_start, b.F, u0) : w.f + 1;
      while (__ldg(b.seg_start + f + 1) <= u) ++f;  // (empty filters)
      seg_enter(b, f, w);
      const double M = filter_M(b, f);
      // all weights zero (flagged), or a filter that is not resampled: the identity
      live = resampled(b.resample, f);
      if (own_prefix && live && !(M > -DBL_MAX) && u == w.s0 && lane == 0) {
        b.fSd[f] = 0.0;
        flag_error(b.err, RS_ERR_ZERO_WEIGHT);
      }
      live = live && M > -DBL_MAX;
      if (live && own_prefix) {
        warp_own_prefix<T, V>(b, f, w.s0, w.s1 - w.s0, u - w.s0, w.hi - w.lo, static_cast<T>(M),
                              sh_tab, Ps, Pn, S, scale);
      } else if (live) {
        S = load_v_cg<V>(b.fS + f);
        scale = load_v_cg<V>(b.fscale + f);
      }
      live = live && vto_double(S) > 0.0;
      wc = ctx_staged<T, V>(live ? M : 0.0, sh_tab);  // (the table was staged at the start)
      if (live) {
        if constexpr (SCHEME == RS_SYSTEMATIC)
          u_sys = Path<T, V>::draw_u(
              draw(with_tag(base_keys, static_cast<uint32_t>(f), SCHEME), 0u, 0u));
      }
    }
    const int64_t base = w.lo + static_cast<int64_t>(u - w.s0) * kSeg;
    uint8_t* const cl = claimed_bits(b, w.f, w.lo);
    if (!live) {
      const int64_t end = min(w.hi, base + kSeg);
      for (int64_t e = base + lane; e < end; e += 32) {
        a[e] = static_cast<int32_t>(e - w.lo);
        if (d) d[e] = static_cast<int32_t>(e - w.lo);
        if (W) W[e] = vzero(V());
      }
      if (cl && base - w.lo + 8 * lane < end - w.lo) cl[((base - w.lo) >> 3) + lane] = 0xFFu;
      continue;
    }
    if (!own_prefix) {
      Ps = load_v_cg<V>(b.P_rec + u + w.f);
      Pn = load_v_cg<V>(b.P_rec + u + w.f + 1);
    }
    if constexpr (SCHEME == RS_MULTINOMIAL) {
      if (d) {  // claims of the search kernel start from the sentinel n
        const int32_t n = static_cast<int32_t>(w.hi - w.lo);
        for (int64_t e = base + lane; e < w.hi && e < base + kSeg; e += 32) d[e] = n;
      }
      emit_seg_W<T, V, V>(lw, w.lo, w.hi, base, wc, vec, Ps, Pn, W);
    } else {
      emit_seg_cumoff<T, V, SCHEME == RS_STRATIFIED>(
          lw, w.lo, w.hi, base, wc, vec, Ps, Pn, S, scale, u_sys,
          with_tag(base_keys, static_cast<uint32_t>(w.f), SCHEME), a, sh.win[warp], cl,
          L2Hint::kEvictFirst);
    }
  }
  grid_exit(bar, target);
}

template <typename T, typename V>
__global__ void __launch_bounds__(kBlock)
batch_search_kernel(const V* __restrict__ W, Batch b, int64_t total, Keys base_keys,
                    int32_t* __restrict__ a, int32_t* __restrict__ d) {
  pdl_wait();
  const int64_t g = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  PartLoc P;
  if (g >= total || !locate_particle(b.off, b.F, b.max_n, g, P)) return;
  if (!resampled(b.resample, P.f) || !(__ldcg(b.fSd + P.f) > 0.0) ||
      !(filter_M(b, P.f) > -DBL_MAX))
    return;  // the identity, written by the emission kernel
  const Keys keys = with_tag(base_keys, static_cast<uint32_t>(P.f), RS_MULTINOMIAL);
  const int32_t k = search_one<T, V>(W + P.lo, P.n, keys, P.i);
  a[g] = k;
  if (d) atomicMin(d + P.lo + k, static_cast<int32_t>(P.i));
}

// The claims' sentinels: d[g] = n of particle g's filter, for the positions [g0, g0 + 256) of one
// warp (eight consecutive per lane), whose filter is looked up once; across a filter boundary
// each position's filter is found by stepping past the offsets it crosses. Positions that
// locate_in rejects get nothing.
constexpr int kFillPer = 8;
__device__ __forceinline__ void fill_sentinels_warp(const int64_t* __restrict__ off, int F,
                                                    int64_t end, int64_t gw,
                                                    int32_t* __restrict__ d) {
  if (gw >= end) return;  // (uniform over the warp)
  int f = filter_of_warp(off, F, gw);
  const int64_t g0 = gw + kFillPer * static_cast<int64_t>(threadIdx.x & 31);
  PartLoc P;
  if (locate_in(off, f, end, gw, P) && P.i + 32 * kFillPer <= P.n && gw + 32 * kFillPer <= end &&
      (reinterpret_cast<uintptr_t>(d + g0) & 15u) == 0) {
    const int32_t n = static_cast<int32_t>(P.n);
    int4* const p4 = reinterpret_cast<int4*>(d + g0);
    p4[0] = make_int4(n, n, n, n);
    p4[1] = make_int4(n, n, n, n);
    return;
  }
  for (int q = 0; q < kFillPer; ++q) {
    const int64_t g = g0 + q;
    if (g >= end) break;
    f = advance_filter(off, F, g, f);
    if (locate_in(off, f, end, g, P)) d[g] = static_cast<int32_t>(P.n);
  }
}

// Metropolis steps of filter f (a negative B counts as 0; flagged by the plan).
__device__ __forceinline__ int32_t filter_steps(const int32_t* __restrict__ Bf, int32_t B, int f) {
  const int32_t v = Bf ? __ldg(Bf + f) : B;
  return v < 0 ? 0 : v;
}

// Work of one particle of the batched chains, in units of a chain's step: its B steps and what a
// particle costs besides (its first draw products, log-weight, result and claim).
constexpr int kParticleSteps = 8;
__device__ __forceinline__ unsigned long long particle_work(const uint8_t* flags,
                                                            const int32_t* __restrict__ Bf,
                                                            int32_t B, int f) {
  return resampled(flags, f) ? static_cast<unsigned long long>(filter_steps(Bf, B, f)) + kParticleSteps
                             : 2ull;
}

// Plan of the per-particle schemes (CTA 0): the batch's end (limit: 0 if its offsets descend) and,
// with work given (the staged chains), the exclusive prefix over the filters of their work,
// work[0 .. F], and the chunk counter reset; rejected filters and negative B are flagged and get no
// work. The other CTAs write the claims' sentinels (d given).
constexpr int kChainBlock = 1024;
__global__ void __launch_bounds__(kChainBlock)
batch_chain_plan_kernel(const int64_t* __restrict__ off, int F, int64_t total,
                        const int32_t* __restrict__ Bf, int32_t B,
                        const uint8_t* __restrict__ flags, unsigned long long* work,
                        unsigned int* counter, int32_t* __restrict__ d, int32_t* limit, int* err) {
  pdl_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t end = batch_end(off, F, total);
  if (blockIdx.x > 0) {
    const int64_t warps = static_cast<int64_t>(gridDim.x - 1) * (kChainBlock / 32);
    for (int64_t w = static_cast<int64_t>(blockIdx.x - 1) * (kChainBlock / 32) + warp;
         w * (32 * kFillPer) < end; w += warps)
      fill_sentinels_warp(off, F, end, w * (32 * kFillPer), d);
    return;
  }
  __shared__ unsigned long long sh[kChainBlock / 32];
  const int chunk = (F + kChainBlock - 1) / kChainBlock;
  const int f0 = min(F, static_cast<int>(threadIdx.x) * chunk), f1 = min(F, f0 + chunk);
  auto filter_work = [&](int f) -> unsigned long long {  // (~0: rejected)
    const int64_t n = filter_size(off, f, end);
    return n < 0 ? ~0ull : static_cast<unsigned long long>(n) * particle_work(flags, Bf, B, f);
  };
  unsigned long long local = 0;
  bool down = false, rejected = false;
  for (int f = f0; f < f1; ++f) {
    down |= descends(off, f);
    if (!work) continue;  // (the other kernels check the filter of each of their particles)
    const unsigned long long w = filter_work(f);
    if (w != ~0ull) local += w;
    rejected |= w == ~0ull || (w > 0 && resampled(flags, f) && (Bf ? __ldg(Bf + f) : B) < 0);
  }
  // (positions before the first filter belong to none: the other kernels report them too)
  if (work && threadIdx.x == 0) rejected |= end > 0 && __ldg(off) > 0;
  if (rejected) flag_error(err, RS_ERR_ARG);
  unsigned long long incl = local;
#pragma unroll
  for (int dd = 1; dd < 32; dd <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, dd);
    if (lane >= dd) incl += y;
  }
  if (lane == 31) sh[warp] = incl;
  down = __syncthreads_or(down);
  if (threadIdx.x == 0) *limit = down ? 0 : static_cast<int32_t>(end);
  if (!work) return;
  unsigned long long p = incl - local;
  for (int k = 0; k < warp; ++k) p += sh[k];
  if (down) p = 0;
  for (int f = f0; f < f1; ++f) {
    work[f] = p;
    const unsigned long long w = filter_work(f);
    if (w != ~0ull && !down) p += w;
  }
  if (f1 == F && f0 < F) work[F] = p;
  if (threadIdx.x == 0) *counter = 0u;
}

// ---------------------------------------------------------------------------------------
// Metropolis chains of all filters with the log-weights in shared memory.
//
// A chain's proposals are random 4-byte reads of its filter's log-weights. With one thread per
// particle and CTAs of any filter on an SM, half of those reads missed L1 and the kernel ran at
// the L2's rate of random sectors (4096 filters of 256 .. 65536 particles, 2.5 G steps: 5.3 ms).
// Here one CTA of 1024 threads per SM stages the log-weights of a window of whole filters (up to
// kChainCap values, 224 KB; of a longer filter the first kChainCap, the rest is read from
// memory) and runs the chains of its particles from there (4.05 ms: 42 instructions and 61 cycles
// a step on each SM quarter, of which the 8 wide products of its half Philox block and the
// product of its index take about 45 in the multiplier: 5 and 4 cycles each, measured).
//
// The particles of the batch are cut into chunks of equal work (steps plus kParticleSteps a
// particle, batch_chain_plan_kernel), taken in order from a counter: the first half of the
// chunks covers 9/10 of the work, the second half the rest, so that the last one to end is
// short. A chunk holds whole turns of the CTA's 1024 chains where it can: the end of a window
// waits for its slowest warp (32 chunks per CTA instead of 16: 4.65 against 4.51 ms a call). Inside
// a window every warp takes the next 32 particles from a shared counter (filters of one window may
// differ in B). Every particle's chain and claim are those of batch_mcmc_kernel.
// ---------------------------------------------------------------------------------------
static_assert(kBatchMaxN < (1 << 24), "half_index<true>");
constexpr int kChainCap = 57344;                            // staged log-weights
constexpr size_t kChainSmem = sizeof(float) * (kChainCap + 4);  // (+ the alignment shift)
constexpr int kChainBlocks = 2;                             // blocks of a chain drawn together
constexpr int kChainChunks = 16;                            // chunks per CTA, at most

__global__ void __launch_bounds__(kChainBlock, 1)
batch_chain_kernel(const float* __restrict__ lw, const int64_t* __restrict__ off, int F,
                   int64_t total, const int32_t* __restrict__ Bf, int32_t B, Keys base_keys,
                   const uint8_t* __restrict__ flags,
                   const unsigned long long* __restrict__ work, unsigned int* counter,
                   int32_t* __restrict__ a, int32_t* __restrict__ d, int* err) {
  pdl_wait();
  extern __shared__ __align__(16) float sh_lw[];
  __shared__ unsigned int sh_chunk, sh_group;
  __shared__ int sh_f[2], sh_i[2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned long long W = __ldg(work + F);
  if (W == 0) return;
  // chunks: four turns of the CTA's threads each where there are (one turn: 243 against 175 us for
  // 150 filters of 256 .. 65536, the chunks of the highest B too few chains for the CTA), at
  // least one per CTA
  const unsigned long long G = gridDim.x;
  unsigned long long K = static_cast<unsigned long long>(batch_end(off, F, total)) / (4 * kChainBlock);
  K = K < G ? G : K > kChainChunks * G ? kChainChunks * G : K;
  const bool tapered = K >= 8 * G;  // (fewer chunks: all alike)
  const unsigned long long K1 = tapered ? K / 2 : K, W1 = tapered ? W / 10 * 9 : W;
  for (;;) {
    __syncthreads();  // (the previous chunk's shared state has been read)
    if (threadIdx.x == 0) sh_chunk = atomicAdd(counter, 1u);
    __syncthreads();
    const unsigned long long c = sh_chunk;
    if (c >= K) return;
    if (warp < 2) {  // the chunk's first particle (warp 0) and the next chunk's (warp 1)
      const unsigned long long b = c + warp;
      const unsigned long long X = b < K1 ? W1 / K1 * b : b < K ? W1 + (W - W1) / (K - K1) * (b - K1)
                                                               : W;
      int f = F, i = 0;
      if (X < W) {
        f = filter_of_warp(work, F, X);
        // whole turns of the CTA's threads where a chunk holds several, else whole warps
        const unsigned long long per = particle_work(flags, Bf, B, f);
        const int turn = W / K >= 4 * kChainBlock * per ? kChainBlock : 32;
        i = static_cast<int>((X - __ldg(work + f)) / per) & -turn;
      }
      if (lane == 0) {
        sh_f[warp] = f;
        sh_i[warp] = i;
      }
    }
    __syncthreads();
    int f = sh_f[0], i = sh_i[0];
    const int fe = sh_f[1], ie = sh_i[1];
    while (f < fe || (f == fe && i < ie)) {  // one window of filters (uniform over the CTA)
      if (__ldg(work + f + 1) == __ldg(work + f)) {  // empty or malformed: no particles
        ++f;
        i = 0;
        continue;
      }
      const ChainWindow w = chain_window(off, total, f, i, fe, ie, kChainCap);
      const int64_t lo = w.lo;
      const int f1 = w.f1, staged = w.staged;
      const int pad = static_cast<int>(lo & 3);  // shared index = particle - lo + pad
      __syncthreads();  // (the previous window has been read)
      if (threadIdx.x == 0) sh_group = 0u;
      if ((reinterpret_cast<uintptr_t>(lw) & 15u) == 0) {  // 128-bit loads of whole quadruples
        const float4* const src = reinterpret_cast<const float4*>(lw + (lo - pad));
        const int q1 = (staged + pad) >> 2;  // quadruples that end inside the window
        float4* const dst = reinterpret_cast<float4*>(sh_lw);
#pragma unroll 4
        for (int q = threadIdx.x; q < q1; q += kChainBlock) dst[q] = __ldg(src + q);
        for (int e = 4 * q1 + threadIdx.x; e < staged + pad; e += kChainBlock)
          if (e >= pad) sh_lw[e] = __ldg(lw + (lo - pad) + e);
      } else {
        for (int e = threadIdx.x; e < staged; e += kChainBlock) sh_lw[e + pad] = __ldg(lw + lo + e);
      }
      __syncthreads();
      const int64_t ps = w.ps, pe = w.pe;
      for (;;) {
        unsigned int grp = 0;
        if (lane == 0) grp = atomicAdd(&sh_group, 1u);
        grp = __shfl_sync(0xffffffffu, grp, 0);
        const int64_t gw = ps + 32 * static_cast<int64_t>(grp);
        if (gw >= pe) break;
        const int64_t g = gw + lane;
        if (g < pe) {
          int ff = f;
          if (f1 > f) ff = f + filter_of(off + f, f1 + 1 - f, g);
          PartLoc P;
          if (locate_in(off, ff, total, g, P)) {
            const uint32_t un = static_cast<uint32_t>(P.n), ui = static_cast<uint32_t>(P.i);
            const float* const sw = sh_lw + (pad + static_cast<int>(P.lo - lo));
            int32_t k = static_cast<int32_t>(P.i);  // (not resampled: keeps its particle)
            if (resampled(flags, ff) && in_window(w, P)) {
              const int32_t Bv = filter_steps(Bf, B, ff);
              const Keys keys = with_tag(base_keys, static_cast<uint32_t>(ff), RS_METROPOLIS);
              const float lwi = __ldg(lw + g);
              if (nonfinite_logw(lwi)) flag_error(err, RS_ERR_NONFINITE);
              const float* const lf = lw + P.lo;
              auto all = [&](uint32_t j) { return sw[j]; };
              auto part = [&](uint32_t j) {
                return j < static_cast<uint32_t>(kChainCap) ? sw[j] : __ldg(lf + j);
              };
              k = w.whole
                      ? metropolis_chain<true, kChainBlocks, false>(lwi, all, un, Bv, keys, ui)
                      : metropolis_chain<true, kChainBlocks, false>(lwi, part, un, Bv, keys, ui);
            }
            a[g] = k;
            if (d) atomicMin(d + P.lo + k, static_cast<int32_t>(P.i));
          }
        }
        __syncwarp();
      }
      f = f1 + 1;
      i = 0;
    }
  }
}

// First particle of item q of this thread when each CTA covers blockDim.x * ipt consecutive
// particles, item q being the q-th blockDim.x-wide slice (coalesced for every q).
__device__ __forceinline__ int64_t item_index(int ipt, int q) {
  return (static_cast<int64_t>(blockIdx.x) * ipt + q) * blockDim.x + threadIdx.x;
}

// Metropolis over the particles of all filters, ipt particles per thread, one thread per particle
// (the launch shape is tunable; every particle's chain and claim are the same for any shape).
template <typename T>
__global__ void __launch_bounds__(kMaxTunedBlock, 2)
batch_mcmc_kernel(const T* __restrict__ lw, const int64_t* __restrict__ off, int F,
                  int64_t total, const int32_t* __restrict__ Bf, int32_t B, Keys base_keys,
                  const uint8_t* __restrict__ flags, int32_t* __restrict__ a,
                  int32_t* __restrict__ d, int ipt, int* err) {
  pdl_wait();
  flag_descending(off, F, err);
  for (int q = 0; q < ipt; ++q) {
    const int64_t g = item_index(ipt, q);
    if (g >= total) return;
    PartLoc P;
    if (!locate_particle(off, F, total, g, P)) {
      if (g < __ldg(off + F)) flag_error(err, RS_ERR_ARG);
      continue;
    }
    int32_t k;
    if (!resampled(flags, P.f)) {
      k = static_cast<int32_t>(P.i);  // the filter keeps its particles
    } else {
      int32_t Bv = Bf ? __ldg(Bf + P.f) : B;
      if (Bv < 0) {
        flag_error(err, RS_ERR_ARG);
        Bv = 0;
      }
      const Keys keys = with_tag(base_keys, static_cast<uint32_t>(P.f), RS_METROPOLIS);
      if constexpr (sizeof(T) == 4) k = metropolis_one<true, 2>(lw + P.lo, P.n, Bv, keys, P.i, err);
      else k = metropolis_one(lw + P.lo, P.n, Bv, keys, P.i, err);
    }
    a[g] = k;
    if (d) atomicMin(d + P.lo + k, static_cast<int32_t>(P.i));
  }
}

// Rejection over the particles of all filters (mcmc.cuh), a warp per run of consecutive particles (at
// most 32: a lane each), every lane looking up the filter of its particle; the lanes make attempts
// of their own while more than half of them are busy and share the rest (rejection_tail). Runs of
// 32; of 8 where the batch has fewer than kRejSmallBatch particles, whose warps share them among
// their lanes from the start (64 filters of 256 .. 4096: 40 against 61 us; 2000 of 256 .. 40000: 2398
// against 1451; runs of 64 and 256 before the lanes share: 134 and 288 us against 108 for 200
// filters of up to 20000). The batch's size is known on the device only: the grid covers the
// handle's capacity up to kRejCtas CTAs per SM; larger handles get kRejTurnCtas per SM that take the
// runs in turns (TURNS), so that a small batch on them gets few idle CTAs (64 filters of up to 4096
// on a handle of 2^24: 71.9 -> 45.3 us with Permute). Bound by the latency of the longest particles
// and the gathers of the others.
constexpr int64_t kRejSmallBatch = int64_t{1} << 18;
constexpr int kRejCtas = 256;
constexpr int kRejTurnCtas = 64;
template <typename T, bool TURNS>
__global__ void __launch_bounds__(kBlock, sizeof(T) == 8 ? 4 : 5)
batch_rejection_kernel(const T* __restrict__ lw, const int64_t* __restrict__ off, int F,
                       int64_t total, Keys base_keys, double log_wmax, int64_t max_trials,
                       const uint8_t* __restrict__ flags, int32_t* __restrict__ a,
                       int32_t* __restrict__ d, int* err) {
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int64_t limit = batch_end(off, F, total);
  const int lg = limit < kRejSmallBatch ? 3 : 5;  // (log2 of the run length)
  const int runs = static_cast<int>((limit + (1 << lg) - 1) >> lg);
  flag_descending(off, F, err);
  const RejBound rb = make_bound(log_wmax);
  for (int run = static_cast<int>((blockIdx.x * blockDim.x + threadIdx.x) >> 5); run < runs;
       run += TURNS ? static_cast<int>((gridDim.x * blockDim.x) >> 5) : runs) {  // uniform over the warp
    const int64_t g = (static_cast<int64_t>(run) << lg) + lane;
    PartLoc P;
    Keys keys = base_keys;
    T lwi = T(0);
    bool active = lane < (1 << lg) && g < limit;
    if (active && !locate_in(off, filter_of(off, F, g), limit, g, P)) {
      flag_error(err, RS_ERR_ARG);
      active = false;
    }
    if (active) {
      keys = with_tag(base_keys, static_cast<uint32_t>(P.f), RS_REJECTION);
      lwi = __ldg(lw + g);
      if (nonfinite_logw(lwi)) flag_error(err, RS_ERR_NONFINITE);
      if (!resampled(flags, P.f)) {  // the particle's filter is not resampled: it keeps its place
        a[g] = static_cast<int32_t>(P.i);
        if (d) atomicMin(d + g, static_cast<int32_t>(P.i));
        active = false;
      }
    }
    uint64_t s = 0;  // attempts made (max_trials < 2^32, but s + kRejBatch may pass 2^32)
    while (__popc(__ballot_sync(0xffffffffu, active)) > 16) {
      if (!active) continue;
      int64_t j = P.i;
      bool over = false;
      bool settled = rejection_attempts<kRejBatch>(lw + P.lo, P.n, rb, keys, P.i,
                                                   static_cast<uint32_t>(s), lwi, max_trials, j, over);
      s += kRejBatch;
      if (!settled && s >= static_cast<uint64_t>(max_trials)) {
        flag_error(err, RS_ERR_REJECTION_CAP);
        j = P.i;
        settled = true;
      }
      if (settled) {
        if (over) flag_error(err, RS_ERR_BOUND_VIOLATED);
        a[g] = static_cast<int32_t>(j);
        if (d) atomicMin(d + P.lo + j, static_cast<int32_t>(P.i));
        active = false;
      }
    }
    RejParticle<T> own{active, 0u, 1u, 0u, 0, s, lwi};
    if (active) {
      own.i = static_cast<uint32_t>(P.i);
      own.n = static_cast<uint32_t>(P.n);
      own.tag = keys.tag;
      own.lo = P.lo;
    }
    rejection_tail<T>(
        own, max_trials, err,
        [&](const RejParticle<T>& R, uint32_t from, int64_t& j, bool& over) {
          Keys rk = base_keys;
          rk.tag = R.tag;
          return rejection_attempts<kRejBatch>(lw + R.lo, R.n, rb, rk, R.i, from, R.lwi, max_trials, j,
                                               over);
        },
        [&](const RejParticle<T>& R, int64_t j) {
          a[R.lo + R.i] = static_cast<int32_t>(j);
          if (d) atomicMin(d + R.lo + j, static_cast<int32_t>(R.i));
        });
  }
}

// Permute of every filter: each warp takes 32 K consecutive slots of the batch, ipt times
// (tunable launch shape). Nearly every warp lies inside one filter: its filter is
// looked up once per warp and its slots run as in the single-filter kernels (permute4_slots;
// SORTED: permute_sorted_slots, the non-decreasing ancestries of stratified and systematic from
// the claimed bits cl of their emission, filter f's bytes at (offsets[f] >> 3) + f). A warp that
// meets a filter boundary takes its slots one by one. Bound by L2 latency of the claims and
// walks, as in the single-filter kernels; looking the filter up per slot instead (a binary
// search of the offsets each) took 350 instructions per slot.
//
// K slots per lane: four for large batches; one for small ones, where it keeps more threads in
// flight (50 filters of up to 5000: 30.8 against 34.9 us a call). The batch's size is known on the
// device only, where the form is chosen; the grid covers the handle's capacity in either form. (By
// the capacity, multinomial over 64 filters of up to 4096 took 26.8 us on a handle of 2^20 instead
// of 24.7; two forms in one kernel cost multinomial over 2000 filters 1 %, 350.6 -> 354.2.) LARGE:
// the handle holds batches of the size for four slots.
constexpr int64_t kBatchSorted4MinN = int64_t{1} << 18;
constexpr int64_t kBatchPermute4MinN = int64_t{1} << 20;
template <bool SORTED> constexpr int64_t permute4_min_n() {
  return SORTED ? kBatchSorted4MinN : kBatchPermute4MinN;
}
constexpr size_t kPermSmemPerWarp = 128 * (sizeof(int2) + sizeof(int32_t));
template <bool SORTED, int K>
__device__ __forceinline__ void batch_permute_slots(const int64_t* __restrict__ off, int F,
                                                    int64_t total, int64_t end,
                                                    const int32_t* __restrict__ a,
                                                    const int32_t* __restrict__ d,
                                                    const uint8_t* __restrict__ cl,
                                                    int32_t* __restrict__ c, int ipt, int32_t* cw,
                                                    int2* pend, int* err) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int q = 0; q < ipt; ++q) {
    // first slot of this warp (of this lane: K * lane further)
    const int64_t gw = K * ((static_cast<int64_t>(blockIdx.x) * ipt + q) * blockDim.x +
                            32 * static_cast<int64_t>(warp));
    if (gw >= end) return;  // (uniform over the warp)
    const int f = filter_of_warp(off, F, gw);
    const int64_t g0 = gw + K * lane;
    PartLoc P;
    const bool ok = locate_in(off, f, total, gw, P);  // (uniform over the warp)
    if (ok && P.i + 32 * K <= P.n) {
      if constexpr (SORTED)
        permute_sorted_slots<K>(a + P.lo, cl + (P.lo >> 3) + f, P.n, c + P.lo, g0 - P.lo, cw, pend,
                                err);
      else if constexpr (K == 4)
        permute4_slots(a + P.lo, d + P.lo, P.n, c + P.lo, g0 - P.lo, pend, err);
      else
        permute_one(a + P.lo, d + P.lo, P.n, c + P.lo, g0 - P.lo, err);
      __syncwarp();  // (the warp's shared lists are rewritten by its next slots)
      continue;
    }
    int fs = f;
    for (int k = 0; k < K; ++k) {
      const int64_t g = g0 + k;
      if (g >= end) break;
      fs = advance_filter(off, F, g, fs);
      if (!locate_in(off, fs, total, g, P)) continue;
      if constexpr (SORTED)
        permute_sorted_one(a + P.lo, cl + (P.lo >> 3) + fs, P.n, c + P.lo, P.i, err);
      else
        permute_one(a + P.lo, d + P.lo, P.n, c + P.lo, P.i, err);
    }
  }
}
template <bool SORTED, bool LARGE>
__global__ void __launch_bounds__(kMaxTunedBlock)
batch_permute_kernel(const int64_t* __restrict__ off, int F, int64_t total,
                     const int32_t* __restrict__ a, const int32_t* __restrict__ d,
                     const uint8_t* __restrict__ cl, int32_t* __restrict__ c, int ipt,
                     const int32_t* limit, int* err) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char sh_perm[];
  int32_t* const cw = reinterpret_cast<int32_t*>(sh_perm + (threadIdx.x >> 5) * kPermSmemPerWarp);
  int2* const pend = reinterpret_cast<int2*>(cw + 128);
  const int64_t end = __ldg(limit);  // (0: the offsets descend, no ancestors were formed)
  if (LARGE && end >= permute4_min_n<SORTED>())
    batch_permute_slots<SORTED, 4>(off, F, total, end, a, d, cl, c, ipt, cw, pend, err);
  else
    batch_permute_slots<SORTED, 1>(off, F, total, end, a, d, cl, c, ipt, cw, pend, err);
}

// Total number of particles of the batch (offsets[F]) is not known on the host without a
// synchronisation, so grids are sized for the handle's capacity and surplus CTAs exit at once.
inline int grid_particles(int64_t cap) { return static_cast<int>((cap + kBlock - 1) / kBlock); }
inline int grid_shaped(int64_t cap, const LaunchCfg& c) {
  const int64_t per = static_cast<int64_t>(c.block) * c.ipt;
  return static_cast<int>((cap + per - 1) / per);
}

// CTAs that write the claims' sentinels beside the plan: 32 warps each, 256 positions a warp and
// turn, two CTAs per SM at most.
inline int fill_grid(int64_t cap) {
  const int64_t want = (cap + 32 * kFillPer * (kChainBlock / 32) - 1) /
                       (32 * kFillPer * (kChainBlock / 32));
  const int64_t most = 2 * static_cast<int64_t>(device_sm_count());
  return static_cast<int>(want < most ? want : most);
}

// Whether the current device grants batch_chain_kernel its shared memory (asked once per device).
inline bool chain_available() {
  static std::mutex mu;
  static int known[64] = {};  // 0: not asked, 1: yes, 2: no
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  std::lock_guard<std::mutex> lock(mu);
  if (known[dev] == 0) {
    const cudaError_t e = cudaFuncSetAttribute(
        batch_chain_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kChainSmem));
    if (e != cudaSuccess) cudaGetLastError();  // (not an error of the call: the other kernel runs)
    known[dev] = e == cudaSuccess ? 1 : 2;
  }
  return known[dev] == 1;
}

const char* const kLblSum[4] = {"batch_sum_f32", "batch_sum_f32c", "batch_sum_f64", "batch_sum_f64n"};
const char* const kLblEmit[4] = {"batch_emit_f32", "batch_emit_f32c", "batch_emit_f64",
                                 "batch_emit_f64n"};
const char* const kLblSearch[4] = {"batch_search_f32", "batch_search_f32c", "batch_search_f64",
                                   "batch_search_f64n"};

const char* const kLblCoop[4] = {"batch_coop_f32", "batch_coop_f32c", "batch_coop_f64",
                                 "batch_coop_f64n"};

// The cooperative form of the batched scan passes (batch_coop_kernel), sized to the resident
// grid; false when the device cannot run it (then the separate kernels run).
template <typename T, typename V, int SCHEME>
bool launch_batched_coop(const Scratch& s, const T* lw, const Batch& b, const Keys& keys,
                         int32_t* a, int32_t* d, V* W, cudaStream_t st, cudaError_t& e) {
  const int cap = coop_capacity(reinterpret_cast<const void*>(batch_coop_kernel<T, V, SCHEME>));
  if (cap < 1) return false;
  // a segment per warp at most: every filter adds at most one partial segment
  const int64_t want = (s.max_n / kSeg + b.F + kWarps) / kWarps;
  const int grid = static_cast<int64_t>(cap) < want ? cap : static_cast<int>(want);
  trace_mark(s.trace, kLblCoop[Path<T, V>::id], st);
  e = coop_launch(batch_coop_kernel<T, V, SCHEME>, grid, st, lw, b, keys, a, d, W, &s.glob->bar);
  return true;
}

template <typename T, typename V>
cudaError_t run_batched_scan(const Scratch& s, int scheme, const T* lw, const Batch& b,
                             int64_t cap_tiles, const Keys& keys, int32_t* a, int32_t* d,
                             cudaStream_t st) {
  constexpr int ai = Path<T, V>::id;
  const int tiles = static_cast<int>(cap_tiles);
  if (s.coop && s.launch_mode != RS_LAUNCH_SEPARATE) {
    cudaError_t e = cudaSuccess;
    V* Wc = static_cast<V*>(s.W);
    bool done;
    switch (scheme) {
      case RS_MULTINOMIAL:
        done = launch_batched_coop<T, V, RS_MULTINOMIAL>(s, lw, b, keys, a, d, Wc, st, e);
        if (done && e == cudaSuccess) {
          trace_mark(s.trace, kLblSearch[ai], st);
          launch_pdl(batch_search_kernel<T, V>, grid_particles(s.max_n), kBlock, st, Wc, b,
                     s.max_n, keys, a, d);
          e = cudaGetLastError();
        }
        break;
      case RS_STRATIFIED:
        done = launch_batched_coop<T, V, RS_STRATIFIED>(s, lw, b, keys, a, d, nullptr, st, e);
        break;
      default:
        done = launch_batched_coop<T, V, RS_SYSTEMATIC>(s, lw, b, keys, a, d, nullptr, st, e);
        break;
    }
    if (done) return e;
  }
  trace_mark(s.trace, "batch_max", st);
  launch_pdl(batch_max_kernel<T>, tiles, kBlock, st, lw, b);
  trace_mark(s.trace, kLblSum[ai], st);
  launch_pdl(batch_sum_kernel<T, V>, tiles, kBlock, st, lw, b);
  trace_mark(s.trace, "batch_prefix", st);
  launch_pdl(batch_prefix_kernel<T, V>, b.F, kBlock, st, b);
  V* W = static_cast<V*>(s.W);
  trace_mark(s.trace, kLblEmit[ai], st);
  switch (scheme) {
    case RS_MULTINOMIAL:
      launch_pdl(batch_emit_kernel<T, V, RS_MULTINOMIAL>, tiles, kBlock, st, lw, b, keys, a, d, W);
      trace_mark(s.trace, kLblSearch[ai], st);
      launch_pdl(batch_search_kernel<T, V>, grid_particles(s.max_n), kBlock, st, W, b, s.max_n, keys,
                                                                            a, d);
      break;
    case RS_STRATIFIED:
      launch_pdl(batch_emit_kernel<T, V, RS_STRATIFIED>, tiles, kBlock, st, lw, b, keys, a, d, nullptr);
      break;
    default:
      launch_pdl(batch_emit_kernel<T, V, RS_SYSTEMATIC>, tiles, kBlock, st, lw, b, keys, a, d, nullptr);
      break;
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_batched(const Scratch& s, int scheme, Acc acc, const void* logw,
                           const int64_t* offsets, int F, const int32_t* Bf, int32_t B,
                           uint64_t seed, uint64_t step, double log_wmax, int64_t max_trials,
                           const uint8_t* flags, int32_t* out, int permute, cudaStream_t st) {
  int32_t* a = permute ? s.a_tmp : out;
  int32_t* d = permute ? s.d : nullptr;
  // a non-decreasing ancestry (stratified, systematic): claimed bits in the claims' buffer
  uint8_t* cl = nullptr;
  if (permute && (scheme == RS_STRATIFIED || scheme == RS_SYSTEMATIC)) {
    cl = reinterpret_cast<uint8_t*>(s.d);
    d = nullptr;
  }
  const bool f64 = acc == Acc::F64 || acc == Acc::F64N;
  const Keys keys = make_keys(seed, step, 0u, static_cast<uint32_t>(scheme));
  // particles are bounded by the capacity; the true total is offsets[F] (checked per filter)
  const int64_t total = s.max_n;
  cudaError_t e = cudaSuccess;
  if (scheme == RS_METROPOLIS || scheme == RS_REJECTION) {
    const LaunchCfg& mc = s.batch_cfg[f64 ? kCfgMetropolisF64 : kCfgMetropolisF32];
    // binary32: the staged chains at the default launch shape; another shape (set or tuned), and
    // binary64, whose chains are bound by their draws (a block a step) and gained nothing from
    // staged sidecars (1000 filters of 256 .. 65536: 2975 against 2946 us; 64 of 64 .. 8000: 128
    // against 116), run one thread per particle
    const bool staged = scheme == RS_METROPOLIS && !f64 && mc.block == kBlock && mc.ipt == 1 &&
                        chain_available();
    auto* work = reinterpret_cast<unsigned long long*>(s.batch_fS);  // F + 1 <= 2 max_filters
    if (d || staged) {
      trace_mark(s.trace, "batch_fill", st);
      launch_pdl(batch_chain_plan_kernel, 1 + (d ? fill_grid(total) : 0), kChainBlock, st, offsets,
                 F, total, Bf, B, flags, staged ? work : nullptr, &s.glob->batch_next, d,
                 &s.glob->batch_limit, s.err);
    }
    trace_mark(s.trace, scheme == RS_METROPOLIS ? (f64 ? "batch_metropolis_f64" : "batch_metropolis_f32")
                                                : (f64 ? "batch_rejection_f64" : "batch_rejection_f32"),
               st);
    if (scheme == RS_REJECTION) {
      const int64_t runs = total < kRejSmallBatch ? (total + 7) / 8
                                                  : std::max((total + 31) / 32, kRejSmallBatch / 8);
      const int64_t ctas = (32 * runs + kBlock - 1) / kBlock;
      const bool turns = ctas > kRejCtas * device_sm_count();
      const int grid = turns ? kRejTurnCtas * device_sm_count() : static_cast<int>(ctas);
      if (f64)
        launch_pdl(turns ? batch_rejection_kernel<double, true> : batch_rejection_kernel<double, false>,
                   grid, kBlock, st, static_cast<const double*>(logw), offsets, F, total, keys,
                   log_wmax, max_trials, flags, a, d, s.err);
      else
        launch_pdl(turns ? batch_rejection_kernel<float, true> : batch_rejection_kernel<float, false>,
                   grid, kBlock, st, static_cast<const float*>(logw), offsets, F, total, keys,
                   log_wmax, max_trials, flags, a, d, s.err);
    } else if (staged) {
      launch_pdl_smem(batch_chain_kernel, device_sm_count(), kChainBlock, kChainSmem, st,
                      static_cast<const float*>(logw), offsets, F, total, Bf, B, keys, flags, work,
                      &s.glob->batch_next, a, d, s.err);
    } else if (f64) {
      launch_pdl(batch_mcmc_kernel<double>, grid_shaped(total, mc), mc.block, st,
                 static_cast<const double*>(logw), offsets, F, total, Bf, B, keys, flags, a, d,
                 mc.ipt, s.err);
    } else {
      launch_pdl(batch_mcmc_kernel<float>, grid_shaped(total, mc), mc.block, st,
                 static_cast<const float*>(logw), offsets, F, total, Bf, B, keys, flags, a, d,
                 mc.ipt, s.err);
    }
  } else {
    Batch b;
    b.off = offsets;
    b.F = F;
    b.max_n = s.max_n;
    b.tile_start = s.batch_tile_start;
    b.seg_start = s.batch_tile_start + s.max_filters + 1;  // (F + 2 entries)
    b.fmax = s.batch_fmax;
    b.fS = s.batch_fS;
    b.fscale = s.batch_fscale;
    b.fSd = s.batch_fSd;
    b.s_rec = s.batch_s_rec;
    b.P_rec = s.batch_P_rec;
    b.resample = flags;
    b.cl = cl;
    b.limit = &s.glob->batch_limit;
    b.err = s.err;
    trace_mark(s.trace, "batch_plan", st);
    launch_pdl(batch_plan_kernel, 1, 1024, st, b);
    // every filter adds at most one partial tile to the max_n / kTile full ones
    const int64_t cap_tiles = s.max_n / kTile + F + 1;
    switch (acc) {
      case Acc::F32:
        e = run_batched_scan<float, float>(s, scheme, static_cast<const float*>(logw), b,
                                           cap_tiles, keys, a, d, st);
        break;
      case Acc::F32C:
        e = run_batched_scan<float, float2>(s, scheme, static_cast<const float*>(logw), b,
                                            cap_tiles, keys, a, d, st);
        break;
      case Acc::F64:
        e = run_batched_scan<double, float2>(s, scheme, static_cast<const double*>(logw), b,
                                             cap_tiles, keys, a, d, st);
        break;
      case Acc::F64N:
        e = run_batched_scan<double, double>(s, scheme, static_cast<const double*>(logw), b,
                                             cap_tiles, keys, a, d, st);
        break;
    }
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e == cudaSuccess && permute) {
    trace_mark(s.trace, "batch_permute", st);
    const LaunchCfg& c = s.batch_cfg[kCfgPermute];
    const int64_t min4 = cl ? permute4_min_n<true>() : permute4_min_n<false>();
    const int grid = grid_shaped(total < min4 ? total : std::max((total + 3) / 4, min4), c);
    const bool large = total >= min4;
    launch_pdl_smem(cl ? (large ? batch_permute_kernel<true, true> : batch_permute_kernel<true, false>)
                       : (large ? batch_permute_kernel<false, true> : batch_permute_kernel<false, false>),
                    grid, c.block, kPermSmemPerWarp * (c.block / 32), st, offsets, F, total, s.a_tmp,
                    s.d, cl, out, c.ipt, &s.glob->batch_limit, s.err);
    e = cudaGetLastError();
  }
  return e;
}

}  // namespace rsk
