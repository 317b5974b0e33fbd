// fused.cu -- the passes of the multinomial, stratified and systematic resamplers of one filter
// (maximum and segment records, segment prefixes, emission) as one persistent cooperative
// kernel.
//
// Each CTA owns a contiguous range of segments; the CTAs are all resident at once (cooperative
// launch) and meet at grid-wide barriers between the phases (see fused_body). The segment
// prefixes are exact fixed-point sums, so they can be assembled in parallel from per-CTA
// totals instead of by one CTA, and each phase calls the same device functions as the
// separate kernels on the same segments: the results are identical. The latency-bound
// particle-parallel steps that follow (the multinomial search, Permute) stay separate
// full-occupancy kernels.
// A barrier waits at most the handle's barrier timeout (then it records RS_ERR_TIMEOUT and proceeds;
// every phase stays bounds-checked, so the kernel still ends); the barrier counter returns
// to 0 at the end of every launch.
#include <cfloat>
#include <type_traits>

#include "common.cuh"
#include "grid.cuh"
#include "internal.h"
#include "tile.cuh"
#include "values.cuh"

namespace rsk {
namespace {

struct FusedArgs {
  int64_t N;
  Keys keys;
  int32_t* a;      // ancestors (systematic / stratified)
  int32_t* d;      // Prepermute claims of the multinomial (set to the sentinel), or nullptr
  uint8_t* cl;     // claimed bits of the particles (systematic / stratified), or nullptr
  void* W;         // multinomial cumulative weights
  int32_t* guide;  // multinomial guide table
  double2* s_rec;  // segment records
  double2* P_rec;  // segment prefixes: exact in-range prefixes (u128), then rounded P_g
  u128* agg;       // per-CTA exact totals (gridDim.x entries)
  ScanGlob* g;
  int* err;
};

// CTA c owns the contiguous segments [c T / G, (c+1) T / G) of the T segments of kSeg particles
// (G = gridDim.x <= T), its warps taking them in turns of kWarps: cutting by segments, not by
// tiles, gives every SM the same work to within a segment a CTA (2^20 particles: 4096 segments on
// 608 CTAs; as 512 tiles some SMs had four, most three).
//   phase 1  the records (m_g, s_g) of its segments (seg_record, each warp its own: the
//            segment's maximum and its weights' sum relative to it), last turn to first,
//            and its largest m_g
//            (an atomic maximum of ordered keys per CTA) -> barrier;
//   phase 2  T_g = s_g exp(m_g - M) (rec_scaled) of its segments and their exact running sum in
//            fixed point (the in-range prefix of each segment, and the CTA total) -> barrier;
//            (compensated binary32, whose records must sum the weights exp(lw - M) themselves:
//            phase 1 forms the maximum only and phase 2 the records relative to M, which then
//            scale by exactly 1);
//   phase 3  every CTA sums the exact CTA totals: those before it (CP) and all (the total);
//            P_g = RN(CP + in-range prefix of g) for its segments and P_{g1} = RN(CP + its
//            own total), which is the P_{g1} the next CTA computes; W^N = RN(total), N / W^N;
//   phase 4  emission of its segments, first to last (it starts on those phase 1 read last,
//            still in L2 when the log-weights exceed half of it), each warp its own.
// Phases 1 and 4 are warp-level work only: no block barrier per turn. The log-weights are read
// twice (phases 1 and 4; three times for compensated binary32), the least the normaliser
// allows. P_g is the exact sum of the T before g rounded once, as in seg_prefix_compute, so the
// results equal those of the separate kernels. Two grid barriers per call (none for one CTA).
//
// Phases 2 and 3 are a chain of short dependent steps that every CTA takes whatever N is (at 2^20
// they were two thirds of the kernel's instructions and about 8 of its 20 us). So a CTA with
// fewer than 32 segments scans them in one warp, records and prefixes of a CTA's segments stay
// in shared memory (up to kCtaSegs of them), the totals before the CTA and the total with its
// binary64 division are finished by two different warps, and the systematic uniform is drawn at
// the start: 2^20 binary32 systematic 26.7 -> 24.7 us a call, 1000 particles 14.4 -> 10.3 with the
// launches queued ahead (alone, such a call was bound by its 14 us on the host then).
constexpr int kCtaSegs = kBlock;  // segments of a CTA whose records and prefixes stay on chip

// The order-preserving key of a log-weight as an unsigned number above 0, and back.
template <typename T> __device__ __forceinline__ T from_key(unsigned long long k) {
  if constexpr (sizeof(T) == 4) return from_ordered_key(static_cast<uint32_t>(k));
  else return from_ordered_key(k);
}

// Inclusive sum over the lanes of a warp.
__device__ __forceinline__ u128 warp_incl_scan_u128(u128 v) {
#pragma unroll
  for (int dd = 1; dd < 32; dd <<= 1) {
    const u128 y = shfl_up_u128(v, dd);
    if ((threadIdx.x & 31) >= dd) v += y;
  }
  return v;
}

template <typename T, typename V, int SCHEME>
__device__ __forceinline__ void fused_body(const T* __restrict__ lw, const FusedArgs& A,
                                           unsigned int& target) {
  __shared__ SegSh sh;
  __shared__ float2 sh_tab[64];
  __shared__ unsigned long long sh_key[kWarps];
  __shared__ u128 sh_sum[2 * kWarps];
  __shared__ double2 sh_rp[kCtaSegs + 1];  // records, then rounded prefixes, of the CTA's segments
  __shared__ typename Path<T, V>::U sh_u;
  const int64_t N = A.N;
  const int T_segs = static_cast<int>((N + kSeg - 1) / kSeg);
  const int G = static_cast<int>(gridDim.x), c = static_cast<int>(blockIdx.x);
  const int g0 = static_cast<int>(static_cast<int64_t>(c) * T_segs / G);  // this CTA's segments
  const int g1 = static_cast<int>(static_cast<int64_t>(c + 1) * T_segs / G);
  const int nseg = g1 - g0;
  const bool on_chip = (T_segs + G - 1) / G <= kCtaSegs;  // (uniform over the grid)
  const bool one_warp = nseg < 32;
  const int turns = (nseg + kWarps - 1) / kWarps;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t e0 = static_cast<int64_t>(g0) * kSeg;
  const int64_t e1 = min(static_cast<int64_t>(g1) * kSeg, N);
  const int64_t off = kPer * static_cast<int64_t>(threadIdx.x);
  const bool vec = (reinterpret_cast<uintptr_t>(lw) & 15u) == 0;
  double2* const recs = on_chip ? sh_rp : A.s_rec + g0;
  if (threadIdx.x < 64) sh_tab[threadIdx.x] = kExp2Frac64[threadIdx.x];
  if constexpr (SCHEME == RS_SYSTEMATIC)
    if (threadIdx.x == kBlock - 1) sh_u = Path<T, V>::draw_u(draw(A.keys, 0u, 0u));
  __syncthreads();

  // ---- phase 1: segment records, last turn to first (and the Prepermute sentinel of the
  // multinomial claims); the next segment's log-weights are loaded while this one is reduced.
  // Without kTileRef, the maximum only (the records follow once M is known) ----------------
  const int last_turn = turns - (kWarps * (turns - 1) + warp < nseg ? 1 : 2);  // (of this warp)
  const int64_t lane0 = e0 + static_cast<int64_t>(kSeg) * warp + kPer * lane;  // (turn 0)
  {
    unsigned long long key;  // of this warp's largest log-weight
    bool bad = false;
    if constexpr (Path<T, V>::kTileRef) {
      long long cm = max_key(neg_inf<T>());
      // (two segments ahead for binary32, 64 KB in flight on an SM: 2^24 63.5 -> 62.5 us)
      constexpr int kAhead = sizeof(T) == 4 ? 2 : 1;
      T xn[kAhead][kPer];
#pragma unroll
      for (int h = 0; h < kAhead; ++h)
        if (last_turn >= h)
          load_per(lw, lane0 + static_cast<int64_t>(kTile) * (last_turn - h), 0, N, vec, xn[h],
                   L2Hint::kEvictLast);
      for (int t = last_turn; t >= 0; t -= kAhead) {
#pragma unroll
        for (int h = 0; h < kAhead; ++h) {
          if (t < h) break;
          T x[kPer];
#pragma unroll
          for (int q = 0; q < kPer; ++q) x[q] = xn[h][q];
          if (t - h >= kAhead)
            load_per(lw, lane0 + static_cast<int64_t>(kTile) * (t - h - kAhead), 0, N, vec, xn[h],
                     L2Hint::kEvictLast);
          const long long k = seg_record<T, V>(x, sh_tab, recs + kWarps * (t - h) + warp, bad);
          cm = k > cm ? k : cm;
        }
      }
      key = ordered_key(key_to<T>(cm));
    } else {
      float mf = -INFINITY;  // (binary32 inputs)
      for (int t = 0; t <= last_turn; ++t) {
        T x[kPer];
        load_per(lw, lane0 + static_cast<int64_t>(kTile) * t, 0, N, vec, x, L2Hint::kEvictLast);
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
          bad |= !(x[q] <= FLT_MAX);  // NaN or +inf
          mf = fmaxf(mf, static_cast<float>(x[q]));
        }
      }
      key = __reduce_max_sync(0xffffffffu, ordered_key(mf));
    }
    if constexpr (SCHEME == RS_MULTINOMIAL) {
      if (A.d) {
        int32_t sv[kPer];
#pragma unroll
        for (int q = 0; q < kPer; ++q) sv[q] = static_cast<int32_t>(N);
        for (int64_t i0 = e0 + off; i0 < e1; i0 += kTile)
          store_per(A.d + i0, sv, e1 - i0 < kPer ? static_cast<int>(e1 - i0) : kPer);
      }
    }
    if (bad) flag_error(A.err, RS_ERR_NONFINITE);
    if (lane == 0) sh_key[warp] = key;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < kWarps; ++w) key = sh_key[w] > key ? sh_key[w] : key;
      if (G > 1) atomicMax(&A.g->scan_key, key);
      else sh_key[0] = key;
    }
  }
  if (G > 1) grid_barrier(&A.g->bar, target, A.err);
  else __syncthreads();
  const T Mt = from_key<T>(G > 1 ? __ldcg(&A.g->scan_key) : sh_key[0]);
  const double M = static_cast<double>(Mt);
  const bool zero = sizeof(T) == 4 ? is_neg_inf(Mt) : !(M > -DBL_MAX);  // (M > -DBL_MAX, in binary32)
  u128* LP = reinterpret_cast<u128*>(A.P_rec);  // (not on_chip) in-range exact prefixes, then P_g

  // ---- phase 2: segment totals relative to M and their exact running sum -------------------
  const WeightCtx wc = ctx_staged<T, V>(zero ? 0.0 : M, sh_tab);
  u128 run = 0;  // the exact total of this CTA's segments (one_warp: in warp 0)
  u128 lp0 = 0;  // the exact in-range prefix of segment g0 + threadIdx.x
  if (!zero) {
    if constexpr (!Path<T, V>::kTileRef) {  // the records, relative to M, last turn to first
      bool bad = false;
      for (int t = last_turn; t >= 0; --t) {
        const int g = g0 + kWarps * t + warp;
        seg_record<T, V>(lw, 0, N, static_cast<int64_t>(g) * kSeg, sh_tab, vec, recs + (g - g0), bad,
                         max_key(Mt), L2Hint::kEvictLast);
      }
      __syncthreads();  // (lane 0 of each warp stored them; all threads read them below)
    }
    if (one_warp) {
      if (warp == 0) {
        const u128 f = lane < nseg ? to_fixed(rec_scaled_of<T, V>(recs[lane], Mt, sh_tab)) : u128(0);
        const u128 incl = warp_incl_scan_u128(f);
        lp0 = incl - f;
        run = (static_cast<u128>(__shfl_sync(0xffffffffu, static_cast<uint64_t>(incl >> 64), 31)) << 64) |
              __shfl_sync(0xffffffffu, static_cast<uint64_t>(incl), 31);
      }
    } else {
      for (int gb = 0; gb < nseg; gb += kBlock) {
        const int g = gb + static_cast<int>(threadIdx.x);
        u128 f = 0;
        if (g < nseg) f = to_fixed(rec_scaled_of<T, V>(on_chip ? recs[g] : __ldcg(recs + g), Mt, sh_tab));
        u128 tot;
        const u128 ex = block_excl_scan_u128(f, sh_sum, tot);
        if (!on_chip && g < nseg) st_u128(LP + g0 + g, run + ex);
        if (gb == 0) lp0 = ex;
        run += tot;
      }
    }
    if (threadIdx.x == 0) st_u128(A.agg + c, run);
  }
  if (G > 1) grid_barrier(&A.g->bar, target, A.err);
  else __syncthreads();

  // ---- phase 3: the total and this CTA's segment prefixes ----------------------------------
  if (zero) {  // all weights zero (flagged): every particle keeps itself
    if (c == 0 && threadIdx.x == 0) {
      A.g->S_d = 0.0;
      A.g->M = M;
      A.g->all_zero = 1;
      flag_error(A.err, RS_ERR_ZERO_WEIGHT);
    }
    if constexpr (SCHEME != RS_MULTINOMIAL) {  // (the search kernel writes the identity)
      for (int64_t i = e0 + threadIdx.x; i < e1; i += kBlock) A.a[i] = static_cast<int32_t>(i);
      if (A.cl)  // every slot claimed (e0 is a multiple of 8)
        for (int64_t b = (e0 >> 3) + threadIdx.x; b < ((e1 + 7) >> 3); b += kBlock) A.cl[b] = 0xFFu;
    }
    return;  // uniform over the grid
  }
  __shared__ double2 sh_S, sh_scale, sh_pend;
  __shared__ bool sh_zero;
  __shared__ Guide sh_gd;
  {
    u128 CP = 0, TOT = 0;  // this thread's, then this warp's, part of the sums over the CTAs
    for (int k = threadIdx.x; k < G; k += kBlock) {
      const u128 v = ld_u128_cg(A.agg + k);
      TOT += v;
      if (k < c) CP += v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      CP += shfl_xor_u128(CP, o);
      TOT += shfl_xor_u128(TOT, o);
    }
    if (lane == 0) {
      sh_sum[warp] = CP;
      sh_sum[kWarps + warp] = TOT;
    }
    __syncthreads();
    // the prefixes: of segment g0 + threadIdx.x (one_warp: warp 0 has them all) and of g1
    if (!one_warp || warp == 0) {
      CP = 0;
#pragma unroll
      for (int k = 0; k < kWarps; ++k) CP += sh_sum[k];
      for (int g = threadIdx.x; g <= nseg; g += kBlock) {
        const u128 lp = g == nseg ? run : (on_chip || g < kBlock) ? lp0 : ld_u128_cg(LP + g0 + g);
        const V P = fixed_to(CP + lp, V(), kFixFrac);
        if (on_chip) store_v<V>(sh_rp + g, P);
        else if (g < nseg || c == G - 1) store_v<V>(A.P_rec + g0 + g, P);
        if (g == nseg) store_v<V>(&sh_pend, P);
      }
    }
    // the total, N / total and the guide step (a binary64 division takes about a microsecond),
    // in the last warp
    if (threadIdx.x == kBlock - 32) {
      TOT = 0;
#pragma unroll
      for (int k = 0; k < kWarps; ++k) TOT += sh_sum[kWarps + k];
      const V S0 = fixed_to(TOT, V(), kFixFrac);
      const double Sd0 = vto_double(S0);
      const V scale0 = vfrom_double(__ddiv_rn(static_cast<double>(N), Sd0), V());
      store_v<V>(&sh_S, S0);
      store_v<V>(&sh_scale, scale0);
      sh_zero = !(Sd0 > 0.0);
      if constexpr (SCHEME == RS_MULTINOMIAL) sh_gd = make_guide(Sd0, N);
      if (c == 0) {  // read by the search kernel and the host-side callers
        store_v<V>(&A.g->S_raw, S0);
        store_v<V>(&A.g->scale_raw, scale0);
        A.g->S_d = Sd0;
        A.g->M = M;
        A.g->all_zero = !(Sd0 > 0.0);
        if constexpr (SCHEME == RS_MULTINOMIAL) {
          A.g->guide_step = sh_gd.step;
          A.g->guide_inv_step = sh_gd.inv_step;
        }
        if (!(Sd0 > 0.0)) flag_error(A.err, RS_ERR_ZERO_WEIGHT);
      }
    }
    __syncthreads();
  }
  const V S = load_v<V>(&sh_S), scale = load_v<V>(&sh_scale);
  const bool all_zero = sh_zero;
  // the kernels that follow (search, Permute) may launch now; they wait for this grid's end
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (all_zero) {  // the total rounds to zero: every particle keeps itself
    if constexpr (SCHEME != RS_MULTINOMIAL) {
      for (int64_t i = e0 + threadIdx.x; i < e1; i += kBlock) A.a[i] = static_cast<int32_t>(i);
      if (A.cl)
        for (int64_t b = (e0 >> 3) + threadIdx.x; b < ((e1 + 7) >> 3); b += kBlock) A.cl[b] = 0xFFu;
    }
    return;
  }

  // ---- phase 4: emission of this CTA's segments, each warp its own (no block-level
  // synchronisation) -------------------------------------------------------------------------
  typename Path<T, V>::U u_sys = typename Path<T, V>::U();
  Guide gd;
  if constexpr (SCHEME == RS_MULTINOMIAL) gd = sh_gd;
  else if constexpr (SCHEME == RS_SYSTEMATIC) u_sys = sh_u;
  for (int g = g0 + warp; g < g1; g += kWarps) {
    const int64_t base = static_cast<int64_t>(g) * kSeg;
    const V Ps = on_chip ? load_v<V>(sh_rp + (g - g0)) : load_v_cg<V>(A.P_rec + g);
    const V Pn = g + 1 == g1 ? load_v<V>(&sh_pend)
                             : on_chip ? load_v<V>(sh_rp + (g + 1 - g0)) : load_v_cg<V>(A.P_rec + g + 1);
    if constexpr (SCHEME == RS_MULTINOMIAL) {
      emit_seg_W_guide<T, V>(lw, 0, N, base, wc, vec, Ps, Pn, gd, static_cast<V*>(A.W), A.guide,
                             sh.win[warp], L2Hint::kEvictFirst);
    } else {
      emit_seg_cumoff<T, V, SCHEME == RS_STRATIFIED>(lw, 0, N, base, wc, vec, Ps, Pn, S, scale,
                                                      u_sys, A.keys, A.a, sh.win[warp], A.cl,
                                                      L2Hint::kEvictFirst);
    }
  }
}

// CTAs of kBlock threads that share an SM (the cooperative grid holds so many on each): four for
// binary32 log-weights and the multinomial (64 registers), three for the stratified and systematic
// of binary64 log-weights, whose emission keeps more values in flight (80 registers; 3000001
// particles, double-float: 92.2 -> 90.2 us, IEEE 700001: 85.8 -> 78.9; see launch_fused for the
// sizes where four take one turn; compensated binary32 at 2^20 is faster with four).
template <typename T, int SCHEME>
constexpr int fused_ctas() {
  return sizeof(T) == 4 || SCHEME == RS_MULTINOMIAL ? 4 : 3;
}
template <typename T, typename V, int SCHEME, int CTAS>
__global__ void __launch_bounds__(kBlock, CTAS) fused_scan_kernel(const T* __restrict__ lw, FusedArgs A) {
  unsigned int target = 0;
  fused_body<T, V, SCHEME>(lw, A, target);
  // the last CTA to end returns the shared state to its start (every CTA has read the key)
  if (gridDim.x > 1 && threadIdx.x == 0 &&
      atomicAdd(&A.g->bar.count, 1u) == target + gridDim.x - 1) {
    A.g->scan_key = 0ull;
    atomicExch(&A.g->bar.count, 0u);
  }
}

template <typename T, typename V, int SCHEME, int CTAS = fused_ctas<T, SCHEME>()>
int fused_capacity() {
  static int cap = -1;  // identical devices assumed
  if (cap < 0) {
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fused_scan_kernel<T, V, SCHEME, CTAS>,
                                                      kBlock, 0) != cudaSuccess)
      return 0;
    cap = per_sm * sms;
  }
  return cap;
}

template <typename T, typename V, int SCHEME, int CTAS = fused_ctas<T, SCHEME>()>
cudaError_t launch_fused(const Scratch& s, const T* lw, const FusedArgs& A, cudaStream_t st) {
  int64_t grid = fused_capacity<T, V, SCHEME, CTAS>();
  if (grid > s.max_blocks) grid = s.max_blocks;
  // a full turn of the warps each; half a turn for native binary64, which is bound by the
  // binary64 pipes of the SMs it reaches (20000 particles: 51 -> 33 us), while the others lose by
  // more CTAs at the barriers (2^20 binary32: 27.2 -> 29.0 us)
  constexpr int64_t per = std::is_same_v<V, double> ? kWarps / 2 : kWarps;
  const int64_t want = ((A.N + kSeg - 1) / kSeg + per - 1) / per;
  if constexpr (CTAS == 3 && per == kWarps) {
    // a fourth CTA on an SM (64 registers) where it makes one turn of the warps of two: double-float
    // at 2^20 (4096 segments, 456 x 8 warps) systematic 42.7 -> 39.0 us with Permute, stratified
    // 47.3 -> 43.9; from two turns on the registers win (stratified 3600000: 92.7 against 95.3)
    int64_t more = fused_capacity<T, V, SCHEME, 4>();
    if (more > s.max_blocks) more = s.max_blocks;
    if (grid >= 1 && want > grid && want <= more)
      return launch_fused<T, V, SCHEME, 4>(s, lw, A, st);
  }
  if (grid > want) grid = want;
  if (grid < 1) return cudaErrorCooperativeLaunchTooLarge;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(grid));
  cfg.blockDim = dim3(kBlock);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fused_scan_kernel<T, V, SCHEME, CTAS>, lw, A);
}

template <typename T, typename V>
int capacity(int scheme) {
  switch (scheme) {
    case RS_MULTINOMIAL: return fused_capacity<T, V, RS_MULTINOMIAL>();
    case RS_STRATIFIED: return fused_capacity<T, V, RS_STRATIFIED>();
    default: return fused_capacity<T, V, RS_SYSTEMATIC>();
  }
}

template <typename T, typename V>
cudaError_t dispatch(const Scratch& s, int scheme, const T* lw, const FusedArgs& A,
                     cudaStream_t st) {
  switch (scheme) {
    case RS_MULTINOMIAL: return launch_fused<T, V, RS_MULTINOMIAL>(s, lw, A, st);
    case RS_STRATIFIED: return launch_fused<T, V, RS_STRATIFIED>(s, lw, A, st);
    default: return launch_fused<T, V, RS_SYSTEMATIC>(s, lw, A, st);
  }
}

const char* const kLblFused[4][3] = {
    {"fused_multinomial_f32", "fused_stratified_f32", "fused_systematic_f32"},
    {"fused_multinomial_f32c", "fused_stratified_f32c", "fused_systematic_f32c"},
    {"fused_multinomial_f64", "fused_stratified_f64", "fused_systematic_f64"},
    {"fused_multinomial_f64n", "fused_stratified_f64n", "fused_systematic_f64n"}};
}  // namespace

bool fused_available(const Scratch& s, int scheme, Acc acc) {
  if (!s.coop) return false;
  switch (acc) {
    case Acc::F32: return capacity<float, float>(scheme) > 0;
    case Acc::F32C: return capacity<float, float2>(scheme) > 0;
    case Acc::F64: return capacity<double, float2>(scheme) > 0;
    case Acc::F64N: return capacity<double, double>(scheme) > 0;
  }
  return false;
}

cudaError_t launch_fused_passes(const Scratch& s, int scheme, Acc acc, const void* logw,
                                int64_t N, const Keys& keys, int32_t* a_out, int32_t* d,
                                uint8_t* cl, cudaStream_t st) {
  FusedArgs A;
  A.N = N;
  A.keys = keys;
  A.a = a_out;
  A.d = d;
  A.cl = scheme == RS_MULTINOMIAL ? nullptr : cl;
  A.W = s.W;
  A.guide = s.guide;
  A.s_rec = s.rec;
  A.P_rec = s.rec + seg_cap(s.max_tiles);
  A.agg = reinterpret_cast<u128*>(s.irec);  // at least max_blocks entries >= gridDim.x
  A.g = s.glob;
  A.err = s.err;
  trace_mark(s.trace, kLblFused[static_cast<int>(acc)][scheme], st);
  switch (acc) {
    case Acc::F32:
      return dispatch<float, float>(s, scheme, static_cast<const float*>(logw), A, st);
    case Acc::F32C:
      return dispatch<float, float2>(s, scheme, static_cast<const float*>(logw), A, st);
    case Acc::F64:
      return dispatch<double, float2>(s, scheme, static_cast<const double*>(logw), A, st);
    case Acc::F64N:
      return dispatch<double, double>(s, scheme, static_cast<const double*>(logw), A, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace rsk
