// ess.cu -- effective sample size of a weight vector, ESS = (sum w)^2 / sum w^2 with the
// weights w_i = exp(lw_i - max lw) of Appendix E, the quantity that decides when an adaptive
// particle filter resamples (Section 4.3 discusses resampling every step against on demand).
// One cooperative launch: maximum -> grid barrier -> per-CTA sums of w and w^2; the CTA that
// finishes last adds the per-CTA totals exactly (128-bit fixed point, all its threads) and
// divides; the same sums give the log of the weight total, M + log sum w.
// A thread takes quadruples of consecutive log-weights and keeps its first ones in registers
// between the two passes, so that up to about two million binary32 log-weights are read once.
// Latency-bound at these sizes: the loads, one barrier, two block reductions (with 4-byte loads,
// a second barrier and a maximum over all CTAs' maxima 2^20 binary32 log-weights took 20.6 us).
//
// Also here: the bootstrap filter's copy by the ancestry, propagation, weighting and ESS as one
// such launch (lgssm_step_ess_kernel).
#include <cfloat>

#include "common.cuh"
#include "dfexp.cuh"
#include "grid.cuh"
#include "internal.h"
#include "model.cuh"
#include "tile.cuh"
#include "values.cuh"

namespace rsk {
namespace {

constexpr int kEssCtas = 4;  // CTAs of kBlock threads per SM

// Binary32 weight of one log-weight given the maximum (the ESS needs no more precision).
__device__ __forceinline__ float ess_weight(float x, float Mf, float2) {
  return is_neg_inf(x) ? 0.0f : exp_pinned(__fsub_rn(x, Mf));
}
__device__ __forceinline__ float ess_weight(double x, float, float2 M2) {
  return is_neg_inf(x) ? 0.0f : exp_pinned(add22_accurate(split_f64(x), neg2(M2)).x);
}

// Maximum of the grid's log-weights from every thread's own maximum m (NaN left out): one atomic
// maximum of order-preserving keys per CTA, then the grid barrier. Every thread gets it (-inf
// when all weights are zero).
template <typename T>
__device__ __forceinline__ T grid_max(T m, ScanGlob* g, unsigned int& target, int* err) {
  __shared__ unsigned long long sh_key[kWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long k = ordered_key(m);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, k, o);
    k = y > k ? y : k;
  }
  if (lane == 0) sh_key[warp] = k;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kWarps; ++w) k = sh_key[w] > k ? sh_key[w] : k;
    atomicMax(&g->ess_key, k);
  }
  grid_barrier(&g->bar, target, err);
  const unsigned long long all = __ldcg(&g->ess_key);
  if constexpr (sizeof(T) == 4) return from_ordered_key(static_cast<uint32_t>(all));
  else return from_ordered_key(all);
}

// The grid's sums of w and w^2 from every thread's, and the outputs: exact per CTA from its
// warps' two-float sums on; the last CTA to arrive adds the CTAs' totals and resets the shared
// state for the next launch.
__device__ __forceinline__ void ess_finish(float2 s1, float2 s2, double M, ScanGlob* g, u128* agg,
                                           double* ess_out, double* log_total_out, int* err) {
  __shared__ float2 sh_s[kWarps][2];
  __shared__ u128 sh_u[2 * kWarps];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s1 = vadd(s1, vshfl_xor(s1, o));
    s2 = vadd(s2, vshfl_xor(s2, o));
  }
  if (lane == 0) {
    sh_s[warp][0] = s1;
    sh_s[warp][1] = s2;
  }
  __syncthreads();
  if (warp == 0) {  // lanes 0 .. kWarps - 1: the warps' sums of w; the next kWarps: of w^2
    static_assert(2 * kWarps <= 32, "one lane per sum");
    u128 v = lane < 2 * kWarps ? to_fixed(sh_s[lane & (kWarps - 1)][lane / kWarps]) : u128(0);
#pragma unroll
    for (int o = kWarps / 2; o > 0; o >>= 1) v += shfl_xor_u128(v, o);
    if (lane == 0 || lane == kWarps) st_u128(agg + 2 * blockIdx.x + lane / kWarps, v);
    __threadfence();
    __syncwarp();
    if (lane == 0) last = atomicAdd(&g->ess_ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  u128 a1 = 0, a2 = 0;
  for (int b = threadIdx.x; b < static_cast<int>(gridDim.x); b += kBlock) {
    a1 += ld_u128_cg(agg + 2 * b);
    a2 += ld_u128_cg(agg + 2 * b + 1);
  }
  block_sum2_u128(a1, a2, sh_u);
  if (lane == 0 && warp < 2) {  // (the binary64 division and logarithm in two warps)
    const double S1 = fixed_to_double(a1, kFixFrac), S2 = fixed_to_double(a2, kFixFrac);
    const bool zero = !(M > -DBL_MAX) || !(S2 > 0.0);
    if (warp == 0) {
      if (ess_out) *ess_out = zero ? 0.0 : __ddiv_rn(__dmul_rn(S1, S1), S2);
      if (zero) flag_error(err, RS_ERR_ZERO_WEIGHT);
      g->ess_key = 0ull;
      g->ess_ticket = 0u;
    } else if (log_total_out) {
      *log_total_out = zero ? -static_cast<double>(INFINITY) : M + log(S1);
    }
  }
}

// Quadruples of log-weights that a thread keeps between the passes.
template <typename T> constexpr int ess_kept() { return sizeof(T) == 4 ? 4 : 2; }

template <typename T>
__global__ void __launch_bounds__(kBlock, kEssCtas)
ess_kernel(const T* __restrict__ lw, int64_t N, ScanGlob* g, u128* agg, double* ess_out,
           double* log_total_out, int* err) {
  constexpr int K = ess_kept<T>();
  unsigned int target = 0;
  const int64_t stride = 4 * static_cast<int64_t>(gridDim.x) * kBlock;
  const int64_t i0 = 4 * (static_cast<int64_t>(blockIdx.x) * kBlock + threadIdx.x);
  const bool vec = (reinterpret_cast<uintptr_t>(lw) & 15u) == 0;
  T kept[K][4];
  T m = neg_inf<T>();
  bool bad = false;
  auto look = [&](const T (&x)[4]) {  // (positions past N read as -inf)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      bad |= nonfinite_logw(x[q]);
      if constexpr (sizeof(T) == 4) m = fmaxf(m, x[q]);  // (skips NaN)
      else if (!is_nan(x[q]) && max_key(x[q]) > max_key(m)) m = x[q];
    }
  };
#pragma unroll
  for (int r = 0; r < K; ++r) load4(lw, i0 + r * stride, 0, N, vec, kept[r]);
#pragma unroll
  for (int r = 0; r < K; ++r) look(kept[r]);
  for (int64_t i = i0 + K * stride; i < N; i += stride) {
    T x[4];
    load4(lw, i, 0, N, vec, x);
    look(x);
  }
  if (bad) flag_error(err, RS_ERR_NONFINITE);
  const double M = static_cast<double>(grid_max(m, g, target, err));
  // two-float sums of w and w^2 per thread, then per CTA
  float2 s1 = make_float2(0.0f, 0.0f), s2 = make_float2(0.0f, 0.0f);
  if (M > -DBL_MAX) {
    const float Mf = static_cast<float>(M);
    const float2 M2 = split_f64(M);
    auto add = [&](const T (&x)[4], int64_t i) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (i + q < N) {
          const float w = ess_weight(x[q], Mf, M2);
          s1 = add21(s1, w);
          s2 = add21(s2, __fmul_rn(w, w));
        }
      }
    };
#pragma unroll
    for (int r = 0; r < K; ++r) add(kept[r], i0 + r * stride);
    for (int64_t i = i0 + K * stride; i < N; i += stride) {
      T x[4];
      load4(lw, i, 0, N, vec, x);
      add(x, i);
    }
  }
  ess_finish(s1, s2, M, g, agg, ess_out, log_total_out, err);
  grid_exit(&g->bar, target);
}

// One step of the bootstrap filter around its resampling, as one cooperative launch: x_i <-
// x_{c_i} (copy_ancestors_kernel; c null: no copy), propagation and log-weight
// (lgssm_step_kernel with accumulate = 0), and the ESS and log weight total of the new
// log-weights (ess_kernel). All rows are read before the grid barrier of the maximum and written
// after it, which makes the copy and the propagation one pass in place; the log-weights stay in
// registers for the sums (K quadruples a thread). Reads c and x, writes x and logw once (16 bytes
// a particle) where the three kernels moved 36. About 270 instructions a particle, half of them
// the noise (Philox, logarithm, cosine), a third the two-float sums: at 2^20 23 us under the
// profiler against 41 for the three kernels; a bootstrap step 59 -> 51 us.
template <int K>
__global__ void __launch_bounds__(kBlock, kEssCtas)
lgssm_step_ess_kernel(float* __restrict__ x, const int32_t* __restrict__ c, uint32_t N, int init,
                      float phi, float sigma_x, float sigma_0, float y, float inv_2vy, Keys keys,
                      float* __restrict__ logw, ScanGlob* g, u128* agg, double* ess_out,
                      double* log_total_out, int* err) {
  unsigned int target = 0;
  // (N <= 4 K threads of the grid < 2^31: 32-bit indices)
  const uint32_t stride = 4 * gridDim.x * kBlock;
  const uint32_t i0 = 4 * (blockIdx.x * kBlock + threadIdx.x);
  const bool vec = ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(c) |
                     reinterpret_cast<uintptr_t>(logw)) & 15u) == 0;
  float xn[K][4], l[K][4];  // (l: the noise, then the log-weights)
  float m = -INFINITY;
  bool bad = false, bad_c = false;
  int32_t src[K][4];
#pragma unroll
  for (int r = 0; r < K; ++r) {
    const uint32_t i = i0 + r * stride;
    if (c && vec && i + 4 <= N) {
      const int4 v = __ldg(reinterpret_cast<const int4*>(c + i));
      src[r][0] = v.x; src[r][1] = v.y; src[r][2] = v.z; src[r][3] = v.w;
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        src[r][q] = c && i + q < N ? __ldg(c + i + q) : static_cast<int32_t>(i + q);
    }
  }
#pragma unroll
  for (int r = 0; r < K; ++r)  // (the noise while the ancestors are on their way)
    if (i0 + r * stride < N) {
#pragma unroll
      for (int q = 0; q < 4; ++q) l[r][q] = normal_draw(keys, i0 + r * stride + q);
    }
#pragma unroll
  for (int r = 0; r < K; ++r) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t i = i0 + r * stride + q;
      xn[r][q] = 0.0f;
      if (i < N && !init) {
        int32_t s = src[r][q];
        if (static_cast<uint32_t>(s) >= N || (s != static_cast<int32_t>(i) && __ldg(c + s) != s)) {
          bad_c = true;  // not from Permute: left alone
          s = static_cast<int32_t>(i);
        }
        xn[r][q] = x[s];
      }
    }
  }
#pragma unroll
  for (int r = 0; r < K; ++r) {
    const uint32_t i = i0 + r * stride;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float z = l[r][q];
      l[r][q] = -INFINITY;
      if (i + q < N) {
        const float xi = init ? sigma_0 * z : fmaf(phi, xn[r][q], sigma_x * z);
        const float e = y - xi;
        xn[r][q] = xi;
        l[r][q] = -(e * e) * inv_2vy;
        bad |= nonfinite_logw(l[r][q]);
        m = fmaxf(m, l[r][q]);
      }
    }
    if (vec && i + 4 <= N) {
      *reinterpret_cast<float4*>(logw + i) = make_float4(l[r][0], l[r][1], l[r][2], l[r][3]);
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (i + q < N) logw[i + q] = l[r][q];
    }
  }
  if (bad) flag_error(err, RS_ERR_NONFINITE);
  if (bad_c) flag_error(err, RS_ERR_ARG);
  const float Mf = grid_max(m, g, target, err);  // (every row of x has been read)
#pragma unroll
  for (int r = 0; r < K; ++r) {
    const uint32_t i = i0 + r * stride;
    if (vec && i + 4 <= N) {
      *reinterpret_cast<float4*>(x + i) = make_float4(xn[r][0], xn[r][1], xn[r][2], xn[r][3]);
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (i + q < N) x[i + q] = xn[r][q];
    }
  }
  float2 s1 = make_float2(0.0f, 0.0f), s2 = make_float2(0.0f, 0.0f);
  if (!is_neg_inf(Mf)) {
#pragma unroll
    for (int r = 0; r < K; ++r) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (i0 + r * stride + q < N) {
          const float w = ess_weight(l[r][q], Mf, make_float2(0.0f, 0.0f));
          s1 = add21(s1, w);
          s2 = add21(s2, __fmul_rn(w, w));
        }
      }
    }
  }
  ess_finish(s1, s2, static_cast<double>(Mf), g, agg, ess_out, log_total_out, err);
  grid_exit(&g->bar, target);
}

// Grid of these kernels: a quadruple per thread, at most kEssCtas CTAs per SM (and the totals'
// room in the scratch).
int ess_grid(const Scratch& s, int64_t N, int cap) {
  if (cap > s.max_blocks) cap = s.max_blocks;
  if (cap > seg_cap(s.max_tiles)) cap = static_cast<int>(seg_cap(s.max_tiles));  // agg below
  const int64_t want = (N + 4 * kBlock - 1) / (4 * kBlock);
  return static_cast<int>(want < cap ? want : cap);
}
u128* ess_totals(const Scratch& s) {  // 2 * grid <= 2 * seg_cap(max_tiles) entries
  return reinterpret_cast<u128*>(s.rec);
}

}  // namespace

cudaError_t launch_ess(const Scratch& s, bool f64, const void* logw, int64_t N, double* ess,
                       double* log_total, cudaStream_t st) {
  const void* k = f64 ? reinterpret_cast<const void*>(ess_kernel<double>)
                      : reinterpret_cast<const void*>(ess_kernel<float>);
  const int cap = coop_capacity(k);
  if (!s.coop || cap < 1) return cudaErrorNotSupported;
  const int grid = ess_grid(s, N, cap);
  trace_mark(s.trace, f64 ? "ess_f64" : "ess_f32", st);
  if (f64)
    return coop_launch(ess_kernel<double>, grid, st, static_cast<const double*>(logw), N, s.glob,
                       ess_totals(s), ess, log_total, s.err);
  return coop_launch(ess_kernel<float>, grid, st, static_cast<const float*>(logw), N, s.glob,
                     ess_totals(s), ess, log_total, s.err);
}

cudaError_t launch_lgssm_step_ess(const Scratch& s, float* x, const int32_t* c, int64_t N,
                                  int init, float phi, float sigma_x, float y, float sigma_y,
                                  uint64_t seed, uint64_t step, uint32_t filter, float* logw,
                                  double* ess, double* log_total, cudaStream_t st) {
  const int cap = s.coop ? coop_capacity(reinterpret_cast<const void*>(lgssm_step_ess_kernel<4>)) : 0;
  const int grid = cap > 0 ? ess_grid(s, N, cap) : 0;
  const int64_t per = 4 * static_cast<int64_t>(grid) * kBlock;  // particles of one quadruple each
  if (grid < 1 || N > 4 * per) {  // more than the registers hold: the three kernels
    cudaError_t e = cudaSuccess;
    if (c) e = launch_copy_ancestors(s, x, 1, c, N, st);
    if (e == cudaSuccess)
      e = launch_lgssm_step(s, x, N, init, 0, phi, sigma_x, y, sigma_y, seed, step, filter, logw, st);
    if (e == cudaSuccess) e = launch_ess(s, false, logw, N, ess, log_total, st);
    return e;
  }
  const LgssmConsts k = lgssm_consts(phi, sigma_x, sigma_y);
  trace_mark(s.trace, "lgssm_step_ess", st);
  const auto kernel = N <= per       ? lgssm_step_ess_kernel<1>
                      : N <= 2 * per ? lgssm_step_ess_kernel<2>
                                     : lgssm_step_ess_kernel<4>;
  return coop_launch(kernel, grid, st, x, c, static_cast<uint32_t>(N), init, phi, sigma_x, k.sigma_0, y, k.inv_2vy,
                     make_keys(seed, step, filter, 5u), logw, s.glob, ess_totals(s), ess, log_total,
                     s.err);
}

}  // namespace rsk
