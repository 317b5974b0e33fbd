// mcmc.cuh -- per-particle bodies of the collective-free resamplers of Section 2: the
// Metropolis chain of Code 2 and the rejection loop of Code 3, shared by the single-filter
// and batched kernels. Binary64 decisions are made on the binary32 pipes with an exact
// fallback (same outcome as the binary64 definition).
#pragma once

#include <cstdint>

#include "common.cuh"

namespace rsk {
namespace {

// ---------------------------------------------------------------------------------------
// The acceptance test u < exp_pinned(delta) (delta < 0) without evaluating the pinned
// polynomial in almost every case. e = 2^(delta log2 e) from the hardware approximation
// (PTX ex2.approx) is within a relative 1e-5 of exp(delta) for delta >= -86.5: rounding
// delta * log2 e (relative 2^-24, plus 2^-25.6 for log2 e in binary32) moves the exponent by
// at most 86.5 * 8e-8 = 7e-6 in relative terms of the result, the approximation itself is
// accurate to about 2^-22, and exp_pinned is within 2^-22 of exp. exp_pinned(delta) therefore
// lies in [e (1 - 2^-15), e (1 + 2^-15)] (a margin of about 4x), so u below the lower end
// accepts, u at or above the upper end rejects, and only u inside the band (probability
// about 6e-5 e) evaluates exp_pinned: the decision is that of u < exp_pinned(delta) always.
// Below -86.5 exp_pinned is 0 and NaN compares false, so the test is false there.
// ---------------------------------------------------------------------------------------
constexpr float kExpBand = 0x1p-15f;

__device__ __forceinline__ float exp_band_estimate(float delta) {
  float e;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(__fmul_rn(delta, 0x1.715476p+0f)));
  return e;
}

// 2^32 exp(delta), the scaling an addition inside the product (an FMA: one rounding of
// delta log2 e + 32, whose magnitude is below 2^7: 2^-18, so still within a relative 1e-5).
__device__ __forceinline__ float exp_band_estimate32(float delta) {
  float e;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(__fmaf_rn(delta, 0x1.715476p+0f, 32.0f)));
  return e;
}

// The binary32 acceptance test u < exp_pinned(delta), u = (w0 >> 8) 2^-24, from the band: with
// e = 2^32 exp(delta) and v = w0 rounded towards zero to binary32, which is at most 256 above
// 2^32 u, the test is v < e wherever |v - e| > v b + 256, b = 2^-15 / (1 - 2^-15) rounded up: then
// e (1 - 2^-15) > v, or e (1 + 2^-15) < v - 256. Where that does not hold `amb` is set (and stays
// set): probability about 6e-5 v / 2^32 a test, and every test of a NaN and of u = 0 against
// exp(delta) < 2^-24. A rise of any size, an infinite e included, is decided; with the margin taken
// from e instead of v, e = inf was not, and steps of chains that rise by more than 66 were taken
// twice (64 filters of 4096 log-weights spread over +-100, B = 29: 53 -> 26 us). Four operations
// after the exponential, no branch.
constexpr float kExpBandOfV = 0x1.0004p-15f;
__device__ __forceinline__ bool band_accept(uint32_t w0, float delta, bool& amb) {
  const float e = exp_band_estimate32(delta);
  const float v = __uint2float_rz(w0);
  const float d = __fsub_rn(v, e);
  amb |= !(fabsf(d) > __fmaf_rn(v, kExpBandOfV, 256.0f));
  return d < 0.0f;
}

// The same by definition.
__device__ __forceinline__ bool u_below_exp_exact(uint32_t w0, float delta) {
  return delta >= -86.5f && half_u01_f32(w0) < exp_pinned(delta);
}

// u < w^j / w^k from log-weights, by definition: a ratio >= 1 or a zero-weight current state
// accepts.
__device__ __noinline__ bool metropolis_accept_exact(float lwk, float lwj, uint32_t w0) {
  if (lwk == neg_inf<float>()) return true;
  const float delta = lwj - lwk;
  return delta >= 0.0f || u_below_exp_exact(w0, delta);
}

// ---------------------------------------------------------------------------------------
// Binary64 decisions on the binary32 pipes. GB300 runs binary64 arithmetic at 1/57 of the
// binary32 rate, so the binary64 test  u < exp(lw_j - lw_k)  is first decided with binary32
// arithmetic and a rigorous error bound, and evaluated exactly (binary64 subtraction,
// pinned binary64 exp, 53-bit u) only when u falls inside the uncertainty band. The outcome
// is therefore identical to the binary64 definition; the band has relative width about
// 2^-21 + 2^-23 (|lw_j| + |lw_k|), so the exact path runs for a few draws per million.
// ---------------------------------------------------------------------------------------

// Truncation of a finite binary64 to binary32 with integer operations only: |x - f| <
// 2^-23 |x| + 2^-126. Returns false (f unusable) for inf, NaN or |x| >= 2^128.
__device__ __forceinline__ bool f64_to_f32_trunc(double x, float& f) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
  const unsigned int sign = static_cast<unsigned int>(b >> 32) & 0x80000000u;
  const int e = static_cast<int>((b >> 52) & 0x7ffu);
  if (e == 0x7ff) return false;
  const int fe = e - 1023 + 127;
  if (fe >= 255) return false;
  if (fe <= 0) {  // below the binary32 normal range (or zero): 0, absolute error < 2^-126
    f = __uint_as_float(sign);
    return true;
  }
  const unsigned int m = static_cast<unsigned int>((b >> 29) & 0x7fffffu);
  f = __uint_as_float(sign | (static_cast<unsigned int>(fe) << 23) | m);
  return true;
}

// Order-preserving signed key of a binary64 (for exact comparisons without the FP64 pipe).
__device__ __forceinline__ long long f64_key(double x) {
  const long long b = __double_as_longlong(x);
  return b >= 0 ? b : (b ^ 0x7fffffffffffffffLL);
}

// Decides u < exp_pinned(lwj - lwk) for lwj < lwk, lwk > -inf, with u = 53-bit u01 of x.
// lwj_f / lwk_f are binary32 truncations (valid flags as returned above).
__device__ __noinline__ bool exact_f64_less_exp(double lwj, double lwk, uint4 x) {
  return u01_f64(x) < exp_pinned(__dsub_rn(lwj, lwk));
}

// The filter of f64_accept_lt on usable truncations lwj_f, lwk_f: true / false where they
// decide, else exact() -- the binary64 test, which the caller evaluates only then (so its
// binary64 log-weights are read only then).
template <typename Exact>
__device__ __forceinline__ bool f64_filter_lt(float lwj_f, float lwk_f, uint4 x, const Exact& exact) {
  const float df = __fsub_rn(lwj_f, lwk_f);  // <= 0 up to rounding
  // bound on |df - (lwj - lwk)|: both truncations, the subtraction's rounding, margin
  const float E = __fmaf_ru(fabsf(lwj_f) + fabsf(lwk_f), 0x1p-23f,
                            __fmaf_ru(fabsf(df), 0x1p-24f, 0x1p-124f));
  if (!(E < 0.01f)) return exact();
  // u lies in [x0 2^-32, (x0 + 1) 2^-32)
  const float u_lo = __fmul_rn(__uint2float_rd(x.x), 0x1p-32f);
  const float u_hi = __fmul_rn(__fadd_ru(__uint2float_ru(x.x), 1.0f), 0x1p-32f);
  if (!(df >= -86.5f)) {  // exp(df) < 2^-124: the binary64 ratio is below e^-86 < 2^-32 <= u
    if (x.x != 0u) return false;
    return exact();
  }
  // ef = exp(df) within a relative 1e-5 (exp_band_estimate); exp(lwj - lwk) within
  // ef * exp(+-E) * (1 +- 1e-5) (1 +- 2^-52): m bounds all of it
  const float ef = exp_band_estimate(df);
  const float m = __fmaf_ru(E, 1.02f, kExpBand);
  const float lo = __fmul_rd(ef, __fsub_rd(1.0f, m));
  const float hi = __fmul_ru(ef, __fadd_ru(1.0f, m));
  if (u_hi < lo) return true;
  if (u_lo >= hi) return false;
  return exact();
}

__device__ __forceinline__ bool f64_accept_lt(double lwj, float lwj_f, bool okj, double lwk,
                                              float lwk_f, bool okk, uint4 x) {
  if (!(okj && okk)) return exact_f64_less_exp(lwj, lwk, x);
  return f64_filter_lt(lwj_f, lwk_f, x, [&] { return exact_f64_less_exp(lwj, lwk, x); });
}

// ---------------------------------------------------------------------------------------
// Binary32 sidecar of binary64 log-weights. The binary64 chains gather a 4-byte sidecar per
// proposal instead of the 8-byte log-weight: the truncation of lw_j to binary32 when usable,
// -inf for lw_j = -inf, a NaN otherwise (NaN, +inf, or beyond the binary32 range). Truncation
// is monotone, so t_j > t_k implies lw_j > lw_k and t_j < t_k implies lw_j < lw_k; the
// binary64 values are read only when the sidecars are equal or NaN, and for the exact
// fallback of the filter. Every decision equals the one taken from the binary64 values.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ float f64_sidecar(double x) {
  float f;
  if (f64_to_f32_trunc(x, f)) return f;
  return is_neg_inf(x) ? -INFINITY : __int_as_float(0x7fffffff);
}

constexpr int kUnroll64 = 4;  // binary64 chains (2 measured slower)
// Log-weights of which two of this size put the filter's bound past 0.01 (2 * 41943 * 2^-23).
constexpr float kWide64 = 41000.0f;

// S consecutive steps (S = 1 or even, s even) of a binary32 chain of e steps in state (k, lwk), with
// S = 2 and without ZEROS those of them below e: the blocks drawn and their proposals gathered
// together, then the decisions from the band (band_accept: a ratio >= 1 is e >= 2^32 (1 - 1e-5),
// never rejected by it). If any of them was undecided they are taken again by definition: one branch
// for S steps. With ZEROS a state of zero weight accepts without that branch, which is taken from
// the proposals at hand (200003 particles, 99 of 100 of weight zero, B = 29: 46 -> 30 us). Without,
// such a state is decided there where the proposal's weight is zero too, and undecided steps are
// drawn and gathered again: the staged chains take that form, which the operation a step and the
// registers held for the branch cost 4 %.
template <int S, bool SMALL, bool ZEROS, typename Gather>
__device__ __forceinline__ void metropolis_steps(uint32_t& k, float& lwk, const Gather& gather,
                                                 uint32_t n, int32_t s, int32_t e, const Keys& keys,
                                                 const DrawRow& row) {
  uint32_t w[S], j[S];
  float lwj[S];
#pragma unroll
  for (int q = 0; q < S; q += 2) {
    const uint4 x = draw(keys, row, (static_cast<uint32_t>(s) >> 1) + q / 2);
    w[q] = x.x;
    j[q] = half_index<SMALL>(x.x, x.y, n);
    lwj[q] = gather(j[q]);
    if constexpr (S > 1) {
      w[q + 1] = x.z;
      j[q + 1] = half_index<SMALL>(x.z, x.w, n);
      lwj[q + 1] = gather(j[q + 1]);
    }
  }
  const uint32_t k0 = k;
  const float lwk0 = lwk;
  bool amb = false;
#pragma unroll
  for (int q = 0; q < S; ++q) {
    bool yes;
    if constexpr (ZEROS) {
      const bool none = lwk == -INFINITY;
      bool open = false;
      yes = band_accept(w[q], __fsub_rn(lwj[q], lwk), open) || none;
      amb |= open && !none;
    } else {
      yes = band_accept(w[q], __fsub_rn(lwj[q], lwk), amb);
    }
    if (yes && (S != 2 || ZEROS || q == 0 || s + 1 < e)) {
      k = j[q];
      lwk = lwj[q];
    }
  }
  if (amb) {
    k = k0;
    lwk = lwk0;
#pragma unroll 1
    for (int32_t t = s; t < s + S && t < e; ++t) {
      uint32_t w0, jt;
      float lwt;
      if constexpr (ZEROS) {
        w0 = w[0];
        jt = j[0];
        lwt = lwj[0];
#pragma unroll
        for (int q = 1; q < S; ++q) {  // (the next step's to the front: no indexing)
          w[q - 1] = w[q];
          j[q - 1] = j[q];
          lwj[q - 1] = lwj[q];
        }
      } else {
        const uint4 x = draw(keys, row, static_cast<uint32_t>(t >> 1));
        w0 = (t & 1) ? x.z : x.x;
        jt = half_index<SMALL>(w0, (t & 1) ? x.w : x.y, n);
        lwt = gather(jt);
      }
      if (metropolis_accept_exact(lwk, lwt, w0)) {
        k = jt;
        lwk = lwt;
      }
    }
  }
}

// Metropolis chain of particle i over n < 2^31 (SMALL: n < 2^24) binary32 log-weights (Code 2),
// from the state i with log-weight lwk; gather(j) reads the log-weight of proposal j. B steps;
// steps 2m and 2m + 1 take the two halves of the block of counter (i, m) (half_u01_f32,
// half_index), so a chain draws ceil(B / 2) blocks. P blocks (2 P proposals) are issued together.
// Returns the ancestor.
template <bool SMALL, int P, bool ZEROS, typename Gather>
__device__ __forceinline__ int32_t metropolis_chain(float lwk, const Gather& gather, uint32_t n,
                                                    int32_t B, const Keys& keys, uint32_t i) {
  uint32_t k = i;
  const DrawRow row = draw_row(keys, i);
  int32_t s = 0;
  for (; s + 2 * P <= B; s += 2 * P)
    metropolis_steps<2 * P, SMALL, ZEROS>(k, lwk, gather, n, s, B, keys, row);
  if constexpr (ZEROS) {
    if constexpr (P > 1)
      for (; s + 2 <= B; s += 2)
        metropolis_steps<2, SMALL, ZEROS>(k, lwk, gather, n, s, B, keys, row);
    // an odd last step gathers one proposal from memory (with the block's other one 10^6 particles
    // took 9.6 instead of 6.4 us at B = 1, 39.8 instead of 36.8 with Permute at B = 5)
    if (s < B) metropolis_steps<1, SMALL, ZEROS>(k, lwk, gather, n, s, B, keys, row);
  } else {  // (from shared memory it costs less than the code for it)
    for (; s < B; s += 2) metropolis_steps<2, SMALL, ZEROS>(k, lwk, gather, n, s, B, keys, row);
  }
  return static_cast<int32_t>(k);
}

// The chain of particle i with its proposals gathered from the log-weights themselves.
template <bool SMALL, int P>
__device__ __forceinline__ int32_t metropolis_one(const float* __restrict__ lw, int64_t n,
                                                  int32_t B, const Keys& keys, int64_t i,
                                                  int* err) {
  const float lwi = __ldg(lw + i);
  if (nonfinite_logw(lwi)) flag_error(err, RS_ERR_NONFINITE);
  const auto gather = [&](uint32_t j) { return __ldg(lw + j); };
  return metropolis_chain<SMALL, P, true>(lwi, gather, static_cast<uint32_t>(n), B, keys,
                                          static_cast<uint32_t>(i));
}

// A Metropolis step of a binary64 chain, by definition: state lwk, proposal lwj, u from the words x.
__device__ __forceinline__ bool f64_step_accept(double lwk, double lwj, uint2 x) {
  const long long kk = f64_key(lwk), kj = f64_key(lwj), none = f64_key(-INFINITY);
  if (kk == none || kj >= kk) return true;  // zero-weight state, or ratio >= 1
  return kj != none && exact_f64_less_exp(lwj, lwk, make_uint4(x.x, x.y, 0u, 0u));
}

// A Metropolis step of a binary64 chain decided from sidecars (f64_sidecar): state k with
// sidecar tk, proposal j with tj, u from the words x; the binary64 log-weights lw[k], lw[j] are read
// only when the sidecars cannot decide.
__device__ __forceinline__ bool sc_step_accept(const double* __restrict__ lw, uint32_t k, float tk,
                                               uint32_t j, float tj, uint2 x) {
  if (tk == -INFINITY) return true;     // zero-weight state (tk = -inf iff lw_k = -inf)
  if (tj > tk) return true;             // lw_j > lw_k: ratio above 1
  const uint4 x4 = make_uint4(x.x, x.y, 0u, 0u);
  bool open = true, yes = false;        // (equal sidecars or a NaN: undecided)
  if (tj < tk) {
    if (tj == -INFINITY) return false;  // zero-weight proposal
    open = false;
    yes = f64_filter_lt(tj, tk, x4, [&] { open = true; return false; });
  }
  return open ? f64_step_accept(__ldg(lw + k), __ldg(lw + j), x) : yes;
}

// The same decision from the sidecars tj, tk and the band alone in almost every case, without
// branches: with e = 2^32 exp(tj - tk), v = x0 rounded towards zero to binary32 (2^32 u lies in
// [v, v + 257)) and m the filter's relative margin (f64_filter_lt), the step accepts iff v < e
// wherever |v - e| > v m' + 260, m' >= m / (1 - m), and the truncations' bound E is below 0.01 (so m
// below 0.0103): then e (1 - m) > v + 257, or e (1 + m) < v. Elsewhere `amb` is set (and stays set): a
// zero-weight state, a NaN, wide bounds, u next to the ratio. Equal sidecars and ratios above 1, of
// any size, are covered by the same inequality. A zero-weight proposal is e = 0, rejected, from any
// state of non-zero weight. (The chain of tests took about 45 instructions, this 16.)
__device__ __forceinline__ bool band_accept_sc(uint32_t x0, float tj, float tk, bool& amb) {
  const float df = __fsub_rn(tj, tk);
  const float E = __fmaf_ru(fabsf(tj) + fabsf(tk), 0x1p-23f,
                            __fmaf_ru(fabsf(df), 0x1p-24f, 0x1p-124f));
  const float e = exp_band_estimate32(df);
  const float v = __uint2float_rz(x0);
  const float d = __fsub_rn(v, e);
  const float w = __fmaf_ru(v, __fmaf_ru(E, 1.04f, 1.02f * kExpBand), 260.0f);
  amb |= !(fabsf(d) > w && E < 0.01f) && !(is_neg_inf(tj) && tk > -INFINITY);
  return d < 0.0f;
}

// metropolis_chain for n < 2^31 binary64 log-weights lw from the state i with sidecar tk:
// gather(j) reads the sidecar of proposal j (4 bytes instead of 8). Steps kUnroll64 at a time
// from the band; if any of them was undecided their decisions are taken again from the proposals at
// hand: by sc_step_accept, or, from a state so large that the filter cannot hold (unnormalised
// log-likelihoods: every step is decided so), by definition on the binary64 log-weights, read
// together. The decisions, and so the ancestor, are those of the binary64 definition. 200003
// particles near -10^6, B = 29: 343 -> 268 us; log-weights spread over +-100: 51 -> 28 (rises above
// 66 were undecided, and undecided steps were drawn and gathered again one by one).
template <typename Gather>
__device__ __forceinline__ int32_t metropolis_chain_sc(const double* __restrict__ lw, float tk,
                                                       const Gather& gather, uint32_t n,
                                                       int32_t B, const Keys& keys, uint32_t i) {
  uint32_t k = i;
  const DrawRow row = draw_row(keys, i);
  for (int32_t s = 0; s < B; s += kUnroll64) {
    uint2 x[kUnroll64];  // (the words of u)
    uint32_t j[kUnroll64];
    float tj[kUnroll64];
#pragma unroll
    for (int q = 0; q < kUnroll64; ++q) {
      if (s + q < B) {
        const uint4 r = draw(keys, row, static_cast<uint32_t>(s + q));
        x[q] = make_uint2(r.x, r.y);
        j[q] = uniform_index(r, n);
        tj[q] = gather(j[q]);
      }
    }
    const uint32_t k0 = k;
    const float tk0 = tk;
    bool amb = false;
#pragma unroll
    for (int q = 0; q < kUnroll64; ++q) {
      if (s + q < B && band_accept_sc(x[q].x, tj[q], tk, amb)) {
        k = j[q];
        tk = tj[q];
      }
    }
    if (amb) {
      k = k0;
      tk = tk0;
      if (fabsf(tk) > kWide64 && tk != -INFINITY) {
        double lwk = __ldg(lw + k), lwj[kUnroll64];
#pragma unroll
        for (int q = 0; q < kUnroll64; ++q) lwj[q] = s + q < B ? __ldg(lw + j[q]) : 0.0;
#pragma unroll
        for (int q = 0; q < kUnroll64; ++q) {
          if (s + q < B && f64_step_accept(lwk, lwj[q], x[q])) {
            k = j[q];
            tk = tj[q];
            lwk = lwj[q];
          }
        }
      } else {
#pragma unroll
        for (int q = 0; q < kUnroll64; ++q) {
          if (s + q < B && sc_step_accept(lw, k, tk, j[q], tj[q], x[q])) {
            k = j[q];
            tk = tj[q];
          }
        }
      }
    }
  }
  return static_cast<int32_t>(k);
}

// The chain of particle i with its proposals gathered from the binary64 log-weights (batched
// chains, which have no sidecars in memory).
__device__ __forceinline__ int32_t metropolis_one(const double* __restrict__ lw, int64_t n,
                                                  int32_t B, const Keys& keys, int64_t i,
                                                  int* err) {
  const double lwi = __ldg(lw + i);
  if (nonfinite_logw(lwi)) flag_error(err, RS_ERR_NONFINITE);
  return metropolis_chain_sc(lw, f64_sidecar(lwi),
                             [&](uint32_t j) { return f64_sidecar(__ldg(lw + j)); },
                             static_cast<uint32_t>(n), B, keys, static_cast<uint32_t>(i));
}

// The chain of particle i with its proposals gathered from the sidecars lwf in memory.
__device__ __forceinline__ int32_t metropolis_one_sc(const double* __restrict__ lw,
                                                     const float* __restrict__ lwf, int64_t n,
                                                     int32_t B, const Keys& keys, int64_t i,
                                                     int* err) {
  const double lwi = __ldg(lw + i);
  if (nonfinite_logw(lwi)) flag_error(err, RS_ERR_NONFINITE);
  return metropolis_chain_sc(lw, f64_sidecar(lwi), [&](uint32_t j) { return __ldg(lwf + j); },
                             static_cast<uint32_t>(n), B, keys, static_cast<uint32_t>(i));
}

// Rejection loop of particle i (Code 3): attempt 0 proposes j = i, attempt s >= 1 a uniform
// j; binary64 attempts draw from counter (i, s), binary32 ones from half s mod 2 of the block
// of counter (i, floor(s/2)) (half_u01_f32, half_index); accept when u < exp(lw^j - log w_max).
// A log-weight above the bound is flagged and accepted; max_trials attempts without
// acceptance keep i and flag the cap.
//
// ---------------------------------------------------------------------------------------
// Rejection with warp refill. Trial counts vary per particle (a geometric tail, Section 2.2),
// and a warp would wait for its slowest lane. Instead every warp owns a run of particles and
// a lane that settles its particle takes the next unstarted one of the run, so all lanes stay
// busy. Attempt s of particle i always uses the same draw: the result does not depend on the
// schedule.
// ---------------------------------------------------------------------------------------

// The bound log w_max in the forms the attempts compare against. clamp: partial rejection
// control (Section 2.2): the attempts sample v = min(w, v_max) with v_max = the bound, so a
// weight above it is the clamped weight v_max (ratio 1, accepted, not an error).
struct RejBound {
  double lwmax;
  float lwmax_rn;  // RN(log w_max) in binary32 (the binary32 scheme's bound)
  float lwmax_f;   // truncation (the binary64 scheme's filter)
  bool okm;
  long long km;
  bool clamp;
};
__device__ __forceinline__ RejBound make_bound(double log_wmax, bool clamp = false) {
  RejBound r;
  r.clamp = clamp;
  r.lwmax = log_wmax;
  r.lwmax_rn = static_cast<float>(log_wmax);
  r.okm = f64_to_f32_trunc(log_wmax, r.lwmax_f);
  r.km = f64_key(log_wmax);
  return r;
}

// Decision of one rejection attempt with the uniform's word w0 (binary32) or draw x (binary64) and
// proposal log-weight lwj: accept when u < exp(lw^j - log w_max); a log-weight above the bound
// is accepted and, unless clamped, sets over (which the caller flags if the attempt counts).
__device__ __forceinline__ bool rejection_accept(const RejBound& rb, uint32_t w0, float lwj,
                                                 bool& over) {
  const float delta = lwj - rb.lwmax_rn;
  if (delta > 0.0f) {
    over |= !rb.clamp;
    return true;
  }
  if (delta == 0.0f) return true;
  bool amb = false;
  const bool yes = band_accept(w0, delta, amb);
  return amb ? u_below_exp_exact(w0, delta) : yes;
}

__device__ __forceinline__ bool rejection_accept(const RejBound& rb, uint4 x, double lwj,
                                                 bool& over) {
  const long long kj = f64_key(lwj);
  if (kj > rb.km && !is_nan(lwj)) {  // above the bound (NaN never compares)
    over |= !rb.clamp;
    return true;
  }
  if (kj == rb.km) return true;  // ratio exactly 1
  if (kj == f64_key(-INFINITY) || is_nan(lwj)) return false;
  float lwj_f;
  const bool okj = f64_to_f32_trunc(lwj, lwj_f);
  return f64_accept_lt(lwj, lwj_f, okj, rb.lwmax, rb.lwmax_f, rb.okm, x);
}

// rejection_accept for a binary64 proposal decided from its sidecar tj (f64_sidecar); the
// binary64 log-weight lw[j] is read only when the sidecar cannot decide. Same decision.
__device__ __forceinline__ bool rejection_accept_sc(const RejBound& rb, uint4 x,
                                                    const double* __restrict__ lw, int64_t j,
                                                    float tj, bool& over) {
  if (!(tj == tj) || !rb.okm || tj == rb.lwmax_f) return rejection_accept(rb, x, __ldg(lw + j), over);
  if (tj > rb.lwmax_f) {  // lw_j above the bound
    over |= !rb.clamp;
    return true;
  }
  if (tj == -INFINITY) return false;
  return f64_filter_lt(tj, rb.lwmax_f, x,
                       [&] { return exact_f64_less_exp(__ldg(lw + j), rb.lwmax, x); });
}

// Attempts a lane issues together (rejection_attempts): 2 measured 7-16 % faster than 1 at
// N = 2^20 (y = 2 and 4); 4 is faster still at y = 4 but slower at y = 2, where most particles
// settle within two attempts.
constexpr int kRejBatch = 2;

// Attempts s .. s + K - 1 of particle i (those below max_trials) with their draws and
// proposal gathers issued together -- the draws are counter-based, so they do not depend on
// the outcome of earlier attempts -- then decided in order: the first accepted one is the
// result, exactly as attempting one at a time. Returns true with j when one accepts.
template <int K, typename T>
__device__ __forceinline__ bool rejection_attempts(const T* __restrict__ lw, int64_t n,
                                                   const RejBound& rb, const Keys& keys,
                                                   int64_t i, uint32_t s, T lwi,
                                                   int64_t max_trials, int64_t& j, bool& over) {
  uint4 x[K];
  int64_t jq[K];
  T lwj[K];
#pragma unroll
  for (int q = 0; q < K; ++q) {
    const uint32_t sq = s + static_cast<uint32_t>(q);
    x[q] = draw(keys, static_cast<uint32_t>(i), sq);
    jq[q] = (sq > 0) ? uniform_index(x[q], static_cast<uint32_t>(n)) : i;
    lwj[q] = (sq > 0) ? __ldg(lw + jq[q]) : lwi;
  }
#pragma unroll
  for (int q = 0; q < K; ++q) {
    if (static_cast<int64_t>(s) + q >= max_trials) return false;
    if (rejection_accept(rb, x[q], lwj[q], over)) {
      j = jq[q];
      return true;
    }
  }
  return false;
}

// The same for binary32 log-weights, whose attempts 2m and 2m + 1 share the block of counter
// (i, m) (s even, K even): K / 2 blocks for K attempts.
template <int K>
__device__ __forceinline__ bool rejection_attempts(const float* __restrict__ lw, int64_t n,
                                                   const RejBound& rb, const Keys& keys,
                                                   int64_t i, uint32_t s, float lwi,
                                                   int64_t max_trials, int64_t& j, bool& over) {
  static_assert(K % 2 == 0, "whole blocks");
  uint32_t w[K];
  float lwj[K];
  int64_t jq[K];
#pragma unroll
  for (int p = 0; p < K / 2; ++p) {
    const uint4 x = draw(keys, static_cast<uint32_t>(i), s / 2 + static_cast<uint32_t>(p));
    const uint32_t s0 = s + 2 * static_cast<uint32_t>(p);
    jq[2 * p] = (s0 > 0) ? half_index<false>(x.x, x.y, static_cast<uint32_t>(n)) : i;
    w[2 * p] = x.x;
    jq[2 * p + 1] = half_index<false>(x.z, x.w, static_cast<uint32_t>(n));
    w[2 * p + 1] = x.z;
    lwj[2 * p] = (s0 > 0) ? __ldg(lw + jq[2 * p]) : lwi;
    lwj[2 * p + 1] = __ldg(lw + jq[2 * p + 1]);
  }
#pragma unroll
  for (int q = 0; q < K; ++q) {
    if (static_cast<int64_t>(s) + q >= max_trials) return false;
    if (rejection_accept(rb, w[q], lwj[q], over)) {
      j = jq[q];
      return true;
    }
  }
  return false;
}

// rejection_attempts for binary64 log-weights with their sidecars lwf (ti: the sidecar of
// particle i's own log-weight): the proposals gather 4 bytes instead of 8; same outcome.
template <int K>
__device__ __forceinline__ bool rejection_attempts_sc(const double* __restrict__ lw,
                                                      const float* __restrict__ lwf, int64_t n,
                                                      const RejBound& rb, const Keys& keys,
                                                      int64_t i, uint32_t s, float ti,
                                                      int64_t max_trials, int64_t& j, bool& over) {
  uint4 x[K];
  int64_t jq[K];
  float tj[K];
#pragma unroll
  for (int q = 0; q < K; ++q) {
    const uint32_t sq = s + static_cast<uint32_t>(q);
    x[q] = draw(keys, static_cast<uint32_t>(i), sq);
    jq[q] = (sq > 0) ? uniform_index(x[q], static_cast<uint32_t>(n)) : i;
    tj[q] = (sq > 0) ? __ldg(lwf + jq[q]) : ti;
  }
#pragma unroll
  for (int q = 0; q < K; ++q) {
    if (static_cast<int64_t>(s) + q >= max_trials) return false;
    if (rejection_accept_sc(rb, x[q], lw, jq[q], tj[q], over)) {
      j = jq[q];
      return true;
    }
  }
  return false;
}

// ---------------------------------------------------------------------------------------
// The end of a warp's run: no particle left to take in and at most half of its lanes still busy.
// The trial counts have a geometric tail, and a lane alone makes two attempts per round of
// dependent steps (draw, gather, decision: about a microsecond), so the longest particle of a
// call set its time (100000 particles at y = 4: 880 attempts, 432 us). The draws are counted, not
// drawn in turn, so here the lanes share the particles that are left: with m particles each gets
// the largest power of two of lanes <= 32 / m, lane r of a group takes attempts s + 2r and
// s + 2r + 1, and the first accepted one in attempt order is the result, exactly as one lane
// would have found it (attempts after it leave no trace: `over` counts only for the winner).
// ---------------------------------------------------------------------------------------
// One particle of a warp: local index i of the n particles from lo on, its attempts made so far,
// its log-weight and the counter tag of its filter.
template <typename T>
struct RejParticle {
  bool active;
  uint32_t i, n, tag;
  int64_t lo;
  uint64_t s;
  T lwi;
};

__device__ __forceinline__ uint64_t shfl_u64(uint64_t v, int src) {
  const uint32_t lo = __shfl_sync(0xffffffffu, static_cast<uint32_t>(v), src);
  const uint32_t hi = __shfl_sync(0xffffffffu, static_cast<uint32_t>(v >> 32), src);
  return (static_cast<uint64_t>(hi) << 32) | lo;
}

// attempts(P, s, j, over): rejection_attempts of particle P from attempt s on; settle(P, j): its
// result. Called by all 32 lanes, each with its own particle (or inactive).
template <typename T, typename Attempts, typename Settle>
__device__ __forceinline__ void rejection_tail(RejParticle<T> own, int64_t max_trials, int* err,
                                               const Attempts& attempts, const Settle& settle) {
  const int lane = threadIdx.x & 31;
  const uint64_t most = static_cast<uint64_t>(max_trials);
  for (;;) {
    const unsigned mask = __ballot_sync(0xffffffffu, own.active);
    if (mask == 0u) return;
    const int m = __popc(mask);
    const int lg = 31 - __clz(32 / m), g = 1 << lg;
    const int grp = lane >> lg, r = lane & (g - 1);
    const int src = grp < m ? static_cast<int>(__fns(mask, 0, grp + 1)) : 0;  // the group's owner
    RejParticle<T> P;
    P.i = __shfl_sync(0xffffffffu, own.i, src);
    P.n = __shfl_sync(0xffffffffu, own.n, src);
    P.tag = __shfl_sync(0xffffffffu, own.tag, src);
    P.lo = static_cast<int64_t>(shfl_u64(static_cast<uint64_t>(own.lo), src));
    P.s = shfl_u64(own.s, src);
    P.lwi = __shfl_sync(0xffffffffu, own.lwi, src);
    const uint64_t s = P.s + 2 * static_cast<uint64_t>(r);
    bool acc = false, over = false;
    int64_t j = 0;
    if (grp < m && s < most) acc = attempts(P, static_cast<uint32_t>(s), j, over);
    const unsigned won = __ballot_sync(0xffffffffu, acc);
    const unsigned ones = g == 32 ? 0xffffffffu : (1u << g) - 1u;
    if (acc && __ffs(won & (ones << (grp << lg))) == lane + 1) {
      settle(P, j);
      if (over) flag_error(err, RS_ERR_BOUND_VIOLATED);
    }
    if (own.active) {
      const int rank = __popc(mask & ((1u << lane) - 1u));
      own.s += 2 * static_cast<uint64_t>(g);
      if (won & (ones << (rank << lg))) {
        own.active = false;
      } else if (own.s >= most) {
        flag_error(err, RS_ERR_REJECTION_CAP);
        settle(own, static_cast<int64_t>(own.i));
        own.active = false;
      }
    }
  }
}
static_assert(kRejBatch == 2, "two attempts per lane and round");

}  // namespace
}  // namespace rsk
