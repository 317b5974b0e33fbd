// ragged.cuh -- index arithmetic of a ragged batch (F filters in CSR layout, filter f owning the
// particles off[f] .. off[f+1]-1) that the kernels and the host can both run: from a particle to
// its filter, and the windows of filters whose log-weights a CTA stages. No CUDA header is needed
// to compile it for the host.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define RSK_BOTH __host__ __device__ __forceinline__
#else
#define RSK_BOTH inline
#endif

namespace rsk {
constexpr int64_t kBatchMaxN = 1 << 20;  // particles of one filter of a batched call, at most
namespace {

template <typename T>
RSK_BOTH T ld_ro(const T* p) {
#ifdef __CUDA_ARCH__
  return __ldg(p);
#else
  return *p;
#endif
}

// Particle g of the batch -> (filter f, its first particle lo, its size n, local index i).
struct PartLoc {
  int f;
  int64_t lo, n, i;
};

// Filter holding global position g: the last f with off[f] <= g (off has F + 1 entries).
RSK_BOTH int filter_of(const int64_t* __restrict__ off, int F, int64_t g) {
  int lo = 0, hi = F;  // invariant: off[lo] <= g < off[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (ld_ro(off + mid) <= g) lo = mid; else hi = mid;
  }
  return lo;
}

// One past the last position that a filter may hold: off[F], at most the handle's max_n.
RSK_BOTH int64_t batch_end(const int64_t* __restrict__ off, int F, int64_t max_n) {
  const int64_t e = ld_ro(off + F);
  return e < max_n ? e : max_n;
}

// Particles of filter f, -1 for one that is rejected (RS_ERR_ARG): it begins before 0, ends past
// the batch's end or is too long. (No two accepted filters share a position, and together they hold
// at most `end` particles, exactly if no offset is below the one before it: see descends.)
RSK_BOTH int64_t filter_size(const int64_t* __restrict__ off, int f, int64_t end) {
  const int64_t lo = ld_ro(off + f), hi = ld_ro(off + f + 1), n = hi - lo;
  return lo >= 0 && n >= 0 && hi <= end && n <= kBatchMaxN ? n : -1;
}

// An offset below the one before it: the filters then overlap, and their tiles and segments can
// outnumber the scratch. The plans give such a batch no work.
RSK_BOTH bool descends(const int64_t* __restrict__ off, int f) {
  return ld_ro(off + f + 1) < ld_ro(off + f);
}

// Position g in filter f; false for filters that are rejected and positions outside them.
RSK_BOTH bool locate_in(const int64_t* __restrict__ off, int f, int64_t end, int64_t g,
                        PartLoc& P) {
  P.f = f;
  P.lo = ld_ro(off + f);
  const int64_t hi = ld_ro(off + f + 1);
  P.n = hi - P.lo;
  P.i = g - P.lo;
  return P.lo >= 0 && hi <= end && P.n > 0 && P.n <= kBatchMaxN && P.i >= 0 && P.i < P.n;
}

// Window of the staged chains (batch_chain_kernel): from position i of filter f, the filters
// f .. f1 (whole ones while cap values hold them) up to the chunk's end (fe, ie): their values
// lo .. lo + staged - 1 go to shared memory, their particles ps .. pe - 1 are run. Filter f must
// be one that the plan accepted.
struct ChainWindow {
  int f1;
  bool whole;       // all len values are staged (else: the first cap of filter f, the only one)
  int staged;
  int64_t lo, len, ps, pe;
};
RSK_BOTH ChainWindow chain_window(const int64_t* __restrict__ off, int64_t end, int f, int i,
                                  int fe, int ie, int cap) {
  ChainWindow w;
  w.lo = ld_ro(off + f);
  const int64_t n = ld_ro(off + f + 1) - w.lo;
  w.f1 = f;
  int hi = ie > 0 ? fe : fe - 1;  // (the last filter with particles of this chunk)
  while (w.f1 < hi) {
    const int mid = (w.f1 + hi + 1) >> 1;
    const int64_t e = ld_ro(off + mid + 1), len = e - w.lo;
    if (len <= cap && len >= n && e <= end) w.f1 = mid; else hi = mid - 1;
  }
  w.len = ld_ro(off + w.f1 + 1) - w.lo;
  w.whole = w.len <= cap;
  w.staged = static_cast<int>(w.whole ? w.len : cap);
  w.ps = w.lo + i;
  w.pe = w.f1 == fe ? ld_ro(off + fe) + ie : w.lo + w.len;
  return w;
}

// Whether filter P lies inside the window, lo .. lo + len - 1, so that its value j is the window's
// value P.lo - lo + j. Offsets that do not ascend could bring a window filters that begin before it
// or end after it; nothing outside the staged values is read for them. (Their plan gives such a
// batch no work; this does not rely on it.)
RSK_BOTH bool in_window(const ChainWindow& w, const PartLoc& P) {
  return P.lo >= w.lo && P.lo + P.n <= w.lo + w.len;
}

}  // namespace
}  // namespace rsk
