// The ragged batches' index arithmetic (csrc/ragged.cuh) on the host. chain_chunk: the windows of one
// chunk of a batch are taken as a CTA of the batched Metropolis kernel takes them, and every index
// that its chains may form is checked against the staged and the global range. batch_sizes: the
// filters' sizes as the plans accept them.
#include "ragged.cuh"

using namespace rsk;

// Chunk (f, i) .. (fe, ie) of the batch; work: exclusive prefix of the filters' work (equal
// entries: a filter that the plan rejects, or empty). visits[g] counts the chains run at particle
// g, staged[g] those whose filter is wholly staged. Returns 0, or 1 for a shared index outside
// the staged values, 2 for a global one outside [0, total).
extern "C" int chain_chunk(const int64_t* off, int F, int64_t total, const int64_t* work, int f,
                           int i, int fe, int ie, int cap, int32_t* visits, int32_t* staged) {
  while (f < fe || (f == fe && i < ie)) {
    if (work[f + 1] == work[f]) {
      ++f;
      i = 0;
      continue;
    }
    const ChainWindow w = chain_window(off, total, f, i, fe, ie, cap);
    if (w.staged < 0 || w.staged > cap) return 1;
    if (w.lo < 0 || w.lo + w.staged > total) return 2;
    for (int64_t g = w.ps; g < w.pe; ++g) {
      const int ff = w.f1 > f ? f + filter_of(off + f, w.f1 + 1 - f, g) : f;
      PartLoc P;
      if (!locate_in(off, ff, total, g, P)) continue;
      if (g >= total) return 2;
      ++visits[g];
      if (!in_window(w, P)) continue;
      if (w.whole) ++staged[g];
      for (int64_t j = 0; j < P.n; j += P.n > 64 ? P.n / 61 : 1) {
        const int64_t s = P.lo - w.lo + j;  // the shared index of value j
        if (w.whole || j < cap) {
          if (s < 0 || s >= w.staged) return 1;
        } else if (P.lo + j < 0 || P.lo + j >= total) {
          return 2;
        }
      }
    }
    f = w.f1 + 1;
    i = 0;
  }
  return 0;
}

// n[f]: particles of filter f that the plan gives work, 0 for a rejected one or a void batch;
// returns 1 if the call is to be reported, +2 if the batch is void.
extern "C" int batch_sizes(const int64_t* off, int F, int64_t max_n, int64_t* n) {
  const int64_t end = batch_end(off, F, max_n);
  bool down = false, rejected = false;
  for (int f = 0; f < F; ++f) {
    n[f] = filter_size(off, f, end);
    rejected |= n[f] < 0;
    down |= descends(off, f);
    if (n[f] < 0) n[f] = 0;
  }
  if (down)
    for (int f = 0; f < F; ++f) n[f] = 0;
  return (rejected ? 1 : 0) + (down ? 2 : 0);
}
