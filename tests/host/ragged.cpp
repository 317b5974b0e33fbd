// The staged chains' index arithmetic (csrc/ragged.cuh) on the host: the windows of one chunk of
// a batch are taken as a CTA of the batched Metropolis kernel takes them, and every index that
// its chains may form is checked against the staged and the global range.
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
