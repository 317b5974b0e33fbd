// A stand-in for the CUDA runtime header in host builds of the library's warp-level code: the 32
// lanes of a warp run as coroutines of one thread that change places at every warp-wide
// operation, and the rounded operations are the host's (compiled without contraction).
#pragma once

#include <ucontext.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <functional>
#include <vector>

#define __device__
#define __forceinline__ inline
#define __global__
#define __shared__ static

struct int2 { int x, y; };
struct alignas(16) int4 { int x, y, z, w; };
struct float2 { float x, y; };
inline int4 make_int4(int x, int y, int z, int w) { return {x, y, z, w}; }
inline float2 make_float2(float x, float y) { return {x, y}; }

inline int max(int a, int b) { return a > b ? a : b; }
inline int min(int a, int b) { return a < b ? a : b; }
inline int __clz(unsigned v) { return v ? __builtin_clz(v) : 32; }
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
inline double __dadd_rn(double a, double b) { return a + b; }
inline double __dsub_rn(double a, double b) { return a - b; }
inline double __dmul_rn(double a, double b) { return a * b; }
inline float __double2float_rn(double x) { return static_cast<float>(x); }

namespace host_warp {
struct Warp {
  ucontext_t main, lane[32];
  std::vector<char> stack[32];
  uint64_t slot[2][32];  // the values exchanged by alternate operations
  int op[32];
  bool done[32];
  int current = 0;
  std::function<void(int)> body;
};
inline Warp* self = nullptr;
inline void entry(int lane) {
  self->body(lane);
  self->done[lane] = true;
  swapcontext(&self->lane[lane], &self->main);
}
// Runs body(lane) for the 32 lanes; a lane gives way at each warp-wide operation, which it passes
// when all lanes have reached it.
inline void run(const std::function<void(int)>& body) {
  static Warp w;
  self = &w;
  w.body = body;
  for (int l = 0; l < 32; ++l) {
    w.stack[l].resize(1 << 16);
    w.op[l] = 0;
    w.done[l] = false;
    getcontext(&w.lane[l]);
    w.lane[l].uc_stack.ss_sp = w.stack[l].data();
    w.lane[l].uc_stack.ss_size = w.stack[l].size();
    w.lane[l].uc_link = nullptr;
    makecontext(&w.lane[l], reinterpret_cast<void (*)()>(entry), 1, l);
  }
  for (bool any = true; any;) {
    any = false;
    for (int l = 0; l < 32; ++l) {
      if (w.done[l]) continue;
      any = true;
      w.current = l;
      swapcontext(&w.main, &w.lane[l]);
    }
  }
}
// Publishes v; returns every lane's value of this operation.
inline const uint64_t* exchange(uint64_t v) {
  const int l = self->current, b = self->op[l]++ & 1;
  self->slot[b][l] = v;
  swapcontext(&self->lane[l], &self->main);
  return self->slot[b];
}
struct ThreadIdx {
  struct X { operator int() const { return self->current; } } x;
};
}  // namespace host_warp
inline host_warp::ThreadIdx threadIdx;

template <typename T> T host_shfl(T v, int src) {
  uint64_t u = 0;
  std::memcpy(&u, &v, sizeof v);
  const uint64_t* all = host_warp::exchange(u);
  std::memcpy(&v, &all[src & 31], sizeof v);
  return v;
}
template <typename T> T __shfl_sync(unsigned, T v, int src) { return host_shfl(v, src); }
template <typename T> T __shfl_up_sync(unsigned, T v, int d) {
  const int l = host_warp::self->current;
  return host_shfl(v, l >= d ? l - d : l);
}
template <typename T> T __shfl_xor_sync(unsigned, T v, int m) {
  return host_shfl(v, host_warp::self->current ^ m);
}
inline unsigned __ballot_sync(unsigned, bool p) {
  const uint64_t* all = host_warp::exchange(p);
  unsigned m = 0;
  for (int l = 0; l < 32; ++l) m |= static_cast<unsigned>(all[l] != 0) << l;
  return m;
}
inline bool __any_sync(unsigned m, bool p) { return __ballot_sync(m, p) != 0; }
inline void __syncwarp() { host_warp::exchange(0); }
