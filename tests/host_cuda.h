// Enough of CUDA's device language for a host compiler to run kernels of this library, block by block, on
// the CPU: a thread is a fiber that runs to its next warp or block collective.  Stands in for ptx.cuh.
//
// Cell<T> is a shared-memory word that reports data races: an access by one lane and a write by another
// with no __syncwarp() or __syncthreads() between them.  Votes and shuffles order no memory.
#pragma once
#include <ucontext.h>
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <vector>

#define __global__ static
#define __device__
#define __host__
#define __forceinline__ inline
#define __launch_bounds__(...)
#define __shared__ static
#define __align__(n) alignas(n)
#define asm(...) host_mma(d, a0, a1, a2, a3, b0, b1, c)

struct float2 { float x, y; };
struct alignas(16) float4 { float x, y, z, w; };
struct alignas(16) uint4 { uint32_t x, y, z, w; };
inline float2 make_float2(float x, float y) { return {x, y}; }
struct Dim { unsigned x; };
static Dim threadIdx, blockIdx, blockDim, gridDim;

namespace host {

struct Word10 { uint32_t v[10]; };
enum Wait { READY, WARP, BLOCK, DONE };
struct Fiber {
  ucontext_t ctx;
  Wait wait;
  const char* what;
  Word10 in;
};
struct Warp { Word10 snap[32]; int epoch; };

static std::vector<Fiber> fibers;
static std::vector<Warp> warps;
static std::vector<char> stacks;
static ucontext_t scheduler;
static std::function<void()> body;
static int current, races, mmas, matches, tests, epochs;   // mmas, matches: by any warp; epochs: begun so far
constexpr size_t kStack = 64 * 1024;

inline void die(const char* why) { std::fprintf(stderr, "host_cuda: %s\n", why); std::abort(); }
inline void entry() { body(); fibers[current].wait = DONE; swapcontext(&fibers[current].ctx, &scheduler); }
inline Warp& warp() { return warps[current / 32]; }
inline void yield(Wait w, const char* what) {
  fibers[current].wait = w;
  fibers[current].what = what;
  const int me = current;
  swapcontext(&fibers[me].ctx, &scheduler);
}
// A collective of the whole warp: every lane's words, as they were when the last lane came.
inline const Word10* all_lanes(const char* what, const Word10& in) {
  fibers[current].in = in;
  yield(WARP, what);
  return warp().snap;
}
inline void run_block(int threads) {
  fibers.resize(threads);
  warps.resize((threads + 31) / 32);
  for (Warp& w : warps) w.epoch = ++epochs;
  stacks.resize(threads * kStack);
  for (int i = 0; i < threads; ++i) {
    Fiber& f = fibers[i];
    getcontext(&f.ctx);
    f.ctx.uc_stack = {};
    f.ctx.uc_stack.ss_sp = &stacks[i * kStack];
    f.ctx.uc_stack.ss_size = kStack;
    f.ctx.uc_link = nullptr;
    f.wait = READY;
    makecontext(&f.ctx, entry, 0);
  }
  for (bool live = true; live;) {
    bool ran = false;
    live = false;
    for (int w = 0; w * 32 < threads; ++w) {
      const int lo = 32 * w, hi = std::min(threads, lo + 32);
      for (current = lo; current < hi; ++current)
        if (fibers[current].wait == READY) {
          threadIdx.x = current;
          swapcontext(&scheduler, &fibers[current].ctx);
          ran = true;
        }
      int waiting = 0, done = 0;
      const char* what = nullptr;
      for (int i = lo; i < hi; ++i) {
        done += fibers[i].wait == DONE;
        if (fibers[i].wait != WARP) continue;
        if (what && std::strcmp(what, fibers[i].what) != 0) die("lanes of a warp wait at different collectives");
        what = fibers[i].what;
        ++waiting;
      }
      live = live || done < hi - lo;
      if (waiting == 0) continue;
      if (waiting != hi - lo) die("a collective that not every lane of the warp reaches");
      for (int i = lo; i < hi; ++i) { warps[w].snap[i - lo] = fibers[i].in; fibers[i].wait = READY; }
      if (std::strcmp(what, "__syncwarp") == 0) warps[w].epoch = ++epochs;
      ran = true;
    }
    if (!ran && live) {                               // every live thread is at the block's barrier
      for (Fiber& f : fibers) if (f.wait == WARP || f.wait == DONE) die("a thread misses __syncthreads()");
      for (Fiber& f : fibers) f.wait = READY;
      for (Warp& w : warps) w.epoch = ++epochs;
    }
  }
}
template <typename F>
inline void launch(unsigned grid, unsigned block, F&& kernel) {
  gridDim.x = grid;
  blockDim.x = block;
  body = kernel;
  for (blockIdx.x = 0; blockIdx.x < grid; ++blockIdx.x) run_block((int)block);
}

template <typename T>
struct Cell {                                         // a shared word that one warp uses
  T v;
  int write_epoch, write_lane, read_epoch;
  uint32_t readers;
  operator T() {
    const int lane = current % 32, e = warp().epoch;
    if (write_epoch == e && write_lane != lane) ++races;
    if (read_epoch != e) { read_epoch = e; readers = 0; }
    readers |= 1u << lane;
    return v;
  }
  T operator=(T x) {
    const int lane = current % 32, e = warp().epoch;
    if (write_epoch == e && write_lane != lane) ++races;
    if (read_epoch == e && (readers & ~(1u << lane))) ++races;
    write_epoch = e;
    write_lane = lane;
    return v = x;
  }
  T operator=(Cell& o) { return *this = (T)o; }
};

}  // namespace host

template <typename T> inline uint32_t host_bits(T x) { uint32_t u = 0; std::memcpy(&u, &x, sizeof(T)); return u; }
template <typename T> inline T host_from(uint32_t u) { T x; std::memcpy(&x, &u, sizeof(T)); return x; }
template <typename T> inline const host::Word10* host_collect(const char* what, T x) {
  static_assert(sizeof(T) <= 4, "32-bit values");
  return host::all_lanes(what, {{host_bits(x)}});
}
inline int host_lane() { return host::current % 32; }

inline void __syncwarp() { host_collect("__syncwarp", 0); }
inline void __syncthreads() { host::yield(host::BLOCK, "__syncthreads"); }
template <typename T> inline T __shfl_sync(unsigned, T x, int from) {
  return host_from<T>(host_collect("__shfl_sync", x)[from & 31].v[0]);
}
template <typename T> inline T __shfl_up_sync(unsigned, T x, int by) {
  const int lane = host_lane();
  const host::Word10* w = host_collect("__shfl_up_sync", x);
  return lane < by ? x : host_from<T>(w[lane - by].v[0]);
}
template <typename T> inline T __shfl_xor_sync(unsigned, T x, int mask) {
  const int lane = host_lane();
  if constexpr (sizeof(T) == 8) {
    uint64_t u;
    std::memcpy(&u, &x, 8);
    const host::Word10* w = host::all_lanes("__shfl_xor_sync", {{(uint32_t)u, (uint32_t)(u >> 32)}});
    u = w[lane ^ mask].v[0] | (uint64_t)w[lane ^ mask].v[1] << 32;
    std::memcpy(&x, &u, 8);
    return x;
  } else {
    return host_from<T>(host_collect("__shfl_xor_sync", x)[lane ^ mask].v[0]);
  }
}
inline unsigned __ballot_sync(unsigned, int p) {
  const host::Word10* w = host_collect("__ballot_sync", p != 0 ? 1 : 0);
  unsigned b = 0;
  for (int i = 0; i < 32; ++i) b |= w[i].v[0] << i;
  return b;
}
inline int __any_sync(unsigned m, int p) { return __ballot_sync(m, p) != 0; }
inline int __all_sync(unsigned m, int p) { return __ballot_sync(m, p) == m; }
inline unsigned __match_any_sync(unsigned, int x) {
  host::matches += host_lane() == 0;
  const host::Word10* w = host_collect("__match_any_sync", x);
  unsigned b = 0;
  for (int i = 0; i < 32; ++i) b |= (w[i].v[0] == (uint32_t)x ? 1u : 0u) << i;
  return b;
}
inline int __reduce_add_sync(unsigned, int x) {
  const host::Word10* w = host_collect("__reduce_add_sync", x);
  int s = 0;
  for (int i = 0; i < 32; ++i) s += (int)w[i].v[0];
  return s;
}
inline int __popc(unsigned x) { return __builtin_popcount(x); }
inline int __ffs(unsigned x) { return __builtin_ffs((int)x); }
inline int __clz(unsigned x) { return x ? __builtin_clz(x) : 32; }
inline float __uint_as_float(uint32_t u) { return host_from<float>(u); }
inline float __int_as_float(int u) { return host_from<float>((uint32_t)u); }
inline uint32_t __float_as_uint(float f) { return host_bits(f); }
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline int atomicAdd(int* p, int x) { const int o = *p; *p += x; return o; }
inline uint32_t atomicOr(uint32_t* p, uint32_t x) { const uint32_t o = *p; *p |= x; return o; }

struct __nv_bfloat16 { uint16_t b; };
inline __nv_bfloat16 __float2bfloat16_rn(float f) {
  uint32_t u = host_bits(f);
  if ((u & 0x7fffffffu) > 0x7f800000u) return {0x7fff};
  u += 0x7fffu + ((u >> 16) & 1u);
  return {(uint16_t)(u >> 16)};
}
inline float __bfloat162float(__nv_bfloat16 x) { return __uint_as_float((uint32_t)x.b << 16); }

// mma.m16n8k16, bf16 operands.  Every product and the accumulator are off by up to 2^-22 of the largest of
// them in the tensor core; here all errors go upwards, against a filter that keeps negative results.
inline void host_mma(float* d, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1,
                     const float* c) {
  const int lane = host_lane(), g = lane >> 2, q = lane & 3;
  host::mmas += lane == 0;
  const float c0[4] = {c[0], c[1], c[2], c[3]};
  const host::Word10* w = host::all_lanes("mma", {{a0, a1, a2, a3, b0, b1}});
  auto half = [](uint32_t x, int h) { return __uint_as_float(h ? x & 0xffff0000u : x << 16); };
  for (int e = 0; e < 4; ++e) {
    const int row = g + 8 * (e >> 1), col = 2 * q + (e & 1);
    double s = c0[e], top = std::fabs((double)c0[e]);
    for (int k = 0; k < 16; ++k) {
      const int t = (k % 8) / 2, h = k & 1;
      const double p = (double)half(w[(row % 8) * 4 + t].v[2 * (k / 8) + row / 8], h) * half(w[col * 4 + t].v[4 + k / 8], h);
      s += p;
      top = std::max(top, std::fabs(p));
    }
    d[e] = (float)(s + 17 * std::ldexp(top, -22));
  }
}

namespace gnn {
enum : uint32_t { DEV_ERR_INDEX_RANGE = 1u, DEV_ERR_TIMEOUT = 2u, DEV_ERR_CAPACITY = 4u };
inline void pdl_wait() {}
inline void pdl_trigger_small() {}
inline uint32_t pack_bf16x2(float a, float b) {
  return (uint32_t)__float2bfloat16_rn(a).b | (uint32_t)__float2bfloat16_rn(b).b << 16;
}
}  // namespace gnn
