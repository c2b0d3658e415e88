// Runs CUDA kernels on the host, one CTA after another, each thread a fiber that runs until its next
// barrier, shuffle, ballot or __syncwarp. Which warp runs next is the caller's to choose, so that an
// order in which a missing barrier shows can be had every time. Only what the kernels under test use.
#pragma once

#include <stdint.h>
#include <string.h>
#include <ucontext.h>

#include <memory>
#include <vector>

struct int2 { int32_t x, y; };
struct int4 { int32_t x, y, z, w; };
struct uint2 { uint32_t x, y; };
struct uint4 { uint32_t x, y, z, w; };
inline int4 make_int4(int32_t x, int32_t y, int32_t z, int32_t w) { return {x, y, z, w}; }
inline uint2 make_uint2(uint32_t x, uint32_t y) { return {x, y}; }
inline uint4 make_uint4(uint32_t x, uint32_t y, uint32_t z, uint32_t w) { return {x, y, z, w}; }

namespace emu {

struct Dim { unsigned x; };
struct Warp { uint32_t arrived = 0; uint64_t in[32], out[32]; };
struct Fiber {
  ucontext_t ctx;
  std::unique_ptr<char[]> stack;
  unsigned tid;
  int wait;  // 0 ready, 1 for its warp, 2 for the block, 3 finished
};

inline constexpr size_t kStack = 64 << 10;
inline std::vector<Fiber> fibers;
inline std::vector<Warp> warps;
inline ucontext_t home;
inline Fiber* self = nullptr;
inline unsigned at_barrier = 0;
inline Dim block_idx{0}, grid_dim{0};
alignas(1024) inline unsigned char shared_mem[256 << 10];
inline void (*entry)(void*) = nullptr;
inline void* entry_arg = nullptr;
// Whose turn it is: 0 the lowest warp that can run, 1 the highest, others a random one (the seed).
inline uint32_t order = 0, rnd = 1;
inline bool stuck = false;

inline void yield(int wait) {
  self->wait = wait;
  swapcontext(&self->ctx, &home);
}

inline void start() {
  entry(entry_arg);
  yield(3);
}

// All lanes of a warp hand in a value; every lane may then read the others'.
inline const uint64_t* collect(uint64_t v) {
  Warp& w = warps[self->tid / 32];
  const unsigned lane = self->tid & 31;
  w.in[lane] = v;
  w.arrived |= 1u << lane;
  if (w.arrived == 0xffffffffu) {
    w.arrived = 0;
    memcpy(w.out, w.in, sizeof(w.in));
    for (unsigned l = 0; l < 32; l++) fibers[self->tid / 32 * 32 + l].wait = 0;
    yield(0);
  } else {
    yield(1);
  }
  return w.out;
}

template <typename T>
uint64_t bits_of(T v) {
  uint64_t b = 0;
  memcpy(&b, &v, sizeof(T));
  return b;
}
template <typename T>
T from_bits(uint64_t b) {
  T v;
  memcpy(&v, &b, sizeof(T));
  return v;
}

inline void barrier() {
  if (++at_barrier == fibers.size()) {
    at_barrier = 0;
    for (Fiber& f : fibers) f.wait = 0;
    yield(0);
  } else {
    yield(2);
  }
}

inline Fiber* next() {
  const size_t nw = warps.size();
  const size_t first = order > 1 ? (rnd = rnd * 1664525u + 1013904223u, (rnd >> 8) % nw) : 0;
  for (size_t k = 0; k < nw; k++) {
    const size_t w = order == 1 ? nw - 1 - k : (first + k) % nw;
    for (unsigned l = 0; l < 32; l++)
      if (fibers[w * 32 + l].wait == 0) return &fibers[w * 32 + l];
  }
  return nullptr;
}

template <typename F>
void launch(unsigned grid, unsigned block, F body) {
  grid_dim.x = grid;
  entry = [](void* p) { (*static_cast<F*>(p))(); };
  entry_arg = &body;
  rnd = order;
  for (unsigned b = 0; b < grid && !stuck; b++) {
    block_idx.x = b;
    memset(shared_mem, 0xa5, sizeof(shared_mem));
    at_barrier = 0;
    warps.assign(block / 32, Warp{});
    fibers.resize(block);
    for (unsigned t = 0; t < block; t++) {
      Fiber& f = fibers[t];
      if (!f.stack) f.stack.reset(new char[kStack]);
      f.tid = t;
      f.wait = 0;
      getcontext(&f.ctx);
      f.ctx.uc_stack.ss_sp = f.stack.get();
      f.ctx.uc_stack.ss_size = kStack;
      f.ctx.uc_link = nullptr;
      makecontext(&f.ctx, start, 0);
    }
    while (Fiber* f = next()) {
      self = f;
      swapcontext(&home, &f->ctx);
    }
    for (const Fiber& f : fibers) stuck = stuck || f.wait != 3;  // threads left waiting for others
  }
}

}  // namespace emu

#define threadIdx (emu::Dim{emu::self->tid})
#define blockIdx emu::block_idx
#define gridDim emu::grid_dim
#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
#define __restrict__
#define __grid_constant__
#define __launch_bounds__(...)
#define __align__(n) alignas(n)
#define __shared__ static
inline void __syncthreads() { emu::barrier(); }
inline void __syncwarp() { emu::collect(0); }
inline uint32_t __ballot_sync(uint32_t, bool p) {
  const uint64_t* o = emu::collect(p);
  uint32_t m = 0;
  for (int l = 0; l < 32; l++) m |= (uint32_t)o[l] << l;
  return m;
}
template <typename T>
T __shfl_sync(uint32_t, T v, int from) { return emu::from_bits<T>(emu::collect(emu::bits_of(v))[from & 31]); }
template <typename T>
T __shfl_up_sync(uint32_t, T v, int by) {
  const int lane = emu::self->tid & 31;
  return emu::from_bits<T>(emu::collect(emu::bits_of(v))[lane >= by ? lane - by : lane]);
}
template <typename T>
T __shfl_xor_sync(uint32_t, T v, int by) {
  return emu::from_bits<T>(emu::collect(emu::bits_of(v))[(emu::self->tid & 31) ^ by]);
}
inline uint32_t __reduce_add_sync(uint32_t, uint32_t v) {
  const uint64_t* o = emu::collect(v);
  uint32_t s = 0;
  for (int l = 0; l < 32; l++) s += (uint32_t)o[l];
  return s;
}
inline uint32_t __reduce_or_sync(uint32_t, uint32_t v) {
  const uint64_t* o = emu::collect(v);
  uint32_t s = 0;
  for (int l = 0; l < 32; l++) s |= (uint32_t)o[l];
  return s;
}
inline int __popc(uint32_t v) { return __builtin_popcount(v); }
inline int __popcll(uint64_t v) { return __builtin_popcountll(v); }
inline int __ffs(uint32_t v) { return __builtin_ffs((int)v); }
inline uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)((uint64_t)a * b >> 32); }
inline uint64_t __umul64hi(uint64_t a, uint64_t b) { return (uint64_t)((unsigned __int128)a * b >> 64); }
inline double __dmul_rn(double a, double b) { return a * b; }
inline double __dadd_rn(double a, double b) { return a + b; }
template <typename T>
T __ldg(const T* p) { return *p; }
template <typename T>
T __ldcg(const T* p) { return *p; }
template <typename T, typename V>
T atomicAdd(T* p, V v) { const T was = *p; *p = was + (T)v; return was; }
template <typename T, typename V>
T atomicOr(T* p, V v) { const T was = *p; *p = was | (T)v; return was; }
template <typename T, typename V, typename W>
T atomicCAS(T* p, V expect, W v) { const T was = *p; if (was == (T)expect) *p = (T)v; return was; }

typedef int cudaError_t;
typedef void* cudaStream_t;
enum { cudaSuccess = 0, cudaErrorInvalidValue = 1, cudaFuncAttributeMaxDynamicSharedMemorySize = 8 };
inline cudaError_t cudaGetLastError() { return cudaSuccess; }
template <typename K>
cudaError_t cudaFuncSetAttribute(K, int, int) { return cudaSuccess; }
inline cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { memset(p, v, n); return cudaSuccess; }
