// Stream-ordered device memory of one call. Host code.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>
#include <cstdint>
#include <cstdio>
#include <vector>

#include "stc.h"

namespace stc {

stc_status report_error(stc_status s, const char* msg);

// A context's memory pool and what it holds.
struct DevicePool {
  size_t budget = 0;  // 0 = no cap
  cudaMemPool_t pool = nullptr;
  std::atomic<size_t> held{0};
};

// Scratch from the context's pool. Everything still held when the arena dies is returned to the pool
// in stream order; `keep` hands a block to a result instead. In a context without a budget, small
// requests share slabs of kSlab bytes: a call makes some thirty of them, at about a microsecond of host
// time each to take and to return. (A budget counts every request for itself.) A slab lives as long as
// the arena: what `keep` and `release` take are blocks, and a piece of a slab is none, although the
// first piece has the slab's address.
struct Arena {
  static constexpr size_t kSlab = 1 << 20, kSlabMost = 1 << 16;
  DevicePool* ctx;
  cudaStream_t s;
  struct Block { void* p; size_t bytes; bool slab; };
  std::vector<Block> blocks;
  char* slab = nullptr;
  size_t slab_left = 0;
  Arena(DevicePool* c, cudaStream_t st) : ctx(c), s(st) {}
  // Whether a request is a piece of a slab, and the bytes that it takes there.
  static size_t piece(size_t bytes) { return (bytes + 255) & ~(size_t)255; }
  static bool shares_slab(const DevicePool* c, size_t bytes) {
    return bytes != 0 && piece(bytes) <= kSlabMost && !c->budget;
  }
  Arena(const Arena&) = delete;
  Arena& operator=(const Arena&) = delete;
  ~Arena() {
    for (auto& b : blocks) {
      cudaFreeAsync(b.p, s);
      ctx->held -= b.bytes;
    }
  }
  template <typename T>
  stc_status alloc(T** out, size_t count) {
    if (!shares_slab(ctx, count * sizeof(T))) return alloc_own(out, count);
    const size_t bytes = piece(count * sizeof(T));
    if (bytes > slab_left) {
      char* p = nullptr;
      if (alloc_own(&p, kSlab) != STC_OK) return alloc_own(out, count);
      blocks.back().slab = true;
      slab = p;
      slab_left = kSlab;
    }
    *out = reinterpret_cast<T*>(slab);
    slab += bytes;
    slab_left -= bytes;
    return STC_OK;
  }
  // A block of its own, which `keep` and `release` can find.
  template <typename T>
  stc_status alloc_own(T** out, size_t count) {
    *out = nullptr;
    const size_t bytes = count * sizeof(T);
    if (bytes == 0) return STC_OK;
    const size_t after = ctx->held.fetch_add(bytes) + bytes;
    char msg[160];
    if (ctx->budget && after > ctx->budget) {
      ctx->held -= bytes;
      snprintf(msg, sizeof(msg), "request of %zu bytes exceeds the context budget (%zu of %zu held)", bytes,
               after - bytes, ctx->budget);
      return report_error(STC_ERR_OUT_OF_MEMORY, msg);
    }
    void* p = nullptr;
    const cudaError_t e = cudaMallocFromPoolAsync(&p, bytes, ctx->pool, s);
    if (e != cudaSuccess) {
      ctx->held -= bytes;
      cudaGetLastError();
      snprintf(msg, sizeof(msg), "device allocation of %zu bytes failed: %s", bytes, cudaGetErrorString(e));
      return report_error(STC_ERR_OUT_OF_MEMORY, msg);
    }
    blocks.push_back({p, bytes, false});
    *out = static_cast<T*>(p);
    return STC_OK;
  }
  // Gives one block back, in stream order. A piece of a slab stays until the arena dies.
  void release(void* p) {
    const size_t b = keep(p);
    if (!b) return;
    cudaFreeAsync(p, s);
    ctx->held -= b;
  }
  // Takes one block out of the arena, to be given back by its new owner. 0: p is no block.
  size_t keep(void* p) {
    for (size_t i = 0; i < blocks.size(); i++)
      if (blocks[i].p == p && !blocks[i].slab) {
        const size_t b = blocks[i].bytes;
        blocks.erase(blocks.begin() + i);
        return b;
      }
    return 0;
  }
};

// The bytes that an arena holds after the same requests, none given back: what a call will hold at its
// peak, counted without making it.
struct ArenaBytes {
  const DevicePool* ctx;
  uint64_t held = 0;
  size_t slab_left = 0;
  explicit ArenaBytes(const DevicePool* c) : ctx(c) {}
  void alloc(uint64_t bytes) {
    if (!Arena::shares_slab(ctx, bytes)) {
      held += bytes;
      return;
    }
    const size_t b = Arena::piece(bytes);
    if (b > slab_left) {
      held += Arena::kSlab;
      slab_left = Arena::kSlab;
    }
    slab_left -= b;
  }
  void alloc_own(uint64_t bytes) { held += bytes; }
};

}  // namespace stc
