"""A call's device memory (csrc/arena.h) on the host, over a pool that counts: what is given back early,
what a result keeps, that a slab outlives every piece of it, and what a sequence of requests will hold."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUNTIME = r"""
#pragma once
#include <stdlib.h>
typedef int cudaError_t;
typedef void* cudaStream_t;
typedef void* cudaMemPool_t;
enum { cudaSuccess = 0, cudaErrorMemoryAllocation = 2 };
inline int taken = 0, given = 0;
inline size_t limit = ~(size_t)0;
inline cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) {
  if (n > limit) return cudaErrorMemoryAllocation;
  taken++;
  *p = malloc(n);
  return cudaSuccess;
}
inline cudaError_t cudaFreeAsync(void* p, cudaStream_t) { given++; free(p); return cudaSuccess; }
inline cudaError_t cudaGetLastError() { return cudaSuccess; }
inline const char* cudaGetErrorString(cudaError_t) { return "out of memory"; }
"""

MAIN = r"""
#include "arena.h"
#include <string.h>
#define CHECK(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
static int errors = 0;
stc_status stc::report_error(stc_status s, const char*) { errors++; return s; }
int main() {
  using namespace stc;
  DevicePool pool;
  char *first, *second, *third, *big, *own;
  {
    Arena ar(&pool, nullptr);
    CHECK(ar.alloc(&first, 1000) == STC_OK && ar.alloc(&second, 1000) == STC_OK);
    CHECK(taken == 1 && second == first + 1024);
    // The first piece has its slab's address: giving it back must leave the slab alone.
    ar.release(first);
    CHECK(given == 0 && ar.keep(first) == 0 && ar.keep(second) == 0);
    CHECK(ar.alloc(&third, 1000) == STC_OK && taken == 1 && third == second + 1024);
    memset(first, 1, 1000), memset(second, 2, 1000), memset(third, 3, 1000);
    CHECK(ar.alloc(&big, 1 << 20) == STC_OK && ar.alloc_own(&own, 300) == STC_OK && taken == 3);
    ar.release(big);
    CHECK(given == 1 && pool.held == Arena::kSlab + 300);
    CHECK(ar.keep(own) == 300 && ar.keep(own) == 0);
  }
  CHECK(given == 2 && pool.held == 300);  // the kept block is its new owner's
  cudaFreeAsync(own, nullptr);
  pool.held -= 300;
  // No memory for a slab: a block of the request's own size, and that can be given back.
  limit = 5000;
  {
    Arena ar(&pool, nullptr);
    CHECK(ar.alloc(&first, 4000) == STC_OK && errors == 1 && pool.held == 4000);
    ar.release(first);
    CHECK(pool.held == 0 && ar.alloc(&first, 6000) == STC_ERR_OUT_OF_MEMORY && first == nullptr);
  }
  // Under a budget every request counts for itself.
  limit = ~(size_t)0;
  pool.budget = 5000;
  {
    Arena ar(&pool, nullptr);
    CHECK(ar.alloc(&first, 4000) == STC_OK && pool.held == 4000 && ar.alloc(&second, 1001) == STC_ERR_OUT_OF_MEMORY);
    ar.release(first);
    CHECK(pool.held == 0 && ar.alloc(&second, 5000) == STC_OK);
  }
  CHECK(pool.held == 0 && taken == given);
  // The bytes counted for a sequence of requests are those that an arena holds after it.
  for (int budget = 0; budget < 2; budget++) {
    pool.budget = budget ? (size_t)1 << 40 : 0;
    Arena ar(&pool, nullptr);
    ArenaBytes count(&pool);
    unsigned x = 12345;
    for (int i = 0; i < 400; i++) {
      x = x * 1664525u + 1013904223u;
      const size_t n = i % 7 == 0 ? x >> 12 : x >> 17;  // up to 2^20 and 2^15
      if (i % 29 == 0) {
        CHECK(ar.alloc_own(&own, n) == STC_OK);
        count.alloc_own(n);
      } else {
        CHECK(ar.alloc(&own, n) == STC_OK);
        count.alloc(n);
      }
      CHECK(count.held == pool.held);
    }
  }
  return 0;
}
"""


def test_arena(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = tmp_path / "arena"
    subprocess.run(["g++", "-std=c++20", "-I", str(tmp_path), "-I", os.path.join(ROOT, "paper_2410_10094_gb300", "csrc"),
                    "-I", os.path.join(ROOT, "include"), str(tmp_path / "main.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
