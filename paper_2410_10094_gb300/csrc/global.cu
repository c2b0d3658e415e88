// Contraction and accumulation into one device-wide open-addressing table (Section 2.4.2
// contraction; Section 4.3 probing table sized from the exact product count), followed
// by the writeback of occupied slots as COO output (Section 2.5).
//
// This is the "leave X ungrouped" form noted at the end of Section 4.4: every product
// goes to one global table keyed on the full output key. It is chosen when the output
// key space is small enough for the whole table to stay in L2.
#include "launch.h"

namespace stc {

namespace {

constexpr int kExThreads = 256;
constexpr int kExTile = 2048;  // products per merge-path tile
constexpr int kCpThreads = 256;

// Linear probing (Section 2.3.1) with a compare-and-swap claim of empty slots. A slot's key
// only ever changes from empty to its final key, so a stale read can only show "empty"
// and is then settled by the CAS. The probe sequence is bounded by the table size.
__device__ __forceinline__ void table_add(u64* __restrict__ keys, double* __restrict__ vals, u64 mask, u64 key,
                                          double v, uint32_t* status) {
  u64 slot = mix64(key) & mask;
  for (u64 probe = 0; probe <= mask; probe++) {
    u64 cur = __ldcg(keys + slot);
    if (cur == kEmpty64) {
      const u64 prev = atomicCAS(keys + slot, kEmpty64, key);
      cur = (prev == kEmpty64) ? key : prev;
    }
    if (cur == key) {
      atomicAdd(vals + slot, v);
      return;
    }
    slot = (slot + 1) & mask;
  }
  atomicOr(status, kStatTableFull);
}

// Cooperative probing: a tile of G consecutive lanes inserts its lanes' keys one at a time.
// The table is read as buckets of G consecutive slots (G·8 contiguous bytes of the key array,
// one 32-byte sector for G = 4); every lane of the tile reads one slot of the bucket and two
// ballots tell the whole tile whether the key is there and where the first free slot is. A
// key is placed in the first free slot of the first bucket of its probe sequence that has
// one, so a key is found in the bucket where it would be placed: the invariant of linear
// probing (Section 2.3.1) over buckets instead of slots. A lost claim reads the bucket again.
// Every lane of the warp calls this (`has` false for lanes without a product); `done` and the
// ballots' masks are uniform over a tile, so the tile's lanes stay converged where they
// exchange values.
template <int G>
__device__ __forceinline__ void table_add_coop(u64* __restrict__ keys, double* __restrict__ vals, u64 mask, bool has,
                                               u64 key, double v, uint32_t* status) {
  constexpr unsigned kFull = 0xffffffffu;
  const unsigned lane = lane_id();
  const unsigned base = lane & ~(unsigned)(G - 1);
  const unsigned tmask = (G == 32) ? kFull : (((1u << G) - 1u) << base);
  const unsigned r = lane - base;
  const u64 bmask = mask / G;  // buckets - 1 (the capacity is a power of two >= G)
  bool todo = has;
  while (__any_sync(kFull, todo)) {
    const unsigned pend = __ballot_sync(kFull, todo) & tmask;
    const int src = pend ? __ffs(pend) - 1 : (int)lane;
    const u64 k = __shfl_sync(kFull, key, src);
    const double x = __shfl_sync(kFull, v, src);
    if ((int)lane == src) todo = false;
    bool done = pend == 0;
    u64 b = (mix64(k) & mask) / G;
    u64 steps = 0;
    while (__any_sync(kFull, !done)) {
      const u64 cur = done ? kEmpty64 : __ldcg(keys + b * G + r);
      const unsigned hit = __ballot_sync(kFull, !done && cur == k) & tmask;
      const unsigned emp = __ballot_sync(kFull, !done && cur == kEmpty64) & tmask;
      if (done) continue;
      if (hit) {
        if ((int)lane == __ffs(hit) - 1) atomicAdd(vals + b * G + r, x);
        done = true;
      } else if (emp) {
        const int e = __ffs(emp) - 1;
        u64 prev = 0;
        if ((int)lane == e) prev = atomicCAS(keys + b * G + r, kEmpty64, k);
        prev = __shfl_sync(tmask, prev, e);
        if (prev == kEmpty64 || prev == k) {
          if ((int)lane == e) atomicAdd(vals + b * G + r, x);
          done = true;
        }
      } else {
        b = (b + 1) & bmask;
        if (++steps > bmask) {
          if (lane == base) atomicOr(status, kStatTableFull);
          done = true;
        }
      }
    }
  }
}

// The largest a in [0, n) with pre[a] <= p, given pre[0] <= p, by all lanes of a warp: 33 ways per
// round of loads.
__device__ __forceinline__ int64_t warp_upper(const u64* __restrict__ pre, int64_t n, u64 p) {
  int64_t a = 0, b = n;  // pre[a] <= p < pre[b]
  while (b - a > 1) {
    const int64_t w = (b - a + 32) / 33;
    const int64_t at = a + w * ((int64_t)lane_id() + 1);
    const int64_t k = __popc(__ballot_sync(0xffffffffu, at < b && pre[at] <= p));
    a += w * k;
    if (a + w < b) b = a + w;
  }
  return a;
}

// The owners of 32 consecutive products g0 + lane of a warp: the largest a in [0, n) with
// pre[a] <= g0 + lane, where pre (shared memory, pre[0] <= g0) increases by at least one per entry.
// The first owner by a search of all lanes; the others from where the entries after it begin.
__device__ __forceinline__ int warp_owners(const u64* pre, int n, u64 g0) {
  const int lane = (int)lane_id();
  int a = 0, b = n;  // pre[a] <= g0 < pre[b]
  while (b - a > 1) {
    const int w = (b - a + 32) / 33;
    const int at = a + w * (lane + 1);
    a += w * __popc(__ballot_sync(0xffffffffu, at < b && pre[at] <= g0));
    if (a + w < b) b = a + w;
  }
  const u64 d = a + 1 + lane < n ? pre[a + 1 + lane] - g0 : 32;
  const uint32_t begins = __reduce_or_sync(0xffffffffu, d < 32 ? 1u << d : 0u);
  return a + __popc(begins & (0xffffffffu >> (31 - lane)));
}

// Each CTA takes tiles of kExTile consecutive products. Products are numbered by the
// survivors' exclusive prefix `wpre`: survivor s owns products [wpre[s], wpre[s+1]), its
// r-th product pairs it with slot ystart[s] + r of its Y run. Within a tile, thread t
// handles products t, t+256, ...; consecutive threads read consecutive Y slots.
// G = 1: each lane probes on its own (table_add); G > 1: tiles of G lanes probe buckets together
// (table_add_coop). The loop over a tile's products is uniform over each warp, so all lanes reach the
// cooperative probe.
template <int G>
__global__ void __launch_bounds__(kExThreads) expand_global_kernel(
    const u64* __restrict__ wpre, int64_t ns, u64 P, const u64* __restrict__ sfk, const uint32_t* __restrict__ systart,
    const double* __restrict__ sv, const u64* __restrict__ yfk, const double* __restrict__ yv, u64 FY,
    GlobalTable t, uint32_t* status) {
  __shared__ u64 s_pre[kExTile + 1];
  __shared__ int64_t s_lo, s_hi;
  const unsigned warp = threadIdx.x >> 5;
  const u64 ntiles = (P + kExTile - 1) / kExTile;
  for (u64 tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const u64 p0 = tile * kExTile;
    const u64 p1 = (p0 + kExTile < P) ? p0 + kExTile : P;
    if (warp < 2) {
      const int64_t at = warp_upper(wpre, ns, warp ? p1 - 1 : p0);
      if (lane_id() == 0) (warp ? s_hi : s_lo) = at;
    }
    __syncthreads();
    const int64_t lo = s_lo;
    const int n = (int)(s_hi - lo) + 1;
    for (int k = threadIdx.x; k <= n; k += kExThreads) s_pre[k] = wpre[lo + k];
    __syncthreads();
    for (u64 g0 = p0 + (threadIdx.x & ~31u); g0 < p1; g0 += kExThreads) {
      const u64 g = g0 + lane_id();
      const bool has = g < p1;
      u64 key = 0;
      double prod = 0.0;
      if (has) {
        int a = 0, b = n - 1;
        while (a < b) {
          const int mid = (a + b + 1) >> 1;
          if (s_pre[mid] <= g) a = mid; else b = mid - 1;
        }
        const int64_t s = lo + a;
        const u64 j = (u64)__ldg(systart + s) + (g - s_pre[a]);
        key = __ldg(sfk + s) * FY + __ldg(yfk + j);
        prod = __dmul_rn(__ldg(sv + s), __ldg(yv + j));
      }
      if (G == 1) {
        if (has) table_add(t.keys, t.vals, t.mask, key, prod, status);
      } else {
        table_add_coop<G>(t.keys, t.vals, t.mask, has, key, prod, status);
      }
    }
    __syncthreads();
  }
}

// ---- the expansion without a host read and without a prefix over all survivors: the survey has
// summed the products per block of kSurvivorBlock survivors; one CTA scans those sums, and a tile's
// CTA scans the run lengths of the one to three blocks that its products lie in.
constexpr int kBpThreads = 1024;
__global__ void __launch_bounds__(kBpThreads) block_prefix_kernel(const u64* __restrict__ bsum, u64* __restrict__ bpre,
                                                                  const unsigned* __restrict__ dns) {
  __shared__ u64 s_warp[32];
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  const unsigned nb = (*dns + kSurvivorBlock - 1) / kSurvivorBlock;
  u64 run = 0;
  for (unsigned b0 = 0; b0 < nb; b0 += kBpThreads) {
    const unsigned i = b0 + threadIdx.x;
    const u64 v = i < nb ? bsum[i] : 0;
    u64 x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u64 y = __shfl_up_sync(0xffffffffu, x, o);
      if ((int)lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    u64 t = s_warp[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u64 y = __shfl_up_sync(0xffffffffu, t, o);
      if ((int)lane >= o) t += y;
    }
    const u64 total = __shfl_sync(0xffffffffu, t, 31);
    const u64 before = warp ? __shfl_sync(0xffffffffu, t, warp - 1) : 0;
    if (i < nb) bpre[i] = run + before + x - v;
    run += total;
    __syncthreads();
  }
  if (threadIdx.x == 0) bpre[nb] = run;
}

// An array of a whole output space of up to 2^18 keys, in place of a table. Key k lies at k * kSpread
// mod the array's length, a power of two, so that the keys of one output row, of which a few may get
// most of the products, lie on lines far apart: additions to one 128-byte line take their turns. 4e7
// products on one row of 130 keys of 2,000 x 130: 1.14 ms for the contraction, 9.9 with the rows in
// order, 1.26 in a table; 4e7 uniform products on 512 x 512: 0.60, 0.51 and 0.84 (all with tiles of 1,024
// products; with larger ones, kBxTileMost, 1.05 and 1.21 by array and table, and 0.38 and 0.57).
constexpr uint32_t kSpread = 0x9e3779b1u;  // odd; 2^32 over the golden ratio
constexpr uint32_t inverse_of(uint32_t odd) {
  uint32_t x = odd;  // the right inverse mod 8; every step doubles the bits that are right
  for (int i = 0; i < 4; i++) x *= 2u - odd * x;
  return x;
}
constexpr uint32_t kUnspread = inverse_of(kSpread);
static_assert(kSpread * kUnspread == 1u, "the inverse mod 2^32, and so mod every smaller power of two");
// A cell that no product has met holds -0.0, to which any sum adds up as itself; products of -0.0 are
// added as +0.0, after which no sum is -0.0.
constexpr long long kNoSum = (long long)0x8000000000000000ull;

__global__ void __launch_bounds__(kExThreads) clear_space_kernel(double* __restrict__ vals, u64 n) {
  for (u64 i = (u64)blockIdx.x * kExThreads + threadIdx.x; i < n; i += (u64)gridDim.x * kExThreads) vals[i] = -0.0;
}

// Products per tile, at least, and at most: a tile scans whole blocks of survivors for the products that
// it takes of them, so that many products come in larger tiles, about eight per CTA. 2.04e10 products of
// some thousand per survivor on 262,144 outputs: 213 -> 105 ms by array, 305 -> 173 by table.
constexpr u64 kBxTile = 1024, kBxTileMost = 65536;

// Adds one product to the output space: the hash table, probed by G lanes together (see
// expand_global_kernel), or with G = 0 an array of the whole space.
template <int G>
__global__ void __launch_bounds__(kExThreads) expand_blocks_kernel(const u64* __restrict__ bpre, Survivors sv,
                                                                   const u64* __restrict__ yfk,
                                                                   const double* __restrict__ yv, u64 FY,
                                                                   GlobalTable t, uint32_t* status) {
  constexpr int IT = kSurvivorBlock / kExThreads, NW = kExThreads / 32;
  const int64_t ns = (int64_t)*sv.count;
  if (ns == 0) return;
  const int64_t nb = (ns + kSurvivorBlock - 1) / kSurvivorBlock;
  const u64 P = bpre[nb];
  __shared__ u64 s_pre[kSurvivorBlock];
  __shared__ u64 s_warp[NW];
  __shared__ int64_t s_lo;
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  const u64 share = P / ((u64)gridDim.x * 8) / kBxTile * kBxTile;
  const u64 size = share < kBxTile ? kBxTile : (share < kBxTileMost ? share : kBxTileMost);
  const u64 ntiles = (P + size - 1) / size;
  for (u64 tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const u64 p0 = tile * size;
    const u64 p1 = (p0 + size < P) ? p0 + size : P;
    if (warp == 0) {
      const int64_t at = warp_upper(bpre, nb, p0);
      if (lane == 0) s_lo = at;
    }
    __syncthreads();
    for (int64_t blk = s_lo; blk < nb; blk++) {
      const u64 q0 = bpre[blk], q1 = bpre[blk + 1];
      if (q0 >= p1) break;  // uniform
      // The block's run lengths, IT consecutive ones per thread, scanned.
      const int64_t s0 = blk * kSurvivorBlock;
      u64 w[IT], sum = 0;
#pragma unroll
      for (int i = 0; i < IT; i++) {
        const int64_t s = s0 + threadIdx.x * IT + i;
        w[i] = sum;
        sum += s < ns ? __ldg(sv.w + s) : 0u;
      }
      u64 x = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const u64 y = __shfl_up_sync(0xffffffffu, x, o);
        if ((int)lane >= o) x += y;
      }
      if (lane == 31) s_warp[warp] = x;
      __syncthreads();
      u64 before = q0 + x - sum;
      for (unsigned k = 0; k < warp; k++) before += s_warp[k];
#pragma unroll
      for (int i = 0; i < IT; i++) s_pre[threadIdx.x * IT + i] = before + w[i];
      __syncthreads();
      const int n = (int)(ns - s0 < (int64_t)kSurvivorBlock ? ns - s0 : (int64_t)kSurvivorBlock);
      const u64 a0 = q0 > p0 ? q0 : p0, a1 = q1 < p1 ? q1 : p1;
      int e0 = 0, e1 = n;  // a larger tile looks among the entries that its own products have
      if (size > kBxTile) {
        e0 = __shfl_sync(0xffffffffu, warp_owners(s_pre, n, a0), 0);
        e1 = __shfl_sync(0xffffffffu, warp_owners(s_pre, n, a1 - 1), 0) + 1;
      }
      for (u64 g0 = a0 + warp * 32; g0 < a1; g0 += kExThreads) {
        const int a = e0 + warp_owners(s_pre + e0, e1 - e0, g0);
        const u64 g = g0 + lane;
        const bool has = g < a1;
        u64 key = 0;
        double prod = 0.0;
        if (has) {
          const int64_t s = s0 + a;
          const u64 j = (u64)__ldg(sv.ystart + s) + (g - s_pre[a]);
          key = __ldg(sv.fk + s) * FY + __ldg(yfk + j);
          prod = __dmul_rn(__ldg(sv.v + s), __ldg(yv + j));
        }
        if (G == 0) {
          if (has) atomicAdd(t.vals + (((uint32_t)key * kSpread) & (uint32_t)t.mask), __dadd_rn(prod, 0.0));
        } else if (G == 1) {
          if (has) table_add(t.keys, t.vals, t.mask, key, prod, status);
        } else {
          table_add_coop<G < 2 ? 2 : G>(t.keys, t.vals, t.mask, has, key, prod, status);
        }
      }
      __syncthreads();  // the block's prefix is rewritten
    }
    __syncthreads();  // and s_lo
  }
}

// ---- large output key spaces. A product that claims a new key writes
// its output entry at once; the table holds keys and output positions, and no values, so there is no
// pass over it afterwards. A product whose key is there already goes to a list (the slot and the
// value), and is added to the slot's entry by a kernel of its own, once every position is known.
// Each thread takes kDirectItems products of a tile together: their searches, gathers and claims
// overlap. One atomic per tile reserves the positions of its new keys, and one the repeats' places.
constexpr int kDirectItems = 4;
constexpr int kDirectTile = kDirectItems * kExThreads;
__global__ void __launch_bounds__(kExThreads, 4) expand_direct_kernel(
    const u64* __restrict__ wpre, int64_t ns, u64 P, const u64* __restrict__ sfk, const uint32_t* __restrict__ systart,
    const double* __restrict__ sv, const u64* __restrict__ yfk, const double* __restrict__ yv, u64 FY, DirectTable t,
    const __grid_constant__ OutPlan op, int32_t* __restrict__ coords, double* __restrict__ vals, u64 out_cap,
    u64* __restrict__ nz, uint32_t* status) {
  constexpr int NW = kExThreads / 32, D = kDirectItems;
  __shared__ u64 s_pre[kDirectTile + 1];
  __shared__ int64_t s_lo, s_hi;
  __shared__ uint32_t s_warp[NW];
  __shared__ u64 s_base, s_rbase;
  __shared__ bool s_look;
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  const uint64_t pol = policy_evict_first();
  const u64 ntiles = (P + kDirectTile - 1) / kDirectTile;
  bool look = true;
  for (u64 tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const u64 p0 = tile * kDirectTile;
    const u64 p1 = (p0 + kDirectTile < P) ? p0 + kDirectTile : P;
    if (warp < 2) {
      const int64_t at = warp_upper(wpre, ns, warp ? p1 - 1 : p0);
      if (lane == 0) (warp ? s_hi : s_lo) = at;
    }
    __syncthreads();
    const int64_t lo = s_lo;
    const int n = (int)(s_hi - lo) + 1;
    for (int k = threadIdx.x; k <= n; k += kExThreads) s_pre[k] = wpre[lo + k];
    __syncthreads();
    u64 key[D], j[D];
    double v[D];
    uint32_t slot[D];
    uint32_t state = 0;  // bit u: product u claimed its key; bit 16 + u: its key was there
#pragma unroll
    for (int u = 0; u < D; u++) {
      const u64 g0 = p0 + (u64)u * kExThreads + warp * 32, g = g0 + lane;
      if (g0 < p1) {
        const int a = warp_owners(s_pre, n, g0);
        if (g < p1) {
          const int64_t s = lo + a;
          j[u] = (u64)__ldg(systart + s) + (g - s_pre[a]);
          key[u] = __ldg(sfk + s);
          v[u] = __ldg(sv + s);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < D; u++)
      if (p0 + (u64)u * kExThreads + threadIdx.x < p1) {
        key[u] = key[u] * FY + __ldg(yfk + j[u]);
        v[u] = __dmul_rn(v[u], __ldg(yv + j[u]));
      }
    // The first probes of all of a thread's products are issued together; the few that meet another key
    // go on one by one. The claims that find a key there already take their turns at it, so the slots
    // are looked at first, except after a tile most of whose products were new: 6e7 products of 1.0 per
    // key 5.53 against 5.80 ms with a look first, of 10 per key 4.37 against 3.61.
    u64 cur[D];
#pragma unroll
    for (int u = 0; u < D; u++) {
      slot[u] = 0;
      cur[u] = 0;
      if (p0 + (u64)u * kExThreads + threadIdx.x < p1) {
        slot[u] = (uint32_t)(mix64(key[u]) & t.mask);
        cur[u] = look ? __ldcg(t.keys + slot[u]) : kEmpty64;
      }
    }
#pragma unroll
    for (int u = 0; u < D; u++)
      if (p0 + (u64)u * kExThreads + threadIdx.x < p1 && cur[u] == kEmpty64)
        cur[u] = atomicCAS(t.keys + slot[u], kEmpty64, key[u]);
#pragma unroll
    for (int u = 0; u < D; u++) {
      if (p0 + (u64)u * kExThreads + threadIdx.x >= p1) continue;
      u64 probe = 0;
      while (cur[u] != kEmpty64 && cur[u] != key[u] && probe++ < t.mask) {
        slot[u] = (uint32_t)((slot[u] + 1) & t.mask);
        cur[u] = __ldcg(t.keys + slot[u]);
        if (cur[u] == kEmpty64) cur[u] = atomicCAS(t.keys + slot[u], kEmpty64, key[u]);
      }
      if (cur[u] == kEmpty64)
        state |= 1u << u;
      else if (cur[u] == key[u])
        state |= 0x10000u << u;
      else
        atomicOr(status, kStatTableFull);
    }
    // The tile's new keys: positions in the order of (warp, product of the thread, lane).
    uint32_t mine = 0, rank[D];
#pragma unroll
    for (int u = 0; u < D; u++) {
      const uint32_t m = __ballot_sync(0xffffffffu, (state >> u) & 1u);
      rank[u] = mine + __popc(m & lanemask_lt());
      mine += __popc(m);
    }
    uint32_t reps = 0, rrank[D];
#pragma unroll
    for (int u = 0; u < D; u++) {
      const uint32_t m = __ballot_sync(0xffffffffu, (state >> (16 + u)) & 1u);
      rrank[u] = reps + __popc(m & lanemask_lt());
      reps += __popc(m);
    }
    if (lane == 0) s_warp[warp] = mine | (reps << 16);  // both at most kDirectTile
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t run = 0;
      for (int w = 0; w < NW; w++) {
        const uint32_t c = s_warp[w];
        s_warp[w] = run;
        run += c;
      }
      s_base = run & 0xffffu ? atomicAdd(nz, (u64)(run & 0xffffu)) : 0;
      s_rbase = run >> 16 ? atomicAdd(t.nreps, (u64)(run >> 16)) : 0;
      s_look = run >> 16 > (run & 0xffffu);
    }
    __syncthreads();
    look = s_look;
    const u64 base = s_base + (s_warp[warp] & 0xffffu), rbase = s_rbase + (s_warp[warp] >> 16);
#pragma unroll
    for (int u = 0; u < D; u++) {
      if ((state >> u) & 1u) {
        const u64 pos = base + rank[u];
        t.pos[slot[u]] = (uint32_t)pos;
        if (pos < out_cap)
          store_output(coords, vals, pos, key[u], v[u], op, pol);
        else
          atomicOr(status, kStatOutOverflow);
      }
      if ((state >> (16 + u)) & 1u) {
        t.rep_slot[rbase + rrank[u]] = slot[u];
        t.rep_val[rbase + rrank[u]] = v[u];
      }
    }
    __syncthreads();  // the tile's shared arrays are rewritten by the next
  }
}

// Additions to one 128-byte line of the outputs take their turns, about 1.5 ns each, and the outputs of
// few keys share few lines (in a table their slots lay apart). So where the repeats are at least four
// per key and CTA, each CTA first sums its own in shared memory: 2e7 products on 196 keys 3.52 -> 0.74 ms
// for the contraction, 6e7 on 576 4.53 -> 1.84.
constexpr uint32_t kFewKeys = 1024;
__global__ void __launch_bounds__(kExThreads) add_repeats_kernel(DirectTable t, double* __restrict__ vals, u64 out_cap,
                                                                 const u64* __restrict__ nz) {
  __shared__ double s_sum[kFewKeys];
  const u64 n = *t.nreps, keys = *nz;
  const bool few = keys <= kFewKeys && keys <= out_cap && n >= 4 * keys * gridDim.x;
  if (few) {
    for (uint32_t k = threadIdx.x; k < keys; k += kExThreads) s_sum[k] = 0.0;
    __syncthreads();
  }
  for (u64 i = (u64)blockIdx.x * kExThreads + threadIdx.x; i < n; i += (u64)gridDim.x * kExThreads) {
    const uint32_t pos = t.pos[t.rep_slot[i]];
    if (few)
      atomicAdd(s_sum + pos, t.rep_val[i]);
    else if (pos < out_cap)
      atomicAdd(vals + pos, t.rep_val[i]);
  }
  if (few) {
    __syncthreads();
    for (uint32_t k = threadIdx.x; k < keys; k += kExThreads)
      if (s_sum[k] != 0.0) atomicAdd(vals + k, s_sum[k]);
  }
}

// Each CTA takes 2048 consecutive slots at a time (8 per thread, coalesced), ranks the
// occupied ones with a block scan and reserves their output positions with one atomic.
constexpr int kCpItems = 8;
// In an array of the whole space the occupied cells are those that hold a sum.
__global__ void __launch_bounds__(kCpThreads) compact_global_kernel(GlobalTable t, OutPlan op,
                                                                    int32_t* __restrict__ coords,
                                                                    double* __restrict__ vals, u64 out_cap,
                                                                    u64* __restrict__ nz, uint32_t* status) {
  constexpr int NW = kCpThreads / 32;
  __shared__ uint32_t s_warp[NW + 1];
  __shared__ u64 s_base;
  const int64_t cap = (int64_t)t.mask + 1;
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  for (int64_t base = (int64_t)blockIdx.x * kCpThreads * kCpItems; base < cap;
       base += (int64_t)gridDim.x * kCpThreads * kCpItems) {
    u64 k[kCpItems];
    uint32_t cnt = 0;
#pragma unroll
    for (int it = 0; it < kCpItems; it++) {
      const int64_t i = base + (int64_t)it * kCpThreads + threadIdx.x;
      k[it] = kEmpty64;
      if (i < cap) {
        if (t.keys)
          k[it] = __ldcs(t.keys + i);
        else if (__double_as_longlong(t.vals[i]) != kNoSum)
          k[it] = ((uint32_t)i * kUnspread) & (uint32_t)t.mask;
      }
      cnt += k[it] != kEmpty64;
    }
    uint32_t x = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if ((int)lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t run = 0;
      for (int w = 0; w < NW; w++) {
        const uint32_t v = s_warp[w];
        s_warp[w] = run;
        run += v;
      }
      s_base = run ? atomicAdd(nz, (u64)run) : 0;
    }
    __syncthreads();
    u64 pos = s_base + s_warp[warp] + x - cnt;
#pragma unroll
    for (int it = 0; it < kCpItems; it++) {
      if (k[it] == kEmpty64) continue;
      if (pos < out_cap) {
        const int64_t i = base + (int64_t)it * kCpThreads + threadIdx.x;
        store_coords(k[it], op, coords + pos * (u64)op.order);
        vals[pos] = __ldcs(t.vals + i);
      } else {
        atomicOr(status, kStatOutOverflow);
      }
      pos++;
    }
    __syncthreads();  // s_warp and s_base are rewritten by the next round
  }
}

}  // namespace

namespace {
using ExpandKernel = void (*)(const u64*, int64_t, u64, const u64*, const uint32_t*, const double*, const u64*,
                              const double*, u64, GlobalTable, uint32_t*);
ExpandKernel expand_for(int probe) {
  switch (probe) {
    case 4: return expand_global_kernel<4>;
    case 8: return expand_global_kernel<8>;
    default: return expand_global_kernel<1>;
  }
}
}  // namespace

cudaError_t launch_expand_global(const u64* wpre, int64_t ns, u64 P, Survivors sv, const u64* yfk, const double* yv,
                                 u64 FY, GlobalTable t, uint32_t* status, int sms, cudaStream_t s, int probe) {
  if (P == 0 || ns <= 0) return cudaSuccess;
  const u64 ntiles = (P + kExTile - 1) / kExTile;
  const u64 cap = (u64)sms * 8;
  const unsigned g = (unsigned)(ntiles < cap ? ntiles : cap);
  expand_for(probe)<<<g, kExThreads, 0, s>>>(wpre, ns, P, sv.fk, sv.ystart, sv.v, yfk, yv, FY, t, status);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_expand_blocks(Survivors sv, u64* bpre, const u64* yfk, const double* yv, u64 FY, GlobalTable t,
                                 uint32_t* status, int sms, cudaStream_t s, int probe) {
  block_prefix_kernel<<<1, kBpThreads, 0, s>>>(sv.bsum, bpre, sv.count);
  auto kern = expand_blocks_kernel<0>;
  if (t.keys)
    kern = probe == 4 ? expand_blocks_kernel<4> : (probe == 8 ? expand_blocks_kernel<8> : expand_blocks_kernel<1>);
  kern<<<(unsigned)sms * 8, kExThreads, 0, s>>>(bpre, sv, yfk, yv, FY, t, status);
  note_launch(2);
  return cudaGetLastError();
}

cudaError_t launch_expand_direct(const u64* wpre, int64_t ns, u64 P, Survivors sv, const u64* yfk, const double* yv,
                                 u64 FY, const DirectTable& t, const OutPlan& op, int32_t* coords, double* vals,
                                 u64 out_cap, u64* nz, uint32_t* status, int sms, cudaStream_t s) {
  if (P == 0 || ns <= 0) return cudaSuccess;
  const u64 ntiles = (P + kDirectTile - 1) / kDirectTile, cap = (u64)sms * 8;
  const unsigned g = (unsigned)(ntiles < cap ? ntiles : cap);
  expand_direct_kernel<<<g, kExThreads, 0, s>>>(wpre, ns, P, sv.fk, sv.ystart, sv.v, yfk, yv, FY, t, op, coords, vals,
                                                out_cap, nz, status);
  add_repeats_kernel<<<g, kExThreads, 0, s>>>(t, vals, out_cap, nz);
  note_launch(2);
  return cudaGetLastError();
}

cudaError_t launch_clear_space(GlobalTable t, int sms, cudaStream_t s) {
  const u64 cap = t.mask + 1, want = (cap + kExThreads * 4 - 1) / (kExThreads * 4), lim = (u64)sms * 8;
  clear_space_kernel<<<(unsigned)(want < lim ? want : lim), kExThreads, 0, s>>>(t.vals, cap);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_compact_global(GlobalTable t, const OutPlan& op, int32_t* coords, double* vals, u64 out_cap, u64* nz, uint32_t* status, int sms, cudaStream_t s) {
  const u64 cap = t.mask + 1;
  const u64 want = (cap + kCpThreads * kCpItems - 1) / (kCpThreads * kCpItems);
  const u64 lim = (u64)sms * 8;
  compact_global_kernel<<<(unsigned)(want < lim ? want : lim), kCpThreads, 0, s>>>(t, op, coords, vals, out_cap, nz,
                                                                                  status);
  note_launch();
  return cudaGetLastError();
}

}  // namespace stc
