// Groups of up to a few thousand products (X entries that share a free key), each output written
// as its first product is formed: the accumulation of a contraction's ordinary groups.
//
// One group, or one segment of 2^16 Y free keys of it, at a time per CTA, four CTAs per SM. The
// group reserves as many output positions as it has products. Pass 1 forms every product once and
// marks its free key in a bitmap: the product that finds its bit clear is its key's first and
// writes the output entry at the next place from the front of the positions; a repeat leaves its
// key and value at the next place from their back and marks the key in a second bitmap. Then the
// repeated keys are ranked, their firsts' places looked up, and every repeat is added to its
// first's entry. The places that the repeats took are what the group leaves over: the CTA's next
// group fills them first. What is left at the end, a few thousand positions per CTA at most, is
// listed as holes and filled from the end of the output (hole_*_kernel).
//
// Products are listed in quarter-slots: up to 8 consecutive Y entries of one X entry's run, four
// to a warp and step, which fills 93% of the lanes at 76 entries per run, where slots of 32 fill
// 82%. A lane without a product reads the entry past Y's last, whose key's bit is always set, so
// that the main loop has no test for it.
//
// What bounds it: without repeats the kernel writes at the rate that a plain kernel storing rows at
// unaligned positions reaches (4.9 TB/s; 6.5 where groups start on 128-byte boundaries): 1.96 ms for
// the 3.65e8 outputs of two 256^4 tensors with 5e6 entries each. The 4.4% repeats cost 0.9 ms more:
// the passes over the first products' keys and the barriers between them, in which a CTA stores
// nothing. Measured on that contraction (accumulation): 2.82 ms, and 0.06 ms for the holes, against
// 3.54 and 0.24 ms with slots of 32, the repeats kept in global memory and every group's holes
// filled; a 4 x 4 x 93 x 36 x 432 tensor of 3e5 entries with itself 2.31 against 3.40 ms.
// A table of 16-bit places per free key in place of the bitmaps and their ranking (128 KB, one CTA
// of 1,024 threads per SM) took 3.4 ms: its phases leave the memory idle between barriers.
#include "launch.h"

namespace stc {

namespace {

constexpr int T = 256, NW = T / 32;
constexpr uint32_t kEntries = T;  // X entries staged at a time
constexpr uint32_t kCap = 8192;   // products of one group segment
constexpr int U = 4;              // slots per warp and step
constexpr uint32_t kStep = NW * U * 4;  // quarter-slots per step
constexpr uint32_t kQuarters = kCap / 8 + kEntries;
constexpr uint32_t kWords = kDenseSeg / 32;
constexpr uint32_t kList = 512;   // repeats kept in shared memory
constexpr uint32_t kHash = 1024;  // table of their keys
constexpr uint32_t kHashEmpty = 0xffffffffu, kNoPlace = 0x8000u;
static_assert(kQuarters % kStep == 0, "the quarter-slot table holds whole steps");
static_assert(kEntries <= 4096 && kCap < 65536, "field widths");

struct StreamSmem {
  uint32_t bits[kWords + 4]; // keys met (and the lanes' without a product, at most key 2^16);
                             // then, at each word, the rank of its first repeated key
  uint32_t rbits[kWords];    // keys met again
  uint2 stab[kQuarters];     // quarter-slots: first Y entry; entries | staged X entry << 4; after
                             // pass 1, rank of a repeated key -> place of its first product
  double rv[kList];          // repeats: values and keys
  uint32_t hash[kHash];      // key of a repeat << 16 | place of its first product
  double sx[kEntries];       // X values
  uint16_t pk[kCap];         // keys of the first products, by place
  uint16_t rk[kList];
  u64 base;                  // positions reserved for the group
  uint32_t warp_tot[NW + 1];
  uint32_t firsts, repeats;  // places given out from the front and from the back
};
static_assert(4 * (sizeof(StreamSmem) + 1024 + 64) <= 228 * 1024, "four CTAs per SM");
static_assert(sizeof(uint2) * kQuarters >= kCap, "the map of ranks fits the quarter-slot table");

// Exclusive block scan of one value per thread; *total receives the sum. Two barriers.
__device__ __forceinline__ uint32_t block_exscan(uint32_t v, uint32_t* total, uint32_t* warp_tot) {
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if ((int)lane >= o) x += y;
  }
  if (lane == 31) warp_tot[warp] = x;
  __syncthreads();
  if (threadIdx.x < 32) {
    const uint32_t t = lane < NW ? warp_tot[lane] : 0u;
    uint32_t inc = t;
#pragma unroll
    for (int o = 1; o < NW; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if ((int)lane >= o) inc += y;
    }
    if (lane < NW) warp_tot[lane] = inc - t;
    if (lane == NW - 1) warp_tot[NW] = inc;
  }
  __syncthreads();
  *total = warp_tot[NW];
  return warp_tot[warp] + x - v;
}

__device__ __forceinline__ uint32_t shared_inc(uint32_t* p) {
  uint32_t at;
  asm volatile("atom.shared.add.u32 %0, [%1], 1;" : "=r"(at) : "r"(smem_addr(p)) : "memory");
  return at;
}

// The slot of a repeat's key in the table.
__device__ __forceinline__ uint32_t hash_find(const uint32_t* hash, uint32_t key) {
  uint32_t h = (key * 0x9e3779b1u) >> 22;
  while (hash[h] >> 16 != key) h = (h + 1) & (kHash - 1);
  return h;
}

// kRows4: order-4 outputs of power-of-two lengths, one 16-byte store per row (kRows22: whose first
// two coordinates are the X part). 3..6: output rows of
// that many coordinates in concatenation order, only the Y part decoded per output (the X part is
// the group's). kRowsAny: every other plan.
constexpr int kRows4 = 0;
constexpr int kRowsAny = 1;
constexpr int kRows22 = 2;

// SEG: several segments (F_Y above 2^16).
template <int ROWS, bool SEG>
__global__ void __launch_bounds__(T, 4)
    group_stream_kernel(const __grid_constant__ GroupArgs a, const uint32_t* __restrict__ yoff, uint32_t nseg,
                        uint32_t seg, const uint32_t* __restrict__ list, uint32_t count,
                        const __grid_constant__ StreamArgs sa) {
  extern __shared__ __align__(16) unsigned char smem[];
  StreamSmem& sm = *reinterpret_cast<StreamSmem*>(smem);
  __shared__ int32_t s_xc[kMaxOutOrder];  // the row's coordinates (its X part)
  uint16_t* const map = reinterpret_cast<uint16_t*>(sm.stab);
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  const uint32_t lt = lanemask_lt();
  const uint64_t keep = policy_evict_last();
  const uint64_t pol = policy_evict_first();
  const uint32_t* const yfk = static_cast<const uint32_t*>(a.yfk);
  const int oz = a.op.order;
  const uint32_t nwords = seg >> 5, dead = sa.dead;
  const uint32_t l8 = lane & 7;
  auto add_hole = [&](u64 pos, uint32_t len) {
    if (len == 0) return;
    sa.holes[atomicAdd(sa.nholes, 1u)] = StreamHole{pos, len};
    atomicAdd(sa.hole_total, (u64)len);
  };
  for (uint32_t i = threadIdx.x; i < kWords; i += T) sm.bits[i] = sm.rbits[i] = 0;
  for (uint32_t i = threadIdx.x; i < kHash; i += T) sm.hash[i] = kHashEmpty;
  __syncthreads();
  if (!SEG && threadIdx.x == 0) sm.bits[dead >> 5] |= 1u << (dead & 31);
  // Prefetched staging of the next group, when it is staged in one piece.
  uint32_t pf_g = 0, pf_x0 = 0, pf_n = 0, pf_ys = 0, pf_w = 0;
  double pf_v = 0.0;
  auto prefetch = [&](uint32_t gi) {
    if (gi >= count) return;
    pf_g = __ldg(list + gi);
    pf_x0 = __ldg(a.goff + pf_g);
    pf_n = __ldg(a.goff + pf_g + 1) - pf_x0;
    if (pf_n <= kEntries && threadIdx.x < pf_n) {
      pf_v = __ldg(a.gx.v + pf_x0 + threadIdx.x);
      if (SEG) {
        pf_ys = __ldg(a.gx.ck + pf_x0 + threadIdx.x);
      } else {
        pf_ys = __ldg(a.gx.ystart + pf_x0 + threadIdx.x);
        pf_w = __ldg(a.gx.w + pf_x0 + threadIdx.x);
      }
    }
  };
  u64 cur = 0;  // the CTA's leftover positions: [cur, cur + left)
  uint32_t left = 0;
  prefetch(blockIdx.x);
  for (uint32_t gi = blockIdx.x; gi < count; gi += gridDim.x) {
    const uint32_t g = pf_g, x0 = pf_x0, xn = pf_n;
    const bool one = xn <= kEntries;
    const uint32_t my_ys = pf_ys, my_w = pf_w;
    const double my_v = pf_v;
    prefetch(gi + gridDim.x);
    const u64 zrow = (u64)g * a.FY;
    // The run of X entry x0 + i in segment q.
    auto run_of = [&](uint32_t i, uint32_t q, uint32_t& ys, uint32_t& w) {
      if (SEG) {
        const u64 bin = (u64)(one ? my_ys : __ldg(a.gx.ck + x0 + i)) * nseg + q;
        ys = __ldg(yoff + bin);
        w = __ldg(yoff + bin + 1) - ys;
      } else {
        ys = one ? my_ys : __ldg(a.gx.ystart + x0 + i);
        w = one ? my_w : __ldg(a.gx.w + x0 + i);
      }
    };
    if (ROWS != kRowsAny && threadIdx.x == 0) {  // published by the staging's barriers
      if (ROWS == kRows4 || ROWS == kRows22) {
#pragma unroll
        for (int q = 0; q < 4; q++) s_xc[q] = out_coord_pow2(zrow, a.op, q);
      } else {
        decode_digits(zrow, a.op, [&](int q, int32_t c) { s_xc[q] = c; });
      }
    }
    for (uint32_t q = 0; q < (SEG ? nseg : 1u); q++) {
      // The counts of the last segment or group were read before the barrier that ends it; the
      // staging's barriers publish the cleared ones. (Every thread derives the leftover positions
      // from its own reading, so the clearing must not overtake a warp that has yet to read.)
      if (threadIdx.x == 0) sm.firsts = sm.repeats = 0;
      // The products, and their positions (a pass of its own for groups of several pieces).
      uint32_t products = 0, r = 0;
      auto reserve = [&](uint32_t n) {  // thread 0
        sm.base = left >= n ? 0 : atomicAdd(a.nz, (u64)n);
      };
      if (!one) {
        for (uint32_t c0 = 0; c0 < xn; c0 += kEntries) {
          uint32_t ys = 0, w = 0, tot;
          if (c0 + threadIdx.x < xn) run_of(c0 + threadIdx.x, q, ys, w);
          block_exscan(w, &tot, sm.warp_tot);
          products += tot;
          __syncthreads();
        }
        if (products == 0) continue;
        if (threadIdx.x == 0) reserve(products);
      }
      u64 da = 0, db = 0;
      const uint32_t dl = left;
      for (uint32_t c0 = 0; c0 < xn; c0 += kEntries) {
        uint32_t ys = 0, w = 0;
        if (c0 + threadIdx.x < xn) {
          sm.sx[threadIdx.x] = one ? my_v : __ldg(a.gx.v + x0 + c0 + threadIdx.x);
          run_of(c0 + threadIdx.x, q, ys, w);
        }
        // Products (high bits) and quarter-slots (low 12 bits) before each entry, in one scan; a
        // group staged in one piece reserves its positions between the scan's barriers.
        const uint32_t nq = (w + 7) >> 3;
        uint32_t x = (w << 12) | nq;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t t = __shfl_up_sync(0xffffffffu, x, o);
          if ((int)lane >= o) x += t;
        }
        if (lane == 31) sm.warp_tot[warp] = x;
        __syncthreads();
        uint32_t t = lane < NW ? sm.warp_tot[lane] : 0u, inc = t;
#pragma unroll
        for (int o = 1; o < NW; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
          if ((int)lane >= o) inc += y;
        }
        const uint32_t tot = __shfl_sync(0xffffffffu, inc, NW - 1);
        const uint32_t before = __shfl_sync(0xffffffffu, inc - t, warp);
        if (one) {
          products = tot >> 12;
          if (threadIdx.x == 0 && products) reserve(products);
        }
        const uint32_t h = tot & 4095u, hpad = (h + kStep - 1) / kStep * kStep;
        uint32_t s = (before + x - ((w << 12) | nq)) & 4095u;
        for (uint32_t k = 0; k < w; k += 8, s++)
          sm.stab[s] = make_uint2(ys + k, (w - k < 8 ? w - k : 8) | (threadIdx.x << 4));
        for (uint32_t i = h + threadIdx.x; i < hpad; i += T) sm.stab[i] = make_uint2(0, 0);
        __syncthreads();
        if (products == 0) continue;
        // Place p is output position p + (p < dl ? da : db).
        r = dl >= products ? 0u : products;
        da = cur;
        db = sm.base - dl;
        int4 xc = make_int4(0, 0, 0, 0);
        if (ROWS == kRows4 || ROWS == kRows22) xc = make_int4(s_xc[0], s_xc[1], s_xc[2], s_xc[3]);
        for (uint32_t qs = warp * (U * 4) + (lane >> 3); qs < hpad; qs += kStep) {
          uint32_t fk[U], e[U], old[U], m[U];
          double v[U];
#pragma unroll
          for (int u = 0; u < U; u++) {
            const uint2 rec = sm.stab[qs + 4 * u];
            const uint32_t j = l8 < (rec.y & 15u) ? rec.x + l8 : sa.ny_entries;
            e[u] = rec.y >> 4;
            fk[u] = ld_keep_u32(yfk + j, keep);
            v[u] = ld_keep_f64(a.yv + j, keep);
          }
#pragma unroll
          for (int u = 0; u < U; u++) {
            if (SEG) {
              old[u] = 0xffffffffu;
              if (fk[u] != dead) {
                fk[u] &= seg - 1;
                old[u] = atomicOr(sm.bits + (fk[u] >> 5), 1u << (fk[u] & 31));
              }
            } else {
              old[u] = atomicOr(sm.bits + (fk[u] >> 5), 1u << (fk[u] & 31));
            }
          }
          uint32_t c = 0;
#pragma unroll
          for (int u = 0; u < U; u++) {
            v[u] = __dmul_rn(sm.sx[e[u]], v[u]);
            m[u] = __ballot_sync(0xffffffffu, !((old[u] >> (fk[u] & 31)) & 1u));
            c += __popc(m[u]);
          }
          uint32_t place0 = 0;
          if (lane == 0) place0 = atomicAdd(&sm.firsts, c);
          place0 = __shfl_sync(0xffffffffu, place0, 0);
          uint32_t again = 0;
#pragma unroll
          for (int u = 0; u < U; u++) {
            if ((m[u] >> lane) & 1u) {
              const uint32_t place = place0 + __popc(m[u] & lt);
              sm.pk[place] = (uint16_t)fk[u];
              const u64 pos = (u64)place + (place < dl ? da : db);
              if constexpr (ROWS == kRows22) {
                const uint32_t z = SEG ? q * seg + fk[u] : fk[u];
                st_stream_v4(a.coords + pos * 4,
                             make_int4(xc.x, xc.y, (int32_t)((z >> sa.rsh[2]) & sa.rmk[2]),
                                       (int32_t)((z >> sa.rsh[3]) & sa.rmk[3])),
                             pol);
                a.vals[pos] = v[u];  // default policy: a repeat may still add to it
              } else if constexpr (ROWS == kRows4) {
                const uint32_t z = SEG ? q * seg + fk[u] : fk[u];
                st_stream_v4(a.coords + pos * 4,
                             make_int4(xc.x | (int32_t)((z >> sa.rsh[0]) & sa.rmk[0]),
                                       xc.y | (int32_t)((z >> sa.rsh[1]) & sa.rmk[1]),
                                       xc.z | (int32_t)((z >> sa.rsh[2]) & sa.rmk[2]),
                                       xc.w | (int32_t)((z >> sa.rsh[3]) & sa.rmk[3])),
                             pol);
                a.vals[pos] = v[u];
              } else if constexpr (ROWS >= 3) {
                int32_t cc[ROWS];
                uint32_t z = SEG ? q * seg + fk[u] : fk[u];
#pragma unroll
                for (int j = 0; j < ROWS; j++) {
                  const int i = ROWS - 1 - j;
                  if (j < sa.ny) {
                    const uint32_t hi = __umulhi(z, sa.ymagic[j]);
                    const uint32_t d = (hi + ((z - hi) >> sa.ysh1[j])) >> sa.ysh2[j];
                    cc[i] = (int32_t)(z - d * sa.ymod[j]);
                    z = d;
                  } else {
                    cc[i] = s_xc[i];
                  }
                }
                int32_t* const dst = a.coords + pos * ROWS;
                if constexpr (ROWS % 2 == 0) {
#pragma unroll
                  for (int i = 0; i < ROWS; i += 2)
                    asm volatile("st.global.L2::cache_hint.v2.s32 [%0], {%1, %2}, %3;" ::"l"(dst + i), "r"(cc[i]),
                                 "r"(cc[i + 1]), "l"(pol)
                                 : "memory");
                } else {
                  const int odd = (int)(pos & 1);  // odd rows start 4 bytes past an 8-byte boundary
                  if (odd) st_stream_s32(dst, cc[0], pol);
#pragma unroll
                  for (int i = 0; i + 1 < ROWS; i += 2) {
                    const int32_t lo = odd ? cc[i + 1] : cc[i], hi = odd ? cc[i + 2] : cc[i + 1];
                    asm volatile("st.global.L2::cache_hint.v2.s32 [%0], {%1, %2}, %3;" ::"l"(dst + i + odd), "r"(lo),
                                 "r"(hi), "l"(pol)
                                 : "memory");
                  }
                  if (!odd) st_stream_s32(dst + ROWS - 1, cc[ROWS - 1], pol);
                }
                a.vals[pos] = v[u];
              } else {
                store_output<false>(a.coords, a.vals, pos, zrow + (SEG ? (u64)q * seg : 0) + fk[u], v[u], a.op, pol);
              }
            } else if (fk[u] != dead) {
              again |= 1u << u;
            }
            place0 += __popc(m[u]);
          }
          // The step's repeats, a lane's one by one (few lanes have any, fewer have two).
#pragma unroll 1
          while (again) {
            const int u = __ffs(again) - 1;
            again &= again - 1;
            uint32_t key = fk[0];
            double val = v[0];
#pragma unroll
            for (int i = 1; i < U; i++)
              if (u == i) key = fk[i], val = v[i];
            const uint32_t at = shared_inc(&sm.repeats);
            if (at < kList) {
              sm.rk[at] = (uint16_t)key;
              sm.rv[at] = val;
            } else {  // beyond the list: at the back of the group's positions
              const uint32_t place = products - 1 - at;
              const u64 pos = (u64)place + (place < dl ? da : db);
              if (oz) a.coords[pos * oz] = (int32_t)key;
              a.vals[pos] = val;
            }
          }
        }
        if (!one) __syncthreads();
      }
      // The barrier orders the CTA's stores (outputs and repeats) before its reads and additions
      // below; no other CTA touches its positions.
      __syncthreads();
      if (products == 0) continue;
      const uint32_t firsts = sm.firsts, reps = sm.repeats;
      if (reps) {
        // The repeated keys: their bits, and a table of them or, where they are many, their ranks
        // (the key marks are no longer needed and hold the ranks). Then the firsts' keys are
        // looked through for them, eight per 16-byte load, and every repeat is added to its
        // first's entry.
        const bool few = reps <= kList;
        auto repeat_key = [&](uint32_t k) {
          if (k < kList) return (uint32_t)sm.rk[k];
          const uint32_t place = products - 1 - k;
          return oz ? (uint32_t)__ldcg(a.coords + ((u64)place + (place < dl ? da : db)) * oz) : 0u;
        };
        for (uint32_t k = threadIdx.x; k < reps; k += T) {
          const uint32_t key = repeat_key(k);
          atomicOr(sm.rbits + (key >> 5), 1u << (key & 31));
          if (few) {
            uint32_t h = (key * 0x9e3779b1u) >> 22;
            for (;;) {  // at most kList of kHash slots are taken
              const uint32_t was = atomicCAS(sm.hash + h, kHashEmpty, key << 16 | kNoPlace);
              if (was == kHashEmpty || was >> 16 == key) break;
              h = (h + 1) & (kHash - 1);
            }
          }
        }
        __syncthreads();
        if (!few) {
          const uint32_t wpt = (nwords + T - 1) / T;
          const uint32_t w0 = threadIdx.x * wpt, w1 = w0 + wpt < nwords ? w0 + wpt : nwords;
          uint32_t sum = 0;
          for (uint32_t w = w0; w < w1; w++) sum += __popc(sm.rbits[w]);
          uint32_t nrk;
          uint32_t rank = block_exscan(sum, &nrk, sm.warp_tot);
          for (uint32_t w = w0; w < w1; w++) {
            sm.bits[w] = rank;
            rank += __popc(sm.rbits[w]);
          }
          __syncthreads();
        }
        for (uint32_t i8 = threadIdx.x; i8 < (firsts + 7) / 8; i8 += T) {
          const uint4 eight = reinterpret_cast<const uint4*>(sm.pk)[i8];
          const uint32_t two[4] = {eight.x, eight.y, eight.z, eight.w};
#pragma unroll
          for (int t = 0; t < 8; t++) {
            const uint32_t i = i8 * 8 + t, fk = (two[t >> 1] >> ((t & 1) * 16)) & 0xffffu;
            const uint32_t rw = sm.rbits[fk >> 5];
            if (((rw >> (fk & 31)) & 1u) && i < firsts) {
              if (few)
                sm.hash[hash_find(sm.hash, fk)] = fk << 16 | i;
              else
                map[sm.bits[fk >> 5] + __popc(rw & ((1u << (fk & 31)) - 1u))] = (uint16_t)i;
            }
          }
        }
        __syncthreads();
        for (uint32_t k = threadIdx.x; k < reps; k += T) {
          const uint32_t key = repeat_key(k);
          uint32_t place = products - 1 - k;
          const double val = k < kList ? sm.rv[k] : __ldcg(a.vals + ((u64)place + (place < dl ? da : db)));
          place = few ? sm.hash[hash_find(sm.hash, key)] & (kNoPlace - 1)
                      : map[sm.bits[key >> 5] + __popc(sm.rbits[key >> 5] & ((1u << (key & 31)) - 1u))];
          atomicAdd(a.vals + ((u64)place + (place < dl ? da : db)), val);
        }
        __syncthreads();
        if (few) {
          for (uint32_t k = threadIdx.x; k < reps; k += T) sm.rbits[sm.rk[k] >> 5] = 0;
          for (uint32_t i = threadIdx.x; i < kHash; i += T) sm.hash[i] = kHashEmpty;
        } else {
          for (uint32_t i = threadIdx.x; i < nwords; i += T) sm.rbits[i] = 0;
        }
      }
      // What the group left over.
      if (firsts < left) {
        const uint32_t rest = left - firsts;  // and positions of its own: keep the larger part
        if (rest >= r) {
          if (threadIdx.x == 0) add_hole(sm.base, r);
          cur += firsts;
          left = rest;
        } else {
          if (threadIdx.x == 0) add_hole(cur + firsts, rest);
          cur = sm.base;
          left = r;
        }
      } else {
        const uint32_t used = firsts - left;
        cur = sm.base + used;
        left = r - used;
      }
      // ---- clear the bitmaps for the next segment or group.
      for (uint32_t i = threadIdx.x; i < nwords; i += T)
        sm.bits[i] = (!SEG && i == dead >> 5) ? 1u << (dead & 31) : 0u;
      __syncthreads();  // also ends the reading of this segment's counts
    }
  }
  if (threadIdx.x == 0) add_hole(cur, left);
}

// Filling the holes. With `tail` hole positions in all, the final count is nnz = reserved - tail: the
// entries at nnz and above (sources) move to the hole positions below (destinations), of which there
// are as many. Sources are taken a window of the tail at a time, in rounds that share one small array,
// so that the filling works with whatever scratch there is.

// A hole's words at and above nnz are marked in place: all ones, in a row's first and last word, is no
// output (coordinates are at least 0 and keys below 2^64 - 1).
__device__ __forceinline__ bool hole_marked(const int32_t* row, int oz) { return (row[0] & row[oz - 1]) == -1; }

// FIRST: holes above nnz are marked, the positions below are numbered through *ndst, and each hole
// becomes {position, number of its first destination << 16 | destinations}. Then the round's
// destinations [base, base + win) are listed: dst[k - base] is the hole that number k lies in.
template <bool FIRST>
__global__ void __launch_bounds__(256) hole_list_kernel(StreamHole* __restrict__ holes,
                                                        const unsigned* __restrict__ nholes,
                                                        const u64* __restrict__ reserved,
                                                        const u64* __restrict__ hole_total, HoleRound rd,
                                                        int32_t* __restrict__ coords, int oz, u64* __restrict__ ndst) {
  const unsigned lane = lane_id(), n = *nholes;
  const u64 nnz = *reserved - *hole_total;
  for (unsigned i = blockIdx.x * 8 + (threadIdx.x >> 5); i < n; i += gridDim.x * 8) {
    StreamHole h = holes[i];
    if (FIRST) {
      const u64 end = h.pos + h.len, cut = end < nnz ? end : (h.pos < nnz ? nnz : h.pos);
      const u64 below = cut - h.pos;
      u64 k = 0;
      if (lane == 0 && below) k = atomicAdd(ndst, below);
      k = __shfl_sync(0xffffffffu, k, 0);
      for (u64 q = cut + lane; q < end; q += 32) coords[q * oz] = coords[q * oz + oz - 1] = -1;
      h.len = k << 16 | below;
      if (lane == 0) holes[i] = h;
    }
    const u64 k0 = h.len >> 16, k1 = k0 + (h.len & 0xffffu);
    const u64 a = k0 > rd.base ? k0 : rd.base, e = k1 < rd.base + rd.win ? k1 : rd.base + rd.win;
    for (u64 k = a + lane; k < e; k += 32) rd.dst[k - rd.base] = i;
  }
}

// The window's entries that are no holes move to the destinations that follow the last round's.
__global__ void __launch_bounds__(256) hole_fill_kernel(const StreamHole* __restrict__ holes,
                                                        const u64* __restrict__ reserved,
                                                        const u64* __restrict__ hole_total, HoleRound rd,
                                                        const u64* __restrict__ ndst, u64* __restrict__ nsrc,
                                                        int32_t* __restrict__ coords, double* __restrict__ vals,
                                                        int oz, uint32_t* status) {
  const u64 tail = *hole_total, last = *ndst;
  const u64 nnz = *reserved - tail;
  const u64 end = tail < rd.at + rd.win ? tail : rd.at + rd.win;
  for (u64 t0 = rd.at + (((u64)blockIdx.x * 256 + threadIdx.x) & ~31ull); t0 < end; t0 += (u64)gridDim.x * 256) {
    const u64 t = t0 + lane_id(), s = nnz + t;
    const bool has = t < end && !hole_marked(coords + s * oz, oz);
    const u64 k = warp_reserve(has, nsrc);
    if (!has) continue;
    if (k >= last) {
      atomicOr(status, kStatOutOverflow);
      continue;
    }
    const StreamHole h = holes[rd.dst[k - rd.base]];
    const u64 d = h.pos + (k - (h.len >> 16));
    if (oz == 4 && ((reinterpret_cast<uintptr_t>(coords) & 15u) == 0)) {
      reinterpret_cast<int4*>(coords)[d] = reinterpret_cast<const int4*>(coords)[s];
    } else {
      for (int q = 0; q < oz; q++) coords[d * oz + q] = coords[s * oz + q];
    }
    vals[d] = vals[s];
  }
}

template <bool SEG>
cudaError_t launch_rows(const GroupArgs& a, const uint32_t* yoff, uint32_t nseg, uint32_t seg, const uint32_t* list,
                        uint32_t count, const StreamArgs& sa, int rows, int sms, cudaStream_t s) {
  auto kern = group_stream_kernel<kRowsAny, SEG>;
  switch (rows) {
    case kRows4: kern = group_stream_kernel<kRows4, SEG>; break;
    case kRows22: kern = group_stream_kernel<kRows22, SEG>; break;
    case 3: kern = group_stream_kernel<3, SEG>; break;
    case 4: kern = group_stream_kernel<4, SEG>; break;
    case 5: kern = group_stream_kernel<5, SEG>; break;
    case 6: kern = group_stream_kernel<6, SEG>; break;
    default: break;
  }
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(StreamSmem));
  if (e != cudaSuccess) return e;
  const uint32_t grid = (uint32_t)sms * 4;
  kern<<<count < grid ? count : grid, T, sizeof(StreamSmem), s>>>(a, yoff, nseg, seg, list, count, sa);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

// F_Y itself where its bit is none of the keys'; no key at all where the keys need the mask.
uint32_t stream_dead_key(u64 FY) { return FY > kDenseSeg ? 0xffffffffu : (uint32_t)FY; }

uint32_t stream_cap() { return kCap; }

// A CTA drops positions at most once per segment, never in its first (it has none left over yet), and
// lists what it has left over at its end.
size_t stream_max_holes(uint32_t count, uint32_t nseg) { return (size_t)count * nseg; }

cudaError_t launch_group_stream(const GroupArgs& a, const uint32_t* yoff, uint32_t nseg, uint32_t seg,
                                const uint32_t* list, uint32_t count, const StreamArgs& sa_in, int sms,
                                cudaStream_t s) {
  if (count == 0) return cudaSuccess;
  if (seg < 64 || seg > kDenseSeg) return cudaErrorInvalidValue;
  StreamArgs sa = sa_in;
  sa.dead = stream_dead_key(a.FY);
  int rows = kRowsAny;
  if (a.op.order == 4 && a.op.pow2 && (reinterpret_cast<uintptr_t>(a.coords) & 15u) == 0) {
    // A coordinate is a bit field of the Y free key or constant over the row.
    rows = kRows4;
    bool y_part[4];
    for (int q = 0; q < 4; q++) {
      const bool of_y = y_part[q] = (1ull << a.op.shift[q]) < a.FY;
      sa.rsh[q] = of_y ? a.op.shift[q] : 0;
      sa.rmk[q] = of_y ? (uint32_t)a.op.mod[q] - 1 : 0;
    }
    if (!y_part[0] && !y_part[1] && y_part[2] && y_part[3]) rows = kRows22;
  } else if (!a.op.pow2 && a.op.ident && a.op.order >= 3 && a.op.order <= 6 &&
             (reinterpret_cast<uintptr_t>(a.coords) & 7u) == 0) {
    // The Y part of the output key has the last ny digits; F_Y is below 2^32 here.
    rows = a.op.order;
    u64 fy = 1;
    for (int j = 0; j < rows && fy < a.FY; j++) {
      const u64 d = a.op.mod[rows - 1 - j];
      const uint32_t l = d <= 1 ? 0 : 64 - (uint32_t)__builtin_clzll(d - 1);
      sa.ymod[j] = (uint32_t)d;
      sa.ymagic[j] = (uint32_t)(((((unsigned __int128)1 << l) - d) << 32) / d + 1);
      sa.ysh1[j] = l < 1 ? l : 1;
      sa.ysh2[j] = l > 1 ? l - 1 : 0;
      sa.ny = j + 1;
      fy *= d;
    }
    if (fy != a.FY) rows = kRowsAny;
  }
  return nseg > 1 ? launch_rows<true>(a, yoff, nseg, seg, list, count, sa, rows, sms, s)
                  : launch_rows<false>(a, yoff, nseg, seg, list, count, sa, rows, sms, s);
}

cudaError_t launch_hole_fill(StreamHole* holes, const unsigned* nholes, const u64* reserved, const u64* hole_total,
                             const HoleRound& rd, u64* counters2, int32_t* coords, double* vals, int oz,
                             uint32_t* status, int sms, cudaStream_t s) {
  if (rd.win == 0 || oz <= 0) return cudaErrorInvalidValue;  // an output without modes has no holes
  const u64 g = (u64)sms * 8, want = (rd.win + 255) / 256;
  auto list = rd.at == 0 ? hole_list_kernel<true> : hole_list_kernel<false>;
  list<<<(unsigned)(want < (u64)sms ? want : (u64)sms), 256, 0, s>>>(holes, nholes, reserved, hole_total, rd, coords, oz,
                                                                     counters2);
  hole_fill_kernel<<<(unsigned)(want < g ? want : g), 256, 0, s>>>(holes, reserved, hole_total, rd, counters2,
                                                                   counters2 + 1, coords, vals, oz, status);
  note_launch(2);
  return cudaGetLastError();
}

}  // namespace stc
