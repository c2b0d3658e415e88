// The larger groups of a batch (beyond the warp-sized tables): their outputs belong to one of many
// problems and are counted exactly before any is written, so that no position is left over.
//
// One group at a time per CTA, its products listed in quarter-slots (up to 8 consecutive Y entries of
// one X entry's run, four to a warp and step). Pass 1 reads the keys and marks them in a bitmap: the
// product that finds its bit clear is its key's first; a product that finds it set marks the key in
// a second bitmap. A ballot per slot records the firsts. Their prefix gives every first its place,
// and one atomic on the problem's counter reserves exactly as many positions. Pass 2 reads keys and
// values, writes the firsts' outputs, and puts the place of those whose key repeats into a small
// table; repeats wait in a list and are added to their firsts' entries after a barrier. Groups with
// more repeats than are listed rank the repeated keys instead, and a third pass adds the repeats.
#include "target.cuh"

namespace stc {

namespace {

constexpr int U = 4;  // slots per warp and step
// Most repeats listed, by groups of up to kListSmall products (larger ones list half as many), and the
// slots of the table of their keys. 3e7 products in groups of 7,700 over 6e4 even keys (some 490 repeats)
// take 0.60 ms listed and 0.30 ranked; in groups of 800 over keys by a Zipf law of exponent 1.0 (some 350)
// 0.54 listed and 0.74 ranked.
constexpr uint32_t kList = 512, kListSmall = 2048, kHash = 1024;
constexpr uint32_t kHashEmpty = 0xffffffffu;

template <int T, uint32_t WORDS, uint32_t CAP>
struct TwoPassSmem {
  static constexpr uint32_t kStep = T / 32 * U * 4;  // quarter-slots per step
  static constexpr uint32_t kQuarters = (CAP / 8 + T + kStep - 1) / kStep * kStep;
  static_assert(CAP < (1u << 16) && CAP / 8 + T < (1u << 13), "places in 16 bits, quarter-slots in 13");
  uint32_t bits[WORDS];    // keys met; then (many repeats) the rank of each word's first repeated key
  uint32_t rbits[WORDS];   // keys met again
  uint2 stab[kQuarters];   // quarter-slots: first Y entry; entries | staged X entry << 4
  uint32_t mask[kQuarters / 4], pref[kQuarters / 4];  // per slot: ballot of the firsts, firsts before it
  double sx[T];
  union {
    struct {
      double rv[kList];        // repeats: values and keys
      uint32_t rk[kList];
      uint32_t hkey[kHash];    // repeated keys and the places of their firsts
      uint16_t hplace[kHash];
    } few;
    uint16_t map[CAP / 2];     // rank of a repeated key -> place of its first
  };
  OutTarget tg;
  u64 base;
  uint32_t warp_tot[T / 32 + 1];
  uint32_t reps, listed;
};

// Exclusive block scan of one value per thread; *total receives the sum. Two barriers.
template <int T>
__device__ __forceinline__ uint32_t block_exscan(uint32_t v, uint32_t* total, uint32_t* warp_tot) {
  constexpr int NW = T / 32;
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
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if ((int)lane >= o) inc += y;
    }
    if (lane < NW) warp_tot[lane] = inc - t;
    if (lane == 31) warp_tot[NW] = inc;
  }
  __syncthreads();
  *total = warp_tot[NW];
  return warp_tot[warp] + x - v;
}

__device__ __forceinline__ uint32_t hash_of(uint32_t key) { return (key * 0x9e3779b1u) >> 22; }

__device__ __forceinline__ void store_target(const OutTarget& t, u64 pos, uint32_t fk, double v, uint64_t pol) {
  if (t.op.split) {
    int32_t* const dst = t.coords + pos * (u64)t.op.order;
    switch (t.op.order) {
      case 4: store_row_split<4>(dst, t.xc, fk, t.op, pol); break;
      case 3: store_row_split<3>(dst, t.xc, fk, t.op, pol); break;
      case 2: store_row_split<2>(dst, t.xc, fk, t.op, pol); break;
      case 5: store_row_split<5>(dst, t.xc, fk, t.op, pol); break;
      case 6: store_row_split<6>(dst, t.xc, fk, t.op, pol); break;
      case 7: store_row_split<7>(dst, t.xc, fk, t.op, pol); break;
      default: store_row_split<8>(dst, t.xc, fk, t.op, pol); break;
    }
    t.vals[pos] = v;  // default policy: a repeat may still add to it
  } else {
    store_output<false>(t.coords, t.vals, pos, t.zrow + fk, v, t.op, pol);
  }
}

template <int T, uint32_t WORDS, uint32_t CAP, int MINB>
__global__ void __launch_bounds__(T, MINB) group_twopass_kernel(GroupArgs a, const uint32_t* __restrict__ list,
                                                                const uint32_t* __restrict__ countp) {
  using Smem = TwoPassSmem<T, WORDS, CAP>;
  constexpr uint32_t kStep = Smem::kStep;
  extern __shared__ __align__(16) unsigned char smem[];
  Smem& sm = *reinterpret_cast<Smem*>(smem);
  const uint32_t count = *countp;
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  const uint32_t lt = lanemask_lt(), l8 = lane & 7;
  const uint64_t keep = policy_evict_last();
  const uint64_t pol = policy_evict_first();
  const uint32_t* const yfk = static_cast<const uint32_t*>(a.yfk);
  for (uint32_t i = threadIdx.x; i < WORDS; i += T) sm.bits[i] = sm.rbits[i] = 0;
  for (uint32_t i = threadIdx.x; i < kHash; i += T) sm.few.hkey[i] = kHashEmpty;
  if (threadIdx.x == 0) {
    sm.reps = sm.listed = 0;
    sm.tg.prob = kNoProb;
  }
  __syncthreads();
  uint32_t pf_g = 0, pf_x0 = 0, pf_n = 0, pf_ys = 0, pf_w = 0;
  double pf_v = 0.0;
  auto prefetch = [&](uint32_t gi) {
    if (gi >= count) return;
    pf_g = __ldg(list + gi);
    pf_x0 = __ldg(a.goff + pf_g);
    pf_n = __ldg(a.goff + pf_g + 1) - pf_x0;
    pf_w = 0;
    if (threadIdx.x < pf_n) {
      pf_v = __ldg(a.gx.v + pf_x0 + threadIdx.x);
      pf_ys = __ldg(a.gx.ystart + pf_x0 + threadIdx.x);
      pf_w = __ldg(a.gx.w + pf_x0 + threadIdx.x);
    }
  };
  prefetch(blockIdx.x);
  for (uint32_t gi = blockIdx.x; gi < count; gi += gridDim.x) {
    const uint32_t g = pf_g, n = pf_n, ys = pf_ys, w = pf_w;
    const double xv = pf_v;
    prefetch(gi + gridDim.x);
    if (warp == 0) {
      resolve_target_warp(a, g, 0, sm.tg);
      if (lane == 0 && sm.tg.op.split) decode_x_part((uint32_t)sm.tg.fx, sm.tg.op, sm.tg.xc);
    }
    sm.sx[threadIdx.x] = xv;
    // Products (high bits) and quarter-slots (low 13) before each entry.
    const uint32_t nq = (w + 7) >> 3;
    uint32_t tot;
    const uint32_t before = block_exscan<T>((w << 13) | nq, &tot, sm.warp_tot);  // its barriers publish tg
    const uint32_t h = tot & 8191u, hpad = (h + kStep - 1) / kStep * kStep;
    if (n > (uint32_t)T || (tot >> 13) > CAP) {  // not binned here
      if (threadIdx.x == 0) atomicOr(a.status, kStatOutOverflow);
      __syncthreads();
      continue;
    }
    uint32_t s = before & 8191u;
    for (uint32_t k = 0; k < w; k += 8, s++)
      sm.stab[s] = make_uint2(ys + k, (w - k < 8 ? w - k : 8) | (threadIdx.x << 4));
    for (uint32_t i = h + threadIdx.x; i < hpad; i += T) sm.stab[i] = make_uint2(0, 0);
    __syncthreads();
    if (n == 1 && a.yuniq != nullptr && a.yuniq[sm.stab[0].x]) {
      // One X entry over a run of all-different free keys: the run scaled by x.
      const uint32_t len = tot >> 13, y0 = sm.stab[0].x;
      if (threadIdx.x == 0) sm.base = atomicAdd(sm.tg.counter, (u64)len);
      __syncthreads();
      const u64 base = sm.base;
      if (base + len <= sm.tg.cap) {
        for (uint32_t j = threadIdx.x; j < len; j += T)
          store_target(sm.tg, base + j, ld_keep_u32(yfk + y0 + j, keep),
                       __dmul_rn(sm.sx[0], ld_keep_f64(a.yv + y0 + j, keep)), pol);
      } else if (threadIdx.x == 0) {
        atomicOr(a.status, kStatOutOverflow);
      }
      __syncthreads();  // tg and the staging are rewritten for the next group
      continue;
    }
    // ---- pass 1: keys.
    uint32_t my_reps = 0;
    for (uint32_t qs = warp * (U * 4); qs < hpad; qs += kStep) {
      uint32_t fk[U], old[U], firsts = 0;
      bool live[U];
#pragma unroll
      for (int u = 0; u < U; u++) {
        const uint2 rec = sm.stab[qs + 4 * u + (lane >> 3)];
        live[u] = l8 < (rec.y & 15u);
        fk[u] = ld_keep_u32(yfk + (live[u] ? rec.x + l8 : 0u), keep);
      }
#pragma unroll
      for (int u = 0; u < U; u++) {
        old[u] = 0xffffffffu;
        if (live[u]) old[u] = atomicOr(sm.bits + (fk[u] >> 5), 1u << (fk[u] & 31));
      }
#pragma unroll
      for (int u = 0; u < U; u++) {
        const bool first = !((old[u] >> (fk[u] & 31)) & 1u);
        const uint32_t m = __ballot_sync(0xffffffffu, first);
        if ((int)lane == u) firsts = m;
        if (live[u] && !first) {
          atomicOr(sm.rbits + (fk[u] >> 5), 1u << (fk[u] & 31));
          my_reps++;
        }
      }
      if (lane < U) sm.mask[qs / 4 + lane] = firsts;
    }
    my_reps = __reduce_add_sync(0xffffffffu, my_reps);
    if (lane == 0 && my_reps) atomicAdd(&sm.reps, my_reps);
    __syncthreads();
    // ---- places: a prefix over the slots, a few consecutive ones per thread.
    const uint32_t nslots = hpad / 4, per = (nslots + T - 1) / T;
    uint32_t sum = 0;
    for (uint32_t i = threadIdx.x * per; i < (threadIdx.x + 1) * per && i < nslots; i++) sum += __popc(sm.mask[i]);
    uint32_t firsts;
    uint32_t run = block_exscan<T>(sum, &firsts, sm.warp_tot);
    if (threadIdx.x == 0) sm.base = atomicAdd(sm.tg.counter, (u64)firsts);
    for (uint32_t i = threadIdx.x * per; i < (threadIdx.x + 1) * per && i < nslots; i++) {
      sm.pref[i] = run;
      run += __popc(sm.mask[i]);
    }
    const uint32_t reps = sm.reps;
    const bool few = reps <= (tot >> 13 <= kListSmall ? kList : kList / 2);
    const uint32_t nwords = (uint32_t)((sm.tg.FY + 31) >> 5);
    if (!few) {  // the key marks are no longer needed and hold the ranks of the repeated keys
      const uint32_t wpt = (nwords + T - 1) / T;
      const uint32_t w0 = threadIdx.x * wpt, w1 = w0 + wpt < nwords ? w0 + wpt : nwords;
      uint32_t rsum = 0, all;
      for (uint32_t i = w0; i < w1; i++) rsum += __popc(sm.rbits[i]);
      __syncthreads();
      uint32_t rank = block_exscan<T>(rsum, &all, sm.warp_tot);
      for (uint32_t i = w0; i < w1; i++) {
        sm.bits[i] = rank;
        rank += __popc(sm.rbits[i]);
      }
    }
    __syncthreads();
    const u64 base = sm.base;
    const bool fits = base + firsts <= sm.tg.cap;
    if (!fits && threadIdx.x == 0) atomicOr(a.status, kStatOutOverflow);
    auto rank_of = [&](uint32_t key) {
      return sm.bits[key >> 5] + __popc(sm.rbits[key >> 5] & ((1u << (key & 31)) - 1u));
    };
    // ---- pass 2: keys and values; the outputs.
    for (uint32_t qs = warp * (U * 4); fits && qs < hpad; qs += kStep) {
      uint32_t fk[U], e[U];
      double v[U];
      bool live[U];
#pragma unroll
      for (int u = 0; u < U; u++) {
        const uint2 rec = sm.stab[qs + 4 * u + (lane >> 3)];
        live[u] = l8 < (rec.y & 15u);
        const uint32_t j = live[u] ? rec.x + l8 : 0u;
        e[u] = rec.y >> 4;
        fk[u] = ld_keep_u32(yfk + j, keep);
        v[u] = ld_keep_f64(a.yv + j, keep);
      }
#pragma unroll
      for (int u = 0; u < U; u++) {
        v[u] = __dmul_rn(sm.sx[e[u]], v[u]);
        const uint32_t m = sm.mask[qs / 4 + u];
        if ((m >> lane) & 1u) {
          const uint32_t place = sm.pref[qs / 4 + u] + __popc(m & lt);
          store_target(sm.tg, base + place, fk[u], v[u], pol);
          if (reps && ((sm.rbits[fk[u] >> 5] >> (fk[u] & 31)) & 1u)) {
            if (few) {
              uint32_t i = hash_of(fk[u]);
              while (atomicCAS(sm.few.hkey + i, kHashEmpty, fk[u]) != kHashEmpty) i = (i + 1) & (kHash - 1);
              sm.few.hplace[i] = (uint16_t)place;
            } else {
              sm.map[rank_of(fk[u])] = (uint16_t)place;
            }
          }
        } else if (few && live[u]) {
          const uint32_t at = atomicAdd(&sm.listed, 1u);
          sm.few.rk[at] = fk[u];
          sm.few.rv[at] = v[u];
        }
      }
    }
    __syncthreads();  // also orders the outputs before the additions to them below
    if (reps && fits) {
      if (few) {
        for (uint32_t k = threadIdx.x; k < reps; k += T) {
          const uint32_t key = sm.few.rk[k];
          uint32_t i = hash_of(key);
          while (sm.few.hkey[i] != key) i = (i + 1) & (kHash - 1);
          atomicAdd(sm.tg.vals + base + sm.few.hplace[i], sm.few.rv[k]);
        }
      } else {
        for (uint32_t qs = warp * (U * 4); qs < hpad; qs += kStep)
          for (int u = 0; u < U; u++) {
            const uint2 rec = sm.stab[qs + 4 * u + (lane >> 3)];
            if (l8 < (rec.y & 15u) && !((sm.mask[qs / 4 + u] >> lane) & 1u)) {
              const uint32_t j = rec.x + l8, key = ld_keep_u32(yfk + j, keep);
              atomicAdd(sm.tg.vals + base + sm.map[rank_of(key)],
                        __dmul_rn(sm.sx[rec.y >> 4], ld_keep_f64(a.yv + j, keep)));
            }
          }
      }
      __syncthreads();
    }
    // ---- clear for the next group.
    for (uint32_t i = threadIdx.x; i < nwords; i += T) sm.bits[i] = 0;
    if (reps) {
      for (uint32_t i = threadIdx.x; i < nwords; i += T) sm.rbits[i] = 0;
      for (uint32_t i = threadIdx.x; i < kHash; i += T) sm.few.hkey[i] = kHashEmpty;
    }
    if (threadIdx.x == 0) sm.reps = sm.listed = 0;
    __syncthreads();
  }
}

template <int T, uint32_t WORDS, uint32_t CAP, int MINB>
cudaError_t launch_one(const GroupArgs& a, const uint32_t* list, const uint32_t* countp, uint32_t count, int sms,
                       cudaStream_t s) {
  if (count == 0) return cudaSuccess;
  constexpr size_t smem = sizeof(TwoPassSmem<T, WORDS, CAP>);
  static_assert(MINB * (smem + 1024) <= 228 * 1024, "CTAs per SM");
  auto kern = group_twopass_kernel<T, WORDS, CAP, MINB>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const uint32_t grid = (uint32_t)sms * MINB;
  kern<<<count < grid ? count : grid, T, smem, s>>>(a, list, countp);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_group_twopass(const GroupArgs& a, const Bins& b, const uint32_t* counts, int sms, cudaStream_t s) {
  const uint32_t* d = b.count + kMaxClasses + 1;
  auto n = [&](int l) { return counts ? counts[kMaxClasses + 1 + l] : kCountOnDevice; };
  cudaError_t e;
  if ((e = launch_one<256, 2048, 8192, 4>(a, b.dense_list[0], d, n(0), sms, s))) return e;
  if ((e = launch_one<512, 8192, 16384, 2>(a, b.dense_list[1], d + 1, n(1), sms, s))) return e;
  return launch_one<1024, 8192, 49152, 1>(a, b.dense_list[2], d + 2, n(2), sms, s);
}

}  // namespace stc
