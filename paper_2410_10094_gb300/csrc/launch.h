// Host-side launchers of the library's kernels. Internal; the public ABI is include/stc.h.
#pragma once

#include "common.cuh"

namespace stc {

using u64 = unsigned long long;

// Kernels launched by the calling thread since the last take_launches() (for the stats).
void note_launch(unsigned n = 1);
unsigned take_launches();

// ------------------------------------------------------------------ scans (scan.cu)
// Exclusive prefix sums: out[0] = 0, out[i] = in[0] + ... + in[i-1], out[n] = total.
// `scratch` holds scan_scratch_elems(n) elements of the output type.
int64_t scan_scratch_elems(int64_t n);
// out2 (may be null) receives out[0..n-1] as well.
cudaError_t scan_u32(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* scratch, cudaStream_t s,
                     uint32_t* out2 = nullptr);
cudaError_t scan_u32_u64(const uint32_t* in, u64* out, int64_t n, u64* scratch, cudaStream_t s);
cudaError_t scan_u64(const u64* in, u64* out, int64_t n, u64* scratch, cudaStream_t s);

// ------------------------------------------------------------------ preparation (prep.cu)
// Contract key of every entry (the LN key of the contract modes): keys[i] = ckey(i).
cudaError_t launch_linearize(const int32_t* coords, int64_t n, const KeyPlan& p, u64* keys,
                             uint32_t* status, int sms, cudaStream_t s);

// Counting sort of arbitrary keys in [0, k): count, then scatter through a cursor copy of
// the offsets. perm[pos] = input index.
cudaError_t launch_key_count(const u64* keys, int64_t n, u64 k, uint32_t* cnt, uint32_t* status,
                             int sms, cudaStream_t s);
cudaError_t launch_key_scatter(const u64* keys, int64_t n, u64 k, uint32_t* cursor, uint32_t* perm,
                               int sms, cudaStream_t s);

// Group Y by contract key (Section 4.2): histogram of ckey, then (after a scan) a scatter
// of each entry's free key and value into its key's run.
// nonempty (may be null): K/32 words, zeroed by the caller, receive the bitmap of the contract
// keys that have at least one Y entry.
cudaError_t launch_y_count(const int32_t* coords, int64_t n, const KeyPlan& p, uint32_t* cnt,
                           uint32_t* status, int sms, cudaStream_t s, uint32_t* nonempty = nullptr);
// yfk receives 32-bit free keys when key32 is set (F_Y < 2^32), 64-bit ones otherwise. 32-bit
// arrays hold n + 1 entries: the last has the key stream_dead_key(FY) and the value 0.
uint32_t stream_dead_key(u64 FY);
cudaError_t launch_y_scatter(const int32_t* coords, const double* vals, int64_t n, const KeyPlan& p, u64 FY,
                             uint32_t* cursor, void* yfk, bool key32, double* yv, int sms, cudaStream_t s);

// The id map of a contract key space of K keys (KeyPlan::idmap, id_map_pairs(K) pairs): Y's contract
// keys marked and ranked. *ids receives their number. scratch: id_map_scratch(K) elements.
constexpr u64 id_map_pairs(u64 K) { return (K + 31) / 32; }
int64_t id_map_scratch(u64 K);
cudaError_t launch_id_map(const int32_t* coords, int64_t n, const KeyPlan& p, u64 K, uint2* map, uint32_t* scratch,
                          uint32_t* ids, uint32_t* status, int sms, cudaStream_t s);

// X entries whose contract key has a non-empty Y run ("survivors"), compacted, with the
// run they will read and the total product count P (Section 4.3).
struct Survivors {
  u64* fk;          // X free key
  uint32_t* ck;     // X contract key (kept only when per-segment runs are needed; may be null)
  uint32_t* ystart; // first slot of the matching Y run
  uint32_t* w;      // run length = products this entry makes
  double* v;        // X value
  unsigned* count;  // number of survivors (device counter)
  u64* bsum;        // null, or products of every block of kSurvivorBlock survivors (zeroed by the caller)
};
constexpr unsigned kSurvivorBlock = 1024;
// With gcnt non-null, also counts survivors per X free key.
// `nonempty` (K / 32 words of scratch, may be null) is used when K <= kNonemptyMaxKeys: a
// bitmap of the contract keys that have a Y run, held in shared memory by the survey so that
// rows without a run skip the lookup; built here from the runs unless nonempty_built (then
// launch_y_count built it).
constexpr u64 kNonemptyMaxKeys = 1ull << 18;
cudaError_t launch_x_survey(const int32_t* coords, const double* vals, int64_t n, const KeyPlan& p,
                            const uint32_t* yoff, u64 K, Survivors sv, u64* P, uint32_t* gcnt, uint32_t* status,
                            uint32_t* nonempty, int sms, cudaStream_t s, bool nonempty_built = false);

// Dense X (Y runs exist for most contract keys): count entries with a run per X free key
// and the products, then place them in group order straight from the input, without an
// intermediate survivor list.
struct GroupedX;
cudaError_t launch_x_count(const int32_t* coords, int64_t n, const KeyPlan& p, const uint32_t* yoff, u64* P,
                           uint32_t* gcnt, uint32_t* status, int sms, cudaStream_t s);
cudaError_t launch_x_scatter_dense(const int32_t* coords, const double* vals, int64_t n, const KeyPlan& p,
                                   const uint32_t* yoff, uint32_t* gcur, GroupedX gx, uint32_t* status, int sms,
                                   cudaStream_t s);

// A tensor in key form split into (free part / FL, free part % FL, contract digits): see
// keyed_split_kernel. K and F are the contract and free key spaces (K * F = prod(shape)).
struct KeySplit {
  u64 K, F, FL;
  int32_t m;
  int32_t trailing;  // contracted modes last (1) or first (0)
  int64_t csize[kMaxOrder];
};
cudaError_t launch_keyed_split(const u64* keys, int64_t n, const KeySplit& ks, int32_t* out, uint32_t* status,
                               int sms, cudaStream_t s);

// ------------------------------------------------------------------ dense ids (ids.cu)
// Distinct keys collected in an open-addressing table and numbered densely (Section 4.1.2).
// keys[slots] (all-ones = empty), flags[slots + 1] (flags[slots] = the all-ones key was
// seen), prefix[slots + 2] = exclusive scan of flags: the id of the key in slot h is
// prefix[h], the all-ones key's is prefix[slots], and prefix[slots + 1] = D, the number of
// distinct keys, which is also the id given to a key the table lacks.
struct IdTable {
  u64* keys;
  uint32_t* flags;
  uint32_t* prefix;
  u64 slots;  // a power of two >= 2n
};
uint64_t id_table_slots(int64_t n);
cudaError_t launch_id_insert_keys(const u64* keys, int64_t n, const IdTable& t, uint32_t* status, int sms,
                                  cudaStream_t s);
// Inserts the contract key of every coordinate row.
cudaError_t launch_id_insert_rows(const int32_t* coords, int64_t n, const KeyPlan& p, const IdTable& t,
                                  uint32_t* status, int sms, cudaStream_t s);
// Flags the occupied slots and scans them into prefix (scratch: scan_scratch_elems(slots + 1)).
cudaError_t launch_id_number(const IdTable& t, uint32_t* scratch, int sms, cudaStream_t s);
cudaError_t launch_id_lookup_keys(const u64* keys, int64_t n, const IdTable& t, uint32_t* ids, int sms,
                                  cudaStream_t s);
// out[i] = (free coordinates of row i, ascending mode order; id of its contract key), nf + 1
// int32 per row. fmask has bit j set for each free mode j.
cudaError_t launch_id_rewrite_rows(const int32_t* coords, int64_t n, const KeyPlan& p, uint32_t fmask, int nf,
                                   const IdTable& t, int32_t* out, uint32_t* status, int sms, cudaStream_t s);

// ------------------------------------------------------------------ one global table (global.cu)
struct GlobalTable {
  u64* keys;    // [cap], kEmpty64 when free; null: an array of the whole output space (cap >= F)
  double* vals; // [cap]
  u64 mask;     // cap - 1, cap a power of two
};
// Expansion with a merge-path split over the survivors' product prefix `wpre` (ns+1
// entries, wpre[ns] = P): every CTA takes an equal share of the P products. probe: lanes that
// probe the table together (1: each lane alone over slots; 4 or 8: tiles over buckets of that
// many slots).
cudaError_t launch_expand_global(const u64* wpre, int64_t ns, u64 P, Survivors sv, const u64* yfk,
                                 const double* yv, u64 FY, GlobalTable t, uint32_t* status, int sms,
                                 cudaStream_t s, int probe);
// The same with everything read on the device (no host read between the survey and the expansion):
// the survivor count, and the products per block of survivors (sv.bsum), whose prefix a first kernel
// writes to bpre (one element more than sv.bsum). t.keys null: t is an array of the whole output space,
// cleared by launch_clear_space.
cudaError_t launch_expand_blocks(Survivors sv, u64* bpre, const u64* yfk, const double* yv, u64 FY, GlobalTable t,
                                 uint32_t* status, int sms, cudaStream_t s, int probe);
cudaError_t launch_clear_space(GlobalTable t, int sms, cudaStream_t s);
// The same for large output key spaces: outputs written as their keys are claimed, repeats listed and
// added by a second kernel.
struct DirectTable {
  u64* keys;           // [mask + 1], kEmpty64 when free
  uint32_t* pos;       // [mask + 1] output position of the slot's key
  u64 mask;            // mask + 1 <= 2^32
  uint32_t* rep_slot;  // [P]
  double* rep_val;     // [P]
  u64* nreps;          // zeroed by the caller
};
cudaError_t launch_expand_direct(const u64* wpre, int64_t ns, u64 P, Survivors sv, const u64* yfk, const double* yv,
                                 u64 FY, const DirectTable& t, const OutPlan& op, int32_t* coords, double* vals,
                                 u64 out_cap, u64* nz, uint32_t* status, int sms, cudaStream_t s);
// Occupied slots -> COO output (coordinates decoded from the key).
cudaError_t launch_compact_global(GlobalTable t, const OutPlan& op, int32_t* coords, double* vals, u64 out_cap,
                                  u64* nz, uint32_t* status, int sms, cudaStream_t s);

// ------------------------------------------------------------------ per-group tables (grouped.cu)
constexpr int kMaxClasses = 5;

struct ClassShape {
  uint32_t slots;    // table slots in shared memory
  uint32_t threads;  // threads per CTA
};
extern const ClassShape kClassShapes32[];  // 32-bit local keys (F_Y < 2^32)
extern const ClassShape kClassShapes64[];  // 64-bit local keys
extern const int kNumClasses32;
extern const int kNumClasses64;

// X survivors in group order: the entries of X free key g are [goff[g], goff[g+1]).
struct GroupedX {
  uint32_t* ystart;
  uint32_t* w;
  double* v;
  uint32_t* ck;  // contract keys (dense-row accumulation only; may be null)
};

// Output of the binning pass.
struct Bins {
  int nclasses;
  u64 tmax[kMaxClasses];      // a group goes to the first class with t <= tmax
  uint32_t* list[kMaxClasses];
  // [kMaxClasses + 4]: classes, overflow groups, stream, rank, stash (batches: the two-pass forms)
  uint32_t* count;
  // Dense rows (single contractions with per-segment runs): groups with t >= dense_min go to
  // the stream list (0), the stash list (2) or the rank list (1) by their size and expected
  // repeats (bin_groups_kernel). A streamed group's output bound is B_g itself.
  uint32_t* dense_list[3];    // null when not used; batches: the two-pass kernel's forms
  u64 dense_min;
  u64 stream_cap;
  u64 stash_cap;
  uint32_t* huge_list;        // overflow groups, their table offsets and capacities
  u64* huge_off;
  u64* huge_cap;
  u64* huge_slots;            // total overflow-table slots
  u64* out_cap;               // sum over groups of min(B_g, F_Y): bound on the output size
  uint32_t* status;
};

// Output region of one problem of a batch.
struct BatchOut {
  u64 FY;
  u64 out_cap;
  int32_t* coords;
  double* vals;
  OutPlan op;  // a whole number of 8-byte words (copied word by word)
};
static_assert(sizeof(OutPlan) % 8 == 0, "OutPlan must be a whole number of 8-byte words");

// Positions reserved for outputs that none took.
struct StreamHole {
  u64 pos;
  u64 len;
};

struct GroupArgs {
  const uint32_t* goff;
  GroupedX gx;
  const void* yfk;  // Y free keys in contract-key order: uint32_t when F_Y < 2^32, else u64
  const double* yv;
  u64 FY;
  OutPlan op;
  int32_t* coords;
  double* vals;
  u64 out_cap;
  u64* nz;
  uint32_t* status;
  // Output regions and counters, one per problem (one entry for a single contraction). For
  // batches also the problem of each group and the group's X free key within that problem
  // (both null for a single contraction, where the group index is the X free key).
  const BatchOut* bout;
  u64* bnz;
  const uint32_t* gprob;
  const u64* gfk;
  // Non-null: yuniq[r] = 1 at the first entry r of every Y run whose free keys are all
  // different (run_unique_kernel). A group of one X entry over such a run has one product per
  // output, and the warp kernels write it as a scaled copy of the run without a table.
  const uint8_t* yuniq;
};

// Where one group's outputs go, resolved once per group.
struct OutTarget {
  u64 FY;        // Y free key space of the group's problem
  u64 fx;        // X free key of the group
  u64 zrow;      // output key of the group's row: fX * F_Y
  u64 base;      // first output position reserved for the group
  u64 cap;       // output capacity of the group's problem
  int32_t* coords;
  double* vals;
  u64* counter;  // the problem's output counter (positions are reserved from it)
  uint32_t prob; // problem whose output plan `op` holds (kNoProb before the first group)
  OutPlan op;
  int32_t xc[8]; // split plans: the group's coordinates, its row's X part
};
constexpr uint32_t kNoProb = 0xffffffffu;

// A count only the device knows (launchers then run a full persistent grid).
constexpr uint32_t kCountOnDevice = 0xffffffffu;

struct HugeGroups {
  uint32_t count;             // number of overflow groups, or kCountOnDevice
  const uint32_t* countp;     // device copy of the count, read by the kernel
  const uint32_t* list;
  const u64* off;
  const u64* cap;
  u64* keys;
  double* vals;
};

cudaError_t launch_x_group_scatter(Survivors sv, uint32_t* gcur, GroupedX gx, int64_t max_ns, int sms,
                                   cudaStream_t s);
// entries (may be null) receives the number of grouped X entries.
cudaError_t launch_bin_groups(u64 FX, const uint32_t* goff, const uint32_t* gw, u64 FY, const Bins& b,
                              unsigned* entries, int sms, cudaStream_t s);
// direct: the shared-memory classes may write outputs as keys are first claimed (needs 32-bit
// keys and output positions below 2^32 in every problem). counts: host copies of the class
// counts (b.count), used to size the grids, or null when only the device knows them. depth:
// 0 the default expansion split of the direct CTA tables, 1 half as many products per lane
// per round.
cudaError_t launch_group_classes(const GroupArgs& a, bool wide_keys, bool direct, const Bins& b,
                                 const uint32_t* counts, int sms, cudaStream_t s, int depth = 0);
cudaError_t launch_group_huge(const GroupArgs& a, const HugeGroups& h, bool wide_keys, int sms, cudaStream_t s);

// ------------------------------------------------------------------ batches (batch.cu)
// One problem of a batch as the device kernels see it.
struct BatchProb {
  const int32_t* xc;
  const double* xv;
  const int32_t* yc;
  const double* yv;
  KeyPlan kx, ky;
  u64 koff;   // first contract-key bin of this problem in the concatenated bins
  u64 fxoff;  // offset of this problem's X free keys in the combined group-key space
  u64 FY;
};

// A probing table giving each distinct group key a number: its slot.
struct IdMap {
  u64* keys;  // [mask + 1], kEmpty64 when free
  u64 mask;
};

struct BatchArgs {
  int n;
  const BatchProb* pb;
  const int64_t* xrow;  // [n + 1] row offsets of X in the flattened row space
  const int64_t* yrow;  // [n + 1]
  const u64* fxoff;     // [n + 1]
  int64_t total_x, total_y;
  u64 bins;             // concatenated contract-key bins
  uint32_t* ycnt;
  uint32_t* yoff;       // [bins + 1]
  uint32_t* ycur;
  void* yfk;
  bool key32;
  double* yv;
  Survivors sv;
  u64* P;               // total products
  u64* Pp;              // [n] products per problem
  IdMap idmap;
  uint32_t* gid;        // [total_x] group number (table slot) of each survivor
  uint32_t* gcnt;       // [table size] survivors per group
  uint32_t* goff;       // [table size + 1]
  uint32_t* gcur;       // [table size]
  u64* pcap;            // [n] output bound per problem
  uint32_t* scan_scratch32;
  uint32_t* status;
  uint8_t* yuniq;       // [total_y] or null: runs with all-different free keys (32-bit keys only)
};

cudaError_t launch_batch_prepare(const BatchArgs& ba, int sms, cudaStream_t s);

// Where one run of a captured batch puts its outputs (written by the host before each replay).
struct BatchLayoutArgs {
  unsigned char* out;  // output block: values of every problem, then coordinates
  u64 out_bytes;       // its size
  u64* huge_keys;      // overflow groups' table
  double* huge_vals;
  u64 huge_cap;        // its slots
};
// Places every problem's output region in the run's block from the exact bounds pcap[n]
// (offs: [n + 1] value offsets, then [n + 1] coordinate offsets, in elements), then clears
// the slots of the overflow table this run uses (a grid of its own); flags kStatOutOverflow
// (and places nothing) when the block is too small.
cudaError_t launch_batch_layout(int n, const u64* pcap, const int32_t* oz, BatchOut* bo, const BatchLayoutArgs* args,
                                u64* offs, const u64* huge_slots, uint32_t* huge_count, uint32_t* status, int sms,
                                cudaStream_t s);
cudaError_t launch_batch_group(const BatchArgs& ba, GroupedX gx, const Bins& b, uint32_t* gprob, u64* gfk, int sms,
                               cudaStream_t s);

// Bitmap-row accumulation: each group's outputs are found one free-key segment at a time
// through a bitmap over the segment's free keys. `yoff` are the per-(contract key, segment)
// run offsets; seg is the segment width (a power of two, 64 <= seg <= kDenseSeg). Groups
// with at most dense_stash_cap() products (per segment) may go to the stash kernel, the others
// to the rank kernel.
constexpr uint32_t kDenseSeg = 65536;
constexpr size_t kBitmapSmemPerCta = 112 * 1024;  // two CTAs per SM
uint32_t dense_stash_cap();

// ------------------------------------------------------------------ batches' larger groups (twopass.cu)
// The list (form) of the two-pass kernel for a group of `products` products by `entries` X entries over
// F_Y free keys, or -1 where the group belongs to the hash tables. Accumulation of 3e7 products in groups
// of one size, the tables' time over the two-pass kernel's:
//   form 0, 800 to 8,000 products: even keys 1.2 to 1.8; keys by a Zipf law of exponent 1.0 0.9 to 1.5, of
//     1.5 0.9 to 1.3; all products on 60 keys 0.7 (1,500) to 1.2
//   form 1, 6,000 to 12,000 products: 1.5 to 1.9; 1.0 to 1.1; 0.7; 0.8 to 1.0
//   form 2, 40,000 products, whose tables lie in global memory: 6 to 10; 3.5 to 6; 1.7 to 2.4; 1.4 to 2.2
//   form 1 at 800, 1,500 and 3,000 products over more than 2^16 keys, where half as many groups are in
//     flight: 0.7, 1.0 and 1.4; 0.7, 0.7 and 0.9; 0.5, 0.6 and 0.6; 0.5, 0.5 and 0.6
// A group's skew is not known before it is accumulated: the lines are those of even keys, so that the
// tables take groups of up to 2,048 products over more than 2^16 keys. (2,048 uneven pairs: 78.3 ms with
// this line at 6,144, 77.7 at 2,048; 256 pairs 10.58 and 10.42.)
// The lead falls as even keys repeat, 1.12 to 1.19 at 2 to 4 products per key and 0.96 to 1.14 at 8, where
// the line is drawn. Groups of the 1,024-slot warp tables lose (the batch of 256 pairs: 15.3 against 13.8
// ms with those above 320 products taken in).
__host__ __device__ constexpr int twopass_list(u64 products, uint32_t entries, u64 FY) {
  if (FY > (1u << 18) || products > 49152 || entries > 1024 || products > 4 * FY) return -1;
  if (FY > (1u << 16) && products <= 2048) return -1;
  if (FY <= (1u << 16) && products <= 8192 && entries <= 256) return 0;
  return products <= 16384 && entries <= 512 ? 1 : 2;
}
// counts: as for launch_group_classes.
cudaError_t launch_group_twopass(const GroupArgs& a, const Bins& b, const uint32_t* counts, int sms, cudaStream_t s);

// ------------------------------------------------------------------ streamed groups (stream.cu)
struct StreamArgs {
  StreamHole* holes;    // [stream_max_holes], of fewer than 2^16 positions each
  unsigned* nholes;
  u64* hole_total;
  uint32_t ny_entries;  // entries of Y; the arrays hold one more (stream_dead_key)
  // Set by launch_group_stream: how the Y free key decodes into the output coordinates.
  uint32_t dead;            // stream_dead_key(F_Y)
  uint32_t rsh[4], rmk[4];  // order-4 power-of-two rows: coordinate q has (key >> rsh) & rmk
  int ny;                   // other rows: digits of the Y part, last mode first
  uint32_t ymod[6], ymagic[6], ysh1[6], ysh2[6];
};
uint32_t stream_cap();  // most products of a streamed group
size_t stream_max_holes(uint32_t count, uint32_t nseg);
cudaError_t launch_group_stream(const GroupArgs& a, const uint32_t* yoff, uint32_t nseg, uint32_t seg,
                                const uint32_t* list, uint32_t count, const StreamArgs& sa, int sms, cudaStream_t s);
// One round of filling the holes: moves entries from the last *hole_total of the *reserved positions
// into the holes before them; after the rounds that cover all *hole_total positions, the outputs are
// the first *reserved - *hole_total. Both counts are read on the device.
struct HoleRound {
  u64 at;         // the window of those positions that this round moves entries from: [at, at + win);
  u64 win;        // the rounds start at 0 and follow one another (part of it may lie past the end)
  u64 base;       // entries moved by the rounds before (counters2[1])
  uint32_t* dst;  // [win] scratch
};
// holes: rewritten by the first round. counters2: zeroed before the first round; destinations and
// entries moved.
cudaError_t launch_hole_fill(StreamHole* holes, const unsigned* nholes, const u64* reserved, const u64* hole_total,
                             const HoleRound& rd, u64* counters2, int32_t* coords, double* vals, int oz,
                             uint32_t* status, int sms, cudaStream_t s);

// Lane-private dense rows for output rows of at most 64 free keys (FY <= 64, 32-bit Y free
// keys): a warp or a CTA per group g in [0, ngroups) (empty groups skipped), outputs in key order.
// products and entries: what they hold.
cudaError_t launch_group_lanerow(const GroupArgs& a, u64 ngroups, uint32_t FY, u64 products, u64 entries, int sms,
                                 cudaStream_t s);
cudaError_t launch_group_dense(const GroupArgs& a, const uint32_t* yoff, uint32_t nseg, uint32_t seg,
                               const uint32_t* stash_list, uint32_t stash_count, const uint32_t* rank_list,
                               uint32_t rank_count, int sms, cudaStream_t s);

}  // namespace stc
