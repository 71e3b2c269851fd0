// Hive hash table kernels for GB300 (sm_103a).
//
// Layout (Section III-A/B of the paper): a bucket is S packed 64-bit words
// (value << 32 | key), S = 32 (256 bytes) or 16 (128 bytes), aligned to its
// size; S one-byte slot tags per bucket (0 = free slot), which are the free
// mask and a filter for lookups; a 32-bit lock per bucket used only by
// eviction; an overflow stash of packed words.  The empty word is all ones
// (key 0xFFFFFFFF).
//
// Kernels:
//   k_ops<MODE,S>  bulk find / insert (steps 1-2) / erase / mixed batch, one op
//                  per lane: both candidate buckets' tags in one round trip,
//                  then the words whose tag matches the key's.  A new key
//                  claims a slot with one CAS on a tag word (WABC, Section
//                  III-E).
//   k_overflow<S>  steps 3-4 for inserts whose two buckets were full: warp per
//                  item, bounded cuckoo eviction under the bucket lock
//                  (Algorithm 3), then the stash.
//   k_maint<S>     stash maintenance: reinsert stash words into buckets that
//                  have room, compact, sort by key (lookups binary-search it).
//   k_split<S>     linear-hashing expansion, warp per bucket pair (Section IV-C1).
//   k_merge<S>     linear-hashing contraction, warp per bucket pair (IV-C2).
//   k_fused<S>     a mixed batch as one concurrent kernel (bucket versions make
//                  lookups safe against eviction chains in flight).
//   k_multi_*      the same phases over many tables in one launch each.
#include <cuda_runtime.h>
#include <stdint.h>

#include "hive_internal.h"
#include "hive_device.cuh"
#include "hive_tags.cuh"

namespace hive {
namespace {

constexpr int kOpsThreads = 256;
#ifndef HIVE_MULTI_MIN_BLOCKS
#define HIVE_MULTI_MIN_BLOCKS 4
#endif
constexpr int kOvfThreads = 256;
constexpr int kMaintThreads = 1024;
constexpr unsigned kMaintSmemWords = 8192;  // 64 KB of words sorted in shared memory

// ----------------------------------------------------------------------------
// Hashing and addressing
// ----------------------------------------------------------------------------

__device__ __forceinline__ uint64_t pack(uint32_t k, uint32_t v) {
  return (static_cast<uint64_t>(v) << 32) | k;
}
__device__ __forceinline__ uint32_t key_of(uint64_t w) { return static_cast<uint32_t>(w); }
__device__ __forceinline__ uint32_t val_of(uint64_t w) { return static_cast<uint32_t>(w >> 32); }

// The two candidate buckets of a key.
struct Cand {
  uint32_t b1, b2;
};
__device__ __forceinline__ Cand cand_of(const View& v, uint32_t key) {
  return Cand{lh_bucket(bithash1(key), v.M, v.p), lh_bucket(bithash2(key), v.M, v.p)};
}

template <int S, bool RO>
__device__ __forceinline__ TagVec<S> ld_tags(const View& v, uint32_t b) {
  return ld_tags_at<S, RO>(v.tags, b);
}

// ----------------------------------------------------------------------------
// Memory access helpers
// ----------------------------------------------------------------------------

// Two words of a bucket while other warps may be writing the table.
__device__ __forceinline__ void ld_frag(const uint64_t* p, uint64_t& a, uint64_t& b) {
  asm volatile("ld.relaxed.gpu.global.L1::no_allocate.v2.u64 {%0, %1}, [%2];"
               : "=l"(a), "=l"(b)
               : "l"(p)
               : "memory");
}
// One slot's word; RO as for ld_tags, `keep` as in View::keep_words.
template <bool RO>
__device__ __forceinline__ uint64_t ld_word(const uint64_t* p, bool keep) {
  uint64_t r;
  const uint64_t pol = keep ? policy_keep() : policy_pass();
  if constexpr (RO)
    asm("ld.global.nc.L2::cache_hint.b64 %0, [%1], %2;" : "=l"(r) : "l"(p), "l"(pol));
  else
    asm volatile("ld.relaxed.gpu.global.L2::cache_hint.b64 %0, [%1], %2;"
                 : "=l"(r)
                 : "l"(p), "l"(pol)
                 : "memory");
  return r;
}

// ----------------------------------------------------------------------------
// Slot claims (WABC, Section III-E / Algorithm 2)
// ----------------------------------------------------------------------------

// A claim owns its slot by the non-zero tag and publishes `word` with a plain
// store: nothing else writes a slot while it is EMPTY (erases, replaces and
// swaps expect a non-EMPTY word).
template <int S>
__device__ __forceinline__ bool publish(const View& v, uint32_t b, uint32_t slot, uint64_t word) {
  if (slot >= S) return false;
  st_relaxed64(v.buckets + static_cast<uint64_t>(b) * S + slot, word);
  return true;
}
template <int S>
__device__ __forceinline__ bool claim_in_word(const View& v, uint32_t b, uint32_t q, uint32_t j,
                                              uint32_t cur, uint32_t tag, uint64_t word) {
  return publish<S>(v, b, claim_tag<S>(v.tags, b, q, j, cur, tag), word);
}
template <int S>
__device__ __forceinline__ bool claim_from(const View& v, uint32_t b, const TagVec<S>& t,
                                           uint32_t fm, uint64_t word, uint32_t rot) {
  return publish<S>(v, b, claim_among<S>(v.tags, b, t, fm, tag_of(key_of(word)), rot), word);
}

// The same with the tags read here.
template <int S>
__device__ __forceinline__ bool claim_bucket(const View& v, uint32_t b, uint64_t word,
                                             uint32_t rot) {
  const TagVec<S> t = ld_tags<S, false>(v, b);
  return claim_from<S>(v, b, t, free_slots<S>(t), word, rot);
}

// Step 2 for an absent key, with the tags of both candidate buckets at hand:
// claims a slot in the bucket the placement rule prefers, else in the other
// (with its tags read again: rare, and keeping both sets costs registers).
// Returns the slot, or S, and its bucket in `b`; the word is not stored yet.
template <int S>
__device__ __forceinline__ uint32_t place_slot(const View& v, uint32_t b1, uint32_t b2,
                                               const TagVec<S>& t1, const TagVec<S>& t2,
                                               uint32_t key, uint32_t& b) {
  const uint32_t m1 = free_slots<S>(t1), m2 = free_slots<S>(t2);
  const uint32_t f1 = __popc(m1), f2 = __popc(m2);
  const bool first1 = v.placement ? (f1 > 0) : (f1 >= f2);
  const uint32_t rot = claim_rot(key), tag = tag_of(key);
  TagVec<S> t;
#pragma unroll
  for (int q = 0; q < S / 4; ++q) t.w[q] = first1 ? t1.w[q] : t2.w[q];
  b = first1 ? b1 : b2;
  const uint32_t slot = claim_among<S>(v.tags, b, t, first1 ? m1 : m2, tag, rot);
  // S: filled up meanwhile, or no room in either when the tags were read
  if (slot < S || b1 == b2 || (first1 ? f2 : f1) == 0) return slot;
  b = first1 ? b2 : b1;
  t = ld_tags<S, false>(v, b);
  return claim_among<S>(v.tags, b, t, free_slots<S>(t), tag, rot);
}
template <int S>
__device__ __forceinline__ bool place_from(const View& v, uint32_t b1, uint32_t b2,
                                           const TagVec<S>& t1, const TagVec<S>& t2,
                                           uint64_t word) {
  uint32_t b;
  const uint32_t slot = place_slot<S>(v, b1, b2, t1, t2, key_of(word), b);
  return publish<S>(v, b, slot, word);
}
template <int S>
__device__ __forceinline__ bool place_new(const View& v, uint32_t b1, uint32_t b2, uint64_t word) {
  const TagVec<S> t1 = ld_tags<S, false>(v, b1);
  const TagVec<S> t2 = ld_tags<S, false>(v, b2);
  return place_from<S>(v, b1, b2, t1, t2, word);
}

// Frees a slot whose word (of key `key`) this thread has just emptied: called
// once the CAS to EMPTY has returned, so a claimer that sees the zero tag
// finds the slot EMPTY.
template <int S>
__device__ __forceinline__ void free_tag(const View& v, uint32_t b, uint32_t slot, uint32_t key) {
  xor_tag<S>(v.tags, b, slot, tag_of(key));
}
// Slot's word changed from a key with tag t0 to one with tag t1.
template <int S>
__device__ __forceinline__ void swap_tag(const View& v, uint32_t b, uint32_t slot, uint32_t k0,
                                         uint32_t k1) {
  xor_tag<S>(v.tags, b, slot, tag_of(k0) ^ tag_of(k1));
}

// The bucket lock serialises evictors of one bucket (Algorithm 3).  The word
// swap it protects is an L2 atomic whose result has returned before the
// unlock; the tag change of the swap is ordered before the unlock by the
// fence in unlock_swapped().
__device__ __forceinline__ bool lock_bucket(const View& v, uint32_t b) {
  for (uint32_t t = 0; t < v.lock_spin_limit; ++t) {
    if (atomicCAS(v.locks + b, 0u, 1u) == 0u) return true;
    __nanosleep(64);
  }
  return false;
}
__device__ __forceinline__ void unlock_bucket(const View& v, uint32_t b) {
  atomicExch(v.locks + b, 0u);
}
__device__ __forceinline__ void unlock_swapped(const View& v, uint32_t b) {
  fence_acq_rel_gpu();
  atomicExch(v.locks + b, 0u);
}

// Stash binary search over the sorted key prefix.
__device__ __forceinline__ bool stash_find(const View& v, uint32_t stash_n, uint32_t key,
                                           uint32_t& pos) {
  uint32_t lo = 0, hi = stash_n;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (__ldg(v.stash_keys + mid) < key)
      lo = mid + 1;
    else
      hi = mid;
  }
  pos = lo;
  return lo < stash_n && __ldg(v.stash_keys + lo) == key;
}

// ----------------------------------------------------------------------------
// Bulk op kernel
// ----------------------------------------------------------------------------

struct LaneCounters {
  int size_delta = 0;
  unsigned replaced = 0, claimed = 0, overflowed = 0, stash_lookups = 0;
  unsigned probes = 0;  // buckets examined
  bool reserved = false, contract = false;
};

// An insert examines both candidate buckets of every live op, and every live
// op ends replaced, claimed or handed on: counting the probes once at the end
// keeps a counter out of the loop.
__device__ __forceinline__ void count_insert_probes(LaneCounters& cnt) {
  cnt.probes = 2 * (cnt.replaced + cnt.claimed + cnt.overflowed);
}

// ---- Shared-memory staging of bucket reads ----
//
// Tables of 32-slot buckets created with a stage_wait_limit probe whole
// buckets instead of tags: the buckets of a warp's 32 ops are copied into its
// 8 KB of shared memory with one bulk copy (TMA) each, counted by the warp's
// mbarrier, and each lane scans its own op's bucket.  A barrier wait that
// does not end within View::stage_spin_limit tries raises the table's sticky
// TIMEOUT error, marks the stage dead and redoes the round by tags; before
// the warp exits it waits up to kMbarSpinLimit tries for the copies still in
// flight.
constexpr uint32_t kMbarSpinLimit = 1u << 22;
__host__ __device__ constexpr int stage_warp_words(int S) { return 2 + 32 * S; }
__host__ __device__ constexpr size_t stage_smem(int S, int threads = kOpsThreads) {
  return static_cast<size_t>(threads / 32) * 8u * stage_warp_words(S);
}

struct Stage {
  uint64_t* bar;   // mbarrier
  uint64_t* buf;   // 32 S words, 16-byte aligned
  uint32_t phase;  // parity of the barrier's current phase
  bool dead;       // a wait gave up: copies may still land, the buffer is not reused
};

// Sets up the calling warp's stage in the kernel's dynamic shared memory
// (`stride` words per warp: its barrier, then its staging words).
__device__ __forceinline__ Stage stage_init(uint64_t* smem, int warp_in_block, int lane,
                                            int stride) {
  Stage sg;
  uint64_t* base = smem + static_cast<size_t>(warp_in_block) * stride;
  sg.bar = base;
  sg.buf = base + 2;
  sg.phase = 0;
  sg.dead = false;
  if (lane == 0) mbar_init(sg.bar, 1);
  __syncwarp();
  return sg;
}

// Before a warp exits: a stage whose wait gave up may still receive bytes;
// wait (bounded) for them so that no copy lands after the block has left.
__device__ __forceinline__ void stage_drain(Stage& sg) {
  if (!sg.dead) return;
  bool ok = false;
  for (uint32_t it = 0; it < kMbarSpinLimit && !ok; ++it) ok = mbar_try_wait(sg.bar, sg.phase ^ 1u);
}

// One staged round (warp-wide): op j (bit j of `need`) copies bucket x of
// lane j to buffer bucket j, then the warp waits (bounded).  A limit below 16
// polls without suspending (mbarrier.test_wait), so that a test can make the
// wait give up while the copies are certainly in flight.  Returns false, with
// the stage marked dead and the error raised, if the wait gave up.
template <int S>
__device__ __forceinline__ bool stage_round(const View& v, Stage& sg, unsigned need, uint32_t x,
                                            int lane) {
  constexpr uint32_t kBucketBytes = S * 8u;
  fence_proxy_async();  // earlier fragment reads of the buffer come before the new copies
  __syncwarp();
  if (lane == 0) mbar_arrive_expect_tx(sg.bar, __popc(need) * kBucketBytes);
  __syncwarp();
  if ((need >> lane) & 1u)
    bulk_g2s(sg.buf + lane * S, v.buckets + static_cast<uint64_t>(x) * S, kBucketBytes, sg.bar);
  bool ok = false;
  if (v.stage_spin_limit < 16) {
    for (uint32_t it = 0; it < v.stage_spin_limit && !ok; ++it) ok = mbar_test_wait(sg.bar, sg.phase);
  } else {
    for (uint32_t it = 0; it < v.stage_spin_limit && !ok; ++it) ok = mbar_try_wait(sg.bar, sg.phase);
  }
  sg.phase ^= 1u;
  if (__any_sync(kFull, !ok)) {
    sg.dead = true;
    if (lane == 0) atomicOr(&v.ctrl->err, kErrTimeout);
    return false;
  }
  return true;
}

// Where an op's key was found.
struct Hit {
  uint64_t word;
  uint32_t b, slot;
  bool ok;
};

// The op's staged bucket `myb`, scanned by its own lane with swizzled 16-byte
// reads (the eight lanes of a shared-memory wavefront read eight different
// bank groups).
template <int S>
__device__ __forceinline__ void scan_staged(const uint64_t* sbuf, int lane, uint32_t myb,
                                            uint32_t key, Hit& h) {
  constexpr int NP = S / 2;
  const uint64_t* B = sbuf + lane * S;
  int ms = -1;
#pragma unroll 8
  for (int k = 0; k < NP; ++k) {
    const int f = (k + lane) & (NP - 1);
    uint64_t a, b;
    lds_frag(B + 2 * f, a, b);
    if (key_of(a) == key) ms = 2 * f;
    if (key_of(b) == key) ms = 2 * f + 1;
  }
  if (ms >= 0) h = Hit{B[ms], myb, static_cast<uint32_t>(ms), true};
}

// The slots `m1` of bucket b1, then `m2` of b2, whose tags match the key:
// reads their words until one holds the key, starting where the key's own
// claim would have (so the slot that holds it tends to come before a false
// match).
template <int S, bool RO, class F>
__device__ __forceinline__ void check_words(const View& v, uint32_t b1, uint32_t b2, uint32_t m1,
                                            uint32_t m2, uint32_t key, Hit& h, bool keep,
                                            F on_hit) {
  const uint32_t rot = claim_rot(key);
  while (m1 | m2) {
    const bool in1 = m1 != 0;
    const uint32_t b = in1 ? b1 : b2;
    const uint32_t p = pick_slot(in1 ? m1 : m2, rot);
    const uint32_t slot = slot_of(p);
    const uint64_t w = ld_word<RO>(v.buckets + static_cast<uint64_t>(b) * S + slot, keep);
    if (key_of(w) == key) {
      h = Hit{w, b, slot, true};
      on_hit();
      return;
    }
    if (in1)
      m1 &= ~(1u << p);
    else
      m2 &= ~(1u << p);
  }
}

template <int S, bool RO>
__device__ __forceinline__ void check_words(const View& v, uint32_t b1, uint32_t b2, uint32_t m1,
                                            uint32_t m2, uint32_t key, Hit& h, bool keep) {
  check_words<S, RO>(v, b1, b2, m1, m2, key, h, keep, [] {});
}

// An erase or replace CAS issued by a probe, checked only at the end of the
// chunk, so that its round trip overlaps the claims after it (an op updates
// at most one slot, so one record per lane).
struct PendCas {
  uint64_t cur, old;
  uint32_t b, slot, kind;  // kind: 0 none, 1 erase, 2 replace
};

template <int S>
__device__ __forceinline__ void resolve_cas(const View& v, const PendCas& pc, LaneCounters& cnt) {
  if (pc.kind == 0) return;
  const bool ok = pc.old == pc.cur;
  if (pc.kind == 1) {
    // Algorithm 4: the slot is published as free once the CAS has emptied it
    if (ok) {
      free_tag<S>(v, pc.b, pc.slot, key_of(pc.cur));
      cnt.size_delta -= 1;
    } else {
      cnt.contract = true;
    }
  } else {
    if (ok)
      cnt.replaced += 1;
    else
      cnt.contract = true;
  }
}

// Acts on a hit: a find takes the value; an erase or replace issues its CAS
// (Algorithm 4 / Algorithm 1).
template <int MODE, int S>
__device__ __forceinline__ void act_on(const View& v, const Hit& h, uint32_t key, uint32_t val,
                                       uint32_t op, uint8_t& st, uint32_t& outv, PendCas& pc) {
  const uint32_t opk = MODE == kModeMixed
                           ? op
                           : (MODE == kModeFind ? OP_FIND
                                                : (MODE == kModeErase ? OP_ERASE : OP_INSERT));
  if (opk == OP_FIND) {
    outv = val_of(h.word);
    st = ST_FOUND;
  } else {
    uint64_t* sp = v.buckets + static_cast<uint64_t>(h.b) * S + h.slot;
    st = opk == OP_ERASE ? ST_ERASED : ST_REPLACED;
    pc.old = atomicCAS(ull(sp), h.word, opk == OP_ERASE ? kEmptyWord : pack(key, val));
    pc.cur = h.word;
    pc.b = h.b;
    pc.slot = h.slot;
    pc.kind = opk == OP_ERASE ? 1u : 2u;
  }
}

// Op arrays of one batch, or of one segment of a multi-table batch.
struct OpPtrs {
  const uint8_t* ops;
  const uint32_t* keys;
  const uint32_t* vals;
  uint32_t* vals_out;
  uint8_t* found;
  uint8_t* status;
};

// Adds a warp's counters to the table of `v` and clears them: one atomic per
// non-zero counter.
__device__ __forceinline__ void flush_counters(const View& v, LaneCounters& cnt, int lane) {
  const int sd = __reduce_add_sync(kFull, static_cast<unsigned>(cnt.size_delta));
  const unsigned rp = __reduce_add_sync(kFull, cnt.replaced);
  const unsigned cl = __reduce_add_sync(kFull, cnt.claimed);
  const unsigned of = __reduce_add_sync(kFull, cnt.overflowed);
  const unsigned rs = __ballot_sync(kFull, cnt.reserved);
  const unsigned ct = __ballot_sync(kFull, cnt.contract);
  const unsigned sl = __reduce_add_sync(kFull, cnt.stash_lookups);
  const unsigned pr = __reduce_add_sync(kFull, cnt.probes);
  if (lane == 0) {
    if (pr) atomicAdd(&v.ctrl->stats[kStProbes], static_cast<unsigned long long>(pr));
    if (sl) atomicAdd(&v.ctrl->stats[kStStashLookups], static_cast<unsigned long long>(sl));
    if (sd) atomicAdd(&v.ctrl->size, static_cast<unsigned long long>(static_cast<long long>(sd)));
    if (rp) atomicAdd(&v.ctrl->stats[kStReplaced], static_cast<unsigned long long>(rp));
    if (cl) atomicAdd(&v.ctrl->stats[kStClaimedFast], static_cast<unsigned long long>(cl));
    if (of) atomicAdd(&v.ctrl->stats[kStOverflowed], static_cast<unsigned long long>(of));
    if (rs) atomicOr(&v.ctrl->err, kErrReserved);
    if (ct) atomicOr(&v.ctrl->err, kErrContract);
  }
  cnt = LaneCounters();
}

// The same for every warp of a block at once, with one atomic per counter
// and block: the counters live in one control block, and an atomic per warp
// and counter at the end of a launch of thousands of warps queued in L2 for
// tens of microseconds.  Every thread of the block calls it; `scratch` is
// 8 free shared-memory words of the calling warp, and warp w's are at
// base + w * stride.
__device__ __forceinline__ void flush_counters_block(const View& v, LaneCounters& cnt, int lane,
                                                     uint64_t* scratch, const uint64_t* base,
                                                     int stride) {
  const int sd = __reduce_add_sync(kFull, static_cast<unsigned>(cnt.size_delta));
  const unsigned rp = __reduce_add_sync(kFull, cnt.replaced);
  const unsigned cl = __reduce_add_sync(kFull, cnt.claimed);
  const unsigned of = __reduce_add_sync(kFull, cnt.overflowed);
  const unsigned sl = __reduce_add_sync(kFull, cnt.stash_lookups);
  const unsigned pr = __reduce_add_sync(kFull, cnt.probes);
  const unsigned rs = __ballot_sync(kFull, cnt.reserved);
  const unsigned ct = __ballot_sync(kFull, cnt.contract);
  __syncwarp();
  if (lane == 0) {
    scratch[0] = pr;
    scratch[1] = sl;
    scratch[2] = static_cast<uint64_t>(static_cast<int64_t>(sd));
    scratch[3] = rp;
    scratch[4] = cl;
    scratch[5] = of;
    scratch[6] = rs ? 1u : 0u;
    scratch[7] = ct ? 1u : 0u;
  }
  __syncthreads();
  const int f = threadIdx.x;
  if (f < 8) {
    uint64_t sum = 0;
    for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) sum += base[w * stride + f];
    if (sum) {
      switch (f) {
        case 0: atomicAdd(&v.ctrl->stats[kStProbes], static_cast<unsigned long long>(sum)); break;
        case 1: atomicAdd(&v.ctrl->stats[kStStashLookups], static_cast<unsigned long long>(sum)); break;
        case 2: atomicAdd(&v.ctrl->size, static_cast<unsigned long long>(sum)); break;
        case 3: atomicAdd(&v.ctrl->stats[kStReplaced], static_cast<unsigned long long>(sum)); break;
        case 4: atomicAdd(&v.ctrl->stats[kStClaimedFast], static_cast<unsigned long long>(sum)); break;
        case 5: atomicAdd(&v.ctrl->stats[kStOverflowed], static_cast<unsigned long long>(sum)); break;
        case 6: atomicOr(&v.ctrl->err, kErrReserved); break;
        default: atomicOr(&v.ctrl->err, kErrContract); break;
      }
    }
  }
  cnt = LaneCounters();
}

// One op's inputs (op code, key, value).
struct OpIn {
  uint32_t op, key, val;
};

template <int MODE>
__device__ __forceinline__ OpIn load_in(const OpPtrs& a, uint32_t c, uint64_t n, int lane) {
  constexpr bool kIns = (MODE == kModeInsert || MODE == kModeMixed);
  const uint32_t i = (c << 5) + lane;
  const bool valid = i < n;
  OpIn in;
  in.op = OP_FIND;
  if (MODE == kModeMixed)
    in.op = valid ? static_cast<uint32_t>(__ldcs(a.ops + i)) : OP_FIND;
  else if (MODE == kModeInsert)
    in.op = OP_INSERT;
  else if (MODE == kModeErase)
    in.op = OP_ERASE;
  if (in.op > OP_ERASE) in.op = OP_FIND;  // unknown op codes read only
  in.key = valid ? __ldcs(a.keys + i) : kEmptyKey;
  in.val = (kIns && valid && in.op == OP_INSERT && a.vals) ? __ldcs(a.vals + i) : 0u;
  return in;
}

// List appends at a high rate go through a per-warp shared-memory buffer: a
// warp gathers entries over several rounds and reserves list space for all it
// holds with one atomicAdd when the next round's entries would not fit.  One
// counter serves the whole list; an atomicAdd on that one word per warp round
// queued behind each other in L2 and held up every warp's memory pipeline.
// (The bulk kernel's own eviction hand-off is rare enough to append directly.)
// A buffer of `cap` entries takes 2 * cap shared-memory words: cap packed
// words, then cap op indices and cap segment tags (u32).
struct OvfBuf {
  uint64_t* words;
  uint32_t* idx;
  uint32_t* seg;
  uint32_t n;       // entries held (warp-uniform)
  uint32_t cap;
};

__device__ __forceinline__ OvfBuf ovf_buf_init(uint64_t* region, uint32_t cap) {
  OvfBuf ob;
  ob.words = region;
  ob.idx = reinterpret_cast<uint32_t*>(region + cap);
  ob.seg = ob.idx + cap;
  ob.n = 0;
  ob.cap = cap;
  return ob;
}

// Moves every buffered entry to the list (warp-wide).
__device__ __forceinline__ void ovf_flush(const List& ovf, OvfBuf& ob, int lane) {
  if (!ob.n) return;
  __syncwarp();
  unsigned base = 0;
  if (lane == 0) base = atomicAdd(ovf.count, ob.n);
  base = __shfl_sync(kFull, base, 0);
  for (uint32_t j = lane; j < ob.n; j += 32) {
    ovf.words[base + j] = ob.words[j];
    ovf.idx[base + j] = ob.idx[j];
    if (ovf.seg) ovf.seg[base + j] = ob.seg[j];
  }
  __syncwarp();
  ob.n = 0;
}

// Adds one round's entries (lanes with `put`) to the buffer, flushing first
// if they would not fit.
__device__ __forceinline__ void ovf_put(const List& ovf, OvfBuf& ob, int lane, bool put,
                                        uint64_t word, uint32_t idx, uint32_t seg) {
  const unsigned om = __ballot_sync(kFull, put);
  if (!om) return;
  if (ob.n + __popc(om) > ob.cap) ovf_flush(ovf, ob, lane);
  if (put) {
    const unsigned r = ob.n + __popc(om & ((1u << lane) - 1u));
    ob.words[r] = word;
    ob.idx[r] = idx;
    ob.seg[r] = seg;
  }
  ob.n += __popc(om);
}

// The final flush of every warp of a block at once: one atomicAdd reserves
// the list space of the whole block.  Every thread of the block calls it.
__device__ __forceinline__ void ovf_flush_block(const List& ovf, OvfBuf& ob, int lane) {
  __shared__ unsigned warp_n[32];
  __shared__ unsigned block_base;
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (lane == 0) warp_n[w] = ob.n;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned tot = 0;
    for (int k = 0; k < nw; ++k) tot += warp_n[k];
    block_base = tot ? atomicAdd(ovf.count, tot) : 0u;
  }
  __syncthreads();
  unsigned base = block_base;
  for (int k = 0; k < w; ++k) base += warp_n[k];
  for (uint32_t j = lane; j < ob.n; j += 32) {
    ovf.words[base + j] = ob.words[j];
    ovf.idx[base + j] = ob.idx[j];
    if (ovf.seg) ovf.seg[base + j] = ob.seg[j];
  }
  __syncwarp();
  ob.n = 0;
}

// Appends the lanes' items with `put` to an eviction list (warp-wide, one atomic).
__device__ __forceinline__ void list_append(const List& l, int lane, bool put, uint64_t word,
                                            uint32_t idx, uint32_t seg) {
  const unsigned m = __ballot_sync(kFull, put);
  if (!m) return;
  const int leader = __ffs(m) - 1;
  unsigned base = 0;
  if (lane == leader) base = atomicAdd(l.count, static_cast<unsigned>(__popc(m)));
  base = __shfl_sync(kFull, base, leader);
  if (put) {
    const unsigned r = base + __popc(m & ((1u << lane) - 1u));
    l.words[r] = word;
    l.idx[r] = idx;
    if (l.seg) l.seg[r] = seg;
  }
}

// A warp's queue of new keys of a mixed batch, in shared memory.  In a batch
// of several chunks per warp the new keys of each (a quarter to a half of the
// ops) wait here, and 32 at a time claim their slots with every lane at work;
// claiming chunk by chunk took as many instructions for a third of the lanes
// (256 tables, 4 M ops: 188 -> 180 us per step).
// Their status is written when they are queued (INSERTED; only a full table
// changes it).  `n` is warp-uniform.
constexpr uint32_t kNewQ = 64;
struct NewQ {
  uint64_t* words;
  uint32_t* idx;
  uint32_t n;
};
constexpr int kNewQWords = kNewQ + kNewQ / 2;
__device__ __forceinline__ NewQ new_q(uint64_t* mine) {
  return NewQ{mine, reinterpret_cast<uint32_t*>(mine + kNewQ), 0};
}

// Claims for the first min(n, 32) queued keys (warp-wide); the rest move to
// the front.  Keys whose two buckets are full go to the eviction list.
template <int S>
__device__ __forceinline__ void claim_queued(const View& v, NewQ& q, const List& ovf, uint32_t seg,
                                             LaneCounters& cnt, int lane) {
  __syncwarp();
  const uint32_t m = q.n < 32 ? q.n : 32u;
  const bool has = static_cast<uint32_t>(lane) < m;
  const uint64_t word = has ? q.words[lane] : kEmptyWord;
  const uint32_t idx = has ? q.idx[lane] : kNoOp;
  const uint32_t rest = q.n - m;
  uint64_t mw = 0;
  uint32_t mi = 0;
  if (static_cast<uint32_t>(lane) < rest) {
    mw = q.words[32 + lane];
    mi = q.idx[32 + lane];
  }
  __syncwarp();
  if (static_cast<uint32_t>(lane) < rest) {
    q.words[lane] = mw;
    q.idx[lane] = mi;
  }
  q.n = rest;
  bool to_ovf = false;
  if (has) {
    const Cand cd = cand_of(v, key_of(word));
    if (place_new<S>(v, cd.b1, cd.b2, word)) {
      cnt.size_delta += 1;
      cnt.claimed += 1;
    } else {
      to_ovf = true;
      cnt.overflowed += 1;
    }
  }
  list_append(ovf, lane, to_ovf, word, idx, seg);
}

// Ops [32c, 32c + 32) of a batch of n ops on the table of `v`, one op per
// lane.  Full-bucket inserts go to the overflow list, tagged with `seg` when
// the list keeps tags.  `pre` holds the chunk's inputs when the caller loaded
// them ahead.
// DEFER (mixed batches): inserts of absent keys do not claim here.  They join
// the list through the warp's buffer `ob`, and k_claim places them once every
// find, erase and replace of the batch has run; their status is written here
// already (INSERTED, which only a full table changes).  With a queue `q` (and
// not DEFER) they wait there instead.
template <int MODE, int S, bool DEFER = false>
__device__ __forceinline__ void run_chunk(const View& v, uint32_t stash_n, const OpPtrs a,
                                          uint32_t c, uint64_t n, const List ovf, uint32_t seg,
                                          LaneCounters& cnt, int lane, Stage* sg = nullptr,
                                          const OpIn* pre = nullptr, OvfBuf* ob = nullptr,
                                          NewQ* q = nullptr) {
  constexpr bool kIns = (MODE == kModeInsert || MODE == kModeMixed);
  constexpr bool kClaim = kIns && !DEFER;
  constexpr bool kRO = MODE == kModeFind;
  const uint32_t i = (c << 5) + lane;
  const bool valid = i < n;
  const OpIn in = pre ? *pre : load_in<MODE>(a, c, n, lane);
  const uint32_t op = in.op, key = in.key, val = in.val;
  const bool reserved = valid && key >= kReservedKeyMin;
  const bool live = valid && !reserved;
  cnt.reserved |= reserved;

  const Cand cd = cand_of(v, key);
  const uint32_t b1 = cd.b1, b2 = cd.b2;
  uint8_t st = reserved ? ST_RESERVED : ST_NOT_FOUND;
  uint32_t outv = 0;
  PendCas pc{0, 0, 0, 0, 0};
  Hit h{0, 0, 0, false};
  TagVec<S> t1, t2;
  bool have_tags = false, acted = false;

  bool probed = false;
  if (sg && !sg->dead) {
    // whole buckets, staged: the BitHash1 bucket, then the BitHash2 bucket
    // of the ops still open
    unsigned need = __ballot_sync(kFull, live);
    probed = need == 0 || stage_round<S>(v, *sg, need, b1, lane);
    if (probed) {
      if (live) scan_staged<S>(sg->buf, lane, b1, key, h);
      if (MODE != kModeInsert) cnt.probes += live;
      need = __ballot_sync(kFull, live && !h.ok);
      probed = need == 0 || stage_round<S>(v, *sg, need, b2, lane);
      if (probed) {
        if (MODE != kModeInsert) cnt.probes += live && !h.ok;
        if (live && !h.ok) scan_staged<S>(sg->buf, lane, b2, key, h);
      }
    }
  }
  if (!probed) {
    // by tags: both buckets' tags in one round trip, then the matching words
    if (live) {
      t1 = ld_tags<S, kRO>(v, b1);
      t2 = ld_tags<S, kRO>(v, b2);
      have_tags = true;
      const uint32_t t4 = tag_of(key) * 0x01010101u;
      const uint32_t m1 = tag_match<S>(t1, t4);
      const uint32_t m2 = b2 != b1 ? tag_match<S>(t2, t4) : 0u;
      // an erase or replace issues its CAS at once, while the word's line is in L2
      check_words<S, kRO>(v, b1, b2, m1, m2, key, h, v.keep_words,
                          [&] { act_on<MODE, S>(v, h, key, val, op, st, outv, pc); });
      acted = h.ok;
    }
    if (MODE != kModeInsert) {  // insert batches: see count_insert_probes()
      cnt.probes += live;
      cnt.probes += live && (!h.ok || h.b != b1);
    }
  }
  bool done = !live || h.ok;
  if (h.ok && !acted) act_on<MODE, S>(v, h, key, val, op, st, outv, pc);

  // The stash (Section IV-A step 4) holds keys that found no bucket room.
  if (!done && stash_n) {
    uint32_t pos;
    cnt.stash_lookups += 1;
    if (stash_find(v, stash_n, key, pos)) {
      uint64_t* sp = v.stash_kv + pos;
      const uint64_t w = ld_relaxed64(sp);
      if (key_of(w) == key) {
        done = true;
        if (op == OP_FIND) {
          outv = val_of(w);
          st = ST_FOUND;
        } else if (op == OP_ERASE) {
          st = ST_ERASED;
          if (atomicCAS(ull(sp), w, kEmptyWord) == w) {
            cnt.size_delta -= 1;
            atomicExch(&v.ctrl->stash_dirty, 1u);
          } else {
            cnt.contract = true;
          }
        } else {
          st = ST_REPLACED;
          if (atomicCAS(ull(sp), w, pack(key, val)) == w) cnt.replaced += 1; else cnt.contract = true;
        }
      }
    }
  }

  // Step 2: claim-then-commit for absent keys.
  bool to_ovf = false;
  bool queued = false;
  if (DEFER && !done && op == OP_INSERT) {
    to_ovf = true;  // k_claim places it
    st = ST_INSERTED;
  } else if (kClaim && MODE == kModeMixed && q && !done && op == OP_INSERT) {
    queued = true;
    st = ST_INSERTED;
  } else if (kClaim && !done && op == OP_INSERT) {
    if (!have_tags) {
      t1 = ld_tags<S, false>(v, b1);
      t2 = ld_tags<S, false>(v, b2);
    }
    if (place_from<S>(v, b1, b2, t1, t2, pack(key, val))) {
      done = true;
      st = ST_INSERTED;
      cnt.size_delta += 1;
      cnt.claimed += 1;
    } else {
      to_ovf = true;
      cnt.overflowed += 1;
    }
  }

  resolve_cas<S>(v, pc, cnt);

  // Hand full-bucket inserts to the eviction kernel (steps 3-4).
  if constexpr (DEFER)
    ovf_put(ovf, *ob, lane, to_ovf, pack(key, val), i, 0);
  else if constexpr (kIns)
    list_append(ovf, lane, to_ovf, pack(key, val), i, seg);
  if constexpr (MODE == kModeMixed && !DEFER) {
    const unsigned qm = __ballot_sync(kFull, queued);
    if (qm) {
      // q->n < 32 here, so the queue holds the new entries
      if (queued) {
        const uint32_t r = q->n + __popc(qm & ((1u << lane) - 1u));
        q->words[r] = pack(key, val);
        q->idx[r] = i;
      }
      q->n += __popc(qm);
    }
  }

  if (valid) {
    if (MODE == kModeFind) {
      __stcs(a.vals_out + i, outv);
      if (a.found) a.found[i] = st == ST_FOUND ? 1 : 0;
    } else {
      if (a.status && (DEFER || !to_ovf)) a.status[i] = st;
      if (MODE == kModeMixed && a.vals_out) __stcs(a.vals_out + i, outv);
    }
  }
  if constexpr (MODE == kModeMixed && !DEFER) {
    if (q && q->n >= 32) claim_queued<S>(v, *q, ovf, seg, cnt, lane);
  }
}

// Resident 256-thread blocks per SM a bulk kernel is built for, which sets its
// register budget (other shapes: the same warps per SM, at least one block).
// Kernels that claim need about 64 registers (five blocks of 48 spill: bulk
// load 4.36 -> 5.00 ms); the others run at six (lookups on a 2^26-slot table
// 1.455 -> 1.441 ms, erases on an L2-resident one 24.6 -> 21.2 us).
__host__ __device__ constexpr int ops_min_blocks(int mode, bool defer, bool staged, int threads) {
  const int b256 = staged ? 3 : (mode == kModeInsert || (mode == kModeMixed && !defer)) ? 4
                            : mode == kModeMixed                                        ? 5
                                                                                        : 6;
  return b256 * kOpsThreads / threads > 0 ? b256 * kOpsThreads / threads : 1;
}

constexpr int kDeferBuf = 128;  // entries of each warp's buffer of new keys

// DEFER (mixed batches): the new keys are claimed by k_claim afterwards.
// THREADS: the block shape (128, 256 or 512 threads; a tuning knob).
// STAGED: whole buckets staged in shared memory instead of tags (tables with
// a stage_wait_limit).
template <int MODE, int S, bool DEFER, int THREADS, bool STAGED>
__global__ void __launch_bounds__(THREADS, ops_min_blocks(MODE, DEFER, STAGED, THREADS))
    k_ops(View v, OpPtrs a, uint64_t n, List ovf, int prefetch_tags) {
  pdl_trigger();
  if (prefetch_tags) prefetch_l2_grid(v.tags, static_cast<uint64_t>(v.nb) * S);
  const int lane = threadIdx.x & 31;
  // n < 2^32 per call, so chunk and op indices fit 32 bits
  const uint32_t warp0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t nchunks = static_cast<uint32_t>((n + 31) >> 5);
  const uint32_t stash_n = v.ctrl->stash_n;
  __shared__ uint64_t sums[(THREADS / 32) * 8];
  // new keys of a deferring batch gather here, so that the list is written in
  // long runs with one atomic per kDeferBuf entries
  __shared__ __align__(16) uint64_t defer_smem[DEFER ? (THREADS / 32) * 2 * kDeferBuf : 1];
  constexpr bool kQueue = MODE == kModeMixed && !DEFER;
  __shared__ uint64_t queue_smem[kQueue ? (THREADS / 32) * kNewQWords : 1];
  NewQ nq = new_q(queue_smem + (kQueue ? (threadIdx.x >> 5) * kNewQWords : 0));
  // one chunk per warp: claim at once, with the tags at hand
  NewQ* const q = kQueue && nchunks > nwarps ? &nq : nullptr;
  OvfBuf ob{};
  if constexpr (DEFER)
    ob = ovf_buf_init(defer_smem + (threadIdx.x >> 5) * 2 * kDeferBuf, kDeferBuf);
  LaneCounters cnt;
  // inputs are loaded one chunk ahead, so their latency hides behind the
  // current chunk's probes and claims
  OpIn nxt{};
  if (warp0 < nchunks) nxt = load_in<MODE>(a, warp0, n, lane);
  if constexpr (STAGED) {
    extern __shared__ __align__(16) uint64_t ops_smem[];
    Stage sg = stage_init(ops_smem, threadIdx.x >> 5, lane, stage_warp_words(S));
    for (uint32_t c = warp0; c < nchunks; c += nwarps) {
      const OpIn cur = nxt;
      if (c + nwarps < nchunks) nxt = load_in<MODE>(a, c + nwarps, n, lane);
      run_chunk<MODE, S, DEFER>(v, stash_n, a, c, n, ovf, 0, cnt, lane, &sg, &cur, &ob, q);
    }
    stage_drain(sg);
  } else {
    for (uint32_t c = warp0; c < nchunks; c += nwarps) {
      const OpIn cur = nxt;
      if (c + nwarps < nchunks) nxt = load_in<MODE>(a, c + nwarps, n, lane);
      run_chunk<MODE, S, DEFER>(v, stash_n, a, c, n, ovf, 0, cnt, lane, nullptr, &cur, &ob, q);
    }
  }
  if constexpr (kQueue)
    while (nq.n) claim_queued<S>(v, nq, ovf, 0, cnt, lane);
  if constexpr (DEFER) ovf_flush_block(ovf, ob, lane);
  if constexpr (MODE == kModeInsert) count_insert_probes(cnt);
  flush_counters_block(v, cnt, lane, sums + (threadIdx.x >> 5) * 8, sums, 8);
}

// Find batches (Section IV-B).  A warp takes G runs of 32 consecutive ops at a
// time, one op per lane and run, with the keys loaded one run ahead.  The
// found flags of G = 4 runs leave as one 4-byte store per lane, assembled from
// the runs' ballots: with the outputs in host memory, whole lines cross the
// CPU-GPU link where G = 1 sends 32-byte pieces (2^22 ops: 145 -> 137 us; the
// link alone takes 115 us for their 21 MB of results).
//
// What bounds it (one GB300, 2^26 lookups, half of them hits, 2^26 slots at
// 95%, S = 32): DRAM serves about 41 G random lines/s, and a hit needs one.
// 3.68 ms when each lookup read whole 256-byte buckets, 1.44 ms by tags; the
// floor is 0.82 ms for the 2^25 hits, and false tag matches (30 of 255 per
// bucket examined) make the rest.  In an L2-resident table the dependent
// chain key -> tags -> word is the cost: 2^20 slots, 1.7 M lookups 77 -> 27 us.
template <int S, int THREADS, int G, bool KEEP>
__global__ void __launch_bounds__(THREADS, ops_min_blocks(kModeFind, false, false, THREADS))
    k_find(View v, const uint32_t* __restrict__ keys, uint64_t n, uint32_t* __restrict__ vals_out,
           uint8_t* __restrict__ found, int prefetch_tags) {
  if (prefetch_tags) prefetch_l2_grid(v.tags, static_cast<uint64_t>(v.nb) * S);
  const int lane = threadIdx.x & 31;
  const uint32_t warp0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t ngroups = static_cast<uint32_t>((n + 32 * G - 1) / (32 * G));
  const uint32_t stash_n = v.ctrl->stash_n;
  const bool wide = G == 4 && (reinterpret_cast<uintptr_t>(found) & 3) == 0;
  __shared__ uint64_t sums[(THREADS / 32) * 8];
  LaneCounters cnt;
  uint32_t nxt = kEmptyKey;
  {
    const uint64_t i = static_cast<uint64_t>(warp0) * G * 32 + lane;
    if (i < n) nxt = __ldcs(keys + i);
  }
  for (uint32_t g = warp0; g < ngroups; g += nwarps) {
    uint32_t fb[G];
    const uint64_t base = static_cast<uint64_t>(g) * G * 32;
    const bool whole = base + 32 * G <= n;
#pragma unroll 1
    for (int j = 0; j < G; ++j) {
      const uint32_t key = nxt;
      const uint64_t i = base + 32 * j + lane;
      {  // the next run's keys: of this group, or the first of the warp's next one
        const uint64_t k = j + 1 < G ? i + 32 : i + (static_cast<uint64_t>(nwarps) * G - (G - 1)) * 32;
        nxt = k < n ? __ldcs(keys + k) : kEmptyKey;
      }
      const bool valid = i < n;
      const bool live = valid && key < kReservedKeyMin;
      cnt.reserved |= valid && !live;
      const Cand cd = cand_of(v, key);
      Hit h{0, 0, 0, false};
      if (live) {
        const TagVec<S> t1 = ld_tags<S, true>(v, cd.b1);
        const TagVec<S> t2 = ld_tags<S, true>(v, cd.b2);
        const uint32_t t4 = tag_of(key) * 0x01010101u;
        check_words<S, true>(v, cd.b1, cd.b2, tag_match<S>(t1, t4),
                             cd.b2 != cd.b1 ? tag_match<S>(t2, t4) : 0u, key, h, KEEP);
      }
      cnt.probes += live;
      cnt.probes += live && (!h.ok || h.b != cd.b1);
      if (live && !h.ok && stash_n) {
        uint32_t pos;
        cnt.stash_lookups += 1;
        if (stash_find(v, stash_n, key, pos)) {
          h.word = ld_relaxed64(v.stash_kv + pos);
          h.ok = key_of(h.word) == key;
        }
      }
      const uint32_t b = __ballot_sync(kFull, h.ok);
#pragma unroll
      for (int k = 0; k < G; ++k)
        if (j == k) fb[k] = b;
      if (valid) {
        __stcs(vals_out + i, h.ok ? val_of(h.word) : 0u);
        if (found && !(wide && whole)) __stcs(found + i, static_cast<uint8_t>(h.ok));
      }
    }
    if (G == 4 && found && wide && whole) {
      // lane l: the flags of ops 4 l .. 4 l + 3 of the group, four bits of
      // run l / 8's ballot, one to each byte
      uint32_t b = fb[0];
#pragma unroll
      for (int k = 1; k < G; ++k)
        if ((lane >> 3) == k) b = fb[k];
      const uint32_t nib = (b >> ((4 * lane) & 31)) & 0xFu;
      __stcs(reinterpret_cast<uint32_t*>(found + base) + lane, (nib * 0x00204081u) & 0x01010101u);
    }
  }
  flush_counters_block(v, cnt, lane, sums + (threadIdx.x >> 5) * 8, sums, 8);
}

// ----------------------------------------------------------------------------
// Bulk inserts into tables larger than L2: claim first, store by region
// ----------------------------------------------------------------------------
//
// A claim touches tags only (L2), but the store of its word costs DRAM two
// random accesses (the line's fill and its write-back), and at 41 G/s these
// bound a bulk load.  When a batch brings several words to each line, they are
// worth collecting: k_insert_part claims slots and writes (word, slot) pairs
// to a list, kPartTile ops to a tile, sorted within the tile by the table
// region that the slot lies in; k_insert_store then stores the words region
// after region, so that each region's lines gather all their words in L2.
// The list costs 12 bytes written and 12 read per new key.  2^26 slots, S = 32:
// first 55.8 M keys of a bulk load 3.24 -> 2.26 ms (claims 1.62, bound by
// instruction issue and L2 accesses; stores 0.6, bound by the sector fills of
// the lines' first words).
constexpr int kPartThreads = 256;
constexpr int kPartTile = 2048;

template <int S>
__global__ void __launch_bounds__(kPartThreads, 4)
    k_insert_part(View v, OpPtrs a, uint64_t n, List ovf, PartList pl, int prefetch_tags) {
  pdl_trigger();
  if (prefetch_tags) prefetch_l2_grid(v.tags, static_cast<uint64_t>(v.nb) * S);
  __shared__ uint64_t words[kPartTile];
  __shared__ uint32_t slots[kPartTile];
  __shared__ uint16_t rank[kPartTile], order[kPartTile];
  __shared__ uint32_t hist[kPartMaxRegions + 1], first[kPartMaxRegions + 1];
  __shared__ uint64_t sums[(kPartThreads / 32) * 8];
  constexpr int kRounds = kPartTile / kPartThreads;
  const int tid = threadIdx.x, lane = tid & 31;
  const uint32_t stash_n = v.ctrl->stash_n;
  const uint32_t ntiles = static_cast<uint32_t>((n + kPartTile - 1) / kPartTile);
  LaneCounters cnt;
  if (blockIdx.x == 0 && tid == 0) v.ctrl->part_next = 0;  // for k_insert_store
  for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    for (uint32_t r = tid; r <= pl.regions; r += kPartThreads) hist[r] = 0;
    __syncthreads();
    const uint64_t base = static_cast<uint64_t>(tile) * kPartTile;
    uint32_t key_n = base + tid < n ? __ldcs(a.keys + base + tid) : kEmptyKey;
    uint32_t val_n = base + tid < n ? __ldcs(a.vals + base + tid) : 0u;
#pragma unroll 1
    for (int j = 0; j < kRounds; ++j) {
      const int o = j * kPartThreads + tid;
      const uint64_t i = base + o;
      const uint32_t key = key_n, val = val_n;
      if (j + 1 < kRounds && i + kPartThreads < n) {
        key_n = __ldcs(a.keys + i + kPartThreads);
        val_n = __ldcs(a.vals + i + kPartThreads);
      }
      const bool valid = i < n;
      const bool reserved = valid && key >= kReservedKeyMin;
      const bool live = valid && !reserved;
      cnt.reserved |= reserved;
      uint8_t st = reserved ? ST_RESERVED : ST_INSERTED;
      bool to_ovf = false;
      uint32_t sid = kNoOp;
      if (live) {
        const Cand cd = cand_of(v, key);
        const TagVec<S> t1 = ld_tags<S, false>(v, cd.b1);
        const TagVec<S> t2 = ld_tags<S, false>(v, cd.b2);
        const uint32_t t4 = tag_of(key) * 0x01010101u;
        // words of this batch may not be stored yet: none of them holds this
        // key (no key is updated twice in a batch)
        Hit h{0, 0, 0, false};
        check_words<S, false>(v, cd.b1, cd.b2, tag_match<S>(t1, t4),
                              cd.b2 != cd.b1 ? tag_match<S>(t2, t4) : 0u, key, h, true);
        uint64_t* sp = v.buckets + static_cast<uint64_t>(h.b) * S + h.slot;
        if (!h.ok && stash_n) {
          uint32_t pos;
          cnt.stash_lookups += 1;
          if (stash_find(v, stash_n, key, pos)) {
            sp = v.stash_kv + pos;
            h.word = ld_relaxed64(sp);
            h.ok = key_of(h.word) == key;
          }
        }
        if (h.ok) {
          st = ST_REPLACED;
          if (atomicCAS(ull(sp), h.word, pack(key, val)) == h.word)
            cnt.replaced += 1;
          else
            cnt.contract = true;
        } else {
          uint32_t b;
          const uint32_t slot = place_slot<S>(v, cd.b1, cd.b2, t1, t2, key, b);
          if (slot < S) {
            sid = b * S + slot;
            cnt.size_delta += 1;
            cnt.claimed += 1;
          } else {
            to_ovf = true;
            cnt.overflowed += 1;
          }
        }
      }
      if (sid != kNoOp) {
        words[o] = pack(key, val);
        rank[o] = static_cast<uint16_t>(atomicAdd(&hist[sid >> pl.shift], 1u));
      }
      slots[o] = sid;
      const unsigned om = __ballot_sync(kFull, to_ovf);
      if (om) {
        const int leader = __ffs(om) - 1;
        unsigned at = 0;
        if (lane == leader) at = atomicAdd(ovf.count, static_cast<unsigned>(__popc(om)));
        at = __shfl_sync(kFull, at, leader) + __popc(om & ((1u << lane) - 1u));
        if (to_ovf) {
          ovf.words[at] = pack(key, val);
          ovf.idx[at] = static_cast<uint32_t>(i);
        }
      }
      if (valid && a.status && !to_ovf) a.status[i] = st;
    }
    __syncthreads();
    // first[r]: where region r starts within the tile (regions <= 4 x 32)
    if (tid < 32) {
      uint32_t carry = 0;
      for (uint32_t r0 = 0; r0 <= pl.regions; r0 += 32) {
        const uint32_t r = r0 + lane;
        const uint32_t x = r < pl.regions ? hist[r] : 0u;
        uint32_t incl = x;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t y = __shfl_up_sync(kFull, incl, d);
          if (lane >= d) incl += y;
        }
        if (r <= pl.regions) {
          first[r] = carry + incl - x;
          pl.off[static_cast<uint64_t>(tile) * (pl.regions + 1) + r] =
              static_cast<uint16_t>(carry + incl - x);
        }
        carry += __shfl_sync(kFull, incl, 31);
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int o = tid; o < kPartTile; o += kPartThreads) {
      const uint32_t sid = slots[o];
      if (sid != kNoOp) order[first[sid >> pl.shift] + rank[o]] = static_cast<uint16_t>(o);
    }
    __syncthreads();
    const uint32_t m = first[pl.regions];
    for (uint32_t k = tid; k < m; k += kPartThreads) {
      const uint32_t o = order[k];
      __stcs(pl.words + base + k, words[o]);
      __stcs(pl.slots + base + k, slots[o]);
    }
    __syncthreads();
  }
  count_insert_probes(cnt);
  flush_counters_block(v, cnt, lane, sums + (tid >> 5) * 8, sums, 8);
}

// Stores the listed words, regions in order.  Blocks take groups of kStoreTiles
// tiles of one region from a counter, so that all of them work on the same few
// megabytes of the table at any time.
constexpr uint32_t kStoreTiles = 32;
template <int S>
__global__ void __launch_bounds__(256) k_insert_store(View v, uint32_t ntiles, PartList pl) {
  pdl_trigger();
  pdl_wait();
  __shared__ uint32_t taken;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t groups = (ntiles + kStoreTiles - 1) / kStoreTiles;
  const uint32_t total = groups * pl.regions;
  for (;;) {
    if (threadIdx.x == 0) taken = atomicAdd(&v.ctrl->part_next, 1u);
    __syncthreads();
    const uint32_t w = taken;
    __syncthreads();
    if (w >= total) break;
    const uint32_t r = w / groups, g = w - r * groups;
#pragma unroll
    for (uint32_t t = 0; t < kStoreTiles / 8; ++t) {
      const uint32_t tile = g * kStoreTiles + t * 8 + warp;
      if (tile >= ntiles) continue;
      const uint16_t* off = pl.off + static_cast<uint64_t>(tile) * (pl.regions + 1) + r;
      const uint32_t lo = off[0], hi = off[1];
      const uint64_t base = static_cast<uint64_t>(tile) * kPartTile;
#pragma unroll 2
      for (uint32_t k = lo + lane; k < hi; k += 32) {
        const uint64_t word = __ldcs(pl.words + base + k);
        const uint32_t sid = __ldcs(pl.slots + base + k);
        v.buckets[sid] = word;
      }
    }
  }
}

// Step 2 for the new keys of a mixed batch (WABC, Section III-E), after the
// bulk kernel has run every find, erase and replace of the batch and listed
// them in `in`: the slots those erases freed are then visible to the claims.
// One item per lane: hash, read the tags of both buckets, claim a free slot of
// the emptier bucket with one CAS (the other bucket next), store the word.
// Nothing moves or erases a word meanwhile, so the claim publishes with a
// plain store.  Items whose two buckets are both full go to `out` for
// eviction (steps 3-4).
constexpr int kClaimThreads = 256;
constexpr int kClaimBuf = 128;  // entries of each warp's buffer of full-bucket items
template <int S>
__global__ void __launch_bounds__(kClaimThreads, 4) k_claim(View v, List in, List out) {
  pdl_trigger();
  pdl_wait();
  __shared__ __align__(16) uint64_t claim_smem[(kClaimThreads / 32) * 2 * kClaimBuf];
  const int lane = threadIdx.x & 31;
  OvfBuf ob = ovf_buf_init(claim_smem + (threadIdx.x >> 5) * 2 * kClaimBuf, kClaimBuf);
  LaneCounters cnt;
  const uint32_t total = *in.count;
  const uint32_t step = gridDim.x * blockDim.x;
  uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  // entries are loaded one step ahead of their claims
  uint64_t word_n = i < total ? __ldcs(in.words + i) : kEmptyWord;
  uint32_t idx_n = i < total ? __ldcs(in.idx + i) : kNoOp;
  for (; i - lane < total; i += step) {
    const uint64_t word = word_n;
    const uint32_t idx = idx_n;
    const bool valid = i < total;
    TagVec<S> t1, t2;
    Cand cd{0, 0};
    if (valid) {
      cd = cand_of(v, key_of(word));
      t1 = ld_tags<S, false>(v, cd.b1);
      t2 = ld_tags<S, false>(v, cd.b2);
    }
    const uint64_t j = static_cast<uint64_t>(i) + step;
    if (j < total) {
      word_n = __ldcs(in.words + j);
      idx_n = __ldcs(in.idx + j);
    }
    bool to_ovf = false;
    if (valid) {
      if (place_from<S>(v, cd.b1, cd.b2, t1, t2, word)) {
        cnt.size_delta += 1;
        cnt.claimed += 1;
      } else {
        to_ovf = true;
        cnt.overflowed += 1;
      }
    }
    ovf_put(out, ob, lane, to_ovf, word, idx, 0);
    if (j - lane >= total) break;  // also keeps i from wrapping
  }
  ovf_flush_block(out, ob, lane);
  flush_counters_block(v, cnt, lane, ob.words, claim_smem, 2 * kClaimBuf);
}

// ----------------------------------------------------------------------------
// Steps 3-4: bounded cuckoo eviction and the overflow stash (Algorithm 3)
// ----------------------------------------------------------------------------

// A chain may end in the stash, so it first reserves a stash word; chains that
// finish in a bucket give the reservation back, so appends never pass
// stash_cap.  When every free word is reserved by running chains, wait for
// them (they end within max_evictions rounds); give up only once the stash is
// really full or after a bounded wait.
__device__ __forceinline__ bool stash_reserve(const View& v) {
  const uint32_t limit = v.lock_spin_limit * 4u;
  for (uint32_t t = 0; t < limit; ++t) {
    const unsigned c = atomicAdd(&v.ctrl->stash_claims, 1u);
    if (c < v.stash_cap) return true;
    atomicSub(&v.ctrl->stash_claims, 1u);
    if (ld_relaxed32(&v.ctrl->stash_tail) >= v.stash_cap) return false;
    __nanosleep(256);
  }
  return false;
}

// Counters of the eviction kernel, kept by lane 0 of a warp, and the stash
// word the warp holds in reserve.  A warp works one item at a time, so one
// reservation covers all its chains: it is kept across items that end in a
// bucket and renewed only after a chain used it for a stash append.
struct OvfCounters {
  unsigned claim = 0, rounds = 0, locks = 0, to = 0, stash = 0, pend = 0, added = 0;
  Ctrl* reserved_in = nullptr;  // control block of the table the reservation belongs to
};

// `lead`: the calling lane leads its group and holds the group's counters.
__device__ __forceinline__ void flush_ovf_counters(const View& v, OvfCounters& oc, bool lead) {
  if (lead) {
    Ctrl* c = v.ctrl;
    if (oc.added) atomicAdd(&c->size, static_cast<unsigned long long>(oc.added));
    if (oc.claim) atomicAdd(&c->stats[kStClaimedSlow], static_cast<unsigned long long>(oc.claim));
    if (oc.rounds) atomicAdd(&c->stats[kStEvictRounds], static_cast<unsigned long long>(oc.rounds));
    if (oc.locks) atomicAdd(&c->stats[kStLockAcquired], static_cast<unsigned long long>(oc.locks));
    if (oc.to) {
      atomicAdd(&c->stats[kStLockTimeouts], static_cast<unsigned long long>(oc.to));
      atomicOr(&c->err, kErrTimeout);
    }
    if (oc.stash) atomicAdd(&c->stats[kStStashed], static_cast<unsigned long long>(oc.stash));
    if (oc.pend) atomicAdd(&c->stats[kStPending], static_cast<unsigned long long>(oc.pend));
  }
  Ctrl* keep = oc.reserved_in;  // a reservation outlives the counters
  oc = OvfCounters();
  oc.reserved_in = keep;
}

// Gives back a warp's unused stash reservation.
__device__ __forceinline__ void release_reservation(OvfCounters& oc, bool lead) {
  if (lead && oc.reserved_in) atomicSub(&oc.reserved_in->stash_claims, 1u);
  oc.reserved_in = nullptr;
}

// A block's pool of stash reservations: one table-wide atomic fills it for
// the groups that will carry an item, and the groups take from it in shared
// memory.  With thousands of groups per launch, one reservation atomic each
// on the single counter serialised in L2 and cost about a fifth of the
// eviction kernel's time.  A taker succeeds only on a positive count; a
// failed take puts its decrement back.
__device__ __forceinline__ bool pool_take(int* pool) {
  if (!pool) return false;
  if (atomicSub(pool, 1) > 0) return true;
  atomicAdd(pool, 1);
  return false;
}

// Fills the pool with up to `want` reservations (thread 0 of the block).
__device__ __forceinline__ int pool_fill(const View& v, unsigned want) {
  if (!want) return 0;
  const unsigned base = atomicAdd(&v.ctrl->stash_claims, want);
  const unsigned got = base >= v.stash_cap ? 0u : min(want, v.stash_cap - base);
  if (got < want) atomicSub(&v.ctrl->stash_claims, want - got);
  return static_cast<int>(got);
}

// Steps 3-4 for one insert whose candidate buckets were full (warp-wide).
// `idx` is the caller's op index (kNoOp for a word moved by a merge); the
// outcome goes to status[idx].  With `resizable`, an insert that finds no room
// at all joins the pending list, else it is reported FULL.
// `pool` (optional): stash words the calling block reserved for its groups
// in one atomic (a shared-memory count), taken before the table-wide
// counter is asked.
template <int S>
__device__ __forceinline__ void overflow_item(const View& v, uint64_t word0, uint32_t idx,
                                              uint32_t seg, uint8_t* status, int resizable,
                                              const List& pend, OvfCounters& oc, int lane,
                                              int* pool = nullptr) {
  // The item belongs to a group of S lanes (a half-warp at S = 16, so a warp
  // carries two chains at once): group lane gl holds slot gl of the bucket in
  // hand, and group lane 0 leads.
  constexpr unsigned kGroupBits = (S >= 32) ? 0xFFFFFFFFu : ((1u << S) - 1u);
  const int gl = lane & (S - 1);
  const int gb = lane - gl;
  const unsigned gmask = kGroupBits << gb;
  auto group_ballot = [&](bool pred) { return (__ballot_sync(gmask, pred) >> gb) & kGroupBits; };
  const uint32_t key0 = key_of(word0);
  const uint32_t b1 = lh_bucket(bithash1(key0), v.M, v.p);
  const uint32_t b2 = lh_bucket(bithash2(key0), v.M, v.p);

  // 0: needs eviction, 1: placed, 2: stashed, 3: no room (pending)
  int outcome = 0;
  // the BitHash1 bucket, read now for the first eviction round: most items
  // here find both buckets still full
  const uint64_t w0 = ld_relaxed64(v.buckets + static_cast<uint64_t>(b1) * S + gl);
  if (gl == 0) {
    // the tags of both buckets in one round trip; claim where a slot is free
    if (place_new<S>(v, b1, b2, word0)) {
      outcome = 1;
      ++oc.claim;
    } else {
      if (oc.reserved_in != v.ctrl) {
        if (oc.reserved_in) atomicSub(&oc.reserved_in->stash_claims, 1u);
        oc.reserved_in = (pool_take(pool) || stash_reserve(v)) ? v.ctrl : nullptr;
      }
      if (!oc.reserved_in) outcome = 3;
    }
  }
  outcome = __shfl_sync(gmask, outcome, 0, S);

  if (outcome == 0) {
    uint64_t cur = word0;
    uint32_t b = b1;
    bool placed = false;
    for (uint32_t r = 0; r < v.max_evictions; ++r) {
      // Look ahead: each lane checks whether the word in its slot could move
      // to its other candidate bucket without a further eviction.
      const uint64_t w = r == 0 ? w0 : ld_relaxed64(v.buckets + static_cast<uint64_t>(b) * S + gl);
      // a free slot of this word's other candidate bucket (32: none), and
      // the tag word it lies in
      uint32_t ap = 32, aw = 0;
      if (w != kEmptyWord) {
        const uint32_t k = key_of(w);
        const uint32_t a1 = lh_bucket(bithash1(k), v.M, v.p);
        const uint32_t a2 = lh_bucket(bithash2(k), v.M, v.p);
        const uint32_t alt = (a1 == b) ? a2 : a1;
        if (alt != b) {
          const TagVec<S> ta = ld_tags<S, false>(v, alt);
          const uint32_t fm = free_slots<S>(ta);
          if (fm) {
            ap = pick_slot(fm, claim_rot(k));
            aw = tag_sel<S>(ta, ap & 7u);
          }
        }
      }
      const unsigned gm = group_ballot(ap < 32u);
      const unsigned occ = group_ballot(w != kEmptyWord);
      const bool has_empty = occ != kGroupBits;
      int res = 0;  // 0: evicted `victim`, 1: placed, 2: lock wait gave up, 3: redo the round
      uint64_t victim = kEmptyWord;
      // victim: an occupied slot whose word can move on at once, else an
      // occupied slot picked by rotation (never an EMPTY one, see
      // claim_in_word; occupied slots stay occupied here)
      uint32_t vs = S;
      if (gm) {
        vs = __ffs(gm) - 1;
      } else if (occ) {
        const uint32_t start = (bithash2(key_of(cur)) + r) & (S - 1);
        const unsigned rot =
            start ? (((occ >> start) | (occ << (S - start))) & kGroupBits) : occ;
        vs = (start + __ffs(rot) - 1) & (S - 1);
      }
      const uint32_t vp = __shfl_sync(gmask, ap, vs & (S - 1), S);
      const uint32_t vw = __shfl_sync(gmask, aw, vs & (S - 1), S);
      if (gl == 0) {
        ++oc.rounds;
        if (!lock_bucket(v, b)) {
          res = 2;
          ++oc.to;
        } else {
          ++oc.locks;
          if (has_empty && claim_bucket<S>(v, b, cur, claim_rot(key_of(cur)))) {
            res = 1;
            unlock_bucket(v, b);
          } else if (vs >= S) {
            res = 3;  // every slot claimed but not yet published: look again
            unlock_bucket(v, b);
          } else {
            victim = atomicExch(ull(v.buckets + static_cast<uint64_t>(b) * S + vs), cur);
            swap_tag<S>(v, b, vs, key_of(victim), key_of(cur));
            unlock_swapped(v, b);
          }
        }
      }
      res = __shfl_sync(gmask, res, 0, S);
      victim = __shfl_sync(gmask, victim, 0, S);
      if (res == 1) {
        placed = true;
        break;
      }
      if (res == 2) break;
      if (res == 3) continue;
      // Re-route the displaced word to its alternate bucket.
      cur = victim;
      const uint32_t kc = key_of(cur);
      const uint32_t a1 = lh_bucket(bithash1(kc), v.M, v.p);
      const uint32_t a2 = lh_bucket(bithash2(kc), v.M, v.p);
      const uint32_t nb = (a1 == b) ? a2 : a1;
      if (nb == b) break;  // both candidates are this bucket: no alternative
      b = nb;
      int ok = 0;
      if (gl == 0)
        ok = vp < 32u ? claim_in_word<S>(v, b, vp & 7u, vp >> 3, vw, tag_of(kc), cur)
                      : claim_bucket<S>(v, b, cur, claim_rot(kc));
      if (__shfl_sync(gmask, ok, 0, S)) {
        placed = true;
        break;
      }
    }
    if (gl == 0) {
      if (placed && oc.reserved_in && ld_relaxed32(&v.ctrl->stash_claims) >= v.stash_cap) {
        // every free stash word is reserved: give this one back so that a
        // waiting group can go on
        atomicSub(&v.ctrl->stash_claims, 1u);
        oc.reserved_in = nullptr;
      }
      if (!placed) {
        oc.reserved_in = nullptr;  // this append uses the reservation
        const unsigned pos = atomicAdd(&v.ctrl->stash_tail, 1u);
        st_relaxed64(v.stash_kv + pos, cur);
        ++oc.stash;
      }
    }
    outcome = placed ? 1 : 2;
  }

  if (gl == 0) {
    if (outcome == 3) {
      ++oc.pend;
      if (resizable) {
        const unsigned pos = atomicAdd(pend.count, 1u);
        pend.words[pos] = word0;
        pend.idx[pos] = idx;
        if (pend.seg) pend.seg[pos] = seg;
      } else {
        atomicOr(&v.ctrl->err, kErrFull);
        if (status && idx != kNoOp) status[idx] = ST_FULL;
      }
    } else if (idx != kNoOp) {
      ++oc.added;
      if (status) status[idx] = ST_INSERTED;
    }
  }
}

#ifndef HIVE_OVF_MIN_BLOCKS
#define HIVE_OVF_MIN_BLOCKS 1  // resident blocks per SM the eviction kernel's registers allow
#endif
template <int S>
__global__ void __launch_bounds__(kOvfThreads, HIVE_OVF_MIN_BLOCKS)
    k_overflow(View v, List in, List pend, int resizable, uint8_t* __restrict__ status) {
  pdl_trigger();
  pdl_wait();
  // one item per group of S lanes at a time
  const int lane = threadIdx.x & 31;
  const unsigned group0 = (blockIdx.x * blockDim.x + threadIdx.x) / S;
  const unsigned ngroups = (gridDim.x * blockDim.x) / S;
  const bool lead = (lane & (S - 1)) == 0;
  const unsigned total = *in.count;
  // one stash reservation for each group of the block that gets an item, and
  // the groups' counters summed in shared memory: a few table-wide atomics
  // per block instead of several per group
  __shared__ int pool;
  __shared__ unsigned sum[7];
  const unsigned gpb = blockDim.x / S;
  if (threadIdx.x == 0) {
    const unsigned first = blockIdx.x * gpb;
    pool = pool_fill(v, total > first ? min(total - first, gpb) : 0u);
  }
  if (threadIdx.x < 7) sum[threadIdx.x] = 0;
  __syncthreads();
  OvfCounters oc;
  for (unsigned it = group0; it < total; it += ngroups)
    overflow_item<S>(v, in.words[it], in.idx[it], 0, status, resizable, pend, oc, lane, &pool);
  if (lead) {
    if (oc.reserved_in) atomicAdd(&pool, 1);  // back to the block's pool
    oc.reserved_in = nullptr;
    const unsigned c[7] = {oc.claim, oc.rounds, oc.locks, oc.to, oc.stash, oc.pend, oc.added};
#pragma unroll
    for (int k = 0; k < 7; ++k)
      if (c[k]) atomicAdd(&sum[k], c[k]);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (pool > 0) atomicSub(&v.ctrl->stash_claims, static_cast<unsigned>(pool));
    OvfCounters b;
    b.claim = sum[0];
    b.rounds = sum[1];
    b.locks = sum[2];
    b.to = sum[3];
    b.stash = sum[4];
    b.pend = sum[5];
    b.added = sum[6];
    flush_ovf_counters(v, b, true);
  }
}

// ----------------------------------------------------------------------------
// Concurrent mixed batch in one kernel (the paper's single-kernel mode)
// ----------------------------------------------------------------------------
//
// Here finds, erases, replaces, claims and eviction chains of one batch run
// at the same time, so a lookup can race with a chain that has taken a word
// out of a bucket and not yet put it down.  Each bucket has a version word:
// bits 0..15 count the chains holding, in transit, a word whose BitHash1
// bucket this is, bits 16..31 count chain steps that finished (modulo 2^16:
// the count lives as long as the table, and its carry leaves the word
// instead of reaching the transit count).  A chain raises the transit count
// of the BitHash1 bucket of the word it is about to swap out (whichever of
// its two buckets that word sits in) and lowers it (bumping the step count)
// once that word sits in its other bucket or in the stash, with a fence on
// each side.  A lookup of key k reads the version of
// k's BitHash1 bucket before probing and again after a miss: one word covers
// every move of k.  The miss stands only if no word was in transit there and
// the version did not move; otherwise the op probes again.  A hit needs no
// check: the word was observed in place.  Because erases now run beside
// chains, a chain swaps its victim with a CAS on the word it read (never
// onto an EMPTY slot); claims then own their slot by its tag alone.
constexpr uint32_t kTransitMask = 0xFFFFu;  // words in transit
constexpr uint32_t kStep = 1u << 16;         // one finished step
constexpr uint32_t kFusedRetryLimit = 1u << 14;

__device__ __forceinline__ void transit_begin(const View& v, uint32_t b) {
  atomicAdd(v.vers + b, 1u);
  fence_acq_rel_gpu();
}
__device__ __forceinline__ void transit_end(const View& v, uint32_t b) {
  fence_acq_rel_gpu();
  atomicAdd(v.vers + b, kStep - 1u);  // one word fewer in transit, one step more
}

// Steps 3-4 for one new key whose candidate buckets had no free slot, inside
// the single-kernel batch.  One chain per lane: the lanes of a warp carry up
// to 32 chains at once, each on its own (they may diverge; a chain holds at
// most one bucket lock at a time and waits for it a bounded number of
// tries).  A chain is a run of dependent round trips, so carrying many at
// once is what keeps the step short; a warp-wide chain left 31 lanes idle
// per round trip.  The caller has already tried both buckets' tags and holds a
// stash reservation in `oc`.  Each round reads the bucket in hand 4 words at
// a time with the tags of those words' other buckets, and stops at the
// first word that could move on at once (the victim); if none could, the
// victim is the first occupied slot from a rotating start.  Under the bucket
// lock the chain claims a free slot of the bucket for its word, or swaps the
// victim out with a CAS on the exact word it re-read (never onto an EMPTY
// slot), marking the version of the victim's BitHash1 bucket as holding a
// word in transit until that word is down again.  Returns 1 placed, 2
// stashed.
template <int S>
__device__ int chain_lane(const View& v, uint64_t word0, uint32_t b1, OvfCounters& oc) {
  uint64_t cur = word0;
  uint32_t b = b1;
  uint32_t held = kNoOp;  // version bucket marked for the word in hand
  bool placed = false;
  for (uint32_t r = 0; r < v.max_evictions; ++r) {
    uint64_t* B = v.buckets + static_cast<uint64_t>(b) * S;
    unsigned occ = 0;
    int vs = -1;
    uint32_t vp = 32, vw = 0;  // free slot of the victim's other bucket, and its tag word
#pragma unroll 1
    for (int f0 = 0; f0 < S; f0 += 4) {
      uint64_t w[4];
      ld_frag(B + f0, w[0], w[1]);
      ld_frag(B + f0 + 2, w[2], w[3]);
      TagVec<S> ta[4];
      bool can[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        can[k] = false;
        if (w[k] != kEmptyWord) {
          occ |= 1u << (f0 + k);
          const Cand a = cand_of(v, key_of(w[k]));
          const uint32_t alt = (a.b1 == b) ? a.b2 : a.b1;
          if (alt != b) {
            ta[k] = ld_tags<S, false>(v, alt);
            can[k] = true;
          }
        }
      }
#pragma unroll
      for (int k = 3; k >= 0; --k)
        if (can[k]) {
          const uint32_t fm = free_slots<S>(ta[k]);
          if (fm) {
            vs = f0 + k;
            vp = pick_slot(fm, claim_rot(key_of(w[k])));
            vw = tag_sel<S>(ta[k], vp & 7u);
          }
        }
      if (vs >= 0) break;
    }
    if (vs < 0 && occ) {
      const uint32_t start = (bithash2(key_of(cur)) + r) & (S - 1);
      const unsigned rot = (occ >> start) | (start ? (occ << (32 - start)) : 0u);
      vs = static_cast<int>((start + __ffs(rot) - 1) & (S - 1));
    }
    int res;  // 0: swapped, 1: placed, 2: lock wait gave up, 3: redo the round
    uint64_t wv = kEmptyWord;
    uint32_t vb = 0;  // BitHash1 bucket of the victim: its version carries the transit mark
    ++oc.rounds;
    if (!lock_bucket(v, b)) {
      res = 2;
      ++oc.to;
    } else {
      ++oc.locks;
      if (claim_bucket<S>(v, b, cur, claim_rot(key_of(cur)))) {
        res = 1;
      } else if (vs < 0) {
        res = 3;
      } else {
        uint64_t* sp = B + vs;
        wv = ld_relaxed64(sp);
        if (wv == kEmptyWord) {
          res = 3;  // claimed and not yet published, or erased: look again
        } else {
          vb = lh_bucket(bithash1(key_of(wv)), v.M, v.p);
          transit_begin(v, vb);
          if (atomicCAS(ull(sp), wv, cur) == wv) {
            swap_tag<S>(v, b, vs, key_of(wv), key_of(cur));
            res = 0;
          } else {
            transit_end(v, vb);
            res = 3;
          }
        }
      }
      if (res == 0)
        unlock_swapped(v, b);
      else
        unlock_bucket(v, b);
    }
    // the word in hand now sits in b (placed or swapped in)
    if ((res == 0 || res == 1) && held != kNoOp) transit_end(v, held);
    if (res == 1) {
      placed = true;
      held = kNoOp;
      break;
    }
    if (res == 2) break;
    if (res == 3) continue;
    held = vb;
    cur = wv;
    const uint32_t kc = key_of(cur);
    const uint32_t a1 = lh_bucket(bithash1(kc), v.M, v.p);
    const uint32_t a2 = lh_bucket(bithash2(kc), v.M, v.p);
    const uint32_t nb = (a1 == b) ? a2 : a1;
    if (nb == b) break;
    b = nb;
    // the free slot seen in the lookahead (only a guess: the victim may have
    // been swapped meanwhile)
    if (vp < 32u ? claim_in_word<S>(v, b, vp & 7u, vp >> 3, vw, tag_of(kc), cur)
                 : claim_bucket<S>(v, b, cur, claim_rot(kc))) {
      transit_end(v, held);
      held = kNoOp;
      placed = true;
      break;
    }
  }
  if (placed && oc.reserved_in && ld_relaxed32(&v.ctrl->stash_claims) >= v.stash_cap) {
    // every free stash word is reserved: give this one back
    atomicSub(&v.ctrl->stash_claims, 1u);
    oc.reserved_in = nullptr;
  }
  if (!placed) {
    oc.reserved_in = nullptr;  // this append uses the reservation
    const unsigned pos = atomicAdd(&v.ctrl->stash_tail, 1u);
    st_relaxed64(v.stash_kv + pos, cur);
    ++oc.stash;
    if (held != kNoOp) transit_end(v, held);
  }
  return placed ? 1 : 2;
}

// A warp's queue of new keys whose two buckets were full, in shared memory:
// kFusedQ packed words, then kFusedQ op indices.  The warp runs their chains
// 32 at a time (one per lane) once 32 are waiting, and the rest before it
// exits.  `n` is warp-uniform.
constexpr uint32_t kFusedQ = 64;
struct EvictQ {
  uint64_t* words;
  uint32_t* idx;
  uint32_t n;
};

// Runs the chains of the first min(n, 32) queued keys, one per lane, and
// moves the rest to the front (warp-wide).  Each key first tries both
// buckets again (slots may have been freed since); the keys still without room
// take a stash reservation for the warp's chains with one atomic, then run
// their chains.  Not inlined: few keys come here, and the chains' registers
// would spill those of the probes (10^6 ops, S = 32: 80 -> 74 us).
template <int S>
__device__ __noinline__ void fused_drain(const View& v, EvictQ& q, uint8_t* status, const List& pend,
                            int resizable, OvfCounters& oc, int lane) {
  __syncwarp();
  const uint32_t m = q.n < 32 ? q.n : 32u;
  const bool has = static_cast<uint32_t>(lane) < m;
  const uint64_t word = has ? q.words[lane] : kEmptyWord;
  const uint32_t idx = has ? q.idx[lane] : kNoOp;
  const uint32_t key = key_of(word);
  const uint32_t b1 = lh_bucket(bithash1(key), v.M, v.p);
  const uint32_t b2 = lh_bucket(bithash2(key), v.M, v.p);
  int out = 0;  // 1 placed, 2 stashed, 3 no room
  if (has) {
    if (place_new<S>(v, b1, b2, word)) {
      out = 1;
      ++oc.claim;
    }
  }
  // a chain may end in the stash, so it holds a reservation (kept by the lane
  // for its later chains unless a stash append uses it)
  const bool need_res = has && out == 0 && oc.reserved_in != v.ctrl;
  const unsigned rm = __ballot_sync(kFull, need_res);
  if (rm) {
    const int leader = __ffs(rm) - 1;
    const unsigned k = __popc(rm);
    unsigned c0 = 0;
    if (lane == leader) c0 = atomicAdd(&v.ctrl->stash_claims, k);
    c0 = __shfl_sync(kFull, c0, leader);
    const unsigned ok_n = c0 >= v.stash_cap ? 0u : min(k, v.stash_cap - c0);
    if (lane == leader && ok_n < k) atomicSub(&v.ctrl->stash_claims, k - ok_n);
    if (need_res) {
      const unsigned rank = __popc(rm & ((1u << lane) - 1u));
      oc.reserved_in = (rank < ok_n || stash_reserve(v)) ? v.ctrl : nullptr;
    }
  }
  if (has && out == 0) out = oc.reserved_in == v.ctrl ? chain_lane<S>(v, word, b1, oc) : 3;
  __syncwarp();
  if (has) {
    if (out == 3) {
      ++oc.pend;
      if (resizable) {
        // placed by the eviction kernel after the table grows; it writes the status
        const unsigned p = atomicAdd(pend.count, 1u);
        pend.words[p] = word;
        pend.idx[p] = idx;
      } else {
        atomicOr(&v.ctrl->err, kErrFull);
        if (status && idx != kNoOp) status[idx] = ST_FULL;
      }
    } else {
      ++oc.added;
      if (status && idx != kNoOp) status[idx] = ST_INSERTED;
    }
  }
  // the keys after the first 32 move to the front
  const uint32_t rest = q.n - m;
  __syncwarp();
  uint64_t mw = 0;
  uint32_t mi = 0;
  if (static_cast<uint32_t>(lane) < rest) {
    mw = q.words[32 + lane];
    mi = q.idx[32 + lane];
  }
  __syncwarp();
  if (static_cast<uint32_t>(lane) < rest) {
    q.words[lane] = mw;
    q.idx[lane] = mi;
  }
  __syncwarp();
  q.n = rest;
}

// Looks the op keys of the `need` lanes up in the stash words appended during
// this kernel, [from, to) (warp-wide).  A lane that finds its key gets its
// position in `pos` and returns true.
__device__ __forceinline__ bool stash_tail_find(const View& v, uint32_t from, uint32_t to,
                                                unsigned need, uint32_t key, int lane,
                                                uint32_t& pos) {
  bool hit = false;
  for (uint32_t base = from; base < to; base += 32) {
    const uint32_t j = base + lane;
    const uint64_t w = j < to ? ld_relaxed64(v.stash_kv + j) : kEmptyWord;
    for (unsigned m = need; m; m &= m - 1) {
      const int src = __ffs(m) - 1;
      const uint32_t kj = __shfl_sync(kFull, key, src);
      const unsigned eq = __ballot_sync(kFull, w != kEmptyWord && key_of(w) == kj);
      if (lane == src && eq && !hit) {
        hit = true;
        pos = base + __ffs(eq) - 1;
      }
    }
  }
  return hit;
}

// A warp's queue of ops that take the checked probe, in shared memory:
// kFusedQ words (value << 32 | key), then kFusedQ words (op << 32 | op index).
// `n` is warp-uniform.
struct OpQ {
  uint64_t* kv;
  uint64_t* oi;
  uint32_t n;
};

// The checked probe of the first min(n, 32) queued ops, one per lane
// (warp-wide); the rest move to the front.  Each attempt reads the version of
// the BitHash1 bucket of every op still open, then the tags of both its
// buckets, the words whose tag matches, and the stash.  A hit is acted on at
// once: a find takes the value (the word was seen in place), an erase or
// replace CASes the word it saw and probes again if the CAS fails (the word
// moved).  A miss stands only if no word of that version was in transit and
// the version did not move; otherwise the op probes again.  New keys then
// claim a slot by a CAS on its tag; keys whose two buckets are full join the
// warp's eviction queue.
template <int S>
__device__ void fused_checked(const View& v, uint32_t stash_n, const OpPtrs& a, OpQ& rq,
                              EvictQ& q, const List& pend, int resizable, LaneCounters& cnt,
                              OvfCounters& oc, unsigned& retries, int lane) {
  __syncwarp();
  const uint32_t mq = rq.n < 32 ? rq.n : 32u;
  const bool has = static_cast<uint32_t>(lane) < mq;
  const uint64_t kv = has ? rq.kv[lane] : 0u;
  const uint64_t oi = has ? rq.oi[lane] : 0u;
  {
    const uint32_t rest = rq.n - mq;
    uint64_t t0 = 0, t1 = 0;
    if (static_cast<uint32_t>(lane) < rest) {
      t0 = rq.kv[32 + lane];
      t1 = rq.oi[32 + lane];
    }
    __syncwarp();
    if (static_cast<uint32_t>(lane) < rest) {
      rq.kv[lane] = t0;
      rq.oi[lane] = t1;
    }
    __syncwarp();
    rq.n = rest;
  }
  const uint32_t op = has ? static_cast<uint32_t>(oi >> 32) : OP_FIND;
  const uint32_t key = has ? key_of(kv) : kEmptyKey;
  const uint32_t val = val_of(kv);
  const uint32_t i = static_cast<uint32_t>(oi);
  const uint32_t b1 = lh_bucket(bithash1(key), v.M, v.p);
  const uint32_t b2 = lh_bucket(bithash2(key), v.M, v.p);
  bool done = !has;
  uint8_t st = ST_NOT_FOUND;
  uint32_t outv = 0;
  bool absent = false;  // a miss that survived the version check
  for (uint32_t attempt = 0;; ++attempt) {
    const bool active = !done && !absent;
    const unsigned need = __ballot_sync(kFull, active);
    if (!need) break;
    if (attempt >= kFusedRetryLimit) {  // never expected: chains end in bounded time
      if (lane == 0) atomicOr(&v.ctrl->err, kErrTimeout);
      break;
    }
    if (attempt) {
      retries += (lane == 0) ? __popc(need) : 0u;
      __nanosleep(64u << min(attempt, 6u));
    }
    const uint32_t v1 = active ? ld_acquire32(v.vers + b1) : 0u;
    // the stash words appended so far by this kernel (read with the probes: a
    // word appended later was in transit from one of the op's buckets, which
    // the second version read catches)
    const uint32_t tail = ld_relaxed32(&v.ctrl->stash_tail);
    PendCas pc{0, 0, 0, 0, 0};
    Hit h{0, 0, 0, false};
    if (active) {
      const TagVec<S> t1 = ld_tags<S, false>(v, b1);
      const TagVec<S> t2 = ld_tags<S, false>(v, b2);
      const uint32_t t4 = tag_of(key) * 0x01010101u;
      check_words<S, false>(v, b1, b2, tag_match<S>(t1, t4),
                            b2 != b1 ? tag_match<S>(t2, t4) : 0u, key, h, v.keep_words);
    }
    cnt.probes += active;
    cnt.probes += active && (!h.ok || h.b != b1);
    if (h.ok) {
      done = true;
      act_on<kModeMixed, S>(v, h, key, val, op, st, outv, pc);
    }
    // an erase or replace is done once its CAS has succeeded
    bool retry = false;
    if (pc.kind) {
      if (pc.old == pc.cur) {
        if (pc.kind == 1) {
          free_tag<S>(v, pc.b, pc.slot, key);
          cnt.size_delta -= 1;
        } else {
          cnt.replaced += 1;
        }
      } else {
        done = false;
        retry = true;
        st = ST_NOT_FOUND;
      }
    }
    // the stash: the sorted prefix, then what this kernel appended
    const bool miss = active && !done && !retry;
    uint32_t pos = 0;
    bool shit = false;
    if (miss && stash_n) {
      cnt.stash_lookups += 1;
      shit = stash_find(v, stash_n, key, pos);
    }
    const unsigned tneed = __ballot_sync(kFull, miss && !shit);
    if (tneed && tail > stash_n) {
      uint32_t tp = 0;
      if (stash_tail_find(v, stash_n, min(tail, v.stash_cap), tneed, key, lane, tp) && miss &&
          !shit) {
        shit = true;
        pos = tp;
      }
    }
    if (shit) {
      uint64_t* sp = v.stash_kv + pos;
      const uint64_t w = ld_relaxed64(sp);
      if (key_of(w) == key) {
        if (op == OP_FIND) {
          done = true;
          outv = val_of(w);
          st = ST_FOUND;
        } else if (op == OP_ERASE) {
          if (atomicCAS(ull(sp), w, kEmptyWord) == w) {
            done = true;
            st = ST_ERASED;
            cnt.size_delta -= 1;
            atomicExch(&v.ctrl->stash_dirty, 1u);
          } else {
            retry = true;
          }
        } else {
          if (atomicCAS(ull(sp), w, pack(key, val)) == w) {
            done = true;
            st = ST_REPLACED;
            cnt.replaced += 1;
          } else {
            retry = true;
          }
        }
      }
    }
    if (active && !done && !retry) {
      fence_acq_rel_gpu();
      const uint32_t w1 = ld_relaxed32(v.vers + b1);
      absent = (v1 & kTransitMask) == 0 && v1 == w1;
    }
  }

  // New keys: claim in the preferred bucket (two-choice), else the other;
  // keys that find both full join the eviction queue.
  bool to_evict = false;
  if (absent && op == OP_INSERT) {
    if (place_new<S>(v, b1, b2, pack(key, val))) {
      st = ST_INSERTED;
      cnt.size_delta += 1;
      cnt.claimed += 1;
    } else {
      to_evict = true;
      cnt.overflowed += 1;
    }
  }
  if (has) {
    if (a.status && !to_evict) a.status[i] = st;
    if (a.vals_out) a.vals_out[i] = outv;
  }
  const unsigned em = __ballot_sync(kFull, to_evict);
  if (em) {
    // q.n < 32 here, so the queue holds the new entries
    if (to_evict) {
      const uint32_t r = q.n + __popc(em & ((1u << lane) - 1u));
      q.words[r] = pack(key, val);
      q.idx[r] = i;
    }
    q.n += __popc(em);
    if (q.n >= 32) fused_drain<S>(v, q, a.status, pend, resizable, oc, lane);
  }
}

// Ops [32c, 32c + 32) of a mixed batch in the single-kernel mode (one op per
// lane).  Finds and erases first probe by tags without reading versions,
// since a hit needs no check (the word was seen in place).  Their misses, and
// erases whose CAS failed (the word moved), join the warp's queue for the
// checked probe; so do all inserts, which mostly miss (new keys) and would
// have to probe again.  The checked probe runs 32 queued ops at a time.
template <int S>
__device__ __forceinline__ void run_chunk_fused(const View& v, uint32_t stash_n, const OpPtrs a,
                                                uint32_t c, uint64_t n, const OpIn& in,
                                                const List pend, int resizable,
                                                LaneCounters& cnt, OvfCounters& oc,
                                                unsigned& retries, int lane, OpQ& rq, EvictQ& q) {
  const uint32_t i = (c << 5) + lane;
  const bool valid = i < n;
  const uint32_t op = in.op, key = in.key, val = in.val;
  const bool reserved = valid && key >= kReservedKeyMin;
  const bool live = valid && !reserved;
  cnt.reserved |= reserved;
  const uint32_t b1 = lh_bucket(bithash1(key), v.M, v.p);
  const uint32_t b2 = lh_bucket(bithash2(key), v.M, v.p);
  const bool open = live && op != OP_INSERT;
  bool done = false;
  uint8_t st = reserved ? ST_RESERVED : ST_NOT_FOUND;
  uint32_t outv = 0;
  PendCas pc{0, 0, 0, 0, 0};
  Hit h{0, 0, 0, false};
  if (open) {
    const TagVec<S> t1 = ld_tags<S, false>(v, b1);
    const TagVec<S> t2 = ld_tags<S, false>(v, b2);
    const uint32_t t4 = tag_of(key) * 0x01010101u;
    check_words<S, false>(v, b1, b2, tag_match<S>(t1, t4), b2 != b1 ? tag_match<S>(t2, t4) : 0u,
                          key, h, v.keep_words);
  }
  cnt.probes += open;
  cnt.probes += open && (!h.ok || h.b != b1);
  if (h.ok) {
    done = true;
    act_on<kModeMixed, S>(v, h, key, val, op, st, outv, pc);
  }
  if (pc.kind) {
    if (pc.old == pc.cur) {
      free_tag<S>(v, pc.b, pc.slot, key);  // erases only here
      cnt.size_delta -= 1;
    } else {
      done = false;
      st = ST_NOT_FOUND;
    }
  }
  const bool to_check = live && !done;
  if (valid && !to_check) {
    if (a.status) a.status[i] = st;
    if (a.vals_out) __stcs(a.vals_out + i, outv);
  }
  const unsigned cm = __ballot_sync(kFull, to_check);
  if (cm) {
    // rq.n < 32 here, so the queue holds the new entries
    if (to_check) {
      const uint32_t r = rq.n + __popc(cm & ((1u << lane) - 1u));
      rq.kv[r] = pack(key, val);
      rq.oi[r] = (static_cast<uint64_t>(op) << 32) | i;
    }
    rq.n += __popc(cm);
    if (rq.n >= 32)
      fused_checked<S>(v, stash_n, a, rq, q, pend, resizable, cnt, oc, retries, lane);
  }
}

// Shared-memory words per warp of the single-kernel batch: the checked-probe
// queue (2 kFusedQ words), then the eviction queue (kFusedQ words and kFusedQ
// indices).
constexpr int kFusedWarpWords = 3 * static_cast<int>(kFusedQ) + static_cast<int>(kFusedQ) / 2;

template <int S>
__global__ void __launch_bounds__(kOpsThreads, 3)
    k_fused(const __grid_constant__ View v, OpPtrs a, uint64_t n, List pend, int resizable) {
  pdl_trigger();
  __shared__ __align__(16) uint64_t fused_smem_words[(kOpsThreads / 32) * kFusedWarpWords];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  uint64_t* mine = fused_smem_words + static_cast<size_t>(wib) * kFusedWarpWords;
  OpQ rq{mine, mine + kFusedQ, 0};
  EvictQ q{mine + 2 * kFusedQ, reinterpret_cast<uint32_t*>(mine + 3 * kFusedQ), 0};
  const uint32_t warp0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t nchunks = static_cast<uint32_t>((n + 31) >> 5);
  const uint32_t stash_n = v.ctrl->stash_n;
  LaneCounters cnt;
  OvfCounters oc;
  unsigned retries = 0;
  // inputs are loaded one chunk ahead
  OpIn nxt{};
  if (warp0 < nchunks) nxt = load_in<kModeMixed>(a, warp0, n, lane);
  for (uint32_t c = warp0; c < nchunks; c += nwarps) {
    const OpIn cur = nxt;
    if (c + nwarps < nchunks) nxt = load_in<kModeMixed>(a, c + nwarps, n, lane);
    run_chunk_fused<S>(v, stash_n, a, c, n, cur, pend, resizable, cnt, oc, retries, lane, rq, q);
  }
  while (rq.n) fused_checked<S>(v, stash_n, a, rq, q, pend, resizable, cnt, oc, retries, lane);
  while (q.n) fused_drain<S>(v, q, a.status, pend, resizable, oc, lane);
  // counters: one atomic per counter and block
  // (and the lanes' unused stash reservations go back in one atomic)
  __shared__ unsigned sum[9];
  if (threadIdx.x < 9) sum[threadIdx.x] = 0;
  __syncthreads();
  {
    const unsigned c9[9] = {oc.claim, oc.rounds, oc.locks, oc.to, oc.stash, oc.pend, oc.added,
                            retries, oc.reserved_in ? 1u : 0u};
    oc.reserved_in = nullptr;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const unsigned t = __reduce_add_sync(kFull, c9[k]);
      if (lane == 0 && t) atomicAdd(&sum[k], t);
    }
  }
  flush_counters_block(v, cnt, lane, mine, fused_smem_words, kFusedWarpWords);
  if (threadIdx.x == 0) {
    OvfCounters b;
    b.claim = sum[0];
    b.rounds = sum[1];
    b.locks = sum[2];
    b.to = sum[3];
    b.stash = sum[4];
    b.pend = sum[5];
    b.added = sum[6];
    flush_ovf_counters(v, b, true);
    if (sum[7]) atomicAdd(&v.ctrl->stats[kStFusedRetries], static_cast<unsigned long long>(sum[7]));
    if (sum[8]) atomicSub(&v.ctrl->stash_claims, sum[8]);
  }
}

// ----------------------------------------------------------------------------
// Stash maintenance (single CTA)
// ----------------------------------------------------------------------------

__device__ __forceinline__ uint32_t sort_key(uint64_t w) { return key_of(w); }

// Bitonic sort of a[0, P) by key (P a power of two), one CTA.
__device__ void block_bitonic(uint64_t* a, unsigned P) {
  for (unsigned k = 2; k <= P; k <<= 1) {
    for (unsigned j = k >> 1; j > 0; j >>= 1) {
      for (unsigned t = threadIdx.x; t < (P >> 1); t += blockDim.x) {
        const unsigned low = t & (j - 1);
        const unsigned i = ((t - low) << 1) | low;
        const unsigned l = i | j;
        const uint64_t x = a[i], y = a[l];
        const bool up = (i & k) == 0;
        if ((sort_key(x) > sort_key(y)) == up) {
          a[i] = y;
          a[l] = x;
        }
      }
      __syncthreads();
    }
  }
}

// One CTA maintains the stash of the table of `v`; `smem` holds
// kMaintSmemWords words.  `mode` (kMaint*): what a resizable table's call
// asks for before the host has seen the batch's outcome.
template <int S>
__device__ void maint_body(const View& v, uint64_t* smem, int mode = 0) {
  __shared__ unsigned s_reins, s_live;
  Ctrl* c = v.ctrl;
  // items wait for growth: the host grows, places them and asks again
  if ((mode & kMaintUnlessPend) && c->pend_n) return;
  if ((mode & kMaintUnlessOvf) && c->ovf_n) return;
  const unsigned tail = c->stash_tail;
  const unsigned sorted = c->stash_n;
  const unsigned dirty = c->stash_dirty || ((mode & kMaintStash) && sorted);
  if (threadIdx.x == 0) {
    s_reins = 0;
    s_live = 0;
  }
  __syncthreads();
  if (threadIdx.x == 0) {  // the next call's op lists start empty
    c->ovf_n = 0;
    c->pend_n = 0;
    c->defer_n = 0;
  }
  if (tail == sorted && !dirty) return;

  // Move stash words back into a candidate bucket that has room.
  unsigned reins = 0;
  for (unsigned j = threadIdx.x; j < tail; j += blockDim.x) {
    const uint64_t w = v.stash_kv[j];
    if (w == kEmptyWord) continue;
    const uint32_t k = key_of(w);
    const uint32_t b1 = lh_bucket(bithash1(k), v.M, v.p);
    const uint32_t b2 = lh_bucket(bithash2(k), v.M, v.p);
    if (place_new<S>(v, b1, b2, w)) {
      v.stash_kv[j] = kEmptyWord;
      ++reins;
    }
  }
  if (reins) atomicAdd(&s_reins, reins);
  __syncthreads();

  unsigned P = 1;
  while (P < tail) P <<= 1;
  if (P <= kMaintSmemWords) {
    for (unsigned j = threadIdx.x; j < P; j += blockDim.x) smem[j] = j < tail ? v.stash_kv[j] : kEmptyWord;
    __syncthreads();
    block_bitonic(smem, P);
    for (unsigned j = threadIdx.x; j < P; j += blockDim.x) v.stash_kv[j] = smem[j];
  } else {
    // [tail, P) is EMPTY by construction: the buffer is a power of two long
    // and every word past the live prefix is reset to EMPTY below.
    block_bitonic(v.stash_kv, P);
  }
  __syncthreads();

  // EMPTY words sort last: the live prefix ends at the first EMPTY word.
  unsigned live = 0;
  for (unsigned j = threadIdx.x; j < P; j += blockDim.x) {
    const uint64_t w = v.stash_kv[j];
    if (w != kEmptyWord) {
      v.stash_keys[j] = key_of(w);
      ++live;
    }
  }
  if (live) atomicAdd(&s_live, live);
  __syncthreads();
  if (threadIdx.x == 0) {
    c->stash_n = s_live;
    c->stash_tail = s_live;
    c->stash_claims = s_live;
    c->stash_dirty = 0;
    if (s_reins) c->stats[kStStashReinserted] += s_reins;
  }
}

template <int S>
__global__ void __launch_bounds__(kMaintThreads) k_maint(View v, int mode,
                                                                Ctrl* __restrict__ host_out) {
  extern __shared__ uint64_t smem[];
  pdl_wait();
  maint_body<S>(v, smem, mode);
  if (host_out) {
    // the control block for a host that waits next, written to its pinned copy
    __syncthreads();
    constexpr int kWords = sizeof(Ctrl) / sizeof(unsigned long long);
    if (threadIdx.x < kWords)
      reinterpret_cast<unsigned long long*>(host_out)[threadIdx.x] =
          reinterpret_cast<const unsigned long long*>(v.ctrl)[threadIdx.x];
  }
}

// ----------------------------------------------------------------------------
// Linear-hashing resize (Section IV-C)
// ----------------------------------------------------------------------------

// The tags of bucket b as bytes, slot by slot (one warp has the bucket to itself).
template <int S>
__device__ __forceinline__ uint8_t* tag_bytes(const View& v, uint32_t b) {
  return reinterpret_cast<uint8_t*>(v.tags) + static_cast<uint64_t>(b) * S;
}

// Expansion: warp w splits bucket src0 + w into its partner src0 + w + half.
// `v` carries the state after this launch.  A word leaves the source bucket
// when neither candidate address equals the source under the new state; it
// then belongs to the partner, where the movers are packed from slot 0 by a
// ballot-rank compaction.
template <int S>
__device__ __forceinline__ void split_pair(const View& v, uint32_t src, uint32_t half, int lane) {
  const uint32_t dst = src + half;
  uint64_t* sb = v.buckets + static_cast<uint64_t>(src) * S;
  uint64_t* db = v.buckets + static_cast<uint64_t>(dst) * S;
  const uint64_t word = lane < S ? sb[lane] : kEmptyWord;
  bool mv = false;
  if (word != kEmptyWord) {
    const uint32_t k = key_of(word);
    const uint32_t a1 = lh_bucket(bithash1(k), v.M, v.p);
    const uint32_t a2 = lh_bucket(bithash2(k), v.M, v.p);
    mv = (a1 != src) && (a2 != src);
  }
  const unsigned mm = __ballot_sync(kFull, mv);
  if (mv) {
    // the partner's slots past the movers stay EMPTY with tag 0, as every
    // bucket outside [0, nb) is kept
    const uint32_t r = __popc(mm & ((1u << lane) - 1u));
    db[r] = word;
    sb[lane] = kEmptyWord;
    tag_bytes<S>(v, dst)[r] = static_cast<uint8_t>(tag_of(key_of(word)));
    tag_bytes<S>(v, src)[lane] = 0;
  }
}

template <int S>
__global__ void __launch_bounds__(256) k_split(View v, uint32_t src0, uint32_t count, uint32_t half) {
  const uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= count) return;
  split_pair<S>(v, src0 + w, half, threadIdx.x & 31);
}

// Contraction pre-check: how many words of the batch's high buckets do not
// fit into the free slots of their low partner, from the tags alone (one
// thread per pair reads two sectors: 32,768 pairs in 3 us, 8.5 when a warp
// read the high bucket's words).  The last block hands the sum and the stash
// fill to the host, zeroes the counts and empties list A for the merge.
template <int S>
__global__ void __launch_bounds__(256) k_merge_excess(View v, uint32_t count, Ctrl* host_out) {
  const uint32_t w = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned ex = 0;
  if (w < count) {
    const uint32_t low = v.p + w;
    const int fr = __popc(free_slots<S>(ld_tags<S, false>(v, low)));
    const int live = S - __popc(free_slots<S>(ld_tags<S, false>(v, low + v.M + 1u)));
    ex = live > fr ? live - fr : 0;
  }
  __shared__ unsigned sum;
  if (threadIdx.x == 0) sum = 0;
  __syncthreads();
  ex = __reduce_add_sync(kFull, ex);
  if ((threadIdx.x & 31) == 0 && ex) atomicAdd(&sum, ex);
  __syncthreads();
  if (threadIdx.x != 0) return;
  Ctrl* c = v.ctrl;
  if (sum) atomicAdd(&c->merge_excess, sum);
  __threadfence();
  if (atomicAdd(&c->count_blocks, 1u) == gridDim.x - 1) {
    host_out->merge_excess = atomicExch(&c->merge_excess, 0u);
    host_out->stash_claims = c->stash_claims;
    c->count_blocks = 0;
    c->ovf_n = 0;
  }
}

// Contraction: warp w merges high bucket (p + w + 2^m) into low bucket p + w,
// `v` carrying the state after this launch.  Live words take the free slots
// of the low bucket in rank order (the r-th free slot); words that do
// not fit go to the overflow list and are placed by the eviction kernel.
template <int S>
__global__ void __launch_bounds__(256) k_merge(View v, uint32_t count, List ovf) {
  const int lane = threadIdx.x & 31;
  const uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= count) return;
  const uint32_t low = v.p + w;
  const uint32_t high = low + v.M + 1u;
  uint64_t* lb = v.buckets + static_cast<uint64_t>(low) * S;
  uint64_t* hb = v.buckets + static_cast<uint64_t>(high) * S;
  const uint64_t word = lane < S ? hb[lane] : kEmptyWord;
  const bool live = word != kEmptyWord;
  const unsigned lm = __ballot_sync(kFull, live);
  const unsigned rank = __popc(lm & ((1u << lane) - 1u));
  const uint32_t fr =
      __ballot_sync(kFull, lane < S && tag_bytes<S>(v, low)[lane & (S - 1)] == 0);
  const unsigned nfree = __popc(fr);
  const bool fits = live && rank < nfree;
  if (fits) {
    uint32_t m = fr;
    for (unsigned t = 0; t < rank; ++t) m &= m - 1u;
    lb[__ffs(m) - 1] = word;
    tag_bytes<S>(v, low)[__ffs(m) - 1] = static_cast<uint8_t>(tag_of(key_of(word)));
  }
  const bool spill = live && !fits;
  const unsigned sm = __ballot_sync(kFull, spill);
  if (sm) {
    const int leader = __ffs(sm) - 1;
    unsigned base = 0;
    if (lane == leader) base = atomicAdd(ovf.count, static_cast<unsigned>(__popc(sm)));
    base = __shfl_sync(kFull, base, leader);
    if (spill) {
      const unsigned r = base + __popc(sm & ((1u << lane) - 1u));
      ovf.words[r] = word;
      ovf.idx[r] = kNoOp;
    }
  }
  if (lane < S) {
    hb[lane] = kEmptyWord;
    tag_bytes<S>(v, high)[lane] = 0;
  }
}

// Inserts among the op codes of a batch: 16 codes per load (the bytes before
// the first 16-byte boundary and after the last one by single loads) and one
// atomic per block.  Reads n bytes once: 2^22 codes in 5 us (25 with a byte
// per load and an atomic per warp).
__global__ void __launch_bounds__(256)
    k_count_inserts(const uint8_t* __restrict__ ops, uint64_t n, Ctrl* ctrl, unsigned* host_out) {
  const uint64_t tid = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const uint64_t step = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  uint64_t head = (16 - (reinterpret_cast<uintptr_t>(ops) & 15)) & 15;
  if (head > n) head = n;
  const uint64_t nv = (n - head) / 16;
  const uint64_t tail0 = head + 16 * nv;
  unsigned c = 0;
  if (tid < head) c += ops[tid] == OP_INSERT;
  if (tid < n - tail0) c += ops[tail0 + tid] == OP_INSERT;
  const uint4* p = reinterpret_cast<const uint4*>(ops + head);
  for (uint64_t i = tid; i < nv; i += step) {
    const uint4 x = __ldg(p + i);  // op code 0 is an insert
    c += __popc(zero_bytes(x.x)) + __popc(zero_bytes(x.y)) + __popc(zero_bytes(x.z)) +
         __popc(zero_bytes(x.w));
  }
  __shared__ unsigned sum;
  if (threadIdx.x == 0) sum = 0;
  __syncthreads();
  c = __reduce_add_sync(kFull, c);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(&sum, c);
  __syncthreads();
  if (threadIdx.x != 0) return;
  if (sum) atomicAdd(&ctrl->n_insert, sum);
  __threadfence();
  // the last block hands the total to the host and leaves both counts at zero
  if (atomicAdd(&ctrl->count_blocks, 1u) == gridDim.x - 1) {
    *host_out = atomicExch(&ctrl->n_insert, 0u);
    ctrl->count_blocks = 0;
  }
}

// ----------------------------------------------------------------------------
// Multi-table batches: many independent tables serviced by one launch per
// phase.  A batch is a list of segments (table, op range); segment s owns the
// 32-op chunks [chunk0_s, chunk0_{s+1}) of the batch.  Each table keeps its own
// control block, so counters, stash and sticky errors stay per table.
// ----------------------------------------------------------------------------

__device__ __forceinline__ OpPtrs seg_ptrs(const MultiSeg& S) {
  return OpPtrs{S.ops, S.keys, S.vals, S.vals_out, nullptr, S.status};
}

// Each warp takes a contiguous run of chunks, so it changes table only at
// segment boundaries and flushes its counters there.  A small batch is a chain
// of dependent reads (segment, op, tags, word), so the segment of the first
// chunk is found 32 ways at a time, and a segment descriptor carries its
// table's view.  The descriptor sits in shared memory: in registers it cost
// 200 bytes of spills per thread.
template <int S>
__global__ void __launch_bounds__(kOpsThreads, HIVE_MULTI_MIN_BLOCKS)
    k_multi_ops(const MultiHdr* __restrict__ hdr, const MultiSeg* __restrict__ segs, List ovf) {
  pdl_trigger();
  __shared__ MultiSeg held[kOpsThreads / 32];
  __shared__ uint64_t queue_smem[(kOpsThreads / 32) * kNewQWords];
  const int lane = threadIdx.x & 31;
  MultiSeg& sg = held[threadIdx.x >> 5];
  const uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
  const uint32_t total = hdr->total_chunks;
  const uint32_t ns = hdr->n_segs;
  const uint32_t c0 = static_cast<uint32_t>(static_cast<uint64_t>(total) * w / nw);
  const uint32_t c1 = static_cast<uint32_t>(static_cast<uint64_t>(total) * (w + 1) / nw);
  if (c0 >= c1) return;
  NewQ nq = new_q(queue_smem + (threadIdx.x >> 5) * kNewQWords);
  NewQ* const q = c1 - c0 > 1 ? &nq : nullptr;
  // the last segment with chunk0 <= c0: [lo, hi) narrows to a 32nd per step
  uint32_t lo = 0, hi = ns;
  while (hi - lo > 1) {
    const uint32_t step = (hi - lo + 31) / 32;
    const uint32_t at = lo + lane * step;
    const unsigned le = __ballot_sync(kFull, at < hi && segs[at < hi ? at : lo].chunk0 <= c0);
    const uint32_t k = 31 - __clz(le);  // lane 0 always holds
    hi = min(hi, lo + (k + 1) * step);
    lo += k * step;
  }
  uint32_t s = lo;
  auto take = [&](uint32_t i) {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(segs + i);
    uint32_t* dst = reinterpret_cast<uint32_t*>(&sg);
    __syncwarp();
    for (uint32_t k = lane; k < sizeof(MultiSeg) / 4; k += 32) dst[k] = __ldg(src + k);
    __syncwarp();
  };
  take(s);
  uint32_t next0 = s + 1 < ns ? segs[s + 1].chunk0 : 0xFFFFFFFFu;
  uint32_t stash_n = sg.v.ctrl->stash_n;
  LaneCounters cnt;
  OpIn nxt = load_in<kModeMixed>(seg_ptrs(sg), c0 - sg.chunk0, sg.n, lane);
  for (uint32_t c = c0; c < c1; ++c) {
    if (next0 <= c) {
      while (nq.n) claim_queued<S>(sg.v, nq, ovf, s, cnt, lane);
      flush_counters(sg.v, cnt, lane);
      do {
        ++s;
      } while (s + 1 < ns && segs[s + 1].chunk0 <= c);
      take(s);
      next0 = s + 1 < ns ? segs[s + 1].chunk0 : 0xFFFFFFFFu;
      stash_n = sg.v.ctrl->stash_n;
      nxt = load_in<kModeMixed>(seg_ptrs(sg), c - sg.chunk0, sg.n, lane);
    }
    const OpIn cur = nxt;
    // the next chunk's inputs, unless another segment starts there
    if (c + 1 < c1 && c + 1 < next0)
      nxt = load_in<kModeMixed>(seg_ptrs(sg), c + 1 - sg.chunk0, sg.n, lane);
    run_chunk<kModeMixed, S>(sg.v, stash_n, seg_ptrs(sg), c - sg.chunk0, sg.n, ovf, s, cnt, lane,
                             nullptr, &cur, nullptr, q);
  }
  while (nq.n) claim_queued<S>(sg.v, nq, ovf, s, cnt, lane);
  flush_counters(sg.v, cnt, lane);
}

// Steps 3-4 for the overflow list of a multi-table batch.  Inserts that find
// no room are reported FULL (a resizable table grows before its next batch).
template <int S>
__global__ void __launch_bounds__(kOvfThreads)
    k_multi_overflow(const MultiSeg* __restrict__ segs, List in) {
  pdl_trigger();
  pdl_wait();
  // one item per group of S lanes at a time
  const int lane = threadIdx.x & 31;
  const unsigned group0 = (blockIdx.x * blockDim.x + threadIdx.x) / S;
  const unsigned ngroups = (gridDim.x * blockDim.x) / S;
  const bool lead = (lane & (S - 1)) == 0;
  const unsigned total = *in.count;
  const List none{nullptr, nullptr, nullptr, nullptr};
  OvfCounters oc;
  for (unsigned it = group0; it < total; it += ngroups) {
    const uint32_t sg = in.seg[it];
    const View v = segs[sg].v;
    overflow_item<S>(v, in.words[it], in.idx[it], sg, segs[sg].status, 0, none, oc, lane);
    flush_ovf_counters(v, oc, lead);
  }
  release_reservation(oc, lead);
}

// One CTA per table of the batch: stash maintenance (exits at once when
// nothing changed), then the table's size and stash fill for the host's resize
// policy (entries of tables outside the batch are left as they were).  The
// grid covers every table of the group, so a captured graph serves batches of
// any composition.  Block 0 also empties the batch's overflow list for the
// next batch.
template <int S>
__global__ void __launch_bounds__(256)
    k_multi_maint(const MultiHdr* __restrict__ hdr, const View* __restrict__ views,
                  const uint32_t* __restrict__ touched, unsigned* __restrict__ ovf_count,
                  unsigned long long* __restrict__ out) {
  extern __shared__ uint64_t smem[];
  pdl_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0) *ovf_count = 0;
  if (blockIdx.x >= hdr->n_touched) return;
  const uint32_t t = touched[blockIdx.x];
  maint_body<S>(views[t], smem);
  __syncthreads();
  if (threadIdx.x == 0) {
    const Ctrl* c = views[t].ctrl;
    out[2 * t] = c->size;
    out[2 * t + 1] = (static_cast<unsigned long long>(c->err) << 32) | c->stash_claims;
  }
}

// One wave of split launches over many tables: warp w runs pair
// w - pair0 of the job whose range holds w.  Jobs of one wave touch disjoint
// buckets (a table appears in a wave with splits of one round only).
template <int S>
__global__ void __launch_bounds__(256)
    k_multi_split(const MultiJob* __restrict__ jobs, uint32_t n_jobs, uint32_t total_pairs,
                  const View* __restrict__ views) {
  const uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= total_pairs) return;
  uint32_t lo = 0, hi = n_jobs;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (jobs[mid].pair0 <= w) lo = mid; else hi = mid;
  }
  const MultiJob J = jobs[lo];
  View v = views[J.table];
  v.M = J.M;
  v.p = J.p;
  split_pair<S>(v, J.src0 + (w - J.pair0), J.half, threadIdx.x & 31);
}

// BitHash1 and BitHash2 of n keys (hive_hash).
__global__ void k_hash(const uint32_t* __restrict__ keys, uint64_t n, uint32_t* __restrict__ h1,
                       uint32_t* __restrict__ h2) {
  for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
    const uint32_t k = __ldcs(keys + i);
    if (h1) __stcs(h1 + i, bithash1(k));
    if (h2) __stcs(h2 + i, bithash2(k));
  }
}

__global__ void k_fill_u32(uint32_t* __restrict__ p, uint64_t n, uint32_t value) {
  for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<uint64_t>(gridDim.x) * blockDim.x)
    p[i] = value;
}

// Launches a kernel on `s`, inside the table's persisting L2 window over the
// slot tags when it has one (a per-launch attribute: the stream is left as
// it was).  DEP: as the dependent of the call's previous kernel (see pdl_wait).
template <bool DEP = false, typename... KArgs, typename... Args>
cudaError_t launch_in_window(const Launch& L, void (*kern)(KArgs...), unsigned grid,
                             unsigned block, size_t smem, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  cfg.attrs = at;
  if (L.l2_bytes) {
    cudaLaunchAttribute& w = at[cfg.numAttrs++];
    w.id = cudaLaunchAttributeAccessPolicyWindow;
    w.val.accessPolicyWindow.base_ptr = L.l2_base;
    w.val.accessPolicyWindow.num_bytes = L.l2_bytes;
    w.val.accessPolicyWindow.hitRatio = L.l2_hit;
    w.val.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
    w.val.accessPolicyWindow.missProp = cudaAccessPropertyStreaming;
  }
  if (DEP) {
    cudaLaunchAttribute& d = at[cfg.numAttrs++];
    d.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    d.val.programmaticStreamSerializationAllowed = 1;
  }
  return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}
template <int MODE, int S, bool DEFER, int THREADS, bool STAGED = false>
cudaError_t launch_ops_tt(const View& v, const OpPtrs& a, uint64_t n, List ovf, const Launch& L,
                          cudaStream_t s) {
  const uint64_t chunks = (n + 31) / 32;
  constexpr uint64_t warps_per_block = THREADS / 32;
  uint64_t blocks = (chunks + warps_per_block - 1) / warps_per_block;
  const int per_sm =
      STAGED ? L.staged_blocks_per_sm : L.ops_blocks_per_sm[MODE + (DEFER ? 1 : 0)];
  const uint64_t cap = static_cast<uint64_t>(L.num_sms) * per_sm;
  if (blocks > cap) blocks = cap;
  if (blocks == 0) blocks = 1;
  const size_t smem = STAGED ? stage_smem(S, THREADS) : 0;
  const int pf = prefetch_tags_rule(n, v.nb, S);
  if constexpr (MODE == kModeFind && !STAGED) {  // finds change no tag: no persisting window
    // groups of four runs once every warp has at least four of them: with
    // fewer, rounding to whole groups leaves warps idle (1.7 M ops on 7296
    // warps: 33 us against 28)
    const bool long_batch = chunks >= cap * warps_per_block * 16;
    auto kern = long_batch ? (v.keep_words ? k_find<S, THREADS, 4, true> : k_find<S, THREADS, 4, false>)
                           : (v.keep_words ? k_find<S, THREADS, 1, true> : k_find<S, THREADS, 1, false>);
    kern<<<static_cast<unsigned>(blocks), THREADS, 0, s>>>(v, a.keys, n, a.vals_out, a.found, pf);
    return cudaGetLastError();
  } else
  return launch_in_window(L, k_ops<MODE, S, DEFER, THREADS, STAGED>, static_cast<unsigned>(blocks),
                          THREADS, smem, s, v, a, n, ovf, pf);
}

template <int MODE, int S, bool DEFER = false>
cudaError_t launch_ops_t(View v, const uint8_t* ops, const uint32_t* keys,
                         const uint32_t* vals, uint64_t n, uint32_t* vals_out, uint8_t* found,
                         uint8_t* status, List ovf, const Launch& L, cudaStream_t s) {
  const OpPtrs a{ops, keys, vals, vals_out, found, status};
  if (MODE != kModeFind && n * 16 >= static_cast<uint64_t>(v.nb) * S) v.keep_words = 1;
  if constexpr (S == 32) {
    if (L.staged) return launch_ops_tt<MODE, S, DEFER, 256, true>(v, a, n, ovf, L, s);
  }
  switch (L.ops_threads) {
    case 128:
      return launch_ops_tt<MODE, S, DEFER, 128>(v, a, n, ovf, L, s);
    case 512:
      return launch_ops_tt<MODE, S, DEFER, 512>(v, a, n, ovf, L, s);
    default:
      return launch_ops_tt<MODE, S, DEFER, 256>(v, a, n, ovf, L, s);
  }
}

template <int S>
cudaError_t launch_ops_s(int mode, const View& v, const uint8_t* ops, const uint32_t* keys,
                         const uint32_t* vals, uint64_t n, uint32_t* vals_out, uint8_t* found,
                         uint8_t* status, List ovf, const Launch& L, cudaStream_t s, bool defer) {
  switch (mode) {
    case kModeFind:
      return launch_ops_t<kModeFind, S>(v, ops, keys, vals, n, vals_out, found, status, ovf, L, s);
    case kModeInsert:
      return launch_ops_t<kModeInsert, S>(v, ops, keys, vals, n, vals_out, found, status, ovf, L, s);
    case kModeErase:
      return launch_ops_t<kModeErase, S>(v, ops, keys, vals, n, vals_out, found, status, ovf, L, s);
    default:
      if (defer)
        return launch_ops_t<kModeMixed, S, true>(v, ops, keys, vals, n, vals_out, found, status, ovf,
                                                 L, s);
      return launch_ops_t<kModeMixed, S>(v, ops, keys, vals, n, vals_out, found, status, ovf, L, s);
  }
}

}  // namespace

cudaError_t launch_fused(View v, const uint8_t* ops, const uint32_t* keys,
                         const uint32_t* vals, uint64_t n, uint32_t* vals_out, uint8_t* status,
                         List pend, int resizable, const Launch& L, cudaStream_t s) {
  // words stay in L2 only for a batch of an op or more per line (2^22 ops on
  // 2^26 slots 629 -> 616 us; 10^6 ops on 2^24 slots 147 us, 152 kept)
  v.keep_words = n * 16 >= static_cast<uint64_t>(v.nb) * v.S;
  const uint64_t chunks = (n + 31) / 32;
  const uint64_t warps_per_block = kOpsThreads / 32;
  uint64_t blocks = (chunks + warps_per_block - 1) / warps_per_block;
  const uint64_t cap = static_cast<uint64_t>(L.num_sms) * L.fused_blocks_per_sm;
  if (blocks > cap) blocks = cap;
  if (blocks == 0) blocks = 1;
  const OpPtrs a{ops, keys, vals, vals_out, nullptr, status};
  if (v.S == 16)
    k_fused<16><<<static_cast<unsigned>(blocks), kOpsThreads, 0, s>>>(v, a, n, pend, resizable);
  else
    k_fused<32><<<static_cast<unsigned>(blocks), kOpsThreads, 0, s>>>(v, a, n, pend, resizable);
  return cudaGetLastError();
}

cudaError_t launch_ops(int mode, const View& v, const uint8_t* ops, const uint32_t* keys,
                       const uint32_t* vals, uint64_t n, uint32_t* vals_out, uint8_t* found,
                       uint8_t* status, List ovf, const Launch& L, cudaStream_t s, bool defer) {
  if (v.S == 16)
    return launch_ops_s<16>(mode, v, ops, keys, vals, n, vals_out, found, status, ovf, L, s, defer);
  return launch_ops_s<32>(mode, v, ops, keys, vals, n, vals_out, found, status, ovf, L, s, defer);
}

uint64_t part_tiles(uint64_t n) { return (n + kPartTile - 1) / kPartTile; }

template <int S>
static cudaError_t load_part_kernels() {
  cudaFuncAttributes a;
  const cudaError_t e = cudaFuncGetAttributes(&a, k_insert_part<S>);
  return e != cudaSuccess ? e : cudaFuncGetAttributes(&a, k_insert_store<S>);
}
cudaError_t prepare_insert_part(int S) {
  return S == 16 ? load_part_kernels<16>() : load_part_kernels<32>();
}

cudaError_t launch_insert_part(const View& v, const uint32_t* keys, const uint32_t* vals,
                               uint64_t n, uint8_t* status, List ovf, const PartList& pl,
                               const Launch& L, cudaStream_t s) {
  const OpPtrs a{nullptr, keys, vals, nullptr, nullptr, status};
  const uint32_t ntiles = static_cast<uint32_t>(part_tiles(n));
  // as many warps per SM as the plain insert kernel runs (config blocks_per_sm)
  const int per_sm = L.ops_blocks_per_sm[kModeInsert] * L.ops_threads / kPartThreads;
  const unsigned cap = static_cast<unsigned>(L.num_sms) * (per_sm > 4 ? 4 : per_sm < 1 ? 1 : per_sm);
  const unsigned blocks = ntiles < cap ? ntiles : cap;
  const int pf = prefetch_tags_rule(n, v.nb, v.S);
  cudaError_t e;
  if (v.S == 16)
    e = launch_in_window(L, k_insert_part<16>, blocks, kPartThreads, 0, s, v, a, n, ovf, pl, pf);
  else
    e = launch_in_window(L, k_insert_part<32>, blocks, kPartThreads, 0, s, v, a, n, ovf, pl, pf);
  if (e != cudaSuccess) return e;
  const unsigned sb = static_cast<unsigned>(L.num_sms) * 8;
  if (v.S == 16) return launch_dependent(k_insert_store<16>, sb, 256, 0, s, v, ntiles, pl);
  return launch_dependent(k_insert_store<32>, sb, 256, 0, s, v, ntiles, pl);
}

cudaError_t launch_claim(const View& v, List in, uint64_t n, List out, const Launch& L,
                         cudaStream_t s) {
  if (!n) return cudaSuccess;
  uint64_t blocks = (n + kClaimThreads - 1) / kClaimThreads;
  const uint64_t cap = static_cast<uint64_t>(L.num_sms) * L.claim_blocks_per_sm;
  if (blocks > cap) blocks = cap;
  if (v.S == 16)
    return launch_in_window<true>(L, k_claim<16>, static_cast<unsigned>(blocks), kClaimThreads, 0, s, v,
                            in, out);
  return launch_in_window<true>(L, k_claim<32>, static_cast<unsigned>(blocks), kClaimThreads, 0, s, v, in,
                          out);
}

cudaError_t launch_overflow(const View& v, List in, List pend, int resizable, uint8_t* status,
                            const Launch& L, cudaStream_t s) {
  const unsigned blocks = static_cast<unsigned>(L.num_sms * L.ovf_blocks_per_sm);
  if (v.S == 16)
    return launch_in_window<true>(L, k_overflow<16>, blocks, kOvfThreads, 0, s, v, in, pend, resizable,
                            status);
  return launch_in_window<true>(L, k_overflow<32>, blocks, kOvfThreads, 0, s, v, in, pend, resizable,
                          status);
}

cudaError_t launch_maintenance(const View& v, cudaStream_t s, int mode, Ctrl* host_out) {
  constexpr size_t smem = kMaintSmemWords * sizeof(uint64_t);
  if (v.S == 16) return launch_dependent(k_maint<16>, 1, kMaintThreads, smem, s, v, mode, host_out);
  return launch_dependent(k_maint<32>, 1, kMaintThreads, smem, s, v, mode, host_out);
}

cudaError_t launch_split(const View& v_new, uint32_t src0, uint32_t count, uint32_t half,
                         cudaStream_t s) {
  if (!count) return cudaSuccess;
  const unsigned blocks = (count * 32u + 255u) / 256u;
  if (v_new.S == 16)
    k_split<16><<<blocks, 256, 0, s>>>(v_new, src0, count, half);
  else
    k_split<32><<<blocks, 256, 0, s>>>(v_new, src0, count, half);
  return cudaGetLastError();
}

cudaError_t launch_merge_excess(const View& v_new, uint32_t count, Ctrl* host_out,
                                cudaStream_t s) {
  if (!count) return cudaSuccess;
  const unsigned blocks = (count + 255u) / 256u;
  if (v_new.S == 16)
    k_merge_excess<16><<<blocks, 256, 0, s>>>(v_new, count, host_out);
  else
    k_merge_excess<32><<<blocks, 256, 0, s>>>(v_new, count, host_out);
  return cudaGetLastError();
}

cudaError_t launch_merge(const View& v_new, uint32_t count, List ovf, cudaStream_t s) {
  if (!count) return cudaSuccess;
  const unsigned blocks = (count * 32u + 255u) / 256u;
  if (v_new.S == 16)
    k_merge<16><<<blocks, 256, 0, s>>>(v_new, count, ovf);
  else
    k_merge<32><<<blocks, 256, 0, s>>>(v_new, count, ovf);
  return cudaGetLastError();
}

cudaError_t launch_count_inserts(const uint8_t* ops, uint64_t n, Ctrl* ctrl, unsigned* host_out,
                                 cudaStream_t s) {
  if (!n) return cudaSuccess;
  uint64_t blocks = (n / 16 + 255) / 256;
  if (blocks > 152 * 4) blocks = 152 * 4;
  if (blocks == 0) blocks = 1;
  k_count_inserts<<<static_cast<unsigned>(blocks), 256, 0, s>>>(ops, n, ctrl, host_out);
  return cudaGetLastError();
}

cudaError_t launch_hash(const uint32_t* keys, uint64_t n, uint32_t* h1, uint32_t* h2,
                        cudaStream_t s) {
  if (!n) return cudaSuccess;
  uint64_t blocks = (n + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  k_hash<<<static_cast<unsigned>(blocks), 256, 0, s>>>(keys, n, h1, h2);
  return cudaGetLastError();
}

cudaError_t launch_fill_u32(uint32_t* p, uint64_t n, uint32_t value, cudaStream_t s) {
  if (!n) return cudaSuccess;
  uint64_t blocks = (n + 255) / 256;
  if (blocks > 8192) blocks = 8192;
  k_fill_u32<<<static_cast<unsigned>(blocks), 256, 0, s>>>(p, n, value);
  return cudaGetLastError();
}

cudaError_t launch_multi_ops(int S, const MultiHdr* hdr, const MultiSeg* segs, List ovf,
                             const Launch& L, cudaStream_t s) {
  const unsigned blocks = static_cast<unsigned>(L.num_sms * L.multi_blocks_per_sm);
  if (S == 16)
    k_multi_ops<16><<<blocks, kOpsThreads, 0, s>>>(hdr, segs, ovf);
  else
    k_multi_ops<32><<<blocks, kOpsThreads, 0, s>>>(hdr, segs, ovf);
  return cudaGetLastError();
}

namespace {
// A batch's descriptors (tens of kilobytes) by a kernel that reads them over
// the CPU-GPU link: a copy engine's turn between kernels costs 4 us more.
__global__ void __launch_bounds__(1024)
    k_stage(uint4* __restrict__ dst, const uint4* __restrict__ src, uint32_t n) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = src[i];
}
}  // namespace
cudaError_t launch_stage(void* dst, const void* src, size_t bytes, cudaStream_t s) {
  const uint32_t n = static_cast<uint32_t>((bytes + 15) / 16);
  if (!n) return cudaSuccess;
  k_stage<<<(n + 1023) / 1024, 1024, 0, s>>>(static_cast<uint4*>(dst),
                                             static_cast<const uint4*>(src), n);
  return cudaGetLastError();
}
cudaError_t launch_multi_overflow(int S, const MultiSeg* segs, List in, const Launch& L,
                                  cudaStream_t s) {
  const unsigned blocks = static_cast<unsigned>(L.num_sms * L.ovf_blocks_per_sm);
  if (S == 16) return launch_dependent(k_multi_overflow<16>, blocks, kOvfThreads, 0, s, segs, in);
  return launch_dependent(k_multi_overflow<32>, blocks, kOvfThreads, 0, s, segs, in);
}

cudaError_t launch_multi_maint(int S, const MultiHdr* hdr, const View* views,
                               const uint32_t* touched, uint32_t max_tables, unsigned* ovf_count,
                               unsigned long long* out, cudaStream_t s) {
  if (!max_tables) return cudaSuccess;
  constexpr size_t smem = kMaintSmemWords * sizeof(uint64_t);
  if (S == 16)
    return launch_dependent(k_multi_maint<16>, max_tables, 256, smem, s, hdr, views, touched,
                            ovf_count, out);
  return launch_dependent(k_multi_maint<32>, max_tables, 256, smem, s, hdr, views, touched,
                          ovf_count, out);
}

cudaError_t launch_multi_split(int S, const MultiJob* jobs, uint32_t n_jobs, uint32_t total_pairs,
                               const View* views, cudaStream_t s) {
  if (!total_pairs) return cudaSuccess;
  const unsigned blocks = static_cast<unsigned>((static_cast<uint64_t>(total_pairs) * 32 + 255) / 256);
  if (S == 16)
    k_multi_split<16><<<blocks, 256, 0, s>>>(jobs, n_jobs, total_pairs, views);
  else
    k_multi_split<32><<<blocks, 256, 0, s>>>(jobs, n_jobs, total_pairs, views);
  return cudaGetLastError();
}

namespace {
// Resident blocks of the bulk kernels of one shape.
template <int S, int T, int MODE, bool DEFER = false>
cudaError_t occupancy_mode(Launch* L) {
  int b = 0;
  cudaError_t e;
  if constexpr (MODE == kModeFind)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_find<S, T, 4, false>, T, 0);
  else
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_ops<MODE, S, DEFER, T, false>, T, 0);
  L->ops_blocks_per_sm[MODE + (DEFER ? 1 : 0)] = b > 0 ? b : 1;
  return e;
}
template <int S, int T>
cudaError_t occupancy_ops(Launch* L) {
  cudaError_t e = occupancy_mode<S, T, kModeFind>(L);
  if (e == cudaSuccess) e = occupancy_mode<S, T, kModeInsert>(L);
  if (e == cudaSuccess) e = occupancy_mode<S, T, kModeErase>(L);
  if (e == cudaSuccess) e = occupancy_mode<S, T, kModeMixed>(L);
  if (e == cudaSuccess) e = occupancy_mode<S, T, kModeMixed, true>(L);
  return e;
}

// The same for the staged kernels (32-slot buckets, 256 threads).
template <int MODE, bool DEFER>
cudaError_t staged_limits(int* least) {
  constexpr int smem = static_cast<int>(stage_smem(32));
  cudaError_t e = cudaFuncSetAttribute(k_ops<MODE, 32, DEFER, 256, true>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  int b = 0;
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_ops<MODE, 32, DEFER, 256, true>, 256,
                                                      smem);
  if (b < 1) b = 1;
  if (b < *least) *least = b;
  return e;
}

template <int S>
cudaError_t occupancy_s(Launch* L) {
  int b = 0;
  cudaError_t e = L->ops_threads == 128   ? occupancy_ops<S, 128>(L)
                  : L->ops_threads == 512 ? occupancy_ops<S, 512>(L)
                                          : occupancy_ops<S, 256>(L);
  if (e != cudaSuccess) return e;
  if (S == 32 && L->staged) {
    int least = 64;
    e = staged_limits<kModeFind, false>(&least);
    if (e == cudaSuccess) e = staged_limits<kModeInsert, false>(&least);
    if (e == cudaSuccess) e = staged_limits<kModeErase, false>(&least);
    if (e == cudaSuccess) e = staged_limits<kModeMixed, false>(&least);
    if (e == cudaSuccess) e = staged_limits<kModeMixed, true>(&least);
    if (e != cudaSuccess) return e;
    L->staged_blocks_per_sm = least;
  }
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_fused<S>, kOpsThreads, 0);
  if (e != cudaSuccess) return e;
  L->fused_blocks_per_sm = b > 0 ? b : 1;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_multi_ops<S>, kOpsThreads, 0);
  if (e != cudaSuccess) return e;
  L->multi_blocks_per_sm = b > 0 ? b : 1;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_overflow<S>, kOvfThreads, 0);
  if (e != cudaSuccess) return e;
  L->ovf_blocks_per_sm = b > 0 ? b : 1;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_claim<S>, kClaimThreads, 0);
  if (e != cudaSuccess) return e;
  L->claim_blocks_per_sm = b > 0 ? b : 1;
  const int smem = static_cast<int>(kMaintSmemWords * sizeof(uint64_t));
  e = cudaFuncSetAttribute(k_multi_maint<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_maint<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}
}  // namespace

cudaError_t query_occupancy(Launch* L, int S) {
  if (L->ops_threads != 128 && L->ops_threads != 512) L->ops_threads = 256;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&L->num_sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  return S == 16 ? occupancy_s<16>(L) : occupancy_s<32>(L);
}

}  // namespace hive

