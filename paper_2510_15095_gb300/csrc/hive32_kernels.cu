// Hive table with 32-bit entries (Section III-B: with 32-bit entries -- a
// key-only set, or a 16-bit key with a 16-bit value -- a 32-slot bucket is
// 128 bytes, one cache line, half the bytes of a probe of the 64-bit table).
//
// Same algorithm as the 64-bit table, fixed capacity:
//   k32_ops<MODE, LAYOUT>  bulk find / insert (steps 1-2) / erase / mixed, one
//                          op per lane by slot tags (hive_tags.cuh).
//   k32_overflow<LAYOUT>   steps 3-4: bounded cuckoo eviction under the
//                          bucket lock, warp per item (one slot per lane),
//                          then the stash.
//   k32_maint<LAYOUT>      stash maintenance: reinsert, sort by key, compact.
// The empty word is all ones; its key (0xFFFF or 0xFFFFFFFF) is reserved.
#include <cuda_runtime.h>
#include <stdint.h>

#include "hive_device.cuh"
#include "hive_internal.h"
#include "hive_tags.cuh"

namespace hive {
namespace {

constexpr int kS32 = 32;                   // slots per bucket
constexpr uint32_t kEmpty32 = 0xFFFFFFFFu;  // empty slot
constexpr int kOps32Threads = 256;
constexpr int kMaint32Threads = 1024;
constexpr unsigned kMaint32SmemWords = 16384;  // 64 KB of words sorted in shared memory

// Entry layouts.
template <int LAYOUT>
struct E32;
template <>
struct E32<HIVE32_KEY16_VAL16> {  // value << 16 | key
  static __device__ __forceinline__ uint32_t key(uint32_t w) { return w & 0xFFFFu; }
  static __device__ __forceinline__ uint32_t val(uint32_t w) { return w >> 16; }
  static __device__ __forceinline__ uint32_t pack(uint32_t k, uint32_t v) { return (v << 16) | k; }
  // keys 0xFFFE and 0xFFFF are reserved; keys and values must fit 16 bits
  static __device__ __forceinline__ bool reserved(uint32_t k, uint32_t v) {
    return k >= 0xFFFEu || v > 0xFFFFu;
  }
};
template <>
struct E32<HIVE32_KEY_ONLY> {  // the key itself
  static __device__ __forceinline__ uint32_t key(uint32_t w) { return w; }
  static __device__ __forceinline__ uint32_t val(uint32_t) { return 0u; }
  static __device__ __forceinline__ uint32_t pack(uint32_t k, uint32_t) { return k; }
  static __device__ __forceinline__ bool reserved(uint32_t k, uint32_t) { return k >= 0xFFFFFFFEu; }
};

__device__ __forceinline__ void st_relaxed32(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
struct Counters32 {
  int size_delta = 0;
  unsigned replaced = 0, claimed = 0, overflowed = 0, probes = 0;
  bool reserved = false, contract = false;
};

// Adds the counters of every warp of a block to the table with one atomic per
// non-zero counter and block.  Every thread of the block calls it.
__device__ __forceinline__ void flush32_block(const View32& v, const Counters32& c, int lane) {
  __shared__ uint64_t sums[kOps32Threads / 32][7];
  uint64_t* mine = sums[threadIdx.x >> 5];
  const int sd = __reduce_add_sync(kFull, static_cast<unsigned>(c.size_delta));
  const unsigned rp = __reduce_add_sync(kFull, c.replaced);
  const unsigned cl = __reduce_add_sync(kFull, c.claimed);
  const unsigned of = __reduce_add_sync(kFull, c.overflowed);
  const unsigned pr = __reduce_add_sync(kFull, c.probes);
  const unsigned rs = __ballot_sync(kFull, c.reserved);
  const unsigned ct = __ballot_sync(kFull, c.contract);
  if (lane == 0) {
    mine[0] = pr;
    mine[1] = static_cast<uint64_t>(static_cast<int64_t>(sd));
    mine[2] = rp;
    mine[3] = cl;
    mine[4] = of;
    mine[5] = rs ? 1u : 0u;
    mine[6] = ct ? 1u : 0u;
  }
  __syncthreads();
  const int f = threadIdx.x;
  if (f >= 7) return;
  unsigned long long sum = 0;
  for (int w = 0; w < kOps32Threads / 32; ++w) sum += sums[w][f];
  if (!sum) return;
  switch (f) {
    case 0: atomicAdd(&v.ctrl->stats[kStProbes], sum); break;
    case 1: atomicAdd(&v.ctrl->size, sum); break;
    case 2: atomicAdd(&v.ctrl->stats[kStReplaced], sum); break;
    case 3: atomicAdd(&v.ctrl->stats[kStClaimedFast], sum); break;
    case 4: atomicAdd(&v.ctrl->stats[kStOverflowed], sum); break;
    case 5: atomicOr(&v.ctrl->err, kErrReserved); break;
    default: atomicOr(&v.ctrl->err, kErrContract); break;
  }
}

// A slot's entry; `keep` as in View::keep_words (RO: no kernel writes the table
// meanwhile).
template <bool RO>
__device__ __forceinline__ uint32_t ld_entry(const uint32_t* p, bool keep) {
  uint32_t r;
  const uint64_t pol = keep ? policy_keep() : policy_pass();
  if constexpr (RO)
    asm("ld.global.nc.L2::cache_hint.b32 %0, [%1], %2;" : "=r"(r) : "l"(p), "l"(pol));
  else
    asm volatile("ld.relaxed.gpu.global.L2::cache_hint.b32 %0, [%1], %2;"
                 : "=r"(r)
                 : "l"(p), "l"(pol)
                 : "memory");
  return r;
}

// Claims (step 2): the tag makes the slot the claimer's, which publishes its
// entry with a plain store (see hive_tags.cuh).
__device__ __forceinline__ bool publish32(const View32& v, uint32_t b, uint32_t slot,
                                          uint32_t word) {
  if (slot >= kS32) return false;
  st_relaxed32(v.buckets + static_cast<uint64_t>(b) * kS32 + slot, word);
  return true;
}
__device__ __forceinline__ bool claim32_bucket(const View32& v, uint32_t b, uint32_t key,
                                               uint32_t word) {
  const TagVec<kS32> t = ld_tags_at<kS32, false>(v.tags, b);
  return publish32(v, b,
                   claim_among<kS32>(v.tags, b, t, free_slots<kS32>(t), tag_of(key),
                                     claim_rot(key)),
                   word);
}
// The bucket with more free slots first, then the other with its tags read again.
__device__ __forceinline__ bool place32_from(const View32& v, uint32_t b1, uint32_t b2,
                                             const TagVec<kS32>& t1, const TagVec<kS32>& t2,
                                             uint32_t key, uint32_t word) {
  const uint32_t m1 = free_slots<kS32>(t1), m2 = free_slots<kS32>(t2);
  const uint32_t f1 = __popc(m1), f2 = __popc(m2);
  const bool first1 = f1 >= f2;
  TagVec<kS32> t;
#pragma unroll
  for (int q = 0; q < kS32 / 4; ++q) t.w[q] = first1 ? t1.w[q] : t2.w[q];
  const uint32_t b = first1 ? b1 : b2;
  if (publish32(v, b,
                claim_among<kS32>(v.tags, b, t, first1 ? m1 : m2, tag_of(key), claim_rot(key)),
                word))
    return true;
  if (b1 == b2 || (first1 ? f2 : f1) == 0) return false;
  return claim32_bucket(v, first1 ? b2 : b1, key, word);
}
__device__ __forceinline__ bool place32(const View32& v, uint32_t b1, uint32_t b2, uint32_t key,
                                        uint32_t word) {
  const TagVec<kS32> t1 = ld_tags_at<kS32, false>(v.tags, b1);
  const TagVec<kS32> t2 = ld_tags_at<kS32, false>(v.tags, b2);
  return place32_from(v, b1, b2, t1, t2, key, word);
}

__device__ __forceinline__ bool stash32_find(const View32& v, uint32_t stash_n, uint32_t key,
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

// Acts on a found word `cur` in slot sp of bucket b (or in the stash when
// b == kNoOp): find, erase or replace.
template <int LAYOUT>
__device__ __forceinline__ void act32(const View32& v, uint32_t opk, uint32_t* sp, uint32_t b,
                                      uint32_t slot, uint32_t cur, uint32_t key, uint32_t val,
                                      uint8_t& st, uint32_t& outv, Counters32& cnt) {
  using E = E32<LAYOUT>;
  if (opk == OP_FIND) {
    outv = E::val(cur);
    st = ST_FOUND;
  } else if (opk == OP_ERASE) {
    st = ST_ERASED;
    if (atomicCAS(sp, cur, kEmpty32) == cur) {
      if (b != kNoOp)
        xor_tag<kS32>(v.tags, b, slot, tag_of(key));
      else
        atomicExch(&v.ctrl->stash_dirty, 1u);
      cnt.size_delta -= 1;
    } else {
      cnt.contract = true;
    }
  } else {
    st = ST_REPLACED;
    const uint32_t nw = E::pack(key, val);
    if (nw == cur || atomicCAS(sp, cur, nw) == cur)
      cnt.replaced += 1;
    else
      cnt.contract = true;
  }
}

// One op's inputs.
struct In32 {
  uint32_t op, key, val;
};
template <int MODE>
__device__ __forceinline__ In32 load32(const Ops32& a, uint32_t c, uint64_t n, int lane) {
  constexpr bool kIns = (MODE == kModeInsert || MODE == kModeMixed);
  const uint32_t i = (c << 5) + lane;
  const bool valid = i < n;
  In32 in;
  in.op = MODE == kModeMixed ? (valid ? static_cast<uint32_t>(__ldcs(a.ops + i)) : OP_FIND)
                             : (MODE == kModeFind    ? OP_FIND
                                : MODE == kModeErase ? OP_ERASE
                                                     : OP_INSERT);
  if (in.op > OP_ERASE) in.op = OP_FIND;
  in.key = valid ? __ldcs(a.keys + i) : 0u;
  in.val = 0;
  if (kIns && valid && in.op == OP_INSERT && a.vals) in.val = __ldcs(a.vals + i);
  return in;
}

// Appends the flagged lanes' items to the eviction list.
__device__ __forceinline__ void append32(const List32& l, int lane, bool has, uint32_t word,
                                         uint32_t idx) {
  const unsigned om = __ballot_sync(kFull, has);
  if (!om) return;
  const int leader = __ffs(om) - 1;
  unsigned base = 0;
  if (lane == leader) base = atomicAdd(l.count, static_cast<unsigned>(__popc(om)));
  base = __shfl_sync(kFull, base, leader);
  if (has) {
    const unsigned r = base + __popc(om & ((1u << lane) - 1u));
    l.words[r] = word;
    l.idx[r] = idx;
  }
}

// A warp's queue of a mixed batch's new keys, in shared memory: they wait for
// 32 of their kind, so that the claims of a batch with one insert in four
// ops are not made by a quarter of the lanes in each chunk (a set of 2^25
// slots at 90%, 2^23 ops: 387 -> 325 us; staged buckets took 365).  Their
// status is written when they are queued (INSERTED; the eviction pass writes
// it again).
// `n` is warp-uniform and below 32 between chunks.
constexpr uint32_t kNewQ32 = 64;
struct NewQ32 {
  uint32_t* words;
  uint32_t* idx;
  uint32_t n;
};

// Claims for the first min(n, 32) queued keys (warp-wide); the rest move to
// the front.
template <int LAYOUT>
__device__ __forceinline__ void claim32_queued(const View32& v, NewQ32& q, const List32& ovf,
                                               Counters32& cnt, int lane) {
  using E = E32<LAYOUT>;
  __syncwarp();
  const uint32_t m = q.n < 32 ? q.n : 32u, rest = q.n - m;
  const bool has = static_cast<uint32_t>(lane) < m;
  const uint32_t word = has ? q.words[lane] : kEmpty32;
  const uint32_t idx = has ? q.idx[lane] : kNoOp;
  uint32_t mw = 0, mi = 0;
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
    const uint32_t key = E::key(word);
    if (place32(v, lh_bucket(bithash1(key), v.M, v.p), lh_bucket(bithash2(key), v.M, v.p), key,
                word)) {
      cnt.size_delta += 1;
      cnt.claimed += 1;
    } else {
      to_ovf = true;
      cnt.overflowed += 1;
    }
  }
  append32(ovf, lane, to_ovf, word, idx);
}

// Ops [32c, 32c + 32) of a batch, one op per lane: the tags of both candidate
// buckets in one round trip, then the entries whose tag matches.  With a queue
// `q`, the new keys of a mixed batch wait there for their claims.
template <int MODE, int LAYOUT>
__device__ __forceinline__ void run_chunk32(const View32& v, uint32_t stash_n, const Ops32 a,
                                            uint32_t c, uint64_t n, const List32 ovf,
                                            Counters32& cnt, const In32& in, int lane,
                                            NewQ32* q) {
  using E = E32<LAYOUT>;
  constexpr bool kIns = (MODE == kModeInsert || MODE == kModeMixed);
  constexpr bool kRO = MODE == kModeFind;
  const uint32_t i = (c << 5) + lane;
  const bool valid = i < n;
  const uint32_t op = in.op, key = in.key, val = in.val;
  const bool reserved = valid && E::reserved(key, op == OP_INSERT ? val : 0u);
  const bool live = valid && !reserved;
  cnt.reserved |= reserved;
  const uint32_t b1 = lh_bucket(bithash1(key), v.M, v.p);
  const uint32_t b2 = lh_bucket(bithash2(key), v.M, v.p);
  bool done = !live;
  uint8_t st = reserved ? ST_RESERVED : ST_NOT_FOUND;
  uint32_t outv = 0;
  TagVec<kS32> t1, t2;
  uint32_t slot = kS32, hb = b1, cur = 0;
  if (live) {
    t1 = ld_tags_at<kS32, kRO>(v.tags, b1);
    t2 = ld_tags_at<kS32, kRO>(v.tags, b2);
    const uint32_t t4 = tag_of(key) * 0x01010101u;
    uint32_t m1 = tag_match<kS32>(t1, t4);
    uint32_t m2 = b2 != b1 ? tag_match<kS32>(t2, t4) : 0u;
    const uint32_t rot = claim_rot(key);
    while (m1 | m2) {
      const bool in1 = m1 != 0;
      const uint32_t b = in1 ? b1 : b2;
      const uint32_t p = pick_slot(in1 ? m1 : m2, rot);
      const uint32_t w = ld_entry<kRO>(v.buckets + static_cast<uint64_t>(b) * kS32 + slot_of(p),
                                       v.keep_words);
      if (E::key(w) == key) {
        slot = slot_of(p);
        hb = b;
        cur = w;
        break;
      }
      if (in1)
        m1 &= ~(1u << p);
      else
        m2 &= ~(1u << p);
    }
  }
  const bool hit = slot < kS32;
  if (MODE != kModeInsert) {
    cnt.probes += live;
    cnt.probes += live && (!hit || hb != b1);
  }
  if (hit) {
    done = true;
    act32<LAYOUT>(v, op, v.buckets + static_cast<uint64_t>(hb) * kS32 + slot, hb, slot, cur, key,
                  val, st, outv, cnt);
  }

  // the stash (step 4) holds keys that found no bucket room
  if (!done && stash_n) {
    uint32_t pos;
    if (stash32_find(v, stash_n, key, pos)) {
      const uint32_t w = ld_relaxed32(v.stash_kv + pos);
      if (w != kEmpty32 && E::key(w) == key) {
        done = true;
        act32<LAYOUT>(v, op, v.stash_kv + pos, kNoOp, 0, w, key, val, st, outv, cnt);
      }
    }
  }

  // step 2: claim for absent keys
  bool to_ovf = false;
  if (kIns && q) {
    const bool fresh = !done && op == OP_INSERT;
    const unsigned nm = __ballot_sync(kFull, fresh);
    if (fresh) {
      const uint32_t r = q->n + __popc(nm & ((1u << lane) - 1u));
      q->words[r] = E::pack(key, val);
      q->idx[r] = i;
      st = ST_INSERTED;
    }
    q->n += __popc(nm);
  } else if (kIns) {
    if (!done && op == OP_INSERT) {
      if (place32_from(v, b1, b2, t1, t2, key, E::pack(key, val))) {
        st = ST_INSERTED;
        cnt.size_delta += 1;
        cnt.claimed += 1;
      } else {
        to_ovf = true;
        cnt.overflowed += 1;
      }
    }
    append32(ovf, lane, to_ovf, E::pack(key, val), i);
  }
  if (valid) {
    if (MODE == kModeFind) {
      if (a.vals_out) __stcs(a.vals_out + i, outv);
      if (a.found) a.found[i] = st == ST_FOUND ? 1 : 0;
    } else {
      if (a.status && !to_ovf) a.status[i] = st;
      if (MODE == kModeMixed && a.vals_out) __stcs(a.vals_out + i, outv);
    }
  }
  if (kIns && q && q->n >= 32) claim32_queued<LAYOUT>(v, *q, ovf, cnt, lane);
}

// What bounds it (one GB300, a set of 2^25 slots at 90%, 128 MB of entries and
// 32 MB of tags): random accesses in L2 and, past its capacity, DRAM.  Against
// whole 128-byte buckets staged in shared memory: 30 M inserts 1.58 -> 1.09
// ms, 60 M lookups (half hits) 1.22 -> 0.86 ms and, with half the keys gone,
// 1.32 -> 0.76 ms; 15 M erases 0.46 -> 0.62 ms (the entry, its CAS and the tag
// are three dependent accesses where the old probe had two).  Mixed batches at
// four blocks per SM: five and six spill (2^26 slots, 2^24 ops: 1.20 -> 1.32 and
// 1.45 ms).
template <int MODE, int LAYOUT>
__global__ void __launch_bounds__(kOps32Threads, (MODE == kModeInsert || MODE == kModeMixed) ? 4 : 6)
    k32_ops(View32 v, Ops32 a, uint64_t n, List32 ovf, int prefetch_tags) {
  pdl_trigger();
  if (prefetch_tags) prefetch_l2_grid(v.tags, static_cast<uint64_t>(v.nb) * kS32);
  const int lane = threadIdx.x & 31;
  const uint32_t warp0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t nchunks = static_cast<uint32_t>((n + 31) >> 5);
  const uint32_t stash_n = v.ctrl->stash_n;
  Counters32 cnt;
  constexpr bool kQueue = MODE == kModeMixed;
  __shared__ uint32_t queue[kQueue ? (kOps32Threads / 32) * 2 * kNewQ32 : 1];
  uint32_t* mine = queue + (kQueue ? (threadIdx.x >> 5) * 2 * kNewQ32 : 0);
  NewQ32 nq{mine, mine + kNewQ32, 0};
  // one chunk per warp: claim at once, with the tags at hand
  NewQ32* const q = kQueue && nchunks > nwarps ? &nq : nullptr;
  // inputs are loaded one chunk ahead
  In32 nxt{};
  if (warp0 < nchunks) nxt = load32<MODE>(a, warp0, n, lane);
  for (uint32_t c = warp0; c < nchunks; c += nwarps) {
    const In32 in = nxt;
    if (c + nwarps < nchunks) nxt = load32<MODE>(a, c + nwarps, n, lane);
    run_chunk32<MODE, LAYOUT>(v, stash_n, a, c, n, ovf, cnt, in, lane, q);
  }
  if constexpr (kQueue)
    while (nq.n) claim32_queued<LAYOUT>(v, nq, ovf, cnt, lane);
  // an insert examines both buckets of every live op, which ends in one of these
  if (MODE == kModeInsert) cnt.probes = 2 * (cnt.replaced + cnt.claimed + cnt.overflowed);
  flush32_block(v, cnt, lane);
}

// ---- steps 3-4 -------------------------------------------------------------

struct Ovf32 {
  unsigned claim = 0, rounds = 0, locks = 0, to = 0, stash = 0, pend = 0, added = 0;
  bool reserved = false;
};

__device__ __forceinline__ bool lock32(const View32& v, uint32_t b) {
  for (uint32_t t = 0; t < v.lock_spin_limit; ++t) {
    if (atomicCAS(v.locks + b, 0u, 1u) == 0u) return true;
    __nanosleep(64);
  }
  return false;
}
__device__ __forceinline__ bool stash32_reserve(const View32& v) {
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

// One overflowing insert, warp-wide (lane i holds slot i of the bucket in
// hand).  Mirrors the 64-bit eviction kernel: claim, else a bounded chain of
// locked exchanges with a lookahead victim, else the stash, else FULL.
template <int LAYOUT>
__device__ __forceinline__ void overflow32_item(const View32& v, uint32_t word0, uint32_t idx,
                                                uint8_t* status, Ovf32& oc, int lane) {
  using E = E32<LAYOUT>;
  const uint32_t key0 = E::key(word0);
  const uint32_t b1 = lh_bucket(bithash1(key0), v.M, v.p);
  const uint32_t b2 = lh_bucket(bithash2(key0), v.M, v.p);
  int outcome = 0;  // 0: evict, 1: placed, 2: stashed, 3: no room
  if (lane == 0) {
    if (place32(v, b1, b2, key0, word0)) {
      outcome = 1;
      ++oc.claim;
    } else {
      if (!oc.reserved) oc.reserved = stash32_reserve(v);
      if (!oc.reserved) outcome = 3;
    }
  }
  outcome = __shfl_sync(kFull, outcome, 0);
  if (outcome == 0) {
    uint32_t cur = word0, b = b1;
    bool placed = false;
    for (uint32_t r = 0; r < v.max_evictions; ++r) {
      const uint32_t w = ld_relaxed32(v.buckets + static_cast<uint64_t>(b) * kS32 + lane);
      // a free slot of this entry's other candidate bucket (32: none), and
      // the tag word it lies in
      uint32_t ap = 32, aw = 0;
      if (w != kEmpty32) {
        const uint32_t k = E::key(w);
        const uint32_t a1 = lh_bucket(bithash1(k), v.M, v.p);
        const uint32_t a2 = lh_bucket(bithash2(k), v.M, v.p);
        const uint32_t alt = (a1 == b) ? a2 : a1;
        if (alt != b) {
          const TagVec<kS32> ta = ld_tags_at<kS32, false>(v.tags, alt);
          const uint32_t fm = free_slots<kS32>(ta);
          if (fm) {
            ap = pick_slot(fm, claim_rot(k));
            aw = tag_sel<kS32>(ta, ap & 7u);
          }
        }
      }
      const unsigned gm = __ballot_sync(kFull, ap < 32u);
      const unsigned occ = __ballot_sync(kFull, w != kEmpty32);
      const bool has_empty = occ != kFull;
      // victim: an occupied slot whose entry can move on at once, else an
      // occupied slot picked by rotation (never an EMPTY one: its claimer
      // publishes with a plain store; occupied slots stay occupied here)
      uint32_t vs = kS32;
      if (gm)
        vs = __ffs(gm) - 1;
      else if (occ)
        vs = pick_slot(occ, (bithash2(E::key(cur)) + r) & (kS32 - 1));
      const uint32_t vp = __shfl_sync(kFull, ap, vs & (kS32 - 1));
      const uint32_t vw = __shfl_sync(kFull, aw, vs & (kS32 - 1));
      int res = 0;
      uint32_t victim = kEmpty32;
      if (lane == 0) {
        ++oc.rounds;
        if (!lock32(v, b)) {
          res = 2;
          ++oc.to;
        } else {
          ++oc.locks;
          if (has_empty && claim32_bucket(v, b, E::key(cur), cur)) {
            res = 1;
          } else if (vs >= kS32) {
            res = 3;  // every slot claimed but not yet published: look again
          } else {
            victim = atomicExch(v.buckets + static_cast<uint64_t>(b) * kS32 + vs, cur);
            xor_tag<kS32>(v.tags, b, vs, tag_of(E::key(victim)) ^ tag_of(E::key(cur)));
            fence_acq_rel_gpu();  // the tag change comes before the unlock
          }
          atomicExch(v.locks + b, 0u);
        }
      }
      res = __shfl_sync(kFull, res, 0);
      victim = __shfl_sync(kFull, victim, 0);
      if (res == 1) {
        placed = true;
        break;
      }
      if (res == 2) break;
      if (res == 3) continue;
      cur = victim;
      const uint32_t kc = E::key(cur);
      const uint32_t a1 = lh_bucket(bithash1(kc), v.M, v.p);
      const uint32_t a2 = lh_bucket(bithash2(kc), v.M, v.p);
      const uint32_t nb = (a1 == b) ? a2 : a1;
      if (nb == b) break;
      b = nb;
      int ok = 0;
      if (lane == 0)
        ok = vp < 32u ? publish32(v, b,
                                  claim_tag<kS32>(v.tags, b, vp & 7u, vp >> 3, vw, tag_of(kc)), cur)
                      : claim32_bucket(v, b, kc, cur);
      if (__shfl_sync(kFull, ok, 0)) {
        placed = true;
        break;
      }
    }
    if (lane == 0) {
      if (placed && oc.reserved && ld_relaxed32(&v.ctrl->stash_claims) >= v.stash_cap) {
        atomicSub(&v.ctrl->stash_claims, 1u);
        oc.reserved = false;
      }
      if (!placed) {
        oc.reserved = false;
        const unsigned pos = atomicAdd(&v.ctrl->stash_tail, 1u);
        st_relaxed32(v.stash_kv + pos, cur);
        ++oc.stash;
      }
    }
    outcome = placed ? 1 : 2;
  }
  if (lane == 0) {
    if (outcome == 3) {
      ++oc.pend;
      atomicOr(&v.ctrl->err, kErrFull);
      if (status) status[idx] = ST_FULL;
    } else {
      ++oc.added;
      if (status) status[idx] = ST_INSERTED;
    }
  }
}

template <int LAYOUT>
__global__ void __launch_bounds__(256) k32_overflow(View32 v, List32 in, uint8_t* status) {
  pdl_trigger();
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const unsigned warp0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const unsigned nwarps = (gridDim.x * blockDim.x) >> 5;
  const unsigned total = *in.count;
  Ovf32 oc;
  for (unsigned it = warp0; it < total; it += nwarps)
    overflow32_item<LAYOUT>(v, in.words[it], in.idx[it], status, oc, lane);
  if (lane == 0) {
    Ctrl* c = v.ctrl;
    if (oc.reserved) atomicSub(&c->stash_claims, 1u);
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
}

// ---- stash maintenance (single CTA) -----------------------------------------

template <int LAYOUT>
__device__ __forceinline__ uint64_t sort_key32(uint32_t w) {
  // EMPTY sorts last
  return w == kEmpty32 ? ~0ull : static_cast<uint64_t>(E32<LAYOUT>::key(w));
}

template <int LAYOUT>
__device__ void bitonic32(uint32_t* a, unsigned P) {
  for (unsigned k = 2; k <= P; k <<= 1) {
    for (unsigned j = k >> 1; j > 0; j >>= 1) {
      for (unsigned t = threadIdx.x; t < (P >> 1); t += blockDim.x) {
        const unsigned low = t & (j - 1);
        const unsigned i = ((t - low) << 1) | low;
        const unsigned l = i | j;
        const uint32_t x = a[i], y = a[l];
        const bool up = (i & k) == 0;
        if ((sort_key32<LAYOUT>(x) > sort_key32<LAYOUT>(y)) == up) {
          a[i] = y;
          a[l] = x;
        }
      }
      __syncthreads();
    }
  }
}

template <int LAYOUT>
__global__ void __launch_bounds__(kMaint32Threads) k32_maint(View32 v) {
  extern __shared__ uint32_t smem_m32[];
  pdl_wait();
  using E = E32<LAYOUT>;
  __shared__ unsigned s_reins, s_live;
  Ctrl* c = v.ctrl;
  const unsigned tail = c->stash_tail;
  const unsigned sorted = c->stash_n;
  const unsigned dirty = c->stash_dirty;
  if (threadIdx.x == 0) {
    s_reins = 0;
    s_live = 0;
    c->ovf_n = 0;
  }
  __syncthreads();
  if (tail == sorted && !dirty) return;
  unsigned reins = 0;
  for (unsigned j = threadIdx.x; j < tail; j += blockDim.x) {
    const uint32_t w = v.stash_kv[j];
    if (w == kEmpty32) continue;
    const uint32_t k = E::key(w);
    const uint32_t b1 = lh_bucket(bithash1(k), v.M, v.p);
    const uint32_t b2 = lh_bucket(bithash2(k), v.M, v.p);
    if (place32(v, b1, b2, k, w)) {
      v.stash_kv[j] = kEmpty32;
      ++reins;
    }
  }
  if (reins) atomicAdd(&s_reins, reins);
  __syncthreads();
  unsigned P = 1;
  while (P < tail) P <<= 1;
  if (P <= kMaint32SmemWords) {
    for (unsigned j = threadIdx.x; j < P; j += blockDim.x)
      smem_m32[j] = j < tail ? v.stash_kv[j] : kEmpty32;
    __syncthreads();
    bitonic32<LAYOUT>(smem_m32, P);
    for (unsigned j = threadIdx.x; j < P; j += blockDim.x) v.stash_kv[j] = smem_m32[j];
  } else {
    bitonic32<LAYOUT>(v.stash_kv, P);  // [tail, P) is EMPTY by construction
  }
  __syncthreads();
  unsigned live = 0;
  for (unsigned j = threadIdx.x; j < P; j += blockDim.x) {
    const uint32_t w = v.stash_kv[j];
    if (w != kEmpty32) {
      v.stash_keys[j] = E::key(w);
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

// Resident blocks per SM of each bulk kernel, per layout and mode (set once
// per process by setup32; every GPU of the machine is the same model).
int g_occ32[2][4] = {{1, 1, 1, 1}, {1, 1, 1, 1}};

template <int MODE, int LAYOUT>
cudaError_t launch32_t(const View32& v, const Ops32& a, uint64_t n, const List32& ovf,
                       int num_sms, cudaStream_t s) {
  const uint64_t chunks = (n + 31) / 32;
  uint64_t blocks = (chunks + (kOps32Threads / 32) - 1) / (kOps32Threads / 32);
  const uint64_t cap = static_cast<uint64_t>(num_sms) * g_occ32[LAYOUT][MODE];
  if (blocks > cap) blocks = cap;
  if (blocks == 0) blocks = 1;
  k32_ops<MODE, LAYOUT><<<static_cast<unsigned>(blocks), kOps32Threads, 0, s>>>(
      v, a, n, ovf, prefetch_tags_rule(n, v.nb, kS32));
  return cudaGetLastError();
}

template <int LAYOUT>
cudaError_t launch32_l(int mode, const View32& v, const Ops32& a, uint64_t n, const List32& ovf,
                       int num_sms, cudaStream_t s) {
  switch (mode) {
    case kModeFind:
      return launch32_t<kModeFind, LAYOUT>(v, a, n, ovf, num_sms, s);
    case kModeInsert:
      return launch32_t<kModeInsert, LAYOUT>(v, a, n, ovf, num_sms, s);
    case kModeErase:
      return launch32_t<kModeErase, LAYOUT>(v, a, n, ovf, num_sms, s);
    default:
      return launch32_t<kModeMixed, LAYOUT>(v, a, n, ovf, num_sms, s);
  }
}

template <int MODE, int LAYOUT>
cudaError_t setup32_mode() {
  int b = 0;
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      &b, k32_ops<MODE, LAYOUT>, kOps32Threads, 0);
  g_occ32[LAYOUT][MODE] = b > 0 ? b : 1;
  return e;
}

template <int LAYOUT>
cudaError_t setup32_l(int* blocks_per_sm) {
  cudaError_t e = setup32_mode<kModeFind, LAYOUT>();
  if (e == cudaSuccess) e = setup32_mode<kModeInsert, LAYOUT>();
  if (e == cudaSuccess) e = setup32_mode<kModeErase, LAYOUT>();
  if (e == cudaSuccess) e = setup32_mode<kModeMixed, LAYOUT>();
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k32_maint<LAYOUT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(kMaint32SmemWords * 4));
  *blocks_per_sm = g_occ32[LAYOUT][kModeInsert];
  return e;
}

}  // namespace

cudaError_t launch32_ops(int mode, const View32& v, const Ops32& a, uint64_t n, const List32& ovf,
                         int num_sms, cudaStream_t s) {
  return v.layout == HIVE32_KEY_ONLY
             ? launch32_l<HIVE32_KEY_ONLY>(mode, v, a, n, ovf, num_sms, s)
             : launch32_l<HIVE32_KEY16_VAL16>(mode, v, a, n, ovf, num_sms, s);
}

cudaError_t launch32_overflow(const View32& v, const List32& in, uint8_t* status, int blocks,
                              cudaStream_t s) {
  if (v.layout == HIVE32_KEY_ONLY)
    return launch_dependent(k32_overflow<HIVE32_KEY_ONLY>, blocks, 256, 0, s, v, in, status);
  return launch_dependent(k32_overflow<HIVE32_KEY16_VAL16>, blocks, 256, 0, s, v, in, status);
}

cudaError_t launch32_maint(const View32& v, cudaStream_t s) {
  const size_t smem = kMaint32SmemWords * 4;
  if (v.layout == HIVE32_KEY_ONLY)
    return launch_dependent(k32_maint<HIVE32_KEY_ONLY>, 1, kMaint32Threads, smem, s, v);
  return launch_dependent(k32_maint<HIVE32_KEY16_VAL16>, 1, kMaint32Threads, smem, s, v);
}

cudaError_t setup32(int layout, int* blocks_per_sm) {
  return layout == HIVE32_KEY_ONLY ? setup32_l<HIVE32_KEY_ONLY>(blocks_per_sm)
                                   : setup32_l<HIVE32_KEY16_VAL16>(blocks_per_sm);
}

}  // namespace hive
