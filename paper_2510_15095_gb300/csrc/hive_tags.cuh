// Slot tags: the one-byte filter and free mask of every slot, shared by the
// tables with 64-bit and with 32-bit entries.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "hive_device.cuh"

namespace hive {
namespace {

// Each slot has a one-byte tag in an array of its own: 0 while the slot is
// free, else a byte in [1, 255] computed from the slot's key.  The S tags of
// a bucket are 32 (S = 32) or 16 (S = 16) bytes, at most one memory sector,
// so a lookup reads one sector per candidate bucket and then only the words
// whose tag matches: one word for a hit, and one in about 255 / S buckets for
// a false match.  Random reads bound every bulk kernel here: measured on one
// GB300, DRAM serves 40-50 G random accesses/s whether each moves 32 or 128
// bytes, L2 serves 290 G/s of 32-byte sectors, and the tags of a 2^26-slot
// table (64 MB) fit in L2 where its words (512 MB) do not.
//
// The tags are also the authority on free slots (WABC, Section III-E): a
// claim is one CAS that replaces a zero byte of a tag word by the key's tag,
// and the claimer then owns the slot and publishes the word with a plain
// store.  Every later change of a tag byte is an XOR with (old tag ^ new
// tag), so changes of neighbouring slots in one tag word never undo each
// other.  A chain that swaps a word lets its XOR reach memory before it
// unlocks the bucket (transient sums of two pending XORs could read as 0).
// At the end of every kernel a slot is EMPTY iff its tag is 0.

__device__ __forceinline__ uint32_t tag_of(uint32_t key) {
  // the high bits of a multiplicative hash, independent of the bucket bits
  return 1u + __umulhi(key * 0x9E3779B1u, 255u);
}

template <int S>
struct TagVec {
  uint32_t w[S / 4];
};

// L2 priorities: tags stay (every op reads 2 S bytes of them); words stay or go
// first as View::keep_words says (an op reads one of 8 bytes, and in a table
// beyond L2 the next op that wants its line is far away).  Measured: lookups
// on 2^26 slots 1.77 -> 1.51 ms with the words sent first, bulk load 4.08 ->
// 3.67 ms and a resize stream's bulk kernel 870 -> 582 us with the tags kept.
__device__ __forceinline__ uint64_t policy_keep() {
  uint64_t p;
  asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t policy_pass() {
  uint64_t p;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}

// Whether a batch of n ops on nb buckets first asks L2 for the whole tag array
// in sequential pieces: when its probes would touch about every second bucket
// or more, and while L2 (129 MB) holds the tags beside the words.  Asked for ->
// left to the probes, 2^22 ops: lookups on 2^26 slots, 64 MB of tags, level
// (S = 16 81.4 -> 80.1 us, S = 32 88.7 -> 88.4); with 128 MB of tags (2^27
// slots) and 256 MB, lookups S = 16 151 -> 145 us and 231 -> 204, S = 32
// 157 -> 150 and 238 -> 211, 32-bit entries 157 -> 151 and 238 -> 210, mixed
// ops S = 16 1056 -> 1042 and 971 -> 930.
inline bool prefetch_tags_rule(uint64_t n, uint64_t nb, uint64_t slots_per_bucket) {
  return n * 4 >= nb && nb * slots_per_bucket <= (96ull << 20);
}

// The tags of bucket b.  RO: through the read-only path (no kernel writes
// tags meanwhile); otherwise a relaxed load, which never returns a stale
// cached copy.
template <int S, bool RO>
__device__ __forceinline__ TagVec<S> ld_tags_at(const uint32_t* tags, uint32_t b) {
  TagVec<S> t;
  const uint32_t* p = tags + static_cast<uint64_t>(b) * (S / 4);
  const uint64_t pol = policy_keep();
  if constexpr (S == 32) {
    if constexpr (RO)
      asm("ld.global.nc.L2::cache_hint.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8], %9;"
          : "=r"(t.w[0]), "=r"(t.w[1]), "=r"(t.w[2]), "=r"(t.w[3]), "=r"(t.w[4]), "=r"(t.w[5]),
            "=r"(t.w[6]), "=r"(t.w[7])
          : "l"(p), "l"(pol));
    else
      asm volatile(
          "ld.relaxed.gpu.global.L2::cache_hint.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8], %9;"
          : "=r"(t.w[0]), "=r"(t.w[1]), "=r"(t.w[2]), "=r"(t.w[3]), "=r"(t.w[4]), "=r"(t.w[5]),
            "=r"(t.w[6]), "=r"(t.w[7])
          : "l"(p), "l"(pol)
          : "memory");
  } else {
    if constexpr (RO)
      asm("ld.global.nc.L2::cache_hint.v4.b32 {%0, %1, %2, %3}, [%4], %5;"
          : "=r"(t.w[0]), "=r"(t.w[1]), "=r"(t.w[2]), "=r"(t.w[3])
          : "l"(p), "l"(pol));
    else
      asm volatile("ld.relaxed.gpu.global.L2::cache_hint.v4.b32 {%0, %1, %2, %3}, [%4], %5;"
                   : "=r"(t.w[0]), "=r"(t.w[1]), "=r"(t.w[2]), "=r"(t.w[3])
                   : "l"(p), "l"(pol)
                   : "memory");
  }
  return t;
}

// 0x80 in every byte of x that is zero (exact in every byte; this and the
// shorter test in tag_match are the usual byte-parallel zero tests).
__device__ __forceinline__ uint32_t zero_bytes(uint32_t x) {
  return ~(((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x | 0x7F7F7F7Fu);
}

// Slot sets are 32-bit masks in tag order: bit 8 j + q stands for byte j of
// tag word q, which is slot 4 q + j.  Consecutive bits lie in different tag
// words, so claims that start at different bits rarely meet in one word.
__device__ __forceinline__ uint32_t slot_of(uint32_t p) { return ((p & 7u) << 2) | (p >> 3); }

// Slots that may hold the tag in all four bytes of `t4`: every slot whose tag
// equals it, and possibly the slot after one of these when its tag differs
// from it in the lowest bit only (the borrow of the byte below reaches it).
// One operation less per tag word than the exact test; a lookup compares
// the words' keys anyway.
template <int S>
__device__ __forceinline__ uint32_t tag_match(const TagVec<S>& t, uint32_t t4) {
  uint32_t m = 0;
#pragma unroll
  for (int q = 0; q < S / 4; ++q) {
    const uint32_t x = t.w[q] ^ t4;
    m = (m >> 1) + ((x - 0x01010101u) & ~x & 0x80808080u);
  }
  return S == 32 ? m : m >> 4;
}
// Slots whose tag is 0 (exact: a claim may only take a zero byte).
template <int S>
__device__ __forceinline__ uint32_t free_slots(const TagVec<S>& t) {
  uint32_t m = 0;
#pragma unroll
  for (int q = 0; q < S / 4; ++q) m = (m >> 1) + zero_bytes(t.w[q]);
  return S == 32 ? m : m >> 4;
}

// The first set bit of slot set m at or after bit `rot`, cyclically (m != 0).
__device__ __forceinline__ uint32_t pick_slot(uint32_t m, uint32_t rot) {
  return (__ffs(__funnelshift_r(m, m, rot)) - 1 + rot) & 31u;
}
// Tag word q of t, for q known only at run time.
template <int S>
__device__ __forceinline__ uint32_t tag_sel(const TagVec<S>& t, uint32_t q) {
  uint32_t x = t.w[0];
#pragma unroll
  for (int k = 1; k < S / 4; ++k)
    if (q == k) x = t.w[k];
  return x;
}

// Where a key's claims start in a bucket: spreads the claims of concurrent
// inserts into one bucket over its tag words.
__device__ __forceinline__ uint32_t claim_rot(uint32_t key) { return (key * 0x85EBCA6Bu) >> 27; }

// Claims a free byte of tag word q of bucket b for `tag`, where the word was
// last seen as `cur` with byte j zero.  Returns the slot, or S when the word
// has filled up.  Algorithm 2 restores its bit when it loses the race; here a
// lost CAS changes nothing, and the claim goes on from the value the CAS
// returned.  A CAS fails only because another op of the batch changed the
// word, so the loop ends.
template <int S>
__device__ __forceinline__ uint32_t claim_tag(uint32_t* tags, uint32_t b, uint32_t q, uint32_t j,
                                              uint32_t cur, uint32_t tag) {
  uint32_t* tw = tags + static_cast<uint64_t>(b) * (S / 4) + q;
  for (;;) {
    const uint32_t old = atomicCAS(tw, cur, cur | (tag << (8 * j)));
    if (old == cur) return 4 * q + j;
    const uint32_t z = zero_bytes(old);
    if (!z) return S;
    cur = old;
    j = (__ffs(z) - 1) >> 3;
  }
}
// Claims a slot of bucket b for a key with tag `tag` among the free slots
// `fm` of its tags `t`, read moments ago (the CAS is the authority), starting
// at bit `rot`.  Returns the slot or S.
template <int S>
__device__ __forceinline__ uint32_t claim_among(uint32_t* tags, uint32_t b, const TagVec<S>& t,
                                                uint32_t fm, uint32_t tag, uint32_t rot) {
  while (fm) {
    const uint32_t p = pick_slot(fm, rot);
    const uint32_t q = p & 7u;
    const uint32_t slot = claim_tag<S>(tags, b, q, p >> 3, tag_sel<S>(t, q), tag);
    if (slot < S) return slot;
    fm &= ~(0x01010101u << q);  // that word is full now
  }
  return S;
}

// The tag word of a slot, and the XOR that changes its tag by `d` (a tag, to
// free the slot of a key whose word the caller has just emptied, or the XOR of
// an old and a new tag).
template <int S>
__device__ __forceinline__ void xor_tag(uint32_t* tags, uint32_t b, uint32_t slot, uint32_t d) {
  if (d) atomicXor(tags + static_cast<uint64_t>(b) * (S / 4) + (slot >> 2), d << (8 * (slot & 3u)));
}

}  // namespace
}  // namespace hive
