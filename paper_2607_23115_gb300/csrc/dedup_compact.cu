// First-occurrence resolution, stream compaction, packing and insertion for
// one dedup call over one or more payloads (paper Sec. 4.1.2: a chunk that is
// not resident travels in full and becomes reusable).
//
// The result must equal deciding the chunks one at a time, payload after
// payload, in ascending order.  Given the probe/verify outcome against the
// cache as it was when the call started (kHit0 or not), that rule reduces to:
//   * any other chunk is a hit iff an earlier chunk of the call has the same
//     length and bytes; its leader is the first such chunk;
//   * the misses are the leaders, inserted in ascending order at
//     slot = slots_used + rank;
//   * a hit on a leader from an earlier payload is, for its own payload, a hit
//     on the cache (that payload's call would have found the insert);
//   * a leader counts as a verify reject iff the cache had a key+length
//     candidate for it, or an earlier leader of the call has its key+length.
//
// Two launches follow the hash kernel of a batch, a large call, and a call of a
// KEY16 or evicting cache.  k_dedup, cooperative or on few blocks, with phases
// separated by bounded grid barriers:
//   A  outputs are cleared; every non-resident chunk claims the entry of its
//      (key, length) in a per-call table and posts its number as the group
//      minimum;
//   B  each unresolved chunk compares itself (whole warp, 16-byte loads) with
//      its group's minimum: equal -> duplicate, number == minimum -> leader
//      of this round, else it stays for the next round (different bytes under
//      one key: a true 64-bit collision, or KEY16 test mode);
//   C  group minima of the remaining chunks are reset and re-posted (A);
//   D  leaders are counted per contiguous block range; the exclusive rank of
//      every chunk (and of every stored miss) follows from the block totals
//      plus warp ballots.
// k_pack, a regular launch of one wave, then writes hit masks, miss indices,
// chunk slots and per-payload counters, copies every miss by rank to the
// packed output and its arena slot and inserts it into the index; its last
// block publishes the counters and results and leaves the per-call state
// zeroed for the next call.  Where no chunk missed, k_dedup publishes itself.
//
// One launch follows it for another call of one payload that is not large:
// k_resolve_direct (k_resolve_pack for paper identifiers), which does all of
// that.
//
// A call with few, short chunks runs instead as one single-block kernel,
// k_small_call: the staged hash, then k_dedup's and k_pack's steps with a
// grid of one block (every grid barrier a block barrier), so that the call
// costs one launch and no kernel boundary.
#include <algorithm>

#include "gleam_internal.cuh"
#include "staged_hash.cuh"

namespace gleam {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
#ifndef GLEAM_COPY_VEC
#define GLEAM_COPY_VEC 8
#endif
#ifndef GLEAM_DEDUP_BLOCKS_PER_SM
#define GLEAM_DEDUP_BLOCKS_PER_SM 3
#endif
#ifndef GLEAM_DEDUP_CHUNKS_PER_BLOCK
#define GLEAM_DEDUP_CHUNKS_PER_BLOCK 1024
#endif
#ifndef GLEAM_CHAIN_PREFETCH
#define GLEAM_CHAIN_PREFETCH 1
#endif
#ifndef GLEAM_PACK_MINBLOCKS
#define GLEAM_PACK_MINBLOCKS 3
#endif
#if GLEAM_PACK_MINBLOCKS > 1
#define GLEAM_PACK_BOUNDS __launch_bounds__(kThreads, GLEAM_PACK_MINBLOCKS)
#else
#define GLEAM_PACK_BOUNDS __launch_bounds__(kThreads)
#endif
constexpr int kCopyVec = GLEAM_COPY_VEC;  // 16-byte vectors per lane in flight while copying
// In-call duplicates of at most this many bytes are compared kSmallCmpWays at a time.
#ifndef GLEAM_SMALL_CMP_WAYS
#define GLEAM_SMALL_CMP_WAYS 2
#endif
constexpr uint32_t kSmallCmpBytes = 1024;
constexpr uint32_t kSmallCmpWays = GLEAM_SMALL_CMP_WAYS;

__device__ __forceinline__ uint32_t ldcg_u32(const uint32_t* p) { return __ldcg(p); }

__device__ __forceinline__ bool differ16(uint4 x, uint4 y) {
  return (x.x != y.x) | (x.y != y.y) | (x.z != y.z) | (x.w != y.w);
}

// Bytes [m, m + 16) of the 32 bytes a, b (m < 16).
__device__ __forceinline__ uint4 shifted16(uint4 a, uint4 b, uint32_t m) {
  uint32_t y0, y1, y2, y3, y4;
  switch (m >> 2) {
    case 0: y0 = a.x, y1 = a.y, y2 = a.z, y3 = a.w, y4 = b.x; break;
    case 1: y0 = a.y, y1 = a.z, y2 = a.w, y3 = b.x, y4 = b.y; break;
    case 2: y0 = a.z, y1 = a.w, y2 = b.x, y3 = b.y, y4 = b.z; break;
    default: y0 = a.w, y1 = b.x, y2 = b.y, y3 = b.z, y4 = b.w; break;
  }
  const uint32_t r = (m & 3) * 8;
  return make_uint4(__funnelshift_r(y0, y1, r), __funnelshift_r(y1, y2, r),
                    __funnelshift_r(y2, y3, r), __funnelshift_r(y3, y4, r));
}

// The 16 bytes at p of any alignment, by the aligned 16-byte pieces that hold
// them (both must be readable).
__device__ __forceinline__ uint4 load16_any(const uint8_t* p) {
  const uint32_t m = (uint32_t)((uintptr_t)p & 15);
  const uint4* a = reinterpret_cast<const uint4*>(p - m);
  if (m == 0) return __ldg(a);
  return shifted16(__ldg(a), __ldg(a + 1), m);
}

// warp_equal for chunks of any alignment: 16 bytes at a time put together from
// aligned pieces (load16_any) where those lie inside both chunks, the bytes at
// either end one by one.  Out of line.
__device__ __noinline__ bool warp_equal_any(const uint8_t* x, const uint8_t* y, uint32_t len) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t k_lo = 1, k_hi = len < 32 ? 1u : (len - 16) >> 4;  // 16-byte steps [k_lo, k_hi)
  bool diff = false;
  for (uint32_t k0 = k_lo; k0 < k_hi; k0 += 64) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const uint32_t k = k0 + r * 32 + lane;
      if (k < k_hi) diff |= differ16(load16_any(x + 16ull * k), load16_any(y + 16ull * k));
    }
    if (__any_sync(0xffffffffu, diff)) return false;
  }
  for (uint32_t k = lane; k < min(len, 16u * k_lo); k += 32) diff |= (x[k] != y[k]);
  for (uint32_t k = 16 * k_hi + lane; k < len; k += 32) diff |= (x[k] != y[k]);
  return !__any_sync(0xffffffffu, diff);
}

// Whole-warp byte equality of two chunks.
__device__ bool warp_equal(const uint8_t* x, const uint8_t* y, uint32_t len) {
  if ((((uintptr_t)x | (uintptr_t)y) & 15) != 0) return warp_equal_any(x, y, len);
  const uint32_t lane = threadIdx.x & 31;
  bool diff = false;
  const uint32_t nv = len >> 4;
  const uint4* xv = reinterpret_cast<const uint4*>(x);
  const uint4* yv = reinterpret_cast<const uint4*>(y);
  for (uint32_t k0 = 0; k0 < nv; k0 += 128) {
    uint4 u[4], w[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const uint32_t k = k0 + r * 32 + lane;
      if (k < nv) {
        u[r] = __ldcs(xv + k);
        w[r] = __ldcs(yv + k);
      } else {
        u[r] = make_uint4(0, 0, 0, 0);
        w[r] = u[r];
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) diff |= differ16(u[r], w[r]);
    if (__any_sync(0xffffffffu, diff)) return false;
  }
  for (uint32_t k = (nv << 4) + lane; k < len; k += 32) diff |= (x[k] != y[k]);
  return !__any_sync(0xffffffffu, diff);
}

// Whole-warp copy of len bytes at s to d1 and, if not null, to d2, in 16-byte
// stores put together from the aligned 16-byte pieces of the payload that
// hold them; s of any alignment, d1 and d2 of one alignment.  The bytes
// before d1's first 16-byte boundary, and those at the payload's ends whose
// pieces reach past it, go one by one.  Byte by byte throughout, the copies of
// 26 MB of misses at 8-byte alignment took 1,035 us of a 1,489 us call (40
// payloads, 260 MB, a tenth of their 16 KiB chunks changed); the second load
// of each lane is its neighbour's first, so it comes from L1.
__device__ __noinline__ void warp_copy_any(uint8_t* d1, uint8_t* d2, const uint8_t* s,
                                           uint32_t len, const PayloadDesc& P) {
  const uint8_t *lo = P.buf, *hi = P.buf + P.n;
  const uint32_t lane = threadIdx.x & 31;
  uint32_t head = (uint32_t)(0 - (uintptr_t)d1) & 15u;
  const uint32_t m = (uint32_t)((uintptr_t)(s + head) & 15);
  if (m && s + head - m < lo) head += 16;
  uint32_t nv = len > head ? (len - head) >> 4 : 0u;
  if (nv && m && s + head - m + 16ull * nv + 16 > hi) --nv;
  const uint32_t tail = min(len, head) + (nv << 4);
  for (uint32_t k0 = 0; k0 < nv; k0 += 128) {
    uint4 u[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const uint32_t k = k0 + r * 32 + lane;
      if (k < nv) u[r] = load16_any(s + head + 16ull * k);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const uint32_t k = k0 + r * 32 + lane;
      if (k < nv) {
        __stcs(reinterpret_cast<uint4*>(d1 + head) + k, u[r]);
        if (d2) __stcs(reinterpret_cast<uint4*>(d2 + head) + k, u[r]);
      }
    }
  }
  auto bytes = [&](uint32_t k0, uint32_t k1) {
    for (uint32_t k = k0 + lane; k < k1; k += 32) {
      const uint8_t b = s[k];
      d1[k] = b;
      if (d2) d2[k] = b;
    }
  };
  bytes(0, min(len, head));
  bytes(tail, len);
}

// Whole-warp copy of a piece of a chunk to the packed output and to its arena
// slot (d2 == nullptr: to the packed output only).  The path of copies that cannot
// be bulk copies (host or managed memory, unaligned addresses): out of line,
// away from the code that every call runs.  P: the piece's payload.
__device__ __noinline__ void warp_copy2(uint8_t* d1, uint8_t* d2, const uint8_t* s, uint32_t len,
                                        const PayloadDesc& P) {
  if ((((uintptr_t)d1 | (uintptr_t)d2 | (uintptr_t)s) & 15) != 0) {
    const bool apart = d2 && (((uintptr_t)d1 ^ (uintptr_t)d2) & 15) != 0;
    warp_copy_any(d1, apart ? nullptr : d2, s, len, P);
    if (apart) warp_copy_any(d2, nullptr, s, len, P);
    return;
  }
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t nv = len >> 4;
  const uint4* sv = reinterpret_cast<const uint4*>(s);
  uint4* d1v = reinterpret_cast<uint4*>(d1);
  uint4* d2v = reinterpret_cast<uint4*>(d2);
  for (uint32_t k0 = 0; k0 < nv; k0 += 32 * kCopyVec) {
    uint4 u[kCopyVec];
#pragma unroll
    for (int r = 0; r < kCopyVec; ++r) {
      const uint32_t k = k0 + r * 32 + lane;
      if (k < nv) u[r] = __ldg(sv + k);
    }
#pragma unroll
    for (int r = 0; r < kCopyVec; ++r) {
      const uint32_t k = k0 + r * 32 + lane;
      if (k < nv) {
        __stcs(d1v + k, u[r]);
        if (d2) __stcs(d2v + k, u[r]);
      }
    }
  }
  for (uint32_t k = (nv << 4) + lane; k < len; k += 32) {
    const uint8_t b = s[k];
    d1[k] = b;
    if (d2) d2[k] = b;
  }
}

// ---- bulk asynchronous copies (k_pack's miss copies) -------------------------
//
// Lane 0 of a warp moves the warp's misses through kPackBufs shared-memory
// buffers of kPackPiece bytes: a bulk copy (the TMA engine, no registers)
// brings a piece in and signals an mbarrier with its byte count, then two bulk
// copies write it to the packed output and the arena slot.  Up to kPackBufs
// pieces are in flight per warp across chunk boundaries.  Needs 16-byte
// aligned addresses; a chunk's last len % 16 bytes are copied by its lane.
// Steps of the misses' copies that k_pack's warps take from the call's counter:
// 32 pieces, and kFineStep pieces from kFinePerWarp pieces per warp before the
// end.  With 32 throughout, the 85,000 pieces of four Llama-3-8B layers with
// 10% of their chunks changed were 2,663 steps for 3,648 warps; pass of that
// upload 718 us so, 702 us with these (712 us with 16 pieces per warp left to
// the fine steps), of a 256 MiB payload of 1 KiB chunks that repeat 292 -> 283
// us (289 us with 32 per warp).
constexpr unsigned long long kFinePerWarp = 64, kFineStep = 8;
#ifndef GLEAM_PACK_BULK
#define GLEAM_PACK_BULK 1
#endif
constexpr uint32_t kPackPiece = 2048;
constexpr uint32_t kPackBufs = 4;
struct PackMeta {
  unsigned long long src, d1, d2;
  uint32_t len, pad;
};
// per warp: the buffers, then the mbarriers (64 B), then the batch's metadata;
// a multiple of 128 bytes so that every warp's buffers start 128-byte aligned
constexpr uint32_t kPackWarpBytes =
    (kPackBufs * kPackPiece + 64 + 32 * (uint32_t)sizeof(PackMeta) + 127) & ~127u;
constexpr uint32_t kPackSmem = kWarps * kPackWarpBytes;

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes,
                                          uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void bulk_store(void* dst, uint32_t src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() {
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
template <int N>
__device__ __forceinline__ void bulk_wait_all() {
  asm volatile("cp.async.bulk.wait_group %0;" ::"n"(N) : "memory");
}
// Until at most n (0..3; more waits for 3) newest bulk store groups still read
// shared memory.
__device__ __forceinline__ void bulk_wait_read_n(uint32_t n) {
  if (n == 0) bulk_wait_read<0>();
  else if (n == 1) bulk_wait_read<1>();
  else if (n == 2) bulk_wait_read<2>();
  else bulk_wait_read<3>();
}
static_assert(kPackBufs == 4, "bulk_wait_read_n covers up to kPackBufs - 1 pending groups");

// Ring state of one warp's lane 0, kept across its batches of 32 misses.
struct PackRing {
  uint32_t issued, consumed, phase;
};

// After a wait for a piece has run out: the limit for the pieces still in flight
// to land, however short the call's own limit.  A block that ended before them
// would leave copies under way into shared memory that another block may own.
constexpr unsigned long long kLandNs = 1000000000ULL;

// Lane 0: the whole-16-byte part of chunks 0..m-1 of `meta`; false if a
// piece did not arrive within limit_ns (the pieces still in flight have then
// been waited for).
__device__ bool bulk_copy_batch(const PackMeta* meta, uint32_t m, uint32_t bufs, uint32_t bars,
                                PackRing& ring, unsigned long long limit_ns) {
  auto nbytes = [&](uint32_t j) { return meta[j].len & ~15u; };
  uint32_t ij = 0, ioff = 0, cj = 0, coff = 0;  // issue and consume cursors
  while (ij < m && nbytes(ij) == 0) ++ij;
  cj = ij;
  while (cj < m) {
    while (ring.issued - ring.consumed < kPackBufs && ij < m) {
      const uint32_t b = ring.issued % kPackBufs;
      // the store that last read buffer b (piece issued - kPackBufs) must be done reading
      if (ring.issued >= kPackBufs) bulk_wait_read_n(kPackBufs - 1 - (ring.issued - ring.consumed));
      const uint32_t nb = nbytes(ij);
      const uint32_t bytes = min(kPackPiece, nb - ioff);
      mbar_expect_tx(bars + 8 * b, bytes);
      bulk_load(bufs + b * kPackPiece, reinterpret_cast<const uint8_t*>(meta[ij].src) + ioff, bytes,
                bars + 8 * b);
      ++ring.issued;
      ioff += bytes;
      if (ioff == nb) {
        ioff = 0;
        do ++ij;
        while (ij < m && nbytes(ij) == 0);
      }
    }
    const uint32_t b = ring.consumed % kPackBufs;
    if (!mbar_wait(bars + 8 * b, (ring.phase >> b) & 1u, limit_ns)) {
      for (uint32_t k = ring.consumed; k < ring.issued; ++k) {  // let the loads land
        const uint32_t bb = k % kPackBufs;
        mbar_wait(bars + 8 * bb, (ring.phase >> bb) & 1u, max(limit_ns, kLandNs));
        ring.phase ^= 1u << bb;
      }
      ring.consumed = ring.issued;
      return false;
    }
    ring.phase ^= 1u << b;
    const uint32_t nb = nbytes(cj);
    const uint32_t bytes = min(kPackPiece, nb - coff);
    bulk_store(reinterpret_cast<uint8_t*>(meta[cj].d1) + coff, bufs + b * kPackPiece, bytes);
    if (meta[cj].d2) bulk_store(reinterpret_cast<uint8_t*>(meta[cj].d2) + coff, bufs + b * kPackPiece, bytes);
    bulk_commit();
    ++ring.consumed;
    coff += bytes;
    if (coff == nb) {
      coff = 0;
      do ++cj;
      while (cj < m && nbytes(cj) == 0);
    }
  }
  return true;
}

__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// The rest of an insert's linear probe in KEY16 mode, from `pos` (the probe's
// `probe`-th position): all chunks of one 16-bit key share a home position,
// so an insert walks the cluster of the key's earlier entries.  The slot words
// of the next kScanEntries entries are read at once and the first that was
// free is claimed: one round trip per kScanEntries entries instead of one per
// entry.  While a call inserts, entries only go from free to used (evictions
// finish before), so an entry read as used stays used and is passed over
// safely; a claim that loses the race moves on to the next entry.  (With full
// 64-bit keys the entry after a used home is mostly free, and claiming it
// directly is one round trip fewer.)  False if the table is full.
constexpr uint32_t kScanEntries = 8;
__device__ __noinline__ bool index_insert_scan(IndexEntry* index, uint64_t mask,
                                               unsigned long long key, uint32_t slot,
                                               uint32_t len, uint64_t pos, uint64_t probe) {
  while (probe <= mask) {
    uint32_t free_bits = 0;
#pragma unroll
    for (uint32_t k = 0; k < kScanEntries; ++k)
      free_bits |= (ldcg_u32(&index[(pos + k) & mask].slot) == kEmptySlot ? 1u : 0u) << k;
    if (free_bits == 0) {
      pos = (pos + kScanEntries) & mask;
      probe += kScanEntries;
      continue;
    }
    const uint32_t k = __ffs(free_bits) - 1;
    probe += k;
    if (probe > mask) break;
    pos = (pos + k) & mask;
    if (atomicCAS(&index[pos].slot, kEmptySlot, slot) == kEmptySlot) {
      index[pos].key = key;
      index[pos].len = len;
      return true;
    }
    pos = (pos + 1) & mask;
    ++probe;
  }
  return false;
}

// Claims a free index entry for (key, slot, len); false if the table is full.
// scan: the rest of the probe by index_insert_scan (KEY16 index keys).
// place: the probe starts that many entries after the key's home position.
// With KEY16 classes the misses of a call that share an index key (and
// length) have the places 0 .. n-1, so each starts at its own entry instead
// of walking past the others; an entry stays reachable from the home
// position: a free entry left between the home position and a miss's entry
// (at place q) would have been taken by the miss whose place is q.
__device__ bool index_insert(IndexEntry* index, uint64_t mask, unsigned long long key,
                             uint32_t slot, uint32_t len, bool scan = false,
                             uint32_t place = 0) {
  uint64_t pos = (mix64(key) + place) & mask;
  for (uint64_t probe = 0; probe <= mask; ++probe) {
    const uint32_t old = atomicCAS(&index[pos].slot, kEmptySlot, slot);
    if (old == kEmptySlot) {
      index[pos].key = key;
      index[pos].len = len;
      return true;
    }
    pos = (pos + 1) & mask;
    if (scan) return index_insert_scan(index, mask, key, slot, len, pos, probe + 1);
  }
  return false;
}

// index_insert in two halves: the first claim attempt at the key's home
// position (issued early; its result is not waited for until it is needed),
// then, given that attempt's result, the entry's fields or the rest of the
// probe.  Together they do what index_insert does.
struct PendingInsert {
  uint64_t pos;
  uint32_t old;
};
__device__ __forceinline__ PendingInsert index_insert_begin(IndexEntry* index, uint64_t mask,
                                                            unsigned long long key, uint32_t slot) {
  const uint64_t pos = mix64(key) & mask;
  return PendingInsert{pos, atomicCAS(&index[pos].slot, kEmptySlot, slot)};
}
__device__ bool index_insert_end(IndexEntry* index, uint64_t mask, unsigned long long key,
                                 uint32_t slot, uint32_t len, PendingInsert p, bool scan = false) {
  uint64_t pos = p.pos;
  uint32_t old = p.old;
  for (uint64_t probe = 0;;) {
    if (old == kEmptySlot) {
      index[pos].key = key;
      index[pos].len = len;
      return true;
    }
    if (++probe > mask) return false;
    pos = (pos + 1) & mask;
    if (scan) return index_insert_scan(index, mask, key, slot, len, pos, probe);
    old = atomicCAS(&index[pos].slot, kEmptySlot, slot);
  }
}

// Finds or claims the per-call group entry of (key, len) for chunk g;
// *claimed tells whether g claimed it (else another chunk of the group did).
// cas_first: claim without reading the entry first (one round trip fewer
// where entries are mostly free; the read spares a contended entry the
// atomics of every chunk of a large group).
__device__ uint32_t group_entry(const DedupArgs& a, uint32_t g, unsigned long long k,
                                uint32_t len, bool* claimed = nullptr, bool cas_first = false) {
  uint64_t pos = mix64(k ^ ((unsigned long long)len << 40)) & a.tbl_mask;
  for (uint64_t probe = 0; probe <= a.tbl_mask; ++probe) {
    uint32_t o = cas_first && probe == 0 ? 0u : ldcg_u32(&a.tbl[pos].owner);
    if (o == 0) {
      // a free entry is all zeros: the claim posts the claimant's minimum too
      const unsigned long long old =
          atomicCAS(reinterpret_cast<unsigned long long*>(&a.tbl[pos]), 0ull,
                    (unsigned long long)~g << 32 | (unsigned long long)(g + 1));
      if (old == 0) {
        if (claimed) *claimed = true;
        return (uint32_t)pos;
      }
      o = (uint32_t)old;
    }
    if (a.ch.key[o - 1] == k && a.ch.len[o - 1] == len) {
      if (claimed) *claimed = false;
      return (uint32_t)pos;
    }
    pos = (pos + 1) & a.tbl_mask;
  }
  return 0xFFFFFFFFu;  // cannot happen: the table has >= 2 Ntot entries
}

// KEY16 with XXH64 keys: finds or claims chunk g's entry in the per-call table
// of (16-bit index key, length) classes.
__device__ uint32_t class_entry(const DedupArgs& a, uint32_t g, unsigned long long k16,
                                uint32_t len) {
  uint64_t pos = mix64(k16 ^ ((unsigned long long)len << 40)) & a.tbl_mask;
  for (uint64_t probe = 0; probe <= a.tbl_mask; ++probe) {
    uint32_t o = ldcg_u32(&a.cls_tbl[pos].owner);
    if (o == 0) {
      o = atomicCAS(&a.cls_tbl[pos].owner, 0u, g + 1);
      if (o == 0) return (uint32_t)pos;
    }
    if ((a.ch.key[o - 1] & 0xFFFFull) == k16 && a.ch.len[o - 1] == len) return (uint32_t)pos;
    pos = (pos + 1) & a.tbl_mask;
  }
  return 0xFFFFFFFFu;  // cannot happen: the table has >= 2 Ntot entries
}

// The index key of a group key (KEY16 mode: its low 16 bits).
__device__ __forceinline__ unsigned long long index_key(const DedupArgs& a,
                                                        unsigned long long k) {
  return a.key16 ? (k & 0xFFFFull) : k;
}

__device__ __forceinline__ const PayloadDesc& desc(const DedupArgs& a, uint32_t p) {
  return a.count > 1 ? a.table[p] : a.one;
}

template <typename T>
__device__ __forceinline__ T block_sum(T v, T* red) {
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  T t = 0;
#pragma unroll
  for (int k = 0; k < kWarps; ++k) t += red[k];
  return t;
}

// Sum of v over the lanes of `peers`, added to *dst by the one lane of the
// group whose dst is not null.
__device__ __forceinline__ void add_in_group(unsigned long long* dst, unsigned peers, uint32_t v) {
  const uint32_t sum = __reduce_add_sync(peers, v);
  if (dst && sum) atomicAdd(dst, sum);
}

// ---- LRU eviction (paper Sec. 4.1.3; reading R16) ---------------------------
//
// The K slots to evict are the K smallest (last use, slot number) among the
// used slots whose last use is before this call (the call's own hits were
// stamped with its clock value in phase A).  The cut-off stamp is found by a
// two-pass radix select on its high and low 16 bits; the victims are then the
// slots older than the cut-off plus the lowest-numbered slots at it.  Their
// index and hint-table entries are removed without tombstones surviving the
// call: each is first replaced by a tombstone, then every cluster (maximal
// run of occupied entries) that holds one is rebuilt by its single owner
// thread, moving each live entry, in cluster order, to the first hole between
// its home position and itself, and finally the remaining tombstones become
// empty.  Clusters shrink but never merge, so owners never meet.

// Rebuilds the cluster that starts at `start` (its predecessor is empty).
__device__ void compact_cluster(IndexEntry* t, unsigned long long mask, unsigned long long start) {
  unsigned long long len = 0;
  bool any = false;
  for (unsigned long long q = start; len <= mask; q = (q + 1) & mask, ++len) {
    const uint32_t sl = t[q].slot;
    if (sl == kEmptySlot) break;
    any |= sl == kTombSlot;
  }
  if (!any) return;
  for (unsigned long long k = 0; k < len; ++k) {
    const unsigned long long q = (start + k) & mask;
    const IndexEntry e = t[q];
    if (e.slot == kTombSlot) continue;
    for (unsigned long long j = mix64(e.key) & mask; j != q; j = (j + 1) & mask) {
      if (t[j].slot == kTombSlot) {
        t[j] = e;
        t[q].slot = kTombSlot;
        break;
      }
    }
  }
}

// Exclusive block-wide prefix of per-thread flags, in thread order, for one
// 256-slot step; returns the thread's offset and adds the step's total to
// *running (shared arrays: kWarps counts + offsets).
__device__ __forceinline__ uint32_t block_rank(bool f, uint32_t* cnt, uint32_t* off,
                                               unsigned long long* running_total) {
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t b = __ballot_sync(0xffffffffu, f);
  if (lane == 0) cnt[w] = __popc(b);
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t acc = 0;
    for (int k = 0; k < kWarps; ++k) {
      off[k] = acc;
      acc += cnt[k];
    }
    cnt[0] = acc;
  }
  __syncthreads();
  const uint32_t r = off[w] + __popc(b & ((1u << lane) - 1u));
  const uint32_t step = cnt[0];
  __syncthreads();
  *running_total += step;
  return r;
}

// The cut-off stamp by a two-pass radix select on its high and low 16 bits, and
// how many candidates at it are victims; false if a grid barrier failed.  Out
// of line: for stamps that lru_evict's one pass by age does not tell apart.
// The bins hold that pass's counts.
__device__ __noinline__ bool lru_radix_cut(const DedupArgs& a, uint32_t G, uint32_t bid,
                                           unsigned long long slots0, unsigned long long K,
                                           unsigned long long* sred, uint32_t* off,
                                           uint32_t* cut, unsigned long long* ties) {
  static_assert(kLruBins == kThreads * kThreads, "one part of kThreads bins per thread");
  const uint32_t lane = threadIdx.x & 31;
  const unsigned long long tid = (unsigned long long)bid * kThreads + threadIdx.x;
  const unsigned long long nth = (unsigned long long)G * kThreads;
  const uint32_t now = a.epoch;
  if (!grid_barrier(a.ctl, G, a.wait_ns, false)) return false;  // every block has read the bins
  for (unsigned long long q = tid; q < kLruBins; q += nth) a.bins[q] = 0u;
  if (!grid_barrier(a.ctl, G, a.wait_ns, false)) return false;
  uint32_t hi_bin = 0;
  unsigned long long below = 0;
  for (int pass = 0; pass < 2; ++pass) {
    for (unsigned long long base = tid - lane; base < slots0; base += nth) {
      const unsigned long long sl = base + lane;
      uint32_t key = 0xFFFFFFFFu;
      if (sl < slots0) {
        const uint32_t u = __ldcg(&a.last_use[sl]);
        if (u != now && (pass == 0 || (u >> 16) == hi_bin)) key = pass == 0 ? (u >> 16) : (u & 0xFFFFu);
      }
      const unsigned peers = __match_any_sync(0xffffffffu, key);
      if (key != 0xFFFFFFFFu && lane == (uint32_t)(__ffs(peers) - 1))
        atomicAdd(&a.bins[key], (uint32_t)__popc(peers));
    }
    if (!grid_barrier(a.ctl, G, a.wait_ns, false)) return false;
    if (bid == 0) {
      // the bin holding the K-th candidate: partial sums of 256 bins per
      // thread (16-byte loads), the part holding it, then that part's bins
      constexpr uint32_t kPer = kLruBins / kThreads;
      const uint4* b4 = reinterpret_cast<const uint4*>(a.bins + threadIdx.x * kPer);
      unsigned long long part = 0;
#pragma unroll 16
      for (uint32_t j = 0; j < kPer / 4; ++j) {
        const uint4 v = __ldcg(b4 + j);
        part += (unsigned long long)v.x + v.y + v.z + v.w;
      }
      sred[threadIdx.x] = part;
      __syncthreads();
      const unsigned long long target = K - below;  // >= 1 candidates in this range
      if (threadIdx.x == 0) {
        unsigned long long acc = 0;
        uint32_t pi = 0;
        while (pi + 1 < (uint32_t)kThreads && acc + sred[pi] < target) acc += sred[pi++];
        off[0] = pi;
        sred[kThreads - 1] = acc;  // candidates before part pi (its own sum is no longer needed)
      }
      __syncthreads();
      const uint32_t pi = off[0];
      const unsigned long long acc0 = sred[kThreads - 1];
      __syncthreads();
      sred[threadIdx.x] = __ldcg(&a.bins[pi * kPer + threadIdx.x]);
      __syncthreads();
      if (threadIdx.x == 0) {
        unsigned long long acc = acc0;
        uint32_t j = 0;
        while (j + 1 < kPer && acc + sred[j] < target) acc += sred[j++];
        const uint32_t bin = pi * kPer + j;
        if (pass == 0) {
          a.ctl->lru_hi = bin;
          a.ctl->lru_below = acc;
        } else {
          a.ctl->lru_cut = (hi_bin << 16) | bin;
          a.ctl->lru_below = below + acc;
          a.ctl->lru_ties = target - acc;
        }
      }
      __syncthreads();
      uint4* z4 = reinterpret_cast<uint4*>(a.bins);
      for (uint32_t j = threadIdx.x; j < kLruBins / 4; j += kThreads) z4[j] = make_uint4(0, 0, 0, 0);
    }
    if (!grid_barrier(a.ctl, G, a.wait_ns, false)) return false;
    hi_bin = __ldcg(&a.ctl->lru_hi);
    below = __ldcg(&a.ctl->lru_below);
  }
  *cut = __ldcg(&a.ctl->lru_cut);
  *ties = __ldcg(&a.ctl->lru_ties);
  return true;
}

// Ages (calls since the last use) that have a bin of their own; bin 0 holds
// stamps later than this call's (the clock was set back), the last bin all
// greater ages.  Bin b is word b + kAgeBase: the sixteen bins of a thread
// (lru_evict) are then four 16-byte loads.
constexpr uint32_t kAgeBins = 16 * kThreads;
constexpr uint32_t kAgeBase = 3;
static_assert(kAgeBins + kAgeBase < kLruBins, "the bins' array holds them");

// Selects and removes the K victims; false if a grid barrier failed.
__device__ bool lru_evict(const DedupArgs& a, uint32_t G, uint32_t bid,
                          unsigned long long slots0, unsigned long long K,
                          unsigned long long* sred, uint32_t* cnt, uint32_t* off,
                          unsigned long long* red64) {
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned long long tid = (unsigned long long)bid * kThreads + threadIdx.x;
  const unsigned long long nth = (unsigned long long)G * kThreads;
  const uint32_t now = a.epoch;

  // The cut-off stamp: one histogram of the candidates' ages, from which every
  // block finds the bin of the K-th oldest.  A warp adds up a run of slots of
  // one age before it touches the bin.
  {
    uint32_t run = 0xFFFFFFFFu, run_cnt = 0;
    for (unsigned long long base = tid - lane; base < slots0; base += nth) {
      const unsigned long long sl = base + lane;
      uint32_t bin = 0xFFFFFFFFu;
      if (sl < slots0) {
        const uint32_t u = __ldcg(&a.last_use[sl]);
        if (u != now) bin = u > now ? 0u : min(now - u, kAgeBins);
      }
      const unsigned have = __ballot_sync(0xffffffffu, bin != 0xFFFFFFFFu);
      if (!have) continue;
      const uint32_t b0 = __shfl_sync(0xffffffffu, bin, __ffs(have) - 1);
      if (__ballot_sync(0xffffffffu, bin == b0) == have) {
        if (b0 != run) {
          if (run_cnt && lane == 0) atomicAdd(&a.bins[kAgeBase + run], run_cnt);
          run = b0;
          run_cnt = 0;
        }
        run_cnt += __popc(have);
      } else {
        const unsigned peers = __match_any_sync(0xffffffffu, bin);
        if (bin != 0xFFFFFFFFu && lane == (uint32_t)(__ffs(peers) - 1))
          atomicAdd(&a.bins[kAgeBase + bin], (uint32_t)__popc(peers));
      }
    }
    if (run_cnt && lane == 0) atomicAdd(&a.bins[kAgeBase + run], run_cnt);
  }
  if (!grid_barrier(a.ctl, G, a.wait_ns, false)) return false;
  uint32_t cut = 0;
  unsigned long long ties = 0;
  {
    // thread i: the bins of ages kAgeBins - 16 i down to kAgeBins - 16 i - 15
    uint32_t v[16], sum = 0;
    const uint4* b4 = reinterpret_cast<const uint4*>(a.bins + kAgeBase + kAgeBins -
                                                     16 * threadIdx.x - 15);
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
      const uint4 x = __ldcg(b4 + k);
      v[4 * k] = x.x, v[4 * k + 1] = x.y, v[4 * k + 2] = x.z, v[4 * k + 3] = x.w;
      sum += x.x + x.y + x.z + x.w;
    }
    uint32_t incl = sum;
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
      const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += x;
    }
    if (lane == 31) cnt[w] = incl;
    if (threadIdx.x == 0) off[0] = 0;  // the bin of the K-th oldest; 0: in no thread's
    __syncthreads();
    unsigned long long older = incl - sum;
    for (uint32_t k = 0; k < w; ++k) older += cnt[k];
    if (older < K && K <= older + sum) {
#pragma unroll
      for (uint32_t k = 0; k < 16; ++k) {
        const uint32_t c = v[15 - k];
        if (older < K && K <= older + c) {
          off[0] = kAgeBins - 16 * threadIdx.x - k;
          sred[0] = K - older;
        }
        older += c;
      }
    }
    __syncthreads();
    const uint32_t bin = off[0];
    cut = now - bin;
    ties = sred[0];
    __syncthreads();
    if (bin == 0 || bin == kAgeBins) {
      if (!lru_radix_cut(a, G, bid, slots0, K, sred, off, &cut, &ties)) return false;
    }
  }

  // per contiguous slot range: candidates older than the cut-off, and at it
  const unsigned long long per = ((slots0 + G - 1) / G + 31) & ~31ull;
  const unsigned long long lo = min(slots0, bid * per);
  const unsigned long long hi = min(slots0, lo + per);
  {
    uint32_t nlt = 0, ntie = 0;
    for (unsigned long long sl = lo + threadIdx.x; sl < hi; sl += kThreads) {
      const uint32_t u = __ldcg(&a.last_use[sl]);
      if (u != now) {
        nlt += u < cut;
        ntie += u == cut;
      }
    }
    const unsigned long long t_lt = block_sum<unsigned long long>(nlt, red64);
    const unsigned long long t_tie = block_sum<unsigned long long>(ntie, red64);
    if (threadIdx.x == 0) {
      a.bcount[bid] = (uint32_t)t_tie;
      a.bcount[G + bid] = (uint32_t)t_lt;
    }
  }
  if (!grid_barrier(a.ctl, G, a.wait_ns, false)) return false;
  // every block has read the ages' bins
  for (unsigned long long q = tid; q <= kAgeBase + kAgeBins; q += nth) a.bins[q] = 0u;
  {
    unsigned long long tie_before = 0, lt_before = 0;
    for (uint32_t j = threadIdx.x; j < bid; j += kThreads) {
      tie_before += __ldcg(&a.bcount[j]);
      lt_before += __ldcg(&a.bcount[G + j]);
    }
    tie_before = block_sum<unsigned long long>(tie_before, red64);
    lt_before = block_sum<unsigned long long>(lt_before, red64);
    unsigned long long vrun = lt_before + min(ties, tie_before), trun = tie_before;
    unsigned long long vbytes = 0;
    for (unsigned long long t0 = lo; t0 < hi; t0 += kThreads) {
      const unsigned long long sl = t0 + threadIdx.x;
      const uint32_t u = sl < hi ? __ldcg(&a.last_use[sl]) : now;
      const bool tie = u != now && u == cut;
      const unsigned long long tb = trun;
      const uint32_t tr = block_rank(tie, cnt, off, &trun);
      const bool victim = (u != now && u < cut) || (tie && tb + tr < ties);
      const unsigned long long vb = vrun;
      const uint32_t vr = block_rank(victim, cnt, off, &vrun);
      if (victim && vb + vr < K) {  // always: the counts above add up to K
        a.victims[vb + vr] = (uint32_t)sl;
        a.vflag[sl] = 1;
        vbytes += a.slot_len[sl];
      }
    }
    vbytes = block_sum<unsigned long long>(vbytes, red64);
    if (threadIdx.x == 0 && vbytes) atomicAdd(&a.ctl->acc_victim_bytes, vbytes);
  }
  if (!grid_barrier(a.ctl, G, a.wait_ns, false)) return false;

  // the victims' entries leave the index and the hint table; kTabWays entries
  // of each per thread at a time, so that their loads wait together
  constexpr uint32_t kTabWays = 4;
  const unsigned long long tsize = a.index_mask + 1;
  for (unsigned long long q0 = tid; q0 < tsize; q0 += kTabWays * nth) {
    uint32_t s1[kTabWays], s2[kTabWays];
#pragma unroll
    for (uint32_t k = 0; k < kTabWays; ++k) {
      const unsigned long long q = q0 + k * nth;
      s1[k] = q < tsize ? a.index[q].slot : kEmptySlot;
      s2[k] = q < tsize ? a.hints[q].slot : kEmptySlot;
    }
    bool f1[kTabWays], f2[kTabWays];
#pragma unroll
    for (uint32_t k = 0; k < kTabWays; ++k) {
      f1[k] = s1[k] < slots0 && a.vflag[s1[k]];
      f2[k] = s2[k] < slots0 && a.vflag[s2[k]];
    }
#pragma unroll
    for (uint32_t k = 0; k < kTabWays; ++k) {
      const unsigned long long q = q0 + k * nth;
      if (f1[k]) a.index[q].slot = kTombSlot;
      if (f2[k]) a.hints[q].slot = kTombSlot;
    }
  }
  if (!grid_barrier(a.ctl, G, a.wait_ns, false)) return false;
  for (unsigned long long q0 = tid; q0 < tsize; q0 += kTabWays * nth) {
    bool f1[kTabWays], f2[kTabWays];  // a cluster begins here
#pragma unroll
    for (uint32_t k = 0; k < kTabWays; ++k) {
      const unsigned long long q = q0 + k * nth;
      f1[k] = f2[k] = false;
      if (q < tsize) {
        const unsigned long long prev = (q + tsize - 1) & a.index_mask;
        f1[k] = a.index[q].slot != kEmptySlot && a.index[prev].slot == kEmptySlot;
        f2[k] = a.hints[q].slot != kEmptySlot && a.hints[prev].slot == kEmptySlot;
      }
    }
#pragma unroll 1
    for (uint32_t k = 0; k < kTabWays; ++k) {
      if (f1[k]) compact_cluster(a.index, a.index_mask, q0 + k * nth);
      if (f2[k]) compact_cluster(a.hints, a.index_mask, q0 + k * nth);
    }
  }
  if (!grid_barrier(a.ctl, G, a.wait_ns, false)) return false;
#pragma unroll 4
  for (unsigned long long q = tid; q < tsize; q += nth) {
    if (a.index[q].slot == kTombSlot) a.index[q].slot = kEmptySlot;
    if (a.hints[q].slot == kTombSlot) a.hints[q].slot = kEmptySlot;
  }
  for (unsigned long long r = tid; r < K; r += nth) a.vflag[a.victims[r]] = 0;
  return true;
}

// Posts ~g as a candidate minimum of group entry `e` (0xFFFFFFFF: none), one
// atomic per group of lanes that share the entry.  Called by the whole warp.
template <typename Entry>
__device__ __forceinline__ void post_minimum(Entry* tbl, uint32_t e, uint32_t g,
                                             unsigned peers) {
  const uint32_t m = __reduce_max_sync(peers, e != 0xFFFFFFFFu ? ~g : 0u);
  // a group of many chunks (all-zero chunks, say) would queue its atomics on
  // one address: skip the atomic when a smaller number is already posted
  if (e != 0xFFFFFFFFu && (threadIdx.x & 31) == (uint32_t)(__ffs(peers) - 1) &&
      ldcg_u32(&tbl[e].minv) < m)
    atomicMax(&tbl[e].minv, m);
}
__device__ __forceinline__ void post_minimum(CallEntry* tbl, uint32_t e, uint32_t g) {
  post_minimum(tbl, e, g, __match_any_sync(0xffffffffu, e));
}

// KEY16 classes: posts ~g as a candidate minimum of class entry `e`
// (0xFFFFFFFF: none) and returns the lane's place among the misses of the
// class (counted in the entry), one atomic of each kind per group of lanes
// that share the entry.  Called by the whole warp.
__device__ __forceinline__ uint32_t post_class(ClassEntry* tbl, uint32_t e, uint32_t g) {
  const uint32_t lane = threadIdx.x & 31;
  const unsigned peers = __match_any_sync(0xffffffffu, e);
  post_minimum(tbl, e, g, peers);
  const int first = __ffs(peers) - 1;
  uint32_t base = 0;
  if (e != 0xFFFFFFFFu && lane == (uint32_t)first)
    base = atomicAdd(&tbl[e].count, (uint32_t)__popc(peers));
  return __shfl_sync(0xffffffffu, base, first) + __popc(peers & ((1u << lane) - 1u));
}
__device__ __forceinline__ void post_minimum(const DedupArgs& a, uint32_t e, uint32_t g) {
  post_minimum(a.tbl, e, g);
}

// The first-occurrence resolution and miss ranks of a call, run by block
// `bid` of a grid of G co-resident blocks.  claimed: the caller has done
// phase A (claims and minima posted, outputs cleared) and passed a grid
// barrier since, with outcome `ok0`.  True if no chunk missed; *hits_ok then
// tells whether the block's barrier was passed and no error recorded.
__device__ __forceinline__ bool resolve_rank(const DedupArgs& a, uint32_t G, uint32_t bid,
                                             bool claimed = false, bool ok0 = true,
                                             bool* hits_ok = nullptr) {
  __shared__ unsigned long long red64[kWarps];
  __shared__ uint32_t warp_cnt[kWarps];
  __shared__ uint32_t warp_off[kWarps];
  __shared__ uint32_t swarp_cnt[kWarps];
  __shared__ uint32_t swarp_off[kWarps];
  __shared__ unsigned long long s_slots0;
  __shared__ unsigned long long sred[kThreads];
  __shared__ int s_err1, s_any;  // s_any: a chunk of the block's is not a cache hit
  // chunks of a block's contiguous range; here, and the range's bounds taken after
  // the rounds, so that the compares' loads find registers (1 GiB of 64 KiB
  // chunks, half of them copies: 201 us the kernel, 286 with the bounds live)
  __shared__ uint32_t s_per;

  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t tid = bid * kThreads + threadIdx.x;
  const uint32_t nth = G * kThreads;
  const uint32_t N = (uint32_t)a.Ntot;
  const bool skip = (int)bid == a.skip_block;
  const ChunkArrays& ch = a.ch;

  // thread 0's read of the slot count completes while phase A runs
  const unsigned long long my_slots0 =
      threadIdx.x == 0 ? *(volatile const unsigned long long*)&a.dstats[ST_SLOTS_USED] : 0ull;

  // the rounds count the misses of every range as they find them (a warp step's
  // 32 chunks lie in one range), so that the ranks need no counting pass and no
  // barrier after it; a grid of one, and KEY16 classes, whose rejects wait for
  // every miss's class, count them afterwards
  const bool counted = !claimed && !a.classes && G > 1;

  // ---- A: clear outputs, round-1 claims; LRU: stamp the slots hit ----------
  if (!claimed) {
    if (threadIdx.x == 0) {
      s_any = 0;
      s_per = (uint32_t)((((uint64_t)N + G - 1) / G + 31) & ~31ull);
    }
    __syncthreads();
    if (counted)
      for (uint32_t j = tid; j < 2 * G; j += nth) a.bcount[j] = 0;
    unsigned long long distinct = 0;
    for (uint32_t p = tid; p < a.count; p += nth) {
      gleam_result_t* r = desc(a, p).result;
      if (r) {
        r->n_miss = 0;
        r->n_hit_cache = 0;
        r->n_hit_intra = 0;
        r->verify_rejects = 0;
        r->miss_bytes = 0;
      }
    }
    // warp-uniform steps, so that chunks of one group in a warp post their
    // minimum with one atomic (all-zero chunks, say, share a group)
    for (uint32_t base = tid - lane; base < N; base += nth) {
      const uint32_t g = base + lane;
      uint32_t post = 0xFFFFFFFFu;  // group entry that gets this chunk's number
      if (g < N) {
        // every operand at once: the claim below then waits for none of them
        const uint8_t st = ch.status[g];
        const unsigned long long key = ch.key[g];
        const uint32_t len = ch.len[g];
        const PayloadDesc& P = desc(a, ch.pidx[g]);
        const unsigned long long i = g - P.chunk_base;
        if ((i & 31) == 0) P.mask[i >> 5] = 0;
        if (st != kHit0) s_any = 1;
        if (st == kHit0) {
          ch.res[g] = kResHit0;
          if (a.lru) {  // the first chunk to stamp a slot keeps its old value
            const uint32_t old = atomicExch(&a.last_use[ch.ent[g]], a.epoch);
            ch.old[g] = old;
            distinct += old != a.epoch;
          }
        } else if (st == kUncached) {  // never cached: a miss of its own, in no group
          ch.ent[g] = 0xFFFFFFFFu;
          ch.res[g] = kResLeader | kResNoSlot | 1u;
        } else {
          bool mine = false;  // a claim posts the claimant's own number
          const uint32_t e = group_entry(a, g, key, len, &mine);
          if (e == 0xFFFFFFFFu) {
            atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_INTERNAL);
            ch.ent[g] = 0xFFFFFFFFu;
            ch.res[g] = kResLeader | 1u;
          } else {
            ch.ent[g] = e;
            ch.res[g] = kResUnresolved;
            if (!mine) post = e;
          }
        }
      }
      post_minimum(a, post, g);
    }
    if (a.lru) {
      distinct = block_sum<unsigned long long>(distinct, red64);
      if (threadIdx.x == 0 && distinct) atomicAdd(&a.ctl->acc_distinct, distinct);
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_any) *(volatile unsigned int*)&a.ctl->any_miss = 1u;
  }
  bool any_miss = true;
  bool ok = claimed ? ok0 : grid_barrier(a.ctl, G, a.wait_ns, skip, &any_miss);
  // nothing but cache hits, as far as a block whose wait ran out can know: no
  // rounds and no ranks (and no misses counted)
  if (!any_miss) {
    if (G == 1) {  // its barrier did not read the error word
      if (threadIdx.x == 0) s_err1 = ld_volatile_s32(&a.ctl->err);
      __syncthreads();
      ok = ok && s_err1 == 0;
    }
    if (hits_ok) *hits_ok = ok;
    return true;
  }

  // ---- B/C: rounds until every chunk is a hit, duplicate or leader ---------
  uint32_t round = 1;
  while (ok) {
    bool stay = false;  // one of this thread's chunks is left for the next round
    if (tid == 0) atomicExch(&a.ctl->unres[(round + 1) % 3], 0u);
    // W chunks per warp step: 32, or fewer when there are too few chunks to
    // give every warp a step (large chunks), so the compares spread over the grid
    const uint32_t nwarps = nth / 32;
    uint32_t W = 32;
    while (W > 1 && (unsigned long long)N < (unsigned long long)nwarps * W) W >>= 1;
    for (uint32_t base = (tid / 32) * W; base < N; base += nwarps * W) {
      const uint32_t g = base + lane;
      bool need = false, lead = false;
      uint32_t m = 0;
      const uint32_t res0 = lane < W && g < N ? ldcg_u32(&ch.res[g]) : kResHit0;
      if (res0 == kResUnresolved) {
        m = ~ldcg_u32(&a.tbl[ch.ent[g]].minv);
        if (m == g) {
          ch.res[g] = kResLeader | round;
          lead = true;
        } else if (m > g) {  // the group minimum can only be below g: table damaged
          atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_INTERNAL);
          ch.res[g] = kResLeader | round;
          lead = true;
        } else if (ch.hint[g] != ch.hint[m]) {
          // different first 512 bytes (the prefix hints differ), so different
          // chunks: no byte compare, the chunk waits for a later round
          atomicAdd(&a.ctl->unres[round % 3], 1u);
          stay = true;
        } else {
          need = true;
        }
      }
      if (counted) {
        // (phase A made leaders of the chunks that are never cached)
        const bool first = round == 1 && (res0 & kResLeader);
        const unsigned mb = __ballot_sync(0xffffffffu, lead || first);
        const unsigned sb = __ballot_sync(0xffffffffu, lead || (first && !(res0 & kResNoSlot)));
        if (lane == 0 && mb) {
          const uint32_t range = base / s_per;
          atomicAdd(&a.bcount[range], (uint32_t)__popc(mb));
          if (sb) atomicAdd(&a.bcount[G + range], (uint32_t)__popc(sb));
        }
      }
      if (a.classes) {
        // KEY16: a new leader (a miss) claims the class of its 16-bit index
        // key and length, posts its number there and takes its place among
        // the class's misses (where its index insert starts); after the last
        // round a class minimum below a leader's number is an earlier miss of
        // its index key and length (a reject).  Groups are whole fingerprints, so
        // nearly all leaders are found in the first round, while the other warps
        // compare their duplicates.
        uint32_t cpost = 0xFFFFFFFFu;
        if (lead) {
          cpost = class_entry(a, g, ch.key[g] & 0xFFFFull, ch.len[g]);
          if (cpost == 0xFFFFFFFFu) atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_INTERNAL);
        }
        const uint32_t place = post_class(a.cls_tbl, cpost, g);
        if (lead) ch.cls[g] = cpost | ((unsigned long long)place << 32);
      }
      uint32_t todo = __ballot_sync(0xffffffffu, need);
      // every lane fetches its own chunk's operands at once, so that each
      // compare below waits for its bytes only, not for their addresses first
      unsigned long long xs = 0, ys = 0;
      uint32_t ln = 0;
      if (need) {
        xs = ch.src[g];
        ys = ch.src[m];
        ln = ch.len[g];
      }
      // duplicates of at most kSmallCmpBytes (whole 16-byte pieces, aligned
      // operands) are compared up to kSmallCmpWays at a time, every lane loading
      // its pieces of all of them before any result is needed; the others one
      // by one
      unsigned small = __ballot_sync(0xffffffffu, need && ln <= kSmallCmpBytes && (ln & 15) == 0 &&
                                                      ((xs | ys) & 15) == 0);
      auto settle = [&](int j, bool eq) {
        if (lane == (uint32_t)j) {
          if (eq) {
            ch.ent[g] = m;  // the leader, for the hit's classification
            ch.res[g] = kResDup;
          } else {
            atomicAdd(&a.ctl->unres[round % 3], 1u);
            stay = true;
          }
        }
      };
      while (kSmallCmpWays > 1 && __popc(small) >= 2) {
        int js[kSmallCmpWays];
        uint32_t cnt = 0;
        while (cnt < kSmallCmpWays && small) {
          js[cnt++] = __ffs(small) - 1;
          small &= small - 1;
        }
        uint4 u[kSmallCmpWays][kSmallCmpBytes / 512], v[kSmallCmpWays][kSmallCmpBytes / 512];
#pragma unroll
        for (uint32_t c = 0; c < kSmallCmpWays; ++c) {
          if (c < cnt) {
            const uint4* x = reinterpret_cast<const uint4*>(__shfl_sync(0xffffffffu, xs, js[c]));
            const uint4* y = reinterpret_cast<const uint4*>(__shfl_sync(0xffffffffu, ys, js[c]));
            const uint32_t np = __shfl_sync(0xffffffffu, ln, js[c]) >> 4;
#pragma unroll
            for (uint32_t r = 0; r < kSmallCmpBytes / 512; ++r) {
              const uint32_t k = r * 32 + lane;
              u[c][r] = k < np ? __ldcs(x + k) : make_uint4(0, 0, 0, 0);
              v[c][r] = k < np ? __ldcs(y + k) : make_uint4(0, 0, 0, 0);
            }
          }
        }
#pragma unroll
        for (uint32_t c = 0; c < kSmallCmpWays; ++c) {
          if (c < cnt) {
            bool diff = false;
#pragma unroll
            for (uint32_t r = 0; r < kSmallCmpBytes / 512; ++r)
              diff |= (u[c][r].x != v[c][r].x) | (u[c][r].y != v[c][r].y) |
                      (u[c][r].z != v[c][r].z) | (u[c][r].w != v[c][r].w);
            settle(js[c], !__any_sync(0xffffffffu, diff));
            todo &= ~(1u << js[c]);
          }
        }
      }
      while (todo) {
        const int j = __ffs(todo) - 1;
        todo &= todo - 1;
        const uint8_t* x = reinterpret_cast<const uint8_t*>(__shfl_sync(0xffffffffu, xs, j));
        const uint8_t* y = reinterpret_cast<const uint8_t*>(__shfl_sync(0xffffffffu, ys, j));
        const uint32_t len = __shfl_sync(0xffffffffu, ln, j);
        settle(j, warp_equal(x, y, len));
      }
    }
    if (G == 1) {  // the block's own count, without the round trip to the counter
      if (!__syncthreads_or(stay)) break;
    } else {
      ok = grid_barrier(a.ctl, G, a.wait_ns, false);
      if (!ok) break;
      if (ldcg_u32(&a.ctl->unres[round % 3]) == 0) break;
    }
    for (uint32_t g = tid; g < N; g += nth)
      if (ldcg_u32(&ch.res[g]) == kResUnresolved) a.tbl[ch.ent[g]].minv = 0;
    ok = grid_barrier(a.ctl, G, a.wait_ns, false);
    if (!ok) break;
    for (uint32_t base = tid - lane; base < N; base += nth) {
      const uint32_t g = base + lane;
      post_minimum(a, g < N && ldcg_u32(&ch.res[g]) == kResUnresolved ? ch.ent[g] : 0xFFFFFFFFu, g);
    }
    ok = grid_barrier(a.ctl, G, a.wait_ns, false);
    ++round;
  }

  // contiguous chunk range of each block, for the ranks
  const uint64_t per = (((uint64_t)N + G - 1) / G + 31) & ~31ull;
  const uint32_t lo = (uint32_t)min((uint64_t)N, bid * per);
  const uint32_t hi = (uint32_t)min((uint64_t)N, lo + per);
  // A verify reject: the cache had a key+length candidate, or an earlier miss of
  // the call has this key and length (another leader of a later round; with
  // classes, an earlier leader of the class).  And the miss's entry of the group
  // table is left zeroed for the next call: every claimed entry belongs to a
  // group with at least one leader.
  auto settle_leader = [&](uint32_t g, uint32_t r) {
    bool earlier;
    if (a.classes) {
      const uint32_t cl = (uint32_t)ch.cls[g];  // in range unless the call failed
      earlier = cl <= a.tbl_mask && ~ldcg_u32(&a.cls_tbl[cl].minv) < g;
    } else {
      earlier = (r & kResRoundMask) > 1;
    }
    const bool rej = !(r & kResNoSlot) && (ch.status[g] == kMissCand || earlier);
    if (rej) ch.res[g] = r | kResReject;
    const uint32_t e = ch.ent[g];
    if (e != 0xFFFFFFFFu) a.tbl[e] = CallEntry{0u, 0u};
  };

  // ---- D1: misses per contiguous block range --------------------------------
  unsigned long long before = 0, total = 0, sbefore = 0, stotal = 0, evict = 0;
  if (ok && !counted) {
    uint32_t cnt = 0, scnt = 0;
    for (uint32_t g = lo + threadIdx.x; g < hi; g += kThreads) {
      const uint32_t r = ldcg_u32(&ch.res[g]);
      if (r & kResLeader) {
        ++cnt;
        if (!(r & kResNoSlot)) ++scnt;
        settle_leader(g, r);
      }
    }
    const unsigned long long c = block_sum<unsigned long long>(cnt, red64);
    const unsigned long long sc = block_sum<unsigned long long>(scnt, red64);
    if (G == 1) {
      total = c;
      stotal = sc;
    } else {
      if (threadIdx.x == 0) {
        a.bcount[bid] = (uint32_t)c;
        a.bcount[G + bid] = (uint32_t)sc;
      }
      ok = grid_barrier(a.ctl, G, a.wait_ns, false);
    }
  }
  if (threadIdx.x == 0) s_slots0 = my_slots0;
  __syncthreads();
  const unsigned long long slots0 = s_slots0;
  // ---- D2: exclusive miss rank of every chunk; per-payload start ranks ------
  if (ok && G > 1) {
    for (uint32_t j = threadIdx.x; j < G; j += kThreads) {
      const uint32_t v = ldcg_u32(&a.bcount[j]);
      const uint32_t sv = ldcg_u32(&a.bcount[G + j]);
      total += v;
      stotal += sv;
      if (j < bid) {
        before += v;
        sbefore += sv;
      }
    }
    before = block_sum<unsigned long long>(before, red64);
    total = block_sum<unsigned long long>(total, red64);
    sbefore = block_sum<unsigned long long>(sbefore, red64);
    stotal = block_sum<unsigned long long>(stotal, red64);
  }
  if (ok) {
    if (stotal > a.nslots - slots0) {
      // LRU: evict the missing slots among those this call did not hit
      evict = stotal - (a.nslots - slots0);
      if (!a.lru || evict > slots0 - __ldcg(&a.ctl->acc_distinct)) {
        if (threadIdx.x == 0) atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_CAPACITY);
        ok = false;
      }
    }
  }
  if (ok && a.classes) {
    // every read of the class table happened before the last barrier: the
    // grid clears the call's whole table with plain 16-byte stores (a
    // clear per chunk would first load the chunk's class entry)
    uint4* t4 = reinterpret_cast<uint4*>(a.cls_tbl);
    const unsigned long long n4 = a.tbl_mask + 1;  // one 16-byte store per entry
    for (unsigned long long e = tid; e < n4; e += nth) t4[e] = make_uint4(0u, 0u, 0u, 0u);
  }
  if (ok) {
    unsigned long long running = before, srunning = sbefore;
    uint32_t n_ahead = 0;  // misses that the hash kernel wrote where they belong
    for (uint32_t t = lo; t < hi; t += kThreads) {
      const uint32_t g = t + threadIdx.x;
      const bool valid = g < hi;
      const uint32_t rv = valid ? ldcg_u32(&ch.res[g]) : 0u;
      const bool miss = valid && (rv & kResLeader);
      const bool stored = miss && !(rv & kResNoSlot);
      if (counted && miss) settle_leader(g, rv);
      const uint32_t mb = __ballot_sync(0xffffffffu, miss);
      const uint32_t sb = __ballot_sync(0xffffffffu, stored);
      if (lane == 0) {
        warp_cnt[w] = __popc(mb);
        swarp_cnt[w] = __popc(sb);
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        uint32_t acc = 0, sacc = 0;
        for (int k = 0; k < kWarps; ++k) {
          warp_off[k] = acc;
          acc += warp_cnt[k];
          swarp_off[k] = sacc;
          sacc += swarp_cnt[k];
        }
        warp_cnt[0] = acc;
        swarp_cnt[0] = sacc;
      }
      __syncthreads();
      const uint32_t below = (1u << lane) - 1u;
      if (valid) {
        const uint32_t r = (uint32_t)(running + warp_off[w] + __popc(mb & below));
        ch.rank[g] = r;
        if (miss) ch.order[r] = g;
        if (stored) {
          const uint32_t sr = (uint32_t)(srunning + swarp_off[w] + __popc(sb & below));
          ch.srank[g] = sr;
          n_ahead += a.spec_active && evict == 0 && sr == g && ch.spec[g];
        }
        const uint32_t p = ch.pidx[g];
        if (g == desc(a, p).chunk_base) a.pstart[p] = r;
      }
      running += warp_cnt[0];
      srunning += swarp_cnt[0];
      __syncthreads();
    }
    if (a.spec_active) {
      const unsigned long long s = block_sum<unsigned long long>(n_ahead, red64);
      if (threadIdx.x == 0 && s) atomicAdd(&a.ctl->spec_ahead, s);
    }
    // no barrier: what reads the ranks follows a kernel boundary or a barrier
    // of its own, and an eviction's first barrier comes before it writes
    // anything that a slower block may still read here
  }
  if (ok && evict && G == 1) {  // its barriers did not read the error word
    if (threadIdx.x == 0) s_err1 = ld_volatile_s32(&a.ctl->err);
    __syncthreads();
    ok = s_err1 == 0;
  }
  if (ok && evict) ok = lru_evict(a, G, bid, slots0, evict, sred, warp_cnt, warp_off, red64);
  // totals for k_pack (the capacity check above left them unpublished on error)
  if (ok && bid == 0 && threadIdx.x == 0) {
    a.ctl->acc_misses = total;
    a.ctl->acc_stored = stotal;
    a.ctl->evict_k = evict;
  }
  return false;
}

// After an error, by the call's last block: what the failed call may have left is
// taken back.  Its group entries, where the error stopped the leaders before they
// cleared them (the whole group table, and class table); an eviction's histogram
// and flags; and, if the call failed while it copied, the last uses that its hits
// stamped and its index entries: those of slots from slots0 on, the slots used
// before the call (they filled free entries, so the tables are then what they
// were; what an eviction removed stays removed).  Out of line: rare, and kept out
// of the code that every call runs.
__device__ __noinline__ void clear_after_error(const DedupArgs& a, int err,
                                               unsigned long long slots0) {
  for (unsigned long long e = threadIdx.x; e <= a.tbl_mask; e += kThreads) {
    a.tbl[e].owner = 0u;
    a.tbl[e].minv = 0u;
    if (a.classes) a.cls_tbl[e] = ClassEntry{0u, 0u, 0u, 0u};
  }
  if (a.lru) {  // an eviction that stopped half-way may have left these set
    for (uint32_t j = threadIdx.x; j < kLruBins; j += kThreads) a.bins[j] = 0u;
    for (unsigned long long j = threadIdx.x; j < a.nslots; j += kThreads) a.vflag[j] = 0;
  }
  if (err == (int)GLEAM_ERR_CAPACITY) return;  // found before the copies
  if (a.lru)
    for (unsigned long long g = threadIdx.x; g < a.Ntot; g += kThreads)
      if (a.ch.status[g] == kHit0 && a.ch.old[g] != a.epoch)
        a.last_use[a.ch.ent[g]] = a.ch.old[g];
#pragma unroll 4
  for (unsigned long long q = threadIdx.x; q <= a.index_mask; q += kThreads) {
    const uint32_t s1 = a.index[q].slot, s2 = a.hints[q].slot;
    if (s1 < kTombSlot && s1 >= slots0) a.index[q].slot = kEmptySlot;
    if (s2 < kTombSlot && s2 >= slots0) a.hints[q].slot = kEmptySlot;
  }
}

// The end of a call, run by every block of its last kernel (finish_call): the
// last block to get here publishes the counters and results and leaves the
// per-call state (group table, control block) as the next call expects it.
// total/stored/evict/vbytes: the call's misses, stored misses, evicted slots and
// their bytes; s_sum: a grid of one block's sums (hits, intra hits, rejects, miss
// bytes, stored bytes, chunks written ahead, of them used), else the control
// block's.
//
// Whether the calling block is the last of n to count itself here; what the
// others wrote before is then visible to it.  Called by every thread.
__device__ __forceinline__ bool last_to_arrive(unsigned int* count, uint32_t n) {
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    if (n == 1) {  // the block barrier already orders the block's own writes
      s_last = 1;
    } else {
      __threadfence();
      s_last = atomicAdd(count, 1u) == n - 1;
    }
  }
  __syncthreads();
  if (!s_last) return false;
  if (n > 1) __threadfence();
  return true;
}

__device__ __forceinline__ void publish_call(const DedupArgs& a, bool one,
                                             unsigned long long slots0,
                                             unsigned long long total,
                                             unsigned long long s_stored,
                                             unsigned long long evict,
                                             unsigned long long s_vbytes,
                                             const unsigned long long* s_sum) {
  const uint32_t N = (uint32_t)a.Ntot;
  const int err = ld_volatile_s32(&a.ctl->err);
  if (threadIdx.x == 0) {
    const unsigned long long misses = total;
    const unsigned long long hc = one ? s_sum[0] : __ldcg(&a.ctl->acc_hits_cache);
    const unsigned long long hi2 = one ? s_sum[1] : __ldcg(&a.ctl->acc_hits_intra);
    const unsigned long long rej = one ? s_sum[2] : __ldcg(&a.ctl->acc_rejects);
    const unsigned long long mbytes = one ? s_sum[3] : __ldcg(&a.ctl->acc_miss_bytes);
    const unsigned long long sbytes = one ? s_sum[4] : __ldcg(&a.ctl->acc_stored_bytes);
    const unsigned long long stored = s_stored;
    const unsigned long long vbytes = s_vbytes;
    const unsigned long long spec = one ? s_sum[5] : __ldcg(&a.ctl->spec_tried);
    const unsigned long long spec_used = one ? s_sum[6] : __ldcg(&a.ctl->spec_used);
    if (err == 0 && a.spec_state) {
      // automatic write-through: stays on while at least half of the chunks
      // written ahead were used; once off, tried again after 256 calls
      uint32_t* st = a.spec_state;
      if (spec) {
        st[0] = 2 * spec_used >= spec ? 1u : 0u;
        st[1] = 0;
      } else if (st[0] == 0 && ++st[1] >= 256) {
        st[0] = 1;
        st[1] = 0;
      }
      *a.spec_mirror = st[0];
    }
    if (err == 0) {  // no reads: the counters change by atomic adds
      atomicAdd(&a.dstats[ST_CALLS], a.ncalls);
      atomicAdd(&a.dstats[ST_CHUNKS], (unsigned long long)N);
      atomicAdd(&a.dstats[ST_HITS_CACHE], hc);
      atomicAdd(&a.dstats[ST_HITS_INTRA], hi2);
      atomicAdd(&a.dstats[ST_MISSES], misses);
      atomicAdd(&a.dstats[ST_INSERTS], stored);
      atomicAdd(&a.dstats[ST_REJECTS], rej);
      a.dstats[ST_SLOTS_USED] = slots0 + stored - evict;
      atomicAdd(&a.dstats[ST_BYTES_USED], sbytes - vbytes);
      atomicAdd(&a.dstats[ST_EVICTIONS], evict);
      if (spec) atomicAdd(&a.dstats[ST_SPEC_CHUNKS], spec);
    }
    gleam_result_t* t = a.total;
    t->status = err;
    t->n_miss = err ? 0 : misses;
    t->n_hit_cache = err ? 0 : hc;
    t->n_hit_intra = err ? 0 : hi2;
    t->verify_rejects = err ? 0 : rej;
    t->miss_bytes = err ? 0 : mbytes;
  }
  for (uint32_t p = threadIdx.x; p < a.count; p += kThreads) {
    gleam_result_t* r = desc(a, p).result;
    if (!r) continue;
    r->status = err;
    if (err) {
      r->n_miss = 0;
      r->n_hit_cache = 0;
      r->n_hit_intra = 0;
      r->verify_rejects = 0;
      r->miss_bytes = 0;
    }
  }
  // Leave the per-call state as the next call expects it: the group table
  // (cleared entry by entry by the leaders, or here in full after an error
  // that may have stopped them) and the control block.
  if (err) clear_after_error(a, err, slots0);
  __syncthreads();
  if (threadIdx.x == 0) {
    DevCtl* c = a.ctl;
    c->bar_count = 0;
    c->copy_next = 0;
    c->err = 0;
    c->unres[0] = c->unres[1] = c->unres[2] = 0;
    c->shared_groups = 0;
    c->any_miss = 0;
    c->hits_done = 0;
    c->acc_hits_cache = c->acc_hits_intra = c->acc_rejects = 0;
    c->acc_misses = c->acc_miss_bytes = 0;
    c->acc_stored = c->acc_stored_bytes = 0;
    c->acc_distinct = c->evict_k = c->lru_below = c->lru_ties = c->acc_victim_bytes = 0;
    c->lru_hi = c->lru_cut = 0;
    c->spec_tried = c->spec_used = c->spec_ahead = 0;
    c->done = 0;
  }
  __threadfence();
}

// Every block of the grid is counted, not only the G that share the work (the
// others get there by leave_general_to; where G is 1, so is the grid).
__device__ __forceinline__ void finish_call(const DedupArgs& a, uint32_t G,
                                            unsigned long long slots0,
                                            unsigned long long total,
                                            unsigned long long s_stored,
                                            unsigned long long evict,
                                            unsigned long long s_vbytes,
                                            const unsigned long long* s_sum) {
  if (last_to_arrive(&a.ctl->done, G == 1 ? 1u : gridDim.x))
    publish_call(a, G == 1, slots0, total, s_stored, evict, s_vbytes, s_sum);
}

// The rest of a call whose every chunk is a cache hit (DevCtl::any_miss), done
// by k_dedup after its first phase: hit masks of ones, the matched slots, and
// counts that follow from the payloads' sizes, without the rounds, ranks,
// sums and atomics of the other calls; k_pack then finds the call published
// and returns.  498 MB of 4 KiB chunks in 148 payloads, all cached: 195 us the
// call without it, 192 with (194 and 183 while a k_dedup of this grid was
// launched early).  Had the hash kernel stored the flag, once per warp that held
// a miss, k_dedup could leave its first phase too (2 us less), but the stores to
// one address cost 256 MiB of 1 KiB chunks 5%.  Out of line.
//
// ok: the block passed its barrier and saw no error.  The blocks need not agree on
// that (a wait may run out as the last block arrives), so each is counted
// whatever it saw, and the last of them decides by the error word: after an
// error the call stays unpublished, and k_pack ends it as it ends any failed one.
__device__ __noinline__ void publish_all_hits(const DedupArgs& a, uint32_t G, uint32_t bid,
                                              bool ok) {
  __shared__ unsigned long long red64[kWarps];
  __shared__ unsigned long long s_sum[7];
  const uint32_t N = (uint32_t)a.Ntot;
  const uint32_t tid = bid * kThreads + threadIdx.x, nth = G * kThreads;
  const ChunkArrays& ch = a.ch;
  const unsigned long long slots0 =
      *(volatile const unsigned long long*)&a.dstats[ST_SLOTS_USED];
  for (uint32_t p = ok ? tid : a.count; p < a.count; p += nth) {
    const PayloadDesc& P = desc(a, p);
    gleam_result_t* r = P.result;
    if (!r) continue;
    r->n_miss = 0;
    r->n_hit_cache = P.nchunks;
    r->n_hit_intra = 0;
    r->verify_rejects = 0;
    r->miss_bytes = 0;
  }
  uint32_t n_spec = 0;
#pragma unroll 4
  for (uint32_t g = ok ? tid : N; g < N; g += nth) {
    const PayloadDesc& P = desc(a, ch.pidx[g]);
    const unsigned long long i = g - P.chunk_base, left = P.nchunks - i;
    if ((i & 31) == 0)
      P.mask[i >> 5] = left >= 32 ? 0xffffffffu : (1u << (uint32_t)left) - 1u;
    if (P.chunk_slot) P.chunk_slot[i] = ch.ent[g];
    n_spec += a.spec_active && ch.spec[g];
  }
  const unsigned long long b_spec =
      a.spec_active ? block_sum<unsigned long long>(n_spec, red64) : 0ull;
  if (threadIdx.x == 0) {
    if (G == 1) {
      for (int k = 0; k < 7; ++k) s_sum[k] = 0;
      s_sum[0] = N;
      s_sum[5] = b_spec;
    } else {
      if (bid == 0) atomicAdd(&a.ctl->acc_hits_cache, (unsigned long long)N);
      if (b_spec) atomicAdd(&a.ctl->spec_tried, b_spec);
    }
  }
  if (!last_to_arrive(&a.ctl->hits_done, G) || !ok || ld_volatile_s32(&a.ctl->err) != 0) return;
  __syncthreads();  // every thread has read the error word, which publish_call resets
  if (threadIdx.x == 0) a.ctl->published = 1u;
  publish_call(a, G == 1, slots0, 0ull, 0ull, 0ull, 0ull, s_sum);
}

// Second kernel of the call (a regular launch sized for the copies): hit
// masks, miss indices, chunk slots, per-payload counters, then every miss by
// rank copied by whole warps to the packed output and its arena slot and
// inserted into the index; the last block publishes the counters and results
// and leaves the per-call state zeroed.  Nothing is written after an error.
// kPlain: the misses are copied by whole warps (DedupArgs::plain_copy), a
// variant of its own so that the bulk copies' kernels carry none of its code.
template <bool kPlain>
__device__ __forceinline__ void pack_publish(const DedupArgs& a, uint32_t G, uint32_t bid,
                                             uint8_t* pack_smem) {
  __shared__ unsigned long long red64[kWarps];
  __shared__ unsigned long long s_slots0, s_total, s_evict;
  // a grid of one block keeps its totals here instead of in the control block
  __shared__ unsigned long long s_stored, s_vbytes, s_ahead, s_sum[7];
  __shared__ int s_err;
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t N = (uint32_t)a.Ntot;
  const ChunkArrays& ch = a.ch;
  if (threadIdx.x == 0) {
    s_slots0 = *(volatile const unsigned long long*)&a.dstats[ST_SLOTS_USED];
    s_err = ld_volatile_s32(&a.ctl->err);
    s_total = __ldcg(&a.ctl->acc_misses);
    s_evict = __ldcg(&a.ctl->evict_k);
    s_stored = __ldcg(&a.ctl->acc_stored);
    s_vbytes = __ldcg(&a.ctl->acc_victim_bytes);
    s_ahead = a.spec_active ? __ldcg(&a.ctl->spec_ahead) : 0ull;
    for (int k = 0; k < 7; ++k) s_sum[k] = 0;
  }
  __syncthreads();
  const unsigned long long slots0 = s_slots0;
  const unsigned long long total = s_total;
  const unsigned long long evict = s_evict;
  const bool ok = s_err == 0;
  const uint32_t wbase =
      kPlain ? 0u : (uint32_t)__cvta_generic_to_shared(pack_smem) + w * kPackWarpBytes;
  const uint32_t bufs = wbase, bars = wbase + kPackBufs * kPackPiece;
  PackMeta* meta = reinterpret_cast<PackMeta*>(pack_smem + w * kPackWarpBytes +
                                               kPackBufs * kPackPiece + 64);
  PackRing ring{0u, 0u, 0u};
  if constexpr (!kPlain) {
    if (lane == 0) {
      for (uint32_t b = 0; b < kPackBufs; ++b) mbar_init(bars + 8 * b);
      mbar_fence_init();
    }
    __syncwarp();
  }
  bool bulk_failed = false;
  // slot of the stored miss of stored rank sr: the evicted slots in ascending
  // order, then never-used slots
  auto slot_of = [&](uint32_t sr) -> unsigned long long {
    return sr < evict ? (unsigned long long)__ldcg(&a.victims[sr]) : slots0 + (sr - evict);
  };

  // ---- after an error: give the hit slots their last use back (LRU; the first
  // hit to stamp a slot kept its old value) ------------------------------------
  if (!ok && a.lru) {
    for (unsigned long long g = (unsigned long long)bid * kThreads + threadIdx.x; g < N;
         g += (unsigned long long)G * kThreads)
      if (ch.status[g] == kHit0 && ch.old[g] != a.epoch) a.last_use[ch.ent[g]] = ch.old[g];
  }

  // ---- hit masks, miss indices, chunk slots, counters ------------------------
  if (ok) {
    unsigned long long n_hc = 0, n_hi = 0, n_rej = 0, n_bytes = 0, n_sbytes = 0;
    uint32_t n_spec = 0, n_spec_used = 0;  // write-through: chunks written ahead, used
    // Each warp classifies a contiguous range of chunks (whole 32-chunk
    // steps), so that its steps mostly fall in one payload: the counters of a
    // payload are summed in the warp over its steps and added once where the
    // warp leaves the payload, instead of once per step by every warp on the
    // same few addresses (a one-payload call of a million chunks would queue
    // ~10^5 atomics on one result).
    const unsigned long long nsteps = ((unsigned long long)N + 31) / 32;
    const unsigned long long cw_n = (unsigned long long)G * kWarps;
    const unsigned long long cw = (unsigned long long)bid * kWarps + w;
    const unsigned long long c_lo = nsteps * cw / cw_n * 32;
    const unsigned long long c_hi = min((unsigned long long)N, nsteps * (cw + 1) / cw_n * 32);
    gleam_result_t* acc_res = nullptr;  // the payload whose counters the warp holds
    unsigned long long acc_hc = 0, acc_hi = 0, acc_miss = 0, acc_rej = 0, acc_len = 0;
    auto flush = [&]() {
      if (acc_res && lane == 0) {
        if (acc_hc) atomicAdd((unsigned long long*)&acc_res->n_hit_cache, acc_hc);
        if (acc_hi) atomicAdd((unsigned long long*)&acc_res->n_hit_intra, acc_hi);
        if (acc_miss) atomicAdd((unsigned long long*)&acc_res->n_miss, acc_miss);
        if (acc_rej) atomicAdd((unsigned long long*)&acc_res->verify_rejects, acc_rej);
        if (acc_len) atomicAdd((unsigned long long*)&acc_res->miss_bytes, acc_len);
      }
      acc_res = nullptr;
      acc_hc = acc_hi = acc_miss = acc_rej = acc_len = 0;
    };
    for (unsigned long long t = c_lo; t < c_hi; t += 32) {
      const uint32_t g = (uint32_t)(t + lane);
      const bool valid = t + lane < c_hi;
      const uint32_t r = valid ? ldcg_u32(&ch.res[g]) : 0u;
      const uint32_t p = valid ? ch.pidx[g] : 0xFFFFFFFFu;
      const bool miss = valid && (r & kResLeader);
      bool hc = false, hi2 = false, rej = false;
      uint32_t len = 0, bit = 0;
      unsigned long long mw = 0;  // address of the chunk's hit-mask word, if a hit
      gleam_result_t* res = nullptr;
      if (valid) {
        const PayloadDesc& P = desc(a, p);
        const unsigned long long i = g - P.chunk_base;
        res = P.result;
        if (r & kResHit0) hc = true;
        if (r & kResDup) {
          if (ch.pidx[ch.ent[g]] == p) hi2 = true;  // leader in the same payload
          else hc = true;                           // inserted by an earlier payload
        }
        if (hc || hi2) {
          mw = (unsigned long long)(P.mask + (i >> 5));
          bit = 1u << (i & 31);
        }
        if (P.chunk_slot) {
          uint32_t sl;
          if (r & kResHit0) sl = ch.ent[g];                                      // matched slot
          else if (r & kResDup) sl = (uint32_t)slot_of(__ldcg(&ch.srank[ch.ent[g]]));  // leader's
          else if (r & kResNoSlot) sl = kEmptySlot;                              // never cached
          else sl = (uint32_t)slot_of(ch.srank[g]);                              // its new slot
          P.chunk_slot[i] = sl;
        }
        if (miss) {
          len = ch.len[g];
          P.miss_idx[ch.rank[g] - __ldcg(&a.pstart[p])] = (uint32_t)i;
          rej = (r & kResReject) != 0;
        }
      }
      n_spec += a.spec_active && valid && ch.spec[g];
      n_hc += hc;
      n_hi += hi2;
      n_rej += rej;
      n_bytes += len;
      if (!(r & kResNoSlot)) n_sbytes += len;
      // hit-mask words and per-payload result counters: one atomic per group
      // of lanes that share the word or the payload
      const unsigned mpeers = __match_any_sync(0xffffffffu, mw);
      const uint32_t bits = __reduce_or_sync(mpeers, bit);
      if (mw && lane == (uint32_t)(__ffs(mpeers) - 1)) atomicOr((uint32_t*)mw, bits);
      const unsigned peers = __match_any_sync(0xffffffffu, res ? p : 0xFFFFFFFFu);
      if (peers == 0xffffffffu && res) {  // the whole step in one payload that has a result
        if (res != acc_res) {
          flush();
          acc_res = res;
        }
        acc_hc += __reduce_add_sync(0xffffffffu, (uint32_t)hc);
        acc_hi += __reduce_add_sync(0xffffffffu, (uint32_t)hi2);
        acc_miss += __reduce_add_sync(0xffffffffu, (uint32_t)miss);
        acc_rej += __reduce_add_sync(0xffffffffu, (uint32_t)rej);
        acc_len += __reduce_add_sync(0xffffffffu, len);
      } else {  // payload boundaries: one atomic per group of lanes per counter
        const bool lead = res && lane == (uint32_t)(__ffs(peers) - 1);
        add_in_group((unsigned long long*)(lead ? &res->n_hit_cache : nullptr), peers, hc);
        add_in_group((unsigned long long*)(lead ? &res->n_hit_intra : nullptr), peers, hi2);
        add_in_group((unsigned long long*)(lead ? &res->n_miss : nullptr), peers, miss);
        add_in_group((unsigned long long*)(lead ? &res->verify_rejects : nullptr), peers, rej);
        add_in_group((unsigned long long*)(lead ? &res->miss_bytes : nullptr), peers, len);
      }
    }
    flush();
    // Every miss's bytes, in pieces of kPackPiece bytes: piece k of the miss
    // of rank r is number r * ppc + k (ppc = pieces of a whole chunk; a
    // shorter miss has fewer), and warp gw owns the contiguous numbers
    // [plo, phi), so that a call with few misses still spreads its copies over
    // every warp (one 64 KiB miss is 32 pieces) and a call with many streams
    // whole runs of chunks per warp.  The lanes fetch the metadata of 32
    // pieces at once (mostly one chunk's: the same addresses), then the pieces
    // go to the packed output and the miss's arena slot, all but those of
    // misses the hash kernel already wrote there.
    const unsigned long long nw = (unsigned long long)G * kWarps;
    const unsigned long long gw = (unsigned long long)bid * kWarps + w;
    const unsigned long long ppc = (a.C + kPackPiece - 1) / kPackPiece;
    const unsigned long long npieces = total * ppc;
    const unsigned long long plo = npieces * gw / nw, phi = npieces * (gw + 1) / nw;
    // written ahead by the hash kernel exactly where it belongs: with no
    // eviction, stored rank g means every earlier chunk of the call is a
    // stored miss, so the chunk's packed offset is i*C and its slot
    // slots_used + g, the places it was written to
    auto written_ahead = [&](uint32_t gg, uint32_t sr) {
      return a.spec_active && evict == 0 && sr == gg && ch.spec[gg];
    };
    // Mostly the warps take their steps from a counter of
    // the call instead (each asks for its next step before it copies the
    // current one), so that warps on SMs that copy faster take more: steps of
    // 32 pieces, then, from kFinePerWarp pieces per warp before the end,
    // steps of kFineStep, so that the last steps end together.
    // The static ranges remain where the hash kernel wrote at least half of the
    // misses ahead (the steps then copy little, and the counter's round trip
    // would be most of a step), where a warp has less than a fine step (a batch
    // of 665 misses of 64 KiB, 5.8 pieces a warp: 246 us so, 252 with the
    // counter), and for counts the 32-bit counter cannot hold.
    // Where it wrote all of them ahead (a first load) there is nothing to copy,
    // and no step looks its pieces up to find that out (498 MB in 148 payloads,
    // none cached: 344 -> 341 us).
    const bool grab =
        2 * s_ahead < total && npieces >= kFineStep * nw && npieces < (1ull << 31);
    const unsigned long long coarse =
        npieces > nw * kFinePerWarp ? (npieces - nw * kFinePerWarp) / 32 : 0ull;
    auto step_at = [&](unsigned long long v) {  // first piece of the counter's v-th step
      return v <= coarse ? 32 * v : 32 * coarse + kFineStep * (v - coarse);
    };
    unsigned long long step = plo, step_end = s_ahead == total ? plo : phi;
    if (grab) {
      uint32_t b0 = 0;
      if (lane == 0) b0 = atomicAdd(&a.ctl->copy_next, 1u);
      step = __shfl_sync(0xffffffffu, b0, 0);
      step_end = min(npieces, step_at(step + 1));
      step = step_at(step);
    }
    while (step < (grab ? npieces : step_end)) {
      uint32_t next = 0;
      if (grab && lane == 0) next = atomicAdd(&a.ctl->copy_next, 1u);
      const unsigned long long shi = min(step_end, step + 32);
      const unsigned long long pc = step + lane;
      uint32_t bytes = 0;
      bool copy = false;
      unsigned long long src = 0, d1 = 0, d2 = 0;
      uint32_t pp = 0;
      if (pc < shi) {
        const unsigned long long r = pc / ppc;
        const uint32_t off = (uint32_t)(pc - r * ppc) * kPackPiece;
        const uint32_t gg = ch.order[r];
        const uint32_t ln = ch.len[gg];
        if (off < ln) {
          pp = ch.pidx[gg];
          const PayloadDesc& P = desc(a, pp);
          bytes = min(kPackPiece, ln - off);
          src = ch.src[gg] + off;
          d1 = (unsigned long long)(P.packed + (r - a.pstart[pp]) * a.C + off);
          uint32_t sr = 0xFFFFFFFFu;
          if (!(ch.res[gg] & kResNoSlot)) {  // else sent, never cached
            sr = ch.srank[gg];
            d2 = (unsigned long long)(a.arena + slot_of(sr) * a.C + off);
          }
          copy = !written_ahead(gg, sr);
        }
      }
      const unsigned cmask = __ballot_sync(0xffffffffu, copy);  // lanes whose piece is copied
      const uint32_t m = __popc(cmask);
      if constexpr (!kPlain) {
        if (copy) meta[__popc(cmask & ((1u << lane) - 1u))] = PackMeta{src, d1, d2, bytes, 0u};
        __syncwarp();
        if (lane == 0 && m && !bulk_failed &&
            !bulk_copy_batch(meta, m, bufs, bars, ring, a.wait_ns)) {
          bulk_failed = true;
          atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_TIMEOUT);
        }
        if (copy) {  // the piece's last bytes % 16 (only a miss's last piece has any)
          const uint8_t* sp = reinterpret_cast<const uint8_t*>(src);
          uint8_t* x = reinterpret_cast<uint8_t*>(d1);
          uint8_t* y = reinterpret_cast<uint8_t*>(d2);
          for (uint32_t k = bytes & ~15u; k < bytes; ++k) {
            x[k] = sp[k];
            if (y) y[k] = sp[k];
          }
        }
        __syncwarp();
      }
      for (unsigned todo = kPlain ? cmask : 0u; todo; todo &= todo - 1) {
        const int j = __ffs(todo) - 1;
        const unsigned long long sj = __shfl_sync(0xffffffffu, src, j);
        const unsigned long long xj = __shfl_sync(0xffffffffu, d1, j);
        const unsigned long long yj = __shfl_sync(0xffffffffu, d2, j);
        const uint32_t lj = __shfl_sync(0xffffffffu, bytes, j);
        warp_copy2(reinterpret_cast<uint8_t*>(xj), reinterpret_cast<uint8_t*>(yj),
                   reinterpret_cast<const uint8_t*>(sj), lj,
                   desc(a, __shfl_sync(0xffffffffu, pp, j)));
      }
      if (grab) {
        const unsigned long long v = __shfl_sync(0xffffffffu, next, 0);
        step = step_at(v);
        step_end = min(npieces, step_at(v + 1));
      } else {
        step += 32;
      }
    }
    // Every miss's index and hint-table entries, by rank: warp gw owns the
    // contiguous ranks [lo, hi), each lane inserting its own chunk (32
    // independent probes at a time).
    const unsigned long long lo = total * gw / nw, hi = total * (gw + 1) / nw;
    for (unsigned long long base = lo; base < hi; base += 32) {
      const unsigned long long r = base + lane;
      if (r >= hi) continue;
      const uint32_t gg = ch.order[r];
      if (ch.res[gg] & kResNoSlot) continue;  // sent, never cached
      const uint32_t ln = ch.len[gg];
      const uint32_t sr = ch.srank[gg];
      const unsigned long long slot = slot_of(sr);
      n_spec_used += written_ahead(gg, sr);
      a.slot_len[slot] = ln;
      a.slot_key[slot] = ch.key[gg];
      if (a.lru) a.last_use[slot] = a.epoch;
      if (!index_insert(a.index, a.index_mask, index_key(a, ch.key[gg]), (uint32_t)slot, ln,
                        a.key16, a.classes ? (uint32_t)(ch.cls[gg] >> 32) : 0u))
        atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_INTERNAL);
      if (!a.paper && ln >= kPrefixBytes &&
          !index_insert(a.hints, a.index_mask, ch.hint[gg], (uint32_t)slot, ln))
        atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_INTERNAL);
    }
    if (!kPlain && lane == 0) bulk_wait_all<0>();  // every piece written before the block ends
    n_hc = block_sum<unsigned long long>(n_hc, red64);
    n_hi = block_sum<unsigned long long>(n_hi, red64);
    n_rej = block_sum<unsigned long long>(n_rej, red64);
    n_bytes = block_sum<unsigned long long>(n_bytes, red64);
    n_sbytes = block_sum<unsigned long long>(n_sbytes, red64);
    const unsigned long long b_spec = block_sum<unsigned long long>(n_spec, red64);
    const unsigned long long b_spec_used = block_sum<unsigned long long>(n_spec_used, red64);
    if (threadIdx.x == 0 && G == 1) {
      s_sum[0] = n_hc;
      s_sum[1] = n_hi;
      s_sum[2] = n_rej;
      s_sum[3] = n_bytes;
      s_sum[4] = n_sbytes;
      s_sum[5] = b_spec;
      s_sum[6] = b_spec_used;
    } else if (threadIdx.x == 0) {
      atomicAdd(&a.ctl->acc_hits_cache, n_hc);
      atomicAdd(&a.ctl->acc_hits_intra, n_hi);
      atomicAdd(&a.ctl->acc_rejects, n_rej);
      atomicAdd(&a.ctl->acc_miss_bytes, n_bytes);
      atomicAdd(&a.ctl->acc_stored_bytes, n_sbytes);
      if (b_spec) atomicAdd(&a.ctl->spec_tried, b_spec);
      if (b_spec_used) atomicAdd(&a.ctl->spec_used, b_spec_used);
    }
  }

  finish_call(a, G, slots0, total, s_stored, evict, s_vbytes, s_sum);
}

// ---- one-launch resolve + pack of a one-payload call --------------------------
//
// A call of one payload that is launched chained (few enough chunks to leave
// most of the GPU idle) runs its resolution, ranks, packing and publishing in
// one launch: k_resolve_direct if the hash kernel claimed the misses' (key,
// length) groups as it recorded them, else (paper identifiers, and the
// single-block small call) the steps below.  Block b owns the contiguous chunks
// [b * per, (b + 1) * per), at most one per thread.  Phase 1 classifies them
// and claims their groups (a claim stores the claimant as the group's minimum;
// the group's other chunks post theirs later).  If no chunk of the call
// found its group claimed by another (no in-call duplicate and no key
// collision: the common case), every chunk that is not a cache hit is a miss of
// round one (its own group's first chunk), so after one grid barrier each block
// knows its misses' ranks from the blocks' counts, writes the outputs and
// inserts its misses; after a second barrier every warp of the grid copies its
// share of all misses' bytes (a block's own misses would leave the blocks that
// hold the most of them as the call's tail).  Otherwise the general algorithm
// takes over: the other minima are posted and resolve_rank and pack_publish run
// on the same grid.

// Bit k of the result: byte k of w (k < 4) is not v.
__device__ __forceinline__ uint32_t bytes_not(uint32_t w, uint32_t v) {
  const uint32_t x = w ^ (0x01010101u * v);
  const uint32_t t = (((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x) & 0x80808080u;  // bit 8k+7: byte k != 0
  return ((t >> 7) & 1u) | ((t >> 14) & 2u) | ((t >> 21) & 4u) | ((t >> 28) & 8u);
}

// The general algorithm on the one-launch kernel's grid, for a call with a
// shared group: if the hash kernel claimed the groups (pre), their entries are
// cleared and claimed again by the whole group key and length (a shared tag
// may be two different pairs'); then the group minima are posted, and the
// rounds, ranks and copies of k_dedup and k_pack run.  Out of line, so that
// the common path's code stays compact (the kernel runs once per call, on SMs
// whose instruction caches are cold).  Every thread of blocks 0 .. G-1 calls it,
// the other blocks of the grid call leave_general_to; mine: this thread holds a
// chunk of a group (entry e, group key and length).
template <bool kPlain>
__device__ __noinline__ void resolve_pack_general(const DedupArgs& a, uint32_t G, uint32_t bid,
                                                  uint8_t* smem, bool ok, bool pre, bool mine,
                                                  uint32_t e, unsigned long long key,
                                                  uint32_t len, uint32_t g) {
  if (pre) {
    if (mine && e != 0xFFFFFFFFu)
      *reinterpret_cast<volatile unsigned long long*>(&a.tbl[e]) = 0ull;
    ok = grid_barrier(a.ctl, G, a.wait_ns, false) && ok;
    if (ok && mine) {
      bool claimed = true;
      e = group_entry(a, g, key, len, &claimed, true);
      if (e == 0xFFFFFFFFu) {
        atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_INTERNAL);
        a.ch.res[g] = kResLeader | 1u;
      }
      a.ch.ent[g] = e;
    }
  }
  if (ok) post_minimum(a, mine && e != 0xFFFFFFFFu ? e : 0xFFFFFFFFu, g);  // one chunk per thread
  ok = grid_barrier(a.ctl, G, a.wait_ns, false);
  resolve_rank(a, G, bid, true, ok);
  grid_barrier(a.ctl, G, a.wait_ns, false);
  pack_publish<kPlain>(a, G, bid, smem);
}

// A block of the one-launch kernel that leaves the general algorithm to others.
// It may start after they are through, and decides by shared_groups that it has
// nothing to do: so it is counted at the end of the call like them, the last of
// the whole grid publishes, and no block of the call reads a control block that
// is already the next call's.
__device__ __noinline__ void leave_general_to(const DedupArgs& a) {
  if (!last_to_arrive(&a.ctl->done, gridDim.x)) return;
  publish_call(a, false, __ldcg(&a.dstats[ST_SLOTS_USED]), __ldcg(&a.ctl->acc_misses),
               __ldcg(&a.ctl->acc_stored), __ldcg(&a.ctl->evict_k),
               __ldcg(&a.ctl->acc_victim_bytes), nullptr);
}

template <bool kPlain>
__device__ __forceinline__ void resolve_pack_fast(const DedupArgs& a, uint32_t G, uint32_t bid,
                                                  uint8_t* smem) {
  __shared__ unsigned long long red64[kWarps];
  __shared__ uint32_t wcnt[kWarps], swcnt[kWarps];
  __shared__ unsigned long long s_slots0, s_sum[7];
  __shared__ int s_shared, s_err;
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const ChunkArrays& ch = a.ch;
  const PayloadDesc& P = a.one;
  const uint32_t N = (uint32_t)a.Ntot;
  const uint32_t per = (N + G - 1) / G;  // <= kThreads (the host sizes the grid)
  const uint32_t g = bid * per + threadIdx.x;
  const bool valid = threadIdx.x < per && g < N;
  if (per > kThreads && threadIdx.x == 0) atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_INTERNAL);
  const unsigned long long my_slots0 =
      threadIdx.x == 0 ? *(volatile const unsigned long long*)&a.dstats[ST_SLOTS_USED] : 0ull;
  if (threadIdx.x == 0) s_shared = 0;

  // ---- 1: classify, clear the outputs, claim the groups ----------------------
  if (bid == 0 && threadIdx.x == 0 && P.result) {
    gleam_result_t* r = P.result;
    r->n_miss = r->n_hit_cache = r->n_hit_intra = r->verify_rejects = r->miss_bytes = 0;
  }
  uint8_t st = kMissNoCand;
  uint32_t len = 0, e = 0xFFFFFFFFu;
  unsigned long long key = 0, hint = 0;
  bool lead = false, stored = false, shared = false;
  if (valid) {
    // the chunk's record at once (one round trip, whatever its status)
    st = ch.status[g];
    const unsigned long long key0 = ch.key[g];
    const uint32_t len0 = ch.len[g];
    hint = a.paper ? 0ull : ch.hint[g];
    if ((g & 31) == 0) P.mask[g >> 5] = 0;
    if (st == kHit0) {
      ch.res[g] = kResHit0;
    } else if (st == kUncached) {  // never cached: a miss of its own, in no group
      ch.ent[g] = 0xFFFFFFFFu;
      ch.res[g] = kResLeader | kResNoSlot | 1u;
      lead = true;
      len = len0;
    } else {
      key = key0;
      len = len0;
      bool claimed = true;
      e = group_entry(a, g, key, len, &claimed, true);
      if (e == 0xFFFFFFFFu) {
        atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_INTERNAL);
        ch.res[g] = kResLeader | 1u;
      } else {
        ch.res[g] = kResUnresolved;
      }
      ch.ent[g] = e;
      shared = !claimed;
      lead = stored = true;
    }
  }
  const uint32_t c_b = __syncthreads_count(lead);
  const uint32_t s_b = __syncthreads_count(stored);
  if (__syncthreads_or(shared) && threadIdx.x == 0) {
    s_shared = 1;
    if (G > 1) atomicOr(&a.ctl->shared_groups, 1u);
  }
  bool ok = true;
  if (G > 1 && threadIdx.x == 0) {
    a.bcount[bid] = c_b;
    a.bcount[G + bid] = s_b;
  }
  ok = grid_barrier(a.ctl, G, a.wait_ns, false);
  if (threadIdx.x == 0) {
    if (G > 1) s_shared = (int)ldcg_u32(&a.ctl->shared_groups);
    s_slots0 = my_slots0;
    s_err = G == 1 ? ld_volatile_s32(&a.ctl->err) : 0;
  }
  __syncthreads();
  if (G == 1) ok = s_err == 0;  // a grid of one did not read the error word

  if (s_shared) {
    resolve_pack_general<kPlain>(a, G, bid, smem, ok, false,
                                 valid && st != kHit0 && st != kUncached, e, key, len, g);
    return;
  }

  // ---- 2: the fast path: ranks, outputs, inserts; then copies ----------------
  const unsigned long long slots0 = s_slots0;
  unsigned long long before = 0, total = c_b, sbefore = 0, stotal = s_b;
  if (G > 1) {
    unsigned long long b0 = 0, t0 = 0, sb0 = 0, st0 = 0;
    for (uint32_t j = threadIdx.x; j < G; j += kThreads) {
      const uint32_t v = ldcg_u32(&a.bcount[j]), sv = ldcg_u32(&a.bcount[G + j]);
      t0 += v;
      st0 += sv;
      if (j < bid) {
        b0 += v;
        sb0 += sv;
      }
    }
    before = block_sum<unsigned long long>(b0, red64);
    total = block_sum<unsigned long long>(t0, red64);
    sbefore = block_sum<unsigned long long>(sb0, red64);
    stotal = block_sum<unsigned long long>(st0, red64);
  }
  if (ok && stotal > a.nslots - slots0) {  // every block decides the same
    if (threadIdx.x == 0) atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_CAPACITY);
    ok = false;
  }
  unsigned long long n_hc = 0, n_rej = 0, n_bytes = 0, n_sbytes = 0;
  uint32_t n_spec = 0, n_spec_used = 0;
  unsigned long long ins_slot = ~0ull;  // the slot this thread's stored miss takes
  if (ok) {
    // ranks within the block, in chunk order
    const uint32_t mb = __ballot_sync(0xffffffffu, lead);
    const uint32_t sb = __ballot_sync(0xffffffffu, stored);
    if (lane == 0) {
      wcnt[w] = __popc(mb);
      swcnt[w] = __popc(sb);
    }
    __syncthreads();
    uint32_t woff = 0, swoff = 0;
    for (uint32_t k2 = 0; k2 < w; ++k2) {
      woff += wcnt[k2];
      swoff += swcnt[k2];
    }
    const uint32_t below = (1u << lane) - 1u;
    const unsigned long long r = before + woff + __popc(mb & below);
    const unsigned long long sr = sbefore + swoff + __popc(sb & below);
    const unsigned long long slot = slots0 + sr;
    const bool spec = a.spec_active && valid && ch.spec[g];
    n_spec += spec;
    n_spec_used += spec && stored && sr == g;
    if (lead) {
      P.miss_idx[r] = g;
      ch.order[r] = g;  // for the copies, spread over the grid below
      ch.srank[g] = stored ? (uint32_t)sr : kEmptySlot;
      n_rej += st == kMissCand;
      n_bytes += len;
      if (stored) n_sbytes += len;
    }
    // hit-mask words: one atomic per group of lanes that share a word
    const bool hit = valid && st == kHit0;
    n_hc += hit;
    const unsigned long long mw = hit ? (unsigned long long)(P.mask + (g >> 5)) : 0ull;
    const unsigned mpeers = __match_any_sync(0xffffffffu, mw);
    const uint32_t bits = __reduce_or_sync(mpeers, hit ? 1u << (g & 31) : 0u);
    if (mw && lane == (uint32_t)(__ffs(mpeers) - 1)) atomicOr((uint32_t*)mw, bits);
    if (P.chunk_slot && valid)
      P.chunk_slot[g] = hit ? ch.ent[g] : stored ? (uint32_t)slot : kEmptySlot;
    ins_slot = stored ? slot : ~0ull;
  }
  ok = grid_barrier(a.ctl, G, a.wait_ns, false) && ok;
  if (ok) {
    // each stored miss records its slot and starts its index inserts (the
    // first claim attempts), which complete after the copies below
    const bool ins = ins_slot != ~0ull;
    const bool ins_hint = ins && !a.paper && len >= kPrefixBytes;
    PendingInsert pi{0ull, 0u}, ph{0ull, 0u};
    if (ins) {
      a.slot_len[ins_slot] = len;
      a.slot_key[ins_slot] = key;
      pi = index_insert_begin(a.index, a.index_mask, index_key(a, key), (uint32_t)ins_slot);
      if (ins_hint) ph = index_insert_begin(a.hints, a.index_mask, hint, (uint32_t)ins_slot);
    }
    // every miss's bytes, in pieces of kPackPiece bytes spread over all the
    // grid's warps (piece k of the miss of rank r is number r * ppc + k), all
    // but those of misses the hash kernel already wrote where they belong
    // (stored rank g means every earlier chunk is a stored miss: no eviction
    // here)
    const unsigned long long nw = (unsigned long long)G * kWarps;
    const unsigned long long gw = (unsigned long long)bid * kWarps + w;
    const unsigned long long ppc = (a.C + kPackPiece - 1) / kPackPiece;
    const unsigned long long npieces = total * ppc;
    const unsigned long long plo = npieces * gw / nw, phi = npieces * (gw + 1) / nw;
    const uint32_t wbase =
        kPlain ? 0u : (uint32_t)__cvta_generic_to_shared(smem) + w * kPackWarpBytes;
    const uint32_t bufs = wbase, bars = wbase + kPackBufs * kPackPiece;
    PackMeta* meta = reinterpret_cast<PackMeta*>(smem + w * kPackWarpBytes + kPackBufs * kPackPiece + 64);
    PackRing ring{0u, 0u, 0u};
    bool bulk_failed = false;
    if constexpr (!kPlain) {
      if (lane == 0) {
        for (uint32_t b = 0; b < kPackBufs; ++b) mbar_init(bars + 8 * b);
        mbar_fence_init();
      }
      __syncwarp();
    }
    // pieces [lo, hi) of the call, 32 at a time
    auto copy_range = [&](unsigned long long lo, unsigned long long hi) {
      for (unsigned long long base = lo; base < hi; base += 32) {
        const unsigned long long pc = base + lane;
        uint32_t bytes = 0;
        bool copy = false;
        unsigned long long src = 0, d1 = 0, d2 = 0;
        if (pc < hi) {
          const unsigned long long rr = pc / ppc;
          const uint32_t off = (uint32_t)(pc - rr * ppc) * kPackPiece;
          const uint32_t gg = __ldcg(&ch.order[rr]);
          const uint32_t ln = (uint32_t)min(a.C, P.n - (unsigned long long)gg * a.C);
          if (off < ln) {
            const uint32_t srr = __ldcg(&ch.srank[gg]);
            const bool ahead = a.spec_active && srr == gg && ch.spec[gg];
            if (!ahead) {
              bytes = min(kPackPiece, ln - off);
              src = (unsigned long long)(P.buf + (unsigned long long)gg * a.C + off);
              d1 = (unsigned long long)(P.packed + rr * a.C + off);
              d2 = srr != kEmptySlot ? (unsigned long long)(a.arena + (slots0 + srr) * a.C + off)
                                     : 0ull;
              copy = true;
            }
          }
        }
        const unsigned cmask = __ballot_sync(0xffffffffu, copy);
        if constexpr (!kPlain) {
          if (copy) meta[__popc(cmask & ((1u << lane) - 1u))] = PackMeta{src, d1, d2, bytes, 0u};
          __syncwarp();
          if (lane == 0 && cmask && !bulk_failed &&
              !bulk_copy_batch(meta, __popc(cmask), bufs, bars, ring, a.wait_ns)) {
            bulk_failed = true;
            atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_TIMEOUT);
          }
          if (copy) {  // the piece's last bytes % 16
            const uint8_t* sp = reinterpret_cast<const uint8_t*>(src);
            uint8_t* x = reinterpret_cast<uint8_t*>(d1);
            uint8_t* y = reinterpret_cast<uint8_t*>(d2);
            for (uint32_t k2 = bytes & ~15u; k2 < bytes; ++k2) {
              x[k2] = sp[k2];
              if (y) y[k2] = sp[k2];
            }
          }
          __syncwarp();
        }
        for (unsigned todo = kPlain ? cmask : 0u; todo; todo &= todo - 1) {
          const int j = __ffs(todo) - 1;
          const unsigned long long sj = __shfl_sync(0xffffffffu, src, j);
          const unsigned long long xj = __shfl_sync(0xffffffffu, d1, j);
          const unsigned long long yj = __shfl_sync(0xffffffffu, d2, j);
          const uint32_t lj = __shfl_sync(0xffffffffu, bytes, j);
          warp_copy2(reinterpret_cast<uint8_t*>(xj), reinterpret_cast<uint8_t*>(yj),
                     reinterpret_cast<const uint8_t*>(sj), lj, P);
        }
      }
    };
    if (a.copy_grab) {
      // the pieces taken copy_grab at a time from a counter of the call, the
      // warp's next grab requested before its current one is copied: warps
      // on SMs that copy faster take more
      const uint32_t grab = a.copy_grab;
      uint32_t nxt = 0;
      if (lane == 0) nxt = atomicAdd(&a.ctl->copy_next, grab);
      nxt = __shfl_sync(0xffffffffu, nxt, 0);
      while (nxt < npieces) {
        uint32_t nn = 0;
        if (lane == 0) nn = atomicAdd(&a.ctl->copy_next, grab);
        copy_range(nxt, min(npieces, (unsigned long long)nxt + grab));
        nxt = __shfl_sync(0xffffffffu, nn, 0);
      }
    } else {
#if GLEAM_CHAIN_PREFETCH
      // the warp's source pieces start their way into L2 at once (up to 32),
      // so that the copies below wait for L2 rather than HBM
      if (plo + lane < phi && !a.far) {
        const unsigned long long pc = plo + lane, rr = pc / ppc;
        const uint32_t off = (uint32_t)(pc - rr * ppc) * kPackPiece;
        const uint32_t gg = __ldcg(&ch.order[rr]);
        const uint32_t ln = (uint32_t)min(a.C, P.n - (unsigned long long)gg * a.C);
        const uint8_t* src = P.buf + (unsigned long long)gg * a.C + off;
        if (off < ln && ((uintptr_t)src & 15) == 0) {  // the prefetch wants 16-byte alignment
          const uint32_t pb = min(kPackPiece, ln - off) & ~15u;
          if (pb) prefetch_l2(src, pb);
        }
      }
#endif
      copy_range(plo, phi);
    }
    // each stored miss completes its inserts and frees the group entry it
    // claimed, while the last pieces' stores are still in flight
    if (ins) {
      if (!index_insert_end(a.index, a.index_mask, index_key(a, key), (uint32_t)ins_slot, len, pi,
                            a.key16))
        atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_INTERNAL);
      if (ins_hint &&
          !index_insert_end(a.hints, a.index_mask, hint, (uint32_t)ins_slot, len, ph))
        atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_INTERNAL);
      if (e != 0xFFFFFFFFu) a.tbl[e] = CallEntry{0u, 0u};  // owner and the claim's tag
    }
    if (!kPlain && lane == 0) bulk_wait_all<0>();  // every piece written before the block ends
  }
  n_hc = block_sum<unsigned long long>(n_hc, red64);
  n_rej = block_sum<unsigned long long>(n_rej, red64);
  n_bytes = block_sum<unsigned long long>(n_bytes, red64);
  n_sbytes = block_sum<unsigned long long>(n_sbytes, red64);
  const unsigned long long b_spec = block_sum<unsigned long long>(n_spec, red64);
  const unsigned long long b_spec_used = block_sum<unsigned long long>(n_spec_used, red64);
  if (threadIdx.x == 0 && P.result) {  // the payload's own counters (cleared in phase 1)
    gleam_result_t* res = P.result;
    if (n_hc) atomicAdd((unsigned long long*)&res->n_hit_cache, n_hc);
    if (c_b) atomicAdd((unsigned long long*)&res->n_miss, (unsigned long long)c_b);
    if (n_rej) atomicAdd((unsigned long long*)&res->verify_rejects, n_rej);
    if (n_bytes) atomicAdd((unsigned long long*)&res->miss_bytes, n_bytes);
  }
  if (threadIdx.x == 0) {
    if (G == 1) {
      s_sum[0] = n_hc;
      s_sum[1] = 0;  // no in-call duplicate on this path
      s_sum[2] = n_rej;
      s_sum[3] = n_bytes;
      s_sum[4] = n_sbytes;
      s_sum[5] = b_spec;
      s_sum[6] = b_spec_used;
    } else {
      if (n_hc) atomicAdd(&a.ctl->acc_hits_cache, n_hc);
      if (n_rej) atomicAdd(&a.ctl->acc_rejects, n_rej);
      if (n_bytes) atomicAdd(&a.ctl->acc_miss_bytes, n_bytes);
      if (n_sbytes) atomicAdd(&a.ctl->acc_stored_bytes, n_sbytes);
      if (b_spec) atomicAdd(&a.ctl->spec_tried, b_spec);
      if (b_spec_used) atomicAdd(&a.ctl->spec_used, b_spec_used);
    }
  }
  finish_call(a, G, slots0, total, stotal, 0ull, 0ull, s_sum);
}

// The one-launch path where the hash kernel has claimed the misses' groups
// (DedupArgs::pre_claimed; every miss is then stored, under its 64-bit key: KEY16
// and paper identifiers claim nothing there).  If no group is shared,
// every chunk that is not a cache hit is a miss, so every block reads the
// statuses of the whole call (at most 16 KiB), turns them into a bit per chunk
// with the misses counted before each word, and knows the rank of every miss,
// the chunk of every rank, the hit mask and all of the call's counts: the
// blocks write, copy and insert their shares and meet only at the end, to
// publish.  What bounds it is the chain of round trips (statuses, claims or
// copies, the arrival count, the publishing).
constexpr uint32_t kDirectWords = 2 * kThreads;  // 32 chunks each

struct DirectShared {
  uint32_t bits[kDirectWords];  // chunk 32 w + k is not a cache hit: bit k of word w
  uint16_t before[kDirectWords];  // such chunks before word w
  unsigned long long scan[kWarps];
  unsigned long long slots0;
  int shared, err, last;
};

// Chunk of the r-th miss: the last of nw words with at most r misses before it,
// then its bit.
__device__ __forceinline__ uint32_t direct_miss(const DirectShared& sh, uint32_t nw, uint32_t r) {
  uint32_t lo = 0, hi = nw;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (sh.before[mid] <= r) lo = mid;
    else hi = mid;
  }
  uint32_t b = sh.bits[lo], k = r - sh.before[lo], pos = 0;
#pragma unroll
  for (uint32_t step = 16; step; step >>= 1) {
    const uint32_t c = __popc(b & ((1u << step) - 1u));
    if (k >= c) {
      k -= c;
      pos += step;
      b >>= step;
    }
  }
  return lo * 32 + pos;
}

template <bool kPlain>
__device__ __forceinline__ void resolve_direct(const DedupArgs& a, uint32_t G, uint32_t bid,
                                               uint8_t* smem) {
  __shared__ DirectShared sh;
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const ChunkArrays& ch = a.ch;
  const PayloadDesc& P = a.one;
  const uint32_t N = (uint32_t)a.Ntot, nw = (N + 31) / 32;
  const uint32_t per = (N + G - 1) / G;  // <= kThreads (the host sizes the grid)
  const uint32_t g = bid * per + threadIdx.x;
  const bool valid = threadIdx.x < per && g < N;
  if (threadIdx.x == 0) {
    sh.slots0 = *(volatile const unsigned long long*)&a.dstats[ST_SLOTS_USED];
    sh.shared = (int)ldcg_u32(&a.ctl->shared_groups);
    sh.err = ld_volatile_s32(&a.ctl->err);
    if (per > kThreads || nw > kDirectWords) atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_INTERNAL);
  }
  // the thread's own chunk and its share of the statuses, in one round trip
  unsigned long long key = 0, hint = 0;
  uint32_t e = 0xFFFFFFFFu;
  if (valid) {
    key = ch.key[g];
    hint = ch.hint[g];
    e = ch.ent[g];
  }
  unsigned long long cnt = 0;  // misses of words < kThreads, of the others << 16, rejects << 32
#pragma unroll
  for (uint32_t k = 0; k < 2; ++k) {
    const uint32_t word = k * kThreads + threadIdx.x, c0 = word * 32;
    uint32_t m = 0, rej = 0;
    if (c0 + 32 <= N) {
      const uint4* q = reinterpret_cast<const uint4*>(ch.status + c0);
      const uint4 v[2] = {__ldcg(q), __ldcg(q + 1)};
#pragma unroll
      for (uint32_t h = 0; h < 2; ++h) {
        const uint32_t x[4] = {v[h].x, v[h].y, v[h].z, v[h].w};
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) {
          m |= bytes_not(x[u], kHit0) << (16 * h + 4 * u);
          rej += 4 - __popc(bytes_not(x[u], kMissCand));
        }
      }
    } else {
      for (uint32_t c = c0; c < N; ++c) {
        const uint8_t st = __ldcg(ch.status + c);
        m |= (uint32_t)(st != kHit0) << (c - c0);
        rej += st == kMissCand;
      }
    }
    sh.bits[word] = m;
    cnt += (unsigned long long)__popc(m) << (16 * k) | (unsigned long long)rej << 32;
  }
  unsigned long long incl = cnt;
#pragma unroll
  for (uint32_t o = 1; o < 32; o <<= 1) {
    const unsigned long long v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) sh.scan[w] = incl;
  __syncthreads();
  unsigned long long excl = incl - cnt, all = 0;
#pragma unroll
  for (uint32_t k = 0; k < kWarps; ++k) {
    const unsigned long long v = sh.scan[k];
    if (k < w) excl += v;
    all += v;
  }
  const uint32_t total0 = (uint32_t)all & 0xFFFFu;
  const uint32_t total = total0 + ((uint32_t)all >> 16);
  sh.before[threadIdx.x] = (uint16_t)excl;
  sh.before[kThreads + threadIdx.x] = (uint16_t)(total0 + (uint32_t)(excl >> 16 & 0xFFFFu));
  __syncthreads();
  const unsigned long long slots0 = sh.slots0;
  bool ok = sh.err == 0;
  const bool miss = valid && (sh.bits[g >> 5] >> (g & 31) & 1u);

  if (sh.shared) {
    // a group may be shared: the general algorithm, from cleared outputs, on the
    // first Gg blocks, each with a larger share of the chunks
    const uint32_t Gg = min(G, a.general_blocks);
    if (bid >= Gg) {
      leave_general_to(a);
      return;
    }
    const uint32_t pg = (N + Gg - 1) / Gg;  // <= kThreads, too
    const uint32_t c = bid * pg + threadIdx.x;
    const bool mine = threadIdx.x < pg && c < N;
    if (pg > kThreads && threadIdx.x == 0) atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_INTERNAL);
    for (uint32_t k = bid * kThreads + threadIdx.x; k < nw; k += Gg * kThreads) P.mask[k] = 0;
    if (bid == 0 && threadIdx.x == 0 && P.result) {
      gleam_result_t* r = P.result;
      r->n_miss = r->n_hit_cache = r->n_hit_intra = r->verify_rejects = r->miss_bytes = 0;
    }
    const bool grouped = mine && (sh.bits[c >> 5] >> (c & 31) & 1u);
    if (mine && !grouped) ch.res[c] = kResHit0;
    resolve_pack_general<kPlain>(a, Gg, bid, smem, ok, true, grouped,
                                 grouped ? ch.ent[c] : 0xFFFFFFFFu, grouped ? ch.key[c] : 0ull,
                                 grouped ? ch.len[c] : 0u, c);
    return;
  }

  if (ok && total > a.nslots - slots0) {  // every block decides the same
    if (threadIdx.x == 0) atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_CAPACITY);
    ok = false;
  }
  const unsigned long long last = (unsigned long long)(N - 1) * a.C;  // the last chunk's place
  uint32_t n_spec = 0, n_spec_used = 0;
  if (ok) {
    // each miss records its slot and starts its index inserts (the first claim
    // attempts), which complete after the copies below
    const uint32_t r = miss ? sh.before[g >> 5] + __popc(sh.bits[g >> 5] & ((1u << (g & 31)) - 1u)) : 0u;
    const unsigned long long slot = slots0 + r;
    const uint32_t len = (uint32_t)min(a.C, P.n - (unsigned long long)min(g, N - 1) * a.C);
    const bool ins_hint = miss && len >= kPrefixBytes;
    PendingInsert pi{0ull, 0u}, ph{0ull, 0u};
    if (miss) {
      pi = index_insert_begin(a.index, a.index_mask, key, (uint32_t)slot);
      if (ins_hint) ph = index_insert_begin(a.hints, a.index_mask, hint, (uint32_t)slot);
      P.miss_idx[r] = g;
      a.slot_len[slot] = len;
      a.slot_key[slot] = key;
    }
    if (P.chunk_slot && valid) P.chunk_slot[g] = miss ? (uint32_t)slot : e;
    for (uint32_t k = bid * kThreads + threadIdx.x; k < nw; k += G * kThreads)
      P.mask[k] = ~sh.bits[k] & (k * 32 + 32 <= N ? 0xffffffffu : (1u << (N & 31)) - 1u);
    if (a.spec_active && valid && ch.spec[g]) {
      n_spec = 1;
      n_spec_used = miss && r == g;
    }
    // every miss's bytes, in pieces of kPackPiece bytes spread over all the
    // grid's warps (piece k of the miss of rank r is number r * ppc + k), all
    // but those of misses the hash kernel already wrote where they belong
    // (rank g means every earlier chunk is a miss)
    const unsigned long long warps = (unsigned long long)G * kWarps;
    const unsigned long long gw = (unsigned long long)bid * kWarps + w;
    const unsigned long long ppc = (a.C + kPackPiece - 1) / kPackPiece;
    const unsigned long long npieces = total * ppc;
    const uint32_t wbase =
        kPlain ? 0u : (uint32_t)__cvta_generic_to_shared(smem) + w * kPackWarpBytes;
    const uint32_t bufs = wbase, bars = wbase + kPackBufs * kPackPiece;
    PackMeta* meta =
        reinterpret_cast<PackMeta*>(smem + w * kPackWarpBytes + kPackBufs * kPackPiece + 64);
    PackRing ring{0u, 0u, 0u};
    bool bulk_failed = false;
    if constexpr (!kPlain) {
      if (lane == 0) {
        for (uint32_t b = 0; b < kPackBufs; ++b) mbar_init(bars + 8 * b);
        mbar_fence_init();
      }
      __syncwarp();
    }
    auto copy_range = [&](unsigned long long lo, unsigned long long hi) {  // 32 pieces at a time
      for (unsigned long long base = lo; base < hi; base += 32) {
        const unsigned long long pc = base + lane;
        uint32_t bytes = 0;
        bool copy = false;
        unsigned long long src = 0, d1 = 0, d2 = 0;
        if (pc < hi) {
          const uint32_t rr = (uint32_t)(pc / ppc);
          const uint32_t off = (uint32_t)(pc - rr * ppc) * kPackPiece;
          const uint32_t gg = direct_miss(sh, nw, rr);
          const unsigned long long at = (unsigned long long)gg * a.C;
          const uint32_t ln = (uint32_t)min(a.C, P.n - at);
          if (off < ln && !(a.spec_active && rr == gg && ch.spec[gg])) {
            bytes = min(kPackPiece, ln - off);
            src = (unsigned long long)(P.buf + at + off);
            d1 = (unsigned long long)(P.packed + rr * a.C + off);
            d2 = (unsigned long long)(a.arena + (slots0 + rr) * a.C + off);
            copy = true;
          }
        }
        const unsigned cmask = __ballot_sync(0xffffffffu, copy);
        if constexpr (!kPlain) {
          const uint32_t at = __popc(cmask & ((1u << lane) - 1u));
          if (copy) {
            meta[at] = PackMeta{src, d1, d2, bytes, 0u};
            // the pieces that wait for a buffer are on their way into L2
            if (at >= kPackBufs && bytes >= 16) prefetch_l2(reinterpret_cast<const void*>(src), bytes & ~15u);
          }
          __syncwarp();
          if (lane == 0 && cmask && !bulk_failed &&
              !bulk_copy_batch(meta, __popc(cmask), bufs, bars, ring, a.wait_ns)) {
            bulk_failed = true;
            atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_TIMEOUT);
          }
          if (copy) {  // the piece's last bytes % 16
            const uint8_t* sp = reinterpret_cast<const uint8_t*>(src);
            for (uint32_t k = bytes & ~15u; k < bytes; ++k)
              reinterpret_cast<uint8_t*>(d1)[k] = reinterpret_cast<uint8_t*>(d2)[k] = sp[k];
          }
          __syncwarp();
        } else {
          for (unsigned todo = cmask; todo; todo &= todo - 1) {
            const int j = __ffs(todo) - 1;
            const unsigned long long sj = __shfl_sync(0xffffffffu, src, j);
            const unsigned long long xj = __shfl_sync(0xffffffffu, d1, j);
            const unsigned long long yj = __shfl_sync(0xffffffffu, d2, j);
            const uint32_t lj = __shfl_sync(0xffffffffu, bytes, j);
            warp_copy2(reinterpret_cast<uint8_t*>(xj), reinterpret_cast<uint8_t*>(yj),
                       reinterpret_cast<const uint8_t*>(sj), lj, P);
          }
        }
      }
    };
    if (a.copy_grab) {
      // the pieces taken copy_grab at a time from a counter of the call, the
      // warp's next grab requested before its current one is copied: warps
      // on SMs that copy faster take more
      const uint32_t grab = a.copy_grab;
      uint32_t nxt = 0;
      if (lane == 0) nxt = atomicAdd(&a.ctl->copy_next, grab);
      nxt = __shfl_sync(0xffffffffu, nxt, 0);
      while (nxt < npieces) {
        uint32_t nn = 0;
        if (lane == 0) nn = atomicAdd(&a.ctl->copy_next, grab);
        copy_range(nxt, min(npieces, (unsigned long long)nxt + grab));
        nxt = __shfl_sync(0xffffffffu, nn, 0);
      }
    } else {
      copy_range(npieces * gw / warps, npieces * (gw + 1) / warps);
    }
    // each miss completes its inserts and frees the group entry it claimed,
    // while the last pieces' stores are still in flight
    if (miss) {
      if (!index_insert_end(a.index, a.index_mask, key, (uint32_t)slot, len, pi) ||
          (ins_hint && !index_insert_end(a.hints, a.index_mask, hint, (uint32_t)slot, len, ph)))
        atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_INTERNAL);
      if (e != 0xFFFFFFFFu) a.tbl[e] = CallEntry{0u, 0u};  // owner and the claim's tag
      else atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_INTERNAL);
    }
    if (!kPlain && lane == 0) bulk_wait_all<0>();  // every piece written before the block ends
  }
  if (a.spec_active) {
    __shared__ unsigned long long red64[kWarps];
    const unsigned long long b_spec = block_sum<unsigned long long>(n_spec, red64);
    const unsigned long long b_used = block_sum<unsigned long long>(n_spec_used, red64);
    if (threadIdx.x == 0) {
      if (b_spec) atomicAdd(&a.ctl->spec_tried, b_spec);
      if (b_used) atomicAdd(&a.ctl->spec_used, b_used);
    }
  }

  // ---- the last block publishes -------------------------------------------------
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    sh.last = G == 1 || atomicAdd(&a.ctl->done, 1u) == G - 1;
  }
  __syncthreads();
  if (!sh.last) return;
  __threadfence();
  const int err = ld_volatile_s32(&a.ctl->err);
  if (err) {
    clear_after_error(a, err, slots0);
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const bool tail = sh.bits[nw - 1] >> ((N - 1) & 31) & 1u;  // the last chunk is a miss
    const unsigned long long bytes =
        (unsigned long long)total * a.C - (tail ? last + a.C - P.n : 0ull);
    const unsigned long long rejects = all >> 32, hits = N - total;
    if (a.spec_active || a.spec_state) {
      const unsigned long long spec = __ldcg(&a.ctl->spec_tried);
      if (err == 0 && a.spec_state) {
        // automatic write-through: as in finish_call
        uint32_t* st = a.spec_state;
        if (spec) {
          st[0] = 2 * __ldcg(&a.ctl->spec_used) >= spec ? 1u : 0u;
          st[1] = 0;
        } else if (st[0] == 0 && ++st[1] >= 256) {
          st[0] = 1;
          st[1] = 0;
        }
        *a.spec_mirror = st[0];
      }
      if (err == 0 && spec) atomicAdd(&a.dstats[ST_SPEC_CHUNKS], spec);
      a.ctl->spec_tried = a.ctl->spec_used = 0;
    }
    if (err == 0) {
      atomicAdd(&a.dstats[ST_CALLS], a.ncalls);
      atomicAdd(&a.dstats[ST_CHUNKS], (unsigned long long)N);
      if (hits) atomicAdd(&a.dstats[ST_HITS_CACHE], hits);
      if (rejects) atomicAdd(&a.dstats[ST_REJECTS], rejects);
      if (total) {
        atomicAdd(&a.dstats[ST_MISSES], (unsigned long long)total);
        atomicAdd(&a.dstats[ST_INSERTS], (unsigned long long)total);
        a.dstats[ST_SLOTS_USED] = slots0 + total;
        atomicAdd(&a.dstats[ST_BYTES_USED], bytes);
      }
    }
    for (uint32_t k = 0; k < 2; ++k) {
      gleam_result_t* t = k == 0 ? a.total : P.result;
      if (!t) continue;
      t->status = err;
      t->n_miss = err ? 0 : total;
      t->n_hit_cache = err ? 0 : hits;
      t->n_hit_intra = 0;
      t->verify_rejects = err ? 0 : rejects;
      t->miss_bytes = err ? 0 : bytes;
    }
    // the control block as the next call expects it (no barrier was used)
    DevCtl* c = a.ctl;
    c->copy_next = 0;
    c->err = 0;
    c->shared_groups = 0;
    c->done = 0;
  }
  __threadfence();
}

// Passes with this kernel against one in which the blocks exchanged the misses'
// places through memory and a grid barrier: a Llama-3-8B layer, one call per
// tensor, a tenth of its 64 KiB chunks changed, 575 -> 535 us (overlapping
// calls 346 -> 314); 48 calls of 4 KiB-1 MiB 1,104 -> 1,067; one 64 MiB payload,
// half of its 4 KiB chunks cached, 86.6 -> 81.4.
template <bool kPlain>
__global__ void __launch_bounds__(kThreads) k_resolve_direct(DedupArgs a) {
  extern __shared__ __align__(128) uint8_t rd_smem[];
  pdl_trigger();
  pdl_wait();
  resolve_direct<kPlain>(a, gridDim.x, blockIdx.x, rd_smem);
}

template <bool kPlain>
__global__ void __launch_bounds__(kThreads) k_resolve_pack(DedupArgs a) {
  extern __shared__ __align__(128) uint8_t rp_smem[];
  pdl_trigger();
  pdl_wait();
  resolve_pack_fast<kPlain>(a, gridDim.x, blockIdx.x, rp_smem);
}

#ifndef GLEAM_DEDUP_MINBLOCKS
#define GLEAM_DEDUP_MINBLOCKS 3
#endif
// three co-resident blocks per SM (at most 85 registers): the resolve kernel's
// phases are chains of round trips that want every thread of the grid
__global__ void __launch_bounds__(kThreads, GLEAM_DEDUP_MINBLOCKS) k_dedup(DedupArgs a) {
  pdl_trigger();
  pdl_wait();
  // k_pack's question, answered anew in every call
  if (blockIdx.x == 0 && threadIdx.x == 0) a.ctl->published = 0u;
  bool ok = true;
  if (resolve_rank(a, gridDim.x, blockIdx.x, false, true, &ok))
    publish_all_hits(a, gridDim.x, blockIdx.x, ok);
}

template <bool kPlain>
__global__ void GLEAM_PACK_BOUNDS k_pack(DedupArgs a) {
  extern __shared__ __align__(128) uint8_t pack_smem[];
  pdl_trigger();
  pdl_wait();
  if (ldcg_u32(&a.ctl->published)) return;  // a call of hits alone (publish_all_hits)
  pack_publish<kPlain>(a, gridDim.x, blockIdx.x, pack_smem);
}

// A whole small call in one block: the staged hash of its chunks (kThreads / 4
// at a time), then the resolution and ranks, then the copies, inserts and
// publish, separated by block barriers instead of kernel boundaries and grid
// barriers.  The pack reuses the shared memory of the hash stages.
constexpr uint32_t kSmallGroups = kThreads / 4;
constexpr uint32_t kSmallHashSmem = kSmallGroups * (uint32_t)kGroupBytes;
constexpr uint32_t kSmallSmem = kSmallHashSmem > kPackSmem ? kSmallHashSmem : kPackSmem;


// k_dedup's and k_pack's steps on a grid of one block (several payloads, LRU,
// a class table, or more chunks than threads): out of line, so that the small
// kernel's common path stays compact.
template <bool kPlain>
__device__ __noinline__ void small_call_general(const DedupArgs& a, uint8_t* smem) {
  resolve_rank(a, 1, 0);
  __syncthreads();
  pack_publish<kPlain>(a, 1, 0, smem);
}

//
// One block per SM at least: without saying so the compiler keeps to 102
// registers and waits for more loads one by one (a 6 KB call of hits, back to
// back: 14.8 us against 13.9).
template <bool kAhead, bool kPrefixAsync, bool kMis, bool kPlain>
__global__ void __launch_bounds__(kThreads, 1) k_small_call(HashArgs h, DedupArgs a) {
  extern __shared__ __align__(128) uint8_t small_smem[];
  pdl_trigger();
  if (!h.wait_late) pdl_wait();  // else in staged_range, before the first probe
  // Device-resident payloads are prefetched into L2 at once, lane p taking the
  // whole 16-byte pieces of payload p, 16 KiB at a time, so that the hash
  // stages wait for L2 rather than HBM.
  constexpr uint32_t kPiece = 16u << 10;
  if (!a.far && a.count <= 32 && threadIdx.x < a.count) {
    const PayloadDesc& P = desc(a, threadIdx.x);
    const uint8_t* b0 = P.buf + (kMis ? (0 - (uintptr_t)P.buf) & 15 : 0);
    const unsigned long long skip = b0 - P.buf;
    const unsigned long long nb = P.n > skip ? (P.n - skip) & ~15ull : 0ull;
    for (unsigned long long off = 0; off < nb; off += kPiece)
      prefetch_l2(b0 + off, (uint32_t)min((unsigned long long)kPiece, nb - off));
  }
  const unsigned long long nvb = (h.Ntot * 4 + kThreads - 1) / kThreads;
  for (unsigned long long vb = 0; vb < nvb; ++vb) {
    __syncthreads();  // the previous range's groups are done with the shared memory
    staged_range<true, kAhead, true, kPrefixAsync, kStage, kMis>(h, vb, small_smem);
  }
  __syncthreads();  // every chunk's probe outcome written (and its stage copies landed)
  if (a.count == 1 && !a.lru && !a.classes && a.Ntot <= (unsigned long long)kThreads) {
    // one payload of at most one chunk per thread: the one-launch path's
    // steps, which for a call without duplicates rank the misses by a block
    // scan (no LRU: they stamp no last use)
    resolve_pack_fast<kPlain>(a, 1, 0, small_smem);
  } else {
    small_call_general<kPlain>(a, small_smem);
  }
}

// One warp per record: does the block still hold the recorded chunk's bytes?
__global__ void __launch_bounds__(kThreads) k_block_check(BlockCheckArgs a) {
  const uint32_t lane = threadIdx.x & 31;
  const unsigned long long warp = ((unsigned long long)blockIdx.x * kThreads + threadIdx.x) >> 5;
  const unsigned long long nwarps = ((unsigned long long)gridDim.x * kThreads) >> 5;
  const unsigned long long used = a.dstats[ST_SLOTS_USED];
  uint32_t bad = 0;
  for (unsigned long long r = warp; r < a.nrec; r += nwarps) {
    const unsigned long long off = a.offsets[r];
    const uint32_t slot = a.slots[r];
    bool differs = true;
    if (slot < used) {
      const uint32_t len = a.slot_len[slot];
      if (off <= a.block_bytes && len <= a.block_bytes - off) {
        const uint8_t* x = a.block + off;
        const uint8_t* y = a.arena + (unsigned long long)slot * a.C;
        differs = !warp_equal(x, y, len);
      }
    }
    if (lane == 0) {
      if (a.mismatch) a.mismatch[r] = differs ? 1 : 0;
      bad += differs;
    }
  }
  if (lane == 0 && bad) atomicAdd(a.count, (unsigned long long)bad);
}

__global__ void k_debug_insert(IndexEntry* index, uint64_t index_mask, uint32_t* slot_len,
                               unsigned long long* slot_key, unsigned long long* dstats,
                               unsigned long long key, uint32_t slot, uint32_t len, DevCtl* ctl,
                               uint32_t* last_use, uint32_t epoch) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  if (!index_insert(index, index_mask, key, slot, len)) {
    ctl->err = GLEAM_ERR_INTERNAL;
    return;
  }
  slot_len[slot] = len;
  slot_key[slot] = key;
  if (last_use) last_use[slot] = epoch;
  dstats[ST_SLOTS_USED] = (unsigned long long)slot + 1;
  dstats[ST_INSERTS] += 1;
  dstats[ST_BYTES_USED] += len;
}

// ---- GLEAM_DEBUG_CHECKS --------------------------------------------------------
__global__ void __launch_bounds__(kThreads) k_check_entries(IndexCheckArgs a) {
  const unsigned long long used = a.dstats[ST_SLOTS_USED];
  const unsigned long long n = a.index_mask + 1;
  bool bad = false;
  for (unsigned long long q = (unsigned long long)blockIdx.x * kThreads + threadIdx.x; q < n;
       q += (unsigned long long)gridDim.x * kThreads) {
    const IndexEntry e = a.index[q];
    if (e.slot != kEmptySlot) {
      if (e.slot >= used || e.len != a.slot_len[e.slot]) bad = true;
      else atomicAdd(&a.count[e.slot], 1u);
    }
    const IndexEntry h = a.hints[q];
    if (h.slot != kEmptySlot && (h.slot >= used || h.len != a.slot_len[h.slot])) bad = true;
  }
  if (bad) atomicExch(a.flag, 1u);
}

__global__ void __launch_bounds__(kThreads) k_check_slots(IndexCheckArgs a) {
  const unsigned long long used = a.dstats[ST_SLOTS_USED];
  bool bad = false;
  for (unsigned long long sl = (unsigned long long)blockIdx.x * kThreads + threadIdx.x; sl < used;
       sl += (unsigned long long)gridDim.x * kThreads) {
    bad |= a.count[sl] != 1u;
    a.count[sl] = 0u;
  }
  if (bad) atomicExch(a.flag, 1u);
}

__global__ void k_check_publish(IndexCheckArgs a) {
  if (*(volatile uint32_t*)a.flag == 0u) return;
  for (uint32_t p = threadIdx.x; p < a.npayloads; p += blockDim.x) {
    gleam_result_t* r = a.npayloads > 1 ? a.table[p].result : a.one.result;
    if (r) r->status = GLEAM_ERR_INTERNAL;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a.total->status = GLEAM_ERR_INTERNAL;
    *a.flag = 0u;
  }
}

}  // namespace

cudaError_t launch_index_check(const IndexCheckArgs& a, cudaStream_t s) {
  const unsigned grid = 1024;
  k_check_entries<<<grid, kThreads, 0, s>>>(a);
  k_check_slots<<<grid, kThreads, 0, s>>>(a);
  k_check_publish<<<1, kThreads, 0, s>>>(a);
  return cudaGetLastError();
}

int dedup_threads() { return kThreads; }

int dedup_chunks_per_block() { return GLEAM_DEDUP_CHUNKS_PER_BLOCK; }

// Dynamic shared memory of a pack or one-launch resolve variant: the bulk
// copies' buffers.
constexpr uint32_t pack_smem_bytes(bool plain) { return plain ? 0u : kPackSmem; }

// Co-resident blocks per SM of a kernel (0: unknown).
template <auto kKern>
int blocks_per_sm(uint32_t smem) {
  static PerDevice blocks;
  return blocks.get([smem](int) {
    int nb = 0;
    if (cudaFuncSetAttribute((const void*)kKern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kKern, kThreads, smem) != cudaSuccess)
      return 0;
    return nb;
  });
}

// Co-resident blocks per SM of the pack kernel.
int pack_blocks_per_sm() { return blocks_per_sm<k_pack<false>>(pack_smem_bytes(false)); }

// Co-resident blocks per SM of the one-launch resolve + pack kernel (its grid
// barriers need every block of the grid resident at once).
int resolve_pack_blocks_per_sm() {
  return std::min({blocks_per_sm<k_resolve_pack<false>>(pack_smem_bytes(false)),
                   blocks_per_sm<k_resolve_pack<true>>(pack_smem_bytes(true)),
                   blocks_per_sm<k_resolve_direct<false>>(pack_smem_bytes(false)),
                   blocks_per_sm<k_resolve_direct<true>>(pack_smem_bytes(true))});
}

// Co-resident blocks per SM for the cooperative launch (capped).
int dedup_blocks_per_sm() {
  const int nb = blocks_per_sm<k_dedup>(0);
  return nb < GLEAM_DEDUP_BLOCKS_PER_SM ? nb : GLEAM_DEDUP_BLOCKS_PER_SM;
}

// Every kernel of this file.
cudaError_t load_dedup_kernels() {
  return load_kernels<
      k_dedup, k_pack<false>, k_pack<true>, k_resolve_direct<false>, k_resolve_direct<true>,
      k_resolve_pack<false>, k_resolve_pack<true>, k_small_call<false, false, false, false>,
      k_small_call<false, true, false, false>, k_small_call<false, false, false, true>,
      k_small_call<false, true, false, true>, k_small_call<false, false, true, true>,
      k_small_call<false, true, true, true>, k_small_call<true, false, false, false>,
      k_small_call<true, true, false, false>, k_small_call<true, false, false, true>,
      k_small_call<true, true, false, true>, k_block_check, k_debug_insert, k_check_entries,
      k_check_slots, k_check_publish>();
}

cudaError_t launch_dedup(const DedupArgs& a, int grid, int pack_grid, cudaStream_t s, bool pdl) {
  cudaError_t e;
  // chained, and so small that several caches' calls are resident together:
  // a regular launch, which may start early; else a cooperative one, which
  // starts once all of its blocks fit beside whatever else is running
  pdl = pdl && grid <= kRegularDedupBlocks;
  if (pdl) {
    e = launch_kernel(k_dedup, dim3(grid), dim3(kThreads), 0, s, true, a);
  } else {
    DedupArgs copy = a;
    void* args[] = {&copy};
    e = cudaLaunchCooperativeKernel((void*)k_dedup, dim3(grid), dim3(kThreads), args, 0, s);
  }
  if (e != cudaSuccess) return e;
  auto pack = a.plain_copy ? k_pack<true> : k_pack<false>;
  const uint32_t smem = pack_smem_bytes(a.plain_copy);
  cudaFuncSetAttribute((const void*)pack, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  return launch_kernel(pack, dim3(pack_grid), dim3(kThreads), smem, s, pdl, a);
}

cudaError_t launch_resolve_pack(const DedupArgs& a, int grid, cudaStream_t s) {
  auto kern = a.pre_claimed
                  ? (a.plain_copy ? k_resolve_direct<true> : k_resolve_direct<false>)
                  : (a.plain_copy ? k_resolve_pack<true> : k_resolve_pack<false>);
  const uint32_t smem = pack_smem_bytes(a.plain_copy);
  cudaFuncSetAttribute((const void*)kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  return launch_kernel(kern, dim3(grid), dim3(kThreads), smem, s, true, a);
}

uint32_t small_call_groups() { return kSmallGroups; }

template <bool kAhead, bool kPrefixAsync, bool kMis, bool kPlain>
cudaError_t launch_small(const HashArgs& h, const DedupArgs& a, cudaStream_t s, bool pdl) {
  auto kern = k_small_call<kAhead, kPrefixAsync, kMis, kPlain>;
  cudaFuncSetAttribute((const void*)kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmallSmem);
  return launch_kernel(kern, dim3(1), dim3(kThreads), kSmallSmem, s, pdl, h, a);
}

template <bool kPrefixAsync>
cudaError_t launch_small(const HashArgs& h, const DedupArgs& a, bool aligned, cudaStream_t s,
                         bool pdl) {
  // unaligned payloads: no write-through (its 16-byte stores want aligned ones)
  if (!aligned) return launch_small<false, kPrefixAsync, true, true>(h, a, s, pdl);
  if (a.plain_copy)
    return h.spec_mode ? launch_small<true, kPrefixAsync, false, true>(h, a, s, pdl)
                       : launch_small<false, kPrefixAsync, false, true>(h, a, s, pdl);
  return h.spec_mode ? launch_small<true, kPrefixAsync, false, false>(h, a, s, pdl)
                     : launch_small<false, kPrefixAsync, false, false>(h, a, s, pdl);
}

cudaError_t launch_small_call(const HashArgs& h, const DedupArgs& a, bool aligned,
                              cudaStream_t s, bool pdl) {
  return h.C <= kPrefixAsyncMaxChunk ? launch_small<true>(h, a, aligned, s, pdl)
                                     : launch_small<false>(h, a, aligned, s, pdl);
}

cudaError_t launch_block_check(const BlockCheckArgs& a, cudaStream_t s) {
  if (a.nrec == 0) return cudaSuccess;
  const unsigned long long warps = a.nrec < (1ull << 20) ? a.nrec : (1ull << 20);
  const unsigned grid = (unsigned)((warps * 32 + kThreads - 1) / kThreads);
  k_block_check<<<grid, kThreads, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_debug_insert(IndexEntry* index, uint64_t index_mask, uint32_t* slot_len,
                                unsigned long long* slot_key, unsigned long long* dstats,
                                unsigned long long key, uint32_t slot, uint32_t len, DevCtl* ctl,
                                uint32_t* last_use, uint32_t epoch, cudaStream_t s) {
  k_debug_insert<<<1, 32, 0, s>>>(index, index_mask, slot_len, slot_key, dstats, key, slot, len,
                                  ctl, last_use, epoch);
  return cudaGetLastError();
}

}  // namespace gleam
