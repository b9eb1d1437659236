// Fingerprint + speculative verify of calls that leave most of the GPU idle,
// with the work on a chunk split over a whole warp and a quarter of another.
//
// Such a call waits for one chunk's XXH64 chain: 2,048 dependent rounds for 64
// KiB.  In the staged routine the four lanes that run the chain also fetch,
// compare and multiply their words, about 81 cycles a round with one warp per
// scheduler.  Here each chunk has a warp of its own that does all of that: it
// streams the chunk (and the cached copy) through shared memory, compares the
// two, and leaves every word already multiplied by XXH64's second prime in a
// ring of stages; one warp of the block, four lanes per chunk, only loads those
// products and runs the chain (25-27 cycles a round on its own).
#pragma once

#include <type_traits>

#include "staged_hash.cuh"

namespace gleam {
namespace {

constexpr uint32_t kLoneChunks = 8;     // chunks of a block: the chain warp has four lanes for each
constexpr uint32_t kLoneStage = 1024;   // bytes per stage
constexpr uint32_t kLoneProds = 4;      // stages in the ring of products
// Shared memory of a chunk with kD payload (and cached) stages in flight: the
// ring of products first (32 bytes off a multiple of 128 from chunk to chunk,
// so that four chunks' words meet no bank twice), then the payload's stages (16
// bytes more each, for any alignment) and the cached copy's.
constexpr uint32_t kLonePayStage = kLoneStage + 16;
constexpr uint32_t kLonePay = kLoneProds * kLoneStage;
__host__ __device__ constexpr uint32_t lone_copy(uint32_t depth) {
  return kLonePay + depth * kLonePayStage;
}
__host__ __device__ constexpr uint32_t lone_bytes(uint32_t depth) {
  return ((lone_copy(depth) + depth * kLoneStage + 127) & ~127u) + 32;
}

// One round given the next round's product: rotl(s, 31) * P1 + wp, where s is
// the accumulator plus this round's product.  The high product terms take wp's
// high half first, so that the widening multiply-add comes last (25.1 cycles a
// round in a dependent chain; added up after it 27.9).
__device__ __forceinline__ unsigned long long xround(unsigned long long s, unsigned long long wp) {
  const uint32_t lo = (uint32_t)s, hi = (uint32_t)(s >> 32);
  const uint32_t rl = __funnelshift_l(hi, lo, 31), rh = __funnelshift_l(lo, hi, 31);
  const uint32_t c =
      rh * (uint32_t)kXP1 + (rl * (uint32_t)(kXP1 >> 32) + (uint32_t)(wp >> 32));
  return (unsigned long long)rl * (unsigned long long)(uint32_t)kXP1 +
         ((unsigned long long)c << 32 | (uint32_t)wp);
}

// One of the four chains over the first `full` bytes of the chunk at p, straight
// from memory.  Out of line: only for a fingerprint whose warps gave up waiting.
__device__ __noinline__ unsigned long long chain_from_memory(const uint8_t* p, uint32_t full,
                                                             uint32_t lane) {
  unsigned long long acc = xlane_start(lane);
#pragma unroll 1
  for (uint32_t off = 0; off < full; off += 32)
    acc = xstep(acc, load_word<false>(p + off + 8 * lane));
  return acc;
}

// What the warps of a block tell each other about one chunk.
struct LoneShared {
  unsigned long long full[kLoneProds];   // mbarriers: stage of products complete
  unsigned long long empty[kLoneProds];  // mbarriers: stage of products used
  unsigned long long hinted;             // mbarrier: hint written
  unsigned long long done;               // mbarrier: the fields below written
  unsigned long long hint, hint_key;
  uint32_t hint_slot, differs, ahead, failed;  // failed: a wait of the chunk's warp ran out
};

template <bool kProbe, uint32_t kD>
__global__ void __launch_bounds__(32 * (1 + kLoneChunks), 2) k_hash_lone(HashArgs a, uint32_t per) {
  extern __shared__ __align__(128) uint8_t lone_smem[];
  __shared__ LoneShared sh[kLoneChunks];
  __shared__ unsigned long long s_find[33];
  pdl_trigger();
  if (!a.wait_late) pdl_wait();  // else before the probe, in record_chunk
  const uint32_t w = threadIdx.x >> 5, l = threadIdx.x & 31;
  const unsigned long long g0 = (unsigned long long)blockIdx.x * per;
  const uint32_t cnt = (uint32_t)min((unsigned long long)per, a.Ntot - g0);
  // the chain warp's lanes 4c .. 4c+3, and warp c + 1, hold chunk c
  const uint32_t c = w == 0 ? l >> 2 : w - 1;
  const unsigned long long g = g0 + min(c, cnt - 1);
  uint32_t pid = 0;
  if (a.count > 1) pid = block_find_payload(a.table, a.count, g0, g, s_find);
  if (w > 0 && l == 0) {
    LoneShared& m = sh[w - 1];
    for (uint32_t k = 0; k < kLoneProds; ++k) {
      mbar_init((uint32_t)__cvta_generic_to_shared(&m.full[k]));
      mbar_init((uint32_t)__cvta_generic_to_shared(&m.empty[k]));
    }
    mbar_init((uint32_t)__cvta_generic_to_shared(&m.hinted));
    mbar_init((uint32_t)__cvta_generic_to_shared(&m.done));
    mbar_fence_init();
  }
  __syncthreads();
  if (c >= cnt) return;

  const PayloadDesc& P = a.count > 1 ? a.table[pid] : a.one;
  const uint8_t* buf = P.buf;
  const unsigned long long n = P.n;
  const unsigned long long start = (g - P.chunk_base) * a.C;
  const uint32_t len = (uint32_t)min(a.C, n - start);
  const uint8_t* p = buf + start;
  const uint32_t full = len & ~31u;
  const uint32_t nst = (uint32_t)(((unsigned long long)full + kLoneStage - 1) / kLoneStage);
  const bool speculate = kProbe && len >= kPrefixBytes;
  const unsigned long long slots_used =
      !kProbe ? 0ULL
              : a.wait_late ? ld_acquire_u64(&a.dstats[ST_SLOTS_USED]) : a.dstats[ST_SLOTS_USED];
  LoneShared& m = sh[c];
  const uint32_t full_b = (uint32_t)__cvta_generic_to_shared(m.full);
  const uint32_t empty_b = (uint32_t)__cvta_generic_to_shared(m.empty);
  const uint32_t hinted_b = (uint32_t)__cvta_generic_to_shared(&m.hinted);
  const uint32_t done_b = (uint32_t)__cvta_generic_to_shared(&m.done);
  uint8_t* region = lone_smem + c * lone_bytes(kD);
  auto sbytes = [&](uint32_t t) { return min(kLoneStage, full - t * kLoneStage); };
  bool ok = true;  // no wait has run out

  if (w == 0) {
    // ---- the chain ------------------------------------------------------------
    const uint32_t lane = l & 3;
    const int gbase = l & 28;
    const unsigned gmask = 0xFu << gbase;
    const unsigned wmask = cnt >= 8 ? 0xffffffffu : (1u << (4 * cnt)) - 1;
    const uint32_t top = __reduce_max_sync(wmask, nst);
    const uint32_t whole = full / kLoneStage;  // whole stages; at most one more follows
    constexpr uint32_t kRounds = kLoneStage / 32;
    auto words = [&](uint32_t t) {  // the lane's products of stage t, one every 4
      return reinterpret_cast<const unsigned long long*>(region + t % kLoneProds * kLoneStage) +
             lane;
    };
    auto arrived = [&](uint32_t t) {  // stage t, where the chunk has one; the warp's verdict
      return __all_sync(wmask, t >= nst || mbar_wait(full_b + 8 * (t % kLoneProds),
                                                     (t / kLoneProds) & 1, a.wait_ns));
    };
    unsigned long long acc = xlane_start(lane), hint = 0;
    auto give_hint = [&](unsigned long long pre) {
      const unsigned long long b0 = group_shfl(pre, gmask, gbase + 0);
      const unsigned long long b1 = group_shfl(pre, gmask, gbase + 1);
      const unsigned long long b2 = group_shfl(pre, gmask, gbase + 2);
      const unsigned long long b3 = group_shfl(pre, gmask, gbase + 3);
      hint = b0 ^ xrotl(b1, 16) ^ xrotl(b2, 32) ^ xrotl(b3, 48);
      if (lane == 0) {
        m.hint = hint;
        mbar_arrive(hinted_b);
      }
    };
    // x: the next eight products, loaded eight rounds ahead, also from stage to
    // stage, so that the chain never waits for them; s: the accumulator plus
    // the first of them
    unsigned long long x[8], y[8], s = 0;
    ok = arrived(0);
    if (ok && whole > 0) {
#pragma unroll
      for (uint32_t u = 0; u < 8; ++u) x[u] = words(0)[4 * u];
      s = acc + x[0];
    }
    for (uint32_t t = 0; t < top && ok; ++t) {
      if (t < whole) {
        const unsigned long long* wp = words(t);
#pragma unroll
        for (uint32_t h = 8; h < kRounds; h += 8) {
#pragma unroll
          for (uint32_t u = 0; u < 8; ++u) y[u] = wp[4 * (h + u)];
#pragma unroll
          for (uint32_t u = 1; u < 8; ++u) s = xround(s, x[u]);
          if (h == kPrefixBytes / 32 && t == 0 && speculate) give_hint(xrotl(s, 31) * kXP1);
          s = xround(s, y[0]);
#pragma unroll
          for (uint32_t u = 0; u < 8; ++u) x[u] = y[u];
        }
        __syncwarp(gmask);  // every lane holds the last of the stage
        if (lane == 0) mbar_arrive(empty_b + 8 * (t % kLoneProds));
      }
      ok = arrived(t + 1);
      if (t < whole) {
        const unsigned long long* wn = words(t + 1);
#pragma unroll
        for (uint32_t u = 0; u < 8; ++u) y[u] = ok && t + 1 < whole ? wn[4 * u] : 0;
#pragma unroll
        for (uint32_t u = 1; u < 8; ++u) s = xround(s, x[u]);
        s = xround(s, y[0]);
        acc = s;  // the accumulator itself after the last whole stage
#pragma unroll
        for (uint32_t u = 0; u < 8; ++u) x[u] = y[u];
      } else if (t < nst) {  // a shorter last stage
        const uint32_t rounds = sbytes(t) >> 5;
        unsigned long long pre = 0;
        for (uint32_t r = 0; r < rounds; ++r) {
          acc = xrotl(acc + words(t)[4 * r], 31) * kXP1;
          if (r + 1 == kPrefixBytes / 32) pre = acc;
        }
        if (t == 0 && speculate) give_hint(pre);
      }
    }
    ok = __all_sync(wmask, mbar_wait(done_b, 0, a.wait_ns) && !m.failed) && ok;
    if (!ok) {
      if constexpr (kProbe) {  // the call reports it; nothing of this chunk is used
        atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_TIMEOUT);
        acc = 0;
      } else {  // fingerprints have no status: the chunk once more, without any wait
        acc = chain_from_memory(p, full, lane);
      }
    }
    ChunkEnd e;
    e.g = g, e.p = p, e.len = len, e.lane = lane, e.gbase = gbase, e.pid = pid;
    e.acc = acc, e.hint = hint, e.slots_used = slots_used;
    e.hint_slot = ok ? m.hint_slot : kEmptySlot, e.hint_key = m.hint_key;
    e.diff = m.differs, e.cmp = e.hint_slot != kEmptySlot && m.differs == 0;
    e.ahead = m.ahead != 0;
    record_chunk<kProbe, true, true>(a, e, wmask);
    return;
  }

  // ---- a chunk's own warp: stream, compare, multiply ------------------------------
  uint8_t* const pay = region + kLonePay;
  uint8_t* const cpy = region + lone_copy(kD);
  const uint32_t pay_s = (uint32_t)__cvta_generic_to_shared(pay) + l * 16;
  const uint32_t cpy_s = (uint32_t)__cvta_generic_to_shared(cpy) + l * 16;
  const uint32_t mis = (uint32_t)((uintptr_t)p & 15);
  const uint8_t* const pa = p - mis;
  const uint8_t* q = nullptr;
  bool cmp = false, ahead = false;
  uint8_t *ahead_pk = nullptr, *ahead_ar = nullptr;
  uint32_t hint_slot = kEmptySlot;
  unsigned long long hint_key = 0;
  bool diff = false;
  // Stage t's 16-byte pieces, none of them past the payload's ends.
  auto load_pay = [&](uint32_t t) {
    const uint32_t b = t % kD;
    const uint8_t* src = pa + (unsigned long long)t * kLoneStage;
    const uint32_t dst = pay_s + b * kLonePayStage;
    if (src >= buf && src + kLonePayStage <= buf + n) {  // all inside (and no shorter stage)
#pragma unroll
      for (uint32_t off = 0; off < kLoneStage; off += 512) cp_async16(dst + off, src + off + l * 16);
      if (mis && l == 0) cp_async16(dst + kLoneStage, src + kLoneStage);
      return;
    }
    const uint32_t win = mis + sbytes(t);
    const uint32_t lim = (uint32_t)min((unsigned long long)(buf + n - src),
                                       (unsigned long long)kLonePayStage);
    const uint32_t o0 = src < buf ? 16u : 0u;
    if (o0 && l >= (uint32_t)(buf - src) && l < min(16u, win)) pay[b * kLonePayStage + l] = src[l];
    for (uint32_t off = l * 16; off < win; off += 512) {
      if (off < o0) continue;
      const uint32_t d = dst + off - l * 16;
      if (off + 16 <= lim) cp_async16(d, src + off);
      else cp_async16_upto(d, src + off, lim - off);
    }
  };
  auto load_copy = [&](uint32_t t) {
    const uint32_t sb = sbytes(t), dst = cpy_s + (t % kD) * kLoneStage;
    const uint8_t* src = q + (unsigned long long)t * kLoneStage + l * 16;
#pragma unroll
    for (uint32_t off = 0; off < kLoneStage; off += 512)
      if (off + l * 16 < sb) cp_async16(dst + off, src + off);
  };
  // The 16 payload bytes at off of stage t.
  auto piece = [&](uint32_t t, uint32_t off) {
    const uint8_t* b = pay + (t % kD) * kLonePayStage;
    if (mis == 0) return *reinterpret_cast<const ulonglong2*>(b + off);
    const unsigned long long* q8 =
        reinterpret_cast<const unsigned long long*>(b + (mis & 8) + off);
    ulonglong2 v = make_ulonglong2(q8[0], q8[1]);
    if (mis & 7) {
      const uint32_t s = (mis & 7) * 8;
      v = make_ulonglong2(v.x >> s | v.y << (64 - s), v.y >> s | q8[2] << (64 - s));
    }
    return v;
  };
  // Stage t: its products into their ring (kMul), and its bytes compared with
  // the cached copy's, or written ahead (kSettle).  whole: a whole stage.
  auto use = [&](uint32_t t, auto mul, auto settle, auto whole) {
    constexpr bool kMul = decltype(mul)::value, kSettle = decltype(settle)::value;
    const uint32_t b = t % kLoneProds, sb = decltype(whole)::value ? kLoneStage : sbytes(t);
    if (kMul && t >= kLoneProds) {
      ok = __all_sync(0xffffffffu,
                      mbar_wait(empty_b + 8 * b, (t / kLoneProds + 1) & 1, a.wait_ns));
      if (!ok) return;  // the chain warp may yet read the stage: it stays, and nothing is handed over
    }
    bool d = false;
#pragma unroll
    for (uint32_t k = 0; k < kLoneStage; k += 512) {
      const uint32_t off = k + l * 16;
      if (off < sb) {
        const ulonglong2 v = piece(t, off);
        if (kMul)
          *reinterpret_cast<ulonglong2*>(region + b * kLoneStage + off) =
              make_ulonglong2(v.x * kXP2, v.y * kXP2);
        if (kSettle && cmp) {
          const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(cpy + (t % kD) * kLoneStage + off);
          d |= ((v.x ^ u.x) | (v.y ^ u.y)) != 0;
        }
        if (kSettle && ahead) {
          const unsigned long long o = (unsigned long long)t * kLoneStage + off;
          __stcs(reinterpret_cast<ulonglong2*>(ahead_pk + o), v);
          __stcs(reinterpret_cast<ulonglong2*>(ahead_ar + o), v);
        }
      }
    }
    d = __any_sync(0xffffffffu, d);
    __syncwarp();  // every lane is done with the stage's buffers, its products written
    if (kMul && l == 0) mbar_arrive(full_b + 8 * b);
    if (d) {  // the cached copy is not streamed any further
      diff = true;
      cmp = false;
    }
  };
  using Yes = std::integral_constant<bool, true>;
  using No = std::integral_constant<bool, false>;

  // the first stages: multiplied as they arrive, and kept until the chain warp
  // has the prefix hint
  static_assert(kD >= kLoneProds, "the first products' stages are kept");
#pragma unroll
  for (uint32_t t = 0; t < kD; ++t) {
    if (t < nst) load_pay(t);
    cp_commit();
  }
#pragma unroll
  for (uint32_t t = 0; t < kLoneProds; ++t) {
    cp_wait_upto<kD>(kD - 1 - t);
    __syncwarp();
    if (t < nst) use(t, Yes{}, No{}, No{});
  }
  if (speculate) {
    ok = __all_sync(0xffffffffu, mbar_wait(hinted_b, 0, a.wait_ns));
    if (ok) {
      // one lane looks it up: while calls overlap, the table is being added to
      if (l == 0 && !a.no_hints && slots_used)
        hint_slot = hint_lookup(a.hints, a.index_mask, m.hint, len, slots_used);
      hint_slot = __shfl_sync(0xffffffffu, hint_slot, 0);
      cmp = hint_slot != kEmptySlot;
      // no cached chunk begins like it: a likely miss
      ahead = a.spec_mode != 0 && !cmp && slots_used + g < a.nslots;  // no overlap then
    }
    if (cmp) {
      q = a.arena + (unsigned long long)hint_slot * a.C;
      for (uint32_t t = 0; t < min(kD, nst); ++t) load_copy(t);
      hint_key = a.slot_key[hint_slot];
    }
    if (ahead) {
      ahead_pk = P.packed + start;
      ahead_ar = a.arena_w + (slots_used + g) * a.C;
    }
  }
  cp_commit();
  cp_wait<0>();
  __syncwarp();
  if (speculate)
    for (uint32_t t = 0; t < min(kLoneProds, nst); ++t) use(t, No{}, Yes{}, No{});
  // the others; stage t's buffers take stage t + kD as soon as it is used
  uint32_t next = kD;  // first stage not yet asked for
  uint32_t t = kLoneProds;
  {
    // whole stages inside the payload: their loads need no checks
    const uint32_t in_payload = (uint32_t)min(
        (unsigned long long)nst,
        buf + n > pa + 16 ? (unsigned long long)(buf + n - pa - 16) / kLoneStage : 0ull);
    for (; next < min(t + kD - 1, nst); ++next) {
      load_pay(next);
      if (cmp) load_copy(next);
      cp_commit();
    }
    const uint8_t* psrc = pa + (unsigned long long)next * kLoneStage + l * 16;
    const uint8_t* qsrc = q + (unsigned long long)next * kLoneStage + l * 16;
    for (; next == t + kD - 1 && next < min(in_payload, full / kLoneStage) && ok; ++t, ++next) {
      const uint32_t bd = next % kD;
      cp_async16(pay_s + bd * kLonePayStage, psrc);
      cp_async16(pay_s + bd * kLonePayStage + 512, psrc + 512);
      if (mis && l == 0) cp_async16(pay_s + bd * kLonePayStage + kLoneStage, psrc + kLoneStage);
      if (cmp) {
        cp_async16(cpy_s + bd * kLoneStage, qsrc);
        cp_async16(cpy_s + bd * kLoneStage + 512, qsrc + 512);
      }
      cp_commit();
      psrc += kLoneStage;
      qsrc += kLoneStage;
      cp_wait<kD - 1>();
      __syncwarp();
      use(t, Yes{}, Yes{}, Yes{});
    }
  }
  for (; t < nst && ok; ++t) {
    for (; next < min(nst, t + kD); ++next) {
      load_pay(next);
      if (cmp) load_copy(next);
      cp_commit();
    }
    if (t >= kD) {
      cp_wait_upto<kD>(next - 1 - t);
      __syncwarp();
    }
    use(t, Yes{}, Yes{}, No{});
  }
  cp_wait<0>();
  if (ahead && l == 0)  // the bytes past the last whole stripe
    for (uint32_t k = full; k < len; ++k) ahead_pk[k] = ahead_ar[k] = p[k];
  if (l == 0) {
    m.hint_slot = hint_slot;
    m.hint_key = hint_key;
    m.differs = diff;
    m.ahead = ahead;
    m.failed = !ok;
    mbar_arrive(done_b);
  }
}

}  // namespace
}  // namespace gleam
