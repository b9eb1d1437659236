// Fingerprint + index probe + byte verify of every chunk of a payload
// (paper Sec. 4.1.2: hash the source bytes, look the hash up in the set of
// resident chunks; App. B.1: confirm the match so collisions cannot alias).
//
// Mapping: a group of 4 consecutive threads owns one chunk; thread `lane`
// runs XXH64 accumulator lane `lane` on the 8-byte word at 8*lane of each
// 32-byte stripe, so a warp works on 8 chunks and every 32-byte sector it
// touches is used whole.  After the first 512 bytes the group looks its
// prefix hint up and, if a cached chunk began the same way, streams that copy
// alongside the payload and compares as it hashes (speculative verify).  The
// group then probes the index with the full fingerprint; the hinted slot is a
// hit if it is a key+length candidate and compared equal, and any other
// candidate is compared by re-reading both copies.
//
// Kernels: k_hash_probe_staged (chunks stream through shared memory by
// cp.async; a variant for payloads of any alignment), k_hash_lone (few chunks: a
// warp for each, see lone_hash.cuh), and for the paper's
// identifiers k_probe_paper_staged / k_probe_paper (MD5 of the first 128 bytes
// as the key; 16-byte-aligned payloads / any alignment, by direct loads).
#include <algorithm>
#include <cmath>

#include "gleam_internal.cuh"
#include "xxh64_device.cuh"
#include "staged_hash.cuh"
#include "lone_hash.cuh"

namespace gleam {
namespace {

#ifndef GLEAM_HASH_THREADS
#define GLEAM_HASH_THREADS 256
#endif
constexpr int kHashThreads = GLEAM_HASH_THREADS;


template <bool kProbe, bool kAhead, bool kVerify, bool kPrefixAsync = false, int kS = kStage,
          bool kMis = false>
__global__ void __launch_bounds__(kStagedThreads) k_hash_probe_staged(HashArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  pdl_trigger();
  if (!a.wait_late) pdl_wait();  // else in staged_range, before the probe
  const unsigned long long nvb = (a.Ntot * 4 + kStagedThreads - 1) / kStagedThreads;
  for (unsigned long long vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
    __syncthreads();  // the previous range's groups are done with the shared memory
    staged_range<kProbe, kAhead, kVerify, kPrefixAsync, kS, kMis>(a, vb, smem);
  }
}

// Blocks of the kS-stage variant resident at once on the whole GPU (0 if
// unknown).
template <bool kProbe, bool kAhead, bool kVerify, int kS>
int staged_wave_blocks() {
  static PerDevice wave;
  return wave.get([](int dev) {
    constexpr int smem = (kStagedThreads / 4) * group_bytes(kVerify, kS);
    int nsm = 0, occ = 0;
    if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute((const void*)k_hash_probe_staged<kProbe, kAhead, kVerify, false, kS>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &occ, k_hash_probe_staged<kProbe, kAhead, kVerify, false, kS>, kStagedThreads, smem) !=
            cudaSuccess)
      return 0;
    return nsm * occ;
  });
}

template <bool kProbe, bool kAhead, bool kVerify, bool kPrefixAsync = false, int kS = kStage,
          bool kMis = false>
cudaError_t launch_staged(const HashArgs& a, cudaStream_t s, bool pdl) {
  const unsigned long long threads = a.Ntot * 4;
  const unsigned sg = (unsigned)((threads + kStagedThreads - 1) / kStagedThreads);
  if constexpr (kS == kStage && kProbe && !kPrefixAsync && !kMis) {
    // a call whose large chunks all fit one wave of the large-stage variant,
    // unless calls overlap (then the calls in flight share the SMs, and the
    // variant's larger blocks would crowd them out)
    if (a.C >= kBigStageMinChunk && !a.wait_late &&
        (unsigned long long)sg <= (unsigned long long)staged_wave_blocks<kProbe, kAhead, kVerify, kBigStage>())
      return launch_staged<kProbe, kAhead, kVerify, false, kBigStage>(a, s, pdl);
  }
  if constexpr (kVerify && !kPrefixAsync && kS == kStage) {
    if (a.C <= kPrefixAsyncMaxChunk)
      return launch_staged<kProbe, kAhead, kVerify, true, kS, kMis>(a, s, pdl);
  }
  constexpr int smem = (kStagedThreads / 4) * group_bytes(kVerify, kS, kMis);
  // per device and cheap: set on every launch
  cudaFuncSetAttribute(
      (const void*)k_hash_probe_staged<kProbe, kAhead, kVerify, kPrefixAsync, kS, kMis>,
      cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  return launch_kernel(k_hash_probe_staged<kProbe, kAhead, kVerify, kPrefixAsync, kS, kMis>, dim3(sg),
                       dim3(kStagedThreads), smem, s, pdl, a);
}

// ---------------------------------------------------------------------------
// Paper-identifier mode (App. B.1): the key is MD5 (RFC 1321) of the chunk's
// first min(len, 128) bytes, computed by one lane; candidates are then
// compared with the payload directly, so no pass over the whole chunk is
// needed for the key and a chunk without candidates costs only its prefix.
// ---------------------------------------------------------------------------
struct Md5Table {
  uint32_t k[64];  // floor(2^32 * |sin(i + 1)|)
};

__device__ __forceinline__ uint32_t rotl32(uint32_t x, int r) { return (x << r) | (x >> (32 - r)); }

// First 8 digest bytes (little-endian) of MD5 over p[0, m), m <= 128.
__device__ unsigned long long md5_prefix_key(const uint8_t* p, uint32_t m, const uint32_t* K) {
  const uint32_t total = ((m + 8) / 64 + 1) * 64;  // message + 0x80 + padding + length
  const unsigned long long bits = (unsigned long long)m * 8;
  uint32_t a0 = 0x67452301u, b0 = 0xefcdab89u, c0 = 0x98badcfeu, d0 = 0x10325476u;
  for (uint32_t blk = 0; blk < total; blk += 64) {
    uint32_t x[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      uint32_t w = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t q = blk + 4 * j + k;
        uint32_t byte;
        if (q < m) byte = p[q];
        else if (q == m) byte = 0x80u;
        else if (q >= total - 8) byte = (uint32_t)(bits >> (8 * (q - (total - 8)))) & 0xFFu;
        else byte = 0u;
        w |= byte << (8 * k);
      }
      x[j] = w;
    }
    uint32_t a = a0, b = b0, c = c0, d = d0;
#pragma unroll
    for (int i = 0; i < 64; ++i) {
      uint32_t f;
      int g, r;
      if (i < 16) {
        f = (b & c) | (~b & d);
        g = i;
        r = (i & 3) == 0 ? 7 : (i & 3) == 1 ? 12 : (i & 3) == 2 ? 17 : 22;
      } else if (i < 32) {
        f = (d & b) | (~d & c);
        g = (5 * i + 1) & 15;
        r = (i & 3) == 0 ? 5 : (i & 3) == 1 ? 9 : (i & 3) == 2 ? 14 : 20;
      } else if (i < 48) {
        f = b ^ c ^ d;
        g = (3 * i + 5) & 15;
        r = (i & 3) == 0 ? 4 : (i & 3) == 1 ? 11 : (i & 3) == 2 ? 16 : 23;
      } else {
        f = c ^ (b | ~d);
        g = (7 * i) & 15;
        r = (i & 3) == 0 ? 6 : (i & 3) == 1 ? 10 : (i & 3) == 2 ? 15 : 21;
      }
      const uint32_t t = d;
      d = c;
      c = b;
      b = b + rotl32(a + f + K[i] + x[g], r);
      a = t;
    }
    a0 += a;
    b0 += b;
    c0 += c;
    d0 += d;
  }
  return (unsigned long long)a0 | ((unsigned long long)b0 << 32);
}

__global__ void __launch_bounds__(kHashThreads) k_probe_paper(HashArgs a, Md5Table tab) {
  pdl_trigger();
  pdl_wait();
  const unsigned long long g = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 2;
  __shared__ unsigned long long s_scratch[33];
  const uint32_t pid_b =
      a.count > 1 ? block_find_payload(a.table, a.count,
                                       ((unsigned long long)blockIdx.x * blockDim.x) >> 2, g,
                                       s_scratch)
                  : 0u;
  if (g >= a.Ntot) return;  // whole groups leave together
  const uint32_t lane = threadIdx.x & 3;
  const int gbase = threadIdx.x & 28;
  const unsigned gmask = 0xFu << gbase;

  uint32_t pid = 0;
  const uint8_t* buf;
  unsigned long long n, base;
  if (a.count > 1) {
    pid = pid_b;
    buf = a.table[pid].buf;
    n = a.table[pid].n;
    base = a.table[pid].chunk_base;
  } else {
    buf = a.one.buf;
    n = a.one.n;
    base = a.one.chunk_base;
  }
  const unsigned long long start = (g - base) * a.C;
  const uint32_t len = (uint32_t)min(a.C, n - start);
  const uint8_t* p = buf + start;

  unsigned long long key = 0;
  if (lane == 0) key = md5_prefix_key(p, min(len, 128u), tab.k);
  key = group_shfl(key, gmask, gbase);
  if (a.key16) key &= 0xFFFFULL;

  bool hit = false, cand = false;
  uint32_t hit_slot = kEmptySlot;
  if (len >= kPaperMinCached) {
    const unsigned long long slots_used = a.dstats[ST_SLOTS_USED];
    unsigned long long pos = mix64(key) & a.index_mask;
    for (unsigned long long probe = 0; probe <= a.index_mask; ++probe) {
      const IndexEntry e = a.index[pos];
      if (e.slot == kEmptySlot) break;
      if (e.key == key && e.len == len) {
        cand = true;
        if (e.slot >= slots_used) {
          if (lane == 0) atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_INTERNAL);
        } else if (group_equal<false>(p, a.arena + (uint64_t)e.slot * a.C, len, lane, gmask)) {
          hit = true;
          hit_slot = e.slot;
          break;
        }
      }
      pos = (pos + 1) & a.index_mask;
    }
  }
  if (lane == 0) {
    a.ch.status[g] = len < kPaperMinCached ? kUncached : hit ? kHit0 : cand ? kMissCand : kMissNoCand;
    a.ch.key[g] = key;
    a.ch.len[g] = len;
    a.ch.src[g] = (unsigned long long)p;
    a.ch.pidx[g] = pid;
    a.ch.hint[g] = 0;
    if (hit) a.ch.ent[g] = hit_slot;
  }
}

// Staged variant of the paper-identifier probe for 16-byte-aligned payloads.
// Stage 0 of the chunk arrives by cp.async; one lane computes the MD5 key
// from shared memory, the group probes the index, and only if a key+length
// candidate exists do the rest of the chunk and the candidate's copy stream
// through two stages in flight and get compared (each lane compares the
// 16-byte pieces it copied itself, so no cross-lane sync is needed); the
// first difference ends the streaming.  A chunk without a candidate costs one
// stage; further candidates after a mismatch are compared by re-reading.
__global__ void __launch_bounds__(kStagedThreads) k_probe_paper_staged(HashArgs a, Md5Table tab) {
  extern __shared__ __align__(16) uint8_t smem[];
  pdl_trigger();
  pdl_wait();  // the key is known after the first stage: nothing to overlap
  const unsigned long long g = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 2;
  const uint32_t pid_b =
      a.count > 1 ? block_find_payload(a.table, a.count,
                                       ((unsigned long long)blockIdx.x * blockDim.x) >> 2, g,
                                       reinterpret_cast<unsigned long long*>(smem))
                  : 0u;
  if (g >= a.Ntot) return;  // whole groups leave together
  const uint32_t lane = threadIdx.x & 3;
  const int gbase = threadIdx.x & 28;
  const unsigned gmask = 0xFu << gbase;
  uint8_t* region = smem + (threadIdx.x >> 2) * kGroupBytes;
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(region);

  uint32_t pid = 0;
  const uint8_t* buf;
  unsigned long long n, base;
  if (a.count > 1) {
    pid = pid_b;
    buf = a.table[pid].buf;
    n = a.table[pid].n;
    base = a.table[pid].chunk_base;
  } else {
    buf = a.one.buf;
    n = a.one.n;
    base = a.one.chunk_base;
  }
  const unsigned long long start = (g - base) * a.C;
  const uint32_t len = (uint32_t)min(a.C, n - start);
  const uint8_t* p = buf + start;
  const uint32_t full = (len >> 5) * 32;  // bytes in whole stripes
  const uint32_t nst = (full + kStage - 1) / kStage;
  auto sbytes = [&](uint32_t t) { return min((uint32_t)kStage, full - t * kStage); };

  unsigned long long key = 0;
  bool hit = false, cand = false;
  uint32_t hit_slot = kEmptySlot;
  if (len < kPaperMinCached) {  // recorded, never cached: only the key
    if (lane == 0) key = md5_prefix_key(p, min(len, 128u), tab.k);
    key = group_shfl(key, gmask, gbase);
    if (a.key16) key &= 0xFFFFULL;
  } else {
    // stage 0 (the first 512 bytes) -> MD5 of its first 128 bytes
    stage_copy(sbase, p, kStage, lane);
    cp_commit();
    cp_wait<0>();
    __syncwarp(gmask);
    if (lane == 0) key = md5_prefix_key(region, 128u, tab.k);
    key = group_shfl(key, gmask, gbase);
    if (a.key16) key &= 0xFFFFULL;

    // the first key+length candidate
    const unsigned long long slots_used = a.dstats[ST_SLOTS_USED];
    unsigned long long pos = mix64(key) & a.index_mask;
    uint32_t first = kEmptySlot;
    for (unsigned long long probe = 0; probe <= a.index_mask; ++probe) {
      const IndexEntry e = a.index[pos];
      if (e.slot == kEmptySlot) break;
      if (e.key == key && e.len == len) {
        if (e.slot >= slots_used) {
          if (lane == 0) atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_INTERNAL);
        } else {
          first = e.slot;
          break;
        }
      }
      pos = (pos + 1) & a.index_mask;
    }
    if (first != kEmptySlot) {
      cand = true;
      const uint8_t* q = a.arena + (unsigned long long)first * a.C;
      // stream the candidate (and the rest of the payload), two stages in flight
      stage_copy(sbase + kStage, q, kStage, lane);
      cp_commit();
      if (nst > 1) {
        stage_copy(sbase + 2 * kStage, p + kStage, sbytes(1), lane);
        stage_copy(sbase + 3 * kStage, q + kStage, sbytes(1), lane);
      }
      cp_commit();
      bool equal = true;
      for (uint32_t t = 0; t < nst; ++t) {
        cp_wait<1>();  // stage t's group; the one after it may still be in flight
        const uint32_t b = (t & 1) * 2 * kStage;
        unsigned long long d = 0;
#pragma unroll
        for (int j = 0; j < kStage / 64; ++j) {
          const uint32_t off = (uint32_t)j * 64 + lane * 16;
          if (off < sbytes(t)) {
            const uint4 x = *reinterpret_cast<const uint4*>(region + b + off);
            const uint4 y = *reinterpret_cast<const uint4*>(region + b + kStage + off);
            d |= (unsigned long long)((x.x ^ y.x) | (x.y ^ y.y) | (x.z ^ y.z) | (x.w ^ y.w));
          }
        }
        d |= __shfl_xor_sync(gmask, d, 1);
        d |= __shfl_xor_sync(gmask, d, 2);
        if (d) {
          equal = false;
          break;
        }
        if (t + 2 < nst) {  // into the buffers this lane has just read
          stage_copy(sbase + b, p + (unsigned long long)(t + 2) * kStage, sbytes(t + 2), lane);
          stage_copy(sbase + b + kStage, q + (unsigned long long)(t + 2) * kStage, sbytes(t + 2),
                     lane);
        }
        cp_commit();
      }
      cp_wait<0>();
      if (equal) {  // the bytes after the last whole stripe
        unsigned long long d = 0;
        if (lane == 0)
          for (uint32_t k = full; k < len; ++k) d |= (unsigned long long)(p[k] ^ q[k]);
        d |= __shfl_xor_sync(gmask, d, 1);
        d |= __shfl_xor_sync(gmask, d, 2);
        equal = d == 0;
      }
      if (equal) {
        hit = true;
        hit_slot = first;
      } else {  // any further candidates, by re-reading both copies
        pos = (pos + 1) & a.index_mask;
        for (unsigned long long probe = 0; probe <= a.index_mask && !hit; ++probe) {
          const IndexEntry e = a.index[pos];
          if (e.slot == kEmptySlot) break;
          if (e.key == key && e.len == len) {
            if (e.slot >= slots_used) {
              if (lane == 0) atomicCAS(&a.ctl->err, 0, (int)GLEAM_ERR_INTERNAL);
            } else if (group_equal<true>(p, a.arena + (uint64_t)e.slot * a.C, len, lane, gmask)) {
              hit = true;
              hit_slot = e.slot;
            }
          }
          pos = (pos + 1) & a.index_mask;
        }
      }
    }
  }
  if (lane == 0) {
    a.ch.status[g] = len < kPaperMinCached ? kUncached : hit ? kHit0 : cand ? kMissCand : kMissNoCand;
    a.ch.key[g] = key;
    a.ch.len[g] = len;
    a.ch.src[g] = (unsigned long long)p;
    a.ch.pidx[g] = pid;
    a.ch.hint[g] = 0;
    if (hit) a.ch.ent[g] = hit_slot;
  }
}

// SMs of the current GPU; 0 if unknown.
int sm_count() {
  static PerDevice sms;
  return sms.get([](int dev) {
    int v = 0;
    return cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess ? v : 0;
  });
}

// Whether a call hashes with a warp per chunk (k_hash_lone) instead of the
// staged kernel: its chunks fit one wave of it (16 to an SM), so that each is
// a chain that the call waits for.  Per call, back to back, all chunks cached,
// warp per chunk against staged: 64 KiB chunks, 100 / 1,200 / 2,400 of them, 49
// / 60 / 73 us against 84 / 99 / 103; 16 KiB chunks 23 / 28 / 34 against 37 /
// 41 / 45; 4 KiB chunks 12 / 19 / 19 against 16 / 20 / 21; 1 KiB chunks, whose
// 32 rounds are over when the others' second stage arrives, 11.5 / 17.5 / 18.4
// against 11.8 / 16.9 / 16.5.  With more chunks than that the DRAM is the bound
// and the staged kernel streams better (6,658 chunks of 64 KiB: 311 us the
// call, 345 with this one).  Calls that overlap hide each other's chains: only
// large chunks, and few of them, gain there (64 KiB, 100 / 600 chunks: 12 / 20
// us against 25 / 27, but 1,200 chunks 35 against 30).  Payloads in host memory
// stay with the staged kernel, whose 64-byte reads of eight chunks at a time
// cross the CPU-GPU link faster than a chunk's 512 bytes (451 chunks of 64
// KiB: 227 us the call, 314 with this one).
constexpr unsigned long long kLoneMinChunk = 4096, kLoneMinChunkOverlap = 32768;

bool lone_call(const HashArgs& a) {
  const unsigned long long sms = sm_count();
  return !a.far && (a.wait_late ? a.C >= kLoneMinChunkOverlap && a.Ntot <= 4 * sms
                                : a.C >= kLoneMinChunk && a.Ntot <= 2 * kLoneChunks * sms);
}

template <bool kProbe, uint32_t kD>
cudaError_t launch_lone(const HashArgs& a, uint32_t per, cudaStream_t s, bool pdl) {
  // a call on its own asks for a full block's shared memory whatever its
  // chunks, so that the few blocks spread over the SMs, two at most to each
  // (300 chunks of 64 KiB, one to a block: 93 us the call, so 53)
  const uint32_t smem = (a.wait_late ? per * lone_bytes(kD) : kLoneChunks * lone_bytes(4));
  cudaFuncSetAttribute((const void*)k_hash_lone<kProbe, kD>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  return launch_kernel(k_hash_lone<kProbe, kD>, dim3((unsigned)((a.Ntot + per - 1) / per)),
                       dim3(32 * (1 + per)), smem, s, pdl, a, per);
}

template <bool kProbe>
cudaError_t launch_lone(const HashArgs& a, cudaStream_t s, bool pdl) {
  // as few chunks to a block as keep every block resident at once; the fewer,
  // the more stages in flight
  const unsigned long long room = 2ull * sm_count();
  const uint32_t per =
      (uint32_t)std::min<unsigned long long>(kLoneChunks, (a.Ntot + room - 1) / room);
  static_assert(2 * (kLoneChunks * lone_bytes(4) + 3072) <= 228 * 1024 &&
                    6 * lone_bytes(6) <= kLoneChunks * lone_bytes(4) &&
                    4 * lone_bytes(8) <= kLoneChunks * lone_bytes(4),
                "two blocks per SM");
  if (a.wait_late) return launch_lone<kProbe, 4>(a, per, s, pdl);  // calls share the SMs
  if (per <= 4) return launch_lone<kProbe, 8>(a, per, s, pdl);
  if (per <= 6) return launch_lone<kProbe, 6>(a, per, s, pdl);
  return launch_lone<kProbe, 4>(a, per, s, pdl);
}

Md5Table md5_table() {
  Md5Table t;
  for (int i = 0; i < 64; ++i)
    t.k[i] = (uint32_t)std::floor(std::fabs(std::sin((double)(i + 1))) * 4294967296.0);
  return t;
}

}  // namespace

// Every variant that launch_hash may launch.
cudaError_t load_hash_kernels() {
  return load_kernels<
      k_hash_lone<false, 4>, k_hash_lone<false, 6>, k_hash_lone<false, 8>, k_hash_lone<true, 4>,
      k_hash_lone<true, 6>, k_hash_lone<true, 8>,
      k_hash_probe_staged<false, false, false>,
      k_hash_probe_staged<false, false, false, false, kStage, true>,
      k_hash_probe_staged<true, false, false>, k_hash_probe_staged<true, true, false>,
      k_hash_probe_staged<true, false, true>, k_hash_probe_staged<true, true, true>,
      k_hash_probe_staged<true, false, true, true>, k_hash_probe_staged<true, true, true, true>,
      k_hash_probe_staged<true, false, false, false, kStage, true>,
      k_hash_probe_staged<true, false, true, false, kStage, true>,
      k_hash_probe_staged<true, false, true, true, kStage, true>,
      k_hash_probe_staged<true, false, false, false, kBigStage>,
      k_hash_probe_staged<true, true, false, false, kBigStage>,
      k_hash_probe_staged<true, false, true, false, kBigStage>,
      k_hash_probe_staged<true, true, true, false, kBigStage>, k_probe_paper,
      k_probe_paper_staged>();
}

bool hash_is_lone(const HashArgs& a) {
  return a.Ntot > 0 && !(a.index != nullptr && a.paper) && lone_call(a);
}

bool hash_is_staged(const HashArgs& a) { return a.Ntot > 0 && !(a.index != nullptr && a.paper); }

cudaError_t launch_hash(const HashArgs& a, bool aligned, cudaStream_t s, bool pdl) {
  if (a.Ntot == 0) return cudaSuccess;
  const bool probe = a.index != nullptr;
  if (probe && a.paper) {
    static const Md5Table tab = md5_table();
    const unsigned long long threads = a.Ntot * 4;
    if (aligned) {
      const unsigned sg = (unsigned)((threads + kStagedThreads - 1) / kStagedThreads);
      return launch_kernel(k_probe_paper_staged, dim3(sg), dim3(kStagedThreads), kStagedSmem, s,
                           pdl, a, tab);
    }
    const unsigned grid = (unsigned)((threads + kHashThreads - 1) / kHashThreads);
    return launch_kernel(k_probe_paper, dim3(grid), dim3(kHashThreads), 0, s, pdl, a, tab);
  }
  if (lone_call(a)) return probe ? launch_lone<true>(a, s, pdl) : launch_lone<false>(a, s, pdl);
  // no cached copy is streamed when only fingerprints are wanted or the cache
  // holds no chunk (or too few to be worth the hint lookups): the variant
  // without those buffers
  if (!aligned) {  // no write-through: its 16-byte stores want aligned payloads
    if (!probe) return launch_staged<false, false, false, false, kStage, true>(a, s, pdl);
    if (a.no_hints) return launch_staged<true, false, false, false, kStage, true>(a, s, pdl);
    return launch_staged<true, false, true, false, kStage, true>(a, s, pdl);
  }
  if (!probe) return launch_staged<false, false, false>(a, s, pdl);
  if (a.no_hints)
    return a.spec_mode ? launch_staged<true, true, false>(a, s, pdl)
                       : launch_staged<true, false, false>(a, s, pdl);
  return a.spec_mode ? launch_staged<true, true, true>(a, s, pdl)
                     : launch_staged<true, false, true>(a, s, pdl);
}

}  // namespace gleam
