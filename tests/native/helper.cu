// GPU code that only the tests need.
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>
#include <vector>

#include "gleam_internal.cuh"

using namespace gleam;

// Holds smem bytes of shared memory per block for about ns nanoseconds.
__global__ void k_hold(unsigned long long ns) {
  extern __shared__ uint8_t held[];
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  if (threadIdx.x == 0) held[0] = 1;
  do {
    __nanosleep(1000);
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  } while (t - t0 < ns);
}

// k_hold on the stream: a block on every SM where two of them do not fit (more
// than 114 KiB each), else one block.  0 or a CUDA error.
extern "C" int helper_hold(uint64_t smem, uint64_t ns, cudaStream_t stream) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess && (smem == 0 || smem > 227 * 1024 || ns > 1000000000ull))
    e = cudaErrorInvalidValue;
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_hold, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  // the whole of the SM's shared memory, so that other kernels' blocks fit beside it
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_hold, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return (int)e;
  k_hold<<<smem > 114 * 1024 ? sms : 1, 32, smem, stream>>>(ns);
  return (int)cudaGetLastError();
}

// Device memory that starts zeroed (or as given), freed with the object.
template <typename T>
struct Dev {
  T* p = nullptr;
  size_t n;
  explicit Dev(size_t count, const T* from = nullptr) : n(count) {
    if (cudaMalloc(&p, n * sizeof(T)) != cudaSuccess) p = nullptr;
    if (from) cudaMemcpy(p, from, n * sizeof(T), cudaMemcpyHostToDevice);
    else cudaMemset(p, 0, n * sizeof(T));
  }
  ~Dev() { cudaFree(p); }
  std::vector<T> host() const {
    std::vector<T> v(n);
    cudaMemcpy(v.data(), p, n * sizeof(T), cudaMemcpyDeviceToHost);
    return v;
  }
};

// What a call of cache hits alone left behind.
struct HitsOut {
  int64_t status, hits, calls;
  uint64_t mask0, slots_ok, uses_old, uses_new, ctl_left;
};

// The resolve kernel on `grid` blocks and the pack kernel on one, for nch chunks
// that all hit (chunk g slot g, last used at 3) in an evicting cache whose clock
// is at 9, with the control block's barrier count and error word as given.
extern "C" int helper_all_hits(uint32_t grid, uint32_t nch, uint32_t bar_count, int err,
                               uint64_t wait_ns, HitsOut* out) {
  if (nch == 0 || nch > 4096 || grid == 0 || grid > 32) return (int)cudaErrorInvalidValue;
  const uint64_t C = 1024, icap = 8192;
  std::vector<uint32_t> len(nch, (uint32_t)C), ent(nch), use(nch, 3u);
  std::vector<unsigned long long> key(nch, 7ull);
  for (uint32_t g = 0; g < nch; ++g) ent[g] = g;
  std::vector<unsigned long long> stats(ST_COUNT, 0ull);
  stats[ST_SLOTS_USED] = nch;
  std::vector<IndexEntry> none(icap);
  std::memset(none.data(), 0xFF, icap * sizeof(IndexEntry));
  std::vector<uint8_t> st(nch, kHit0);
  DevCtl ctl0{};
  ctl0.bar_count = bar_count;
  ctl0.err = err;
  gleam_result_t res0{};
  res0.status = 77;
  Dev<uint8_t> status(nch, st.data()), spec(nch), vflag(nch), buf(nch * C), packed(nch * C),
      arena(nch * C);
  Dev<unsigned long long> d_key(nch, key.data()), src(nch), hint(nch), cls(nch),
      dstats(ST_COUNT, stats.data()), skey(nch);
  Dev<uint32_t> d_len(nch, len.data()), pidx(nch), res(nch), d_ent(nch, ent.data()), rank(nch),
      order(nch), srank(nch), old(nch), last(nch, use.data()), victims(nch), bins(kLruBins),
      slen(nch, len.data()), bcount(4096), mask((nch + 31) / 32), idx(nch), slots(nch);
  Dev<IndexEntry> index(icap, none.data()), hints(icap, none.data());
  Dev<CallEntry> tbl(8192);
  Dev<DevCtl> ctl(1, &ctl0);
  Dev<gleam_result_t> total(1, &res0);
  DedupArgs a{};
  a.one.buf = buf.p;
  a.one.n = nch * C;
  a.one.nchunks = nch;
  a.one.mask = mask.p;
  a.one.miss_idx = idx.p;
  a.one.packed = packed.p;
  a.one.chunk_slot = slots.p;
  a.count = 1;
  a.Ntot = nch;
  a.C = C;
  a.arena = arena.p;
  a.index = index.p;
  a.hints = hints.p;
  a.index_mask = icap - 1;
  a.nslots = nch;
  a.slot_len = slen.p;
  a.slot_key = skey.p;
  a.dstats = dstats.p;
  a.ch.status = status.p;
  a.ch.key = d_key.p;
  a.ch.len = d_len.p;
  a.ch.src = src.p;
  a.ch.pidx = pidx.p;
  a.ch.res = res.p;
  a.ch.ent = d_ent.p;
  a.ch.rank = rank.p;
  a.ch.hint = hint.p;
  a.ch.order = order.p;
  a.ch.srank = srank.p;
  a.ch.old = old.p;
  a.ch.spec = spec.p;
  a.ch.cls = cls.p;
  a.tbl = tbl.p;
  a.tbl_mask = tbl.n - 1;
  a.bcount = bcount.p;
  a.pstart = bcount.p + 4095;
  a.ctl = ctl.p;
  a.total = total.p;
  a.ncalls = 1;
  a.wait_ns = wait_ns;
  a.skip_block = -1;
  a.lru = 1;
  a.epoch = 9;
  a.last_use = last.p;
  a.vflag = vflag.p;
  a.victims = victims.p;
  a.bins = bins.p;
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = launch_dedup(a, (int)grid, 1, nullptr, false);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) return (int)e;
  const gleam_result_t r = total.host()[0];
  out->status = r.status;
  out->hits = (int64_t)r.n_hit_cache;
  out->calls = (int64_t)dstats.host()[ST_CALLS];
  out->mask0 = mask.host()[0];
  out->slots_ok = out->uses_old = out->uses_new = out->ctl_left = 0;
  const std::vector<uint32_t> sl = slots.host(), lu = last.host();
  for (uint32_t g = 0; g < nch; ++g) {
    out->slots_ok += sl[g] == g;
    out->uses_old += lu[g] == 3;
    out->uses_new += lu[g] == 9;
  }
  DevCtl left = ctl.host()[0];
  left.published = 0;  // each call's first kernel sets it
  const uint8_t* b = reinterpret_cast<const uint8_t*>(&left);
  for (size_t k = 0; k < sizeof(DevCtl); ++k) out->ctl_left += b[k] != 0;
  return 0;
}

// The hash kernel alone over n bytes of device memory in chunks of C, with every
// wait between warps limited to wait_ns.  probe: as a dedup call on an empty
// cache launches it (fingerprints from the chunks' records); else as
// gleam_fingerprint does.  fp: host, one word per chunk; *err: the error recorded.
extern "C" int helper_hash(const uint8_t* d_buf, uint64_t n, uint64_t C, int probe,
                           uint64_t wait_ns, unsigned long long* fp, int* err, int* lone) {
  const uint64_t N = (n + C - 1) / C, icap = 1024;
  if (N == 0 || N > 4096) return (int)cudaErrorInvalidValue;
  std::vector<IndexEntry> none(icap);
  std::memset(none.data(), 0xFF, icap * sizeof(IndexEntry));
  Dev<uint8_t> status(N), spec(N), arena(C);
  Dev<unsigned long long> key(N), src(N), hint(N), out(N), dstats(ST_COUNT), skey(1);
  Dev<uint32_t> len(N), pidx(N), ent(N), res(N);
  Dev<IndexEntry> index(icap, none.data()), hints(icap, none.data());
  Dev<DevCtl> ctl(1);
  HashArgs h{};
  h.one.buf = d_buf;
  h.one.n = n;
  h.one.nchunks = N;
  h.count = 1;
  h.Ntot = N;
  h.C = C;
  h.wait_ns = wait_ns;
  h.ctl = ctl.p;
  if (probe) {
    h.index = index.p;
    h.index_mask = icap - 1;
    h.hints = hints.p;
    h.arena = arena.p;
    h.slot_key = skey.p;
    h.dstats = dstats.p;
    h.ch.status = status.p;
    h.ch.key = key.p;
    h.ch.len = len.p;
    h.ch.src = src.p;
    h.ch.pidx = pidx.p;
    h.ch.res = res.p;
    h.ch.ent = ent.p;
    h.ch.hint = hint.p;
    h.ch.spec = spec.p;
    h.no_hints = 1;
  } else {
    h.fp_out = out.p;
  }
  *lone = hash_is_lone(h);
  const bool aligned = (uintptr_t)d_buf % 16 == 0 && (N == 1 || C % 16 == 0);
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = launch_hash(h, aligned, nullptr, false);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) return (int)e;
  const std::vector<unsigned long long> v = probe ? key.host() : out.host();
  std::memcpy(fp, v.data(), N * 8);
  *err = ctl.host()[0].err;
  return 0;
}

// A kept figure is asked for until it is known, and once from then on: three
// digits, the figure after each of three gets whose question would give 0, 5, 7.
extern "C" int helper_per_device() {
  static PerDevice kept;
  int digits = 0;
  for (int answer : {0, 5, 7}) digits = 10 * digits + kept.get([answer](int) { return answer; });
  return digits;
}
