// kern_small.cu -- the build of a table that fits one SM's shared memory (up
// to 28,000 slots of a pair table), by one block in one launch.
//
// A build over the whole GPU pays a microsecond or two for every step of its
// longest eviction chain (a read from L2, then an atomic there), one launch
// each for the fill, the placement and the insert, and the gaps between them:
// 20,000 keys at LF 0.95 took 7 + 67 us of kernels. One SM holds such a table
// in shared memory, where a step takes tens of nanoseconds, fills it there,
// and writes each line of the table once. What is left is one SM's time for the
// keys, about 3 us per 1000 (and their chains'), so there is a most that it is
// used for (wants_small in ght_api.cu).
//
// The tables are those of the bucketed insert (Sec. III, V): a bucket's
// arrivals are counted in shared memory, and a key takes the slot of its
// arrival number, so slots fill in order. A slot holds its key's index in the
// input (32 bits) until the end: 64-bit exchanges of whole pairs in shared
// memory take ~7 ns of the SM each (20,000 keys of bucket size one took 333
// us), 32-bit ones do not. The values wait in shared memory too where they
// fit, else they are gathered when the table is written.
//   BCHT, set: as the two-phase build, first every key that finds room in
//     H_0, then the rest from H_1 on: the next free slot of the bucket, or the
//     exchange with a random slot, the evicted pair moving on to its next hash.
//   IHT: first the keys that find fewer than t - 1 in their primary, then the
//     rest into the less loaded secondary, or the primary if both are full.
//   P2BHT, load-balanced BCHT, bucket size one: every key in turn.
#include "ght_internal.h"
#include "ght_kernels.cuh"

namespace ght {

namespace {

constexpr int kSmallThreads = 1024;
constexpr int kSmallKeys = 32;  // keys per thread at most: one bit each in its mask of keys left for later
constexpr int kSmallBatch = 8;  // keys a thread has in flight from memory

}  // namespace

constexpr uint32_t kNone = 0xFFFFFFFFu;  // an empty slot

// 227 KB per block, of which the kernel's own variables take less than 1 KB
constexpr uint64_t kSmallSmem = 226u * 1024u;

// keys, one index per slot, and the buckets' counts
uint64_t small_build_smem(int B, uint64_t m, uint64_t n) { return 4u * (n + m * (uint64_t)B + (B > 1 ? m : 0u)); }

template <int SCHEME, int B, bool COUNT, typename S>
__global__ void __launch_bounds__(kSmallThreads, 1)
small_build_kernel(TableView tv, const uint32_t *__restrict__ keys, const uint32_t *__restrict__ values, uint32_t n,
                   uint32_t limit, bool keep_values, PublishedCtrl *__restrict__ host, unsigned long long number) {
  using T = typename S::T;
  extern __shared__ uint32_t sb_smem[];
  uint32_t *skey = sb_smem;           // [n]
  uint32_t *slot = skey + n;          // [m * B]
  uint32_t *cnt = slot + tv.m * B;    // [m] pairs of each bucket
  uint32_t *sval = cnt + (B > 1 ? tv.m : 0u);  // [n], with keep_values
  volatile uint32_t *loads = cnt;
  __shared__ uint32_t s_status;
  __shared__ unsigned long long s_probes, s_retries, s_evictions, s_longest;
  const int tid = threadIdx.x;
  const uint32_t m = tv.m, slots = m * B;
  const int h = tv.h;
  if (tid == 0) {
    s_status = 0u;
    s_probes = s_retries = s_evictions = s_longest = 0ull;
  }
  for (uint32_t i0 = tid; i0 < n; i0 += kSmallThreads * kSmallBatch) {
    uint32_t k[kSmallBatch], v[kSmallBatch];
#pragma unroll
    for (int u = 0; u < kSmallBatch; ++u) {
      const uint32_t i = i0 + u * kSmallThreads;
      k[u] = i < n ? __ldg(keys + i) : 0u;
      v[u] = keep_values && i < n ? __ldg(values + i) : 0u;
    }
#pragma unroll
    for (int u = 0; u < kSmallBatch; ++u) {
      const uint32_t i = i0 + u * kSmallThreads;
      if (i < n) skey[i] = k[u];
      if (keep_values && i < n) sval[i] = v[u];
    }
  }
  for (uint32_t i = tid; i < slots; i += kSmallThreads) slot[i] = kNone;
  if (B > 1)
    for (uint32_t i = tid; i < m; i += kSmallThreads) cnt[i] = 0u;
  uint32_t rng = lane_seed(tv.rng_seed, (uint64_t)tid);
  unsigned long long probes = 0, retries = 0, evictions = 0, longest = 0;
  __syncthreads();

  auto fail = [&](uint32_t bit) { atomicOr(&s_status, bit); };
  auto stop = [&]() {
    return (*(volatile uint32_t *)&s_status & (kStatusBuildFailed | kStatusTimeout | kStatusCorrupt)) != 0u;
  };
  // the lowest hash index under which key k lies in bucket b, h if none
  auto index_in = [&](uint32_t k, uint32_t bk) {
    int i = 0;
    while (i < h && bucket_of(tv.hf, i, k) != bk) ++i;
    return i;
  };
  // add one to bucket b's count if it is still c
  auto claim = [&](uint32_t b, uint32_t c) { return atomicCAS(&cnt[b], c, c + 1u) == c; };

  // What a thread is doing: key x (an index into skey), the bucket it goes to
  // (BCHT, bucket size one) or was evicted from, its exchanges and bucket visits.
  uint32_t x = kNone, b = 0, chain = 0, steps = 0;
  bool again = false;  // the last visit lost a CAS
  // Each of the following takes one step of x and returns whether x is done: it
  // is stored, or the build has failed. A thread takes one step per turn and
  // then its next key, so that a warp's threads don't wait for one another's
  // chains.
  auto give_up = [&](uint32_t bit) {
    fail(bit);
    return true;
  };
  // x took the place of key `old` in bucket b (none: x is stored); BCHT and
  // bucket size one go on with old at its next hash
  auto took = [&](uint32_t old) {
    if (old == kNone) return true;
    const int i = index_in(skey[old], b);
    if (i >= h) return give_up(kStatusCorrupt);
    x = old;
    b = bucket_of(tv.hf, (i + 1) % h, skey[old]);
    return false;
  };
  auto evict = [&](uint32_t at) {
    const uint32_t old = atomicExch(&slot[at], x);
    if (COUNT) evictions++;
    if (++chain > longest) longest = chain;
    return old;
  };
  auto cuckoo = [&]() {  // BCHT at bucket b
    if (++steps > tv.max_steps) return give_up(kStatusTimeout);
    if (COUNT) probes++;
    uint32_t r = loads[b];
    if (r < (uint32_t)B) r = atomicAdd(&cnt[b], 1u);
    // an exchange for a free slot too: an eviction may have come to it first, and its key then moves on
    if (r < (uint32_t)B) return took(atomicExch(&slot[b * B + r], x));
    if (chain >= tv.max_chain) return give_up(kStatusBuildFailed);
    return took(evict(b * B + xorshift32(rng) % B));
  };
  auto two_choice = [&]() {  // P2BHT: the less loaded of two (ties to H_0)
    const uint32_t b0 = bucket_of(tv.hf, 0, skey[x]), b1 = bucket_of(tv.hf, 1, skey[x]);
    steps += 2;
    if (steps > tv.max_steps) return give_up(kStatusTimeout);
    if (COUNT) (steps == 2 ? probes : retries) += 2;
    const uint32_t c0 = loads[b0], c1 = loads[b1];
    if (c0 >= (uint32_t)B && c1 >= (uint32_t)B) return give_up(kStatusBuildFailed);
    const uint32_t bc = c0 <= c1 ? b0 : b1, c = c0 <= c1 ? c0 : c1;
    if (!claim(bc, c)) return false;
    slot[bc * B + c] = x;
    return true;
  };
  // IHT beyond the primary's share: the less loaded secondary (ties to H_1), then the primary
  auto secondary = [&]() {
    const uint32_t k = skey[x], b1 = bucket_of(tv.hf, 1, k), b2 = bucket_of(tv.hf, 2, k);
    const bool first = steps == 1;  // (the primary was visited before)
    steps += 2;
    if (steps > tv.max_steps) return give_up(kStatusTimeout);
    if (COUNT) (first ? probes : retries) += 2;
    const uint32_t c1 = loads[b1], c2 = loads[b2];
    uint32_t bc = c1 <= c2 ? b1 : b2, c = c1 <= c2 ? c1 : c2;
    if (c >= (uint32_t)B) {
      if (COUNT) (first ? probes : retries) += 1;
      bc = bucket_of(tv.hf, 0, k);
      c = loads[bc];
      if (c >= (uint32_t)B) return give_up(kStatusBuildFailed);
    }
    if (!claim(bc, c)) return false;
    slot[bc * B + c] = x;
    return true;
  };
  // load-balanced BCHT: the least loaded candidate (ties to the lowest index),
  // not the bucket b that x was just evicted from; all full: exchange there
  auto balanced = [&]() {
    steps += h;
    if (steps > tv.max_steps) return give_up(kStatusTimeout);
    if (COUNT) (again ? retries : probes) += h;
    uint32_t bc = 0, c = B + 1;
    for (int f = 0; f < h; ++f) {
      const uint32_t bf = bucket_of(tv.hf, f, skey[x]);
      const uint32_t cf = min(loads[bf], (uint32_t)B);
      if (bf != b && cf < c) {
        bc = bf;
        c = cf;
      }
    }
    uint32_t old;
    if (c < (uint32_t)B) {
      again = !claim(bc, c);
      if (again) return false;
      old = atomicExch(&slot[bc * B + c], x);  // (see cuckoo)
    } else if (c > (uint32_t)B || chain >= tv.max_chain) {
      return give_up(kStatusBuildFailed);  // no candidate besides the one it came from, or chain bound
    } else {
      old = evict(bc * B + xorshift32(rng) % B);
    }
    if (old == kNone) return true;
    x = old;
    b = bc;
    return false;
  };
  // bucket size one: exchange, the displaced key moves on; at the chain bound
  // only an empty slot takes it
  auto single = [&]() {
    if (COUNT) probes++;
    if (chain < tv.max_chain) {
      const uint32_t old = atomicExch(&slot[b], x);
      if (old == kNone) return true;
      if (COUNT) evictions++;
      if (++chain > longest) longest = chain;
      return took(old);
    }
    return atomicCAS(&slot[b], kNone, x) == kNone || give_up(kStatusBuildFailed);
  };

  constexpr bool kTwoPhase = SCHEME == kBCHT || SCHEME == kIHT;
  constexpr bool kValues = sizeof(T) == 8;
  uint32_t left = 0u;  // bit j: key j of this thread takes steps
  for (uint32_t i = tid, j = 0; i < n; i += kSmallThreads, ++j) {
    const uint32_t k = skey[i];
    if (k == kEmptyKey) {
      fail(kStatusSentinel);
    } else if (kTwoPhase) {
      const uint32_t h0 = bucket_of(tv.hf, 0, k);
      const uint32_t r = atomicAdd(&cnt[h0], 1u);
      if (COUNT) probes++;
      if (r < limit) slot[h0 * B + r] = i;
      else left |= 1u << j;
    } else {
      left |= 1u << j;
    }
  }
  if (kTwoPhase) {
    __syncthreads();
    for (uint32_t i = tid; i < m; i += kSmallThreads) cnt[i] = min(cnt[i], limit);  // the arrivals that were stored
    __syncthreads();
  }
  for (;;) {
    if (x == kNone) {
      if (left == 0u) break;
      x = (uint32_t)(__ffs(left) - 1) * kSmallThreads + tid;
      left &= left - 1u;
      chain = 0;
      steps = kTwoPhase ? 1u : 0u;
      again = false;
      b = SCHEME == kBCHT_LB ? 0xFFFFFFFFu : bucket_of(tv.hf, SCHEME == kBCHT ? 1 : 0, skey[x]);
    }
    bool done;
    if (SCHEME == kBCHT) done = cuckoo();
    else if (SCHEME == kP2BHT) done = two_choice();
    else if (SCHEME == kIHT) done = secondary();
    else if (SCHEME == kBCHT_LB) done = balanced();
    else done = single();
    if (done) x = kNone;
    if (stop()) break;
  }
  __syncthreads();
  T *dst = reinterpret_cast<T *>(tv.slots);
  for (uint32_t i0 = tid; i0 < slots; i0 += kSmallThreads * kSmallBatch) {
    uint32_t x[kSmallBatch], v[kSmallBatch];
#pragma unroll
    for (int u = 0; u < kSmallBatch; ++u) {
      const uint32_t i = i0 + u * kSmallThreads;
      x[u] = i < slots ? slot[i] : kNone;
      v[u] = kValues && x[u] != kNone ? (keep_values ? sval[x[u]] : __ldg(values + x[u])) : 0u;
    }
#pragma unroll
    for (int u = 0; u < kSmallBatch; ++u) {
      const uint32_t i = i0 + u * kSmallThreads;
      if (i < slots) dst[i] = x[u] == kNone ? S::kEmpty : S::make(skey[x[u]], v[u]);
    }
  }
  if (COUNT) {
    atomicAdd(&s_probes, probes);
    atomicAdd(&s_retries, retries);
    atomicAdd(&s_evictions, evictions);
    atomicMax(&s_longest, longest);
    __syncthreads();
  }
  if (tid < (int)(sizeof(Ctrl) / 8)) reinterpret_cast<unsigned long long *>(tv.ctrl)[tid] = 0ull;
  __syncwarp();
  if (tid == 0) {
    tv.ctrl->status = s_status;
    tv.ctrl->insert_probes = s_probes;
    tv.ctrl->insert_retries = s_retries;
    tv.ctrl->insert_evictions = s_evictions;
    tv.ctrl->longest_chain = s_longest;
  }
  // the host may go on once it sees the number: every line of the table is written
  __threadfence_system();
  __syncthreads();
  if (tid < 32) publish_ctrl(tv.ctrl, host, number, tid);
}

template <int SCHEME, int B, typename S>
static cudaError_t launch_small(const TableView &tv, const uint32_t *k, const uint32_t *v, uint64_t n, uint32_t limit,
                                bool count, PublishedCtrl *host, unsigned long long number, cudaStream_t s) {
  auto kern = count ? small_build_kernel<SCHEME, B, true, S> : small_build_kernel<SCHEME, B, false, S>;
  uint64_t smem = small_build_smem(B, tv.m, n);
  const bool keep_values = sizeof(typename S::T) == 8 && smem + 4u * n <= kSmallSmem;
  if (keep_values) smem += 4u * n;
  const cudaError_t e = allow_smem(kern, kSmallSmem);
  if (e != cudaSuccess) return e;
  kern<<<1, kSmallThreads, smem, s>>>(tv, k, v, (uint32_t)n, limit, keep_values, host, number);
  return cudaGetLastError();
}

// Values that do not fit beside the keys are gathered 4 bytes at a time when the
// table is written. From host memory that takes L1, which the lines fetched over
// the link stay in: none is left beside more than 195 KB. Builds from page-locked
// arrays, us, this / two phases: IHT LF 0.78 21,000 keys (194 KB) 65 / 71, 22,000
// (203 KB) 121 / 72; LF 0.6 18,000 (195 KB) 55 / 60, 19,000 (206 KB) 104 / 59;
// P2BHT LF 0.6 18,000 61 / 60, 19,000 109 / 59.
bool small_build_fits(int B, bool key_slots, uint64_t m, uint64_t n, bool far_values) {
  const uint64_t smem = small_build_smem(B, m, n);
  if (n > (uint64_t)kSmallThreads * kSmallKeys || smem > kSmallSmem) return false;
  return !far_values || key_slots || smem <= 195u * 1024u || smem + 4u * n <= kSmallSmem;
}

cudaError_t launch_small_build(int scheme, int B, bool key_slots, const TableView &tv, const uint32_t *k,
                               const uint32_t *v, uint64_t n, uint32_t limit, bool count, PublishedCtrl *host,
                               unsigned long long number, cudaStream_t s) {
  if (!small_build_fits(B, key_slots, tv.m, n, false)) return cudaErrorInvalidValue;
  if (key_slots) return launch_small<kBCHT, 32, KeySlot>(tv, k, v, n, limit, count, host, number, s);
  if (scheme == kCuckoo1) return launch_small<kCuckoo1, 1, PairSlot>(tv, k, v, n, limit, count, host, number, s);
  if (B == 16) {
    if (scheme == kBCHT) return launch_small<kBCHT, 16, PairSlot>(tv, k, v, n, limit, count, host, number, s);
    if (scheme == kP2BHT) return launch_small<kP2BHT, 16, PairSlot>(tv, k, v, n, limit, count, host, number, s);
    if (scheme == kIHT) return launch_small<kIHT, 16, PairSlot>(tv, k, v, n, limit, count, host, number, s);
    if (scheme == kBCHT_LB) return launch_small<kBCHT_LB, 16, PairSlot>(tv, k, v, n, limit, count, host, number, s);
  }
  if (B == 32) {
    if (scheme == kBCHT) return launch_small<kBCHT, 32, PairSlot>(tv, k, v, n, limit, count, host, number, s);
    if (scheme == kP2BHT) return launch_small<kP2BHT, 32, PairSlot>(tv, k, v, n, limit, count, host, number, s);
    if (scheme == kIHT) return launch_small<kIHT, 32, PairSlot>(tv, k, v, n, limit, count, host, number, s);
    if (scheme == kBCHT_LB) return launch_small<kBCHT_LB, 32, PairSlot>(tv, k, v, n, limit, count, host, number, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ght
