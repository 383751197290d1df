// ght_find_line.cuh -- bulk find of tables with 128-byte buckets (16 pairs or
// 32 keys) with 32-byte loads: the find of every such table whose config names
// no find shape of its own.
//
// A tile of four lanes reads a 128-byte line with one 32-byte load per lane
// (one instruction, each line once in the L1's pipeline), a warp probes 32
// queries at a time, one per lane, and a query that needs another bucket waits
// in shared memory until 32 such queries fill a warp again. So all lanes work
// in every step and a step is short: 178-181 warp instructions for 32
// probes, against 415 in the register find (bucketed_find_kernel) and 392 in
// the staged find (bcht_find_async_kernel), and with 64 registers a thread 32
// warps fit on an SM instead of 16 and 12. That hides the latency of 1024
// lines per SM without query sets in flight: the tables that fit the L2 are
// bound by the SMs' reads from it, the others by DRAM's rate of random lines.
//
// Finds on GB300, us, 2^k queries on a table of 2^k keys, before -> now (half
// present; before: register find up to 2^22 keys, staged find beyond):
//   BCHT 2^20 LF 0.9 41 -> 23, 2^22 LF 0.9 124 -> 59 (13 TB/s from the L2),
//   2^24 LF 0.95 677 -> 312, 2^26 LF 0.9 2400 -> 1990; 2^28 LF 0.99 present
//   9570 -> 9250, absent 19090 -> 18370 (40.1 and 40.8 G lines/s of the 42.2
//   that DRAM gives to random lines); P2BHT 2^24 628 -> 332, IHT 2^24 822 ->
//   416, set of 50M keys 1836 -> 1078.
// Buckets of 32 pairs (two lines, tiles of eight lanes, 64 registers of loads,
// 16 warps per SM) lost to the staged find beyond the L2 (P2BHT 2^24 keys 1640
// against 925) and won nothing inside it (208 / 213), so they keep the others.
#pragma once

#include "ght_find.cuh"
#include "ght_internal.h"

namespace ght {

// 32 bytes of a bucket (four pairs or eight keys) through the read-only path;
// the line is not kept in L1, where random buckets do not meet again.
__device__ __forceinline__ void load32_ro(const void *p, uint32_t (&x)[8]) {
  asm volatile("ld.global.nc.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]), "=r"(x[4]), "=r"(x[5]), "=r"(x[6]), "=r"(x[7])
               : "l"(p));
}

constexpr int kLineFindLanes = 4;  // lanes of a tile: 128 bytes
constexpr int kLineFindThreads = 256;
constexpr int kLineFindWarps = kLineFindThreads / 32;
// queries of a warp that wait for another probe: fewer than 32 are left
// behind, and a step adds at most 32
constexpr int kLineFindWaiting = 64;
// a waiting query is its key and (its place in the warp's slice, next probe);
// h <= 4 leaves 30 bits for the place
constexpr uint32_t kLineFindPlaceBits = 30;

// One probe of 32 queries, lane i owning key k: part(j, x) loads this lane's 32
// bytes of the bucket of tile member j. Sets hit and the found value, and
// empty: whether the bucket has an empty slot, which its last slot shows --
// every insert takes the first empty slot of a bucket in one fixed order that
// ends there, and no slot is ever emptied again.
template <typename S, bool EARLY, typename Part>
__device__ __forceinline__ void line_probe(uint32_t k, int r, int tbase, int lane, Part part, bool &hit, bool &empty,
                                           uint32_t &value) {
  constexpr bool kPairs = sizeof(typename S::T) == 8;
  constexpr int G = kLineFindLanes;
  uint32_t x[G][8], val[G];
  unsigned my_hits = 0u, my_emp = 0u;
#pragma unroll
  for (int j = 0; j < G; ++j) part(j, x[j]);
#pragma unroll
  for (int j = 0; j < G; ++j) {
    const uint32_t kj = __shfl_sync(kFull, k, tbase + j);
    bool h = false;
    val[j] = 1u;
    if (kPairs) {
#pragma unroll
      for (int p = 0; p < 4; ++p)
        if (x[j][2 * p] == kj) {
          h = true;
          val[j] = x[j][2 * p + 1];
        }
    } else {
#pragma unroll
      for (int p = 0; p < 8; ++p) h |= x[j][p] == kj;
    }
    const unsigned hb = __ballot_sync(kFull, h);
    if (r == j) my_hits = hb;
    if (EARLY) {
      const unsigned eb = __ballot_sync(kFull, x[j][kPairs ? 6 : 7] == kEmptyKey);
      if (r == j) my_emp = eb;
    }
  }
  my_hits = (my_hits >> tbase) & ((1u << G) - 1u);
  hit = my_hits != 0u;
  empty = EARLY && ((my_emp >> (tbase + G - 1)) & 1u);
  value = 1u;
  if (kPairs) {
    const int src = hit ? tbase + __ffs(my_hits) - 1 : lane;
#pragma unroll
    for (int j = 0; j < G; ++j) {
      const uint32_t y = __shfl_sync(kFull, val[j], src);
      if (r == j) value = y;
    }
  }
}

// EARLY: BCHT's stop at a bucket with an empty slot (Sec. V-B find); without it
// a query reads its candidates until its key is found (Sec. V-C, V-D).
template <typename S, bool EARLY, bool COUNT>
__global__ void __launch_bounds__(kLineFindThreads, 4)
line_find_kernel(TableView tv, const uint32_t *__restrict__ queries, uint32_t *__restrict__ out, uint64_t n,
                 uint32_t per_warp) {
  constexpr int G = kLineFindLanes;
  __shared__ uint2 s_wait[kLineFindWarps][kLineFindWaiting];
  const int lane = threadIdx.x & 31;
  const int r = lane & (G - 1);
  const int tbase = lane - r;
  const unsigned below = lanemask_lt();
  uint2 *wait = s_wait[threadIdx.x >> 5];
  const uint64_t beg = (((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * per_warp;
  if (beg >= n) return;  // whole warp
  const uint32_t len = (uint32_t)(n - beg < per_warp ? n - beg : per_warp);
  queries += beg;
  out += beg;
  const char *base = reinterpret_cast<const char *>(tv.slots) + r * 32;
  int waiting = 0;
  unsigned long long probes = 0;
  uint32_t next = __ldg(queries + min((uint32_t)lane, len - 1u));
  for (uint32_t c = 0;;) {
    // 32 queries: those that wait, once they fill the warp or the slice is
    // spent, else the next of the slice. Lanes without a query repeat one.
    uint32_t k, at;
    int probe;
    bool valid;
    if (waiting >= 32 || c >= len) {
      if (waiting == 0) break;
      const int take = min(waiting, 32);
      waiting -= take;
      const uint2 e = wait[waiting + min(lane, take - 1)];
      k = e.x;
      at = e.y & ((1u << kLineFindPlaceBits) - 1u);
      probe = (int)(e.y >> kLineFindPlaceBits);
      valid = lane < take;
      __syncwarp();  // read before the step's own entries go there
    } else {
      k = next;
      at = c + lane;
      probe = 0;
      c += 32;
      if (c < len) next = __ldg(queries + min(c + lane, len - 1u));
      valid = at < len && k != kEmptyKey;
      if (at < len && k == kEmptyKey) out[at] = S::missing();  // the sentinel is never a key
    }
    const uint32_t b = bucket_of(tv.hf, probe, k);
    bool hit, empty;
    uint32_t value;
    line_probe<S, EARLY>(
        k, r, tbase, lane,
        [&](int j, uint32_t(&x)[8]) { load32_ro(base + (uint64_t)__shfl_sync(kFull, b, tbase + j) * 128u, x); },
        hit, empty, value);
    if (COUNT && valid) probes++;
    const bool more = valid && !hit && !empty && probe + 1 < tv.h;
    if (valid && !more) out[at] = hit ? value : S::missing();
    const unsigned mb = __ballot_sync(kFull, more);
    if (more) wait[waiting + __popc(mb & below)] = make_uint2(k, at | ((uint32_t)(probe + 1) << kLineFindPlaceBits));
    waiting += __popc(mb);
    __syncwarp();
  }
  if (COUNT) {
    probes = warp_sum(probes);
    if (lane == 0) {
      atomicAdd(&tv.ctrl->find_probes, probes);
      atomicAdd(&tv.ctrl->find_queries, (unsigned long long)len);
    }
  }
}

// Slices of whole chunks; false where a slice's places would not fit their bits.
inline bool line_find_slices(uint64_t n, int blocks, uint32_t *per_warp) {
  const uint64_t warps = (uint64_t)blocks * kLineFindWarps;
  const uint64_t per = ((n + warps - 1) / warps + 31) / 32 * 32;
  *per_warp = (uint32_t)per;
  return per <= (1u << kLineFindPlaceBits);
}

template <typename S>
inline cudaError_t launch_line_find(const TableView &tv, const uint32_t *q, uint32_t *out, uint64_t n, bool early_exit,
                                    bool count, int blocks_per_sm, cudaStream_t s) {
  auto kern = early_exit ? (count ? line_find_kernel<S, true, true> : line_find_kernel<S, true, false>)
                         : (count ? line_find_kernel<S, false, true> : line_find_kernel<S, false, false>);
  int blocks = 0;
  const cudaError_t e = grid_for(kern, n, blocks_per_sm, &blocks);
  if (e != cudaSuccess) return e;
  uint32_t per_warp = 0;
  if (!line_find_slices(n, blocks, &per_warp)) return cudaErrorInvalidValue;
  kern<<<blocks, kLineFindThreads, 0, s>>>(tv, q, out, n, per_warp);
  return cudaGetLastError();
}

}  // namespace ght
