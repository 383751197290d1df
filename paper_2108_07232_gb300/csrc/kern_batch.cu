// kern_batch.cu -- many independent BCHT tables built and queried by single
// launches (the batched form; the paper builds one table at a time).
//
// All tables live in one allocation, each with a descriptor (slots, bucket
// count, hash constants, status word). Keys, values and queries of all tables
// are concatenated; key_offs / query_offs (T+1 entries) give each table's
// range. Work is split over warps exactly as in the single-table kernels; a
// lane finds the table of the item it takes from a per-chunk hint (one
// uniform binary search per 32 items) and reads that table's descriptor.
#include <algorithm>

#include "ght_batch.h"
#include "ght_find_async.cuh"
#include "ght_find_line.cuh"
#include "ght_kernels.cuh"

namespace ght {

// First table whose range contains index i (uniform search over [lo, hi)).
__device__ __forceinline__ uint32_t table_of(const uint64_t *__restrict__ offs, uint32_t lo, uint32_t hi,
                                             uint64_t i) {
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (__ldg(offs + mid) <= i) lo = mid;
    else hi = mid;
  }
  return lo;
}

__device__ __forceinline__ uint32_t advance_table(const uint64_t *__restrict__ offs, uint32_t tb, uint32_t t_hi,
                                                  uint64_t i) {
  while (tb + 1 < t_hi && __ldg(offs + tb + 1) <= i) ++tb;
  return tb;
}

// As table_of for an index a little beyond table tb's first: steps double from tb.
__device__ __forceinline__ uint32_t seek_table(const uint64_t *__restrict__ offs, uint32_t tb, uint32_t t_hi,
                                               uint64_t i) {
  uint32_t step = 1;
  while (tb + step < t_hi && __ldg(offs + tb + step) <= i) {
    tb += step;
    step *= 2;
  }
  return table_of(offs, tb, min(tb + step, t_hi), i);
}

__device__ __forceinline__ uint32_t batch_bucket(const BatchTable &d, int i, uint32_t k) {
  return fastmod(mod_prime((uint64_t)select4(d.a, i) * k + select4(d.c, i)), d.mod);
}

// Input stream of a warp's slice with the table of each chunk's first item.
struct BatchQueue {
  uint64_t base;
  int head;
  uint32_t ta, tb, tc;  // table hint of chunks a, b, c (warp-uniform)
  uint32_t ka, kb, kc, va, vb, vc;
};

template <bool PAIRS>
__device__ __forceinline__ void bq_load(uint32_t &k, uint32_t &v, uint32_t &t, const uint32_t *__restrict__ keys,
                                        const uint32_t *__restrict__ vals, uint64_t at, uint64_t end,
                                        const BatchView &bv, const uint64_t *__restrict__ offs, int lane) {
  k = stream_load(keys, at + lane, end);
  if (PAIRS) v = stream_load(vals, at + lane, end);
  t = offs && at < end ? table_of(offs, bv.t_lo, bv.t_hi, at) : bv.t_lo;  // (an overflow list has no offsets)
}

template <bool PAIRS>
__device__ __forceinline__ uint64_t bq_take(BatchQueue &q, const uint32_t *__restrict__ keys,
                                            const uint32_t *__restrict__ vals, uint64_t end, const BatchView &bv,
                                            const uint64_t *__restrict__ offs, unsigned need, unsigned below,
                                            int lane, uint32_t &key, uint32_t &val, uint32_t &table) {
  const int pos = q.head + __popc(need & below);
  const uint32_t ka = __shfl_sync(kFull, q.ka, pos & 31), kb = __shfl_sync(kFull, q.kb, pos & 31);
  key = pos < 32 ? ka : kb;
  if (PAIRS) {
    const uint32_t va = __shfl_sync(kFull, q.va, pos & 31), vb = __shfl_sync(kFull, q.vb, pos & 31);
    val = pos < 32 ? va : vb;
  }
  const uint64_t at = q.base + (uint64_t)pos;
  table = pos < 32 ? q.ta : q.tb;
  q.head += __popc(need);
  if (q.head >= 32) {
    q.head -= 32;
    q.base += 32;
    q.ka = q.kb;
    q.kb = q.kc;
    q.va = q.vb;
    q.vb = q.vc;
    q.ta = q.tb;
    q.tb = q.tc;
    bq_load<PAIRS>(q.kc, q.vc, q.tc, keys, vals, q.base + 64, end, bv, offs, lane);
  }
  if (!((need >> lane) & 1u) || at >= end) return ~0ull;
  table = advance_table(offs, table, bv.t_hi, at);
  return at;
}

template <bool PAIRS>
__device__ __forceinline__ void bq_init(BatchQueue &q, const uint32_t *__restrict__ keys,
                                        const uint32_t *__restrict__ vals, uint64_t beg, uint64_t end,
                                        const BatchView &bv, const uint64_t *__restrict__ offs, int lane) {
  q.base = beg;
  q.head = 0;
  bq_load<PAIRS>(q.ka, q.va, q.ta, keys, vals, beg, end, bv, offs, lane);
  bq_load<PAIRS>(q.kb, q.vb, q.tb, keys, vals, beg + 32, end, bv, offs, lane);
  bq_load<PAIRS>(q.kc, q.vc, q.tc, keys, vals, beg + 64, end, bv, offs, lane);
}

// Key/value stream of the batched insert: 32-pair chunks claimed from the
// batch's work cursor (all warps stay on the few tables the cursor is in),
// each with the table of its first pair, kept two chunks ahead of use.
struct BatchClaimQueue {
  uint64_t ba, bb, bc;  // index of entry 0 of chunks a, b, c (warp-uniform)
  uint64_t claim_next;  // next chunk of the warp's current claim
  uint32_t claim_left;  // chunks left in that claim
  int head;             // next unused entry of chunk a
  uint32_t ta, tb, tc;  // table of each chunk's first pair
  uint32_t ka, kb, kc, va, vb, vc;
};

__device__ __forceinline__ void bc_init(BatchClaimQueue &q, const uint32_t *__restrict__ keys,
                                        const uint32_t *__restrict__ vals, const ClaimPlan &plan, uint64_t warp,
                                        uint64_t lo, uint64_t shared, uint64_t hi, const BatchView &bv,
                                        const uint64_t *__restrict__ offs, int lane) {
  q.claim_next = lo + warp * plan.first * 32ull;
  q.claim_left = plan.first;
  q.head = 0;
  q.ba = claim_chunk(q.claim_next, q.claim_left, plan, shared, hi, &bv.ctrl->work_cursor, lane);
  q.bb = claim_chunk(q.claim_next, q.claim_left, plan, shared, hi, &bv.ctrl->work_cursor, lane);
  q.bc = claim_chunk(q.claim_next, q.claim_left, plan, shared, hi, &bv.ctrl->work_cursor, lane);
  bq_load<true>(q.ka, q.va, q.ta, keys, vals, q.ba, hi, bv, offs, lane);
  bq_load<true>(q.kb, q.vb, q.tb, keys, vals, q.bb, hi, bv, offs, lane);
  bq_load<true>(q.kc, q.vc, q.tc, keys, vals, q.bc, hi, bv, offs, lane);
}

// Hand the next popc(need) pairs to the lanes in `need`; returns the pair's
// index (~0 for lanes without one) and its table.
__device__ __forceinline__ uint64_t bc_take(BatchClaimQueue &q, const uint32_t *__restrict__ keys,
                                            const uint32_t *__restrict__ vals, const ClaimPlan &plan, uint64_t shared,
                                            uint64_t hi, const BatchView &bv, const uint64_t *__restrict__ offs,
                                            unsigned need, unsigned below, int lane, uint32_t &key, uint32_t &val,
                                            uint32_t &table) {
  const int pos = q.head + __popc(need & below);
  const uint32_t ka = __shfl_sync(kFull, q.ka, pos & 31), kb = __shfl_sync(kFull, q.kb, pos & 31);
  const uint32_t va = __shfl_sync(kFull, q.va, pos & 31), vb = __shfl_sync(kFull, q.vb, pos & 31);
  key = pos < 32 ? ka : kb;
  val = pos < 32 ? va : vb;
  const uint64_t at = pos < 32 ? q.ba + (uint64_t)pos : q.bb + (uint64_t)(pos - 32);
  table = pos < 32 ? q.ta : q.tb;
  q.head += __popc(need);
  if (q.head >= 32) {
    q.head -= 32;
    q.ba = q.bb;
    q.bb = q.bc;
    q.bc = claim_chunk(q.claim_next, q.claim_left, plan, shared, hi, &bv.ctrl->work_cursor, lane);
    q.ka = q.kb;
    q.kb = q.kc;
    q.va = q.vb;
    q.vb = q.vc;
    q.ta = q.tb;
    q.tb = q.tc;
    bq_load<true>(q.kc, q.vc, q.tc, keys, vals, q.bc, hi, bv, offs, lane);
  }
  if (!((need >> lane) & 1u) || at >= hi) return ~0ull;
  if (offs) table = advance_table(offs, table, bv.t_hi, at);
  return at;
}

// ----------------------------------------------------------------------------
// Fill the slots of tables [t_lo, t_hi) and clear their status words.
__global__ void __launch_bounds__(256)
batch_fill_kernel(BatchView bv, uint4 *__restrict__ slots16, uint64_t n16, uint32_t *__restrict__ counters) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint4 e = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += stride) {
    slots16[i] = e;
    if (counters && (i & 7u) == 0u) counters[i >> 3] = 0u;  // one per bucket of 8 pieces
  }
  for (uint64_t t = bv.t_lo + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < bv.t_hi; t += stride)
    bv.tables[t].status = 0u;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    bv.ctrl->work_cursor = 0ull;  // the insert's claims start at zero
    bv.ctrl->reserved[0] = 0ull;  // so does the overflow list
  }
}

// ----------------------------------------------------------------------------
// Ranked first-choice placement of a batch (phase 1 of its build, as
// rank_place_kernel for one table): a key's arrival number at its bucket H_0
// comes from the bucket's counter (bl.counters, one per bucket in slot order),
// numbers below 16 are stored in that slot, the other keys go to the overflow
// list with their table. A key that no longer fits the list marks its table
// (kStatusListFull), which is then built alone, with the same constants and the
// insert of every key: the keys that crowd the list may be another table's. The
// warps take the chunks of 32
// pairs in turn, so the stores and counters in flight stay in the few tables
// that the chunks are in. Build of 512 tables of 2^10..2^20 keys at LF
// 0.8..0.99 (85 M keys): 3.75 ms with the insert of every key, 2.54 now; 64
// tables of 2^12..2^22 keys 2.05 -> 1.29; 512 of 2^10..2^14 0.39 -> 0.26.
template <bool COUNT>
__global__ void __launch_bounds__(256)
batch_place_kernel(BatchView bv, BatchPlace bl, const uint32_t *__restrict__ keys,
                   const uint32_t *__restrict__ values, uint32_t n) {
  // each warp's overflow, appended 32 keys at a time: one reservation each (a
  // reservation per key, all on one address, took longer than the placement)
  __shared__ uint32_t s_over[8][3][64];
  const uint64_t *offs = bv.key_offs;
  const int lane = threadIdx.x & 31;
  uint32_t(*over)[64] = s_over[threadIdx.x >> 5];
  const unsigned below = lanemask_lt();
  int waiting = 0;
  const uint32_t step = gridDim.x * blockDim.x;
  const uint32_t start = blockIdx.x * blockDim.x + (threadIdx.x & ~31u);
  if (start >= n) return;  // whole warp
  auto append = [&](int take) {
    unsigned long long at = 0ull;
    if (lane == 0) at = atomicAdd(&bv.ctrl->reserved[0], (unsigned long long)take);
    at = __shfl_sync(kFull, at, 0) + lane;
    waiting -= take;
    if (lane < take) {
      if (at < bl.cap) {
        bl.k[at] = over[0][waiting + lane];
        bl.v[at] = over[1][waiting + lane];
        bl.table[at] = over[2][waiting + lane];
      } else {
        atomicOr(&bv.tables[over[2][waiting + lane]].status, kStatusListFull);
      }
    }
    __syncwarp();
  };
  const uint64_t lo = __ldg(offs + bv.t_lo);
  keys += lo;
  values += lo;
  unsigned long long placed = 0;
  uint32_t first = table_of(offs, bv.t_lo, bv.t_hi, lo + start);
  uint32_t nk = start + lane < n ? __ldg(keys + start + lane) : 0u;
  uint32_t nv = start + lane < n ? __ldg(values + start + lane) : 0u;
  for (uint32_t c = start;;) {
    const uint32_t i = c + lane, k = nk, v = nv;
    const bool more = c < n - min(n, step);
    if (more) {
      nk = i + step < n ? __ldg(keys + i + step) : 0u;
      nv = i + step < n ? __ldg(values + i + step) : 0u;
    }
    bool overflows = false;
    uint32_t tb = 0;
    if (i < n) {
      tb = advance_table(offs, first, bv.t_hi, lo + i);
      if (k == kEmptyKey) {
        atomicOr(&bv.tables[tb].status, kStatusSentinel);
      } else {
        const BatchTable &d = bv.tables[tb];
        const uint32_t b = batch_bucket(d, 0, k);
        const uint64_t bucket = (uint64_t)(d.slots - bl.slots) / 16u + b;
        const uint32_t r = atomicAdd(bl.counters + bucket, 1u);
        if (COUNT) placed++;
        overflows = r >= 16u;
        if (!overflows) bl.slots[bucket * 16u + r] = ((uint64_t)v << 32) | k;
      }
    }
    const unsigned om = __ballot_sync(kFull, overflows);
    if (overflows) {
      const int x = waiting + __popc(om & below);
      over[0][x] = k;
      over[1][x] = v;
      over[2][x] = tb;
    }
    waiting += __popc(om);
    __syncwarp();
    if (waiting >= 32) append(32);
    if (!more) break;
    c += step;
    first = seek_table(offs, first, bv.t_hi, lo + c);
  }
  if (waiting > 0) append(waiting);
  if (COUNT) {
    placed = warp_sum(placed);
    if (lane == 0) atomicAdd(&bv.ctrl->insert_probes, placed);
  }
}

// ----------------------------------------------------------------------------
// BCHT bulk build of every table in [t_lo, t_hi) (Sec. III-A, V-B), with the
// turn structure, chunk claims (the batch's work cursor, zeroed by the fill),
// key-word gathers and register bound of the single-table insert kernel.
//
// LIST: the pairs are the overflow list of the batch's placement (bl), of the
// length that the control block gives; they start at H_1, H_0 being full.
template <int G, int KPL, bool COUNT, bool LIST>
__global__ void __launch_bounds__(256, insert_min_blocks<16, G, KPL, COUNT>())
batch_insert_kernel(BatchView bv, const uint32_t *__restrict__ keys, const uint32_t *__restrict__ values,
                    ClaimPlan plan, BatchPlace bl) {
  constexpr int B = 16;
  constexpr int PPL = B / G;
  static_assert(B % G == 0 && 32 % G == 0 && (KPL == 1 || KPL == 2), "tile shape");
  const uint64_t *offs = LIST ? nullptr : bv.key_offs;
  const int lane = threadIdx.x & 31;
  const int r = lane & (G - 1);
  const int tbase = lane - r;
  const unsigned tmask = (G == 32 ? kFull : ((1u << G) - 1u)) << tbase;
  const uint64_t gtid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint64_t lo = LIST ? 0ull : __ldg(offs + bv.t_lo);
  const uint64_t hi = LIST ? min(bv.ctrl->reserved[0], (unsigned long long)bl.cap) : __ldg(offs + bv.t_hi);
  if (LIST) {
    keys = bl.k;
    values = bl.v;
    plan = claim_plan(hi, (uint64_t)gridDim.x * (blockDim.x >> 5), true);
  }
  const unsigned below = lanemask_lt();
  const int h = bv.h;

  const uint64_t shared = lo + (uint64_t)gridDim.x * (blockDim.x >> 5) * plan.first * 32ull;

  uint32_t rng = lane_seed(bv.rng_seed, gtid);
  BatchClaimQueue q;
  bc_init(q, keys, values, plan, gtid >> 5, lo, shared, hi, bv, offs, lane);
  bool active[KPL], retrying[KPL];
  uint64_t pair[KPL], old[KPL];
  uint32_t cur[KPL], chain[KPL], steps[KPL], tab[KPL];
  int op[KPL];
#pragma unroll
  for (int s = 0; s < KPL; ++s) {
    active[s] = retrying[s] = false;
    pair[s] = old[s] = 0;
    cur[s] = chain[s] = steps[s] = tab[s] = 0;
    op[s] = 0;
  }
  unsigned long long probes = 0, retries = 0, evictions = 0;

  for (;;) {
#pragma unroll
    for (int s = 0; s < KPL; ++s) {
      // -- resolve the atomic this slot issued on its previous turn
      if (op[s] == 1) {
        if (old[s] == kEmptyPair) active[s] = false;
        else retrying[s] = true;
      } else if (op[s] == 2) {
        if (COUNT) evictions++;
        chain[s]++;
        if (pair_key(old[s]) == kEmptyKey) {
          active[s] = false;
        } else {
          const BatchTable &d = bv.tables[tab[s]];
          const uint32_t from = cur[s], k = pair_key(old[s]);
          pair[s] = old[s];
          int i = -1;
#pragma unroll
          for (int f = 0; f < 4; ++f)
            if (f < h && i < 0 && batch_bucket(d, f, k) == from) i = f;
          if (i < 0) {
            atomicOr(&bv.tables[tab[s]].status, kStatusCorrupt);
            active[s] = false;
          } else {
            cur[s] = batch_bucket(d, (i + 1) % h, k);
          }
        }
      }
      op[s] = 0;
      // -- refill
      const unsigned need = __ballot_sync(kFull, !active[s]);
      if (need != 0u && q.ba + q.head < hi) {
        uint32_t k, val, tb;
        const uint64_t at = bc_take(q, keys, values, plan, shared, hi, bv, offs, need, below, lane, k, val, tb);
        if (at != ~0ull) {
          if (LIST) tb = __ldg(bl.table + at);
          if (k == kEmptyKey) {
            atomicOr(&bv.tables[tb].status, kStatusSentinel);
          } else {
            pair[s] = ((uint64_t)val << 32) | k;
            tab[s] = tb;
            active[s] = true;
            retrying[s] = false;
            chain[s] = steps[s] = 0;
            cur[s] = batch_bucket(bv.tables[tb], LIST ? 1 : 0, k);
          }
        }
      }
      const unsigned act = __ballot_sync(kFull, active[s]);
      if (act == 0u) continue;
      // -- gather: each member's bucket address (its own table)
      uint64_t *myb = active[s] ? bv.tables[tab[s]].slots + (uint64_t)cur[s] * B : nullptr;
      uint32_t v[G][PPL];  // key words only: emptiness is all an insert reads
#pragma unroll
      for (int j = 0; j < G; ++j) {
        uint64_t *bj = reinterpret_cast<uint64_t *>(__shfl_sync(kFull, reinterpret_cast<uintptr_t>(myb), tbase + j));
        if ((act >> (tbase + j)) & 1u)
          load_keys_rw<PPL>(reinterpret_cast<const unsigned long long *>(bj), r, v[j]);
      }
      int my_empty = 0, my_slot = -1;
#pragma unroll
      for (int j = 0; j < G; ++j) {
        const bool aj = (act >> (tbase + j)) & 1u;
        int cnt = 0, slot = -1;
#pragma unroll
        for (int p = 0; p < PPL; ++p) {
          const unsigned em = __ballot_sync(kFull, aj && v[j][p] == kEmptyKey) & tmask;
          cnt += __popc(em);
          if (slot < 0 && em) slot = (__ffs(em) - 1 - tbase) * PPL + p;
        }
        if (lane == tbase + j) {
          my_empty = cnt;
          my_slot = slot;
        }
      }
      uint64_t *target = nullptr;
      if (active[s]) {
        if (COUNT) {
          if (retrying[s]) retries++;
          else probes++;
        }
        if (++steps[s] > bv.max_steps) {
          atomicOr(&bv.tables[tab[s]].status, kStatusTimeout);
          active[s] = false;
        } else if (my_empty > 0) {
          op[s] = 1;
          target = myb + my_slot;
        } else if (chain[s] >= bv.max_chain) {
          atomicOr(&bv.tables[tab[s]].status, kStatusBuildFailed);
          active[s] = false;
        } else {
          op[s] = 2;
          target = myb + (xorshift32(rng) % B);
        }
      }
      if (op[s] == 1) old[s] = cas_pair(target, kEmptyPair, pair[s]);
      else if (op[s] == 2) old[s] = exch_pair(target, pair[s]);
      if (op[s] != 0) retrying[s] = false;
    }
    bool any = false;
#pragma unroll
    for (int s = 0; s < KPL; ++s) any |= active[s];
    if (__ballot_sync(kFull, any) == 0u && q.ba + q.head >= hi) break;
  }
  if (COUNT) {
    probes = warp_sum(probes);
    retries = warp_sum(retries);
    evictions = warp_sum(evictions);
    if (lane == 0) {
      atomicAdd(&bv.ctrl->insert_probes, probes);
      atomicAdd(&bv.ctrl->insert_retries, retries);
      atomicAdd(&bv.ctrl->insert_evictions, evictions);
    }
  }
}

// ----------------------------------------------------------------------------
// BCHT bulk find over tables [t_lo, t_hi) (Sec. V-B find, early exit), with
// the structure of the single-table find kernel.
template <int G, int KPL, bool COUNT>
__global__ void __launch_bounds__(256)
batch_find_kernel(BatchView bv, const uint32_t *__restrict__ queries, uint32_t *__restrict__ out,
                  uint64_t per_warp) {
  constexpr int B = 16;
  constexpr int PPL = B / G;
  static_assert(B % G == 0 && 32 % G == 0 && (KPL == 1 || KPL == 2), "tile shape");
  __shared__ uint32_t s_hit[8][32], s_emp[8][32], s_val[8][32];
  const uint64_t *offs = bv.query_offs;
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const int r = lane & (G - 1);
  const int tbase = lane - r;
  const uint64_t gtid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint64_t lo = __ldg(offs + bv.t_lo), hi = __ldg(offs + bv.t_hi);
  const uint64_t beg = lo + (gtid >> 5) * per_warp;
  if (beg >= hi) return;
  const uint64_t end = beg + per_warp < hi ? beg + per_warp : hi;
  const unsigned below = lanemask_lt();

  BatchQueue q;
  bq_init<false>(q, queries, nullptr, beg, end, bv, offs, lane);
  bool active[KPL];
  uint32_t key[KPL], act[KPL], tab[KPL];
  uint64_t idx[KPL];
  int probe[KPL];
  uint64_t v[KPL][G][PPL];
#pragma unroll
  for (int s = 0; s < KPL; ++s) {
    active[s] = false;
    key[s] = kEmptyKey;
    act[s] = tab[s] = 0u;
    idx[s] = 0;
    probe[s] = 0;
  }
  unsigned long long probes = 0, answered = 0;

  for (;;) {
#pragma unroll
    for (int s = 0; s < KPL; ++s) {
      const unsigned need = __ballot_sync(kFull, !active[s]);
      if (need != 0u && q.base + q.head < end) {
        uint32_t k, unused, tb;
        const uint64_t at = bq_take<false>(q, queries, nullptr, end, bv, offs, need, below, lane, k, unused, tb);
        if (at != ~0ull) {
          if (COUNT) answered++;
          if (k == kEmptyKey) {
            out[at] = kEmptyKey;
          } else {
            active[s] = true;
            key[s] = k;
            idx[s] = at;
            tab[s] = tb;
            probe[s] = 0;
          }
        }
      }
      act[s] = __ballot_sync(kFull, active[s]);
      if (act[s] != 0u) {
        const uint64_t *myb =
            active[s] ? bv.tables[tab[s]].slots + (uint64_t)batch_bucket(bv.tables[tab[s]], probe[s], key[s]) * B
                      : nullptr;
#pragma unroll
        for (int j = 0; j < G; ++j) {
          const uint64_t *bj =
              reinterpret_cast<const uint64_t *>(__shfl_sync(kFull, reinterpret_cast<uintptr_t>(myb), tbase + j));
          if ((act[s] >> (tbase + j)) & 1u) load_part_ro<PPL>(bj, r, v[s][j]);
        }
      }
      const int e = (KPL == 1) ? s : (s + 1) % KPL;
      if (act[e] != 0u) {
        s_hit[wib][lane] = 0u;
        s_emp[wib][lane] = 0u;
        __syncwarp();
#pragma unroll
        for (int j = 0; j < G; ++j) {
          const int owner = tbase + j;
          const uint32_t kj = __shfl_sync(kFull, key[e], owner);
          if ((act[e] >> owner) & 1u) {
#pragma unroll
            for (int p = 0; p < PPL; ++p) {
              const uint32_t sk = pair_key(v[e][j][p]);
              if (sk == kj) {
                s_hit[wib][owner] = 1u;
                s_val[wib][owner] = pair_value(v[e][j][p]);
              }
              if (sk == kEmptyKey) s_emp[wib][owner] = 1u;
            }
          }
        }
        __syncwarp();
        if ((act[e] >> lane) & 1u) {
          if (COUNT) probes++;
          bool finish = false;
          uint32_t result = kEmptyKey;
          if (s_hit[wib][lane]) {
            result = s_val[wib][lane];
            finish = true;
          } else if (s_emp[wib][lane] || ++probe[e] >= bv.h) {
            finish = true;
          }
          if (finish) {
            out[idx[e]] = result;
            active[e] = false;
          }
        }
        act[e] = 0u;
      }
    }
    bool any = false;
#pragma unroll
    for (int s = 0; s < KPL; ++s) any |= active[s];
    if (__ballot_sync(kFull, any) == 0u && q.base + q.head >= end) break;
  }
  if (COUNT) {
    probes = warp_sum(probes);
    answered = warp_sum(answered);
    if (lane == 0) {
      atomicAdd(&bv.ctrl->find_probes, probes);
      atomicAdd(&bv.ctrl->find_queries, answered);
    }
  }
}

// ----------------------------------------------------------------------------
constexpr int kBatchTableBits = 30;  // a waiting query's table, below its next probe (h <= 4)

// The same find with 32-byte loads (the line find, ght_find_line.cuh): 32
// queries per step, those that need another bucket wait in shared memory with
// their table. A step's queries are consecutive, so their tables are found by
// walking on from the last step's first table, and the descriptors come from
// L1.
//
// The warps take the chunks of 32 queries in turn, so that all of them are in
// the same few tables, whose lines then stay in the L2; a slice of the batch
// per warp, as the register find has, keeps every table in use at once (and
// the reads in DRAM). Find of 512 tables of 2^10..2^20 keys (85 M keys, 171 M
// queries, half present): 13.5 ms (register find, two queries per lane; one:
// 11.2) -> 2.5 ms; 64 tables of 2^12..2^22 keys (87 M queries) 6.5 -> 1.3 ms;
// 512 tables of 2^10..2^14 keys (6 M queries, all in the L2) 0.30 -> 0.12 ms.
//
// SEG: segment t's queries are read from bv.src[t] and its answers go to
// bv.dst[t] (the requests of a pool, each with arrays of its own), instead of
// one array each; `queries` and `out` are not used. A burst of 128 requests
// (9.6 M queries, 32 tables of 2^16..2^22 keys), submit to last answer: 1040 us
// with the register find between a gather and a scatter, 534 us now (most of
// it the host's submits and waits).
template <bool COUNT, bool SEG>
__global__ void __launch_bounds__(kLineFindThreads, 4)
batch_line_find_kernel(BatchView bv, const uint32_t *__restrict__ queries, uint32_t *__restrict__ out,
                       uint32_t n) {
  __shared__ uint2 s_wait[kLineFindWarps][kLineFindWaiting];
  __shared__ uint32_t s_table[kLineFindWarps][kLineFindWaiting];
  const uint64_t *offs = bv.query_offs;
  const int lane = threadIdx.x & 31;
  const int r = lane & (kLineFindLanes - 1);
  const int tbase = lane - r;
  const unsigned below = lanemask_lt();
  uint2 *wait = s_wait[threadIdx.x >> 5];
  uint32_t *wait_table = s_table[threadIdx.x >> 5];
  const uint32_t step = gridDim.x * kLineFindThreads;
  const uint32_t start = blockIdx.x * kLineFindThreads + (threadIdx.x & ~31u);
  if (start >= n) return;  // whole warp
  const uint64_t lo = __ldg(offs + bv.t_lo);
  queries += SEG ? 0 : lo;
  out += SEG ? 0 : lo;
  auto query = [&](uint32_t i, uint32_t t) {
    // (a request may be answered in place: each query is read once, before its answer is written)
    if constexpr (SEG) return bv.src[t][lo + i - __ldg(offs + t)];
    else return __ldg(queries + i);
  };
  auto answer = [&](uint32_t i, uint32_t t, uint32_t v) {
    if constexpr (SEG) bv.dst[t][lo + i - __ldg(offs + t)] = v;
    else out[i] = v;
  };
  int waiting = 0;
  unsigned long long probes = 0, answered = 0;
  // the next step's queries and their tables
  uint32_t first = table_of(offs, bv.t_lo, bv.t_hi, lo + start);
  uint32_t next_table = advance_table(offs, first, bv.t_hi, lo + min(start + lane, n - 1u));
  uint32_t next = query(min(start + lane, n - 1u), next_table);
  for (uint32_t c = start;;) {
    uint32_t k, at, tb;
    int probe;
    bool valid;
    if (waiting >= 32 || c >= n) {
      if (waiting == 0) break;
      const int take = min(waiting, 32);
      waiting -= take;
      const uint2 e = wait[waiting + min(lane, take - 1)];
      const uint32_t tp = wait_table[waiting + min(lane, take - 1)];
      k = e.x;
      at = e.y;
      tb = tp & ((1u << kBatchTableBits) - 1u);
      probe = (int)(tp >> kBatchTableBits);
      valid = lane < take;
      __syncwarp();  // read before the step's own entries go there
    } else {
      k = next;
      at = c + lane;
      probe = 0;
      tb = next_table;
      if (c < n - min(n, step)) {
        c += step;
        const uint32_t i = min(c + lane, n - 1u);
        first = seek_table(offs, first, bv.t_hi, lo + c);
        next_table = advance_table(offs, first, bv.t_hi, lo + i);
        next = query(i, next_table);
      } else {
        c = n;
      }
      valid = at < n && k != kEmptyKey;
      if (COUNT && at < n) answered++;
      if (at < n && k == kEmptyKey) answer(at, tb, kEmptyKey);  // the sentinel is never a key
    }
    const BatchTable &d = bv.tables[tb];
    FastMod mod;
    mod.M = __ldg(reinterpret_cast<const unsigned long long *>(&d.mod.M));
    mod.d = __ldg(&d.mod.d);
    const uint32_t b = fastmod(mod_prime((uint64_t)__ldg(&d.a[probe]) * k + __ldg(&d.c[probe])), mod);
    const uint64_t bucket =
        __ldg(reinterpret_cast<const unsigned long long *>(&d.slots)) + (uint64_t)b * (16u * sizeof(uint64_t));
    bool hit, empty;
    uint32_t value;
    line_probe<PairSlot, true>(
        k, r, tbase, lane,
        [&](int j, uint32_t(&x)[8]) {
          load32_ro(reinterpret_cast<const char *>(__shfl_sync(kFull, bucket, tbase + j)) + r * 32, x);
        },
        hit, empty, value);
    if (COUNT && valid) probes++;
    const bool more = valid && !hit && !empty && probe + 1 < bv.h;
    if (valid && !more) answer(at, tb, hit ? value : kEmptyKey);
    const unsigned mb = __ballot_sync(kFull, more);
    if (more) {
      const int i = waiting + __popc(mb & below);
      wait[i] = make_uint2(k, at);
      wait_table[i] = tb | ((uint32_t)(probe + 1) << kBatchTableBits);
    }
    waiting += __popc(mb);
    __syncwarp();
  }
  if (COUNT) {
    probes = warp_sum(probes);
    answered = warp_sum(answered);
    if (lane == 0) {
      atomicAdd(&bv.ctrl->find_probes, probes);
      atomicAdd(&bv.ctrl->find_queries, answered);
    }
  }
}

// ----------------------------------------------------------------------------
// The same find with the bucket parts staged in shared memory (the staged
// find of the single-table path, ght_find_async.cuh): 4-lane tiles, KPL
// query sets per lane in flight, each set's buckets copied by cp.async (two
// 16-byte chunks per lane and tile member, chunk positions swizzled by tile)
// and evaluated KPL - 1 steps after its copies were issued. A query's table
// comes with it from the batch queue; its bucket address from the table's
// descriptor. The tables of a batch are each small but are queried all at
// once, so together their slots exceed the L2 and the reads go to DRAM,
// where the deeper pipeline pays.
template <int KPL, int WARPS, bool COUNT>
__global__ void __launch_bounds__(32 * WARPS)
batch_find_async_kernel(BatchView bv, const uint32_t *__restrict__ queries, uint32_t *__restrict__ out,
                        uint64_t per_warp) {
  constexpr int G = 4;
  constexpr int kChunks = 8;  // 16-byte chunks per 16-pair bucket
  extern __shared__ uint4 bfa_smem[];
  const uint64_t *offs = bv.query_offs;
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const int r = lane & (G - 1);
  const int tbase = lane - r;
  const unsigned swz = (unsigned)(lane >> 2) & 7u;
  const unsigned tmask = ((1u << G) - 1u) << tbase;
  uint4 *wbuf = bfa_smem + (size_t)wib * KPL * 32 * kChunks;
  const uint64_t gtid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint64_t lo = __ldg(offs + bv.t_lo), hi = __ldg(offs + bv.t_hi);
  const uint64_t beg = lo + (gtid >> 5) * per_warp;
  if (beg >= hi) return;  // whole warp
  const uint64_t end = beg + per_warp < hi ? beg + per_warp : hi;
  const unsigned below = lanemask_lt();

  BatchQueue q;
  bq_init<false>(q, queries, nullptr, beg, end, bv, offs, lane);
  bool active[KPL];
  uint32_t key[KPL], act[KPL], tab[KPL];
  uint64_t idx[KPL];
  int probe[KPL];
#pragma unroll
  for (int s = 0; s < KPL; ++s) {
    active[s] = false;
    key[s] = kEmptyKey;
    act[s] = tab[s] = 0u;
    idx[s] = 0;
    probe[s] = 0;
  }
  unsigned long long probes = 0, answered = 0;

  for (;;) {
#pragma unroll
    for (int s = 0; s < KPL; ++s) {
      // -- refill set s from the stream, then issue the copies of its buckets
      const unsigned need = __ballot_sync(kFull, !active[s]);
      if (need != 0u && q.base + q.head < end) {
        uint32_t k, unused, tb;
        const uint64_t at = bq_take<false>(q, queries, nullptr, end, bv, offs, need, below, lane, k, unused, tb);
        if (at != ~0ull) {
          if (COUNT) answered++;
          if (k == kEmptyKey) {
            out[at] = kEmptyKey;  // the sentinel is never a key
          } else {
            active[s] = true;
            key[s] = k;
            idx[s] = at;
            tab[s] = tb;
            probe[s] = 0;
          }
        }
      }
      act[s] = __ballot_sync(kFull, active[s]);
      if (act[s] != 0u) {
        const uint4 *myb = nullptr;
        if (active[s]) {
          const BatchTable &d = bv.tables[tab[s]];
          myb = reinterpret_cast<const uint4 *>(d.slots) + (uint64_t)batch_bucket(d, probe[s], key[s]) * kChunks;
        }
        uint4 *sbuf = wbuf + (size_t)s * 32 * kChunks;
#pragma unroll
        for (int j = 0; j < G; ++j) {
          const int owner = tbase + j;
          const uint4 *src =
              reinterpret_cast<const uint4 *>(__shfl_sync(kFull, reinterpret_cast<uintptr_t>(myb), owner));
          if ((act[s] >> owner) & 1u) {
            uint4 *row = sbuf + owner * kChunks;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const unsigned c = 2u * (unsigned)r + (unsigned)i;
              cp_async16(row + (c ^ swz), src + c);
            }
          }
        }
      }
      cp_async_commit();  // one group per set step, empty or not
      // -- evaluate the set issued KPL - 1 steps ago
      const int e = (s + 1) % KPL;
      cp_async_wait<KPL - 1>();
      __syncwarp();
      if (act[e] != 0u) {
        const uint4 *ebuf = wbuf + (size_t)e * 32 * kChunks;
        bool my_hit = false, my_emp = false;
        uint32_t my_val = kEmptyKey;
#pragma unroll
        for (int j = 0; j < G; ++j) {
          const int owner = tbase + j;
          const uint32_t kj = __shfl_sync(kFull, key[e], owner);
          bool hit = false, emp = false;
          uint32_t hv = 0u;
          if ((act[e] >> owner) & 1u) {
            const uint4 *row = ebuf + owner * kChunks;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const uint4 c = row[(2u * (unsigned)r + (unsigned)i) ^ swz];  // pairs (c.x, c.y), (c.z, c.w)
              if (c.x == kj) {
                hit = true;
                hv = c.y;
              }
              if (c.z == kj) {
                hit = true;
                hv = c.w;
              }
              emp |= c.x == kEmptyKey || c.z == kEmptyKey;
            }
          }
          const unsigned hb = __ballot_sync(kFull, hit) & tmask;
          const unsigned eb = __ballot_sync(kFull, emp) & tmask;
          const uint32_t val = __shfl_sync(kFull, hv, hb ? __ffs(hb) - 1 : lane);
          if (lane == owner) {
            my_hit = hb != 0u;
            my_emp = eb != 0u;
            my_val = val;
          }
        }
        if ((act[e] >> lane) & 1u) {
          if (COUNT) probes++;
          bool finish = false;
          uint32_t result = kEmptyKey;
          if (my_hit) {
            result = my_val;
            finish = true;
          } else if (my_emp || ++probe[e] >= bv.h) {  // BCHT: early exit at a bucket with an empty slot
            finish = true;
          }
          if (finish) {
            out[idx[e]] = result;
            active[e] = false;
          }
        }
        act[e] = 0u;
      }
      __syncwarp();  // set e's buffer is read before the next step reuses it
    }
    bool any = false;
#pragma unroll
    for (int s = 0; s < KPL; ++s) any |= active[s];
    if (__ballot_sync(kFull, any) == 0u && q.base + q.head >= end) break;
  }
  cp_async_wait<0>();
  if (COUNT) {
    probes = warp_sum(probes);
    answered = warp_sum(answered);
    if (lane == 0) {
      atomicAdd(&bv.ctrl->find_probes, probes);
      atomicAdd(&bv.ctrl->find_queries, answered);
    }
  }
}

// ----------------------------------------------------------------------------
template <typename K>
static cudaError_t launch_sliced(K kern, uint64_t items, int blocks_per_sm, cudaStream_t s, int *blocks,
                                 uint64_t *per_warp) {
  cudaError_t e = grid_for(kern, items, blocks_per_sm, blocks);
  if (e != cudaSuccess) return e;
  *per_warp = per_warp_of(items, *blocks);
  return cudaSuccess;
}

cudaError_t launch_batch_fill(const BatchView &bv, uint64_t *slots, uint64_t num_slots, uint32_t *counters,
                              cudaStream_t s) {
  const uint64_t n16 = num_slots / 2;  // every table's slot count is even (b = 16)
  int blocks = 0;
  cudaError_t e = grid_for(batch_fill_kernel, n16 > 0 ? n16 : 1, 0, &blocks);
  if (e != cudaSuccess) return e;
  batch_fill_kernel<<<blocks, kThreads, 0, s>>>(bv, reinterpret_cast<uint4 *>(slots), n16, counters);
  return cudaGetLastError();
}

template <int G, int KPL>
static cudaError_t insert_cfg(const BatchView &bv, const uint32_t *k, const uint32_t *v, uint64_t items,
                              const LaunchOpts &o, cudaStream_t s) {
  auto kern = o.count ? batch_insert_kernel<G, KPL, true, false> : batch_insert_kernel<G, KPL, false, false>;
  int blocks = 0;
  cudaError_t e = grid_for(kern, items, o.blocks_per_sm, &blocks);
  if (e != cudaSuccess) return e;
  kern<<<blocks, kThreads, 0, s>>>(bv, k, v, claim_plan(items, (uint64_t)blocks * (kThreads / 32), true),
                                   BatchPlace());  // the fill zeroed the claim cursor
  return cudaGetLastError();
}

template <int G, int KPL>
static cudaError_t find_cfg(const BatchView &bv, const uint32_t *q, uint32_t *out, uint64_t items,
                            const LaunchOpts &o, cudaStream_t s) {
  auto kern = o.count ? batch_find_kernel<G, KPL, true> : batch_find_kernel<G, KPL, false>;
  int blocks = 0;
  uint64_t pw = 0;
  cudaError_t e = launch_sliced(kern, items, o.blocks_per_sm, s, &blocks, &pw);
  if (e != cudaSuccess) return e;
  kern<<<blocks, kThreads, 0, s>>>(bv, q, out, pw);
  return cudaGetLastError();
}

__device__ __forceinline__ uint32_t segment_of(const uint64_t *__restrict__ offs, uint32_t segs, uint64_t i) {
  uint32_t lo = 0, hi = segs;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (__ldg(offs + mid) <= i) lo = mid;
    else hi = mid;
  }
  return lo;
}

__global__ void __launch_bounds__(256)
segment_gather_kernel(const uint32_t *const *__restrict__ src, const uint64_t *__restrict__ offs, uint32_t segs,
                      uint32_t *__restrict__ dst, uint64_t n) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const uint32_t sg = segment_of(offs, segs, i);
    dst[i] = __ldg(src[sg] + (i - __ldg(offs + sg)));
  }
}

__global__ void __launch_bounds__(256)
segment_scatter_kernel(const uint32_t *__restrict__ src, uint32_t *const *__restrict__ dst,
                       const uint64_t *__restrict__ offs, uint32_t segs, uint64_t n) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const uint32_t sg = segment_of(offs, segs, i);
    dst[sg][i - __ldg(offs + sg)] = src[i];
  }
}

cudaError_t launch_segment_gather(const uint32_t *const *src, const uint64_t *offs, uint32_t segs, uint32_t *dst,
                                  uint64_t n, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  int blocks = 0;
  cudaError_t e = grid_for(segment_gather_kernel, n, 0, &blocks);
  if (e != cudaSuccess) return e;
  segment_gather_kernel<<<blocks, kThreads, 0, s>>>(src, offs, segs, dst, n);
  return cudaGetLastError();
}

cudaError_t launch_segment_scatter(const uint32_t *src, uint32_t *const *dst, const uint64_t *offs, uint32_t segs,
                                   uint64_t n, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  int blocks = 0;
  cudaError_t e = grid_for(segment_scatter_kernel, n, 0, &blocks);
  if (e != cudaSuccess) return e;
  segment_scatter_kernel<<<blocks, kThreads, 0, s>>>(src, dst, offs, segs, n);
  return cudaGetLastError();
}

bool batch_shape_supported(int G, int kpl) {
  return (G == 4 || G == 8 || G == 16) && (kpl == 1 || kpl == 2);
}

bool batch_find_shape_supported(int G, int kpl) { return batch_shape_supported(G, kpl) || (G == 4 && kpl == 6); }

void batch_find_shape(const ght_config *cfg, LaunchOpts *o) {
  o->tile_lanes = cfg && cfg->tile_lanes ? cfg->tile_lanes : 4;
  o->keys_per_lane = cfg && cfg->keys_per_lane ? cfg->keys_per_lane : 2;
  o->line_find = o->tile_lanes == 4 && o->keys_per_lane == 2 && !(cfg && cfg->find_async < 0);
}

// staged find: 6 query sets per lane, 2-warp blocks (24 KB of shared memory per warp)
static cudaError_t find_staged(const BatchView &bv, const uint32_t *q, uint32_t *out, uint64_t items,
                               const LaunchOpts &o, cudaStream_t s) {
  constexpr int kKpl = 6, kWarps = 2;
  auto kern = o.count ? batch_find_async_kernel<kKpl, kWarps, true> : batch_find_async_kernel<kKpl, kWarps, false>;
  const size_t smem = kWarps * find_async_smem_per_warp<kKpl>();
  int blocks = 0;
  cudaError_t e = grid_for_smem(kern, 32 * kWarps, smem, items, o.blocks_per_sm, &blocks);
  if (e != cudaSuccess) return e;
  const uint64_t warps = (uint64_t)blocks * kWarps;
  kern<<<blocks, 32 * kWarps, smem, s>>>(bv, q, out, (items + warps - 1) / warps);
  return cudaGetLastError();
}

static cudaError_t find_lines(const BatchView &bv, const uint32_t *q, uint32_t *out, uint64_t items,
                              const LaunchOpts &o, cudaStream_t s) {
  if (items > kLineFindMost) return find_cfg<4, 2>(bv, q, out, items, o, s);  // 32-bit places
  auto kern = bv.src    ? (o.count ? batch_line_find_kernel<true, true> : batch_line_find_kernel<false, true>)
              : o.count ? batch_line_find_kernel<true, false>
                        : batch_line_find_kernel<false, false>;
  int blocks = 0;
  const cudaError_t e = grid_for(kern, items, o.blocks_per_sm, &blocks);
  if (e != cudaSuccess) return e;
  kern<<<blocks, kLineFindThreads, 0, s>>>(bv, q, out, (uint32_t)items);
  return cudaGetLastError();
}

cudaError_t launch_batch_insert(const BatchView &bv, const uint32_t *k, const uint32_t *v, uint64_t items,
                                const LaunchOpts &o, cudaStream_t s) {
  if (items == 0) return cudaSuccess;
  const int g = o.tile_lanes, kpl = o.keys_per_lane;
  if (g == 16) return kpl == 1 ? insert_cfg<16, 1>(bv, k, v, items, o, s) : insert_cfg<16, 2>(bv, k, v, items, o, s);
  if (g == 8) return kpl == 1 ? insert_cfg<8, 1>(bv, k, v, items, o, s) : insert_cfg<8, 2>(bv, k, v, items, o, s);
  if (g == 4) return kpl == 1 ? insert_cfg<4, 1>(bv, k, v, items, o, s) : insert_cfg<4, 2>(bv, k, v, items, o, s);
  return cudaErrorInvalidValue;
}

cudaError_t launch_batch_place(const BatchView &bv, const BatchPlace &bl, const uint32_t *k, const uint32_t *v,
                               uint64_t items, const LaunchOpts &o, cudaStream_t s) {
  if (items == 0) return cudaSuccess;
  if (items > 0xFFFF0000ull) return cudaErrorInvalidValue;  // 32-bit places
  int blocks = 0;
  auto place = o.count ? batch_place_kernel<true> : batch_place_kernel<false>;
  cudaError_t e = grid_for(place, items, 0, &blocks);
  if (e != cudaSuccess) return e;
  place<<<blocks, kThreads, 0, s>>>(bv, bl, k, v, (uint32_t)items);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  auto insert = o.count ? batch_insert_kernel<16, 1, true, true> : batch_insert_kernel<16, 1, false, true>;
  if ((e = grid_for(insert, std::min<uint64_t>(items, bl.cap), o.blocks_per_sm, &blocks)) != cudaSuccess) return e;
  insert<<<blocks, kThreads, 0, s>>>(bv, nullptr, nullptr, ClaimPlan(), bl);
  return cudaGetLastError();
}

cudaError_t launch_batch_find(const BatchView &bv, const uint32_t *q, uint32_t *out, uint64_t items,
                              const LaunchOpts &o, cudaStream_t s) {
  if (items == 0) return cudaSuccess;
  const int g = o.tile_lanes, kpl = o.keys_per_lane;
  if (bv.src && !(o.line_find && items <= kLineFindMost)) return cudaErrorInvalidValue;
  if (o.line_find) return find_lines(bv, q, out, items, o, s);
  if (g == 16) return kpl == 1 ? find_cfg<16, 1>(bv, q, out, items, o, s) : find_cfg<16, 2>(bv, q, out, items, o, s);
  if (g == 8) return kpl == 1 ? find_cfg<8, 1>(bv, q, out, items, o, s) : find_cfg<8, 2>(bv, q, out, items, o, s);
  if (g == 4 && kpl == 6) return find_staged(bv, q, out, items, o, s);
  if (g == 4) return kpl == 1 ? find_cfg<4, 1>(bv, q, out, items, o, s) : find_cfg<4, 2>(bv, q, out, items, o, s);
  return cudaErrorInvalidValue;
}

}  // namespace ght
