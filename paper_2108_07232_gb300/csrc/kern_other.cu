// kern_other.cu -- instantiations and launchers of the P2BHT, IHT,
// load-balanced BCHT and bucket-size-one cuckoo kernels, plus fill and hash.
#include "ght_internal.h"
#include "ght_kernels.cuh"

namespace ght {

// ----------------------------------------------------------------------------
// Fill (Sec. III-A: initialise all buckets to empty) and reset the control
// block. slots16 covers the 16-byte aligned body; tail8 the last odd pair.
__global__ void fill_kernel(uint4 *__restrict__ slots16, uint64_t n16, uint64_t *__restrict__ tail8,
                            Ctrl *__restrict__ ctrl, uint32_t *__restrict__ counters, uint64_t m) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint4 e = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += stride)
    slots16[i] = e;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) counters[i] = 0u;
  if (blockIdx.x == 0) {
    if (threadIdx.x == 0 && tail8) *tail8 = kEmptyPair;
    if (threadIdx.x < sizeof(Ctrl) / 8) reinterpret_cast<unsigned long long *>(ctrl)[threadIdx.x] = 0ull;
  }
}

__global__ void __launch_bounds__(32)
publish_kernel(const Ctrl *__restrict__ ctrl, PublishedCtrl *__restrict__ host, unsigned long long number) {
  publish_ctrl(ctrl, host, number, (int)threadIdx.x);
}

cudaError_t launch_publish(const Ctrl *ctrl, PublishedCtrl *host, unsigned long long number, cudaStream_t s) {
  publish_kernel<<<1, 32, 0, s>>>(ctrl, host, number);
  return cudaGetLastError();
}

// Bucket indices under each hash function (diagnostic; out is n x h).
__global__ void hash_kernel(TableView tv, const uint32_t *__restrict__ keys, uint32_t *__restrict__ out,
                            uint64_t n) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const uint32_t k = keys[i];
    for (int f = 0; f < tv.h; ++f) out[i * tv.h + f] = bucket_of(tv.hf, f, k);
  }
}

// ----------------------------------------------------------------------------
// Placement by load, for the schemes that put a key into the least loaded of
// its candidates (ties to the lowest hash index): P2BHT (two, Sec. III-B) and
// the load-balanced BCHT (h, Sec. III-A last paragraph).
//
// A bucket's load is its count of arrivals, 4 bytes that stay in L2, instead
// of 128 bytes of bucket: a key reads its candidates' counts, adds one to the
// least by a CAS, and stores its pair in the slot of the old count. The CAS
// fails when the bucket has grown since, and the key looks again: so the
// choices are as balanced as those of the insert, whose CAS into the first
// empty slot fails in the same case. (With a plain add, keys in flight choose
// by old counts, and P2BHT at LF 0.8 failed on tables of up to 2^20 keys.)
// P2BHT fails when all candidates are full; the load-balanced BCHT's keys then
// go to the overflow list, whose insert evicts (Sec. III-A takes the keys in any
// order, so also in this one).
//
// The insert that reads the buckets is bound by its random lines (two or three
// 128-byte reads and a CAS per key); this by the L2's atomics and scattered
// stores. Insert -> placement, us: P2BHT 2^20 keys LF 0.8 120 -> 60, 2^24 1095 ->
// 570, 2^26 4830 -> 2790; load-balanced BCHT 2^22 LF 0.95 424 -> 201 with the
// overflow's insert, 2^24 LF 0.9 1617 -> 644.
template <bool COUNT>
__global__ void __launch_bounds__(256)
load_place_kernel(TableView tv, int B, const uint32_t *__restrict__ keys, const uint32_t *__restrict__ values,
                  uint64_t n, uint32_t *__restrict__ counters, uint32_t *__restrict__ ovf_k,
                  uint32_t *__restrict__ ovf_v, uint64_t cap) {
  constexpr int kPer = 2;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const int h = tv.h;
  unsigned long long probes = 0, retries = 0;
  for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += stride * kPer) {
    uint32_t k[kPer], v[kPer], b[kPer], c[kPer];
    bool open[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const uint64_t i = i0 + u * stride;
      open[u] = i < n;
      k[u] = open[u] ? __ldg(keys + i) : kEmptyKey;
      v[u] = open[u] ? __ldg(values + i) : 0u;
      if (open[u] && k[u] == kEmptyKey) {
        atomicOr(&tv.ctrl->status, kStatusSentinel);
        open[u] = false;
      }
    }
    bool first = true;
    for (uint32_t steps = h;; steps += h) {  // bucket visits of a key, as the inserts count them
      bool any = false;
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        c[u] = 0xFFFFFFFFu;
        any |= open[u];
        if (!open[u]) continue;
        if (COUNT) (first ? probes : retries) += h;
        uint32_t bf[4], cf[4];
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          if (f >= h) continue;
          bf[f] = bucket_of(tv.hf, f, k[u]);
          asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(cf[f]) : "l"(counters + bf[f]) : "memory");
        }
#pragma unroll
        for (int f = 0; f < 4; ++f)
          if (f < h && cf[f] < c[u]) {
            c[u] = cf[f];
            b[u] = bf[f];
          }
      }
      if (!any) break;
      if (steps > tv.max_steps) {
        atomicOr(&tv.ctrl->status, kStatusTimeout);
        break;
      }
      uint32_t was[kPer];
#pragma unroll
      for (int u = 0; u < kPer; ++u)
        if (open[u] && c[u] < (uint32_t)B) was[u] = atomicCAS(counters + b[u], c[u], c[u] + 1u);
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        if (!open[u]) continue;
        if (c[u] < (uint32_t)B) {
          if (was[u] == c[u]) {
            tv.slots[(uint64_t)b[u] * B + c[u]] = PairSlot::make(k[u], v[u]);
            open[u] = false;
          }
        } else {  // every candidate is full
          open[u] = false;
          if (ovf_k) {
            if (COUNT) (first ? probes : retries) -= h;  // the overflow's insert reads them
            const unsigned long long at = atomicAdd(&tv.ctrl->reserved[0], 1ull);
            if (at < cap) {
              ovf_k[at] = k[u];
              ovf_v[at] = v[u];
            }
          } else {
            atomicOr(&tv.ctrl->status, kStatusBuildFailed);
          }
        }
      }
      first = false;
    }
    if ((load_status(tv.ctrl) & (kStatusBuildFailed | kStatusTimeout)) != 0u) break;
  }
  if (COUNT) {
    probes = warp_sum(probes);
    retries = warp_sum(retries);
    if ((threadIdx.x & 31) == 0) {
      atomicAdd(&tv.ctrl->insert_probes, probes);
      atomicAdd(&tv.ctrl->insert_retries, retries);
    }
  }
}

cudaError_t launch_place_by_load(int B, const TableView &tv, const uint32_t *k, const uint32_t *v, uint64_t n,
                                 const PlaceBuffers &pb, bool evicts, bool count, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  auto kern = count ? load_place_kernel<true> : load_place_kernel<false>;
  int blocks = 0;
  const cudaError_t e = grid_for(kern, (n + 1) / 2, 0, &blocks);
  if (e != cudaSuccess) return e;
  kern<<<blocks, kThreads, 0, s>>>(tv, B, k, v, n, pb.counters, evicts ? pb.ovf_k : nullptr,
                                   evicts ? pb.ovf_v : nullptr, pb.cap);
  return cudaGetLastError();
}

template <int S, int B, int G, int KPL>
static cudaError_t insert_kpl(const TableView &tv, const uint32_t *k, const uint32_t *v,
                              uint64_t n, const LaunchOpts &o, cudaStream_t s) {
  auto kern = o.count ? bucketed_insert_kernel<S, B, G, KPL, true> : bucketed_insert_kernel<S, B, G, KPL, false>;
  int blocks = 0;
  cudaError_t e = grid_for(kern, n, o.blocks_per_sm, &blocks);
  if (e != cudaSuccess) return e;
  kern<<<blocks, kThreads, 0, s>>>(tv, k, v, n, o.ordered, o.overflow);
  return cudaGetLastError();
}

template <int S, int B, int G>
static cudaError_t insert_shape(const TableView &tv, const uint32_t *k, const uint32_t *v,
                                uint64_t n, const LaunchOpts &o, cudaStream_t s) {
  return o.keys_per_lane == 1 ? insert_kpl<S, B, G, 1>(tv, k, v, n, o, s) : insert_kpl<S, B, G, 2>(tv, k, v, n, o, s);
}

template <int S, int B, int G, int KPL>
static cudaError_t find_kpl(const TableView &tv, const uint32_t *q, uint32_t *out, uint64_t n,
                            const LaunchOpts &o, cudaStream_t s) {
  auto kern = o.count ? bucketed_find_kernel<S, B, G, KPL, true> : bucketed_find_kernel<S, B, G, KPL, false>;
  int blocks = 0;
  cudaError_t e = grid_for(kern, n, o.blocks_per_sm, &blocks);
  if (e != cudaSuccess) return e;
  kern<<<blocks, kThreads, 0, s>>>(tv, q, out, n, per_warp_of(n, blocks));
  return cudaGetLastError();
}

template <int S, int B, int G>
static cudaError_t find_shape(const TableView &tv, const uint32_t *q, uint32_t *out, uint64_t n,
                              const LaunchOpts &o, cudaStream_t s) {
  return o.keys_per_lane == 1 ? find_kpl<S, B, G, 1>(tv, q, out, n, o, s) : find_kpl<S, B, G, 2>(tv, q, out, n, o, s);
}

bool other_shape_supported(int scheme, int B, int G) {
  if (scheme == kCuckoo1) return B == 1;
  if (scheme == kP2BHT || scheme == kIHT || scheme == kBCHT_LB) return (B == 16 || B == 32) && G == 8;
  return false;
}

#define GHT_DISPATCH_BUCKETED(FN, ...)                                              \
  switch (scheme) {                                                                 \
    case kP2BHT: return B == 16 ? FN<kP2BHT, 16, 8>(__VA_ARGS__) : FN<kP2BHT, 32, 8>(__VA_ARGS__); \
    case kIHT: return B == 16 ? FN<kIHT, 16, 8>(__VA_ARGS__) : FN<kIHT, 32, 8>(__VA_ARGS__);       \
    case kBCHT_LB: return B == 16 ? FN<kBCHT_LB, 16, 8>(__VA_ARGS__) : FN<kBCHT_LB, 32, 8>(__VA_ARGS__); \
    default: return cudaErrorInvalidValue;                                          \
  }

cudaError_t launch_insert_other(int scheme, int B, const TableView &tv, const uint32_t *k,
                                const uint32_t *v, uint64_t n, const LaunchOpts &o, cudaStream_t s) {
  if (scheme == kCuckoo1) {
    auto kern = o.count ? cuckoo1_insert_kernel<true> : cuckoo1_insert_kernel<false>;
    int blocks = 0;
    cudaError_t e = grid_for(kern, n, o.blocks_per_sm, &blocks);
    if (e != cudaSuccess) return e;
    kern<<<blocks, kThreads, 0, s>>>(tv, k, v, n, o.overflow);
    return cudaGetLastError();
  }
  if (!other_shape_supported(scheme, B, o.tile_lanes)) return cudaErrorInvalidValue;
  GHT_DISPATCH_BUCKETED(insert_shape, tv, k, v, n, o, s)
}

cudaError_t launch_find_other(int scheme, int B, const TableView &tv, const uint32_t *q,
                              uint32_t *out, uint64_t n, const LaunchOpts &o, cudaStream_t s) {
  if (scheme == kCuckoo1) {
    auto kern = o.count ? cuckoo1_find_kernel<true> : cuckoo1_find_kernel<false>;
    int blocks = 0;
    cudaError_t e = grid_for(kern, n, o.blocks_per_sm, &blocks);
    if (e != cudaSuccess) return e;
    kern<<<blocks, kThreads, 0, s>>>(tv, q, out, n);
    return cudaGetLastError();
  }
  if (!other_shape_supported(scheme, B, o.tile_lanes)) return cudaErrorInvalidValue;
  GHT_DISPATCH_BUCKETED(find_shape, tv, q, out, n, o, s)
}

// Debug check after a successful build (keys must be unique, Sec. VII): every
// scheme stores a key only in its candidate buckets H_0 .. H_{h-1}, so an
// input key with more than one copy across its distinct candidate buckets was
// passed more than once. Thread per key, every slot of every candidate read.
template <typename S>
__global__ void __launch_bounds__(256)
dup_check_kernel(TableView tv, int B, const uint32_t *__restrict__ keys, uint64_t n) {
  using T = typename S::T;
  const T *slots = reinterpret_cast<const T *>(tv.slots);
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const uint32_t k = __ldg(keys + i);
    if (k == kEmptyKey) continue;  // rejected by the build already
    uint32_t seen[4];
    int copies = 0;
    for (int f = 0; f < tv.h && f < 4; ++f) {
      const uint32_t b = bucket_of(tv.hf, f, k);
      bool again = false;
      for (int g = 0; g < f; ++g) again |= seen[g] == b;
      seen[f] = b;
      if (again) continue;
      for (int j = 0; j < B; ++j) copies += S::key(slots[(uint64_t)b * B + j]) == k;
    }
    if (copies > 1) atomicOr(&tv.ctrl->status, (uint32_t)kStatusDuplicate);
  }
}

cudaError_t launch_dup_check(const TableView &tv, int B, bool key_slots, const uint32_t *keys, uint64_t n,
                             cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  if (B < 1 || B > 32) return cudaErrorInvalidValue;
  int blocks = 0;
  auto kern = key_slots ? dup_check_kernel<KeySlot> : dup_check_kernel<PairSlot>;
  cudaError_t e = grid_for(kern, n, 0, &blocks);
  if (e != cudaSuccess) return e;
  kern<<<blocks, kThreads, 0, s>>>(tv, B, keys, n);
  return cudaGetLastError();
}

cudaError_t launch_fill(const TableView &tv, uint64_t num_slots, cudaStream_t s, uint32_t *counters, uint64_t m) {
  const uint64_t n16 = num_slots / 2;  // slots start 256-byte aligned
  uint64_t *tail = (num_slots & 1) ? tv.slots + (num_slots - 1) : nullptr;
  int blocks = 0;
  cudaError_t e = grid_for(fill_kernel, n16 > 0 ? n16 : 1, 0, &blocks);
  if (e != cudaSuccess) return e;
  fill_kernel<<<blocks, kThreads, 0, s>>>(reinterpret_cast<uint4 *>(tv.slots), n16, tail, tv.ctrl,
                                      counters, counters ? m : 0);
  return cudaGetLastError();
}

cudaError_t launch_hash(const TableView &tv, const uint32_t *k, uint32_t *out, uint64_t n,
                        cudaStream_t s) {
  int blocks = 0;
  cudaError_t e = grid_for(hash_kernel, n, 0, &blocks);
  if (e != cudaSuccess) return e;
  hash_kernel<<<blocks, kThreads, 0, s>>>(tv, k, out, n);
  return cudaGetLastError();
}

}  // namespace ght
