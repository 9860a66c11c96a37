// ws_multi_kernel.cuh -- the persistent multi-table kernel template, included
// only by the per-menu-entry translation units ws_multi_<entry>.cu.
#pragma once
#include "ws_multi.cuh"

namespace ws {

// One warp's share [begin, end) of a chunk of one item: streaming lanes, or
// -- for two-choice tables with plain 32-slot buckets -- 32-op chunks with
// whole-bucket rounds.  Frequent keys (HotKeys) and inserts without the lock
// (LW_INSERT_FRONT) are the single-table kernel's: copies of a Zipf-hot key in
// one item queue on its line here.  Returns the warp's count delta.
template <int SCHEME, bool META, int B, int T, int KIND>
__device__ __forceinline__ int multi_share(const MultiItem& it, u64 begin, u64 end, WarpSmem& sm, int lane) {
  constexpr bool kRounds = (SCHEME == SCHEME_P2) && !META && B == 32;
  const int op = (KIND == KIND_UPSERT) ? it.a.op : 0;
  const bool lockfree = (KIND == KIND_UPSERT) && it.lockfree != 0;
  if constexpr (kRounds) {
    int d = 0;
    for (u64 b = begin; b < end; b += 32)
      d += warp_chunk<SCHEME, META, B, T, KIND>(it.tv, it.a, op, lockfree, b, sm, lane);
    return d;
  } else {
    return warp_stream<SCHEME, META, B, T, KIND>(it.tv, it.a, op, lockfree, begin, end, sm, lane);
  }
}

// Warp copy of n <= kWarpShare elements, all of a lane's loads in flight
// before its stores (one side is host memory, microseconds away).
template <typename V>
__device__ __noinline__ void share_copy(V* dst, const V* src, int n, int lane) {
  constexpr int kEach = kWarpShare / 32;
  V v[kEach];
#pragma unroll
  for (int q = 0; q < kEach; ++q)
    if (q * 32 + lane < n) v[q] = src[q * 32 + lane];
#pragma unroll
  for (int q = 0; q < kEach; ++q)
    if (q * 32 + lane < n) dst[q * 32 + lane] = v[q];
}

// Every warp works alone: its own descriptor, its own place in the queue of
// 256-op shares (the first by its number, the rest from the ticket).  When a
// block took 2048-op chunks together, its warps waited for the slowest of
// eight shares, and for the ticket, chunk and descriptor reads before each
// chunk: 1024 tables of 2^10 to 2^22 slots, 70M ops in four phases, took 2520
// us, now 2257.
//
// Page-locked requests are copied in and out by the warps that serve them, a
// share at a time: a launch's transfers then take no call and no turn on a
// copy engine each, and overlap with other warps' probing.  With one
// copy-engine transfer per request and array (three in, two out, one for the
// live count) they cost about 2 us each on the host and on the engine: 96
// requests of 14,600 ops on average, 32 tables, took 2060 us, of which 1137 us
// in 607 transfers; now they take 1305 us.
template <int SCHEME, bool META, int B, int T, int KIND>
__global__ void __launch_bounds__(kThreads, 4) multi_kernel(MultiGroup g) {
  __shared__ WarpSmem s_w[kWarps];
  __shared__ __align__(16) MultiItem s_it[kWarps];
  static_assert(sizeof(MultiItem) % 8 == 0, "item copy");
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const u32 warps = gridDim.x * kWarps;
  const MultiItem& it = s_it[w];
  u32 cur_item = 0xffffffffu;
  for (u32 unit = blockIdx.x * kWarps + w; unit / kWarps < g.n_chunks;) {  // warp-uniform
    u32 item;
    u64 begin;
    if (g.chunks) {
      const MultiChunk ch = g.chunks[unit / kWarps];
      item = ch.item;
      begin = ch.start;
    } else {
      const u32 gc = g.prefix[g.i0] + unit / kWarps;
      u32 lo = g.i0, hi = g.i1 - 1;  // largest item with prefix[item] <= gc
      while (lo < hi) {
        const u32 mid = (lo + hi + 1) / 2;
        if (g.prefix[mid] <= gc)
          lo = mid;
        else
          hi = mid - 1;
      }
      item = lo;
      begin = (u64)(gc - g.prefix[lo]) * kMultiChunk;
    }
    begin += (u64)(unit % kWarps) * kWarpShare;
    if (item != cur_item) {  // stage the item descriptor once
      const u64* src = reinterpret_cast<const u64*>(g.items + item);
      u64* dst = reinterpret_cast<u64*>(&s_it[w]);
      for (int q = lane; q < (int)(sizeof(MultiItem) / 8); q += 32) dst[q] = src[q];
      cur_item = item;
      __syncwarp();
    }
    if (begin < it.a.n) {
      const int n_here = (int)(it.a.n - begin < (u64)kWarpShare ? it.a.n - begin : (u64)kWarpShare);
      HostOps host = {};
      if (KIND == KIND_MIXED && g.host) host = g.host[item];
      if (KIND == KIND_MIXED && host.keys) {
        share_copy(const_cast<u64*>(it.a.keys) + begin, host.keys + begin, n_here, lane);
        if (host.vals) share_copy(const_cast<u64*>(it.a.vals) + begin, host.vals + begin, n_here, lane);
        share_copy(const_cast<u8*>(it.a.ops) + begin, host.ops + begin, n_here, lane);
        __syncwarp();
      }
      int d = multi_share<SCHEME, META, B, T, KIND>(it, begin, begin + n_here, s_w[w], lane);
      if (KIND != KIND_QUERY) {
        d = __reduce_add_sync(0xffffffffu, d);
        if (lane == 0 && d) {
          const unsigned long long was =
              atomicAdd((unsigned long long*)&it.tv.ctr->count, (unsigned long long)(long long)d);
          // Two-choice and iceberg tables: the next single-table insert reads
          // its load from `live` as long as nothing was erased, and until then
          // `count` only grows.  Left behind, a table filled here looks empty
          // to it: keys then go in without their locks at loads where that
          // is slower and less even.
          if (SCHEME != SCHEME_DOUBLE && d > 0) atomicMax((unsigned long long*)&it.tv.ctr->live, was + d);
        }
      }
      __syncwarp();  // the share's results are written
      if (KIND == KIND_MIXED && g.host) {
        const HostOps out = g.host[item];  // read again: not kept in registers while the share is served
        if (out.keys && out.vals_out) share_copy(out.vals_out + begin, it.a.vals_out + begin, n_here, lane);
        if (out.keys && out.status_out) share_copy(out.status_out + begin, it.a.status_out + begin, n_here, lane);
      }
    }
    if (lane == 0) unit = warps + atomicAdd(g.ticket, 1u);
    unit = __shfl_sync(0xffffffffu, unit, 0);  // every lane is done with s_it
  }
}

template <void (*KERN)(MultiGroup)>
cudaError_t launch_multi_one(const MultiGroup& g, cudaStream_t s, int num_sms) {
  static int occ = 0;
  if (occ == 0) {
    int o = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, KERN, kThreads, 0) != cudaSuccess || o < 1) o = 1;
    occ = o;
  }
  const u64 cap = (u64)occ * (u64)(num_sms > 0 ? num_sms : 1);
  const unsigned grid = (unsigned)(g.n_chunks < cap ? g.n_chunks : cap);
  if (grid == 0) return cudaSuccess;
  KERN<<<grid, kThreads, 0, s>>>(g);
  return cudaGetLastError();
}

template <int SCHEME, bool META, int B, int T>
cudaError_t launch_multi_cfg(int kind, const MultiGroup& g, cudaStream_t s, int num_sms) {
  switch (kind) {
    case KIND_QUERY: return launch_multi_one<multi_kernel<SCHEME, META, B, T, KIND_QUERY>>(g, s, num_sms);
    case KIND_UPSERT: return launch_multi_one<multi_kernel<SCHEME, META, B, T, KIND_UPSERT>>(g, s, num_sms);
    case KIND_ERASE: return launch_multi_one<multi_kernel<SCHEME, META, B, T, KIND_ERASE>>(g, s, num_sms);
    case KIND_MIXED: return launch_multi_one<multi_kernel<SCHEME, META, B, T, KIND_MIXED>>(g, s, num_sms);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ws
