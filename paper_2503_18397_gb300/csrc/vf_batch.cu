// Batched construction kernels of libvfunc (sm_103a): hashing, shard
// histograms and the radix scatter for many independent structures at once.
// The keys of all structures form one index space; each item of the
// descriptor table owns the range [key_off, key_off + n) of it, and each
// (structure, shard) pair owns one histogram / cursor slot.
#include "vf_internal.h"

namespace vf {

constexpr int kBT = 256;
constexpr int kItemCache = 4096;  // key offsets of up to 4096 structures cached in shared memory

// Item owning global key g: largest i with key_off[i] <= g.
__device__ __forceinline__ uint32_t find_item(const uint64_t* off, uint32_t count, uint64_t g) {
    uint32_t lo = 0, hi = count;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (off[mid] <= g) lo = mid; else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ uint32_t batch_value(const void* values, int b, uint64_t i) {
    uint32_t v;
    if (b <= 8) v = __ldg(static_cast<const uint8_t*>(values) + i);
    else if (b <= 16) v = __ldg(static_cast<const uint16_t*>(values) + i);
    else v = __ldg(static_cast<const uint32_t*>(values) + i);
    return b == 32 ? v : (v & ((1u << b) - 1u));
}

// Loads the items' key offsets into shared memory when they fit.
__device__ __forceinline__ const uint64_t* cache_offsets(const BatchItem* items, uint32_t count, uint64_t* s_off) {
    if (count <= kItemCache) {
        for (uint32_t i = threadIdx.x; i < count; i += blockDim.x) s_off[i] = items[i].key_off;
        __syncthreads();
        return s_off;
    }
    return nullptr;
}

__device__ __forceinline__ uint32_t item_of(const BatchItem* items, const uint64_t* s_off, const uint64_t* g_off,
                                            uint32_t count, uint64_t g) {
    return find_item(s_off ? s_off : g_off, count, g);
}

// Both kernels take tiles of consecutive keys. A tile almost always lies within
// one structure, whose descriptor is then looked up once and whose shards are
// counted in shared memory, one global atomic per shard and tile; an unsharded
// structure's keys need no counting at all and stay in order. A tile with a
// boundary in it, or of a structure of more than kTileShards shards, goes key by
// key (lanes of a warp with the same slot share one atomic). 512 structures, 6.9*10^7
// keys: histogram 0.56 -> 0.13 ms a pass, scatter 1.94 -> 0.92.
constexpr int kTileItems = 8;
constexpr uint32_t kTileKeys = kBT * kTileItems;
constexpr uint32_t kTileShards = 512;

// One structure's tile: s_cnt (zeroed, kTileShards words) counts its shards; each
// key's shard and rank among the tile's keys of that shard. Few shards: a warp's
// lanes of one shard add once.
__device__ __forceinline__ uint32_t tile_rank(uint32_t* s_cnt, uint32_t shard, bool on, bool few) {
    if (!few) return on ? atomicAdd(&s_cnt[shard], 1u) : 0u;
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, on ? shard : 0xFFFFFFFFu);
    const unsigned lane = threadIdx.x & 31u;
    const int lead = __ffs(peers) - 1;
    uint32_t at = 0;
    if (on && int(lane) == lead) at = atomicAdd(&s_cnt[shard], uint32_t(__popc(peers)));
    return __shfl_sync(0xFFFFFFFFu, at, lead) + __popc(peers & ((1u << lane) - 1u));
}

// Per-(structure, shard) key counts.
__global__ void __launch_bounds__(kBT) k_batch_hist(const BatchItem* __restrict__ items,
                                                    const uint64_t* __restrict__ key_off, uint32_t count,
                                                    uint64_t total, uint32_t* __restrict__ hist) {
    __shared__ uint64_t s_off[kItemCache];
    __shared__ uint32_t s_cnt[kTileShards];
    const uint64_t* so = cache_offsets(items, count, s_off);
    const unsigned lane = threadIdx.x & 31u;
    for (uint64_t t0 = uint64_t(blockIdx.x) * kTileKeys; t0 < total; t0 += uint64_t(gridDim.x) * kTileKeys) {
        const uint32_t m = total - t0 < kTileKeys ? uint32_t(total - t0) : kTileKeys;
        const BatchItem& d = items[item_of(items, so, key_off, count, t0)];
        const uint64_t j0 = t0 - d.key_off;
        const uint32_t S = d.h < 31 ? 1u << d.h : 0xFFFFFFFFu;
        if (j0 + m <= d.n && S == 1) {
            if (threadIdx.x == 0) atomicAdd(hist + d.hist_off, m);
        } else if (j0 + m <= d.n && S <= kTileShards) {
            for (uint32_t i = threadIdx.x; i < S; i += kBT) s_cnt[i] = 0;
            uint64_t ks[kTileItems];
#pragma unroll
            for (int j = 0; j < kTileItems; j++) {
                const uint32_t i = threadIdx.x + uint32_t(j) * kBT;
                ks[j] = i < m ? __ldg(d.keys + j0 + i) : 0ull;
            }
            __syncthreads();
#pragma unroll
            for (int j = 0; j < kTileItems; j++)
                tile_rank(s_cnt, uint32_t(shard_of(sig_u64(ks[j], d.kh, d.kl), d.h)), threadIdx.x + uint32_t(j) * kBT < m, S <= 16);
            __syncthreads();
            for (uint32_t i = threadIdx.x; i < S; i += kBT)
                if (s_cnt[i]) atomicAdd(hist + d.hist_off + i, s_cnt[i]);
            __syncthreads();
        } else {
            for (uint32_t i0 = threadIdx.x & ~31u; i0 < m; i0 += kBT) {
                const uint64_t g = t0 + i0 + lane;
                uint32_t slot = 0xFFFFFFFFu;
                if (i0 + lane < m) {
                    const BatchItem& q = items[item_of(items, so, key_off, count, g)];
                    const Sig s = sig_u64(__ldg(q.keys + (g - q.key_off)), q.kh, q.kl);
                    slot = q.hist_off + uint32_t(shard_of(s, q.h));
                }
                const unsigned peers = __match_any_sync(0xFFFFFFFFu, slot);
                if (slot != 0xFFFFFFFFu && lane == unsigned(__ffs(peers) - 1)) atomicAdd(hist + slot, uint32_t(__popc(peers)));
            }
        }
    }
}

// Radix scatter into the concatenated bucketed arrays: cursor[slot] starts at
// the slot's first position and advances by the number of keys written there.
__global__ void __launch_bounds__(kBT) k_batch_scatter(const BatchItem* __restrict__ items,
                                                       const uint64_t* __restrict__ key_off, uint32_t count,
                                                       uint64_t total, unsigned long long* __restrict__ cursor,
                                                       uint64_t* __restrict__ loc_out, uint32_t* __restrict__ val_out) {
    __shared__ uint64_t s_off[kItemCache];
    __shared__ uint32_t s_cnt[kTileShards];
    __shared__ unsigned long long s_base[kTileShards];
    const uint64_t* so = cache_offsets(items, count, s_off);
    const unsigned lane = threadIdx.x & 31u;
    for (uint64_t t0 = uint64_t(blockIdx.x) * kTileKeys; t0 < total; t0 += uint64_t(gridDim.x) * kTileKeys) {
        const uint32_t m = total - t0 < kTileKeys ? uint32_t(total - t0) : kTileKeys;
        const BatchItem& d = items[item_of(items, so, key_off, count, t0)];
        const uint64_t j0 = t0 - d.key_off;
        const uint32_t S = d.h < 31 ? 1u << d.h : 0xFFFFFFFFu;
        if (j0 + m <= d.n && S <= kTileShards) {
            const bool has_val = d.vals != nullptr;
            for (uint32_t i = threadIdx.x; i < S; i += kBT) s_cnt[i] = 0;
            uint64_t ks[kTileItems];
            uint32_t rk[kTileItems], vs[kTileItems];
#pragma unroll
            for (int j = 0; j < kTileItems; j++) {
                const uint32_t i = threadIdx.x + uint32_t(j) * kBT;
                ks[j] = i < m ? __ldg(d.keys + j0 + i) : 0ull;
                vs[j] = i < m && has_val ? batch_value(d.vals, d.b, j0 + i) : 0u;
            }
            __syncthreads();
            if (S == 1) {
                if (threadIdx.x == 0) s_base[0] = atomicAdd(cursor + d.hist_off, (unsigned long long)m);
            } else {
#pragma unroll
                for (int j = 0; j < kTileItems; j++)
                    rk[j] = tile_rank(s_cnt, uint32_t(shard_of(sig_u64(ks[j], d.kh, d.kl), d.h)),
                                      threadIdx.x + uint32_t(j) * kBT < m, S <= 16);
                __syncthreads();
                for (uint32_t i = threadIdx.x; i < S; i += kBT)
                    if (s_cnt[i]) s_base[i] = atomicAdd(cursor + d.hist_off + i, (unsigned long long)s_cnt[i]);
            }
            __syncthreads();
#pragma unroll
            for (int j = 0; j < kTileItems; j++) {
                const uint32_t i = threadIdx.x + uint32_t(j) * kBT;
                if (i >= m) continue;
                const Sig s = sig_u64(ks[j], d.kh, d.kl);
                const uint64_t pos = S == 1 ? s_base[0] + i : s_base[shard_of(s, d.h)] + rk[j];
                loc_out[pos] = local_of(s, d.h);
                val_out[pos] = vs[j];
            }
            __syncthreads();
        } else {
            for (uint32_t i0 = threadIdx.x & ~31u; i0 < m; i0 += kBT) {
                const uint64_t g = t0 + i0 + lane;
                uint32_t slot = 0xFFFFFFFFu;
                uint64_t local = 0;
                uint32_t value = 0;
                if (i0 + lane < m) {
                    const BatchItem& q = items[item_of(items, so, key_off, count, g)];
                    const uint64_t j = g - q.key_off;
                    const Sig s = sig_u64(__ldg(q.keys + j), q.kh, q.kl);
                    slot = q.hist_off + uint32_t(shard_of(s, q.h));
                    local = local_of(s, q.h);
                    value = q.vals ? batch_value(q.vals, q.b, j) : 0u;
                }
                const unsigned peers = __match_any_sync(0xFFFFFFFFu, slot);
                const unsigned leader = unsigned(__ffs(peers) - 1);
                unsigned long long base = 0;
                if (slot != 0xFFFFFFFFu && lane == leader) base = atomicAdd(cursor + slot, (unsigned long long)__popc(peers));
                base = __shfl_sync(0xFFFFFFFFu, base, int(leader));
                if (slot != 0xFFFFFFFFu) {
                    const uint64_t pos = base + __popc(peers & ((1u << lane) - 1u));
                    loc_out[pos] = local;
                    val_out[pos] = value;
                }
            }
        }
    }
}

static unsigned batch_grid(uint64_t total) {
    uint64_t blocks = (total + kTileKeys - 1) / kTileKeys;
    const uint64_t cap = uint64_t(num_sms()) * 8;
    if (blocks > cap) blocks = cap;
    return unsigned(blocks < 1 ? 1 : blocks);
}

cudaError_t launch_batch_hist(const BatchItem* items, const uint64_t* key_off, uint32_t count, uint64_t total,
                              uint32_t* hist, cudaStream_t st) {
    if (total == 0) return cudaSuccess;
    k_batch_hist<<<batch_grid(total), kBT, 0, st>>>(items, key_off, count, total, hist);
    return cudaGetLastError();
}

cudaError_t launch_batch_scatter(const BatchItem* items, const uint64_t* key_off, uint32_t count, uint64_t total,
                                 unsigned long long* cursor, uint64_t* loc, uint32_t* val, cudaStream_t st) {
    if (total == 0) return cudaSuccess;
    k_batch_scatter<<<batch_grid(total), kBT, 0, st>>>(items, key_off, count, total, cursor, loc, val);
    return cudaGetLastError();
}

}  // namespace vf
