// Query kernel of libvfunc (sm_103a): signature -> shard (top h bits) ->
// cell offset shard*cells (no offset array, Sec. 4) -> three cells -> XOR
// (eq. MWHC, k = 3) -> [filter: compare with the fingerprint].
//
// Each thread takes kQ keys spaced one grid-stride apart (coalesced key loads)
// and issues all 3*kQ cell loads before using any, so every warp keeps 96
// independent random 32-byte sector reads in flight.
#include <algorithm>

#include "vf_internal.h"

namespace vf {

constexpr int kQThreads = 256;
constexpr int kQ = 4;

template <int WIDTH>
__device__ __forceinline__ uint32_t cell_q(const uint8_t* data, int b, uint64_t i) {
    if constexpr (WIDTH == 8) return __ldg(data + i);
    else if constexpr (WIDTH == 16) return __ldg(reinterpret_cast<const uint16_t*>(data) + i);
    else if constexpr (WIDTH == 32) return __ldg(reinterpret_cast<const uint32_t*>(data) + i);
    else return cell_get_nc(data, b, i);
}

// The answer of one key from its cells' XOR.
template <bool FILTER>
__device__ __forceinline__ void put_answer(void* out, uint64_t i, uint32_t r, uint64_t local, int b) {
    if constexpr (FILTER) {
        static_cast<uint8_t*>(out)[i] = uint8_t(r == fingerprint(local, b));
    } else {
        if (b <= 8) static_cast<uint8_t*>(out)[i] = uint8_t(r);
        else if (b <= 16) static_cast<uint16_t*>(out)[i] = uint16_t(r);
        else static_cast<uint32_t*>(out)[i] = r;
    }
}

// K: vertices per edge (3, or 4 for a 4-uniform fuse graph).
template <int WIDTH, bool FILTER, int K>
__global__ void __launch_bounds__(kQThreads) k_query(const uint64_t* __restrict__ keys, uint64_t m, Geom g,
                                                     const uint8_t* __restrict__ data, void* __restrict__ out) {
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t i0 = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i0 < m; i0 += stride * kQ) {
        uint64_t idx[kQ], loc[kQ], cell[kQ][K];
        bool ok[kQ];
#pragma unroll
        for (int k = 0; k < kQ; k++) {
            idx[k] = i0 + uint64_t(k) * stride;
            ok[k] = idx[k] < m;
            // keys are read once: evict-first, so the cells they probe stay in L2
            const Sig s = ok[k] ? sig_u64(__ldcs(keys + idx[k]), g.kh, g.kl) : Sig{0, 0};
            uint64_t base = shard_of(s, g.h) * g.cells;
            loc[k] = local_of(s, g.h);
            uint64_t v[4];
            edge_of(g, loc[k], v);
#pragma unroll
            for (int j = 0; j < K; j++) cell[k][j] = base + v[j];
        }
        uint32_t x[kQ][K];
#pragma unroll
        for (int k = 0; k < kQ; k++)
#pragma unroll
            for (int j = 0; j < K; j++) x[k][j] = ok[k] ? cell_q<WIDTH>(data, g.b, cell[k][j]) : 0u;
#pragma unroll
        for (int k = 0; k < kQ; k++) {
            if (!ok[k]) continue;
            uint32_t r = x[k][0] ^ x[k][1] ^ x[k][2];
            if constexpr (K == 4) r ^= x[k][3];
            put_answer<FILTER>(out, idx[k], r, loc[k], g.b);
        }
    }
}

// Byte strings: a block takes tiles of consecutive strings through shared
// memory (sig_tile) and probes one key a thread; the resident blocks keep
// enough probes in flight. A tile alternates between loads and remixes, with
// barriers between, so blocks on an SM count (six of 40 registers a thread, not
// five of 48), and blocks of few tiles, which start as others end (3*10^6
// strings: 101 -> 92 us with both; six resident blocks a SM that stay: 102).
template <int WIDTH, bool FILTER, int K>
__global__ void __launch_bounds__(kQThreads, 6) k_query_bytes(const uint8_t* __restrict__ buf,
                                                           const uint64_t* __restrict__ offs, uint64_t m, Geom g,
                                                           const uint8_t* __restrict__ data, void* __restrict__ out) {
    static_assert(kQThreads == kTileStrings, "a string a thread");
    __shared__ StringTile tile;
    const uint64_t total = __ldg(offs + m);
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t t0 = blockIdx.x * uint64_t(blockDim.x); t0 < m; t0 += stride) {
        uint64_t i;
        const Sig s = sig_tile(buf, offs, total, t0, m, tile, g.kh, g.kl, i);
        if (i >= m) continue;
        const uint64_t base = shard_of(s, g.h) * g.cells;
        const uint64_t local = local_of(s, g.h);
        uint64_t v[4];
        edge_of(g, local, v);
        uint32_t r = 0;
#pragma unroll
        for (int j = 0; j < K; j++) r ^= cell_q<WIDTH>(data, g.b, base + v[j]);
        put_answer<FILTER>(out, i, r, local, g.b);
    }
}

template <int WIDTH, bool FILTER>
static void launch_q(bool bytes, const void* keys, const uint64_t* offs, uint64_t m, const Geom& g,
                     const uint8_t* data, void* out, cudaStream_t st) {
    const uint64_t per = uint64_t(kQThreads) * (bytes ? 1 : kQ);
    uint64_t blocks = (m + per - 1) / per;
    uint64_t cap = uint64_t(num_sms()) * (bytes ? 24 : 16);  // bytes: four times what is resident
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    const uint64_t* k64 = static_cast<const uint64_t*>(keys);
    const uint8_t* k8 = static_cast<const uint8_t*>(keys);
    if (g.k == 4) {
        if (bytes) k_query_bytes<WIDTH, FILTER, 4><<<unsigned(blocks), kQThreads, 0, st>>>(k8, offs, m, g, data, out);
        else k_query<WIDTH, FILTER, 4><<<unsigned(blocks), kQThreads, 0, st>>>(k64, m, g, data, out);
    } else if (bytes) {
        k_query_bytes<WIDTH, FILTER, 3><<<unsigned(blocks), kQThreads, 0, st>>>(k8, offs, m, g, data, out);
    } else {
        k_query<WIDTH, FILTER, 3><<<unsigned(blocks), kQThreads, 0, st>>>(k64, m, g, data, out);
    }
}

template <bool FILTER>
static void launch_w(bool bytes, const void* keys, const uint64_t* offs, uint64_t m, const Geom& g,
                     const uint8_t* data, void* out, cudaStream_t st) {
    switch (g.b) {
        case 8: launch_q<8, FILTER>(bytes, keys, offs, m, g, data, out, st); break;
        case 16: launch_q<16, FILTER>(bytes, keys, offs, m, g, data, out, st); break;
        case 32: launch_q<32, FILTER>(bytes, keys, offs, m, g, data, out, st); break;
        default: launch_q<0, FILTER>(bytes, keys, offs, m, g, data, out, st); break;
    }
}

// ------------------------------------------------------- cross-structure batch

constexpr int kReqCache = 4096;
constexpr uint32_t kFewRequests = 1024;  // k_query_few: requests it takes

// The cells' XOR of key i of request r and its answer.
__device__ __forceinline__ void query_one(const QueryReq& r, uint64_t i) {
    const Sig s = sig_u64(__ldcs(r.keys + i), r.g.kh, r.g.kl);
    const uint64_t base = shard_of(s, r.g.h) * r.g.cells;
    const uint64_t local = local_of(s, r.g.h);
    uint64_t v[4];
    edge_of(r.g, local, v);
    if (r.g.b > 32) {  // values wider than 32 bits
        uint64_t y = cell_get64(r.data, r.g.b, base + v[0]) ^ cell_get64(r.data, r.g.b, base + v[1]) ^
                     cell_get64(r.data, r.g.b, base + v[2]);
        if (r.g.k == 4) y ^= cell_get64(r.data, r.g.b, base + v[3]);
        if (r.g.kind == 1) static_cast<uint8_t*>(r.out)[i] = uint8_t(y == fingerprint64(local, r.g.b));
        else static_cast<uint64_t*>(r.out)[i] = y;
        return;
    }
    uint32_t x = cell_get_nc(r.data, r.g.b, base + v[0]) ^ cell_get_nc(r.data, r.g.b, base + v[1]) ^
                 cell_get_nc(r.data, r.g.b, base + v[2]);
    if (r.g.k == 4) x ^= cell_get_nc(r.data, r.g.b, base + v[3]);
    if (r.g.kind == 1) put_answer<true>(r.out, i, x, local, r.g.b);
    else put_answer<false>(r.out, i, x, local, r.g.b);
}

// kQ keys of one request (of a 3-uniform structure) per thread, spaced a block
// apart, with all their cell loads in flight before any is used (as k_query).
template <int WIDTH, bool FILTER>
__device__ __forceinline__ void query_tile(const QueryReq& r, uint64_t i0, uint32_t m) {
    const Geom g = r.g;
    const uint64_t* const keys = r.keys + i0;
    uint64_t loc[kQ], cell[kQ][3];
#pragma unroll
    for (int k = 0; k < kQ; k++) {
        const uint32_t i = threadIdx.x + k * kQThreads;
        const Sig s = i < m ? sig_u64(__ldcs(keys + i), g.kh, g.kl) : Sig{0, 0};
        const uint64_t base = shard_of(s, g.h) * g.cells;
        loc[k] = local_of(s, g.h);
        uint64_t v[4];
        edge_of(g, loc[k], v);
#pragma unroll
        for (int j = 0; j < 3; j++) cell[k][j] = base + v[j];
    }
    uint32_t x[kQ];
#pragma unroll
    for (int k = 0; k < kQ; k++) {
        uint32_t c[3];
#pragma unroll
        for (int j = 0; j < 3; j++) c[j] = threadIdx.x + k * kQThreads < m ? cell_q<WIDTH>(r.data, g.b, cell[k][j]) : 0u;
        x[k] = c[0] ^ c[1] ^ c[2];
    }
#pragma unroll
    for (int k = 0; k < kQ; k++) {
        const uint32_t i = threadIdx.x + k * kQThreads;
        if (i < m) put_answer<FILTER>(r.out, i0 + i, x[k], loc[k], g.b);
    }
}

// The request that key g of the launch belongs to; s_off: the offsets, where they fit
// there (cached).
__device__ __forceinline__ uint32_t request_of(const QueryReq* reqs, const uint64_t* s_off, bool cached, uint32_t count,
                                               uint64_t g) {
    uint32_t lo = 0, hi = count;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        const uint64_t o = cached ? s_off[mid] : reqs[mid].key_off;
        if (o <= g) lo = mid; else hi = mid;
    }
    return lo;
}

// Requests against many resident structures in one launch: request r owns
// keys [key_off, key_off + m) of the launch's key space. Few keys: one a thread,
// each with its own search. At most kFewRequests.
__global__ void __launch_bounds__(kQThreads) k_query_few(const QueryReq* __restrict__ reqs, uint32_t count, uint64_t total) {
    __shared__ uint64_t s_off[kFewRequests];
    for (uint32_t i = threadIdx.x; i < count; i += blockDim.x) s_off[i] = reqs[i].key_off;
    __syncthreads();
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t g = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; g < total; g += stride) {
        const QueryReq& q = reqs[request_of(reqs, s_off, true, count, g)];
        query_one(q, g - q.key_off);
    }
}

// Many: a block takes tiles of consecutive keys; a tile mostly lies within one
// request, whose descriptor is then looked up once for the block and whose keys go
// four a thread (96 requests of 3*10^5 to 1.5*10^6 keys: 1.80 ms with a search and one
// key a thread, 1.07 this way). A tile with a boundary in it is taken key by key.
__global__ void __launch_bounds__(kQThreads, 4) k_query_batch(const QueryReq* __restrict__ reqs, uint32_t count,
                                                           uint64_t total) {
    constexpr uint32_t kTileKeys = kQThreads * kQ;
    __shared__ uint64_t s_off[kReqCache];
    const bool cached = count <= kReqCache;
    if (cached)
        for (uint32_t i = threadIdx.x; i < count; i += blockDim.x) s_off[i] = reqs[i].key_off;
    __syncthreads();
    for (uint64_t t0 = uint64_t(blockIdx.x) * kTileKeys; t0 < total; t0 += uint64_t(gridDim.x) * kTileKeys) {
        const uint32_t m = total - t0 < kTileKeys ? uint32_t(total - t0) : kTileKeys;
        const QueryReq& r = reqs[request_of(reqs, s_off, cached, count, t0)];
        const uint64_t i0 = t0 - r.key_off;
        if (i0 + m <= r.m && r.g.k != 4 && (r.g.b == 8 || r.g.b == 16)) {
            if (r.g.kind == 1) {
                if (r.g.b == 8) query_tile<8, true>(r, i0, m);
                else query_tile<16, true>(r, i0, m);
            } else {
                if (r.g.b == 8) query_tile<8, false>(r, i0, m);
                else query_tile<16, false>(r, i0, m);
            }
        } else if (i0 + m <= r.m && r.g.k != 4 && r.g.b <= 32) {
            if (r.g.kind == 1) query_tile<0, true>(r, i0, m);
            else query_tile<0, false>(r, i0, m);
        } else {
            for (uint32_t i = threadIdx.x; i < m; i += kQThreads) {
                const QueryReq& q = reqs[request_of(reqs, s_off, cached, count, t0 + i)];
                query_one(q, t0 + i - q.key_off);
            }
        }
    }
}

// Up to five blocks of keys an SM, a key a thread: four keys of a thread after one
// another on a quarter of the blocks cost more than they save. Device time, us, a key a
// thread and tiles: one request of 1000 keys 5.6, 8.7 (wider than 32 bits 6.2, 10.3;
// 4-uniform 6.1, 10.3), of 10^5 8.1, 8.5 (8.7, 11.7), of 2*10^5 10.6, 10.2, of 3*10^5 14.0, 10.1; 100 of
// 500 9.9, 13.3; 300 of 500 10.6, 15.2; 700 of 500 22.5, 19.5; 10 of 20,000 10.9, 13.8, of
// 30,000 14.8, 13.0. And not where every block would read thousands of offsets for a few
// keys: 1000 of 64 13.4, 16.0; 3000 of 64 22.8, 18.6.
constexpr uint32_t kFewBlocks = 5;

cudaError_t launch_query_batch(const QueryReq* reqs, uint32_t count, uint64_t total, cudaStream_t st) {
    if (total == 0 || count == 0) return cudaSuccess;
    const bool few = count <= kFewRequests && total <= uint64_t(num_sms()) * kFewBlocks * kQThreads;
    const uint64_t per = uint64_t(kQThreads) * (few ? 1 : kQ), cap = uint64_t(num_sms()) * 16;
    const unsigned blocks = unsigned(std::min((total + per - 1) / per, cap));
    if (few) k_query_few<<<blocks, kQThreads, 0, st>>>(reqs, count, total);
    else k_query_batch<<<blocks, kQThreads, 0, st>>>(reqs, count, total);
    return cudaGetLastError();
}

cudaError_t launch_query(int key_kind, const void* keys, const uint64_t* offs, uint64_t m, const Geom& g,
                         const uint8_t* data, void* out, cudaStream_t st) {
    if (m == 0) return cudaSuccess;
    bool bytes = key_kind != 0;
    if (g.b > 32) return launch_query_wide(keys, bytes ? offs : nullptr, m, g, data, out, st);
    if (g.kind == 1) launch_w<true>(bytes, keys, offs, m, g, data, out, st);
    else launch_w<false>(bytes, keys, offs, m, g, data, out, st);
    return cudaGetLastError();
}

}  // namespace vf
