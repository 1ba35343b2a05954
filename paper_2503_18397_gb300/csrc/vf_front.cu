// Fuse-regime peeling of libvfunc (sm_103a), the waves: one cluster of CTAs per
// shard in synchronous rounds over vertex words in L2, with one cluster-wide
// exchange per round and no counter that more than one CTA takes.
//
// A fuse shard peels as two waves that move inward from its ends (Sec. 4.5):
// about 8000 dependent rounds of ~1000 edges at 12.5M keys. The first
// kFrontHead rounds, in which every degree-one vertex's short cascade is peeled
// (a third of the edges), are launches of their own over all shards' lists. From
// there on a round's latency counts, not bandwidth, and k_front_peel is built
// around the round's dependent chain:
//   claim bit and signature of the frontier's edges (one L2 trip, both in
//   flight together, sent before the round's exchange is waited for)
//   -> the edge's other vertices -> their fetch-and-adds (one L2 trip, whose
//   results are the next frontier) -> the CTA's list in shared memory.
// The exchange: every CTA sends its frontier's size to every CTA of the
// cluster with st.async, which also completes that CTA's mbarrier: one one-way
// message per pair orders the rounds, tells every CTA the round's total (the
// exit test, equal in all CTAs) and where its records start (the sum of the
// sizes before its own). No fence is needed: what a round hands to the next in
// global memory is fetch-and-adds whose results have come back. (A
// barrier.cluster with release and acquire costs ~650 cycles.)
// The wait for it is bounded. A CTA whose wait runs out leaves a mark with every CTA
// of the cluster before it comes to its next cluster barrier, and all of them leave
// the peel behind that barrier, whichever of theirs it meets: the marks that name
// a barrier are the same for all behind it.
//
// Vertex words, claims and records are the worklist solver's. An edge claimed
// for a vertex at the end of round r is removed in round r+1. A round's
// entries take the shard's record slots behind those of the rounds before, in
// list order, empty where the claim failed. A vertex that an edge of round r
// frees is peeled in a later round, so decreasing slot order is a reverse
// peeling order, as the assignment needs it.
//
// The CTA whose fetch-and-add frees a vertex keeps it, so sizes drift apart
// as the waves branch and die out; when one CTA holds well more than the mean
// (front_uneven; every CTA sees the same sizes), the round's pushes are dealt out over the
// cluster through distributed shared memory, behind a full cluster barrier.
//
// Measured (one GB300, b = 8; peel per attempt, worklist -> this): 2^20 keys 2.92 ->
// 2.59 ms, 10^8 (8 shards) 32.2 -> 26.8, 3*10^8 (16) 49.7 -> 27.0, 10^9 (64) 188 -> 86;
// 4-uniform 10^8 14.9 -> 13.1, 3*10^8 56.5 -> 24.7 (and where it is slower: front_pays). A round takes ~4300 cycles at 10^8:
// ~1100 to the claims and signatures, ~1400 to the removals, ~450 waiting for
// the slowest CTA, the rest between them (a remote fetch-and-add also costs an
// SM ~3.3 cycles a lane, L2 or distributed shared memory alike, and a CTA has
// ~64 entries a round). With many shards random DRAM sectors bound it: more
// than 16 clusters at once gain little at 10^9 keys.
#include <algorithm>
#include <mutex>

#include "vf_internal.h"

namespace vf {

constexpr int kFrWork = 256;            // threads that hold frontier entries
constexpr int kFrT = kFrWork + 32;      // and the warp that exchanges the sizes
constexpr uint32_t kFrList = 2048;      // frontier entries a CTA holds in shared memory, per buffer
constexpr uint32_t kFrMaxC = 16;        // CTAs per cluster
constexpr uint32_t kFrHole = 0xFFFFFFFFu;
constexpr int kFrHeadT = 1024;          // threads of a head round's block (one block per list)
constexpr uint32_t kFrHeadPer = 4;      // entries a thread has in flight there (2: +0.15 ms at 10^8 keys)

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return uint32_t(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ uint32_t map_to_cta(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Stores v in a peer's shared memory and counts 4 bytes on the peer's mbarrier.
__device__ __forceinline__ void post_u32(uint32_t remote, uint32_t v, uint32_t remote_mbar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(remote), "r"(v),
                 "r"(remote_mbar)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t mbar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(mbar), "r"(parity)
        : "memory");
    return ok != 0;
}

// A frontier entry on its way: vertex and edge (shard-local), the edge's
// signature, value and claim word as it was, then its other vertices in edge order.
template <int K>
struct FrontItem {
    uint64_t local;
    uint32_t v, e, value, cold;
    uint32_t o[K - 1];
    bool on;  // holds an entry; after front_others: holds an edge to remove
};

// Claims the entry's edge and loads its signature (and value).
template <int K, bool VAL>
__device__ __forceinline__ void front_fetch(FrontItem<K>& x, const FrontArgs& a, uint2 ve, unsigned long long st0, uint32_t ns) {
    x.v = ve.x;
    x.e = ve.y;
    x.on = ve.y < ns;
    if (!x.on) {  // impossible for exact words: touch nothing
        atomicOr(a.err, kErrCapacity);
        return;
    }
    const uint32_t e = uint32_t(st0) + ve.y;  // a group holds fewer than 2^32 edges
    x.cold = atomicOr(a.claimed + (e >> 5), 1u << (e & 31u));
    x.local = __ldg(a.loc + e);
    if (VAL) x.value = __ldg(a.val + e);
}

template <int K>
__device__ __forceinline__ void front_others(FrontItem<K>& x, const Geom& g, unsigned long long st0) {
    const uint32_t lgs = uint32_t(g.lg_seg), smask = (1u << lgs) - 1u;
    const uint32_t v0 = uint32_t(mulhi(x.local, g.span));
    const uint32_t s1 = (v0 >> lgs) + 1u;
    const uint64_t rm = mix64(x.local ^ kEdgeSalt);
    uint32_t vv[K];
    vv[0] = v0;
    vv[1] = (s1 << lgs) + (uint32_t(rm) & smask);
    vv[2] = ((s1 + 1u) << lgs) + (uint32_t(rm >> 32) & smask);
    if constexpr (K == 4) vv[3] = ((s1 + 2u) << lgs) + (uint32_t(mix64(x.local ^ kEdgeSalt2)) & smask);
    bool past = false;
#pragma unroll
    for (int k = 0; k < K - 1; k++) {
        past = past || vv[k] == x.v;
        x.o[k] = past ? vv[k + 1] : vv[k];
    }
    x.on = !((x.cold >> ((uint32_t(st0) + x.e) & 31u)) & 1u);
}

// The entry's record, in shard slot `slot`.
template <int K, bool VAL>
__device__ __forceinline__ void front_record(const FrontItem<K>& x, const FrontArgs& a, uint32_t base, uint32_t cells, uint32_t slot) {
    if (slot >= cells) return;  // at most one entry per vertex: impossible, and reported by the caller
    uint4* const rec = a.rec + base + slot;
    if (x.on) {
        *rec = make_uint4(base + x.v, base + x.o[0], base + x.o[1],
                          VAL ? x.value : fingerprint_slice(x.local, a.g.b, a.g.fpb, a.g.fps));
        if constexpr (K == 4) a.rec3[uint64_t(base) + slot] = base + x.o[2];
    } else {
        rec->x = kFrHole;
    }
}

// ------------------------------------------------------------------ head

// List `list` (shard s, rank k of lg_cta: list s * C + k), buffer buf.
__device__ __forceinline__ uint2* front_list(const FrontArgs& a, uint32_t list, uint32_t buf) {
    return a.lists + (uint64_t(list) * 2 + buf) * a.list_cap;
}

// Round 0: the vertices of degree one, each list those of its share of the cells.
__global__ void __launch_bounds__(kFrHeadT) k_front_scan(FrontArgs a) {
    __shared__ uint32_t s_cnt;
    const uint32_t tid = threadIdx.x, lane = tid & 31u;
    const uint32_t C = 1u << a.lg_cta, list = blockIdx.x, s = list >> a.lg_cta, rank = list & (C - 1u);
    const uint32_t cells = uint32_t(a.g.cells), quads = cells / 4;
    if (tid == 0) s_cnt = 0;
    __syncthreads();
    const uint4* const W4 = reinterpret_cast<const uint4*>(a.W + uint64_t(s) * cells);
    const uint32_t per = (quads + C - 1) / C, q0 = min(quads, rank * per), q1 = min(quads, q0 + per);
    uint2* const out = front_list(a, list, 0);
    for (uint32_t c = q0 + (tid & ~31u); c < q1; c += kFrHeadT) {
        const uint32_t q = c + lane;
        const uint4 w = q < q1 ? __ldcg(W4 + q) : make_uint4(0, 0, 0, 0);
        const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
        uint32_t mine = 0;
#pragma unroll
        for (int j = 0; j < 4; j++) mine += (ws[j] & 31u) == 1u;
        uint32_t incl = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, d);
            if (lane >= uint32_t(d)) incl += y;
        }
        uint32_t at = 0;
        if (lane == 31 && incl) at = atomicAdd(&s_cnt, incl);
        at = __shfl_sync(0xFFFFFFFFu, at, 31) + incl - mine;
#pragma unroll
        for (int j = 0; j < 4; j++)
            if ((ws[j] & 31u) == 1u) {
                if (at < a.list_cap) out[at] = make_uint2(4u * q + j, ws[j] >> 5);
                else atomicOr(a.err, kErrFrontier);
                at++;
            }
    }
    __syncthreads();
    if (tid == 0) a.list_n[list] = min(s_cnt, a.list_cap);
}

// Round r of every list: entries in buffer r & 1, list_n[r], records behind rcv[r].
template <int K, bool VAL>
__global__ void __launch_bounds__(kFrHeadT) k_front_head(FrontArgs a, uint32_t r) {
    __shared__ uint32_t s_cnt;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, below = (1u << lane) - 1u;
    const uint32_t C = 1u << a.lg_cta, list = blockIdx.x, s = list >> a.lg_cta, rank = list & (C - 1u);
    const uint32_t lists = a.S << a.lg_cta;
    // Degrees that wrapped in the incidence make every word worthless as an index.
    if (*reinterpret_cast<const volatile uint32_t*>(a.err_before) != 0) return;
    if (tid == 0) s_cnt = 0;
    __syncthreads();
    const uint32_t cells = uint32_t(a.g.cells), base = s * cells;
    const uint32_t* const cnt = a.list_n + uint64_t(r) * lists;
    const uint32_t sz = lane < C ? __ldcg(cnt + (s << a.lg_cta) + lane) : 0u;
    const uint32_t before = __ldcg(a.rcv + uint64_t(r) * a.S + s);
    const uint32_t total = __reduce_add_sync(0xFFFFFFFFu, sz);
    const uint32_t at = before + __reduce_add_sync(0xFFFFFFFFu, lane < rank ? sz : 0u);
    const uint32_t n = __shfl_sync(0xFFFFFFFFu, sz, rank);
    const unsigned long long st0 = __ldg(a.start + s);
    const uint32_t ns = uint32_t(__ldg(a.start + s + 1) - st0);
    uint32_t* const W = a.W + base;
    const uint2* const in = front_list(a, list, r & 1u);
    uint2* const out = front_list(a, list, (r + 1) & 1u);
    if (rank == 0 && tid == 0) {
        a.rcv[uint64_t(r + 1) * a.S + s] = before + total;
        if (before + total > cells) atomicOr(a.err, kErrFrontier);
    }
    for (uint32_t i0 = tid & ~31u; i0 < n; i0 += kFrHeadT * kFrHeadPer) {
        FrontItem<K> x[kFrHeadPer];
        uint32_t w[kFrHeadPer][K - 1];
#pragma unroll
        for (uint32_t j = 0; j < kFrHeadPer; j++) {
            const uint32_t i = i0 + j * kFrHeadT + lane;
            x[j].on = false;
            if (i < n) front_fetch<K, VAL>(x[j], a, __ldcg(in + i), st0, ns);
        }
#pragma unroll
        for (uint32_t j = 0; j < kFrHeadPer; j++) {
            if (x[j].on) front_others(x[j], a.g, st0);
#pragma unroll
            for (int k = 0; k < K - 1; k++)
                w[j][k] = x[j].on ? atomicAdd(W + x[j].o[k], 0u - (1u + (x[j].e << 5))) : 0u;
        }
#pragma unroll
        for (uint32_t j = 0; j < kFrHeadPer; j++) {
            const uint32_t i = i0 + j * kFrHeadT + lane;
            if (i < n) front_record<K, VAL>(x[j], a, base, cells, at + i);
        }
        // one reservation per warp for all the pass frees
        unsigned m[kFrHeadPer][K - 1];
        uint32_t all = 0;
#pragma unroll
        for (uint32_t j = 0; j < kFrHeadPer; j++)
#pragma unroll
            for (int k = 0; k < K - 1; k++) {
                w[j][k] -= 1u + (x[j].e << 5);
                m[j][k] = __ballot_sync(0xFFFFFFFFu, x[j].on && (w[j][k] & 31u) == 1u);
                all += __popc(m[j][k]);
            }
        if (!all) continue;
        uint32_t to = 0;
        if (lane == 0) to = atomicAdd(&s_cnt, all);
        to = __shfl_sync(0xFFFFFFFFu, to, 0);
#pragma unroll
        for (uint32_t j = 0; j < kFrHeadPer; j++)
#pragma unroll
            for (int k = 0; k < K - 1; k++) {
                if ((m[j][k] >> lane) & 1u) {
                    const uint32_t q = to + __popc(m[j][k] & below);
                    if (q < a.list_cap) out[q] = make_uint2(x[j].o[k], w[j][k] >> 5);
                    else atomicOr(a.err, kErrFrontier);
                }
                to += __popc(m[j][k]);
            }
    }
    __syncthreads();
    if (tid == 0) a.list_n[uint64_t(r + 1) * lists + list] = min(s_cnt, a.list_cap);
}

// ------------------------------------------------------------------ waves

// An entry for CTA `peer` of the cluster: its next list is list[] here, cnt its counter (rare: kept out of line).
__device__ __noinline__ void front_deal(const FrontArgs& a, uint32_t cnt, uint32_t list, uint2* beyond, uint32_t peer, uint2 ve) {
    uint32_t ps;
    asm volatile("atom.relaxed.cluster.shared::cluster.add.u32 %0, [%1], 1;"
                 : "=r"(ps)
                 : "r"(map_to_cta(cnt, peer))
                 : "memory");
    if (ps < kFrList) {
        asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(map_to_cta(list + 8u * ps, peer)), "r"(ve.x), "r"(ve.y)
                     : "memory");
    } else if (ps < a.list_cap) {
        beyond[ps] = ve;
    } else {
        atomicOr(a.err, kErrFrontier);
    }
}

// Whether a round whose largest CTA holds `most` of `total` entries deals out what
// it frees: beyond 1.25 times the mean and 48 more (4-uniform 10^8, ~150 entries a
// CTA: 16.9 ms at twice the mean + 64, 12.2 at 1.25 times + 16; 3-uniform, ~64 a
// CTA: 26.1 and 27.1, so the constant keeps small rounds from dealing often).
__device__ __forceinline__ bool front_uneven(uint32_t most, uint32_t total, uint32_t lg_cta) {
    return 4u * most > 5u * (total >> lg_cta) + 4u * 48u;
}

struct FrontShared {
    uint2 list[2][kFrList];                    // (vertex, edge), both shard-local
    __align__(16) uint32_t size[2][kFrMaxC];   // frontier sizes of the round, one per CTA
    __align__(8) unsigned long long mbar[2];   // exchange of even and of odd rounds
    uint32_t cnt[3];                           // frontier counts; round r counts its next one in cnt[(r + 1) % 3]
    uint32_t deal;                             // entries dealt out by this CTA so far
    uint32_t total[2], most[2];                // of the exchange of even and odd rounds: all entries, the largest CTA's
    uint32_t fail[2];                          // a wait of that exchange gave up
    uint2 mark[kFrMaxC];                       // by a CTA whose wait did: the cluster barrier it comes to next (they
                                               // are counted from 1), its exchanges so far
};

// K: vertices per edge (3, or 4 for a 4-uniform fuse graph). VAL: a function.
// ROUNDS: notes where each round's records start (0.5% of the peel at 10^8 keys).
template <int K, bool VAL, bool ROUNDS>
__global__ void __launch_bounds__(kFrT) k_front_peel(FrontArgs a) {
    __shared__ FrontShared sh;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, below = (1u << lane) - 1u;
    uint32_t rank, C, cid, ncl;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
    asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(cid));
    asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(ncl));
    // What earlier launches reported (the same in all CTAs) voids the attempt.
    if (*reinterpret_cast<const volatile uint32_t*>(a.err_before) != 0) return;
    const uint32_t cells = uint32_t(a.g.cells);
    const uint32_t lgs = uint32_t(a.g.lg_seg);
    const bool exchanger = warp == kFrWork / 32;
    const uint32_t mbar_addr = smem_u32(&sh.mbar[0]);
    // where this CTA's size goes in the CTA of this lane's number, and that CTA's mbarrier
    const uint32_t to_size = map_to_cta(smem_u32(&sh.size[0][rank]), lane < C ? lane : 0u);
    const uint32_t to_mbar = map_to_cta(mbar_addr, lane < C ? lane : 0u);
    if (tid == 0) {
        for (int j = 0; j < 2; j++)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar_addr + 8u * j) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        sh.deal = sh.fail[0] = sh.fail[1] = 0;
        for (uint32_t j = 0; j < kFrMaxC; j++) sh.mark[j] = make_uint2(0, 0);
    }
    uint32_t xr = 0;  // exchanges so far: mbar[xr & 1], whose phase parity is (xr >> 1) & 1
    // This CTA's size for exchange x to every CTA (the exchanger's).
    auto post = [&](uint32_t x, uint32_t n) {
        const uint32_t p = x & 1u;
        if (lane < C) post_u32(to_size + 4u * kFrMaxC * p, n, to_mbar + 8u * p);
        if (lane == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar_addr + 8u * p), "r"(4u * C)
                         : "memory");
    };
    // Waits for exchange x, for `most` tests. (The first one on its own: with the limit
    // compared in the only loop the peel takes 1.5% longer, 2^20 keys 2.63 against 2.59 ms.)
    auto await = [&](uint32_t x, uint32_t most) {
        const uint32_t mb = mbar_addr + 8u * (x & 1u), parity = (x >> 1) & 1u;
        if (mbar_try(mb, parity)) return;
        uint32_t polls = 0;
        while (!mbar_try(mb, parity)) {
            if (++polls > most) {
                sh.fail[x & 1u] = 1;
                break;
            }
        }
    };
    uint32_t bars = 0, gone = 0;  // cluster barriers so far; the most exchanges a CTA that gave up had posted
    // A cluster barrier; true, for all CTAs alike: a wait ran out, leave.
    auto meet = [&]() {
        cluster_barrier();
        bars++;
        const volatile uint2& m = sh.mark[lane & (kFrMaxC - 1u)];
        gone = __reduce_max_sync(0xFFFFFFFFu, m.x == bars ? m.y : 0u);
        return gone != 0;
    };
    for (uint32_t s = cid; s < a.S; s += ncl) {
        const uint32_t base = s * cells;
        const unsigned long long st0 = __ldg(a.start + s);
        const uint32_t ns = uint32_t(__ldg(a.start + s + 1) - st0);
        uint32_t* const W = a.W + base;
        // a list beyond shared memory goes on at the same index of this CTA's list of the head
        uint2* const list0 = front_list(a, s * C + rank, 0);
        auto put = [&](uint32_t buf, uint32_t i, uint2 x) {
            if (i < kFrList) sh.list[buf][i] = x;
            else if (i < a.list_cap) list0[buf * a.list_cap + i] = x;
            else atomicOr(a.err, kErrFrontier);
        };
        // kFrontHead is even: the head left its entries in buffer 0
        const uint32_t left = __ldcg(a.list_n + uint64_t(kFrontHead) * (a.S << a.lg_cta) + s * C + rank);
        for (uint32_t i = tid; i < left && i < kFrList; i += kFrT) sh.list[0][i] = __ldcg(list0 + i);
        if (tid < 3) sh.cnt[tid] = tid == 0 ? left : 0u;
        __syncthreads();
        if (meet()) break;  // every CTA's counters (and at first its mbarriers) are ready
        uint32_t before = __ldcg(a.rcv + uint64_t(kFrontHead) * a.S + s);  // record slots taken so far
        // segments whose words and signatures have been asked for: [0, pf_lo) and (pf_hi, T)
        int pf_lo = 0, pf_hi = int(cells >> lgs) - 1;
        uint32_t c0 = 0, c1 = 1, c2 = 2;  // r % 3, (r + 1) % 3, (r + 2) % 3
        uint32_t rounds = 0;  // (the exchanger's)
        bool done = false;
        for (uint32_t cur = 0;; cur ^= 1u) {
            uint32_t n = sh.cnt[c0];
            n = min(n, max(a.list_cap, kFrList));
            const uint32_t x0 = xr++, p = x0 & 1u;
            if (exchanger) {
                if (lane == 0) sh.cnt[c2] = 0;  // last read a round ago; pushed to from the next round on
                post(x0, n);
                if (n > 0) {
                    // while the sizes are on their way: what the waves reach next comes to L2
                    const bool have = lane < n;
                    const uint32_t sg = have ? sh.list[cur][lane].x >> lgs : 0u;
                    const uint32_t T = cells >> lgs;
                    const unsigned ml = __ballot_sync(0xFFFFFFFFu, have && sg < T / 2);
                    const unsigned mr = __ballot_sync(0xFFFFFFFFu, have && sg >= T / 2);
                    const int suml = int(__reduce_add_sync(0xFFFFFFFFu, have && sg < T / 2 ? sg : 0u));
                    const int sumr = int(__reduce_add_sync(0xFFFFFFFFu, have && sg >= T / 2 ? sg : 0u));
                    int t = -1;
                    if (ml && pf_lo < int(T) && (pf_lo - int(a.ahead)) * __popc(ml) <= suml) t = pf_lo++;
                    else if (mr && pf_hi >= 0 && (pf_hi + int(a.ahead)) * __popc(mr) >= sumr) t = pf_hi--;
                    if (t >= 0 && lane == 0) {
                        const uint32_t part = (1u << lgs) >> a.lg_cta;  // words of this CTA's share
                        if (part >= 32)
                            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(W + (uint32_t(t) << lgs) + rank * part),
                                         "r"(part * 4u)
                                         : "memory");
                        const uint32_t pe = a.epsg >> a.lg_cta;  // of ~epsg edges that start in a segment
                        const uint64_t e0 = (st0 + uint64_t(t) * a.epsg + rank * pe) & ~uint64_t(1);
                        const uint32_t bytes = (pe * 8u) & ~15u;
                        if (bytes && e0 + bytes / 8 <= st0 + ns)
                            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a.loc + e0), "r"(bytes) : "memory");
                    }
                }
                await(x0, a.polls);
                const uint32_t sz = lane < C ? sh.size[p][lane] : 0u;
                const uint32_t total = __reduce_add_sync(0xFFFFFFFFu, sz), most = __reduce_max_sync(0xFFFFFFFFu, sz);
                if (lane == 0) sh.total[p] = total, sh.most[p] = most;
                if (ROUNDS && rank == 0 && lane == 0) {  // where the round's records start, for the assignment
                    if (total == 0) a.rc[s * kRcStride + 1] = rounds;
                    else if (rounds < kFrontRounds) a.round[uint64_t(s) * kFrontRounds + rounds] = before;
                    rounds++;
                }
            } else {
                uint32_t i = tid;
                FrontItem<K> x;
                x.on = false;
                auto entry = [&]() { return i < kFrList ? sh.list[cur][i] : __ldcg(list0 + cur * a.list_cap + i); };
                if (i < n) front_fetch<K, VAL>(x, a, entry(), st0, ns);
                if (x.on) front_others(x, a.g, st0);
                // (in vain: the round is finished with sizes as they are, which decide only where
                // records and pushes go, within their rooms: a vote that told a warp's lanes so
                // would cost every round)
                await(x0, a.polls);
                uint32_t at = 0;
                bool deal = false;
                for (uint32_t i0 = 32u * warp; i0 < n; i0 += kFrWork) {
                    uint32_t w[K - 1];
                    const uint32_t dec = 1u + (x.e << 5);
#pragma unroll
                    for (int k = 0; k < K - 1; k++) w[k] = x.on ? atomicAdd(W + x.o[k], 0u - dec) : 0u;
                    if (i0 == 32u * warp) {  // while the removals are on their way: where the round's records go
                        const uint32_t sz = lane < C ? sh.size[p][lane] : 0u;
                        const uint32_t total = __reduce_add_sync(0xFFFFFFFFu, sz);
                        at = before + __reduce_add_sync(0xFFFFFFFFu, lane < rank ? sz : 0u);
                        deal = front_uneven(__reduce_max_sync(0xFFFFFFFFu, sz), total, a.lg_cta);
                    }
                    if (i < n) front_record<K, VAL>(x, a, base, cells, at + i);
                    // the vertices left at degree one join the next list
                    unsigned m[K - 1];
                    uint32_t all = 0;
#pragma unroll
                    for (int k = 0; k < K - 1; k++) {
                        w[k] -= dec;
                        m[k] = __ballot_sync(0xFFFFFFFFu, x.on && (w[k] & 31u) == 1u);
                        all += __popc(m[k]);
                    }
                    if (all) {
                        uint32_t to = 0;
                        if (lane == 0) to = atomicAdd(deal ? &sh.deal : &sh.cnt[c1], all);
                        to = __shfl_sync(0xFFFFFFFFu, to, 0);
#pragma unroll
                        for (int k = 0; k < K - 1; k++) {
                            if ((m[k] >> lane) & 1u) {
                                const uint32_t slot = to + __popc(m[k] & below);
                                const uint2 ve = make_uint2(x.o[k], w[k] >> 5);
                                if (!deal) {
                                    put(cur ^ 1u, slot, ve);
                                } else {  // to the CTAs of the cluster in turn
                                    const uint32_t peer = (slot + rank) & (C - 1u);
                                    front_deal(a, smem_u32(&sh.cnt[c1]), smem_u32(&sh.list[cur ^ 1u][0]),
                                               front_list(a, s * C + peer, cur ^ 1u), peer, ve);
                                }
                            }
                            to += __popc(m[k]);
                        }
                    }
                    i += kFrWork;
                    x.on = false;
                    if (i < n) {
                        front_fetch<K, VAL>(x, a, entry(), st0, ns);
                        if (x.on) front_others(x, a.g, st0);
                    }
                }
            }
            __syncthreads();
            // equal in every CTA that knows the round's sizes, and so are the ways out behind the first
            const uint32_t total = sh.total[p], gave_up = sh.fail[p];
            if (gave_up) {  // (the other exchange's flag is set behind the next barrier at the earliest)
                if (tid == 0) atomicOr(a.err, kErrTimeout);
                if (tid < C)
                    asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(map_to_cta(smem_u32(&sh.mark[rank]), tid)),
                                 "r"(bars + 1u), "r"(xr)
                                 : "memory");
                break;
            }
            if (total == 0) {
                if (rank == 0 && tid == 0) a.rc[s * kRcStride] = before;
                break;
            }
            before += total;
            if (before > cells) {
                if (tid == 0) atomicOr(a.err, kErrFrontier);
                break;
            }
            if (front_uneven(sh.most[p], total, a.lg_cta)) {  // this round's pushes were dealt out
                done = meet();
                if (done) break;
            }
            const uint32_t t = c0;
            c0 = c1, c1 = c2, c2 = t;
        }
        if (done || meet()) break;  // no CTA starts the next shard (or leaves) while a peer still works on this one
    }
    // After a wait ran out: sizes may be on their way still. The CTAs are at most one
    // exchange apart (the next one takes a size of all), so those behind post it too,
    // and no CTA ends before all of both exchanges' sizes have come to it.
    if (gone && exchanger) {
        if (xr < gone) post(xr, 0);
        if (gone > 1) await(gone - 2, kFrontPolls);
        await(gone - 1, kFrontPolls);
    }
}

// ------------------------------------------------------------ assignment

// The records of one round depend on no other of the round: an edge's other
// vertices are freed by its removal, so what is peeled from them comes in a later
// round. So the rounds go back one by one, the waves' by the shard's cluster with a
// cluster barrier behind each, the head's in a launch each; the cells themselves
// hold the values.
// A round of the waves is one trip to L2 for the two values, whose records were
// loaded two rounds ahead, and one barrier; the worklist's dataflow polls a value
// word written by another SM. Measured (b = 8, dataflow -> this): 10^9 keys 62 -> 27
// ms, 4-uniform 8*10^8 38 -> 24. Asking L2 for the next round's cells a round ahead
// was slower (27 -> 34): a CTA's requests, some 200 a round, already count.
constexpr int kFrAssignT = 128;

// The answer of a record: its value and the cells of the edge's other vertices.
template <int K, class T>
__device__ __forceinline__ void front_put(T* cells, uint4 q, uint32_t q3) {
    if (q.x == kFrHole) return;
    uint32_t x = q.w ^ __ldcg(cells + q.y) ^ __ldcg(cells + q.z);
    if constexpr (K == 4) x ^= __ldcg(cells + q3);
    cells[q.x] = T(x);
}

template <int K, class T>
__global__ void __launch_bounds__(kFrAssignT) k_front_assign(FrontArgs a, T* cells) {
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    uint32_t rank, C, s;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
    asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(s));
    const uint32_t end = __ldg(a.rc + s * kRcStride), R = __ldg(a.rc + s * kRcStride + 1);
    const uint32_t* const off = a.round + uint64_t(s) * kFrontRounds;
    const uint4* const rec = a.rec + uint64_t(s) * a.g.cells;
    const uint32_t* const rec3 = K == 4 ? a.rec3 + uint64_t(s) * a.g.cells : nullptr;
    // bound(0), bound(1): the ends of the last round, and so on back
    auto bound = [&](uint32_t k) { return k == 0 ? end : __ldg(off + R - min(k, R)); };
    const uint32_t me = ((warp * C + rank) << 5) + lane, step = C * kFrAssignT;
    auto load = [&](uint32_t i, uint32_t hi, uint4& q, uint32_t& q3) {
        q.x = kFrHole;
        if (i >= hi) return;
        q = __ldcg(rec + i);
        if constexpr (K == 4) q3 = __ldcg(rec3 + i);
    };
    if (R == 0) return;
    uint32_t b0 = bound(0), b1 = bound(1), b2 = bound(2), b3 = bound(3);
    uint4 q, q1, q2;
    uint32_t t = 0, t1 = 0, t2 = 0;
    load(b1 + me, b0, q, t);
    load(b2 + me, b1, q1, t1);
    for (uint32_t k = 0; k < R; k++) {
        const uint32_t b4 = bound(k + 4);
        load(b3 + me, b2, q2, t2);
        front_put<K, T>(cells, q, t);
        for (uint32_t i = b1 + me + step; i < b0; i += step) {
            uint4 x;
            uint32_t x3 = 0;
            load(i, b0, x, x3);
            front_put<K, T>(cells, x, x3);
        }
        cluster_barrier();
        q = q1, q1 = q2, t = t1, t1 = t2;
        b0 = b1, b1 = b2, b2 = b3, b3 = b4;
    }
}

// Round r of the head, every shard's records over gridDim.x / S blocks.
template <int K, class T>
__global__ void __launch_bounds__(kFrWork) k_front_head_assign(FrontArgs a, T* cells, uint32_t r) {
    const uint32_t per = gridDim.x / a.S, s = blockIdx.x / per;
    const uint32_t lo = __ldg(a.rcv + uint64_t(r) * a.S + s), hi = __ldg(a.rcv + uint64_t(r + 1) * a.S + s);
    const uint64_t base = uint64_t(s) * a.g.cells;
    const uint32_t step = per * kFrWork;
    for (uint64_t i = uint64_t(lo) + (blockIdx.x % per) * kFrWork + threadIdx.x; i < hi; i += kFrHeadPer * step) {
        uint4 q[kFrHeadPer];
        uint32_t q3[kFrHeadPer], x[kFrHeadPer];
#pragma unroll
        for (uint32_t j = 0; j < kFrHeadPer; j++) {
            const uint64_t at = i + uint64_t(j) * step;
            q[j] = make_uint4(kFrHole, 0, 0, 0);
            q3[j] = 0;
            if (at < hi) {
                q[j] = __ldcs(a.rec + base + at);
                if constexpr (K == 4) q3[j] = __ldcs(a.rec3 + base + at);
            }
        }
#pragma unroll
        for (uint32_t j = 0; j < kFrHeadPer; j++) {
            x[j] = q[j].w;
            if (q[j].x == kFrHole) continue;
            x[j] ^= __ldcg(cells + q[j].y) ^ __ldcg(cells + q[j].z);
            if constexpr (K == 4) x[j] ^= __ldcg(cells + q3[j]);
        }
#pragma unroll
        for (uint32_t j = 0; j < kFrHeadPer; j++)
            if (q[j].x != kFrHole) cells[q[j].x] = T(x[j]);
    }
}

// ------------------------------------------------------------------ launches

template <int K, bool VAL>
static const void* front_kernel(bool rounds) {
    return rounds ? reinterpret_cast<const void*>(k_front_peel<K, VAL, true>)
                  : reinterpret_cast<const void*>(k_front_peel<K, VAL, false>);
}
static const void* front_kernel(const Geom& g, bool rounds) {
    const bool val = g.kind == 0;
    if (g.k == 4) return val ? front_kernel<4, true>(rounds) : front_kernel<4, false>(rounds);
    return val ? front_kernel<3, true>(rounds) : front_kernel<3, false>(rounds);
}

static cudaLaunchConfig_t front_launch(unsigned cta, unsigned clusters, cudaStream_t st, cudaLaunchAttribute* at,
                                       unsigned threads = kFrT) {
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3(cta * clusters);
    lc.blockDim = dim3(threads);
    lc.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cta;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeClusterSchedulingPolicyPreference;
    at[1].val.clusterSchedulingPolicyPreference = cudaClusterSchedulingPolicyLoadBalancing;
    lc.attrs = at;
    lc.numAttrs = 2;
    return lc;
}

// Where the clusters are faster than the worklist. The worklist has the whole chip at
// work on whatever is ready; a cluster has 16 SMs for its shard and a round's latency
// for its few entries (about 2^(lg_seg - 5); 2^(lg_seg - 3) where the graph is
// 4-uniform). Peel and assignment of an attempt, ms, worklist and clusters:
//  * a few large shards leave most SMs idle, in the head's rounds above all. 3-uniform,
//    one shard: 2^14 cells a segment 4.9, 4.6 (4*10^6 cells), 2^15 5.3, 5.6 (8*10^6), 2^16 9.1,
//    13.8; two: 2^16 20.4, 19.9, 2^17 25.2, 24.9 and 25.8, 32.4 (3, 5*10^7 cells each); four:
//    2^17 34.9, 30.1 and 40.2, 41.3, 2^18 70, 53. 4-uniform: one or two shards: 2^13 10.4, 9.4
//    (one), 10.8, 10.0 (two), 2^14 7.7, 8.4, 8.3, 9.0; four: 2^13 11.7, 10.7, 2^14 9.6, 9.8 and 18.5,
//    19.6, 2^15 40.8, 45.0, 2^16 (beyond L2, where the worklist's wide front costs) 57.6, 51.4; eight: 2^14
//    27.2, 23.8, 2^15 42.6, 28.7.
//  * shards beyond the clusters resident at once (36) wait for one another. 4-uniform,
//    64 shards: 2^10 2.9, 3.6, 2^11 5.4, 4.9, 2^12 11.0, 7.9; 256: 2^10 11.8, 11.9, 2^11 23.0,
//    17.7; 1024: 2^9 8.1, 14.6, 2^10 42, 48, 2^11 89, 65.
//  * rounds of one or two entries a CTA: 16 shards of 11520 cells 0.28, 0.30, of 22272 0.56,
//    0.52.
static bool front_pays(const Geom& g, uint32_t S, uint32_t clusters) {
    if (S > clusters) return g.lg_seg >= 11;
    if (g.cells < 1u << 14) return false;
    if (S >= 8) return true;
    if (g.k == 4) return g.lg_seg <= 13 || (S >= 4 && g.lg_seg >= 16);
    return S >= 4 || g.lg_seg <= (S == 1 ? 14 : 16);
}

bool front_config(const Geom& g, uint32_t S, FrontConfig& cfg) {
    if (g.regime != kRegimeFuse || (g.k != 3 && g.k != 4) || g.lg_seg < 5 || g.lg_seg > 26) return false;
    static std::mutex mu;
    static FrontConfig known[8][64];  // per kernel and device: cta = 0 unknown, ~0u not able
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    const bool rounds = front_assign_fits(g, S);
    const void* fn = front_kernel(g, rounds);
    std::lock_guard<std::mutex> lock(mu);
    FrontConfig& k = known[(rounds ? 4 : 0) + (g.k == 4 ? 2 : 0) + (g.kind == 0 ? 1 : 0)][dev];
    if (k.cta == 0) {
        k.cta = ~0u;
        for (bool r : {false, true})  // (the fault hooks take the one without rounds)
            if (cudaFuncSetAttribute(front_kernel(g, r), cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
                cudaGetLastError();
        for (unsigned c : {kFrMaxC, 8u}) {
            cudaLaunchAttribute at[2]{};
            const cudaLaunchConfig_t lc = front_launch(c, 1, nullptr, at);
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, fn, &lc) == cudaSuccess && n > 0) {
                k.cta = c;
                k.clusters = unsigned(n);
                break;
            }
            cudaGetLastError();
        }
    }
    if (k.cta == ~0u || !front_pays(g, S, k.clusters)) return false;
    cfg.cta = k.cta;
    cfg.clusters = std::max(1u, std::min(S, k.clusters));
    return true;
}

cudaError_t launch_front_peel(const FrontArgs& a, const FrontConfig& cfg, cudaStream_t st) {
    const unsigned lists = a.S << a.lg_cta;
    k_front_scan<<<lists, kFrHeadT, 0, st>>>(a);
    for (uint32_t r = 0; r < kFrontHead; r++) {
        if (a.g.k == 4) {
            if (a.g.kind == 0) k_front_head<4, true><<<lists, kFrHeadT, 0, st>>>(a, r);
            else k_front_head<4, false><<<lists, kFrHeadT, 0, st>>>(a, r);
        } else {
            if (a.g.kind == 0) k_front_head<3, true><<<lists, kFrHeadT, 0, st>>>(a, r);
            else k_front_head<3, false><<<lists, kFrHeadT, 0, st>>>(a, r);
        }
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at[2]{};
    const cudaLaunchConfig_t lc = front_launch(cfg.cta, cfg.clusters, st, at);
    void* args[] = {const_cast<FrontArgs*>(&a)};
    return cudaLaunchKernelExC(&lc, front_kernel(a.g, a.round != nullptr), args);
}

// A round here costs more than a level of the dataflow (~1.6 against ~1.1 us: a
// barrier behind every store), whatever it holds; the dataflow's polls cost more
// the more records are under way at once. The line lies where the shards' segments
// hold 2^20 cells together (4-uniform graphs, whose rounds are some four times as
// wide: 2^18), ms, dataflow and rounds: 10^8 8.9, 12.7; 3*10^8 (2^20) 14.7, 14.8;
// 4*10^8 (2^20) 21.1, 23.6; 6*10^8 (2^21) 30.1, 18.5; 10^9 (2^22) 62, 27; 4-uniform
// 2*10^8 (2^18) 11.3, 11.8; 4*10^8 (2^19) 19.7, 14.6 (the head's records in launches of
// their own take a seventh off the dataflow and leave the line where it is).
constexpr uint64_t kRoundCells = 1u << 20;

bool front_assign_fits(const Geom& g, uint32_t S) {
    if ((g.b != 8 && g.b != 16 && g.b != 32) || S > kFrontRoundShards) return false;
    return (uint64_t(S) << g.lg_seg) << (g.k == 4 ? 2 : 0) > kRoundCells;
}

template <int K, class T>
static cudaError_t assign_head(const FrontArgs& a, T* cells, cudaStream_t st) {
    const unsigned per = std::max(8u, (num_sms() * 8u + a.S - 1) / a.S);
    for (uint32_t r = kFrontHead; r-- > 0;) k_front_head_assign<K, T><<<a.S * per, kFrWork, 0, st>>>(a, cells, r);
    return cudaGetLastError();
}

template <int K, class T>
static cudaError_t assign_rounds(const FrontArgs& a, const FrontConfig& cfg, T* cells, cudaStream_t st) {
    const auto waves = k_front_assign<K, T>;
    cudaError_t e = cudaFuncSetAttribute(waves, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    // a cluster per shard: none waits for another, so they need not all be resident
    cudaLaunchAttribute at[2]{};
    const cudaLaunchConfig_t lc = front_launch(cfg.cta, a.S, st, at, kFrAssignT);
    e = cudaLaunchKernelEx(&lc, waves, a, cells);
    return e != cudaSuccess ? e : assign_head<K>(a, cells, st);
}

template <class T>
static cudaError_t assign_cells(const FrontArgs& a, const FrontConfig* cfg, T* cells, cudaStream_t st) {
    if (!cfg) return a.g.k == 4 ? assign_head<4>(a, cells, st) : assign_head<3>(a, cells, st);
    return a.g.k == 4 ? assign_rounds<4>(a, *cfg, cells, st) : assign_rounds<3>(a, *cfg, cells, st);
}

cudaError_t launch_front_assign(const FrontArgs& a, const FrontConfig* cfg, uint8_t* data, uint64_t cell_base, cudaStream_t st) {
    if (a.g.b == 8) return assign_cells(a, cfg, data + cell_base, st);
    if (a.g.b == 16) return assign_cells(a, cfg, reinterpret_cast<uint16_t*>(data) + cell_base, st);
    return assign_cells(a, cfg, reinterpret_cast<uint32_t*>(data) + cell_base, st);
}

}  // namespace vf
