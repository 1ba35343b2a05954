// LGE-regime solver of libvfunc (sm_103a): one CTA per shard, shards taken
// from a global counter so uneven shards balance across SMs.
//
// Per shard, all synchronisation is block barriers (no spin-waits):
//  1. incidence: degree (8-bit lanes) and XOR of shard-local edge indices
//     (16-bit lanes) per vertex, in shared memory (Sec. 4.3, XOR trick);
//  2. peeling in synchronous rounds; each round first reads every frontier
//     vertex's (degree, XOR) and only then removes edges, so a vertex's only
//     edge is read consistently; edges are claimed with a bit per edge;
//  3. lazy Gaussian elimination of the 2-core (Sec. 3.3, GOV): variables start
//     idle; an equation with one idle variable is solved for it and the
//     variable is eliminated from the other equations; when none is left, the
//     heaviest idle variables are made active (a batch of ~2.5% of the open
//     equations at a time); equations left with no idle variable form the
//     dense system over the active variables;
//  4. the dense equations are carried back through the solves, 32 at a time
//     with one word per variable in shared memory, until only active variables
//     are left in them; the dense rows are reduced a word of columns at a time
//     (free variables = 0); the solved variables are then evaluated forward
//     and the peeled edges' vertices in reverse peel order, all in shared
//     memory, and the cells stored once.
//
// What bounds it: the latency of a shard's dependent steps (a 9.8K-key shard has
// ~25 peel rounds, ~112 elimination rounds, ~100 rounds of solves to walk back and
// forth, ~11 panels), not bandwidth; several CTAs per SM overlap several shards,
// and issue slots are 38% taken at 8192-key shards. So every step is made of
// few barriers, on-chip words and loads sent ahead. Measured (one GB300): one
// 10^4-key build 1836 -> 593 us; 10^7 strings in 1024 shards 9.86 -> 3.8 ms for
// the whole build; 512 batched structures 49.9 -> 28.1 ms with this kernel alone.
//
// Three configurations of the kernel share this code. Shards of at most
// kLgeSmallTaskKeys keys run in the small configuration (192 threads, 72 KB of
// shared memory, three CTAs per SM), larger ones in the medium one (256
// threads, 108 KB, two per SM). A shard whose arrays do not fit is handed,
// unchanged, to the spill list, which the large configuration (512 threads, 200
// KB, one CTA per SM) then solves from the start: all solve the same system, so
// which one ran changes neither the outcome nor the retry count. A launch of no
// more shards than SMs uses the large configuration alone: with an SM to itself
// a shard is done sooner by 512 threads. A shard beyond the solver's pool (active
// variables, dense rows) fails with kErrLgeSize, a capacity error that ends the
// build rather than a retry.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "vf_internal.h"

namespace vf {

constexpr uint32_t kMaxBatch = 256;
// large configuration: 512 threads, 200 KB dynamic shared memory, 1 CTA per SM
constexpr int kBigT = 512;
constexpr uint32_t kBigWords = 50 * 1024;
// medium configuration: 256 threads, 108 KB, 2 CTAs per SM
constexpr int kMidT = 256;
constexpr uint32_t kMidWords = 27 * 1024;
// small configuration: 192 threads, 72 KB, 3 CTAs per SM
constexpr int kSmallT = 192;
constexpr uint32_t kSmallWords = 18 * 1024;
constexpr uint32_t kNone = 0xFFFFFFFFu;
// equation words: the sum of up to three 16-bit variables in bits 3..20, and a mark
constexpr uint32_t kSumMask = 0x001FFFF8u;
constexpr uint32_t kTwin = 0x80000000u;
constexpr uint32_t kLgSeen = 16, kSeenWords = 1u << (kLgSeen - 5);

uint64_t lge_scratch_words_per_cta(uint32_t m_cap, uint32_t v_cap) { return lge_offsets(m_cap, v_cap).total; }

__device__ __forceinline__ uint32_t rhs_of(const LgeArgs& a, const LgeTask& t, uint64_t ge) {
    return t.kind == 0 ? __ldg(a.val + ge) : fingerprint_slice(__ldg(a.loc + ge), t.b, t.fpb, t.fps);
}

__device__ __forceinline__ uint32_t deg_of(const uint32_t* degw, uint32_t v) {
    return (degw[v >> 2] >> ((v & 3u) * 8u)) & 255u;
}
__device__ __forceinline__ uint32_t xr_of(const uint32_t* xrw, uint32_t v) {
    return (xrw[v >> 1] >> ((v & 1u) * 16u)) & 0xFFFFu;
}

// Exclusive scan of cnt[0..len) by one CTA; part: one word per warp of scratch.
// Each thread takes a run of consecutive entries.
__device__ void cta_exclusive_scan(uint32_t* cnt, uint32_t len, uint32_t* part) {
    const uint32_t T = blockDim.x, tid = threadIdx.x, lane = tid & 31u;
    const uint32_t chunk = (len + T - 1) / T;
    const uint32_t lo = min(len, tid * chunk), hi = min(len, lo + chunk);
    uint32_t sum = 0;
    for (uint32_t i = lo; i < hi; i++) sum += cnt[i];
    uint32_t incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= uint32_t(d)) incl += y;
    }
    if (lane == 31) part[tid >> 5] = incl;
    __syncthreads();
    uint32_t run = incl - sum;
    for (uint32_t w = 0; w < (tid >> 5); w++) run += part[w];
    for (uint32_t i = lo; i < hi; i++) {
        const uint32_t x = cnt[i];
        cnt[i] = run;
        run += x;
    }
    __syncthreads();
}

// Barrier `id` (1..15) of n threads.
__device__ __forceinline__ void bar_some(uint32_t id, uint32_t n) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// A slot of *ctr for every lane with `p` (one shared atomic per warp; all
// lanes of the warp call it).
__device__ __forceinline__ uint32_t warp_slot(uint32_t* ctr, bool p) {
    const unsigned m = __ballot_sync(0xFFFFFFFFu, p);
    if (m == 0) return 0;
    const unsigned lane = threadIdx.x & 31u;
    const int lead = __ffs(m) - 1;
    uint32_t at = 0;
    if (int(lane) == lead) at = atomicAdd(ctr, uint32_t(__popc(m)));
    return __shfl_sync(0xFFFFFFFFu, at, lead) + __popc(m & ((1u << lane) - 1u));
}

// The same for counters that differ by lane (key: which one): one atomic per
// distinct key of the warp's lanes with `p`.
__device__ __forceinline__ uint32_t warp_slot_by(uint32_t* ctrs, uint32_t key, bool p) {
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, p ? key : kNone);
    const unsigned lane = threadIdx.x & 31u;
    const int lead = __ffs(peers) - 1;
    uint32_t at = 0;
    if (p && int(lane) == lead) at = atomicAdd(ctrs + key, uint32_t(__popc(peers)));
    return __shfl_sync(0xFFFFFFFFu, at, lead) + __popc(peers & ((1u << lane) - 1u));
}

// Drops the 128-byte L2 lines wholly inside [p, p + words) without writing
// them back (discard.global.L2: the line's contents become undefined).
__device__ __forceinline__ void discard_words(const uint32_t* p, uint64_t words) {
    const uint64_t lo = (reinterpret_cast<uint64_t>(p) + 127u) & ~uint64_t(127);
    const uint64_t hi = (reinterpret_cast<uint64_t>(p + words)) & ~uint64_t(127);
    for (uint64_t x = lo + uint64_t(threadIdx.x) * 128u; x < hi; x += uint64_t(blockDim.x) * 128u)
        asm volatile("discard.global.L2 [%0], 128;" ::"l"(x) : "memory");
}

// Everything a shard wrote to the CTA's slab is dead once the shard is done,
// and every array is written before it is read by the next shard. Without
// this, the 304 slabs resident at once (more than L2 holds) are written back
// to DRAM line by line as they are evicted; discarding them instead keeps L2
// for live lines. `m`, `V`: the finished shard's keys and cells; `lused`:
// words of the dense system's pool it wrote.
__device__ void discard_slab(const uint32_t* scr, const LgeOffsets& o, uint32_t m, uint32_t V, uint64_t lused) {
    const uint64_t mm = m, vv = V;
    discard_words(scr + o.ev, 2 * mm);
    discard_words(scr + o.prec, 2 * mm);
    discard_words(scr + o.proff, vv + 2);
    discard_words(scr + o.lists, 3 * ((vv + 1) / 2));
    discard_words(scr + o.core, mm / 2);
    discard_words(scr + o.eqst, mm);
    discard_words(scr + o.inc_off, vv + 1);
    discard_words(scr + o.inc_list, 3 * mm / 2);
    discard_words(scr + o.vstate, vv);
    discard_words(scr + o.act, vv / 2);
    discard_words(scr + o.actv, o.a_cap);
    discard_words(scr + o.solves, mm);
    discard_words(scr + o.soff, mm + vv + 4);
    discard_words(scr + o.srec, 2 * mm);
    discard_words(scr + o.dense, mm);
    discard_words(scr + o.lc, mm);
    discard_words(scr + o.L, lused < o.lpool ? lused : o.lpool);
}

// Hands task s to the spill list (small configuration) and reports whether
// it did; the large configuration has no spill list and fails the shard.
__device__ __forceinline__ bool spill_task(const LgeArgs& a, uint32_t s) {
    if (!a.spill) return false;
    if (threadIdx.x == 0) a.spill[atomicAdd(&a.stats[5], 1u)] = s;
    return true;
}

template <int kLT, uint32_t kLgeSmemWords, int kMinBlocks>
__global__ void __launch_bounds__(kLT, kMinBlocks) k_lge(LgeArgs a) {
    extern __shared__ __align__(16) uint32_t sm[];
    __shared__ uint32_t s_shard, s_fail;
    __shared__ uint32_t s_cnt[4];
    __shared__ uint32_t s_C, s_nact, s_nbatch, s_dup;
    __shared__ uint32_t s_queue[4], s_solved[4], s_dense[4];  // the elimination's rounds
    __shared__ uint32_t s_hist[256];
    __shared__ uint32_t s_batch[kMaxBatch];
    __shared__ uint32_t s_part[kLT];
    __shared__ uint4 s_piv[32];    // a panel's pivots: row, reduced panel word, combination with itself, column
    __shared__ uint32_t s_pool[64];  // the rows it is looked for in
    __shared__ uint32_t s_tz[128];   // sums of four pivots' combinations, 16 for each four

    const uint32_t tid = threadIdx.x, T = blockDim.x;
    const unsigned lane = tid & 31u, warp = tid >> 5;
    const LgeOffsets o = lge_offsets(a.m_cap, a.v_cap);
    uint32_t* scr = a.scratch + uint64_t(blockIdx.x) * a.scratch_words_per_cta;
    uint2* ev = reinterpret_cast<uint2*>(scr + o.ev);      // an edge's vertices: v0 | v1 << 16, v2
    uint2* prec = reinterpret_cast<uint2*>(scr + o.prec);  // a peeled edge: its vertex | edge << 16, other | other << 16
    uint32_t* proff = scr + o.proff;
    uint16_t* core = reinterpret_cast<uint16_t*>(scr + o.core);
    uint32_t* eqst = scr + o.eqst;
    uint32_t* inc_off = scr + o.inc_off;
    uint16_t* inc_list = reinterpret_cast<uint16_t*>(scr + o.inc_list);
    uint32_t* vstate = scr + o.vstate;
    uint16_t* act = reinterpret_cast<uint16_t*>(scr + o.act);
    uint32_t* actv = scr + o.actv;
    uint32_t* solves = scr + o.solves;
    uint32_t* soff = scr + o.soff;
    uint2* srec = reinterpret_cast<uint2*>(scr + o.srec);  // a solve: variable | edge << 16, other | other << 16
    uint32_t* dense = scr + o.dense;
    uint32_t* lc = scr + o.lc;
    uint32_t* L = scr + o.L;
    // threads of the elimination's rounds: a round has ~50 solves, and a warp
    // without one still issues the round's instructions
    constexpr int kET = kLT < 256 ? kLT : 256;
    constexpr int kGT = kLT % 128 ? kLT / 2 : 128;  // and of a walk over the solves
    // the small configurations hand on a shard whose arrays do not all fit
    constexpr bool kSpills = kLgeSmemWords != kBigWords;
    constexpr uint32_t kBad = kErrUnsolvable | kErrCapacity | kErrLgeSize | kErrDegOverflow | kErrDupKey;

    // The large configuration behind a small one takes its tasks from the
    // spill list (written by the previous launch), otherwise from all tasks.
    const bool from_spill = a.spilled != nullptr;
    const uint32_t ntasks = from_spill ? *a.spilled : a.ntasks;
    // the previous shard's sizes, for discarding its slab lines (uniform)
    uint32_t prev_m = 0, prev_v = 0;
    uint64_t prev_l = 0;
    for (;;) {
        __shared__ uint32_t s_skip;
        // every path to here ends its shard with a barrier; the barrier below
        // orders the discards before the next shard's first slab write
        if (prev_m | prev_v) discard_slab(scr, o, prev_m, prev_v, prev_l);
        prev_m = prev_v = 0;
        prev_l = 0;
        if (tid == 0) {
            const uint32_t q = atomicAdd(&a.stats[from_spill ? 4 : a.ctr], 1u);
            s_shard = q < ntasks ? (from_spill ? a.spill_in[q] : a.task_lo + q) : kNone;
            s_skip = s_shard != kNone &&
                     (*reinterpret_cast<volatile uint32_t*>(a.item_fail + a.tasks[s_shard].item) & kBad) != 0;
            s_fail = 0;
            s_dup = 0;
        }
        __syncthreads();
        const uint32_t s = s_shard;
        if (s == kNone) break;
        if (s_skip) {  // another shard of this structure already failed: the attempt is void
            __syncthreads();
            continue;
        }
        const LgeTask task = a.tasks[s];
        const uint64_t e0 = task.loc_off;
        const uint32_t m = task.m;
        const uint32_t V = task.cells;
        const uint64_t cbase = task.cell_base;
        const int b = task.b;
        uint8_t* const data = task.data;
        Geom gg;
        gg.kh = gg.kl = 0;
        gg.cells = V;
        gg.span = 0;
        gg.lg_seg = 0;
        gg.h = 0;
        gg.regime = kRegimeLge;
        gg.b = b;
        gg.kind = task.kind;
        gg.fpb = task.fpb;
        gg.fps = task.fps;
        gg.k = 3;
        if (m > a.m_cap || V > a.v_cap || V > 65535u || m > 65535u) {
            // (nothing was written to the slab: prev_m, prev_v stay 0)
            if (tid == 0) {
                atomicOr(a.err, kErrCapacity);
                atomicOr(a.item_fail + task.item, kErrCapacity);
            }
            __syncthreads();
            continue;
        }

        // ---------------------------------------------------------------- 1. incidence
        uint32_t* degw = sm;
        uint32_t* xrw = degw + (V + 3) / 4;
        uint32_t* clm = xrw + (V + 1) / 2;
        const uint32_t pw = (V + 3) / 4 + (V + 1) / 2 + (m + 31) / 32;
        // (or of one whose solve records, ~0.6 a key, will not fit beside its values)
        if (pw > kLgeSmemWords || (kSpills && V + 6u * m / 5u > kLgeSmemWords && a.spill)) {
            if (!spill_task(a, s) && tid == 0) {
                atomicOr(a.err, kErrCapacity);
                atomicOr(a.item_fail + task.item, kErrCapacity);
            }
            __syncthreads();
            continue;
        }
        // frontier lists and the edges read off them: behind the counters when they fit
        const uint32_t lw = (V + 1) / 2;
        uint16_t* lists = reinterpret_cast<uint16_t*>(pw + 3 * lw <= kLgeSmemWords ? sm + pw : scr + o.lists);
        uint16_t* const cand = lists + 4 * lw;
        for (uint32_t i = tid; i < pw; i += T) sm[i] = 0;
        prev_m = m;  // the slab is written from here on
        prev_v = V;
        if (tid == 0) {
            s_cnt[0] = s_cnt[1] = s_cnt[2] = s_cnt[3] = 0;
            proff[0] = 0;
        }
        __syncthreads();
        for (uint32_t e = tid; e < m; e += T) {
            uint64_t v[4];
            edge_of(gg, __ldg(a.loc + e0 + e), v);
            ev[e] = make_uint2(uint32_t(v[0]) | uint32_t(v[1]) << 16, uint32_t(v[2]));
#pragma unroll
            for (int k = 0; k < 3; k++) {
                uint32_t vk = uint32_t(v[k]);
                uint32_t sh8 = (vk & 3u) * 8u;
                uint32_t old = atomicAdd(&degw[vk >> 2], 1u << sh8);
                if (((old >> sh8) & 255u) == 255u) s_fail = 1;
                atomicXor(&xrw[vk >> 1], e << ((vk & 1u) * 16u));
            }
        }
        __syncthreads();
        if (s_fail) {
            if (tid == 0) {
                atomicOr(a.err, kErrDegOverflow);
                atomicOr(a.item_fail + task.item, kErrDegOverflow);
            }
            __syncthreads();
            continue;
        }

        // -------------------------------------------------------------------- 2. peel
        for (uint32_t v0 = tid & ~31u; v0 < V; v0 += T) {
            const uint32_t v = v0 + lane;
            const bool one = v < V && deg_of(degw, v) == 1u;
            const uint32_t at = warp_slot(&s_cnt[0], one);
            if (one) lists[at] = uint16_t(v);
        }
        __syncthreads();
        uint32_t fi = 0;
        for (;;) {
            const uint32_t nF = s_cnt[fi];
            if (nF == 0) break;
            const uint16_t* F = lists + (fi ? 2 * lw : 0u);
            uint16_t* G = lists + (fi ? 0u : 2 * lw);
            // 65535 stands for none: an edge index is at most 65534
            for (uint32_t i = tid; i < nF; i += T) {
                const uint32_t v = F[i];
                cand[i] = uint16_t(deg_of(degw, v) == 1u ? xr_of(xrw, v) : 0xFFFFu);
            }
            __syncthreads();
            for (uint32_t i0 = tid & ~31u; i0 < nF; i0 += T) {
                const uint32_t i = i0 + lane;
                const uint32_t e = i < nF ? cand[i] : 0xFFFFu;
                const uint32_t bit = 1u << (e & 31u);
                const bool mine = e != 0xFFFFu && !(atomicOr(&clm[e >> 5], bit) & bit);
                const uint32_t at = warp_slot(&s_cnt[2], mine);
                if (mine) {
                    const uint32_t v = F[i];
                    const uint2 x = __ldcg(ev + e);
                    const uint32_t a0 = x.x & 0xFFFFu, a1 = x.x >> 16;
                    const uint32_t u0 = a0 == v ? a1 : a0, u1 = x.y == v ? a1 : x.y;
                    prec[at] = make_uint2(v | e << 16, u0 | u1 << 16);
#pragma unroll
                    for (int k = 0; k < 2; k++) {
                        const uint32_t u = k ? u1 : u0;
                        const uint32_t sh8 = (u & 3u) * 8u;
                        const uint32_t old = atomicSub(&degw[u >> 2], 1u << sh8);
                        atomicXor(&xrw[u >> 1], e << ((u & 1u) * 16u));
                        if (((old >> sh8) & 255u) == 2u) G[atomicAdd(&s_cnt[fi ^ 1], 1u)] = uint16_t(u);
                    }
                }
            }
            __syncthreads();
            if (tid == 0) {
                s_cnt[3]++;
                proff[s_cnt[3]] = s_cnt[2];
                s_cnt[fi] = 0;
            }
            fi ^= 1;
            __syncthreads();
        }
        const uint32_t peeled = s_cnt[2];
        const uint32_t prounds = s_cnt[3];

        // ---------------------------------------------------- 3. lazy Gaussian elimination
        uint32_t C = 0, A = 0, S = 0, D = 0, R = 0;
        if (peeled < m) {
            if (tid == 0) s_C = 0;
            __syncthreads();
            for (uint32_t f0 = tid & ~31u; f0 < m; f0 += T) {
                const uint32_t e = f0 + lane;
                const bool open = e < m && !((clm[e >> 5] >> (e & 31u)) & 1u);
                const uint32_t at = warp_slot(&s_C, open);
                if (open) core[at] = uint16_t(e);
            }
            __syncthreads();
            C = s_C;
            // Variable states and equation states move to shared memory when they
            // fit (the peel's arrays are dead now); otherwise they stay in the slab.
            // Equation word: bits 0-1 idle count, bit 2 done, bits 3.. sum of its idle variables.
            const bool in_smem = uint64_t(V) + C <= kLgeSmemWords;
            if (kSpills && !in_smem && spill_task(a, s)) {
                __syncthreads();
                continue;
            }
            // core equations with their vertices, four loads of a thread in flight
            auto for_core = [&](auto&& f) {
                for (uint32_t j0 = tid; j0 < C; j0 += 4 * T) {
                    uint32_t e[4];
                    uint2 x[4];
#pragma unroll
                    for (uint32_t t = 0; t < 4; t++) e[t] = j0 + t * T < C ? core[j0 + t * T] : 0u;
#pragma unroll
                    for (uint32_t t = 0; t < 4; t++) x[t] = __ldcg(ev + e[t]);
#pragma unroll
                    for (uint32_t t = 0; t < 4; t++)
                        if (j0 + t * T < C) f(j0 + t * T, x[t]);
                }
            };
            // vst: first the core degrees, then the list cursors, then the variable
            // states. Written for both places they may be in (the compiler then
            // uses shared-memory instructions for the usual one).
            auto eliminate_all = [&](uint32_t* const vst, uint32_t* const est) {
            // a bit per hashed vertex triple: equations that find theirs set may repeat another
            uint32_t* const seen = in_smem && V + C + kSeenWords <= kLgeSmemWords ? sm + V + C : nullptr;
            for (uint32_t v = tid; v < V; v += T) vst[v] = 0;
            for (uint32_t i = tid; i < 256; i += T) s_hist[i] = 0;
            if (seen)
                for (uint32_t i = tid; i < kSeenWords; i += T) seen[i] = 0;
            __syncthreads();
            for_core([&](uint32_t j, uint2 x) {
                const uint32_t v0 = x.x & 0xFFFFu, v1 = x.x >> 16, v2 = x.y;
                atomicAdd(&vst[v0], 1u);
                atomicAdd(&vst[v1], 1u);
                atomicAdd(&vst[v2], 1u);
                uint32_t twin = kTwin;
                if (seen) {
                    const uint32_t h = (x.x * 0x9E3779B1u + x.y * 0x85EBCA77u) >> (32 - kLgSeen);
                    if (!((atomicOr(&seen[h >> 5], 1u << (h & 31u)) >> (h & 31u)) & 1u)) twin = 0;
                }
                est[j] = ((v0 + v1 + v2) << 3) | 3u | twin;
            });
            __syncthreads();
            // activation order: core degree, heaviest first (counting sort)
            for (uint32_t v0 = tid & ~31u; v0 < V; v0 += T) {
                const uint32_t d = v0 + lane < V ? vst[v0 + lane] : 0u;
                warp_slot_by(s_hist, min(d, 255u), d != 0);
            }
            __syncthreads();
            if (warp == 0) {  // s_hist[d]: variables of larger core degree
                uint32_t x[8], sum = 0;
#pragma unroll
                for (int k = 0; k < 8; k++) {
                    x[k] = s_hist[255 - (8 * lane + k)];
                    sum += x[k];
                }
                uint32_t incl = sum;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, d);
                    if (lane >= unsigned(d)) incl += y;
                }
                uint32_t run = incl - sum;
#pragma unroll
                for (int k = 0; k < 8; k++) {
                    s_hist[255 - (8 * lane + k)] = run;
                    run += x[k];
                }
                if (lane == 31) s_nact = run;
            }
            __syncthreads();
            for (uint32_t v0 = tid & ~31u; v0 < V; v0 += T) {
                const uint32_t v = v0 + lane;
                const uint32_t d = v < V ? vst[v] : 0u;
                const uint32_t at = warp_slot_by(s_hist, min(d, 255u), d != 0);
                if (d) act[at] = uint16_t(v);
            }
            __syncthreads();
            cta_exclusive_scan(vst, V, s_part);
            // The incidence offsets (at most 3C) go to shared memory as 16-bit
            // entries after the states when they fit, and so does the incidence
            // list: the elimination rounds then wait on no memory beyond it.
            uint16_t* ioff16 = nullptr;
            uint32_t used = V + C;
            if (in_smem && 3ull * C < 65536 && uint64_t(used) + (V + 2) / 2 <= kLgeSmemWords) {
                ioff16 = reinterpret_cast<uint16_t*>(sm + used);
                used += (V + 2) / 2;
            }
            constexpr uint32_t kQueueRoom = 1024;  // words kept for the round queues
            uint16_t* ilist = inc_list;
            if (ioff16 && uint64_t(used) + (3 * C + 1) / 2 + kQueueRoom <= kLgeSmemWords) {
                ilist = reinterpret_cast<uint16_t*>(sm + used);
                used += (3 * C + 1) / 2;
            }
            if (ioff16) {
                for (uint32_t v = tid; v < V; v += T) ioff16[v] = uint16_t(vst[v]);
                if (tid == 0) ioff16[V] = uint16_t(3 * C);
            } else {
                for (uint32_t v = tid; v < V; v += T) inc_off[v] = vst[v];
                if (tid == 0) inc_off[V] = 3 * C;
            }
            __syncthreads();
            for_core([&](uint32_t j, uint2 x) {
                ilist[atomicAdd(&vst[x.x & 0xFFFFu], 1u)] = uint16_t(j);
                ilist[atomicAdd(&vst[x.x >> 16], 1u)] = uint16_t(j);
                ilist[atomicAdd(&vst[x.y], 1u)] = uint16_t(j);
            });
            auto off_of = [&](uint32_t v) -> uint32_t { return ioff16 ? uint32_t(ioff16[v]) : __ldcg(&inc_off[v]); };
            __syncthreads();
            for (uint32_t v = tid; v < V; v += T) vst[v] = 0;
            // Duplicate keys (Sec. 4.4-4.5): equal local signatures in a shard are
            // the same key. Identical edges never peel, so every duplicate is in
            // the core, next to its copies in the incidence list of its first
            // vertex; the copy of smallest index stays. A filter's copies carry
            // the same fingerprint, a function's copies are dropped when their
            // values agree; a key with two values has no solution at any seed
            // and ends the build (kErrDupKey). Of every two copies one is a twin
            // (it found their bit set), and copies have the same vertex sum: only
            // such pairs' signatures are compared.
            for_core([&](uint32_t j, uint2 x) {
                const uint32_t wj = est[j];
                if (!(wj & kTwin)) return;
                const uint32_t v = x.x & 0xFFFFu, w = wj & kSumMask;
                const uint32_t q1 = off_of(v + 1);
                for (uint32_t q = off_of(v); q < q1; q++) {
                    const uint32_t j2 = ilist[q];
                    if (j2 == j || (est[j2] & kSumMask) != w) continue;
                    const uint32_t e = core[j], e2 = core[j2];
                    if (__ldg(a.loc + e0 + e2) != __ldg(a.loc + e0 + e)) continue;
                    if (task.kind == 0 && __ldg(a.val + e0 + e2) != __ldg(a.val + e0 + e)) {
                        s_fail = 3;
                    } else if (!(atomicOr(&est[e < e2 ? j2 : j], 4u) & 4u)) {
                        atomicAdd(&s_dup, 1u);  // done: no equation of its own
                    }
                }
            });
            __syncthreads();
            if (s_fail == 3) return;
            for (uint32_t j = tid; j < C; j += T) est[j] &= ~kTwin;
            // The rest of shared memory holds the first qcap entries of the two
            // round queues; entries beyond stay in the slab's queues.
            uint32_t qcap = 0;
            uint32_t* sq0 = nullptr;
            if (in_smem) {
                used = (used + 3) & ~3u;
                qcap = used < kLgeSmemWords ? (kLgeSmemWords - used) / 2 : 0;
                sq0 = sm + used;
            }
            uint16_t* const gq = reinterpret_cast<uint16_t*>(scr + o.lists);
            const uint32_t gq1 = 2 * ((a.v_cap + 1) / 2);
            // Counters of a round, one set for each r mod 4 (a set is cleared two
            // rounds before its round and read after its round's only barrier):
            // queue entries for the round, its solves, its dense equations.
            auto qread = [&](uint32_t q, uint32_t i) -> uint32_t { return i < qcap ? sq0[q * qcap + i] : gq[(q ? gq1 : 0u) + i]; };
            uint32_t r = 0, ns = 0, nd = 0, na = 0, apos = 0;  // round; solves, dense equations, active variables so far
            // Removes variable u (now solved from equation `skip`, or active) from
            // its other equations, four lanes taking an entry each of its incidence
            // list: an equation left with one idle variable joins the next round's
            // queue, one left with none joins the dense system. One fetch-and-add
            // per entry, whose result says all; an equation that is done takes the
            // update too (it is never read again).
            auto remove_var = [&](uint32_t u, uint32_t skip) {
                const uint32_t q1 = off_of(u + 1), dec = (u << 3) + 1u;
                for (uint32_t q = off_of(u) + (lane & 3u); q < q1; q += 4) {
                    const uint32_t k = ilist[q];
                    if (k == skip) continue;
                    const uint32_t old = atomicSub(&est[k], dec);
                    if (old & 4u) continue;
                    const uint32_t c = (old & 3u) - 1u;
                    if (c == 1u) {
                        const uint32_t idx = atomicAdd(&s_queue[(r + 1) & 3u], 1u), nq = (r + 1) & 1u;
                        if (idx < qcap) sq0[nq * qcap + idx] = k;
                        else gq[(nq ? gq1 : 0u) + idx] = uint16_t(k);
                    } else if (c == 0u) {
                        atomicOr(&est[k], 4u);
                        dense[nd + atomicAdd(&s_dense[r & 3u], 1u)] = k;
                    }
                }
            };
            if (tid < 4) s_queue[tid] = s_solved[tid] = s_dense[tid] = 0;
            if (tid == 0) soff[0] = 0;
            const uint32_t max_rounds = m + V + 2;
            __syncthreads();
            if (tid < kET) {
            const uint32_t open = C - s_dup;
            for (;;) {
                const uint32_t rem = open - ns - nd;
                if (rem == 0) break;
                if (r >= max_rounds) {
                    if (tid == 0) s_fail = 2;
                    break;
                }
                const uint32_t nF = s_queue[r & 3u];
                if (nF == 0) {
                    // Activate the next heaviest idle variables that still occur in
                    // open equations: the block examines a window of the activation
                    // order in parallel and keeps the first K eligible ones.
                    // batches of 2.5% of the open equations: smaller batches end with
                    // slightly fewer active variables but need many more rounds (per
                    // 9.8K-key shard, 1%: 194 rounds, 655 active; 2.5%: 112 and 704,
                    // 4% fewer cycles)
                    const uint32_t K = max(1u, min(kMaxBatch, rem / 40u));
                    const uint32_t wn = min(uint32_t(kET), s_nact - apos);
                    bool elig = false;
                    uint32_t v = 0;
                    if (tid < wn) {
                        v = act[apos + tid];
                        if (vst[v] == 0) {
                            const uint32_t q1 = off_of(v + 1);
                            for (uint32_t q = off_of(v); q < q1 && !elig; q += 4) {
                                uint32_t ks[4];
#pragma unroll
                                for (uint32_t t = 0; t < 4; t++) ks[t] = q + t < q1 ? uint32_t(ilist[q + t]) : kNone;
#pragma unroll
                                for (uint32_t t = 0; t < 4; t++) elig |= ks[t] != kNone && (est[ks[t]] & 4u) == 0;
                            }
                        }
                    }
                    const unsigned bal = __ballot_sync(0xFFFFFFFFu, elig);
                    if (lane == 0) s_part[warp] = __popc(bal);
                    bar_some(1, kET);
                    uint32_t rank = __popc(bal & ((1u << lane) - 1u)), tot = 0;
                    for (uint32_t w = 0; w < kET / 32; w++) {
                        const uint32_t x = s_part[w];
                        if (w < warp) rank += x;
                        tot += x;
                    }
                    if (elig && rank < K) s_batch[rank] = v;
                    if (elig && rank == K - 1) s_nbatch = apos + tid + 1;  // new scan position
                    bar_some(1, kET);
                    const uint32_t nb = min(K, tot);
                    apos = tot >= K ? s_nbatch : apos + wn;
                    if (na + nb > o.a_cap || (nb == 0 && apos >= s_nact)) {
                        if (tid == 0) s_fail = 2;
                        break;
                    }
                    for (uint32_t i = tid / 4; i < nb; i += kET / 4) {
                        const uint32_t u = s_batch[i];
                        if ((tid & 3u) == 0) {
                            vst[u] = 1;
                            actv[na + i] = u;
                        }
                        remove_var(u, kNone);
                    }
                    na += nb;
                } else {
                    // Queue entries dealt out over the warps; a warp then takes its
                    // solves eight at a time. (No barrier in between: an equation of
                    // this queue has one idle variable, and whoever solves that
                    // variable elsewhere leaves the equation with none.)
                    for (uint32_t i0 = 0; i0 < nF; i0 += kET) {
                        const uint32_t i = i0 + lane * (kET / 32) + warp;
                        const uint32_t j = i < nF ? qread(r & 1u, i) : 0u;
                        const uint32_t w = i < nF ? est[j] : 4u;
                        const uint32_t x = w >> 3;
                        const bool won = (w & 7u) == 1u && atomicCAS(&vst[x], 0u, 2u) == 0u;
                        const unsigned mw = __ballot_sync(0xFFFFFFFFu, won);
                        if (mw == 0) continue;
                        uint32_t at = 0;
                        if (lane == 0) at = atomicAdd(&s_solved[r & 3u], uint32_t(__popc(mw)));
                        at = __shfl_sync(0xFFFFFFFFu, at, 0);
                        const uint32_t mine = __popc(mw & ((1u << lane) - 1u));
                        if (won) {
                            s_part[32 * warp + mine] = (j << 16) | x;
                            solves[ns + at + mine] = (j << 16) | x;
                            atomicOr(&est[j], 4u);
                        }
                        __syncwarp();
                        for (uint32_t g = lane / 4; g < uint32_t(__popc(mw)); g += 8) {
                            const uint32_t sv = s_part[32 * warp + g];
                            remove_var(sv & 0xFFFFu, sv >> 16);
                        }
                        __syncwarp();
                    }
                }
                if (tid == 0) s_queue[(r + 2) & 3u] = s_solved[(r + 2) & 3u] = s_dense[(r + 2) & 3u] = 0;
                bar_some(1, kET);
                ns += s_solved[r & 3u];
                nd += s_dense[r & 3u];
                r++;
                if (tid == 0) soff[r] = ns;
            }
            if (tid == 0) s_batch[0] = na, s_batch[1] = ns, s_batch[2] = nd, s_batch[3] = r;
            }
            __syncthreads();
            A = s_batch[0], S = s_batch[1], D = s_batch[2], R = s_batch[3];
            };
            if (kSpills || in_smem) eliminate_all(sm, sm + V);
            else eliminate_all(vstate, eqst);
            if (s_fail) {
                const uint32_t bad = s_fail == 3 ? kErrDupKey : kErrLgeSize;
                if (tid == 0) {
                    atomicOr(a.err, bad);
                    atomicOr(a.item_fail + task.item, bad);
                }
                __syncthreads();
                continue;
            }
        }
        const uint32_t AW = (A + 31) / 32, DW = (D + 31) / 32;
        const uint32_t RS = AW | 1u;  // odd row stride: conflict-free shared-memory rows
        // The dense system: rows, then right-hand sides, panel words, combinations
        // and pivot flags (a word per row each), the column map, a panel's pivot
        // rows and their sums in fours. In shared memory when it fits, else its
        // rows are in the slab behind the column-major matrix (large shards only).
        const uint64_t cm_words = (uint64_t(A) * DW + 3) & ~uint64_t(3);
        const uint64_t rows_words = uint64_t(D) * RS;
        const uint32_t PS = (AW + 3) & ~3u;  // stride of a panel's pivot rows
        const uint32_t flat_words = (4 * D + A + 3u) & ~3u;
        const uint32_t small_words = flat_words + (32 + 128) * PS;
        if (small_words > kLgeSmemWords && spill_task(a, s)) {  // nothing of this shard has left the slab yet
            __syncthreads();
            continue;
        }
        // (S * AW is more than is stored: a limit of its own, which shards of random keys
        // do not come to)
        if (uint64_t(S) * AW > o.lpool || cm_words + rows_words > o.lpool || small_words > kLgeSmemWords) {
            if (tid == 0) {
                atomicOr(a.err, kErrLgeSize);
                atomicOr(a.item_fail + task.item, kErrLgeSize);
            }
            __syncthreads();
            continue;
        }
        // ------------------------------------------------------ 4. dense system, values
        // Shared memory holds the solve records, the rounds' offsets and one word
        // per variable when they fit; the dense system takes their place in between.
        const uint32_t rec_words = (2 * S + 3) & ~3u, off_words = (R / 2 + 4) & ~3u;
        const uint32_t rb = rec_words + off_words;
        const bool rec_smem = uint64_t(rb) + V <= kLgeSmemWords;
        const bool rows_smem = rows_words + small_words <= kLgeSmemWords;
        if (kSpills && !(rec_smem && rows_smem) && spill_task(a, s)) {  // nothing of this shard has left the slab yet
            __syncthreads();
            continue;
        }
        uint16_t* const off16 = reinterpret_cast<uint16_t*>(sm + rec_words);
        // One record per solve, gathered for all solves at once: the variable, its
        // equation's edge and the two other variables.
        for (uint32_t si = tid; si < S; si += T) {
            const uint32_t sv = __ldcg(&solves[si]);
            const uint32_t x = sv & 0xFFFFu, e = core[sv >> 16];
            const uint2 q = __ldcg(ev + e);
            const uint32_t a0 = q.x & 0xFFFFu, a1 = q.x >> 16;
            srec[si] = make_uint2(x | e << 16, (a0 == x ? a1 : a0) | (q.y == x ? a1 : q.y) << 16);
        }
        __syncthreads();
        // Written for every place its arrays may be in, as the elimination.
        // false: the system has no solution.
        auto solve_all = [&](uint32_t* const vx, uint2* const rec, uint32_t* const rows) -> bool {
        // (and the first solve of every round that has one, s_cnt[3] rounds)
        auto load_records = [&]() {
            if (!rec_smem) return;
            if (warp == 0) {
                uint32_t n = 0;
                for (uint32_t r0 = 0; r0 < R; r0 += 32) {
                    const uint32_t r = r0 + lane;
                    const uint32_t o0 = r < R ? __ldcg(&soff[r]) : 0u, o1 = r < R ? __ldcg(&soff[r + 1]) : 0u;
                    const unsigned m = __ballot_sync(0xFFFFFFFFu, o1 > o0);
                    if (o1 > o0) off16[n + __popc(m & ((1u << lane) - 1u))] = uint16_t(o0);
                    n += __popc(m);
                }
                if (lane == 0) {
                    off16[n] = uint16_t(S);
                    s_cnt[3] = n;
                }
            }
            for (uint32_t si = tid; si < S; si += T) rec[si] = __ldcg(srec + si);
        };
        // The rounds of solves, first to last or back, with a barrier behind each. A
        // round is short (some 60 solves), so its latency is what counts: the next
        // round's records and the bounds of the one after are on their way while
        // this one is worked on (420 -> 160 cycles a round).
        // Run by gt threads (this one is gtid of them) that share barrier `bar`.
        auto walk = [&](auto back_c, uint32_t* const vx, uint32_t gt, uint32_t gtid, uint32_t bar, auto&& f) {
            constexpr bool back = decltype(back_c)::value;
            if (rec_smem) {
                const uint32_t n = s_cnt[3];
                uint32_t k = 0;
                auto bound = [&](uint32_t i) -> uint32_t {  // i-th bound met on the way
                    const uint32_t j = min(i, n);
                    return off16[back ? n - j : j];
                };
                uint32_t b0 = bound(0), b1 = bound(1), b2 = bound(2);
                auto first = [&](uint32_t x, uint32_t y) { return (back ? y : x) + gtid; };
                auto last = [&](uint32_t x, uint32_t y) { return back ? x : y; };
                uint2 q = make_uint2(0, 0);
                if (first(b0, b1) < last(b0, b1)) q = rec[first(b0, b1)];
                for (; k < n; k++) {
                    const uint32_t si = first(b0, b1), hi = last(b0, b1);
                    const bool on = si < hi;
                    const uint32_t c = on ? vx[q.x & 0xFFFFu] : 0u;
                    uint2 nq = make_uint2(0, 0);
                    if (first(b1, b2) < last(b1, b2)) nq = rec[first(b1, b2)];
                    const uint32_t b3 = bound(k + 3);
                    if (on) f(q, c);
                    for (uint32_t sj = si + gt; sj < hi; sj += gt) {
                        const uint2 x = rec[sj];
                        f(x, vx[x.x & 0xFFFFu]);
                    }
                    bar_some(bar, gt);
                    q = nq, b0 = b1, b1 = b2, b2 = b3;
                }
            } else {
                for (uint32_t k = 0; k < R; k++) {
                    const uint32_t r = back ? R - 1 - k : k;
                    const uint32_t lo = __ldcg(&soff[r]), hi = __ldcg(&soff[r + 1]);
                    if (hi == lo) continue;
                    for (uint32_t si = lo + gtid; si < hi; si += gt) {
                        const uint2 x = rec[si];
                        f(x, vx[x.x & 0xFFFFu]);
                    }
                    bar_some(bar, gt);
                }
            }
        };
        // Values of the solved variables: vx[x] starts as its equation's
        // right-hand side, the active variables as given.
        auto forward = [&]() {
            if (tid < kGT)
                walk(std::false_type{}, vx, kGT, tid, 1,
                     [&](uint2 q, uint32_t c) { vx[q.x & 0xFFFFu] = c ^ vx[q.y & 0xFFFFu] ^ vx[q.y >> 16]; });
            __syncthreads();
        };
        load_records();
        __syncthreads();
        if (D > 0) {
            // constant terms: every active variable 0
            for (uint32_t v = tid; v < V; v += T) vx[v] = 0;
            __syncthreads();
            for (uint32_t si = tid; si < S; si += T) {
                const uint32_t q = rec[si].x;
                vx[q & 0xFFFFu] = rhs_of(a, task, e0 + (q >> 16));
            }
            __syncthreads();
            forward();
            for (uint32_t d = tid; d < D; d += T) {
                const uint32_t e = core[__ldcg(&dense[d])];
                const uint2 q = __ldcg(ev + e);
                lc[d] = rhs_of(a, task, e0 + e) ^ vx[q.x & 0xFFFFu] ^ vx[q.x >> 16] ^ vx[q.y];
            }
            // Coefficients: 32 dense equations at a time are carried back through the
            // solves in reverse order (bit d of vx[v]: equation d contains v): a
            // solved variable's bits pass to the two others of its equation. What
            // is left stands on active variables: a column of the system each.
            // (Carrying the columns forward, one coefficient row per solve, takes
            // as many bits per solve as there are active variables, 2.5 times the
            // dense equations, and the rows do not fit in shared memory.)
            // As many groups of threads as have room for a word per variable take
            // 32 equations each at the same time.
            __syncthreads();
            const uint32_t groups = rec_smem ? max(1u, min(min(DW, uint32_t(kLT / kGT)), (kLgeSmemWords - rb) / V)) : 1u;
            const uint32_t gt = groups > 1 ? kGT : kET;  // one group alone takes the elimination's threads
            const uint32_t grp = tid / gt, gtid = tid % gt;
            if (grp < groups) {
                uint32_t* const gx = vx + grp * V;
                for (uint32_t w = grp; w < DW; w += groups) {
                    for (uint32_t v = gtid; v < V; v += gt) gx[v] = 0;
                    bar_some(1 + grp, gt);
                    if (gtid < 32 && 32 * w + gtid < D) {
                        const uint2 q = __ldcg(ev + core[__ldcg(&dense[32 * w + gtid])]);
                        atomicXor(&gx[q.x & 0xFFFFu], 1u << gtid);
                        atomicXor(&gx[q.x >> 16], 1u << gtid);
                        atomicXor(&gx[q.y], 1u << gtid);
                    }
                    bar_some(1 + grp, gt);
                    walk(std::true_type{}, gx, gt, gtid, 1 + grp, [&](uint2 q, uint32_t c) {
                        if (c) {
                            atomicXor(&gx[q.y & 0xFFFFu], c);
                            atomicXor(&gx[q.y >> 16], c);
                        }
                    });
                    for (uint32_t c = gtid; c < A; c += gt) L[uint64_t(w) * A + c] = gx[__ldcg(&actv[c])];
                    bar_some(1 + grp, gt);
                }
            }
            __syncthreads();
            uint32_t* const small = sm;
            uint32_t* const rhs = small;
            uint32_t* const pan = rhs + D;    // a panel's word of each row
            uint32_t* const comb = pan + D;   // the panel's pivot rows to add to each row
            uint32_t* const pivf = comb + D;
            uint32_t* const colrow = pivf + D;
            uint32_t* const pbuf = small + flat_words;  // pivot rows as the panel found them
            uint32_t* const tab = pbuf + 32 * PS;       // every sum of pivot rows 4g .. 4g + 3, 16 each
            // rows from columns: a warp turns 32 columns x 32 rows with ballots
            for (uint32_t blk = warp; blk < AW * DW; blk += kLT / 32) {
                const uint32_t cw = blk / DW, w = blk % DW;
                const uint32_t c = 32 * cw + lane;
                const uint32_t bits = c < A ? __ldcg(&L[uint64_t(w) * A + c]) : 0u;
                uint32_t mine = 0;
#pragma unroll
                for (uint32_t d = 0; d < 32; d++) {
                    const uint32_t row = __ballot_sync(0xFFFFFFFFu, (bits >> d) & 1u);
                    if (lane == d) mine = row;
                }
                if (32 * w + lane < D) rows[uint64_t(32 * w + lane) * RS + cw] = mine;
            }
            for (uint32_t d = tid; d < D; d += T) {
                rhs[d] = __ldcg(&lc[d]);
                pivf[d] = 0;
            }
            for (uint32_t c = tid; c < A; c += T) colrow[c] = kNone;
            __syncthreads();
            // Gauss-Jordan over GF(2), a word of columns (a panel) at a time. One warp
            // reduces the panel's words of 64 unused rows in registers, two a lane,
            // and finds up to 32 pivots with no barrier (64 random rows hardly ever
            // lack one for a column); what every other row has to take up then
            // follows from its own panel word, and the rest of every row is brought
            // up to date once, from the sums of the pivot rows in fours. Columns
            // the 64 rows had no pivot for are looked at again with the rows that
            // still have bits in them. Once every row is a pivot no later column
            // can have one (its active variable stays free, 0): the loop ends there.
            uint32_t npiv = 0;
            for (uint32_t cw = 0; cw < AW && npiv < D; cw++) {
                for (uint32_t d = tid; d < D; d += T) pan[d] = rows[uint64_t(d) * RS + cw];
                const uint32_t w0 = cw + 1, wn = AW - w0;  // words behind the panel
                for (;;) {
                    if (tid == 0) s_cnt[0] = 0;
                    __syncthreads();
                    for (uint32_t d0 = tid & ~31u; d0 < D; d0 += T) {
                        const uint32_t d = d0 + lane;
                        const bool cand = d < D && !pivf[d] && pan[d];
                        const uint32_t at = warp_slot(&s_cnt[0], cand);
                        if (cand && at < 64) s_pool[at] = d;
                    }
                    __syncthreads();
                    const uint32_t np = min(s_cnt[0], 64u);
                    if (np == 0) break;
                    if (warp == 0) {
                        uint32_t row[2], x[2], y[2] = {0, 0}, mine[2] = {kNone, kNone};
#pragma unroll
                        for (int t = 0; t < 2; t++) {
                            const uint32_t i = lane + 32 * t;
                            row[t] = i < np ? s_pool[i] : kNone;
                            x[t] = i < np ? pan[row[t]] : 0u;
                        }
                        uint32_t k = 0;
                        for (uint32_t c = 0; c < 32; c++) {
                            const unsigned h0 = __ballot_sync(0xFFFFFFFFu, mine[0] == kNone && ((x[0] >> c) & 1u));
                            const unsigned h1 = __ballot_sync(0xFFFFFFFFu, mine[1] == kNone && ((x[1] >> c) & 1u));
                            if (!(h0 | h1)) continue;
                            const int p = __ffs(h0 ? h0 : h1) - 1;
                            const uint32_t px = __shfl_sync(0xFFFFFFFFu, h0 ? x[0] : x[1], p);
                            const uint32_t py = __shfl_sync(0xFFFFFFFFu, h0 ? y[0] : y[1], p) ^ (1u << k);
#pragma unroll
                            for (int t = 0; t < 2; t++) {
                                if (int(lane) == p && (t == 0) == (h0 != 0)) {
                                    mine[t] = k | (c << 8);
                                } else if ((x[t] >> c) & 1u) {
                                    x[t] ^= px;
                                    y[t] ^= py;
                                }
                            }
                            k++;
                        }
#pragma unroll
                        for (int t = 0; t < 2; t++)
                            if (mine[t] != kNone) {
                                const uint32_t j = mine[t] & 255u, c = mine[t] >> 8;
                                s_piv[j] = make_uint4(row[t], x[t], y[t] ^ (1u << j), c);
                                pivf[row[t]] = 2u + j;  // a pivot of this panel
                                colrow[32 * cw + c] = row[t];
                            }
                        if (lane == 0) s_cnt[1] = k;
                    }
                    __syncthreads();
                    const uint32_t k = s_cnt[1];
                    npiv += k;
                    if (k == 32) {  // pivot j stands in column j: its combinations in fours, too
                        if (tid < 128) {
                            uint32_t z = 0;
#pragma unroll
                            for (uint32_t t = 0; t < 4; t++)
                                if ((tid >> t) & 1u) z ^= s_piv[tid / 16 * 4 + t].z;
                            s_tz[tid] = z;
                        }
                        __syncthreads();
                    }
                    for (uint32_t d = tid; d < D; d += T) {
                        const uint32_t own = pivf[d];
                        uint32_t x = pan[d], y = 0;
                        if (own >= 2) {
                            const uint4 p = s_piv[own - 2];
                            y = p.z ^ (1u << (own - 2));
                            // bits left stand in columns that the 64 rows had no pivot
                            // for; a row of the next pass may, and this one takes it up
                            x = p.y & ~(1u << p.w);
                            pivf[d] = 1;
                        } else if (k == 32) {
#pragma unroll
                            for (uint32_t g = 0; g < 8; g++) y ^= s_tz[g * 16 + ((x >> (4 * g)) & 15u)];
                            x = 0;
                        } else {
                            const uint32_t was = x;
                            for (uint32_t j = 0; j < k; j++) {
                                const uint4 p = s_piv[j];
                                const uint32_t f = 0u - ((was >> p.w) & 1u);
                                x ^= f & p.y;
                                y ^= f & p.z;
                            }
                        }
                        pan[d] = x;
                        comb[d] = y;
                    }
                    for (uint32_t j = warp; j < k; j += kLT / 32)
                        for (uint32_t w = lane; w <= wn; w += 32)
                            pbuf[j * PS + w] = w < wn ? rows[uint64_t(s_piv[j].x) * RS + w0 + w] : rhs[s_piv[j].x];
                    __syncthreads();
                    const uint32_t groups = (k + 3) / 4;
                    for (uint32_t i = warp; i < groups * 16; i += kLT / 32) {
                        const uint32_t j0 = i / 16 * 4, n4 = min(4u, k - j0);
                        const uint32_t* pb = pbuf + j0 * PS;
                        for (uint32_t w = lane; w <= wn; w += 32) {
                            uint32_t x = 0;
#pragma unroll
                            for (uint32_t t = 0; t < 4; t++)
                                if (t < n4 && ((i >> t) & 1u)) x ^= pb[t * PS + w];
                            tab[i * PS + w] = x;
                        }
                    }
                    __syncthreads();
                    for (uint32_t q = 0; 4 * q <= wn; q++)
                        for (uint32_t d = tid; d < D; d += T) {
                            const uint32_t c = comb[d];
                            if (!c) continue;
                            uint32_t x[4] = {0, 0, 0, 0};
                            for (uint32_t g = 0; g < groups; g++) {
                                const uint4 y = *reinterpret_cast<const uint4*>(tab + (g * 16 + ((c >> (4 * g)) & 15u)) * PS + 4 * q);
                                x[0] ^= y.x, x[1] ^= y.y, x[2] ^= y.z, x[3] ^= y.w;
                            }
                            uint32_t* row = rows + uint64_t(d) * RS + w0 + 4 * q;
#pragma unroll
                            for (uint32_t t = 0; t < 4; t++) {
                                if (4 * q + t < wn) row[t] ^= x[t];
                                else if (4 * q + t == wn) rhs[d] ^= x[t];
                            }
                        }
                    if (k == 32 || npiv == D) break;
                }
                __syncthreads();
            }
            for (uint32_t d = tid; d < D; d += T)
                if (!pivf[d] && rhs[d] != 0) s_fail = 1;
            __syncthreads();
            if (s_fail) return false;
            // the active variables' values leave the region before the values enter it
            for (uint32_t c = tid; c < A; c += T) lc[c] = colrow[c] != kNone ? rhs[colrow[c]] : 0u;
            __syncthreads();
            load_records();
        }
        // Values of every variable: active, solved in solve order, then the peeled
        // edges' vertices in reverse peel order.
        for (uint32_t v = tid; v < V; v += T) vx[v] = 0;
        __syncthreads();
        if (D > 0)
            for (uint32_t c = tid; c < A; c += T) vx[__ldcg(&actv[c])] = __ldcg(&lc[c]);
        for (uint32_t si = tid; si < S; si += T) {
            const uint32_t q = rec[si].x;
            vx[q & 0xFFFFu] = rhs_of(a, task, e0 + (q >> 16));
        }
        for (uint32_t i = tid; i < peeled; i += T) {
            const uint32_t q = __ldcg(prec + i).x;
            vx[q & 0xFFFFu] = rhs_of(a, task, e0 + (q >> 16));
        }
        __syncthreads();
        forward();
        for (uint32_t r = prounds; r-- > 0;) {
            const uint32_t lo = __ldcg(&proff[r]), hi = __ldcg(&proff[r + 1]);
            for (uint32_t i = lo + tid; i < hi; i += T) {
                const uint2 q = __ldcg(prec + i);
                vx[q.x & 0xFFFFu] ^= vx[q.y & 0xFFFFu] ^ vx[q.y >> 16];
            }
            __syncthreads();
        }
        const uint32_t vmask = b == 32 ? 0xFFFFFFFFu : ((1u << b) - 1u);
        for (uint32_t v = tid; v < V; v += T) cell_put_zero(data, b, cbase + v, vx[v] & vmask);
        return true;
        };
        prev_l = rows_smem ? cm_words : cm_words + rows_words;
        bool solved;
        if (kSpills || (rec_smem && rows_smem)) solved = solve_all(sm + rb, reinterpret_cast<uint2*>(sm), sm + small_words);
        else solved = solve_all(rec_smem ? sm + rb : V <= kLgeSmemWords ? sm : vstate, rec_smem ? reinterpret_cast<uint2*>(sm) : srec,
                                rows_smem ? sm + small_words : L + cm_words);
        if (!solved) {
            if (tid == 0) {
                atomicOr(a.err, kErrUnsolvable);
                atomicOr(a.item_fail + task.item, kErrUnsolvable);
            }
            __syncthreads();
            continue;
        }
        if (tid == 0) {
            atomicAdd(&a.stats[0], peeled);
            atomicAdd(&a.stats[1], C - s_dup);
            if (s_dup) {
                atomicAdd(&a.stats[3], s_dup);
                if (a.item_dup) atomicAdd(a.item_dup + task.item, s_dup);
            }
        }
        __syncthreads();
    }
}

#define VF_LGE_SMALL k_lge<kSmallT, kSmallWords, 3>
#define VF_LGE_MID k_lge<kMidT, kMidWords, 2>
#define VF_LGE_BIG k_lge<kBigT, kBigWords, 1>

enum LgeCfg { kCfgSmall = 0, kCfgMid = 1, kCfgBig = 2 };

// Resident CTAs of one configuration on the whole GPU (attributes set once per device).
static unsigned resident(LgeCfg c) {
    static std::atomic<uint64_t> done{0};
    static unsigned per_sm[3] = {1, 1, 1};
    int dev = 0;
    cudaGetDevice(&dev);
    const uint64_t bit = uint64_t(1) << (dev & 63);
    if (!(done.load() & bit)) {
        int p[3] = {0, 0, 0};
        cudaFuncSetAttribute(VF_LGE_SMALL, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmallWords * 4));
        cudaFuncSetAttribute(VF_LGE_MID, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kMidWords * 4));
        cudaFuncSetAttribute(VF_LGE_BIG, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kBigWords * 4));
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p[0], VF_LGE_SMALL, kSmallT, kSmallWords * 4);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p[1], VF_LGE_MID, kMidT, kMidWords * 4);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p[2], VF_LGE_BIG, kBigT, kBigWords * 4);
        for (int i = 0; i < 3; i++) per_sm[i] = unsigned(p[i] < 1 ? 1 : p[i]);
        done.fetch_or(bit);
    }
    return per_sm[c] * unsigned(num_sms());
}

unsigned lge_grid() { return std::max(resident(kCfgSmall), std::max(resident(kCfgMid), resident(kCfgBig))); }

uint32_t lge_partition(std::vector<LgeTask>& tasks, uint64_t small_keys) {
    auto mid = std::stable_partition(tasks.begin(), tasks.end(),
                                     [small_keys](const LgeTask& t) { return t.m > small_keys; });
    return uint32_t(mid - tasks.begin());
}

cudaError_t launch_lge(const LgeArgs& a, unsigned grid, cudaStream_t st) {
    if (a.ntasks == 0) return cudaSuccess;
    // the large configuration alone: no spill list, or no more shards than SMs
    // (a shard on an SM of its own is done sooner by 512 threads)
    if (!a.spill || (a.ntasks <= unsigned(num_sms()))) {
        LgeArgs only = a;
        only.spill = nullptr;
        only.spilled = nullptr;
        only.task_lo = 0;
        only.ctr = 2;
        VF_LGE_BIG<<<std::min(grid, resident(kCfgBig)), kBigT, kBigWords * 4, st>>>(only);
        return cudaGetLastError();
    }
    // tasks[0, n_mid): medium configuration, counter word 2; the rest: small
    // configuration, counter word 6; then the spill list (counter word 4)
    const uint32_t n_mid = std::min(a.n_mid, a.ntasks);
    if (n_mid > 0) {
        LgeArgs mid = a;
        mid.spilled = nullptr;
        mid.ntasks = n_mid;
        mid.task_lo = 0;
        mid.ctr = 2;
        VF_LGE_MID<<<std::min(std::min(grid, resident(kCfgMid)), n_mid), kMidT, kMidWords * 4, st>>>(mid);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (a.ntasks > n_mid) {
        LgeArgs small = a;
        small.spilled = nullptr;
        small.ntasks = a.ntasks - n_mid;
        small.task_lo = n_mid;
        small.ctr = 6;
        VF_LGE_SMALL<<<std::min(std::min(grid, resident(kCfgSmall)), small.ntasks), kSmallT, kSmallWords * 4, st>>>(
            small);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    LgeArgs last = a;
    last.spill = nullptr;
    last.spilled = a.stats + 5;
    last.spill_in = a.spill;
    last.task_lo = 0;
    last.ctr = 4;
    VF_LGE_BIG<<<std::min(grid, resident(kCfgBig)), kBigT, kBigWords * 4, st>>>(last);
    return cudaGetLastError();
}

}  // namespace vf
