// Load-time and per-superstep helper kernels:
//  * out-degrees (PageRank's MSGGen divides by them);
//  * initial vertex values and cache (ghost) fills;
//  * synchronization caching and skipping between partitions (Section
//    III-B, Algorithm 3): changed ∩ boundary -> global data queue (sorted by
//    id) -> the caches of the partitions that read those vertices; the
//    exchange is skipped on the device when the queue is empty everywhere.
#include "frontier.cuh"

#include <algorithm>

namespace gxp {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

// ----------------------------------------------------------- out-degree

// Sources below kOutdegHot are counted in shared memory and flushed once per
// block: atomics on one address serialize, and power-law generators that do
// not permute ids (R-MAT) put their hubs at the lowest ids (the hottest
// R-MAT 22 source has ~160K out-edges, which took ~1 ms of global atomics).
// 16.8 M edges of a million-vertex R-MAT graph take 191 us read one source a
// thread and 214 us read four: the reads do not bound it. A single partition's
// CSC is therefore counted chunk by chunk behind its copy from the host (189 us
// in eight chunks, next to 363 us of copies). Above them a warp adds once per
// distinct source: loading 16.8 M edges that all leave one vertex above takes
// 0.58 ms so and 10.7 ms with an atomic an edge; uniform sources 0.50 ms either way.
constexpr uint32_t kOutdegHot = 8192;

// kCheck: ids of n_local and above are not counted but reported (bit 1 of err).
template <bool kCheck>
__global__ void __launch_bounds__(256) k_outdeg(const uint32_t* __restrict__ src, uint64_t n_edges, uint32_t n_own,
                                                uint32_t v_begin, const uint32_t* __restrict__ ghost_gid,
                                                uint32_t* __restrict__ outdeg, uint32_t* err) {
    __shared__ uint32_t hot[kOutdegHot];
    for (uint32_t i = threadIdx.x; i < kOutdegHot; i += blockDim.x) hot[i] = 0u;
    __syncthreads();
    bool bad = false;
    auto count = [&](uint32_t u) {
        if (kCheck && u >= n_own) {
            bad = true;
            return;
        }
        const uint32_t g = u < n_own ? v_begin + u : ghost_gid[u - n_own];
        if (g < kOutdegHot) {
            atomicAdd(&hot[g], 1u);
            return;
        }
        const unsigned peers = __match_any_sync(__activemask(), g);
        if ((threadIdx.x & 31) == (unsigned)(__ffs(peers) - 1)) atomicAdd(&outdeg[g], (uint32_t)__popc(peers));
    };
    // four sources a load (src is 16-byte aligned)
    const uint64_t t0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x, stride = (uint64_t)gridDim.x * blockDim.x;
    const uint4* src4 = reinterpret_cast<const uint4*>(src);
    for (uint64_t e = t0; e < n_edges / 4u; e += stride) {
        const uint4 u = __ldg(src4 + e);
        count(u.x);
        count(u.y);
        count(u.z);
        count(u.w);
    }
    for (uint64_t e = (n_edges & ~3ull) + t0; e < n_edges; e += stride) count(src[e]);
    if (kCheck && bad) atomicOr(err, 2u);
    __syncthreads();
    const uint32_t n_hot = kCheck ? min(kOutdegHot, n_own) : kOutdegHot;
    for (uint32_t i = threadIdx.x; i < n_hot; i += blockDim.x)
        if (hot[i]) atomicAdd(&outdeg[i], hot[i]);
}

__global__ void k_validate(const uint32_t* __restrict__ col_ptr, uint32_t n_own,
                           const uint32_t* __restrict__ src, uint64_t n_edges, uint32_t n_local,
                           uint32_t* err) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < n_edges; e += stride)
        if (src[e] >= n_local) atomicOr(err, kErrBounds);
    for (uint64_t v = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; v < n_own; v += stride)
        if (col_ptr[v] > col_ptr[v + 1]) atomicOr(err, kErrInput);
    if (blockIdx.x == 0 && threadIdx.x == 0 && (col_ptr[0] != 0u || (uint64_t)col_ptr[n_own] != n_edges))
        atomicOr(err, kErrInput);
}

// offsets imported as given: col_ptr (u64) -> u32 with its checks (bit 0 of
// err: not running from 0 to n_edges or decreasing)
__global__ void k_csc_offsets(const uint64_t* __restrict__ cp64, uint32_t n, uint64_t n_edges,
                              uint32_t* __restrict__ cp32, uint32_t* err) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t v = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; v <= n; v += stride) {
        const uint64_t c = cp64[v];
        const bool bad = c > n_edges || (v == 0 && c != 0) || (v == n && c != n_edges) || (v < n && cp64[v + 1] < c);
        if (bad) atomicOr(err, 1u);
        cp32[v] = (uint32_t)c;
    }
}

// ------------------------------------------------------- initial values


// The initial state of a run (BeginArgs) in one launch: a run used to take
// nine operations (~35 us of enqueueing) to set it up.
__global__ void __launch_bounds__(256) k_begin(const BeginArgs a) {
    const uint32_t t0 = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
    const bool pr = a.algo == Algo::PR, personalized = pr && a.source != kInf;
    auto rank0 = [&](uint32_t v) { return personalized ? (v == a.source ? 1.0f : 0.0f) : a.r0; };
    // the value other vertices gather of vertex v
    auto value = [&](uint32_t v) -> uint32_t {
        if (a.algo == Algo::SSSP) return v == a.source ? 0u : kInf;
        if (!pr) return a.label_of ? a.label_of[v] : v;   // CC / LP labels are input ids
        const uint32_t od = a.outdeg[v];
        return __float_as_uint(od ? __fdiv_rn(rank0(v), (float)od) : 0.0f);
    };
    for (uint64_t v = t0; v < a.n; v += stride) {
        const uint32_t x = value((uint32_t)v);
        a.own[0][v] = x;
        if (pr) a.rank[v] = rank0((uint32_t)v);
        else a.own[1][v] = x;
    }
    for (uint64_t g = t0; g < a.n_ghost; g += stride) a.ghost[g] = value(a.ghost_gid[g]);
    const uint32_t words = (a.n + 31u) / 32u;
#pragma unroll
    for (int k = 0; k < 5; ++k)
        if (a.clear[k])
            for (uint32_t i = t0; i < words; i += stride) a.clear[k][i] = 0u;
    for (uint32_t slot = blockIdx.x; slot < (uint32_t)kStatRing; slot += gridDim.x) {
        unsigned long long* z = reinterpret_cast<unsigned long long*>(a.stats + slot);
        for (uint32_t i = threadIdx.x; i < sizeof(StepStats) / 8; i += blockDim.x) z[i] = 0ull;
    }
    if (blockIdx.x != 0) return;
    __syncthreads();   // slot 0 is block 0's
    if (a.seed != kInf) {
        const uint32_t deg = a.out_ptr[a.seed + 1] - a.out_ptr[a.seed], items = frontier_items(deg);
        for (uint32_t k = threadIdx.x; k < items; k += blockDim.x) {
            if (k < a.fc.list_cap) a.fc.list_out[k] = make_uint2(a.seed, k);
            else atomicOr(a.fc.err, kErrBounds);
        }
        if (threadIdx.x == 0) a.stats->list_ne = list_pack(items, deg);
    } else if (threadIdx.x == 0) {
        a.stats->list_ne = a.list_ne;
    }
    if (threadIdx.x == 0) {
        // the identity slots that empty SELL slots read
        a.own[0][a.n] = a.identity;
        a.own[1][a.n] = a.identity;
        a.ghost[a.n_ghost] = a.identity;
        if (pr)   // every dangling vertex starts with the same rank: an exact multiple
            a.stats->dangling_fx[0] = personalized ? (a.outdeg[a.source] ? 0ull : fx_of(1.0f))
                                                   : *a.n_dangling * fx_of(a.r0);
    }
}

__global__ void __launch_bounds__(256) k_count_dangling(const uint32_t* __restrict__ outdeg, uint32_t n,
                                                        unsigned long long* out) {
    uint32_t c = 0;
    for (uint64_t v = blockIdx.x * 256ull + threadIdx.x; v < n; v += gridDim.x * 256ull) c += outdeg[v] == 0u;
    c = __reduce_add_sync(kFull, c);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, (unsigned long long)c);
}

__global__ void __launch_bounds__(32) k_step_sums(const StepStats* ring, uint64_t first, const uint32_t* err,
                                                  StepReport* out) {
    const uint64_t slot = (first + blockIdx.x) % kStatRing;
    report_step(ring + slot, &out->sum[slot], err, &out->err);
}

__global__ void k_init_ghosts(uint32_t n_ghost, const uint32_t* __restrict__ gid,
                              const uint32_t* __restrict__ own, uint32_t* __restrict__ ghost) {
    for (uint32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < n_ghost; g += gridDim.x * blockDim.x)
        ghost[g] = own[gid[g]];
}

// ----------------------------------------------------------------- sync

__device__ __forceinline__ uint32_t range_mask(uint32_t w, uint32_t v_lo, uint32_t v_hi) {
    const uint32_t base = w * 32u;
    const uint32_t lo = v_lo > base ? v_lo - base : 0u;
    const uint32_t hi = v_hi < base + 32u ? v_hi - base : 32u;
    if (hi <= lo) return 0u;
    const uint32_t upper = hi == 32u ? kFull : ((1u << hi) - 1u);
    return upper & ~((1u << lo) - 1u);
}

constexpr int kSyncBlock = 256;

template <int kThreads = kSyncBlock>
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t x, uint32_t* s_warp, uint32_t& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t v = lane < kThreads / 32 ? s_warp[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, v, o);
            if (lane >= o) v += y;
        }
        if (lane < kThreads / 32) s_warp[lane] = v;
    }
    __syncthreads();
    const uint32_t warp_off = warp ? s_warp[warp - 1] : 0u;
    total = s_warp[kThreads / 32 - 1];
    __syncthreads();
    return warp_off + incl - x;
}

// Whether the exchange is skipped (Section III-B3) and whether it lists the
// changed copies, from the counts the superstep left: the changed boundary
// vertices are counted where they change, so this is one warp's sum rather
// than a pass over the bitmaps (9.8 us a superstep of 3 M vertices). Also
// reports the superstep's sums to the host.
__device__ __forceinline__ unsigned long long boundary_total(const StepStats* st) {   // by one warp
    const int lane = threadIdx.x & 31;
    unsigned long long grand = __ldcg(&st->boundary[lane]) + __ldcg(&st->boundary[lane + 32]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) grand += __shfl_xor_sync(kFull, grand, o);
    return grand;
}
__device__ __forceinline__ void sync_decide(const SyncArgs& a) {   // by one warp
    StepStats* st = a.stats_out;
    const unsigned long long grand = boundary_total(st);
    if ((threadIdx.x & 31) == 0) {
        st->boundary_changed = grand;
        st->skipped = grand == 0 ? 1ull : 0ull;
        st->exchanged = 1ull;
        // the next superstep pulls anyway when its frontier would be too much
        // work to push: its own vertices' items and out-edges, plus at least
        // one item per changed boundary vertex for the copies that would join
        // (each has a copy somewhere); then the copies are not listed. Nor
        // are they when the superstep did not list its own vertices.
        bool list = a.fc.list_out != nullptr && __ldcg(&st->unlisted) == 0ull;
        if (list && a.fc.direction == GXP_DIR_AUTO) {
            const unsigned long long ne = __ldcg(&st->list_ne);
            list = ((ne >> 32) + (ne & 0xFFFFFFFFull) + grand) * (unsigned long long)a.fc.push_div <= a.fc.total_edges;
        }
        st->list_copies = list ? 1ull : 0ull;
    }
    __syncwarp();
    report_step(st, a.report, a.err, a.report_err);
}
__global__ void __launch_bounds__(32) k_sync_decide(const SyncArgs a) { sync_decide(a); }

// Changed ∩ boundary per block of bitmap words; the last block of a
// partition turns its counts into offsets in the partition's queue.
__global__ void __launch_bounds__(kSyncBlock) k_sync_count(const SyncArgs a) {
    __shared__ uint32_t s_warp[kSyncBlock / 32];
    __shared__ bool s_last;
    if (a.stats_out->skipped) return;   // uniform
    const uint32_t p = blockIdx.y;
    const PartDev P = a.parts[p];
    const uint32_t v_lo = P.v_begin, v_hi = P.v_begin + P.n_own;
    const uint32_t w_lo = v_lo >> 5, w_hi = (v_hi + 31u) >> 5;
    const uint32_t w = w_lo + blockIdx.x * kSyncBlock + threadIdx.x;
    uint32_t c = 0;
    if (P.n_own && w < w_hi) c = __popc(a.changed_bits[w] & a.boundary_bits[w] & range_mask(w, v_lo, v_hi));
    uint32_t total;
    block_excl_scan(c, s_warp, total);
    if (threadIdx.x == 0) {
        a.block_counts[p * a.blocks_x + blockIdx.x] = total;
        __threadfence();
        s_last = atomicAdd(a.done_ctr + p, 1u) == gridDim.x - 1u;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    uint32_t run = 0;
    for (uint32_t b0 = 0; b0 < a.blocks_x; b0 += kSyncBlock) {
        const uint32_t b = b0 + threadIdx.x;
        const uint32_t x = b < a.blocks_x ? __ldcg(&a.block_counts[p * a.blocks_x + b]) : 0u;
        uint32_t tot;
        const uint32_t ex = block_excl_scan(x, s_warp, tot);
        if (b < a.blocks_x) a.block_offsets[p * a.blocks_x + b] = run + ex;
        run += tot;
    }
    if (threadIdx.x == 0) {
        a.part_counts[p] = run;
        a.done_ctr[p] = 0u;
    }
}

// The pairs of a warp's 32 words (each lane's `bits` of word w) at positions
// pos of each lane.
__device__ __forceinline__ void write_queue(const SyncArgs& a, uint32_t bits, uint32_t pos, uint32_t w) {
    // A warp writes its 32 words' pairs one word at a time, lane l taking the
    // word's bit l: the word's vertices are 32 consecutive ids, so the value
    // load is one 128-byte line and the pairs land at consecutive positions
    // (a thread walking its own word wrote 32 scattered runs per store).
    const uint32_t lane = threadIdx.x & 31u;
    unsigned todo = __ballot_sync(kFull, bits != 0u);
    while (todo) {
        const int j = __ffs(todo) - 1;
        todo &= todo - 1u;
        const uint32_t bj = __shfl_sync(kFull, bits, j);
        const uint32_t pj = __shfl_sync(kFull, pos, j);
        const uint32_t wj = __shfl_sync(kFull, w, j);
        if ((bj >> lane) & 1u) {
            const uint32_t gid = wj * 32u + lane;
            const uint32_t at = pj + __popc(bj & ((1u << lane) - 1u));
            a.gdq_ids[at] = gid;
            a.gdq_vals[at] = a.own_val[gid];
        }
    }
}

// Write each partition's global data queue (ascending ids): the changed
// boundary vertices with their new values.
__global__ void __launch_bounds__(kSyncBlock) k_sync_write(const SyncArgs a) {
    __shared__ uint32_t s_warp[kSyncBlock / 32];
    if (a.stats_out->skipped) return;   // uniform: Section III-B3 skip
    const uint32_t p = blockIdx.y;
    const PartDev P = a.parts[p];
    const uint32_t v_lo = P.v_begin, v_hi = P.v_begin + P.n_own;
    const uint32_t w_lo = v_lo >> 5, w_hi = (v_hi + 31u) >> 5;
    const uint32_t w = w_lo + blockIdx.x * kSyncBlock + threadIdx.x;
    uint32_t bits = 0;
    if (P.n_own && w < w_hi) bits = a.changed_bits[w] & a.boundary_bits[w] & range_mask(w, v_lo, v_hi);
    uint32_t total;
    uint32_t pos = block_excl_scan(__popc(bits), s_warp, total);
    if (P.n_own == 0 || blockIdx.x * kSyncBlock >= w_hi - w_lo) return;
    pos += a.block_offsets[p * a.blocks_x + blockIdx.x] + (uint32_t)a.gdq_base[p];
    write_queue(a, bits, pos, w);
}

// The decision and the queues in one launch, a CTA per partition that scans
// its words 1,024 at a time: for partitions of at most kQueueWords words,
// where a launch costs more than the scan (partitions of 65,536 vertices:
// decide + count + write 7 us, this 4).
constexpr int kQueueBlock = 1024;
constexpr uint32_t kQueueWords = 4096;
__global__ void __launch_bounds__(kQueueBlock) k_sync_queue(const SyncArgs a) {
    __shared__ uint32_t s_warp[kQueueBlock / 32];
    const uint32_t p = blockIdx.x;
    const bool none = boundary_total(a.stats_out) == 0ull;   // every warp sums
    if (p == 0 && threadIdx.x < 32) sync_decide(a);
    if (none) return;   // uniform: Section III-B3 skip
    const PartDev P = a.parts[p];
    const uint32_t v_lo = P.v_begin, v_hi = P.v_begin + P.n_own;
    const uint32_t w_lo = v_lo >> 5, w_hi = P.n_own ? (v_hi + 31u) >> 5 : w_lo;
    uint32_t run = 0;
    for (uint32_t w0 = w_lo; w0 < w_hi; w0 += kQueueBlock) {
        const uint32_t w = w0 + threadIdx.x;
        const uint32_t bits = w < w_hi ? a.changed_bits[w] & a.boundary_bits[w] & range_mask(w, v_lo, v_hi) : 0u;
        uint32_t total;
        const uint32_t pos = block_excl_scan<kQueueBlock>((uint32_t)__popc(bits), s_warp, total);
        write_queue(a, bits, run + pos + (uint32_t)a.gdq_base[p], w);
        run += total;
    }
    if (threadIdx.x == 0) a.part_counts[p] = run;
}

// Caching (Section III-B): every cached copy of an uploaded vertex takes its
// new value. Each partition's cache list is sorted by global id, so a thread
// per cached copy reads the changed bits and the owners' values in
// ascending order and writes the cache sequentially.
// With a cache budget only the kept copies (pull_list) are refreshed here.
// With frontier lists on, every copy whose vertex changed (cached or not)
// also joins the next frontier as slot n_vertices + g: the partition that
// holds it relaxes its in-edges from that vertex if the next superstep pushes.
__global__ void k_sync_pull(const SyncArgs a) {
    if (a.stats_out->skipped) return;   // uniform: Section III-B3 skip
    const bool list = a.stats_out->list_copies != 0ull;   // decided by k_sync_decide for every CTA
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto pull = [&](uint32_t g) -> bool {   // copy g takes its owner's new value if it changed
        const uint32_t gid = a.ghost_gid[g];
        const bool ch = ((a.changed_bits[gid >> 5] >> (gid & 31u)) & 1u) != 0u;
        // not cached: downloaded when used (lru.cu)
        if (ch && (!a.cached || (a.cached[g] & 1u))) a.ghost[g] = a.own_val[gid];
        return ch;
    };
    if (!list) {
        // four copies per thread and round, their loads issued together: a
        // thread keeps four independent chains (id -> changed bit -> value)
        // in flight instead of one
        const uint64_t stride = (uint64_t)gridDim.x * blockDim.x, n = a.n_pull;
        for (uint64_t g0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; g0 < n; g0 += 4u * stride) {
            uint32_t gid[4], word[4], val[4];
            bool wr[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) gid[k] = g0 + k * stride < n ? a.ghost_gid[g0 + k * stride] : 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) word[k] = g0 + k * stride < n ? a.changed_bits[gid[k] >> 5] : 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint64_t g = g0 + k * stride;
                // not cached: downloaded when used (lru.cu)
                wr[k] = g < n && ((word[k] >> (gid[k] & 31u)) & 1u) != 0u && (!a.cached || (a.cached[g] & 1u));
                val[k] = wr[k] ? a.own_val[gid[k]] : 0u;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (wr[k]) a.ghost[g0 + k * stride] = val[k];
        }
        return;
    }
    // The changed copies join the next frontier. A CTA takes a contiguous
    // chunk: pass 1 pulls and counts their items, one atomic reserves the
    // CTA's range of the list (one per warp made the list counter a
    // same-address bottleneck), pass 2 writes the items 256 copies at a time
    // at block-scanned offsets.
    __shared__ uint32_t s_items[8], s_edges[8];
    __shared__ unsigned long long s_base;
    const uint64_t per = ((((uint64_t)a.n_pull + gridDim.x - 1) / gridDim.x) + 255) & ~255ull;
    const uint64_t lo = min((uint64_t)a.n_pull, (uint64_t)blockIdx.x * per), hi = min((uint64_t)a.n_pull, lo + per);
    if (lo >= hi) return;   // uniform over the CTA
    auto degree = [&](uint32_t g) { return __ldg(a.out_ptr + a.n_vertices + g + 1) - __ldg(a.out_ptr + a.n_vertices + g); };
    uint32_t items = 0, edges = 0;
    for (uint64_t g = lo + threadIdx.x; g < hi; g += blockDim.x) {
        if (pull((uint32_t)g)) {
            const uint32_t d = degree((uint32_t)g);
            items += frontier_items(d);
            edges += d;
        }
    }
    items = __reduce_add_sync(0xFFFFFFFFu, items);
    edges = __reduce_add_sync(0xFFFFFFFFu, edges);
    if (lane == 0) {
        s_items[warp] = items;
        s_edges[warp] = edges;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t ti = 0, te = 0;
        for (int w = 0; w < 8; ++w) {
            ti += s_items[w];
            te += s_edges[w];
        }
        s_base = ti ? atomicAdd(&a.stats_out->list_ne, list_pack(ti, te)) >> 32 : 0ull;
    }
    __syncthreads();
    unsigned long long run = s_base;
    for (uint64_t r0 = lo; r0 < hi; r0 += blockDim.x) {
        const uint64_t g = r0 + threadIdx.x;
        bool ch = false;
        if (g < hi) {
            const uint32_t gid = a.ghost_gid[g];
            ch = ((a.changed_bits[gid >> 5] >> (gid & 31u)) & 1u) != 0u;
        }
        const uint32_t nit = ch ? frontier_items(degree((uint32_t)g)) : 0u;
        const uint32_t incl = warp_inclusive_scan(nit, lane);
        __syncthreads();   // the previous round's totals are read
        if (lane == 31) s_items[warp] = incl;
        __syncthreads();
        uint32_t before = 0, round = 0;
        for (int w = 0; w < 8; ++w) {
            if (w < warp) before += s_items[w];
            round += s_items[w];
        }
        if (round) frontier_write(a.fc, run + before, incl, nit, a.n_vertices + (uint32_t)g, lane);
        run += round;
    }
}

}  // namespace

cudaError_t launch_outdeg(const PartDev& p, const uint32_t* src, const uint32_t* ghost_gid,
                          uint32_t* outdeg, cudaStream_t s) {
    if (p.n_edges == 0) return cudaSuccess;
    // a few blocks per SM: each flushes its shared counters once
    const uint64_t blocks = std::min<uint64_t>((p.n_edges + 255) / 256, 152ull * 4);
    k_outdeg<false><<<(unsigned)blocks, 256, 0, s>>>(src, p.n_edges, p.n_own, p.v_begin, ghost_gid, outdeg, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_validate_csc(const uint32_t* col_ptr, uint32_t n_own, const uint32_t* src,
                                uint64_t n_edges, uint32_t n_local, uint32_t* err, cudaStream_t s) {
    const uint64_t work = std::max<uint64_t>(std::max<uint64_t>(n_edges, n_own), 1);
    const uint64_t blocks = std::min<uint64_t>((work + 255) / 256, 152ull * 16);
    k_validate<<<(unsigned)blocks, 256, 0, s>>>(col_ptr, n_own, src, n_edges, n_local, err);
    return cudaGetLastError();
}

cudaError_t launch_csc_offsets(const uint64_t* cp64, uint32_t n, uint64_t n_edges, uint32_t* cp32, uint32_t* err,
                               cudaStream_t s) {
    k_csc_offsets<<<(unsigned)std::min<uint64_t>(((uint64_t)n + 256) / 256, 152ull * 16), 256, 0, s>>>(cp64, n, n_edges,
                                                                                                       cp32, err);
    return cudaGetLastError();
}

cudaError_t launch_csc_sources(const uint32_t* src, uint64_t n_edges, uint32_t n_local, uint32_t* outdeg, uint32_t* err,
                               cudaStream_t s) {
    if (n_edges == 0) return cudaSuccess;
    const uint64_t blocks = std::min<uint64_t>((n_edges + 255) / 256, 152ull * 4);
    k_outdeg<true><<<(unsigned)blocks, 256, 0, s>>>(src, n_edges, n_local, 0u, nullptr, outdeg, err);
    return cudaGetLastError();
}

cudaError_t launch_begin(const BeginArgs& a, cudaStream_t s) {
    const uint64_t items = std::max<uint64_t>(a.n, a.n_ghost);
    const uint32_t blocks = (uint32_t)std::min<uint64_t>((items + 255) / 256, 152u * 8);
    k_begin<<<blocks, 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_count_dangling(const uint32_t* outdeg, uint32_t n, unsigned long long* out, cudaStream_t s) {
    const cudaError_t e = cudaMemsetAsync(out, 0, 8, s);
    if (e != cudaSuccess) return e;
    k_count_dangling<<<std::min<uint32_t>((n + 255) / 256, 152u * 8), 256, 0, s>>>(outdeg, n, out);
    return cudaGetLastError();
}

cudaError_t load_step_sums() {
    cudaFuncAttributes at;
    return cudaFuncGetAttributes(&at, k_step_sums);
}

cudaError_t launch_step_sums(const StepStats* ring, uint64_t first, uint64_t last, const uint32_t* err, StepReport* out,
                             cudaStream_t s) {
    if (last < first || last - first >= (uint64_t)kStatRing) return cudaErrorInvalidValue;
    k_step_sums<<<(unsigned)(last - first + 1), 32, 0, s>>>(ring, first, err, out);
    return cudaGetLastError();
}

cudaError_t launch_init_ghosts(Algo, uint32_t n_ghost, const uint32_t* gid, const uint32_t* own,
                               uint32_t* ghost, cudaStream_t s) {
    if (n_ghost == 0) return cudaSuccess;
    const uint32_t blocks = std::min<uint32_t>((n_ghost + 255) / 256, 152u * 8);
    k_init_ghosts<<<blocks, 256, 0, s>>>(n_ghost, gid, own, ghost);
    return cudaGetLastError();
}

cudaError_t launch_sync(const SyncArgs& a, uint32_t, cudaStream_t s) {
    if (a.n_parts == 0 || a.blocks_x == 0) return cudaSuccess;
    if (a.queue && a.max_words <= kQueueWords) {
        k_sync_queue<<<a.n_parts, kQueueBlock, 0, s>>>(a);
    } else {
        k_sync_decide<<<1, 32, 0, s>>>(a);
    }
    if (a.queue && a.max_words > kQueueWords) {
        dim3 grid(a.blocks_x, a.n_parts);
        k_sync_count<<<grid, kSyncBlock, 0, s>>>(a);
        k_sync_write<<<grid, kSyncBlock, 0, s>>>(a);
    }
    if (a.n_pull)
        k_sync_pull<<<std::min<uint32_t>((a.n_pull + 255) / 256, 152u * 16), 256, 0, s>>>(a);
    return cudaGetLastError();
}


}  // namespace gxp
