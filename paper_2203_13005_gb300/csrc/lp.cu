// Mode-label propagation superstep: the paper's LP workload (Section V-A)
// as the three template functions of Section IV-A1 with MSGGen = l[u],
// MSGMerge = the mode of a vertex's incoming labels (ties to the smallest
// label) and MSGApply = take it. Jacobi order: labels are read from the
// previous superstep's buffer and written to the other one.
//
//  * rows with 1..32 in-edges: slices of 32 rows, a row per lane. The lane
//    gathers its row's labels (a coalesced load of sources per column), sorts
//    them in registers with an odd-even merge network of the slice's width
//    and scans the runs: about 15 instructions per edge of 32 rows, so the
//    gathers set the pace. (Windows of 32 adjacent edges, one per lane, with
//    __match_any_sync per window were bound by that instruction: ER 2^20 in 8
//    partitions 169 us a superstep.)
//  * rows with 33..256 in-edges: a warp per row, 257..2048: a CTA per row,
//    up to 65,536: a CTA of 1,024 threads per row. All count the labels in a
//    shared-memory hash table (open addressing; a slot is taken by one
//    compare-and-swap, which also counts the label's first occurrence; a
//    warp's lanes that carry its first lane's label, once labels settle most
//    of them, count as one) and reduce (count, -label) over it. The largest
//    class makes several passes, each over the labels of one range of a
//    second hash, so that a 16,384-slot table holds them;
//  * hub rows (more in-edges): each chunk of 2048 is counted the same way
//    and its counts are added into the hub's global hash table; segments of
//    4096 slots that a label entered this superstep, spread over all CTAs,
//    reduce the tables into a 64-bit maximum per hub and empty them, and a
//    thread per hub applies.
//
// One partition: a row whose in-neighbours all kept their labels keeps its
// own, so once few labels change k_lp_mark marks the rows a change reaches
// (the changed vertices' out-neighbours) and the kernels skip the others.
// On R-MAT 20 (33.5 M edges) twelve of fifteen supersteps change a few
// hundred labels.
#include "frontier.cuh"

#include <algorithm>

namespace gxp {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kLpBlock = 256;
constexpr int kLpWarps = kLpBlock / 32;
constexpr int kGatherUnroll = 4;
constexpr int kBigBlock = 1024;
constexpr uint32_t kBigSlots = 16384;      // 128 KB of keys and counts
constexpr uint32_t kBigPerPass = 8192;     // labels a pass aims at
constexpr uint32_t kBigProbes = 256;       // of a label in a pass, in the first kBigTries tries
constexpr uint32_t kBigTries = 8;
constexpr uint32_t kAllProbes = 2 * kLpChunk - 1;   // of a label in the tables of shorter rows, all of their slots
constexpr uint32_t kLpHash = 0x9E3779B1u;  // a label's first slot: the top bits of its product

// the label of in-edge source s of partition P (previous superstep)
__device__ __forceinline__ uint32_t lp_label(const LpArgs& a, const LpPart& P, uint32_t s) {
    return s < P.n_own ? __ldg(a.own_cur + P.v_begin + s) : __ldg(a.ghost + P.ghost_base + (s - P.n_own));
}

// a min-label superstep after a quiet one changes nothing: the same holds
// here (same labels in, same labels out), so such a superstep returns at once
__device__ __forceinline__ bool lp_quiet(const LpArgs& a, int lane) {
    if (!a.skip_if_quiet) return false;
    unsigned long long c = a.stats_in->changed[lane] + a.stats_in->changed[lane + 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(kFull, c, o);
    return c == 0ull;
}

// Whether only the marked rows are recomputed (the same in every thread of
// the superstep's kernels): the vertices changed by the previous superstep
// have at most an eighth of the edges. Marking costs an atomic per out-edge,
// a recomputed row several instructions per in-edge; the eighth is the push
// direction's line.
__device__ __forceinline__ bool lp_sparse(const LpArgs& a) {
    return a.active != nullptr && !a.all_rows && (a.stats_in->list_ne & 0xFFFFFFFFull) * 8ull <= a.n_edges;
}

__device__ __forceinline__ bool lp_marked(const LpArgs& a, uint32_t g) {
    return (__ldg(a.active + (g >> 5)) >> (g & 31u)) & 1u;
}

// what a thread adds up: changed rows and the out-edges of their vertices, and
// (if only the marked rows are recomputed) the in-edges of the rows
struct LpAcc {
    uint32_t changed = 0, edges = 0, boundary = 0, read = 0;
};

// MSGApply
__device__ __forceinline__ void lp_apply(const LpArgs& a, uint32_t g, uint32_t label, LpAcc& acc) {
    const uint32_t old = a.own_cur[g];
    a.own_nxt[g] = label;
    if (label == old) return;
    ++acc.changed;
    if (a.active) acc.edges += __ldg(a.out_ptr + g + 1) - __ldg(a.out_ptr + g);
    if (a.changed_bits) atomicOr(a.changed_bits + (g >> 5), 1u << (g & 31u));
    if (a.boundary_bits) acc.boundary += (__ldg(a.boundary_bits + (g >> 5)) >> (g & 31u)) & 1u;
}

// a warp's sums into the superstep's stats
__device__ __forceinline__ void lp_count(const LpArgs& a, const LpAcc& acc, int lane, uint64_t slot) {
    const uint32_t c = __reduce_add_sync(kFull, acc.changed), e = __reduce_add_sync(kFull, acc.edges),
                   b = __reduce_add_sync(kFull, acc.boundary), r = __reduce_add_sync(kFull, acc.read);
    if (lane != 0) return;
    if (r) atomicAdd(&a.stats_out->push_edges, (unsigned long long)r);
    if (c == 0u) return;
    atomicAdd(&a.stats_out->changed[slot % kStatLanes], (unsigned long long)c);
    if (e) atomicAdd(&a.stats_out->list_ne, (unsigned long long)e);
    if (b) atomicAdd(&a.stats_out->boundary[slot % kStatLanes], (unsigned long long)b);
}

// (count, -label) as one key: the larger key is the more frequent label,
// and among equally frequent ones the smaller
__device__ __forceinline__ unsigned long long mode_key(uint32_t count, uint32_t label) {
    return ((unsigned long long)count << 32) | (unsigned long long)(~label);
}

// Start of a superstep (one partition): the bitmaps of the next superstep
// cleared and, when few labels changed, the rows those changes reach marked.
// A warp takes 32 vertices and walks the out-edges of the changed ones.
__global__ void __launch_bounds__(kLpBlock) k_lp_mark(const LpArgs a) {
    const int lane = threadIdx.x & 31;
    if (lp_quiet(a, lane)) return;
    const uint32_t words = (a.n_vertices + 31u) / 32u;
    for (uint32_t i = blockIdx.x * kLpBlock + threadIdx.x; i < words; i += gridDim.x * kLpBlock) {
        a.active_next[i] = 0u;
        a.changed_next[i] = 0u;
    }
    if (!lp_sparse(a)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) a.stats_out->pushed = 2ull;
    const uint32_t n_warps = gridDim.x * kLpWarps;
    for (uint32_t w = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; w < words; w += n_warps) {
        const uint32_t bits = __ldg(a.changed_prev + w);
        if (bits == 0u) continue;
        if (lane == 0) atomicOr(a.active + w, bits);   // their other buffer is brought up to date
        for (uint32_t b = bits; b; b &= b - 1u) {
            const uint32_t v = w * 32u + (uint32_t)(__ffs(b) - 1);
            const uint32_t e1 = __ldg(a.out_ptr + v + 1);
            for (uint32_t e = __ldg(a.out_ptr + v) + (uint32_t)lane; e < e1; e += 32u) {
                const uint32_t d = __ldg(a.out_dst + e);
                atomicOr(a.active + (d >> 5), 1u << (d & 31u));
            }
        }
    }
}

// Ascending sort of N registers: Batcher's odd-even merge sorting network
// (K. E. Batcher, Sorting networks and their applications, 1968), one
// template instance per comparator distance K of merge size P, so that every
// index is a constant. Entries known to be kInf at the end cost nothing:
// min(x, kInf) folds away.
template <int N, int P, int K>
__device__ __forceinline__ void sort_step(uint32_t (&x)[N]) {
#pragma unroll
    for (int t = K % P; t < N - K; ++t) {
        if ((t - K % P) % (2 * K) < K && t / (2 * P) == (t + K) / (2 * P)) {
            const uint32_t lo = min(x[t], x[t + K]), hi = max(x[t], x[t + K]);
            x[t] = lo;
            x[t + K] = hi;
        }
    }
    if constexpr (K > 1) sort_step<N, P, K / 2>(x);
    else if constexpr (2 * P < N) sort_step<N, 2 * P, 2 * P>(x);
}

// One slice of at most W columns: lane l's row.
template <bool kOnePart, int W>
__device__ __forceinline__ void lp_slice(const LpArgs& a, const LpPart& P, const SellSlice& sl, uint32_t row, bool want,
                                         int lane, LpAcc& acc) {
    constexpr int N = W <= 4 ? 4 : W <= 8 ? 8 : W <= 16 ? 16 : 32;   // the network's size
    const uint32_t* col = P.sell + sl.off + lane;
    uint32_t x[N];
#pragma unroll
    for (int k = 0; k < W; ++k) x[k] = (uint32_t)k < sl.width ? __ldcs(col + 32 * k) : kInf;
#pragma unroll
    for (int k = 0; k < W; ++k) {
        if constexpr (kOnePart) x[k] = (uint32_t)k < sl.width ? __ldg(a.own_cur + x[k]) : kInf;   // padding: the identity slot
        else x[k] = (uint32_t)k < sl.width ? lp_label(a, P, x[k]) : kInf;
    }
#pragma unroll
    for (int k = W; k < N; ++k) x[k] = kInf;
    sort_step<N, 1, 1>(x);
    // runs of equal labels, ascending: the first longest one is the mode
    uint32_t best = 1u, mode = x[0], run = 1u;
#pragma unroll
    for (int k = 1; k < W; ++k) {
        run = x[k] == x[k - 1] ? run + 1u : 1u;
        if (run > best && x[k] != kInf) {
            best = run;
            mode = x[k];
        }
    }
    if (want && mode != kInf) lp_apply(a, P.v_begin + row, mode, acc);   // (a row without in-edges keeps its label)
}

// kOnePart: one partition (no cached copies): every source is a local
// index into the label array
template <bool kOnePart>
__global__ void __launch_bounds__(kLpBlock) k_lp_slices(const LpArgs a) {
    const int lane = threadIdx.x & 31;
    if (blockIdx.x == 0 && a.stats_clear != nullptr) {
        // zero the ring slot two supersteps ahead (never read or written by this one)
        unsigned long long* z = reinterpret_cast<unsigned long long*>(a.stats_clear);
        for (uint32_t i = threadIdx.x; i < sizeof(StepStats) / 8; i += kLpBlock) z[i] = 0ull;
    }
    if (!kOnePart)   // (one partition: k_lp_mark)
        for (uint64_t i = (uint64_t)blockIdx.x * kLpBlock + threadIdx.x; i <= a.n_vertices / 32u;
             i += (uint64_t)gridDim.x * kLpBlock)
            a.changed_next[i] = 0u;
    if (lp_quiet(a, lane)) return;
    const bool sparse = kOnePart && lp_sparse(a);
    const uint64_t w0 = ((uint64_t)blockIdx.x * kLpBlock + threadIdx.x) >> 5;
    const uint64_t nw = ((uint64_t)gridDim.x * kLpBlock) >> 5;
    LpAcc acc;
    for (uint64_t i = w0; i < a.n_slices; i += nw) {
        const SellSlice sl = a.slices[i];
        const LpPart P = a.parts[kOnePart ? 0 : sl.part];
        const uint32_t row = __ldg(P.perm + sl.row0 + lane);
        bool want = row != kSellPad;
        if (sparse) {
            want = want && lp_marked(a, row);
            if (!__any_sync(kFull, want)) continue;
            if (want) acc.read += __ldg(a.col_ptr + row + 1) - __ldg(a.col_ptr + row);
        }
        switch ((sl.width + 3u) / 4u) {
            case 1: lp_slice<kOnePart, 4>(a, P, sl, row, want, lane, acc); break;
            case 2: lp_slice<kOnePart, 8>(a, P, sl, row, want, lane, acc); break;
            case 3: lp_slice<kOnePart, 12>(a, P, sl, row, want, lane, acc); break;
            case 4: lp_slice<kOnePart, 16>(a, P, sl, row, want, lane, acc); break;
            case 5: lp_slice<kOnePart, 20>(a, P, sl, row, want, lane, acc); break;
            case 6: lp_slice<kOnePart, 24>(a, P, sl, row, want, lane, acc); break;
            case 7: lp_slice<kOnePart, 28>(a, P, sl, row, want, lane, acc); break;
            default: lp_slice<kOnePart, 32>(a, P, sl, row, want, lane, acc); break;
        }
    }
    lp_count(a, acc, lane, w0);
}

// add `count` occurrences of `label` to a hub's global hash table of
// 2^log2_size slots (open addressing with linear probing; a table of 2^k >= 2
// n slots, or 2^32, has a free slot for every distinct label, so one is
// always found)
__device__ __forceinline__ uint32_t lp_table_add(uint32_t* keys, uint32_t* counts, uint32_t log2_size,
                                                 uint32_t label, uint32_t count) {
    const uint32_t mask = log2_size >= 32u ? 0xFFFFFFFFu : (1u << log2_size) - 1u;
    uint32_t slot = (label * kLpHash) >> (32u - log2_size);
    for (uint64_t probe = 0; probe <= mask; ++probe) {
        const uint32_t k = atomicCAS(keys + slot, kInf, label);
        if (k == kInf || k == label) {
            atomicAdd(counts + slot, count);
            return slot;
        }
        slot = (slot + 1u) & mask;
    }
    return 0u;
}

// Add a warp's labels (where `has`) to a shared-memory table of 2^log2_size
// slots. A slot's count is its label's occurrences less one, so a label
// that occurs once costs the compare-and-swap alone. `hash` is the label's, its
// top bits the first slot. Returns false for a lane whose label found no slot
// in `probes` + 1 of them. All 32 lanes must call it.
__device__ __forceinline__ bool lp_warp_add(uint32_t* keys, uint32_t* more, uint32_t log2_size, uint32_t label,
                                            uint32_t hash, uint32_t probes, bool has, int lane) {
    const unsigned act = __ballot_sync(kFull, has);
    if (act == 0u) return true;
    // lanes that carry the first lane's label count as one
    const int first = __ffs(act) - 1;
    const uint32_t l0 = __shfl_sync(kFull, label, first);
    const unsigned same = __ballot_sync(kFull, has && label == l0);
    if (!has || (label == l0 && lane != first)) return true;
    const uint32_t c = lane == first ? (uint32_t)__popc(same) : 1u;
    const uint32_t mask = (1u << log2_size) - 1u;
    uint32_t slot = hash >> (32u - log2_size);
    for (uint32_t probe = 0; probe <= probes; ++probe) {
        const uint32_t k = atomicCAS(keys + slot, kInf, label);
        if (k == kInf || k == label) {
            const uint32_t add = k == kInf ? c - 1u : c;
            if (add) atomicAdd(more + slot, add);
            return true;
        }
        slot = (slot + 1u) & mask;
    }
    return false;
}

template <int kThreads>
__device__ __forceinline__ unsigned long long block_max(unsigned long long v, unsigned long long* s_red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(kFull, v, o));
    if (lane == 0) s_red[warp] = v;
    __syncthreads();
    unsigned long long b = 0ull;
    for (int w = 0; w < kThreads / 32; ++w) b = max(b, s_red[w]);
    return b;
}

// Which of a CTA's next kThreads rows (first, first + step, ... below n) are
// wanted, a thread asking for each: a superstep that recomputes few rows then
// costs a look at 32 of them where one row after another would be a chain of
// two loads each. Every thread gets the bits; returns whether there are any.
template <int kThreads>
__device__ __forceinline__ bool lp_wanted(const LpArgs& a, const LpRow* rows, uint64_t first, uint64_t step, uint64_t n,
                                          bool sparse, uint32_t* s_want) {
    const uint64_t mine = first + (uint64_t)threadIdx.x * step;
    const bool want = mine < n && (!sparse || lp_marked(a, __ldg(&rows[mine].g)));
    const unsigned b = __ballot_sync(kFull, want);
    if ((threadIdx.x & 31) == 0) s_want[threadIdx.x >> 5] = b;
    return __syncthreads_or(want) != 0;
}

// Rows of 33..256 in-edges, a warp each (8 rows in flight per CTA): the
// warp counts the row's labels in its own shared-memory hash table (2^k >=
// 2n slots, at most 512), takes the largest (count, -label) over the table
// with a warp reduction and empties it.
__global__ void __launch_bounds__(kLpBlock) k_lp_warp_rows(const LpArgs a) {
    __shared__ uint32_t t_key[kLpWarps][2 * kLpWarpRow], t_more[kLpWarps][2 * kLpWarpRow];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lp_quiet(a, lane)) return;
    const bool sparse = lp_sparse(a);
    uint32_t* keys = t_key[warp];   // a warp's own table: no other warp waits for it
    uint32_t* more = t_more[warp];
    for (uint32_t i = (uint32_t)lane; i < 2 * kLpWarpRow; i += 32u) {
        keys[i] = kInf;
        more[i] = 0u;
    }
    __syncwarp();
    const uint64_t w0 = ((uint64_t)blockIdx.x * kLpBlock + threadIdx.x) >> 5;
    const uint64_t nw = ((uint64_t)gridDim.x * kLpBlock) >> 5;
    LpAcc acc;
    // the warp's next 32 rows, w0, w0 + nw, ...: lane j asks whether row j is wanted
    for (uint64_t r0 = w0; r0 < a.n_warp_rows; r0 += 32u * nw) {
        const uint64_t mine = r0 + (uint64_t)lane * nw;
        const bool want = mine < a.n_warp_rows && (!sparse || lp_marked(a, __ldg(&a.warp_rows[mine].g)));
        for (unsigned todo = __ballot_sync(kFull, want); todo; todo &= todo - 1u) {
            const LpRow r = a.warp_rows[r0 + (uint64_t)(__ffs(todo) - 1) * nw];
            const LpPart P = a.parts[r.part];
            const uint32_t n = r.n;
            uint32_t lg = 1;
            while ((1u << lg) < 2u * n) ++lg;
            for (uint32_t i0 = 0; i0 < n; i0 += 32u * kGatherUnroll) {
                uint32_t sv[kGatherUnroll], lab[kGatherUnroll];
#pragma unroll
                for (int q = 0; q < kGatherUnroll; ++q) {
                    const uint32_t i = i0 + 32u * q + (uint32_t)lane;
                    sv[q] = i < n ? __ldg(P.src + r.e0 + i) : 0u;
                }
#pragma unroll
                for (int q = 0; q < kGatherUnroll; ++q) {
                    const uint32_t i = i0 + 32u * q + (uint32_t)lane;
                    lab[q] = i < n ? lp_label(a, P, sv[q]) : 0u;
                }
#pragma unroll
                for (int q = 0; q < kGatherUnroll; ++q)   // (a table of 2n slots never fills)
                    lp_warp_add(keys, more, lg, lab[q], lab[q] * kLpHash, kAllProbes,
                                i0 + 32u * q + (uint32_t)lane < n, lane);
            }
            __syncwarp();
            unsigned long long best = 0ull;
            for (uint32_t i = (uint32_t)lane; i < (1u << lg); i += 32u) {
                const uint32_t k = keys[i];
                if (k != kInf) {
                    best = max(best, mode_key(more[i] + 1u, k));
                    keys[i] = kInf;
                    more[i] = 0u;
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(kFull, best, o));
            if (lane == 0) {
                lp_apply(a, r.g, ~(uint32_t)best, acc);
                if (sparse) acc.read += n;
            }
            __syncwarp();
        }
    }
    lp_count(a, acc, lane, w0);
}

// Rows of 257..2048 in-edges (hub = kInf) and chunks of 2048 of hub rows: the
// CTA counts the labels in a shared-memory hash table (2^k >= 2n slots),
// then takes the mode (a row) or adds its counts into the hub's table.
__global__ void __launch_bounds__(kLpBlock) k_lp_rows(const LpArgs a) {
    __shared__ uint32_t t_key[2 * kLpChunk], t_more[2 * kLpChunk];
    __shared__ unsigned long long s_red[kLpWarps];
    __shared__ uint32_t s_want[kLpWarps];
    const int tid = threadIdx.x, lane = tid & 31;
    if (lp_quiet(a, lane)) return;
    const bool sparse = lp_sparse(a);
    bool empty = false;   // the table is set up
    LpAcc acc;
    for (uint64_t c0 = blockIdx.x; c0 < a.n_chunks; c0 += (uint64_t)gridDim.x * kLpBlock) {
        if (!lp_wanted<kLpBlock>(a, a.chunks, c0, gridDim.x, a.n_chunks, sparse, s_want)) continue;
        if (!empty) {
            for (uint32_t i = (uint32_t)tid; i < 2 * kLpChunk; i += kLpBlock) {
                t_key[i] = kInf;
                t_more[i] = 0u;
            }
            empty = true;
            __syncthreads();
        }
        for (int wd = 0; wd < kLpWarps; ++wd)
            for (unsigned todo = s_want[wd]; todo; todo &= todo - 1u) {
                const LpRow r = a.chunks[c0 + (uint64_t)(32 * wd + __ffs(todo) - 1) * gridDim.x];
                const LpPart P = a.parts[r.part];
                const uint32_t n = r.n;
                uint32_t lg = 1;
                while ((1u << lg) < 2u * n) ++lg;
                const uint32_t size = 1u << lg;
                for (uint32_t i0 = 0; i0 < n; i0 += (uint32_t)kLpBlock * kGatherUnroll) {
                    uint32_t sv[kGatherUnroll], lab[kGatherUnroll];
#pragma unroll
                    for (int q = 0; q < kGatherUnroll; ++q) {
                        const uint32_t i = i0 + (uint32_t)q * kLpBlock + (uint32_t)tid;
                        sv[q] = i < n ? __ldg(P.src + r.e0 + i) : 0u;
                    }
#pragma unroll
                    for (int q = 0; q < kGatherUnroll; ++q) {
                        const uint32_t i = i0 + (uint32_t)q * kLpBlock + (uint32_t)tid;
                        lab[q] = i < n ? lp_label(a, P, sv[q]) : 0u;
                    }
#pragma unroll
                    for (int q = 0; q < kGatherUnroll; ++q)
                        lp_warp_add(t_key, t_more, lg, lab[q], lab[q] * kLpHash, kAllProbes,
                                    i0 + (uint32_t)q * kLpBlock + (uint32_t)tid < n, lane);
                }
                __syncthreads();
                // read the counts and empty the table for the next row
                unsigned long long best = 0ull;
                for (uint32_t i = (uint32_t)tid; i < size; i += kLpBlock) {
                    const uint32_t k = t_key[i];
                    if (k != kInf) {
                        const uint32_t cnt = t_more[i] + 1u;
                        if (r.hub == kInf) {
                            best = max(best, mode_key(cnt, k));
                        } else {
                            const LpHub H = a.hubs[r.hub];
                            const uint32_t slot = lp_table_add(a.keys + H.table, a.counts + H.table, H.log2_size, k, cnt);
                            a.seg_used[H.seg0 + slot / kLpSegment] = 1u;   // same value from every writer
                        }
                        t_key[i] = kInf;
                        t_more[i] = 0u;
                    }
                }
                if (r.hub == kInf) {
                    best = block_max<kLpBlock>(best, s_red);
                    if (tid == 0) lp_apply(a, r.g, ~(uint32_t)best, acc);
                }
                if (tid == 0 && sparse) acc.read += n;
                __syncthreads();   // the table and s_red are reused by the next row
            }
        __syncthreads();   // s_want is read
    }
    if (tid < 32) lp_count(a, acc, lane, blockIdx.x);
}

// A permutation of the labels for each try but the first: MurmurHash3's 32-bit
// finalizer (A. Appleby) of the label with the try's number mixed in.
__device__ __forceinline__ uint32_t lp_rehash(uint32_t x, uint32_t attempt) {
    x ^= attempt * 0x632BE5ABu;
    x = (x ^ (x >> 16)) * 0x85EBCA6Bu;
    x = (x ^ (x >> 13)) * 0xC2B2AE35u;
    return x ^ (x >> 16);
}

// Rows of 2049..65,536 in-edges, a large CTA each: `passes` sweeps over the
// row, pass p counting the labels whose second hash falls in its range. A
// label that finds no slot within kBigProbes starts the row again with other
// hashes, and with twice as many passes if the table had filled up. Labels can
// be chosen to crowd under one hash (60,000 of them would have needed 262,144
// passes under the first one), but few labels crowd under several: what five
// tries in a row put into one pass is one 2^25th of the 32-bit numbers, 128
// labels. After kBigTries a label may look at every slot. So a row takes at
// most some hundreds of passes.
__global__ void __launch_bounds__(kBigBlock) k_lp_big(const LpArgs a) {
    extern __shared__ uint32_t s_table[];
    uint32_t* t_key = s_table;
    uint32_t* t_more = s_table + kBigSlots;
    __shared__ unsigned long long s_red[kBigBlock / 32];
    __shared__ uint32_t s_want[kBigBlock / 32];
    __shared__ uint32_t s_taken;   // slots, in a try that failed
    const int tid = threadIdx.x, lane = tid & 31;
    if (lp_quiet(a, lane)) return;
    const bool sparse = lp_sparse(a);
    bool empty = false;   // the table is set up
    LpAcc acc;
    for (uint64_t c0 = blockIdx.x; c0 < a.n_big; c0 += (uint64_t)gridDim.x * kBigBlock) {
        if (!lp_wanted<kBigBlock>(a, a.big, c0, gridDim.x, a.n_big, sparse, s_want)) continue;
        if (!empty) {
            for (uint32_t i = (uint32_t)tid; i < kBigSlots; i += kBigBlock) {
                t_key[i] = kInf;
                t_more[i] = 0u;
            }
            empty = true;
            __syncthreads();
        }
        for (int wd = 0; wd < kBigBlock / 32; ++wd)
            for (unsigned todo = s_want[wd]; todo; todo &= todo - 1u) {
                const LpRow r = a.big[c0 + (uint64_t)(32 * wd + __ffs(todo) - 1) * gridDim.x];
                const LpPart P = a.parts[r.part];
                const uint32_t n = r.n;
                uint32_t passes = (n + kBigPerPass - 1) / kBigPerPass;
                uint32_t lg = 12;
                while (lg < 14u && (1u << lg) < 2u * min(n, kBigPerPass)) ++lg;
                const uint32_t size = 1u << lg;
                unsigned long long best = 0ull;
                uint32_t attempt = 0;
                for (uint32_t p = 0; p < passes; ++p) {
                    // count the labels of pass p; false: one found no slot. The first
                    // try is compiled apart, without what the others need.
                    auto count = [&](auto first) {
                        constexpr bool kFirst = decltype(first)::value;
                        const uint32_t probes = kFirst || attempt < kBigTries ? kBigProbes : size - 1u;
                        bool ok = true;
                        for (uint32_t i0 = 0; i0 < n; i0 += (uint32_t)kBigBlock * kGatherUnroll) {
                            uint32_t sv[kGatherUnroll], lab[kGatherUnroll];
#pragma unroll
                            for (int q = 0; q < kGatherUnroll; ++q) {
                                const uint32_t i = i0 + (uint32_t)q * kBigBlock + (uint32_t)tid;
                                sv[q] = i < n ? __ldg(P.src + r.e0 + i) : 0u;
                            }
#pragma unroll
                            for (int q = 0; q < kGatherUnroll; ++q) {
                                const uint32_t i = i0 + (uint32_t)q * kBigBlock + (uint32_t)tid;
                                lab[q] = i < n ? lp_label(a, P, sv[q]) : 0u;
                            }
#pragma unroll
                            for (int q = 0; q < kGatherUnroll; ++q) {
                                const uint32_t key = kFirst ? lab[q] : lp_rehash(lab[q], attempt);
                                const bool mine = i0 + (uint32_t)q * kBigBlock + (uint32_t)tid < n && (kFirst || ok) &&
                                                  __umulhi(key * 0x85EBCA6Bu, passes) == p;
                                ok &= lp_warp_add(t_key, t_more, lg, lab[q], key * kLpHash, probes, mine, lane);
                            }
                        }
                        return ok;
                    };
                    bool ok = attempt == 0u ? count(std::true_type{}) : count(std::false_type{});
                    if (tid == 0) s_taken = 0u;
                    ok = __syncthreads_and(ok);
                    uint32_t taken = 0;
                    for (uint32_t i = (uint32_t)tid; i < size; i += kBigBlock) {
                        const uint32_t k = t_key[i];
                        if (k != kInf) {
                            if (ok) best = max(best, mode_key(t_more[i] + 1u, k));
                            t_key[i] = kInf;
                            t_more[i] = 0u;
                            ++taken;
                        }
                    }
                    if (!ok) {   // again, with other hashes (the same in every thread)
                        taken = __reduce_add_sync(kFull, taken);
                        if (lane == 0) atomicAdd(&s_taken, taken);
                        __syncthreads();
                        if (s_taken > size / 4u * 3u) passes = min(2u * passes, 1u << 30);
                        ++attempt;
                        best = 0ull;
                        p = 0xFFFFFFFFu;   // ++ -> 0
                    }
                    __syncthreads();
                }
                best = block_max<kBigBlock>(best, s_red);
                if (tid == 0) {
                    lp_apply(a, r.g, ~(uint32_t)best, acc);
                    if (sparse) acc.read += n;
                }
                __syncthreads();   // s_red is reused by the next row
            }
        __syncthreads();   // s_want is read
    }
    if (tid < 32) lp_count(a, acc, lane, blockIdx.x + 31u);
}

// hub tables, a segment per CTA: the best (count, -label) of the segment
// goes into the hub's 64-bit maximum, and the segment is emptied
__global__ void __launch_bounds__(kLpBlock) k_lp_segments(const LpArgs a) {
    __shared__ unsigned long long s_red[kLpWarps];
    const int tid = threadIdx.x, lane = tid & 31;
    if (lp_quiet(a, lane)) return;
    for (uint32_t sg = blockIdx.x; sg < a.n_segments; sg += gridDim.x) {
        if (!a.seg_used[sg]) continue;   // no label took a slot here this superstep (uniform in the CTA)
        const LpSegment S = a.segments[sg];
        uint32_t* keys = a.keys + S.slot0;
        uint32_t* counts = a.counts + S.slot0;
        unsigned long long best = 0ull;
        for (uint32_t i = (uint32_t)tid; i < S.n; i += kLpBlock) {
            const uint32_t k = keys[i];
            if (k != kInf) {
                best = max(best, mode_key(counts[i], k));
                keys[i] = kInf;   // empty again for the next superstep
                counts[i] = 0u;
            }
        }
        best = block_max<kLpBlock>(best, s_red);
        if (tid == 0) {
            if (best) atomicMax(a.hub_best + S.hub, best);
            a.seg_used[sg] = 0u;
        }
        __syncthreads();
    }
}

// a thread per hub: apply the mode its segments agreed on (none: the hub
// was not recomputed)
__global__ void k_lp_hubs(const LpArgs a) {
    const int lane = threadIdx.x & 31;
    if (lp_quiet(a, lane)) return;
    LpAcc acc;
    for (uint32_t h = blockIdx.x * blockDim.x + threadIdx.x; h < a.n_hubs; h += gridDim.x * blockDim.x) {
        const unsigned long long best = a.hub_best[h];
        if (best == 0ull) continue;
        a.hub_best[h] = 0ull;
        lp_apply(a, a.hubs[h].g, ~(uint32_t)best, acc);
    }
    lp_count(a, acc, lane, blockIdx.x * 8u + (threadIdx.x >> 5) + 17u);
}

}  // namespace

cudaError_t launch_lp_superstep(const LpArgs& a, cudaStream_t s) {
    if (a.active)
        k_lp_mark<<<(uint32_t)std::min<uint64_t>((a.n_vertices / 32u + 8u) / 8u, 152ull * 8), kLpBlock, 0, s>>>(a);
    // The slices run partition after partition, wide ones first. Where labels
    // and copies do not fit L2 (129 MB) only a grid of a warp per slice keeps
    // to that order, so that one partition's copies are gathered from at a
    // time; where they fit, 4 CTAs an SM stride over the slices. ER graphs in 8
    // partitions, m = 16 n, a run of 14 or 15 supersteps, a warp per slice / 4
    // CTAs an SM: n = 2^24 (537 MB) 19.6 / 26.1 ms, 2^23 (268 MB) 9.4 / 9.7 ms,
    // 2^22 (134 MB) 4.9 / 4.7 ms; one partition of 2^24 (67 MB) 15.8 / 13.5 ms.
    // (64 CTAs an SM, each striding over every partition: 59.5 ms at 2^24.)
    const bool in_order = 4ull * ((uint64_t)a.n_vertices + a.n_ghost) > (160ull << 20);
    const uint32_t g_slices = (uint32_t)std::max<uint64_t>(
        1, std::min<uint64_t>((a.n_slices + 7ull) / 8, in_order ? 1ull << 24 : 152ull * 4));
    if (a.n_parts == 1) k_lp_slices<true><<<g_slices, kLpBlock, 0, s>>>(a);   // also clears the stat slot
    else k_lp_slices<false><<<g_slices, kLpBlock, 0, s>>>(a);                 // two supersteps ahead
    if (a.n_big) {
        const int smem = 8 * (int)kBigSlots;
        const cudaError_t e = cudaFuncSetAttribute(k_lp_big, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        k_lp_big<<<(uint32_t)std::min<uint64_t>(a.n_big, 152ull), kBigBlock, smem, s>>>(a);
    }
    if (a.n_chunks) k_lp_rows<<<(uint32_t)std::min<uint64_t>(a.n_chunks, 152ull * 6), kLpBlock, 0, s>>>(a);
    if (a.n_warp_rows)
        k_lp_warp_rows<<<(uint32_t)std::min<uint64_t>((a.n_warp_rows + 7) / 8, 152ull * 6), kLpBlock, 0, s>>>(a);
    if (a.n_segments)
        k_lp_segments<<<(uint32_t)std::min<uint64_t>(a.n_segments, 152ull * 8), kLpBlock, 0, s>>>(a);
    if (a.n_hubs) k_lp_hubs<<<(uint32_t)std::min<uint64_t>((a.n_hubs + 255) / 256, 152ull * 4), 256, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace gxp
