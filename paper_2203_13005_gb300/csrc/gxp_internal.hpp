// Internal declarations of libgxp: device data layout, kernel launchers and
// the host-side context. Not part of the C-ABI (include/gxp.h is).
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include "gxp.h"

namespace gxp {

constexpr uint32_t kInf = 0xFFFFFFFFu;
constexpr int kBlock = 128;          // threads per superstep CTA (4 independent warps)
constexpr uint32_t kVertexCost = 4;  // merge-path weight of a vertex end when cutting tiles
constexpr int kStatLanes = 64;       // stat accumulators are spread over lanes to
                                     // avoid same-address atomic serialization
constexpr int kStatRing = 64;        // superstep stat slots kept on the device

// Device error word bits (ORed by kernels, read by the host at sync points).
constexpr uint32_t kErrBounds = 1u;
constexpr uint32_t kErrTimeout = 2u;
constexpr uint32_t kErrDrain = 4u;     // a give-up drain ran out before its copies landed
constexpr uint32_t kErrInput = 8u;     // CSC offsets not running from 0 to n_edges, non-decreasing

// Fixed-point scale of the exact global sums (dangling mass, L1 delta):
// an fp32 value x in [0, 2] is held as round(x * 2^60) in a uint64.
constexpr int kFxShift = 60;

enum class Algo : int { SSSP = 0, CC = 1, PR = 2, LP = 3 };

// One edge block ("tile") paired with its vertex block (Section II-B): the
// in-edges [e0, e0+ne) of local destinations [v0, v0+nv) of one partition.
// Blocks are cut at vertex boundaries except inside hub vertices whose
// in-degree exceeds hub_items; such a vertex spans several blocks, and its
// partial merges are combined by the last block to finish it.
struct Tile {
    uint32_t v0;       // first local destination vertex
    uint32_t nv;       // destination vertices touched (incl. an open head/tail)
    uint32_t e0;       // first edge (partition-local CSC index)
    uint32_t ne;       // edge count
    uint32_t part;     // partition index
    uint32_t flags;    // kHeadOpen | kTailOpen
    uint32_t hub_t0;   // kHeadOpen: global index of the tile where the head vertex starts
    uint32_t nparts;   // tile that starts an open tail vertex: tiles that vertex spans
};
constexpr uint32_t kHeadOpen = 1u;
constexpr uint32_t kTailOpen = 2u;

// Sliced-ELL layout of the non-hub rows (SELL-32-sigma): rows are sorted by
// in-degree inside windows of kSellWindow rows and grouped into slices of 32;
// several partitions store a slice's in-edges column-major, a single
// partition as lane groups (sweep_lanes), padded with the partition's
// padding id.
struct SellSlice {
    uint32_t part;     // partition index; one partition: rows of the slice if they are consecutive
                       // vertices (first ..), else 0
    uint32_t row0;     // first entry of the slice in the partition's perm array
    uint32_t width;    // edges per row slot (the slice's largest in-degree)
    uint32_t first;
    uint64_t off;      // first element of the slice in the partition's sell arrays
};
constexpr uint32_t kSellPad = 0xFFFFFFFFu;   // empty row slot of a slice (perm)
// Storage of a slice. `cols` = 0 (several partitions): column by column,
// element k of row slot r at 32 k + r. Else (one partition) a slice wider
// than `cols` columns spreads each row over L lanes, L the smallest power of
// two (at most 32) that brings its columns down to `cols`: the slice is L
// sub-slices of 32 / L rows, edge k of a row in lane k % L of its lane group
// and column k / L, and columns are stored in groups of 4, so that a lane
// reads 4 of its sources with one 128-bit load. kSweepCols: fewer columns, so
// more items and lanes, pad more and measured no faster at any size (R-MAT and
// uniform graphs of 2^19 to 2^24 edges at 4 / 8 / 16, us a run: PageRank R-MAT
// 2^20 edges 263 / 242 / 235, 2^22 468 / 409 / 389, 2^24 1,135 / 946 / 865; SSSP
// 179 / 174 / 167, 238 / 228 / 220, 520 / 492 / 462).
constexpr uint32_t kSweepCols = 16;
__host__ __device__ constexpr uint32_t sweep_lanes(uint32_t width, uint32_t cols) {
    uint32_t l = 1;
    while (l < 32u && width > cols * l) l *= 2;
    return l;
}
// columns a sub-slice stores
__host__ __device__ constexpr uint32_t sweep_cols(uint32_t width, uint32_t lanes) {
    return ((width + lanes - 1) / lanes + 3u) & ~3u;
}
__host__ __device__ constexpr uint64_t sell_words(uint32_t width, uint32_t cols) {
    if (!cols) return 32ull * width;
    const uint32_t l = sweep_lanes(width, cols);
    return 32ull * l * sweep_cols(width, l);
}
constexpr uint32_t kSellWindow = 65536;      // rows sorted by degree within windows of this size

// A slice of the in-edges of one hub row (in-degree above the SELL limit),
// reduced by one warp; the last part of a row to arrive combines all parts.
struct HubPart {
    uint32_t v;        // partition-local destination vertex
    uint32_t part;     // partition index
    uint32_t e0;       // first edge in the partition's hub edge arrays
    uint32_t ne;       // edges in this part
    uint32_t t0;       // global index of the row's first part
    uint32_t nparts;   // parts of this row
    uint32_t pad[2];
};

// Per-partition device view (array in device memory, indexed by Tile::part).
struct PartDev {
    const uint32_t* col_ptr;   // [n_own + 1] CSC offsets, padded to a multiple of 4 + 4
    const uint32_t* src;       // [n_edges] local source index, padded likewise
    const uint32_t* w;         // [n_edges] weights or nullptr
    uint32_t n_own;            // owned vertices
    uint32_t v_begin;          // global id of local vertex 0
    uint32_t n_ghost;          // cached remote vertices (local ids n_own ..)
    uint32_t ghost_base;       // offset of this partition's ghosts in the ghost array
    uint64_t n_edges;
    // sliced-ELL layout (engine path)
    const uint32_t* sell_src;  // slices (sell_words), pad_id in empty slots
    const uint32_t* sell_w;    // weights in the same layout, or nullptr
    const uint32_t* perm;      // slice row slot -> local vertex (kSellPad = empty)
    const uint32_t* hsrc;      // hub rows' in-edges, row after row
    const uint32_t* hw;        // and weights, or nullptr
    // local id of the identity slot that empty SELL slots name: one partition,
    // n_own (own[V], past the last vertex); several, the slot past every
    // partition's cached copies (ghost[n_ghost_total]). The slot holds the
    // merge's identity (0 for sums, INF for minima) and is never written by
    // a superstep, so padding needs no test in the kernel.
    uint32_t pad_id;
    uint32_t pad1;
};

// Accumulators of one superstep (one ring slot).
struct StepStats {
    unsigned long long changed[kStatLanes];
    unsigned long long dangling_fx[kStatLanes];   // sum of fx(r) over out-degree-0 vertices
    unsigned long long l1_fx[kStatLanes];         // sum |fx(r_new) - fx(r_old)|
    unsigned long long boundary[kStatLanes];      // partitions: changed boundary vertices
    unsigned long long boundary_changed;          // pairs uploaded by the sync (all partitions)
    unsigned long long skipped;                   // 1 if the exchange was skipped
    // frontier of the next superstep (min-label algorithms, single partition):
    // items appended to its list (high 32 bits) and the out-edges of the
    // vertices they cover (low 32 bits), advanced together by one atomic
    unsigned long long list_ne;
    unsigned long long pushed;                    // 1: the superstep ran in push direction, 2: LP recomputed some
    unsigned long long push_edges;                //    rows; out-edges relaxed, the rows' in-edges
    unsigned long long exchanged;                 // 1 once the superstep's exchange between
                                                  // partitions ran (skipped or not)
    unsigned long long downloads;                 // copies the superstep used that were not cached
    // 1: the exchange lists the changed cached copies in the next frontier.
    // Decided once by k_sync_decide from the own vertices' appends and the
    // changed boundary vertices: the copies' appends then advance list_ne,
    // so a test each CTA of k_sync_pull made for itself would see a moving
    // count and the CTAs could disagree (some copies listed, others not).
    unsigned long long list_copies;
    // 1: the superstep pulled without listing its changed vertices: with
    // several partitions (FrontierCfg::list_max_changed) the next one must
    // pull too; one partition holds them in a bitmap (SweepArgs::bits), which
    // the next superstep lists if it pushes, reserving list places here
    unsigned long long unlisted;
    unsigned long long list_cursor;
};
// A superstep's stats, summed over their lanes.
struct StepSum {
    unsigned long long changed, dangling_fx, l1_fx, pushed, push_edges;
    unsigned long long boundary_changed, skipped, exchanged, downloads;   // several partitions
};
// What supersteps leave in pinned host memory, by ring slot: written by the
// exchange's decision (several partitions) or by launch_step_sums (one) and
// read once the stream is synchronized, in place of a copy of the ring.
struct StepReport {
    StepSum sum[kStatRing];
    uint32_t err, pad;      // the error word
};
#ifdef __CUDACC__
// by one warp
__device__ __forceinline__ void report_step(const StepStats* st, StepSum* out, const uint32_t* err, uint32_t* err_out) {
    const int lane = threadIdx.x & 31;
    unsigned long long c = __ldcg(&st->changed[lane]) + __ldcg(&st->changed[lane + 32]);
    unsigned long long d = __ldcg(&st->dangling_fx[lane]) + __ldcg(&st->dangling_fx[lane + 32]);
    unsigned long long l = __ldcg(&st->l1_fx[lane]) + __ldcg(&st->l1_fx[lane + 32]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
        d += __shfl_xor_sync(0xFFFFFFFFu, d, o);
        l += __shfl_xor_sync(0xFFFFFFFFu, l, o);
    }
    if (lane != 0) return;
    *out = StepSum{c, d, l, __ldcg(&st->pushed), __ldcg(&st->push_edges), __ldcg(&st->boundary_changed),
                   __ldcg(&st->skipped), __ldcg(&st->exchanged), __ldcg(&st->downloads)};
    *err_out = __ldcg(err);
}
#endif
__host__ __device__ constexpr unsigned long long list_pack(uint32_t items, uint32_t edges) {
    return ((unsigned long long)items << 32) | edges;
}

// Frontier lists: the vertices changed by a superstep, as work items of at
// most kItemEdges out-edges each ({vertex, chunk}: out-edges [32 chunk,
// 32 chunk + 32) of the vertex; a vertex without out-edges has one empty
// item). Per list: at most n_vertices + ceil(n_edges / 32) items (below
// 2^32, or the lists are not used); the out-edges of one list are at most
// n_edges < 2^32, so the packed counter's halves never carry into each other.
constexpr uint32_t kItemEdges = 32;
struct FrontierCfg {
    const uint2* list_in;        // this superstep's frontier (count: stats_in->list_ne >> 32)
    uint2* list_out;             // the next one; nullptr = no frontier lists (pull only)
    uint32_t direction;          // gxp_direction
    uint32_t push_div;
    uint64_t total_edges;
    uint64_t list_cap;           // items each list holds
    uint32_t* err;               // kErrBounds if a list would overflow (never, for valid graphs)
    // A pull superstep lists the vertices it changes (the next frontier) only
    // when the frontier it read was small enough to make a push next likely:
    // at most this many changed vertices, and items + out-edges within
    // kListSlack times the push limit. Listing costs a pull superstep an
    // out-degree load and an item write per changed vertex, which pays only
    // when the next superstep pushes. kAlwaysList: always list.
    uint64_t list_max_changed;
};
constexpr uint64_t kAlwaysList = ~0ull;
constexpr uint32_t kListSlack = 4;



// Everything the tile superstep kernel touches (superstep.cu: SSSP or CC over
// one CSC in the caller's memory).
struct SuperstepArgs {
    const Tile* tiles;
    PartDev part;
    uint32_t n_tiles;
    const uint32_t* own_cur;     // [V] current values, padded to a multiple of 4
    uint32_t* own_nxt;           // [V] next values
    uint32_t* part_head;         // [n_tiles] partials of rows split across tiles (value bits)
    uint32_t* part_tail;         // [n_tiles]
    uint32_t* hub_cnt;           // [n_tiles] arrival counters (self-resetting)
    unsigned long long* changed; // [kStatLanes] changed vertices
    uint32_t* err;               // device error word; the kernel does nothing when it is set at its start
    uint64_t timeout_ns;         // limit of any device-side wait
    uint32_t force_timeout;      // injected fault: every wait gives up at once (then drains)
    uint32_t max_items;          // largest tile (merge items)
};

// Everything the superstep kernel of a partitioned graph touches (sell.cu).
struct SellArgs {
    const SellSlice* slices;
    uint32_t n_slices;
    const HubPart* hubs;
    uint32_t n_hubs;
    const PartDev* parts;
    uint32_t n_parts;
    uint32_t n_vertices;         // V: the first cached-copy slot of the push direction
    // superstep t reads value buffer t & 1, stat slot t % kStatRing and
    // frontier list t & 1; it writes buffer / list (t + 1) & 1 and slot t + 1,
    // and clears slot t + 2
    uint32_t* own[2];
    float* rank[2];
    StepStats* stats;            // [kStatRing]
    uint2* lists[2];             // frontier lists (min-label algorithms) or nullptr
    uint64_t step;               // t
    const uint32_t* ghost;
    const uint32_t* outdeg;
    uint32_t* changed_bits;      // bitmap of the vertices this superstep changes
    uint32_t* changed_next;      // the next superstep's, cleared by this one
    const uint32_t* boundary_bits;   // vertices another partition caches
    uint32_t* hub_val;           // [n_hubs] published partials (value bits)
    uint32_t* hub_arrive;        // [n_hubs] arrival counters, indexed by a row's first part
    uint32_t* err;
    uint32_t check_bounds;
    float damping;
    float inv_n;                 // 1 / N
    uint32_t ppr_source;         // PageRank: kInf; personalized PageRank: the source vertex
    uint32_t early_exit;         // 1: a superstep (t > 0) after a quiet one returns at once
    // SSSP / CC: fc.list_out != nullptr turns the frontier lists on (the
    // kernel points list_in / list_out at lists[]); the out-edge copy is
    // what the push direction reads. Its sources are slots: the V vertices,
    // then the cached copies, slot V + g for copy g.
    FrontierCfg fc;
    const uint32_t* out_ptr;     // [slots + 1] out-edge offsets, internal ids
    const uint32_t* out_dst;     // [E] destinations (vertices), grouped by source slot
    const uint32_t* out_w;       // [E] weights, or nullptr (CC)
};

// Everything the superstep kernel of a single-partition graph touches
// (sweep.cu); buffers, lists and stat slots by superstep as in SellArgs.
struct SweepArgs {
    const SellSlice* slices;     // decreasing width
    uint32_t n_slices;
    // slices spread over 32, 16, 8, 4, 2 lanes a row end at n_lanes[0..4];
    // then those wider than 8 columns, 4 and 0
    uint32_t n_lanes[5], n_gt8, n_gt4, n_gt0;
    const HubPart* hubs;
    uint32_t n_hubs;
    const uint32_t *sell_src, *sell_w, *perm, *hsrc, *hw;   // as in PartDev
    uint32_t n_vertices;
    uint32_t n_hot;              // values staged in shared memory: vertices [0, n_hot), a multiple of 4
    uint32_t* own[2];            // [V + 1]: the identity slot is own[V]
    float* rank[2];
    StepStats* stats;
    uint2* lists[2];
    uint32_t* bits[3];           // changed vertices of a pull superstep t: bits[t % 3]
    const uint32_t* outdeg;
    unsigned long long* hub_val; // [n_hubs] published partials: value bits << 32 | 1, zero between supersteps
    uint32_t* hub_arrive;        // [n_hubs] arrival counters, indexed by a row's first part, likewise
    uint32_t* err;
    uint32_t check_bounds;
    float damping;
    float inv_n;
    uint32_t ppr_source;
    FrontierCfg fc;
    const uint32_t *out_ptr, *out_dst, *out_w;
};

// Arguments of the batched multi-source SSSP superstep kernel (one edge block).
constexpr uint32_t kUnitEdges = 256;   // in-edges of one destination per warp work unit
// packed edge (4 bytes): weight << 24 | source, when sources < 2^24 and weights < 256
constexpr uint32_t kPackSrcBits = 24;
inline bool packable(uint64_t n_vertices, uint32_t max_weight) {
    return n_vertices <= (1ull << kPackSrcBits) && max_weight < 256u;
}
// Work units (edges in .z, at most kUnitEdges) longest first, stably: dealt
// out round robin, every warp then gets about as many edges (in destination
// order the warps' shares of R-MAT 20 spread by tens of percent and a
// superstep waited for the longest).
std::vector<uint4> units_longest_first(const std::vector<uint4>& units);
struct MsArgs {
    const uint4* units;          // {dst, first edge (global), edges, split-row flag}
    uint64_t u_begin, u_end;     // this block's units
    const void* edges;           // edges[i] is global edge edge_base + i: (source, weight) uint2,
                                 // or with `packed` one uint32 (weight << 24 | source)
    uint32_t packed;
    uint64_t edge_base;
    uint32_t* dist;              // [V][64]
    const uint32_t* frontier_cur;
    uint32_t* frontier_next;
    unsigned long long* changed; // units that improved a slot (this block's counter)
    unsigned long long* active;  // nullable: running count of in-edges whose source was in the frontier
    uint32_t* slot_improved;     // nullable: [2] bit s of word 0 / s - 32 of word 1 = slot s improved
    uint64_t idle_mask;          // slots to skip (no query in them); 0 = compute all 64
    uint32_t no_sat;             // 1: n_vertices x the largest weight is below 2^32 - 1, no sum saturates
};

// f(integral_constant<int, lanes>) with the lanes of four slots each that hold
// the slots in use (the highest of `busy` decides): 16 for 64 slots down to 1
template <class F>
inline cudaError_t with_slot_lanes(uint64_t busy, F f) {
    if (busy >> 32) return f(std::integral_constant<int, 16>{});
    if (busy >> 16) return f(std::integral_constant<int, 8>{});
    if (busy >> 8) return f(std::integral_constant<int, 4>{});
    if (busy >> 4) return f(std::integral_constant<int, 2>{});
    return f(std::integral_constant<int, 1>{});
}

// Finished query slots whose columns are copied out as result vectors.
struct GatherList {
    uint32_t n;
    uint32_t slot[64];
    uint32_t* out[64];
};

// Arguments of the personalized-PageRank superstep over 64 query slots
// (serving). Matrices are [V][64] fp32, one 256-byte row per vertex.
struct PprArgs {
    const uint4* units;              // {dst, first edge, edges, partial index + 1 | 0}, longest first
    uint64_t n_units;                // covers every vertex (empty rows too)
    const uint32_t* src;             // source id of each edge, destination order
    const uint2* split_rows;         // [n_split_rows + 1] {row, first partial}; last .y = n_partials
    uint32_t n_split_rows;
    const float* inv_outdeg;         // [V] 1 / outdeg, 0 for vertices without out-edges
    const float* msg_cur;            // [V][64] r_t / outdeg
    float* msg_nxt;                  // [V][64]
    float* rank;                     // [V][64] r_{t+1}, written for slots in finish_mask
    float* partial;                  // [n_partials][64]
    const unsigned long long* dang_cur;   // [64] exact dangling mass of r_t per slot
    unsigned long long* dang_next;        // [64] (zeroed before the superstep)
    const float* slot_damping;       // [64]
    const uint32_t* slot_source;     // [64]
    uint64_t active_mask;            // slots holding a query
    uint64_t finish_mask;            // slots whose last superstep this is
};

// Mode-label propagation (lp.cu). Rows by in-degree class: up to kLpSmall in
// 32-row slices, a row per lane; up to kLpWarpRow a warp per row and up to
// kLpChunk a CTA per row, counting labels in shared-memory hash tables; up
// to kLpBig a large CTA per row, in passes over the labels' hash range; more
// (a hub): chunks of kLpChunk counted the same way and added into a global
// hash table of the hub's own, which segments of kLpSegment slots then
// reduce. Rows without in-edges keep their labels and are not listed.
constexpr uint32_t kLpSmall = 32;
constexpr uint32_t kLpWarpRow = 256;
constexpr uint32_t kLpChunk = 2048;
constexpr uint32_t kLpBig = 65536;
constexpr uint32_t kLpSegment = 4096;
struct LpPart {                 // where a row's in-edges and their labels are
    const uint32_t* src;        // row-sorted CSC sources as local ids
    const uint32_t* sell;       // slices of the small rows, column-major
    const uint32_t* perm;       // their row slots -> local vertices
    uint32_t v_begin, n_own, ghost_base, pad;
};
struct LpRow {                  // a row, or a chunk of a hub row
    uint32_t g;                 // value index (global internal id)
    uint32_t part;
    uint32_t e0;                // first in-edge (partition CSC index)
    uint32_t n;                 // in-edges
    uint32_t hub;               // hub index for a hub chunk, else kInf
    uint32_t pad[3];
};
struct LpHub {
    uint32_t g;
    uint32_t log2_size;         // table slots = 2^log2_size >= 2 in-degree
    uint64_t table;             // first slot
    uint32_t seg0;              // its first segment (segment i covers slots [i kLpSegment, ...) of the table)
    uint32_t pad;
};
struct LpSegment {              // kLpSegment slots (or fewer) of one hub's table
    uint32_t hub;
    uint32_t n;
    uint64_t slot0;
};
struct LpArgs {
    const LpPart* parts;
    uint32_t n_parts;           // 1: no cached copies (sources are indices into own_cur)
    const SellSlice* slices;    // rows of 1..kLpSmall in-edges, by partition, wide slices first
    uint32_t n_slices;
    const LpRow* warp_rows;     // kLpSmall < in-edges <= kLpWarpRow
    uint32_t n_warp_rows;
    const LpRow* chunks;        // kLpWarpRow < in-edges <= kLpChunk (hub = kInf), and hub chunks
    uint32_t n_chunks;
    const LpRow* big;           // kLpChunk < in-edges <= kLpBig
    uint32_t n_big;
    const LpHub* hubs;
    uint32_t n_hubs;
    const LpSegment* segments;  // the hub tables cut into segments
    uint32_t n_segments;
    uint32_t* keys;             // hub tables: label per slot (kInf = empty) ...
    uint32_t* counts;           // ... and its count; left empty after each superstep
    unsigned long long* hub_best;   // [n_hubs] best (count, -label) over the segments; zeroed after use
    uint32_t* seg_used;             // [n_segments] 1 once a label took a slot of the segment; cleared after use
    const uint32_t* own_cur;
    uint32_t* own_nxt;
    uint32_t n_ghost;                // all partitions' copies
    const uint32_t* ghost;
    uint32_t* changed_bits;     // bitmap of the vertices this superstep changes, or nullptr
    const StepStats* stats_in;
    StepStats* stats_out;
    StepStats* stats_clear;
    uint32_t skip_if_quiet;     // 1: return at once if the previous superstep changed nothing
    // One partition with an out-edge copy: a row none of whose in-neighbours
    // changed in the previous superstep keeps its label, so when the changed
    // vertices have few out-edges only their out-neighbours (and they
    // themselves, to bring the other buffer up to date) are recomputed.
    // nullptr: every row is recomputed.
    uint32_t* active;           // bitmap of the rows to recompute
    uint32_t* active_next;      // cleared for the next superstep
    uint32_t* changed_next;     // the next superstep's changed_bits, cleared by this one
    const uint32_t* boundary_bits;  // partitions: vertices another one caches
    const uint32_t* changed_prev;   // the previous superstep's changed vertices
    uint32_t all_rows;          // 1: recompute every row (first superstep, values set)
    uint32_t n_vertices;
    uint64_t n_edges;
    const uint32_t *out_ptr, *out_dst;
    const uint32_t* col_ptr;    // one partition: row offsets, for the edges a superstep of some rows reads
};
cudaError_t launch_lp_superstep(const LpArgs& a, cudaStream_t s);

// Arguments of the two sync kernels (changed ∩ boundary -> gdq -> caches).
struct SyncArgs {
    const PartDev* parts;
    uint32_t n_parts;
    const uint32_t* changed_bits;
    const uint32_t* boundary_bits;
    const uint32_t* own_val;          // values after the superstep, [V]
    const uint32_t* ghost_gid;        // [n_ghost] global id of each cached copy (sorted per partition)
    uint32_t n_ghost;                 // cached copies over all partitions
    uint32_t* ghost;                  // [n_ghost] caches to update
    const uint8_t* cached;            // [n_ghost] LRU flags (bit 0: cached), or nullptr = all cached
    uint32_t n_pull;
    uint32_t* gdq_ids;                // [sum of boundary counts]
    uint32_t* gdq_vals;
    const uint64_t* gdq_base;         // [n_parts] offset of each partition's gdq
    uint32_t* block_counts;           // [n_parts * blocks_x]
    uint32_t* block_offsets;          // [n_parts * blocks_x]
    uint32_t* part_counts;            // [n_parts]
    uint32_t* done_ctr;               // [n_parts] arrival counters of the count kernel
    uint32_t queue;                   // 1: write the global data queue (gxp_sync returns it)
    uint32_t max_words;               // bitmap words of the largest partition
    StepSum* report;                  // pinned host memory: the superstep's sums
    const uint32_t* err;
    uint32_t* report_err;
    uint32_t blocks_x;
    StepStats* stats_out;
    // frontier lists on (push direction possible): every cached copy whose
    // vertex changed joins the next frontier as slot n_vertices + g
    FrontierCfg fc;                   // fc.list_out = the next superstep's list, or nullptr
    const uint32_t* out_ptr;          // slot out-edge offsets
    uint32_t n_vertices;
};

// ------------------------------------------------------------ launchers
cudaError_t launch_outdeg(const PartDev& p, const uint32_t* d_src, const uint32_t* d_ghost_gid,
                          uint32_t* d_outdeg, cudaStream_t s);
// A CSC as loaded: the offsets checked (bit 0 of *err: not running from 0 to
// n_edges, non-decreasing) and narrowed to 32 bits; the sources checked (bit 1:
// >= n_local) and counted into outdeg[n_local] (zeroed by the caller)
cudaError_t launch_csc_offsets(const uint64_t* cp64, uint32_t n, uint64_t n_edges, uint32_t* cp32, uint32_t* err,
                               cudaStream_t s);
cudaError_t launch_csc_sources(const uint32_t* src, uint64_t n_edges, uint32_t n_local, uint32_t* outdeg, uint32_t* err,
                               cudaStream_t s);
// sources >= n_local set kErrBounds; offsets that do not run from 0 to n_edges
// without decreasing set kErrInput
cudaError_t launch_validate_csc(const uint32_t* d_col_ptr, uint32_t n_own, const uint32_t* d_src,
                                uint64_t n_edges, uint32_t n_local, uint32_t* d_err, cudaStream_t s);

// The initial state of a run, in one pass: values (both buffers of the
// min-label algorithms and LP; PageRank's ranks and messages), cached copies,
// identity slots, stat ring, bitmaps, and the seed of the frontier.
struct BeginArgs {
    Algo algo;
    uint32_t n, n_ghost;
    uint32_t source;             // SSSP: the source; PPR: likewise; else kInf
    float r0;                    // PageRank's 1 / N
    uint32_t* own[2];
    float* rank;
    const uint32_t* outdeg;
    const uint32_t* label_of;    // CC / LP: input ids of renumbered vertices, or nullptr
    const uint32_t* ghost_gid;
    uint32_t* ghost;
    uint32_t identity;           // of the merge
    StepStats* stats;            // [kStatRing]
    const unsigned long long* n_dangling;   // vertices without out-edges
    uint32_t* clear[5];          // bitmaps of the vertices, or nullptr
    uint32_t seed;               // vertex whose items are the first frontier, or kInf
    const uint32_t* out_ptr;
    FrontierCfg fc;              // list_out: the list the seed goes to
    unsigned long long list_ne;  // the first frontier's count, when no vertex is seeded
};
cudaError_t launch_begin(const BeginArgs& a, cudaStream_t s);
// *out = vertices without out-edges
cudaError_t launch_count_dangling(const uint32_t* outdeg, uint32_t n, unsigned long long* out, cudaStream_t s);
// report sums of supersteps first .. last (one partition), and the error word
cudaError_t launch_step_sums(const StepStats* ring, uint64_t first, uint64_t last, const uint32_t* err, StepReport* out,
                             cudaStream_t s);
cudaError_t launch_init_ghosts(Algo a, uint32_t n_ghost_total, const uint32_t* ghost_gid_all,
                               const uint32_t* own_cur, uint32_t* ghost, cudaStream_t s);

cudaError_t launch_superstep(Algo a, const SuperstepArgs& args, uint32_t sms, cudaStream_t s);
cudaError_t launch_superstep_sell(Algo a, const SellArgs& args, cudaStream_t s);

// Grid barrier state of a persistent launch (grid_barrier).
struct GridBar {
    unsigned long long count;   // arrivals since it was zeroed; top bit: a wait gave up
};
constexpr uint32_t kRunChunk = 32;   // supersteps per launch of a run (the stat ring holds 64)
// What a launch of several supersteps leaves in pinned host memory. The host
// clears `step` before the launch; a launch that gave up leaves it zero.
struct RunOut {
    uint64_t step;          // supersteps done since gxp_begin
    uint64_t arrived;       // the barrier counter
    uint32_t err, pad;      // the error word
    StepSum sum[kRunChunk]; // of the launch's supersteps
};
// Supersteps t0, t0 + 1, ... below limit, with quiet_stop until one that
// changed nothing (a lone superstep then returns at once after such a one).
struct RunArgs {
    uint64_t t0, limit;
    uint32_t quiet_stop, force;   // force: every barrier wait gives up (an injected fault)
    uint64_t timeout_ns;
    uint64_t arrived;       // the barrier counter's value
    GridBar* bar;           // nullptr: superstep t0 alone, in a launch that waits for nothing
    RunOut* out;
};
// Supersteps of a single-partition graph (sweep.cu), one CTA on each of the
// `sms` multiprocessors (fewer on small graphs), in one launch. If its CTAs don't all get onto the
// device in time, none of them does anything (run.out->step stays zero, and
// the barrier's top bit is set); a later barrier wait past timeout_ns sets
// kErrTimeout in args.err and ends the launch.
cudaError_t launch_sweep(Algo a, const SweepArgs& args, const RunArgs& run, uint32_t sms, cudaStream_t s);
// Load the kernels that a launch per superstep takes besides: the first launch
// of one not loaded yet waits for whatever runs on the device.
cudaError_t load_sweep_list();
cudaError_t load_step_sums();
// Values to stage per CTA.
uint32_t sweep_hot_values(uint64_t n_vertices, uint64_t n_edges, bool by_degree);

cudaError_t launch_sync(const SyncArgs& args, uint32_t max_words, cudaStream_t s);

// LRU-based caching under a budget (lru.cu): the superstep-boundary update of
// every partition's cached copies. Weights saturate at kLruWMax.
constexpr uint32_t kLruWMax = 65535;
constexpr uint32_t kLruBins = kLruWMax + 1;
struct LruPart {
    uint32_t cand;      // candidates (cached or used) at this boundary
    uint32_t w_star;    // the lowest weight kept
    uint32_t ties;      // candidates of weight w_star kept (lowest ids first); kInf = all candidates
    uint32_t pad;
};
struct LruArgs {
    uint32_t n_parts, n_ghost;
    const uint32_t* ghost_base;       // [n_parts + 1] first copy of each partition
    const uint32_t* ghost_gid;        // [n_ghost] vertex of each copy (ascending per partition)
    const uint32_t* reads;            // [n_ghost] the partition's in-edges from that vertex
    uint32_t* weight;                 // [n_ghost]
    uint8_t* flags;                   // [n_ghost] bit 0 cached, bit 1 candidate (transient)
    uint32_t* ghost;                  // [n_ghost] copy values (downloads write here)
    const uint32_t* own_val;          // owners' current values
    // the frontier of the coming superstep: every vertex, a bitmap, or one vertex
    uint32_t frontier_all;
    const uint32_t* frontier_bits;
    uint32_t frontier_one;
    uint32_t capacity;                // copies kept per partition
    uint32_t* hist;                   // [n_parts][kLruBins], zero between boundaries
    LruPart* part_state;              // [n_parts], cand zero between boundaries
    uint32_t* tie;                    // [n_ghost]
    uint32_t* tie_scan;               // [n_ghost + 1]
    uint32_t* scan_scratch;           // (n_ghost + 2047) / 2048 + 1 words
    StepStats* stats_out;             // `downloads` of the coming superstep
    const StepStats* quiet_check;     // non-null: no-op when that superstep changed nothing
};
cudaError_t launch_lru_boundary(const LruArgs& a, uint32_t max_ghosts_per_part, cudaStream_t s);

// push direction (frontier.cu)
struct RowSource;
// out-edge copy of the CSC `in` (rows renumbered as the layout build does):
// out_ptr = exclusive scan of outdeg (internal ids); scratch holds
// out_edges_scratch_words(n, n_edges) words
// (rows: n, sources: n_src >= n; out_ptr[n_src + 1])
cudaError_t launch_out_edges(const RowSource& in, uint32_t n, uint32_t n_src, uint64_t n_edges,
                             const uint32_t* outdeg, uint32_t* out_ptr, uint32_t* scratch, uint32_t* out_dst,
                             uint32_t* out_w, cudaStream_t s);
size_t out_edges_scratch_words(uint32_t n_src, uint64_t n_edges);
// several partitions: the CSC over global rows whose sources are slots
// (own vertex u -> v_begin + u, cached copy u -> V + ghost_base + u - n_own)
// and the out-degree of every slot (counted into outdeg, zeroed first)
cudaError_t launch_unify_csc(const PartDev& p, uint32_t n_vertices, uint64_t edge_base, uint32_t* ucol,
                             uint32_t* usrc, bool last, cudaStream_t s);
cudaError_t launch_slot_degrees(const uint32_t* usrc, uint64_t n_edges, uint32_t n_slots, uint32_t* outdeg,
                                cudaStream_t s);
// every slot whose value is below INF joins the list (partitioned starts)
cudaError_t launch_seed_finite(uint32_t n_vertices, uint32_t n_ghost, const uint32_t* own, const uint32_t* ghost,
                               const uint32_t* out_ptr, const FrontierCfg& f, StepStats* stats, cudaStream_t s);
// f.list_out <- items of vertex `source` (all vertices when source == kInf);
// the counts go to stats->list_ne (zeroed here first)
cudaError_t launch_seed_frontier(uint32_t n, uint32_t source, const uint32_t* out_ptr, const FrontierCfg& f,
                                 StepStats* stats, cudaStream_t s);
// exclusive scan of n u32 counts into out[0..n] (out[n] = total); scratch:
// (n + 2047) / 2048 + 1 words (sell_build.cu)
cudaError_t launch_exclusive_scan_u32(const uint32_t* x, uint32_t n, uint32_t* out, uint32_t* scratch,
                                      cudaStream_t s);

cudaError_t launch_msssp(const MsArgs& a, bool dry, uint32_t grid, cudaStream_t s);
// Persistent resident run (k_msssp_loop): supersteps over the units of `a`
// until one improves nothing or max_steps, one cooperative launch; frontier
// rotates over three bitmaps of `words` words (frontier[0] holds the sources,
// frontier[1] must be zero), changed over four counters (the first two zero);
// *steps_out gets the supersteps run. A grid-barrier wait past timeout_ns (or any, with `force`)
// sets kErrTimeout in *err and ends the launch.
cudaError_t launch_msssp_loop(const MsArgs& a, uint32_t* const frontier[3], unsigned long long* changed,
                              uint64_t words, uint32_t max_steps, GridBar* bar, uint64_t timeout_ns, bool force,
                              uint32_t* err, uint32_t* steps_out, cudaStream_t s);
cudaError_t launch_msssp_init(uint32_t* dist, uint64_t n_vertices, const uint32_t* sources, uint32_t n_sources,
                              uint32_t* frontier, cudaStream_t s);
cudaError_t launch_popc(const uint32_t* bits, uint64_t words, unsigned long long* out, cudaStream_t s);
uint32_t msssp_grid(uint64_t units);

// sliced-ELL build on the device (sell_build.cu)
// The CSC a build reads: row v of the result is input row row_map[v] (or v),
// with its sources renumbered through src_map (or kept).
struct RowSource {
    const uint32_t* col_ptr;
    const uint32_t* src;
    const uint32_t* w;          // nullptr: unweighted
    const uint32_t* row_map;    // nullptr: identity
    const uint32_t* src_map;    // nullptr: identity
};
// rows of col_ptr (the result's offsets) sorted by source into ssrc / sw
// (rows of up to 256 edges by (source, weight), longer ones stably by
// source); sources are below n_src
cudaError_t launch_sort_rows(const uint32_t* col_ptr, uint32_t n, const RowSource& in, uint32_t n_src,
                             uint32_t* ssrc, uint32_t* sw, uint2* scratch_runs, uint32_t* scratch_cnt,
                             cudaStream_t s);   // scratch_runs: n + n_edges / 2048 + 1 entries
// rows of col_ptr (in.row_map and in.src_map set, rows without in-edges last) as
// loaded, sources renumbered
cudaError_t launch_renumber_rows(const uint32_t* col_ptr, uint32_t n, const RowSource& in, uint64_t n_edges,
                                 uint32_t* ssrc, uint32_t* sw, cudaStream_t s);
cudaError_t launch_sell_windows(const uint32_t* col_ptr, uint32_t n, uint32_t H, uint32_t* rows_out,
                                uint32_t* hub_out, uint32_t* nonhub_cnt, uint32_t* hub_cnt, cudaStream_t s);
cudaError_t launch_sell_slices(const uint32_t* col_ptr, uint32_t n, const uint32_t* rows_out,
                               const uint32_t* nonhub_cnt, const uint32_t* slice_base, uint32_t* perm,
                               uint32_t* width, uint64_t* off, uint32_t n_slices, uint32_t cols, cudaStream_t s);
cudaError_t launch_sell_fill(const uint32_t* col_ptr, const uint32_t* ssrc, const uint32_t* sw, const uint32_t* perm,
                             const uint32_t* width, const uint64_t* off, uint32_t n_slices, uint32_t part,
                             uint32_t pad_id, uint32_t cols, uint32_t* sell_src, uint32_t* sell_w, SellSlice* desc,
                             cudaStream_t s);
// a renumbered partition's slices: rows first_row .. n_rows - 1, in order of
// decreasing in-degree (at[w] + s * sell_words(w) is slice s's start if it is w wide)
cudaError_t launch_sell_fill_sorted(const uint32_t* col_ptr, const uint32_t* ssrc, const uint32_t* sw, uint32_t n_rows,
                                    uint32_t first_row, const uint64_t* at, uint32_t n_slices, uint32_t cols,
                                    uint32_t* sell_src, uint32_t* sell_w, SellSlice* desc, cudaStream_t s);
// Hub rows are cut into parts of T edges, a row of more than max_parts of them
// into longer ones. One partition cuts a row into at most kMaxRowParts, about a
// part for each of its kernel's 4,864 warps: the row's last part combines
// them all, a warp's 128 loads a lane. Rows of up to 2 M in-edges (T = 512; 8 M
// at T = 2048) are below it.
constexpr uint32_t kMaxRowParts = 4096;
// exclusive prefix of the parts of hub rows 0 .. n_hub_rows - 1, and their total
cudaError_t launch_hub_offsets(const uint32_t* col_ptr, uint32_t n_hub_rows, uint32_t T, uint32_t max_parts,
                               uint32_t* part_off, cudaStream_t s);
cudaError_t launch_hub_rows(const uint32_t* col_ptr, uint32_t n, const uint32_t* hub_out, const uint32_t* hub_cnt,
                            const uint32_t* hub_base, uint32_t* hub_list, uint32_t n_hub_rows, uint32_t T,
                            uint32_t max_parts, uint32_t* part_off, cudaStream_t s);
cudaError_t launch_hub_parts(const uint32_t* col_ptr, const uint32_t* hub_list, const uint32_t* part_off,
                             uint32_t n_hub_rows, uint32_t T, uint32_t max_parts, uint32_t part, uint32_t part_base,
                             HubPart* hubs, cudaStream_t s);   // hub_list nullptr: rows 0 .. n_hub_rows - 1
// slices by decreasing width (stable); afterwards word b of
// order_slices_starts(scratch, n) holds the number of slices wider than b
// (b <= kOrderExact)
constexpr uint32_t kOrderExact = 1024;
cudaError_t launch_order_slices(const SellSlice* in, uint32_t n, SellSlice* out, uint32_t* scratch, cudaStream_t s);
size_t order_slices_scratch_bytes(uint32_t n);
const uint32_t* order_slices_starts(const uint32_t* scratch, uint32_t n);

// vertex relabelling by decreasing in-degree (sell_build.cu): new2old / old2new
// and the renumbered offsets rcol[n + 1]; scratch: relabel_scratch_bytes.
// *starts (in scratch): word b is the number of vertices of in-degree above b
// (b <= kOrderExact)
size_t relabel_scratch_bytes(uint32_t n);
cudaError_t launch_relabel(const uint32_t* col_ptr, uint32_t n, uint32_t* new2old, uint32_t* old2new, uint32_t* rcol,
                           uint32_t* scratch, const uint32_t** starts, cudaStream_t s);
// out[v] = in[map[v]] (gather) or out[map[v]] = in[v] (scatter)
cudaError_t launch_permute_u32(const uint32_t* in, const uint32_t* map, uint32_t n, uint32_t* out, bool scatter,
                               cudaStream_t s);

// serving (serve.cu): 64-slot personalized PageRank and slot management
cudaError_t launch_ppr_superstep(const PprArgs& a, cudaStream_t s);
uint32_t serve_grid(uint64_t warp_items);   // short-lived blocks for lanes sharing the GPU
// slots in `mask` start a new query: PPR columns get the messages of
// r_0 = e_src and its exact dangling mass; slot_source holds the sources
cudaError_t launch_ppr_slots_init(float* msg_cur, const float* inv_outdeg, uint64_t n_vertices, uint64_t mask,
                                  const uint32_t* slot_source, unsigned long long* dang_cur, cudaStream_t s);
// SSSP columns in `mask` get d = INF except d[src] = 0; sources join the frontier
cudaError_t launch_sssp_slots_init(uint32_t* dist, uint64_t n_vertices, uint64_t mask, const uint32_t* slot_source,
                                   uint32_t* frontier, cudaStream_t s);
// column slot[j] of mat[V][64] -> out[j][0..V) for j < n (row-tile transpose)
cudaError_t launch_gather_columns(const uint32_t* mat, uint64_t n_vertices, const GatherList& list, cudaStream_t s);

// Fixed point -> double (exact for sums below 2^53 units, else rounded once).
__host__ __device__ inline double fx_to_double(unsigned long long v) {
    return (double)v * (1.0 / (double)(1ULL << kFxShift));
}

// Fixed point (2^-60) -> fp32, from its two 32-bit halves (no FP64).
__host__ __device__ inline float fx_to_float(unsigned long long v) {
    const float hi = (float)(uint32_t)(v >> 32), lo = (float)(uint32_t)v;
    return fmaf(hi, 0x1p-28f, lo * 0x1p-60f);
}

// The base terms of a PageRank superstep from the exact dangling mass D of
// its input ranks (fixed point), for damping d and 1 / N: PageRank spreads
// (1-d) + d*D evenly, (1-d)/N + d*D/N to every vertex; personalized PageRank
// returns all of it to the source vertex (base_pr = 0 elsewhere).
// In fp32 only (the FP64 pipe of this GPU is narrow and every warp of the
// superstep forms these terms).
__host__ __device__ inline void pagerank_base(unsigned long long dangling_fx, float d, float inv_n, bool personalized,
                                              float* base_pr, float* base_src) {
    const float mass = fx_to_float(dangling_fx);   // D
    const float spread = fmaf(d, mass, 1.0f - d);
    if (!personalized) {
        *base_pr = *base_src = spread * inv_n;
    } else {
        *base_pr = 0.0f;
        *base_src = spread;
    }
}

#ifdef __CUDACC__
// x >= 0 (fp32) -> x * 2^60 truncated to an integer, exactly, with integer
// operations only; values below 2^-126 count as 0. For x <= 2 the result is
// below 2^62, so sums of up to 2 units of mass cannot overflow.
__device__ __forceinline__ unsigned long long fx_of(float x) {
    const uint32_t b = __float_as_uint(x);
    const int e = (int)((b >> 23) & 0xFFu);
    if (e == 0) return 0ull;
    const unsigned long long m = (unsigned long long)((b & 0x7FFFFFu) | 0x800000u);
    const int sh = e - 150 + kFxShift;
    if (sh >= 0) return m << sh;
    return (-sh) >= 64 ? 0ull : (m >> (-sh));
}
#endif

}  // namespace gxp
