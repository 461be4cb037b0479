// Supersteps of a single-partition graph (SSSP, CC, PageRank, personalized
// PageRank): MSGGen + MSGMerge + MSGApply over the sliced-ELL layout in one
// persistent CTA per SM (fewer for small graphs), one superstep or many per
// launch.
//
// What bounds it: the gathers of the sources' values. On a power-law graph a
// warp's 32 gathers touch ~30 different sectors, so large graphs run at the
// rate of the L1-to-L2 request path (42 M sectors a superstep of R-MAT 22,
// that path 62% busy, 8.4 TB/s from L2) and small ones at the latency of
// chains of dependent loads (descriptor, sources, values, old value). Hence:
//  * one persistent CTA per SM runs all supersteps of a run: a grid barrier
//    (2.7 us) in place of a launch, and no prologue and epilogue per 8 work
//    items;
//  * work items of one size: a row of up to 512 in-edges is spread over as
//    many lanes (1 .. 32) as bring it down to 16 columns (sweep_lanes), so
//    an item is at most two batches of gathers (four for SSSP), and items are
//    dealt out evenly with neither a queue nor a long item to wait for. With whole
//    rows per lane, up to 1,024 columns, the longest slice alone took as long
//    as the superstep should;
//  * a warp's loads run ahead: the next item's descriptor, then its sources,
//    old value and out-degree, are on their way while an item's values are;
//  * the values of the first n_hot vertices are staged in shared memory at
//    the start of a pull superstep. Vertices are renumbered by decreasing
//    in-degree, so those are the hot ones (32,768 of them carry 54% of the
//    gathers of R-MAT 22, 70% of R-MAT 20), and a shared-memory gather costs
//    its bank conflicts where an L1 hit costs a tag look-up per line. Not
//    more of them: the rest of the 256 KB is L1, which holds the misses in
//    flight (R-MAT 22, us a superstep, for 0 / 16,384 / 32,768 / 53,248
//    staged values: 212 / 202 / 191 / 306, measured before the lane groups);
//  * narrow slices (at most 4 or 8 columns) are taken several per item.
// Per superstep, launch gaps included, before (a launch per superstep, one
// warp per slice, 8 warps a CTA) and after: PageRank R-MAT 22 187 -> 153 us,
// 1 M vertices and 16.8 M edges 73 -> 42 us, 200 K vertices and 3.2 M edges
// 31 -> 17 us; a whole SSSP run of R-MAT 22 1,635 -> 1,119 us.
//
// Work items, in order: for PageRank groups of slices of rows without
// in-edges (the min-label algorithms leave such rows alone: both value
// buffers hold their values from the start), parts of hub rows, sub-slices,
// groups of narrow slices.
//
// A pull superstep of SSSP / CC marks its changed vertices in a bitmap and
// counts their out-edges; only when the next superstep pushes is the bitmap
// turned into the list of work items the push reads (listing every dense
// superstep's vertices costs an item write per changed vertex for a list
// that is hardly ever read).
//
// Sums run in the layout's fixed order, so fp32 PageRank is deterministic;
// its global sums (dangling mass, L1 delta) are exact 64-bit fixed point.
#include "frontier.cuh"
#include "grid_sync.cuh"
#include "merge_ops.cuh"

#include <algorithm>

namespace gxp {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kThreads = 1024;   // one CTA per SM: 64 registers a thread
constexpr int kWarps = kThreads / 32;
constexpr int kZeroGroup = 4;      // slices of rows without in-edges per item
// How long the first CTAs of a run wait for the others. Not a cooperative
// launch, which the device holds back until every SM is free at once: beside a
// kernel of 0.3 s on one SM a PageRank run of 0.41 ms took 279 ms. So it takes
// 0.79 ms (0.94 / 1.74 ms with a limit of 200 / 1,000 us, 0.74 ms if every run
// were a launch per superstep); beside a busy query server 0.43 .. 0.56 ms
// with each of the limits. Alone, all of 3,000 runs met; meeting costs 1.6 us.
constexpr uint64_t kGatherNs = 50000;
constexpr uint32_t kMaxHot = 32768;     // staged values: 128 KB, the rest of an SM's 256 KB is L1

// Columns (gathers) in flight per lane. Of 64 registers a thread these spill
// 80 bytes (PageRank), 112 (CC) and 36 (SSSP); more of them spill more and run
// slower: PageRank on R-MAT 22 at 16, 12 and 8 took 207, 179 and 163 us a
// superstep, SSSP at 8 and 4 together 1,002 and 933 us a run.
template <Algo A> constexpr int kCols = A == Algo::SSSP ? 4 : 8;

// Value of source u: from the staged copy below n_hot, else from memory.
// Two predicated loads and no branch, so that a batch's gathers stay in
// flight together.
__device__ __forceinline__ uint32_t gather(uint32_t hot, uint32_t n_hot, const uint32_t* own, uint32_t u) {
    uint32_t x;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.lt.u32 p, %1, %2;\n\t"
        "@p ld.shared.u32 %0, [%3];\n\t"
        "@!p ld.global.ca.u32 %0, [%4];\n\t}"
        : "=r"(x)
        : "r"(u), "r"(n_hot), "r"(hot + 4u * u), "l"(own + u));
    return x;
}

// 16 bytes global -> shared, asynchronously and past L1 (the values are
// written by other SMs between supersteps), and the wait for all of a
// thread's copies.
__device__ __forceinline__ void stage16(uint32_t dst, const uint32_t* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

struct WarpAcc {     // what a lane adds up over a superstep
    uint32_t changed = 0, items = 0, edges = 0;
    unsigned long long l1 = 0ull, dang = 0ull;
};

constexpr uint32_t kSliceWords = sizeof(SellSlice) / 4, kHubWords = sizeof(HubPart) / 4;
static_assert(kSliceWords == 6 && kHubWords == 8 && 4 * kSliceWords <= 32, "descriptor words are spread over a warp");

// n descriptors of W words each from p on, word j in lane j (0 past the end)
__device__ __forceinline__ uint32_t load_words(const void* p, uint32_t n, int lane) {
    return (uint32_t)lane < n ? __ldg(static_cast<const uint32_t*>(p) + lane) : 0u;
}

// State of one superstep, uniform over the grid.
struct Step {
    const uint32_t* own_cur;
    uint32_t* own_nxt;
    const float* rank_cur;
    float* rank_nxt;
    uint32_t* bits;          // changed vertices (pull supersteps with frontier lists)
    uint32_t hot;            // shared-memory address of the staged values
    float base, base_src;    // PageRank base terms
};

// Partials of a hub row a lane asks for at once. One after the other they took
// two thirds of a superstep of one row of 16.8 M in-edges (20 of PageRank 7.3
// ms with 32,768 parts; 3.9 ms with 4 at once; 1.7 ms with at most kMaxRowParts
// parts besides). 4 and more spill registers elsewhere: SSSP of R-MAT 16 takes
// 187.1 us at 3 and 189.8 us at 4.
constexpr uint32_t kPolls = 3;

template <Algo A, bool kCheck>
struct Pull {
    using Op = Ops<A>;
    using T = typename Op::T;
    static constexpr int kU = kCols<A>;
    const SweepArgs& a;
    const Step& s;
    WarpAcc& acc;
    const int lane;

    // kCheck: an id outside the graph (and not the padding id) is reported
    // and replaced by the padding id
    __device__ __forceinline__ uint32_t value(uint32_t u) const {
        if constexpr (kCheck) {
            if (u > a.n_vertices) {
                atomicOr(a.err, kErrBounds);
                u = a.n_vertices;
            }
        }
        return gather(s.hot, a.n_hot, s.own_cur, u);
    }

    // MSGApply of vertex v with merged message m and its operands loaded
    // before: PageRank the old rank and the out-degree, else the old value
    __device__ __forceinline__ bool apply(uint32_t v, T m, uint32_t op0, uint32_t op1) {
        if constexpr (A == Algo::PR) {
            const float rn = fmaf(a.damping, m, v == a.ppr_source ? s.base_src : s.base);
            s.rank_nxt[v] = rn;
            s.own_nxt[v] = __float_as_uint(op1 ? __fdiv_rn(rn, (float)op1) : 0.0f);
            const unsigned long long fn = fx_of(rn), fo = fx_of(__uint_as_float(op0));
            acc.l1 += fn > fo ? fn - fo : fo - fn;
            if (op1 == 0u) acc.dang += fn;
            return false;
        } else {
            const uint32_t nw = min(op0, (uint32_t)m);
            s.own_nxt[v] = nw;
            return nw != op0;
        }
    }
    __device__ __forceinline__ uint32_t operand0(uint32_t v) const {
        if constexpr (A == Algo::PR) return __float_as_uint(__ldca(s.rank_cur + v));
        else return value(v);
    }
    __device__ __forceinline__ uint32_t operand1(uint32_t v) const {
        if constexpr (A == Algo::PR) return __ldg(a.outdeg + v);
        else return 0u;
    }

    // this lane's vertex v changed (has) or not: counts and changed bits
    __device__ __forceinline__ void changed(bool has, uint32_t v) {
        if constexpr (A != Algo::PR) {
            const unsigned chm = __ballot_sync(kFull, has);
            if (!chm || !has) return;
            ++acc.changed;
            if (a.fc.list_out == nullptr) return;
            const uint32_t deg = __ldg(a.out_ptr + v + 1) - __ldg(a.out_ptr + v);
            acc.items += frontier_items(deg);
            acc.edges += deg;
            // one atomic per bitmap word the warp touches
            const unsigned grp = __match_any_sync(chm, v >> 5);
            const unsigned b = __reduce_or_sync(grp, 1u << (v & 31u));
            if (lane == __ffs(grp) - 1) atomicOr(s.bits + (v >> 5), b);
        }
    }

    // vertex of row slot r of the slice whose descriptor starts at lane at of words
    __device__ __forceinline__ uint32_t row_of(uint32_t words, int at, uint32_t r) const {
        const uint32_t n = __shfl_sync(kFull, words, at), first = __shfl_sync(kFull, words, at + 3);
        if (n) return r < n ? first + r : kSellPad;   // consecutive vertices
        return __ldg(a.perm + __shfl_sync(kFull, words, at + 1) + r);
    }

    // A sub-slice: 32 / L rows of L lanes each (lg = log2 L).
    struct Sub {
        uint64_t at;     // the lane's first 128-bit group
        uint32_t cols;   // stored columns
        uint32_t row;    // the row this lane applies, or kSellPad
        uint32_t op0, op1;
    };
    __device__ __forceinline__ Sub sub_of(uint32_t words, uint32_t lg, uint32_t sub) const {
        const uint32_t width = __shfl_sync(kFull, words, 2);
        const uint64_t off = __shfl_sync(kFull, words, 4) | ((uint64_t)__shfl_sync(kFull, words, 5) << 32);
        Sub r;
        r.cols = (((width + (1u << lg) - 1u) >> lg) + 3u) & ~3u;   // sweep_cols
        r.at = (off >> 2) + 8ull * r.cols * sub + lane;
        r.row = row_of(words, 0, sub * (32u >> lg) + ((uint32_t)lane >> lg));
        if ((uint32_t)lane & ((1u << lg) - 1u)) r.row = kSellPad;   // the first lane of a row's group applies it
        r.op0 = r.row != kSellPad ? operand0(r.row) : 0u;
        r.op1 = r.row != kSellPad ? operand1(r.row) : 0u;
        return r;
    }

    // Item i of the sub-slices, all kinds of lane groups in one order (32
    // lanes a row first): its slice, its number in the slice, log2 of its lanes.
    struct Where {
        uint32_t slice, sub, lg;
    };
    __device__ __forceinline__ uint32_t subs_end(int c) const {   // slices of the kinds 0 .. c
        return c < 5 ? a.n_lanes[c] : kU >= 8 ? a.n_gt8 : a.n_gt4;
    }
    __device__ __forceinline__ Where where(uint32_t i) const {
        uint32_t s0 = 0, lg = 5;
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            const uint32_t end = subs_end(c), n = (end - s0) << (5 - c);
            if (lg == 5u - c && i >= n) {   // past this kind
                i -= n;
                s0 = end;
                lg = 4u - c;
            }
        }
        return Where{s0 + (i >> lg), i & ((1u << lg) - 1u), lg};
    }
    __device__ __forceinline__ uint32_t n_subs() const {
        uint32_t s0 = 0, n = 0;
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            n += (subs_end(c) - s0) << (5 - c);
            s0 = subs_end(c);
        }
        return n;
    }

    // Sub-slices first, first + step, ... below n. The next batch's sources
    // (of this item or the next) are on their way while a batch's values are.
    __device__ __forceinline__ void subs(uint32_t n, uint32_t first, uint32_t step) {
        if (first >= n) return;
        constexpr int kG = kU / 4;
        uint4 u4[kG], w4[kG];
        auto load = [&](const Sub& r, uint32_t k0) {
#pragma unroll
            for (int h = 0; h < kG; ++h) {
                const bool in = k0 + 4u * h < r.cols;
                const uint64_t at = r.at + 8u * (k0 + 4u * h);
                u4[h] = in ? ld_stream4(reinterpret_cast<const uint4*>(a.sell_src) + at)
                           : make_uint4(a.n_vertices, a.n_vertices, a.n_vertices, a.n_vertices);
                if constexpr (Op::kWeighted)
                    w4[h] = in ? ld_stream4(reinterpret_cast<const uint4*>(a.sell_w) + at) : make_uint4(0u, 0u, 0u, 0u);
            }
        };
        Where at = where(first);
        uint32_t lg = at.lg;
        Sub cur = sub_of(load_words(a.slices + at.slice, kSliceWords, lane), lg, at.sub);
        load(cur, 0u);
        uint64_t inext = (uint64_t)first + step;
        uint32_t words = 0u;
        auto fetch = [&]() {   // the descriptor of item inext
            if (inext >= n) return;
            at = where((uint32_t)inext);
            words = load_words(a.slices + at.slice, kSliceWords, lane);
        };
        fetch();
        T m = Op::ident();
        uint32_t k0 = 0;
        for (;;) {
            uint32_t x[kU], w[kU];
#pragma unroll
            for (int h = 0; h < kG; ++h) {
                x[4 * h] = value(u4[h].x);
                x[4 * h + 1] = value(u4[h].y);
                x[4 * h + 2] = value(u4[h].z);
                x[4 * h + 3] = value(u4[h].w);
                w[4 * h] = w[4 * h + 1] = w[4 * h + 2] = w[4 * h + 3] = 0u;
                if constexpr (Op::kWeighted) {
                    w[4 * h] = w4[h].x;
                    w[4 * h + 1] = w4[h].y;
                    w[4 * h + 2] = w4[h].z;
                    w[4 * h + 3] = w4[h].w;
                }
            }
            k0 += kU;
            const bool last = k0 >= cur.cols, more = inext < n;
            const uint32_t row = cur.row, op0 = cur.op0, op1 = cur.op1, L = 1u << lg;
            if (!last) {
                load(cur, k0);
            } else if (more) {
                lg = at.lg;
                cur = sub_of(words, lg, at.sub);
                load(cur, 0u);
                k0 = 0;
                inext += step;
                fetch();
            }
#pragma unroll
            for (int q = 0; q < kU; ++q) m = Op::combine(m, Op::gen(x[q], w[q]));
            if (!last) continue;
            for (uint32_t o = L >> 1; o > 0; o >>= 1) m = Op::combine(m, __shfl_xor_sync(kFull, m, o));
            const bool ch = row != kSellPad && apply(row, m, op0, op1);
            changed(ch, row);
            m = Op::ident();
            if (!more) return;
        }
    }

    // kN narrow slices (n of them at the end of their range), all of whose
    // columns (at most kU / kN) are one batch
    template <int kN>
    __device__ __forceinline__ void narrow(uint32_t words, uint32_t n) {
        constexpr int kG = kU / 4 / kN;   // groups of 4 columns per slice
        uint32_t row[kN], op0[kN], op1[kN];
        uint4 u4[kN * kG], w4[kN * kG];
#pragma unroll
        for (int j = 0; j < kN; ++j) {
            const uint32_t width = __shfl_sync(kFull, words, kSliceWords * j + 2);   // 0 past n: no descriptor words
            const uint64_t off = __shfl_sync(kFull, words, kSliceWords * j + 4) |
                                 ((uint64_t)__shfl_sync(kFull, words, kSliceWords * j + 5) << 32);
            row[j] = (uint32_t)j < n ? row_of(words, kSliceWords * j, lane) : kSellPad;
#pragma unroll
            for (int h = 0; h < kG; ++h) {
                const bool in = 4u * h < width;
                const uint64_t at = (off >> 2) + 32u * h + lane;
                u4[j * kG + h] = in ? ld_stream4(reinterpret_cast<const uint4*>(a.sell_src) + at)
                                    : make_uint4(a.n_vertices, a.n_vertices, a.n_vertices, a.n_vertices);
                if constexpr (Op::kWeighted)
                    w4[j * kG + h] = in ? ld_stream4(reinterpret_cast<const uint4*>(a.sell_w) + at)
                                        : make_uint4(0u, 0u, 0u, 0u);
            }
        }
#pragma unroll
        for (int j = 0; j < kN; ++j) {
            op0[j] = row[j] != kSellPad ? operand0(row[j]) : 0u;
            op1[j] = row[j] != kSellPad ? operand1(row[j]) : 0u;
        }
        T m[kN];
        uint32_t x[kN * kG * 4];
#pragma unroll
        for (int g = 0; g < kN * kG; ++g) {
            x[4 * g] = value(u4[g].x);
            x[4 * g + 1] = value(u4[g].y);
            x[4 * g + 2] = value(u4[g].z);
            x[4 * g + 3] = value(u4[g].w);
        }
#pragma unroll
        for (int j = 0; j < kN; ++j) {
            m[j] = Op::ident();
#pragma unroll
            for (int h = 0; h < kG; ++h) {
                const int g = j * kG + h;
                const uint4 w = Op::kWeighted ? w4[g] : make_uint4(0u, 0u, 0u, 0u);
                m[j] = Op::combine(m[j], Op::gen(x[4 * g], w.x));
                m[j] = Op::combine(m[j], Op::gen(x[4 * g + 1], w.y));
                m[j] = Op::combine(m[j], Op::gen(x[4 * g + 2], w.z));
                m[j] = Op::combine(m[j], Op::gen(x[4 * g + 3], w.w));
            }
            const bool ch = row[j] != kSellPad && apply(row[j], m[j], op0[j], op1[j]);
            changed(ch, row[j]);
        }
    }

    // Groups of kN slices [s0, s1): group i holds slices s0 + kN i ..; f(words, slices in the group)
    template <int kN, class F>
    __device__ __forceinline__ void groups(uint32_t s0, uint32_t s1, uint32_t first, uint32_t step, F f) {
        const uint32_t n = (s1 - s0 + kN - 1) / kN;
        auto words_of = [&](uint64_t i) {
            const uint32_t s = s0 + kN * (uint32_t)i;
            return i < n ? load_words(a.slices + s, kSliceWords * min((uint32_t)kN, s1 - s), lane) : 0u;
        };
        uint32_t words = words_of(first);
        for (uint64_t i = first; i < n; i += step) {
            const uint32_t next = words_of(i + step);
            f(words, min((uint32_t)kN, s1 - s0 - kN * (uint32_t)i));
            words = next;
        }
    }

    __device__ __forceinline__ void zero_rows(uint32_t words, uint32_t n) {
        uint32_t v[kZeroGroup], op0[kZeroGroup], op1[kZeroGroup];
#pragma unroll
        for (int j = 0; j < kZeroGroup; ++j)
            v[j] = (uint32_t)j < n ? row_of(words, kSliceWords * j, lane) : kSellPad;
#pragma unroll
        for (int j = 0; j < kZeroGroup; ++j) {
            op0[j] = v[j] != kSellPad ? operand0(v[j]) : 0u;
            op1[j] = v[j] != kSellPad ? operand1(v[j]) : 0u;
        }
#pragma unroll
        for (int j = 0; j < kZeroGroup; ++j)
            if (v[j] != kSellPad) apply(v[j], Op::ident(), op0[j], op1[j]);
    }

    // Hub parts first, first + step, ... below n, lane-strided. The part of a
    // row that arrives last combines all of the row's parts, in part order.
    // A partial is published as one word with its flag, by a relaxed atomic
    // store that relaxed atomic loads poll, so neither it nor the arrival needs
    // a fence; the arrival's answer is looked at one part later,
    // when it has come back, and the last arriver polls the row's words,
    // all of them stored by then, until it sees them.
    struct Row {
        uint32_t v, t0, nparts, arrived;
    };
    __device__ __forceinline__ void hub_parts(uint32_t n, uint32_t first, uint32_t step) {
        if (first >= n) return;
        uint32_t u[kU], w[kU];
        auto load = [&](uint32_t e0, uint32_t ne, uint32_t j0) {
#pragma unroll
            for (int q = 0; q < kU; ++q) {
                const uint32_t j = j0 + (uint32_t)q * 32u + (uint32_t)lane;
                u[q] = j < ne ? ld_stream(a.hsrc + e0 + j) : a.n_vertices;
                if constexpr (Op::kWeighted) w[q] = j < ne ? ld_stream(a.hw + e0 + j) : 0u;
                else w[q] = 0u;
            }
        };
        auto words_of = [&](uint64_t i) { return i < n ? load_words(a.hubs + i, kHubWords, lane) : 0u; };
        uint32_t words = words_of(first);
        uint32_t e0 = __shfl_sync(kFull, words, 2), ne = __shfl_sync(kFull, words, 3);
        load(e0, ne, 0u);
        Row pend{0u, 0u, 0u, 0u};
        for (uint64_t i = first; i < n; i += step) {
            const uint32_t next = words_of(i + step);
            const Row row{__shfl_sync(kFull, words, 0), __shfl_sync(kFull, words, 4), __shfl_sync(kFull, words, 5), 0u};
            T m = Op::ident();
            for (uint32_t j0 = 0;;) {
                uint32_t x[kU], wc[kU];
#pragma unroll
                for (int q = 0; q < kU; ++q) {
                    x[q] = value(u[q]);
                    wc[q] = w[q];
                }
                j0 += 32u * kU;
                const bool more = j0 < ne;
                if (more) {
                    load(e0, ne, j0);
                } else if (i + step < n) {
                    e0 = __shfl_sync(kFull, next, 2);
                    ne = __shfl_sync(kFull, next, 3);
                    load(e0, ne, 0u);
                }
#pragma unroll
                for (int q = 0; q < kU; ++q) m = Op::combine(m, Op::gen(x[q], wc[q]));
                if (!more) break;
            }
            const T total = warp_all<Op>(m);
            combine_if_last(pend);
            pend = row;
            if (row.nparts == 1u) {
                finish(row.v, total);
                pend.nparts = 0u;
            } else if (lane == 0) {
                st_relaxed_gpu(&a.hub_val[i], ((unsigned long long)Op::to_bits(total) << 32) | 1ull);
                pend.arrived = atomicAdd(&a.hub_arrive[row.t0], 1u);
            }
            words = next;
        }
        combine_if_last(pend);
    }
    __device__ __forceinline__ void finish(uint32_t v, T total) {
        const bool ch = lane == 0 && apply(v, total, operand0(v), operand1(v));
        changed(ch, v);
    }
    __device__ __forceinline__ void combine_if_last(const Row& r) {
        if (r.nparts == 0u || __shfl_sync(kFull, r.arrived, 0) != r.nparts - 1u) return;
        T tot = Op::ident();   // parts in a fixed order: lane-strided, then a fixed tree
        for (uint32_t q0 = (uint32_t)lane; q0 < r.nparts; q0 += 32u * kPolls) {
            unsigned long long x[kPolls];
#pragma unroll
            for (uint32_t j = 0; j < kPolls; ++j)
                x[j] = q0 + 32u * j < r.nparts ? ld_relaxed_gpu(&a.hub_val[r.t0 + q0 + 32u * j]) : 1ull;
#pragma unroll
            for (uint32_t j = 0; j < kPolls; ++j) {
                const uint32_t q = q0 + 32u * j;
                if (q >= r.nparts) break;
                for (uint32_t spin = 0; !(x[j] & 1ull); ++spin) {   // stored already: its way to L2
                    if (spin == 1u << 22) {
                        atomicOr(a.err, kErrTimeout);
                        break;
                    }
                    x[j] = ld_relaxed_gpu(&a.hub_val[r.t0 + q]);
                }
                tot = Op::combine(tot, Op::from_bits((uint32_t)(x[j] >> 32)));
                st_relaxed_gpu(&a.hub_val[r.t0 + q], 0ull);   // ready for the next superstep
            }
        }
        if (lane == 0) a.hub_arrive[r.t0] = 0u;
        finish(r.v, warp_all<Op>(tot));
    }
};

// Push superstep of SSSP / CC over the list of work items (at most 32
// out-edges of one vertex each; see push_superstep in frontier.cuh for why it
// equals the pull superstep). A warp collects the vertices it changed in
// shared memory and lists 32 at a time, so the list counter takes an atomic
// per 32 vertices instead of one per step with a change (a same-address
// bottleneck: 190K atomics in R-MAT 22's 6.1 M-edge superstep). A superstep
// of 45 K vertices took 144 us walking 32 edges at a time, 122 us at 4 x 32.
template <bool kW>
__device__ __forceinline__ void push(const SweepArgs& a, const Step& s, const FrontierCfg& fc,
                                     const StepStats* in, StepStats* out, WarpAcc& acc, uint32_t* pend,
                                     int lane) {
    const unsigned long long ne = __ldcg(&in->list_ne);
    const uint64_t n_items = min(ne >> 32, (unsigned long long)fc.list_cap);
    const uint64_t n_warps = (uint64_t)gridDim.x * kWarps;
    const uint64_t warp0 = (uint64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;   // neighbours on other SMs
    const uint64_t per = (n_items + n_warps - 1) / n_warps;
    const uint32_t c = per >= 32u ? 32u : (per ? (uint32_t)per : 1u);
    constexpr int kBatch = 4;
    uint32_t np = 0;   // vertices in pend (uniform over the warp)
    auto flush = [&](uint32_t n) {   // the first n <= 32 of them
        const bool has = (uint32_t)lane < n;
        const uint32_t v = has ? pend[lane] : 0u;
        const uint32_t deg = has ? __ldg(a.out_ptr + v + 1) - __ldg(a.out_ptr + v) : 0u;
        frontier_append(has, v, deg, fc, out, lane);
    };
    for (uint64_t b = warp0 * c; b < n_items; b += n_warps * c) {
        const uint64_t i = b + (uint64_t)lane;
        uint32_t e_lo = 0, n = 0, du = kInf;
        if ((uint32_t)lane < c && i < n_items) {
            const uint2 it = __ldcg(fc.list_in + i);
            const uint32_t u = it.x;
            du = __ldca(s.own_cur + u);
            const uint32_t r1 = __ldg(a.out_ptr + u + 1);
            e_lo = __ldg(a.out_ptr + u) + it.y * kItemEdges;
            n = min(r1 - e_lo, kItemEdges);
            // bring the next buffer up to date at vertex u (values only
            // decrease, so an entry already at or below du needs nothing)
            if (it.y == 0u && __ldcg(s.own_nxt + u) > du) atomicMin(s.own_nxt + u, du);
            if (kW && du == kInf) n = 0;   // unreachable: sends nothing
        }
        const uint32_t incl = warp_inclusive_scan(n, lane);
        const uint32_t excl = incl - n;
        const uint32_t total = __shfl_sync(kFull, incl, 31);
        // kBatch x 32 edges at a time: each is a chain of dependent loads and
        // an atomic, and the chains of a batch overlap
        for (uint32_t k0 = 0; k0 < total; k0 += 32u * kBatch) {
            uint32_t v[kBatch], m[kBatch], nv[kBatch], cv[kBatch];
#pragma unroll
            for (int q = 0; q < kBatch; ++q) {
                const uint32_t k = k0 + 32u * q + (uint32_t)lane;
                const int j = warp_owner(incl, k);
                const uint32_t e = __shfl_sync(kFull, e_lo, j) + (k - __shfl_sync(kFull, excl, j));
                const uint32_t dj = __shfl_sync(kFull, du, j);
                v[q] = k < total ? __ldg(a.out_dst + e) : kInf;
                m[q] = k < total ? push_message<kW>(dj, kW ? __ldg(a.out_w + e) : 0u) : kInf;
            }
#pragma unroll
            for (int q = 0; q < kBatch; ++q) {
                nv[q] = v[q] != kInf ? __ldcg(s.own_nxt + v[q]) : 0u;
                cv[q] = v[q] != kInf ? __ldca(s.own_cur + v[q]) : 0u;
            }
            bool app[kBatch];
#pragma unroll
            for (int q = 0; q < kBatch; ++q) {
                app[q] = false;
                if (m[q] < nv[q] && m[q] < cv[q]) app[q] = atomicMin(s.own_nxt + v[q], m[q]) >= cv[q];
            }
#pragma unroll
            for (int q = 0; q < kBatch; ++q) {
                const unsigned am = __ballot_sync(kFull, app[q]);
                if (!am) continue;
                if (app[q]) pend[np + (uint32_t)__popc(am & ((1u << lane) - 1u))] = v[q];
                np += (uint32_t)__popc(am);
                if (lane == 0) acc.changed += (uint32_t)__popc(am);
                __syncwarp();
                if (np >= 32u) {
                    flush(32u);
                    const uint32_t rest = np - 32u;   // below 32
                    const uint32_t x = (uint32_t)lane < rest ? pend[32 + lane] : 0u;
                    __syncwarp();
                    if ((uint32_t)lane < rest) pend[lane] = x;
                    __syncwarp();
                    np = rest;
                }
            }
        }
    }
    if (np) flush(np);
}

// The frontier a pull superstep left as bits (of slot t - 1's bitmap), as
// work items: each warp takes 32 words (1,024 vertices), counts their items,
// reserves their place with one atomic and writes them.
__device__ __forceinline__ void list_from_bits(const SweepArgs& a, const uint32_t* bits, const FrontierCfg& fc,
                                               StepStats* in, int lane) {
    const uint32_t words = (a.n_vertices + 31u) / 32u;
    const uint32_t n_groups = (words + 31u) / 32u;
    const uint32_t n_warps = gridDim.x * (blockDim.x >> 5);
    for (uint32_t g = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; g < n_groups; g += n_warps) {
        const uint32_t wi = g * 32u + (uint32_t)lane;
        const uint32_t mine = wi < words ? __ldcg(bits + wi) : 0u;
        const unsigned todo = __ballot_sync(kFull, mine != 0u);
        if (!todo) continue;
        auto vertex = [&](int j, uint32_t& v) -> uint32_t {   // items of word j's vertex in this lane
            const uint32_t b = __shfl_sync(kFull, mine, j);
            v = (g * 32u + (uint32_t)j) * 32u + (uint32_t)lane;
            return (b >> lane) & 1u ? frontier_items(__ldg(a.out_ptr + v + 1) - __ldg(a.out_ptr + v)) : 0u;
        };
        uint32_t cnt = 0, v;
        for (unsigned m = todo; m; m &= m - 1u) cnt += vertex(__ffs(m) - 1, v);
        cnt = __reduce_add_sync(kFull, cnt);
        unsigned long long base = 0ull;
        if (lane == 0) base = atomicAdd(&in->list_cursor, (unsigned long long)cnt);
        base = __shfl_sync(kFull, base, 0);
        for (unsigned m = todo; m; m &= m - 1u) {
            const uint32_t nit = vertex(__ffs(m) - 1, v);
            const uint32_t incl = warp_inclusive_scan(nit, lane);
            frontier_write(fc, base, incl, nit, v, lane);
            base += __shfl_sync(kFull, incl, 31);
        }
    }
}

// Whether superstep t pushes, from the stats of slot t; needs_list: its
// frontier is in a bitmap.
__device__ __forceinline__ bool sweep_pushes(const FrontierCfg& f, const StepStats* in, bool* needs_list) {
    *needs_list = false;
    if (f.list_out == nullptr || f.direction == GXP_DIR_PULL) return false;
    if (f.direction != GXP_DIR_PUSH) {
        const unsigned long long ne = __ldcg(&in->list_ne);
        const unsigned long long work = (ne >> 32) + (ne & 0xFFFFFFFFull);
        if (work * (unsigned long long)f.push_div > f.total_edges) return false;
    }
    *needs_list = __ldcg(&in->unlisted) != 0ull;
    return true;
}

// lists of superstep t, and the list its push reads
__device__ __forceinline__ FrontierCfg frontier_of(const SweepArgs& a, uint64_t t) {
    FrontierCfg fc = a.fc;
    fc.list_in = a.lists[t & 1];
    if (fc.list_out) fc.list_out = a.lists[(t + 1) & 1];
    return fc;
}

// the pull superstep t - 1's changed vertices as the list superstep t reads
__device__ __forceinline__ void build_list(const SweepArgs& a, uint64_t t, int lane) {
    FrontierCfg fc = a.fc;
    fc.list_out = a.lists[t & 1];
    list_from_bits(a, a.bits[(t + 2) % 3], fc, a.stats + t % kStatRing, lane);
}

// The supersteps of `run`. Superstep t reads value buffer, list and stat slot
// t, writes t + 1, clears stat slot t + 2 and changed bitmap (t + 1) mod 3; a
// grid barrier ends each superstep but a lone one (run.bar == nullptr, whose
// frontier k_sweep_list has listed).
template <Algo A, bool kCheck>
__global__ void __launch_bounds__(kThreads, 1) k_sweep(const SweepArgs a, const RunArgs run) {
    extern __shared__ __align__(16) uint32_t s_hot[];
    __shared__ unsigned long long s_acc[3];
    __shared__ uint32_t s_cnt[2];   // items, out-edges of the changed vertices
    __shared__ uint32_t s_pend[A == Algo::PR ? 1 : kWarps * 64];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool loop = run.bar != nullptr;
    uint64_t t = run.t0;
    uint64_t arrived = run.arrived;   // at the grid barriers so far
    if (tid < 3) s_acc[tid] = 0ull;
    if (tid < 2) s_cnt[tid] = 0u;
    __syncthreads();   // a push superstep has no other barrier before the warps add to them
    // The grid's barriers wait for CTAs that may not be on an SM yet, and never
    // get there while something else holds it. So nothing is done before all
    // of them have met here, within kGatherNs of the first; else none does
    // anything and the host takes a launch per superstep.
    if (loop && !grid_barrier<true>(run.bar, gridDim.x, arrived, kGatherNs, run.force != 0u, a.err)) return;
    auto clear_ahead = [&]() {   // what superstep t clears for those after it
        if (blockIdx.x == gridDim.x - 1) {
            unsigned long long* z = reinterpret_cast<unsigned long long*>(a.stats + (t + 2) % kStatRing);
            for (uint32_t i = tid; i < sizeof(StepStats) / 8; i += kThreads) z[i] = 0ull;
        }
        if (A != Algo::PR && a.fc.list_out) {
            uint32_t* z = a.bits[(t + 1) % 3];
            const uint32_t words = (a.n_vertices + 31u) / 32u;
            for (uint32_t i = blockIdx.x * kThreads + tid; i < words; i += gridDim.x * kThreads) z[i] = 0u;
        }
    };
    if (A != Algo::PR && !loop && run.quiet_stop) {   // a lone superstep after one that changed nothing
        const StepStats* const in = a.stats + t % kStatRing;
        if (!__any_sync(kFull, (__ldcg(&in->changed[lane]) + __ldcg(&in->changed[lane + 32])) != 0ull)) {
            clear_ahead();
            return;
        }
    }
    for (;;) {
        const StepStats* const in = a.stats + t % kStatRing;
        StepStats* const out = a.stats + (t + 1) % kStatRing;
        const FrontierCfg fc = frontier_of(a, t);
        Step s;
        s.own_cur = a.own[t & 1];
        s.own_nxt = a.own[(t + 1) & 1];
        s.rank_cur = a.rank[t & 1];
        s.rank_nxt = a.rank[(t + 1) & 1];
        s.bits = a.bits[t % 3];
        s.hot = (uint32_t)__cvta_generic_to_shared(s_hot);
        s.base = s.base_src = 0.0f;
        clear_ahead();
        bool pushes = false;
        if constexpr (A != Algo::PR) {
            bool needs_list;
            pushes = sweep_pushes(fc, in, &needs_list);   // the same in every thread of the grid
            if (pushes && needs_list && loop) {
                build_list(a, t, lane);
                if (!grid_barrier(run.bar, gridDim.x, arrived, run.timeout_ns, run.force != 0u, a.err)) return;
            }
            if (blockIdx.x == 0 && tid == 0 && fc.list_out) {
                if (pushes) {
                    out->pushed = 1ull;
                    out->push_edges = __ldcg(&in->list_ne) & 0xFFFFFFFFull;
                } else {
                    out->unlisted = 1ull;
                }
            }
        } else {
            // base terms, from the exact dangling mass of the current ranks
            const unsigned long long sd =
                warp_sum_u62(__ldcg(&in->dangling_fx[lane]) + __ldcg(&in->dangling_fx[lane + 32]));
            pagerank_base(sd, a.damping, a.inv_n, a.ppr_source != kInf, &s.base, &s.base_src);
        }
        WarpAcc acc;
        if (pushes) {
            if constexpr (A != Algo::PR)
                push<Ops<A>::kWeighted>(a, s, fc, in, out, acc, s_pend + warp * 64, lane);
        } else {
            // each CTA starts elsewhere, so that the SMs do not all ask the same L2 slices at once
            const uint32_t n16 = a.n_hot / 4, i0 = (uint32_t)((uint64_t)n16 * blockIdx.x / gridDim.x);
            for (uint32_t k = tid; k < n16; k += kThreads) {
                const uint32_t i = k + i0 < n16 ? k + i0 : k + i0 - n16;
                stage16(s.hot + 16u * i, s.own_cur + 4u * i);
            }
            Pull<A, kCheck> p{a, s, acc, lane};
            constexpr int kU = kCols<A>;
            // Items of a kind cost the same, so they are dealt out evenly:
            // warp w of the grid takes every n_warps-th, each kind starting
            // where the one before it ended. Neighbouring warps are on
            // different SMs, so a partial round is spread over all of them.
            const uint32_t n_warps = gridDim.x * kWarps, w0 = (uint32_t)warp * gridDim.x + blockIdx.x;
            uint32_t used = 0;   // warps taken by the rounds so far, mod n_warps
            auto deal = [&](uint32_t n) {   // this warp's first of n items
                const uint32_t f = w0 >= used ? w0 - used : w0 + n_warps - used;
                used = (uint32_t)(((uint64_t)used + n) % n_warps);
                return f;
            };
            if constexpr (A == Algo::PR)   // these gather nothing: done while the staged values arrive
                p.template groups<kZeroGroup>(a.n_gt0, a.n_slices,
                                              deal((a.n_slices - a.n_gt0 + kZeroGroup - 1) / kZeroGroup), n_warps,
                                              [&](uint32_t wd, uint32_t n) { p.zero_rows(wd, n); });
            stage_wait();
            __syncthreads();
            p.hub_parts(a.n_hubs, deal(a.n_hubs), n_warps);
            {
                const uint32_t n = p.n_subs();
                p.subs(n, deal(n), n_warps);
            }
            constexpr int kN4 = kU / 4;
            if constexpr (kU >= 8)
                p.template groups<1>(a.n_gt8, a.n_gt4, deal(a.n_gt4 - a.n_gt8), n_warps,
                                     [&](uint32_t wd, uint32_t n) { p.template narrow<1>(wd, n); });
            p.template groups<kN4>(a.n_gt4, a.n_gt0, deal((a.n_gt0 - a.n_gt4 + kN4 - 1) / kN4), n_warps,
                                   [&](uint32_t wd, uint32_t n) { p.template narrow<kN4>(wd, n); });
        }
        // lane sums -> warp -> CTA -> one global atomic each
        const uint32_t n_changed = __reduce_add_sync(kFull, acc.changed);
        if constexpr (A == Algo::PR) {
            acc.l1 = warp_sum_u62(acc.l1);
            acc.dang = warp_sum_u62(acc.dang);
        } else {
            acc.items = __reduce_add_sync(kFull, acc.items);
            acc.edges = __reduce_add_sync(kFull, acc.edges);
        }
        if (lane == 0) {
            if (n_changed) atomicAdd(&s_acc[0], (unsigned long long)n_changed);
            if (acc.l1) atomicAdd(&s_acc[1], acc.l1);
            if (acc.dang) atomicAdd(&s_acc[2], acc.dang);
            if (acc.items) atomicAdd(&s_cnt[0], acc.items);
            if (acc.edges) atomicAdd(&s_cnt[1], acc.edges);
        }
        __syncthreads();
        if (tid == 0) {
            const uint32_t ln = blockIdx.x % kStatLanes;
            if (s_acc[0]) atomicAdd(&out->changed[ln], s_acc[0]);
            if (s_acc[1]) atomicAdd(&out->l1_fx[ln], s_acc[1]);
            if (s_acc[2]) atomicAdd(&out->dangling_fx[ln], s_acc[2]);
            if (s_cnt[0]) atomicAdd(&out->list_ne, list_pack(s_cnt[0], s_cnt[1]));
            s_acc[0] = s_acc[1] = s_acc[2] = 0ull;
            s_cnt[0] = s_cnt[1] = 0u;
        }
        if (!loop) return;
        if (!grid_barrier(run.bar, gridDim.x, arrived, run.timeout_ns, run.force != 0u, a.err)) return;
        ++t;   // supersteps done; slot t holds the last one's counts
        bool more = t < run.limit;
        if (more && run.quiet_stop) {   // every warp reads the counts itself
            const StepStats* st = a.stats + t % kStatRing;
            const unsigned long long c = __ldcg(&st->changed[lane]) + __ldcg(&st->changed[lane + 32]);
            more = __any_sync(kFull, c != 0ull);
        }
        if (more) continue;
        if (blockIdx.x == 0) {   // report: warp w sums superstep run.t0 + w's stats
            const uint64_t mine = run.t0 + (uint32_t)warp;
            if (mine < t) {
                const StepStats* st = a.stats + (mine + 1) % kStatRing;
                report_step(st, &run.out->sum[warp], a.err, &run.out->err);
            }
            if (tid == 0) {
                run.out->arrived = arrived;
                run.out->step = t;
            }
        }
        return;
    }
}
static_assert(kRunChunk <= kWarps, "a warp reports each superstep of a launch");

// before a superstep of its own launch: the list its push reads
__global__ void __launch_bounds__(256) k_sweep_list(const SweepArgs a, uint64_t t) {
    bool needs_list;
    const FrontierCfg fc = frontier_of(a, t);
    if (sweep_pushes(fc, a.stats + t % kStatRing, &needs_list) && needs_list) build_list(a, t, threadIdx.x & 31);
}

template <Algo A, bool kCheck>
cudaError_t launch_t(const SweepArgs& args, const RunArgs& run, uint32_t ctas, cudaStream_t s) {
    const void* fn = (const void*)k_sweep<A, kCheck>;
    const size_t smem = 4 * (size_t)args.n_hot;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * (int)kMaxHot);
    if (e != cudaSuccess) return e;
    SweepArgs a = args;
    RunArgs r = run;
    void* params[] = {&a, &r};
    return cudaLaunchKernel(fn, dim3(ctas), dim3(kThreads), params, smem, s);
}

}  // namespace

cudaError_t load_sweep_list() {
    cudaFuncAttributes at;
    return cudaFuncGetAttributes(&at, k_sweep_list);
}

// All values of a graph that fits, else of a renumbered graph's first
// vertices (its hottest), else none. Staging takes ~2 us for 128 KB, which a
// small graph's gathers do not win back: a staged value per 128 edges.
uint32_t sweep_hot_values(uint64_t n_vertices, uint64_t n_edges, bool by_degree) {
    const uint64_t all = (n_vertices + 1 + 3) & ~3ull;   // with the identity slot
    const uint64_t worth = std::min<uint64_t>(kMaxHot, (n_edges / 128) & ~3ull);
    if (all <= worth) return (uint32_t)all;
    return by_degree ? (uint32_t)worth : 0u;
}

cudaError_t launch_sweep(Algo alg, const SweepArgs& args, const RunArgs& run, uint32_t sms, cudaStream_t s) {
    uint32_t at = 0;   // the item ranges follow one another
    for (uint32_t end : {args.n_lanes[0], args.n_lanes[1], args.n_lanes[2], args.n_lanes[3], args.n_lanes[4],
                         args.n_gt8, args.n_gt4, args.n_gt0, args.n_slices}) {
        if (end < at) return cudaErrorInvalidValue;
        at = end;
    }
    if (args.n_hot > kMaxHot || args.n_hot % 4 || sms == 0) return cudaErrorInvalidValue;
    if (run.bar && (run.limit <= run.t0 || run.limit - run.t0 > kRunChunk || !run.out)) return cudaErrorInvalidValue;
    // A CTA for every kWarps items at least: on a small graph the barriers of
    // fewer CTAs cost less than a warp's second item. Runs of many supersteps
    // of little work, an item or more a CTA / 16 / 32 (us a superstep): SSSP
    // along a path of 20,000 vertices 9.3 / - / 7.1, on a 300 x 300 mesh 10.0 /
    // 10.0 / 8.7; PageRank of R-MAT 12 9.9 / 8.6 / 9.4. (64: 6.9, 8.1, -, but a
    // warp's items then follow one another on graphs that fill the chip.)
    uint64_t items = args.n_hubs + (args.n_slices - args.n_lanes[4]);
    for (int c = 0; c < 5; ++c) items += (uint64_t)(args.n_lanes[c] - (c ? args.n_lanes[c - 1] : 0u)) << (5 - c);
    const uint32_t ctas = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(sms, (items + kWarps - 1) / kWarps));
    const bool chk = args.check_bounds != 0;
    if (!run.bar && alg != Algo::PR && args.fc.list_out && args.fc.direction != GXP_DIR_PULL) {
        k_sweep_list<<<sms, 256, 0, s>>>(args, run.t0);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    switch (alg) {
        case Algo::SSSP: return chk ? launch_t<Algo::SSSP, true>(args, run, ctas, s)
                                    : launch_t<Algo::SSSP, false>(args, run, ctas, s);
        case Algo::CC: return chk ? launch_t<Algo::CC, true>(args, run, ctas, s)
                                  : launch_t<Algo::CC, false>(args, run, ctas, s);
        case Algo::PR: return chk ? launch_t<Algo::PR, true>(args, run, ctas, s)
                                  : launch_t<Algo::PR, false>(args, run, ctas, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace gxp
