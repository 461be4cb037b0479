// Superstep kernel of partitioned graphs over the sliced-ELL layout: MSGGen +
// MSGMerge + MSGApply (Section IV-A1's algorithm template) in pull form, one
// warp per work item (one partition has its own kernel, sweep.cu).
// For SSSP and CC the same grid runs the push direction instead when the
// frontier is small (frontier.cuh); the choice is made on the device from
// the previous superstep's frontier size.
//
//  * slice of 32 non-hub rows (the edge block of Section II-B, laid out
//    column-major): lane i owns row i. For each of the slice's `width` edge
//    slots the warp reads 32 consecutive source ids (one coalesced 128-byte
//    load), gathers the sources' values with up to kUnroll independent loads
//    in flight per lane, and folds the messages into a per-lane register in
//    the row's edge order (MSGMerge without shuffles or shared memory). Then
//    each lane applies its row (MSGApply); the changed bits of a warp are
//    grouped per bitmap word with __match_any_sync and ORed in with one
//    atomic per word.
//  * hub part: up to kHubPartEdges in-edges of one high-in-degree row,
//    reduced lane-strided in registers and by a fixed warp tree; the last part
//    of a row to arrive combines all parts in part order and applies.
//
// Sums run in a fixed order, so fp32 PageRank is deterministic; PageRank's
// global sums (dangling mass, L1 delta) are exact 64-bit fixed point.
#include "frontier.cuh"
#include "merge_ops.cuh"

#include <algorithm>

namespace gxp {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kSellBlock = 256;
constexpr int kSellWarps = kSellBlock / 32;

// Gathers in flight per lane and the CTAs per SM the registers are fitted to.
// PageRank at 12 and 5 (48 registers) measured 181 us per R-MAT 22 superstep
// on one partition against 197 us for 8 at 6 CTAs.
template <Algo A> struct Tune { static constexpr int kUnroll = 8, kMinBlocks = 6; };
template <> struct Tune<Algo::SSSP> { static constexpr int kUnroll = 8, kMinBlocks = 5; };
template <> struct Tune<Algo::PR> { static constexpr int kUnroll = 12, kMinBlocks = 5; };

// The value of local source u of partition P: an owned vertex, a cached
// copy, or (the padding id of empty slots) the identity slot.
struct Source {
    const uint32_t* own;    // own_cur + v_begin
    const uint32_t* copy;   // ghost + ghost_base - n_own: copy(u) for u >= n_own
    uint32_t n_own;
    __device__ __forceinline__ Source(const uint32_t* own_cur, const uint32_t* ghost, const PartDev& P)
        : own(own_cur + P.v_begin), copy(ghost + P.ghost_base - (ptrdiff_t)P.n_own), n_own(P.n_own) {}
    __device__ __forceinline__ const uint32_t* at(uint32_t u) const {
        return u < n_own ? own + u : copy + u;
    }
};

// One CTA's share of superstep t over the sliced-ELL layout (see the top of
// the file). kCheck: range-check every source id (gxp_config.check_bounds),
// setting kErrBounds instead of loading.
template <Algo A, bool kCheck>
__global__ void __launch_bounds__(kSellBlock, Tune<A>::kMinBlocks) k_sell(const SellArgs a) {
    using Op = Ops<A>;
    using T = typename Op::T;
    constexpr int kU = Tune<A>::kUnroll;
    const uint64_t t = a.step;
    const uint32_t vb = blockIdx.x;
    __shared__ unsigned long long s_acc[4];
    __shared__ uint32_t s_done;
    __shared__ uint32_t s_ftot[kSellWarps], s_fedges[kSellWarps];   // frontier items, out-edges per warp
    __shared__ unsigned long long s_fbase;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // superstep t reads value buffer t & 1 and stat slot t, writes the others
    const uint32_t* const own_cur = a.own[t & 1];
    uint32_t* const own_nxt = a.own[(t + 1) & 1];
    const float* const rank_cur = a.rank[t & 1];
    float* const rank_nxt = a.rank[(t + 1) & 1];
    const StepStats* const stats_in = a.stats + t % kStatRing;
    StepStats* const stats_out = a.stats + (t + 1) % kStatRing;
    FrontierCfg fc = a.fc;
    fc.list_in = a.lists[t & 1];
    if (fc.list_out) fc.list_out = a.lists[(t + 1) & 1];
    if (vb == 0) {
        // zero the ring slot two supersteps ahead (never read or written by this one)
        unsigned long long* z = reinterpret_cast<unsigned long long*>(a.stats + (t + 2) % kStatRing);
        for (uint32_t i = tid; i < sizeof(StepStats) / 8; i += kSellBlock) z[i] = 0ull;
    }
    for (uint64_t i = (uint64_t)vb * kSellBlock + tid; i <= a.n_vertices / 32u; i += (uint64_t)gridDim.x * kSellBlock)
        a.changed_next[i] = 0u;
    __shared__ bool s_quiet, s_list;
    if (tid == 0) {
        s_acc[0] = s_acc[1] = s_acc[2] = s_acc[3] = 0ull;
        s_done = 0u;
        s_quiet = false;
        s_list = true;
    }
    const bool gate = fc.list_out != nullptr && fc.list_max_changed != kAlwaysList;
    if (((a.early_exit && t > 0) || gate) && warp == 0) {
        // the vertices the previous superstep changed (this one's frontier)
        const unsigned long long c = warp_sum_u62(stats_in->changed[lane] + stats_in->changed[lane + 32]);
        if (lane == 0) {
            // min-label algorithms at a fixed point: nothing can change any more
            if (a.early_exit && t > 0 && c == 0ull) s_quiet = true;
            if (gate) {   // the same inputs, so the same choice, in every CTA
                const unsigned long long ne = stats_in->list_ne;
                const unsigned long long work = (ne >> 32) + (ne & 0xFFFFFFFFull);
                s_list = c <= fc.list_max_changed &&
                         work * (unsigned long long)fc.push_div <= (unsigned long long)kListSlack * fc.total_edges;
            }
        }
    }
    // PageRank base terms, from the exact dangling mass of the current ranks
    // (every warp forms them itself: no wait on another warp's loads)
    float base = 0.0f, base_src = 0.0f;
    if constexpr (A == Algo::PR) {
        const unsigned long long sd = warp_sum_u62(stats_in->dangling_fx[lane] + stats_in->dangling_fx[lane + 32]);
        pagerank_base(sd, a.damping, a.inv_n, a.ppr_source != kInf, &base, &base_src);
    }
    __syncthreads();
    if (s_quiet) return;   // same for every thread of the grid
    const float damping = a.damping;

    uint32_t n_changed = 0, n_boundary = 0;
    unsigned long long l1 = 0ull, dang = 0ull;

    // MSGApply of local vertex v of partition P with merged message m
    auto apply = [&](const PartDev& P, uint32_t v, T m) -> bool {
        const uint32_t gid = P.v_begin + v;
        if constexpr (A == Algo::PR) {
            const float rn = fmaf(damping, m, gid == a.ppr_source ? base_src : base);
            const float ro = rank_cur[gid];
            const uint32_t od = a.outdeg[gid];
            rank_nxt[gid] = rn;
            const float c = od ? __fdiv_rn(rn, (float)od) : 0.0f;
            const uint32_t cb = __float_as_uint(c);
            own_nxt[gid] = cb;
            const unsigned long long fn = fx_of(rn), fo = fx_of(ro);
            l1 += fn > fo ? fn - fo : fo - fn;
            if (od == 0u) dang += fn;
            return cb != own_cur[gid];
        } else {
            const uint32_t old = own_cur[gid];
            const uint32_t nw = min(old, (uint32_t)m);
            own_nxt[gid] = nw;
            return nw != old;
        }
    };
    // kCheck: a source id outside the partition's ids (and not its padding id)
    // is reported and replaced by the padding id
    auto checked = [&](const PartDev& P, uint32_t u) -> uint32_t {
        if constexpr (kCheck) {
            if (u >= P.n_own + P.n_ghost && u != P.pad_id) {
                atomicOr(a.err, kErrBounds);
                return P.pad_id;
            }
        }
        return u;
    };

    const uint32_t gw = vb * kSellWarps + (uint32_t)warp;
    bool f_has = false;   // pull direction with frontier lists: this lane's changed vertex
    uint32_t f_v = 0;
    bool pushed = false;
    if constexpr (A != Algo::PR) {
        if (push_chosen(fc, stats_in)) {   // same choice in every thread of the grid
            const uint32_t c = push_superstep<Op::kWeighted>(fc, a.out_ptr, a.out_dst, a.out_w, own_cur, own_nxt,
                                                             a.ghost, a.n_vertices, a.changed_bits, a.boundary_bits, n_boundary, stats_in,
                                                             stats_out, gw, (uint64_t)gridDim.x * kSellWarps, lane);
            if (lane == 0) n_changed += c;
            pushed = true;
        } else if (!s_list && vb == 0 && tid == 0) {
            stats_out->unlisted = 1ull;   // the next superstep pulls
        }
    }
    if (pushed) {
        // the frontier's out-edges were relaxed above
    } else if (gw < a.n_hubs) {
        // ============================================================ hub part
        const HubPart hp = a.hubs[gw];
        const PartDev P = a.parts[hp.part];
        const Source S(own_cur, a.ghost, P);
        const uint32_t* src = P.hsrc + hp.e0;
        const uint32_t* wts = P.hw + hp.e0;
        T acc = Op::ident();
        auto hbatch = [&](uint32_t j0) {   // in-edges [j0, j0 + 32 kU) of the part, lane-strided
            uint32_t u[kU], x[kU], wv[kU];
#pragma unroll
            for (int q = 0; q < kU; ++q) {
                const uint32_t j = j0 + (uint32_t)q * 32u + (uint32_t)lane;
                const bool in = j < hp.ne;
                u[q] = in ? ld_stream(src + j) : 0u;
                wv[q] = (Op::kWeighted && in) ? ld_stream(wts + j) : 0u;
            }
#pragma unroll
            for (int q = 0; q < kU; ++q)
                x[q] = j0 + (uint32_t)q * 32u + (uint32_t)lane < hp.ne ? __ldg(S.at(checked(P, u[q])))
                                                                        : Op::to_bits(Op::ident());
#pragma unroll
            for (int q = 0; q < kU; ++q)
                if (j0 + (uint32_t)q * 32u + (uint32_t)lane < hp.ne) acc = Op::combine(acc, Op::gen(x[q], wv[q]));
        };
        for (uint32_t jb = 0; jb < hp.ne; jb += 32u * kU) hbatch(jb);
        T total = warp_all<Op>(acc);
        bool do_apply = hp.nparts == 1u;
        if (!do_apply) {
            uint32_t last = 0;
            if (lane == 0) {
                __stcg(&a.hub_val[gw], Op::to_bits(total));
                last = arrive_acq_rel(&a.hub_arrive[hp.t0]) == hp.nparts - 1u ? 1u : 0u;
            }
            last = __shfl_sync(kFull, last, 0);
            if (last) {
                __threadfence();
                T tot = Op::ident();   // parts in a fixed order: lane-strided, then a fixed tree
                for (uint32_t q = (uint32_t)lane; q < hp.nparts; q += 32u)
                    tot = Op::combine(tot, Op::from_bits(__ldcg(&a.hub_val[hp.t0 + q])));
                total = warp_all<Op>(tot);
                if (lane == 0) a.hub_arrive[hp.t0] = 0u;   // ready for the next superstep
                do_apply = true;
            }
        }
        const bool ch = do_apply && lane == 0 && apply(P, hp.v, total);
        if (ch) {
            ++n_changed;
            const uint32_t g = P.v_begin + hp.v;
            atomicOr(&a.changed_bits[g >> 5], 1u << (g & 31u));
            n_boundary += (__ldg(a.boundary_bits + (g >> 5)) >> (g & 31u)) & 1u;
        }
        if constexpr (A != Algo::PR) {
            if (ch && fc.list_out) {   // the vertex joins the next frontier
                f_has = true;
                f_v = P.v_begin + hp.v;
            }
        }
    } else if (gw - a.n_hubs < a.n_slices) {
        // =============================================================== slice
        const SellSlice sl = a.slices[gw - a.n_hubs];
        const PartDev P = a.parts[sl.part];
        const Source S(own_cur, a.ghost, P);
        const uint32_t row = P.perm[sl.row0 + lane];
        T acc = Op::ident();
        auto batch = [&](uint32_t k0, uint32_t ncols) {   // columns [k0, k0 + ncols), k0 % kU == 0
            uint32_t u[kU], x[kU], wv[kU];
            // column by column, 128-byte warp loads
            const uint32_t* col = P.sell_src + sl.off + lane;
            const uint32_t* wcol = P.sell_w + sl.off + lane;
#pragma unroll
            for (int q = 0; q < kU; ++q) {
                const bool in = (uint32_t)q < ncols;
                u[q] = in ? ld_stream(col + 32u * (k0 + q)) : 0u;
                wv[q] = (Op::kWeighted && in) ? ld_stream(wcol + 32u * (k0 + q)) : 0u;
            }
#pragma unroll
            for (int q = 0; q < kU; ++q)
                x[q] = (uint32_t)q < ncols ? __ldg(S.at(checked(P, u[q]))) : Op::to_bits(Op::ident());
#pragma unroll
            for (int q = 0; q < kU; ++q)
                if ((uint32_t)q < ncols) acc = Op::combine(acc, Op::gen(x[q], wv[q]));
        };
        // whole batches of kU columns (kU gathers in flight per lane), then the rest
        const uint32_t full = sl.width - sl.width % kU;
        uint32_t kb = 0;
        for (; kb < full; kb += kU) batch(kb, kU);
        if (kb < sl.width) batch(kb, sl.width - kb);
        const bool ch = row != kSellPad && apply(P, row, acc);
        const unsigned chm = __ballot_sync(kFull, ch);
        if (lane == 0) n_changed += __popc(chm);
        if constexpr (A != Algo::PR) {
            if (ch && fc.list_out) {
                f_has = true;
                f_v = P.v_begin + row;
            }
        }
        if (ch) {
            // one atomic per bitmap word touched by this warp
            const uint32_t g = P.v_begin + row;
            const unsigned grp = __match_any_sync(chm, g >> 5);
            const unsigned bits = __reduce_or_sync(grp, 1u << (g & 31u));
            if ((uint32_t)lane == (uint32_t)(__ffs(grp) - 1)) {
                atomicOr(&a.changed_bits[g >> 5], bits);
                n_boundary += (uint32_t)__popc(bits & __ldg(a.boundary_bits + (g >> 5)));
            }
        }
    }

    if constexpr (A != Algo::PR) {
        if (fc.list_out && !pushed && s_list) {   // uniform over the grid
            // the changed vertices join the next frontier: one atomic per CTA
            // reserves the CTA's items, each warp writes its own; a vertex's
            // items cover the out-edges of its slot
            const uint32_t deg = f_has ? __ldg(a.out_ptr + f_v + 1) - __ldg(a.out_ptr + f_v) : 0u;
            const uint32_t nit = f_has ? frontier_items(deg) : 0u;
            const uint32_t incl = warp_inclusive_scan(nit, lane);
            const uint32_t edges = __reduce_add_sync(kFull, deg);
            if (lane == 31) {
                s_ftot[warp] = incl;
                s_fedges[warp] = edges;
            }
            __syncthreads();
            if (tid == 0) {
                uint32_t items = 0, e = 0;
                for (int w = 0; w < kSellWarps; ++w) {
                    const uint32_t t = s_ftot[w];
                    s_ftot[w] = items;   // -> the warp's offset in the CTA's range
                    items += t;
                    e += s_fedges[w];
                }
                s_fbase = items ? atomicAdd(&stats_out->list_ne, list_pack(items, e)) >> 32 : 0ull;
            }
            __syncthreads();
            if (__shfl_sync(kFull, incl, 31)) frontier_write(fc, s_fbase + s_ftot[warp], incl, nit, f_v, lane);
        }
    }

    // warp totals -> CTA totals in shared memory; the last warp flushes them
    const unsigned long long c64 = __reduce_add_sync(kFull, n_changed), b64 = __reduce_add_sync(kFull, n_boundary);
    if constexpr (A == Algo::PR) {
        l1 = warp_sum_u62(l1);
        dang = warp_sum_u62(dang);
    }
    if (lane == 0) {
        if (c64) atomicAdd(&s_acc[0], c64);
        if (l1) atomicAdd(&s_acc[1], l1);
        if (dang) atomicAdd(&s_acc[2], dang);
        if (b64) atomicAdd(&s_acc[3], b64);
        __threadfence_block();
        if (atomicAdd(&s_done, 1u) == (uint32_t)kSellWarps - 1u) {
            __threadfence_block();
            const unsigned long long x0 = atomicAdd(&s_acc[0], 0ull), x1 = atomicAdd(&s_acc[1], 0ull),
                                     x2 = atomicAdd(&s_acc[2], 0ull), x3 = atomicAdd(&s_acc[3], 0ull);
            const uint32_t ln = vb % kStatLanes;
            if (x0) atomicAdd(&stats_out->changed[ln], x0);
            if (x1) atomicAdd(&stats_out->l1_fx[ln], x1);
            if (x2) atomicAdd(&stats_out->dangling_fx[ln], x2);
            if (x3) atomicAdd(&stats_out->boundary[ln], x3);
        }
    }
}

}  // namespace

template <Algo A>
static void launch_sell(const SellArgs& args, uint32_t grid, cudaStream_t s) {
    if (args.check_bounds) k_sell<A, true><<<grid, kSellBlock, 0, s>>>(args);
    else k_sell<A, false><<<grid, kSellBlock, 0, s>>>(args);
}

cudaError_t launch_superstep_sell(Algo alg, const SellArgs& args, cudaStream_t s) {
    // an empty layout still runs one block: it clears the stat slot two
    // supersteps ahead
    const uint64_t work = (uint64_t)args.n_hubs + args.n_slices;
    const uint32_t grid = (uint32_t)std::max<uint64_t>(1, (work + kSellWarps - 1) / kSellWarps);
    switch (alg) {
        case Algo::SSSP: launch_sell<Algo::SSSP>(args, grid, s); break;
        case Algo::CC: launch_sell<Algo::CC>(args, grid, s); break;
        case Algo::PR: launch_sell<Algo::PR>(args, grid, s); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace gxp
