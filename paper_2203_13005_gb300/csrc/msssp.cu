// Batched multi-source SSSP superstep: up to 64 Bellman-Ford instances (one
// per source, Section V-A's multi-source SSSP-BF) advance together in one
// pass over the edges, so every edge block read from memory (or streamed by
// the pipeline shuffle of Section III-A) serves all sources.
//
// Layout: dist[v][64] uint32 (one 256-byte row per vertex); an edge is a
// (source, weight) uint2 in destination order, or one uint32 (weight << 24 |
// source) when sources and weights fit, halving the bytes every superstep
// reads (and streams). Work unit = up to kUnitEdges in-edges of one
// destination, a warp each; a lane holds four slots (a 128-bit load), so LG
// lanes hold a row (16 for 64 slots, fewer when only the first slots are in
// use) and the warp works on 32 / LG edges at once:
//   MSGGen   the warp reads 32 in-edges at once (one per lane, coalesced),
//            tests each source against the frontier (changed in the
//            previous superstep) and compacts the active ones into shared
//            memory; each lane group then reads the rows of its share of them
//            (8 in flight per lane) and adds w, saturating below INF.
//            A unit with no active in-edge ends there (no row traffic);
//   MSGMerge per-slot minimum in registers, then over the lane groups;
//   MSGApply new = min(old, merged) is stored in place (rows split over
//            several units use atomicMin), and a destination with any
//            improved slot sets its frontier bit for the next superstep.
// What bounds it: instruction issue and, for the many short rows of a
// power-law graph, the chain unit -> edges -> frontier bits -> rows. So a
// warp reads 32 unit descriptors at a time and is always two units ahead with
// the edges and one with the frontier bits, and the old row travels with the
// source rows. R-MAT 20, 64 sources, 99 M active edges: with two slots a lane,
// a shuffle pair per edge and no look-ahead a run took 7.4 ms (41
// instructions per active edge, 56% of issue slots); 5.4 ms so, and 4.6 ms
// with the units longest first (a quarter of the warps' time was spent at the
// superstep's barrier); 32 / 16 / 5 / 1 sources 7.4 / 6.8 / 5.9 / 4.5 -> 3.3 /
// 2.9 / 2.6 / 2.0 ms.
// Slots in idle_mask (no query) are skipped. In-place updates only ever
// lower distances, so the fixed point equals the per-source Bellman-Ford
// result; superstep counts may be below Jacobi's.
#include <algorithm>

#include "grid_sync.cuh"
#include "gxp_internal.hpp"

namespace gxp {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kMsBlock = 256;
constexpr int kMsWarps = kMsBlock / 32;

// d + w, saturating below INF; INF stays. kNoSat: no finite sum reaches INF.
template <bool kNoSat>
__device__ __forceinline__ uint32_t relax(uint32_t acc, uint32_t d, uint32_t w) {
    const uint32_t s = d + w;
    if constexpr (kNoSat) {
        return s >= w ? min(acc, s) : acc;   // only INF + w wraps (and INF + 0 is INF)
    } else {
        if (d == kInf) return acc;
        return min(acc, s < d || s == kInf ? kInf - 1u : s);
    }
}

template <bool kPacked>
__device__ __forceinline__ uint2 load_edge(const void* base, uint64_t i) {
    if (kPacked) {
        const uint32_t p = __ldg(static_cast<const uint32_t*>(base) + i);
        return make_uint2(p & ((1u << kPackSrcBits) - 1u), p >> kPackSrcBits);
    }
    return __ldg(static_cast<const uint2*>(base) + i);
}

// The rows of active edges [i, n) of `list` (kQ steps of 32 / LG edges), merged into acc.
template <int LG, int kQ, bool kNoSat>
__device__ __forceinline__ void merge_rows(const uint4* dist, const uint2* list, uint32_t i, uint32_t n, uint32_t sub,
                                           uint32_t l, uint4& acc) {
    constexpr uint32_t kPer = 32 / LG;
    uint4 row[kQ];
    uint32_t w[kQ];
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        const uint32_t k = i + (uint32_t)q * kPer + sub;
        row[q] = make_uint4(kInf, kInf, kInf, kInf);
        w[q] = 0u;
        if (k < n) {
            const uint2 e = list[k];
            w[q] = e.y;
            row[q] = dist[(uint64_t)e.x * 16u + l];
        }
    }
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        acc.x = relax<kNoSat>(acc.x, row[q].x, w[q]);
        acc.y = relax<kNoSat>(acc.y, row[q].y, w[q]);
        acc.z = relax<kNoSat>(acc.z, row[q].z, w[q]);
        acc.w = relax<kNoSat>(acc.w, row[q].w, w[q]);
    }
}

// One block's share of a superstep (the units u_begin + warp, + n_warps, ...
// of the grid). kLoop: called by the persistent loop, which reads frontier
// bits written earlier in the same launch, so through coherent loads.
template <int LG, bool kDry, bool kPacked, bool kLoop, bool kNoSat>
__device__ __forceinline__ void msssp_block(const MsArgs& a) {
    constexpr uint32_t kPer = 32 / LG;   // edges the warp works on at once
    __shared__ uint32_t s_imp[2], s_done;
    __shared__ unsigned long long s_changed, s_active;
    __shared__ uint2 s_list[kMsWarps][32];
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 2) s_imp[threadIdx.x] = 0u;
    if (threadIdx.x == 0) {
        s_changed = 0ull;
        s_active = 0ull;
        s_done = 0u;
    }
    __syncthreads();
    uint2* const list = s_list[threadIdx.x >> 5];
    const uint4* const dist = reinterpret_cast<const uint4*>(a.dist);
    const uint32_t l = (uint32_t)lane % LG, sub = (uint32_t)lane / LG;   // slots 4l .. 4l + 3, the sub-th of kPer edges
    const uint32_t busy = (uint32_t)(~a.idle_mask >> (4u * l)) & 15u;    // of my four slots
    uint32_t imp_lo = 0u, imp_hi = 0u;   // improved slots 0..31 / 32..63 (bit = slot)
    const uint32_t warp0 = (blockIdx.x * kMsBlock + threadIdx.x) >> 5;
    const uint32_t n_warps = (gridDim.x * kMsBlock) >> 5;
    uint32_t changed_units = 0;
    unsigned long long n_active = 0;   // active in-edges this warp walked (the same in every lane)
    auto edge_at = [&](uint64_t e, uint32_t i, uint32_t len) {
        return i < len ? load_edge<kPacked>(a.edges, e + i) : make_uint2(0u, 0u);
    };
    auto bits_of = [&](uint2 ed, uint32_t i, uint32_t len) {   // the frontier word of the edge's source
        const uint32_t* p = a.frontier_cur + (ed.x >> 5);
        return i < len ? (kLoop ? __ldca(p) : __ldg(p)) : 0u;
    };
    for (uint64_t base = a.u_begin + warp0; base < a.u_end; base += 32ull * n_warps) {
        // the warp's next 32 units, one descriptor per lane: {v, first edge (global), edges, split flag}
        const uint64_t mine = base + (uint64_t)lane * n_warps;
        uint4 un = mine < a.u_end ? a.units[mine] : make_uint4(0u, (uint32_t)a.edge_base, 0u, 0u);
        const int n_units = (int)min(32ull, (unsigned long long)((a.u_end - base + n_warps - 1) / n_warps));
        auto first_of = [&](int j) { return (uint64_t)__shfl_sync(kFull, un.y, j & 31) - a.edge_base; };
        auto len_of = [&](int j) { return j < n_units ? __shfl_sync(kFull, un.z, j & 31) : 0u; };   // j is uniform
        uint2 e0 = edge_at(first_of(0), lane, len_of(0)), e1 = edge_at(first_of(1), lane, len_of(1));
        uint32_t f0 = bits_of(e0, lane, len_of(0));
        for (int j = 0; j < n_units; ++j) {
            const uint32_t v = __shfl_sync(kFull, un.x, j), len = __shfl_sync(kFull, un.z, j),
                           split = __shfl_sync(kFull, un.w, j);
            const uint64_t e = first_of(j);
            uint2 my = e0;
            uint32_t fw = f0;
            // look ahead: the next unit's frontier words, the edges of the one after
            f0 = bits_of(e1, lane, len_of(j + 1));
            e0 = e1;
            e1 = edge_at(first_of(j + 2), lane, len_of(j + 2));
            uint4 acc = make_uint4(kInf, kInf, kInf, kInf), old = acc;
            bool any = false;
            for (uint32_t b = 0;;) {
                const bool act = b + (uint32_t)lane < len && ((fw >> (my.x & 31u)) & 1u);
                const uint32_t mask = __ballot_sync(kFull, act);
                if (mask) {
                    const uint32_t n = (uint32_t)__popc(mask);
                    if (!any && !kDry && (uint32_t)lane < LG) old = dist[(uint64_t)v * 16u + l];
                    any = true;
                    n_active += n;
                    if (act) list[__popc(mask & ((1u << lane) - 1u))] = my;
                    __syncwarp();
                    for (uint32_t i = 0; i < n; i += 8u * kPer) {
                        if (n - i > 4u * kPer) merge_rows<LG, 8, kNoSat>(dist, list, i, n, sub, l, acc);
                        else if (n - i > kPer) merge_rows<LG, 4, kNoSat>(dist, list, i, n, sub, l, acc);
                        else merge_rows<LG, 1, kNoSat>(dist, list, i, n, sub, l, acc);
                    }
                    __syncwarp();   // the list is read
                }
                b += 32u;
                if (b >= len) break;
                my = edge_at(e, b + lane, len);
                fw = bits_of(my, b + lane, len);
            }
            if (!any) continue;   // no in-edge from the frontier: nothing to merge or apply
#pragma unroll
            for (int o = LG; o < 32; o <<= 1) {   // over the lane groups
                acc.x = min(acc.x, __shfl_xor_sync(kFull, acc.x, o));
                acc.y = min(acc.y, __shfl_xor_sync(kFull, acc.y, o));
                acc.z = min(acc.z, __shfl_xor_sync(kFull, acc.z, o));
                acc.w = min(acc.w, __shfl_xor_sync(kFull, acc.w, o));
            }
            if (kDry) {
                changed_units += (acc.x == 0u && acc.y == 0u && acc.z == 0u && acc.w == 0u);   // keeps the loads live
                continue;
            }
            uint32_t four = 0u;   // my slots that improved
            if ((uint32_t)lane < LG) {
                four = ((acc.x < old.x ? 1u : 0u) | (acc.y < old.y ? 2u : 0u) | (acc.z < old.z ? 4u : 0u) |
                        (acc.w < old.w ? 8u : 0u)) & busy;
                if (split) {   // row split across units: combine with atomics
                    uint32_t* d = a.dist + (uint64_t)v * 64u + 4u * l;
                    if (four & 1u) atomicMin(d, acc.x);
                    if (four & 2u) atomicMin(d + 1, acc.y);
                    if (four & 4u) atomicMin(d + 2, acc.z);
                    if (four & 8u) atomicMin(d + 3, acc.w);
                } else if (four) {
                    reinterpret_cast<uint4*>(a.dist)[(uint64_t)v * 16u + l] =
                        make_uint4(four & 1u ? acc.x : old.x, four & 2u ? acc.y : old.y, four & 4u ? acc.z : old.z,
                                   four & 8u ? acc.w : old.w);
                }
            }
            const uint32_t lo = __reduce_or_sync(kFull, lane < 8 ? four << (4 * lane) : 0u);
            const uint32_t hi = LG > 8 ? __reduce_or_sync(kFull, lane >= 8 && lane < 16 ? four << (4 * lane - 32) : 0u) : 0u;
            if (lo | hi) {
                if (lane == 0) atomicOr(&a.frontier_next[v >> 5], 1u << (v & 31u));
                ++changed_units;
                imp_lo |= lo;
                imp_hi |= hi;
            }
        }
    }
    // block totals in shared memory; the block's last warp to finish issues
    // one global atomic per word (no barrier: early warps leave at once)
    if (lane == 0) {
        if (changed_units) atomicAdd(&s_changed, (unsigned long long)changed_units);
        if (n_active && a.active) atomicAdd(&s_active, n_active);
        if (imp_lo) atomicOr(&s_imp[0], imp_lo);
        if (imp_hi) atomicOr(&s_imp[1], imp_hi);
        __threadfence_block();
        const bool last = atomicAdd(&s_done, 1u) == (uint32_t)kMsWarps - 1u;
        if (last) {
            __threadfence_block();
            const unsigned long long c = atomicAdd(&s_changed, 0ull);
            if (c) atomicAdd(a.changed, c);
            if (a.active) {
                const unsigned long long na = atomicAdd(&s_active, 0ull);
                if (na) atomicAdd(a.active, na);
            }
            const uint32_t i0 = atomicOr(&s_imp[0], 0u), i1 = atomicOr(&s_imp[1], 0u);
            if (!kDry && a.slot_improved != nullptr) {
                if (i0) atomicOr(&a.slot_improved[0], i0);
                if (i1) atomicOr(&a.slot_improved[1], i1);
            }
        }
    }
}

template <int LG, bool kDry, bool kPacked, bool kNoSat>
__global__ void __launch_bounds__(kMsBlock, 4) k_msssp(const MsArgs a) {
    msssp_block<LG, kDry, kPacked, false, kNoSat>(a);
}

// Persistent form of a resident batched run: one cooperative launch runs
// supersteps until one improves nothing (or max_steps). Superstep t reads
// frontier F[t % 3], sets bits in F[(t + 1) % 3] and counts its changed
// units in changed[t % 4]; meanwhile every CTA clears its share of F[(t + 2)
// % 3], which superstep t - 1 read and superstep t + 1 writes, and block 0
// clears changed[(t + 2) % 4] (every CTA read the counter of superstep t - 2
// before it arrived at the barrier that ended superstep t - 1), so one grid
// barrier per superstep orders everything. The distances are updated in
// place, as in the launch-per-superstep form.
template <int LG, bool kNoSat>
__global__ void __launch_bounds__(kMsBlock, 4)
    k_msssp_loop(MsArgs a, uint32_t* f0, uint32_t* f1, uint32_t* f2, unsigned long long* changed, uint64_t words,
                 uint32_t max_steps, GridBar* bar, uint64_t timeout_ns, uint32_t force, uint32_t* err,
                 uint32_t* steps_out) {
    uint32_t* const F[3] = {f0, f1, f2};
    __shared__ uint32_t s_more;
    for (uint32_t t = 0; t < max_steps; ++t) {
        a.frontier_cur = F[t % 3];
        a.frontier_next = F[(t + 1) % 3];
        a.changed = changed + t % 4;
        uint32_t* const clear = F[(t + 2) % 3];
        for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words; i += (uint64_t)gridDim.x * blockDim.x)
            clear[i] = 0u;
        if (blockIdx.x == 0 && threadIdx.x == 0) changed[(t + 2) % 4] = 0ull;
        msssp_block<LG, false, false, true, kNoSat>(a);
        uint64_t arrived = (uint64_t)t * gridDim.x;
        if (!grid_barrier(bar, gridDim.x, arrived, timeout_ns, force != 0u, err)) return;
        if (threadIdx.x == 0) s_more = __ldcg(changed + t % 4) != 0ull ? 1u : 0u;
        __syncthreads();
        if (!s_more || t + 1 == max_steps) {
            if (blockIdx.x == 0 && threadIdx.x == 0) *steps_out = t + 1;
            return;
        }
    }
}

__global__ void k_msssp_init(uint32_t* dist, uint64_t n_vertices) {
    const uint64_t total = n_vertices * 64u;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < total; i += (uint64_t)gridDim.x * blockDim.x)
        dist[i] = kInf;
}

// slot s of vertex sources[s] starts at 0 and the source is on the frontier
__global__ void k_msssp_sources(uint32_t* dist, const uint32_t* sources, uint32_t n_sources, uint32_t* frontier) {
    for (uint32_t s = threadIdx.x; s < n_sources; s += blockDim.x) {
        dist[(uint64_t)sources[s] * 64u + s] = 0u;
        atomicOr(&frontier[sources[s] >> 5], 1u << (sources[s] & 31u));
    }
}

__global__ void k_popc(const uint32_t* bits, uint64_t words, unsigned long long* out) {
    unsigned long long c = 0;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < words; i += (uint64_t)gridDim.x * blockDim.x)
        c += __popc(bits[i]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(kFull, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
}

}  // namespace

cudaError_t launch_msssp(const MsArgs& a, bool dry, uint32_t grid, cudaStream_t s) {
    if (a.u_end <= a.u_begin) return cudaSuccess;
    return with_slot_lanes(~a.idle_mask, [&](auto lanes) {
        constexpr int LG = decltype(lanes)::value;
        auto go = [&](auto packed, auto nosat) {
            constexpr bool kP = decltype(packed)::value, kN = decltype(nosat)::value;
            if (dry) k_msssp<LG, true, kP, kN><<<grid, kMsBlock, 0, s>>>(a);
            else k_msssp<LG, false, kP, kN><<<grid, kMsBlock, 0, s>>>(a);
        };
        using Y = std::true_type;
        using N = std::false_type;
        if (a.packed) a.no_sat ? go(Y{}, Y{}) : go(Y{}, N{});
        else a.no_sat ? go(N{}, Y{}) : go(N{}, N{});
        return cudaGetLastError();
    });
}

cudaError_t launch_msssp_init(uint32_t* dist, uint64_t n_vertices, const uint32_t* sources, uint32_t n_sources,
                              uint32_t* frontier, cudaStream_t s) {
    k_msssp_init<<<1216, 256, 0, s>>>(dist, n_vertices);
    k_msssp_sources<<<1, 64, 0, s>>>(dist, sources, n_sources, frontier);
    return cudaGetLastError();
}

cudaError_t launch_popc(const uint32_t* bits, uint64_t words, unsigned long long* out, cudaStream_t s) {
    k_popc<<<608, 256, 0, s>>>(bits, words, out);
    return cudaGetLastError();
}

cudaError_t launch_msssp_loop(const MsArgs& a, uint32_t* const frontier[3], unsigned long long* changed,
                              uint64_t words, uint32_t max_steps, GridBar* bar, uint64_t timeout_ns, bool force,
                              uint32_t* err, uint32_t* steps_out, cudaStream_t s) {
    if (a.u_end <= a.u_begin || max_steps == 0 || a.packed) return cudaErrorInvalidValue;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    return with_slot_lanes(~a.idle_mask, [&](auto lanes) {
        constexpr int LG = decltype(lanes)::value;
        const void* fn = a.no_sat ? (const void*)k_msssp_loop<LG, true> : (const void*)k_msssp_loop<LG, false>;
        int per_sm = 0;
        const cudaError_t oe = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kMsBlock, 0);
        if (oe != cudaSuccess) return oe;
        const uint64_t resident = (uint64_t)sms * (uint64_t)per_sm;
        if (resident == 0) return cudaErrorNotSupported;
        const uint32_t grid = (uint32_t)std::min<uint64_t>(msssp_grid(a.u_end - a.u_begin), resident);
        MsArgs args = a;
        uint32_t* f0 = frontier[0];
        uint32_t* f1 = frontier[1];
        uint32_t* f2 = frontier[2];
        uint32_t fo = force ? 1u : 0u;
        void* params[] = {&args, &f0, &f1, &f2, &changed, &words, &max_steps, &bar, &timeout_ns, &fo, &err, &steps_out};
        return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kMsBlock), params, 0, s);
    });
}

uint32_t msssp_grid(uint64_t units) {
    const uint64_t warps = std::max<uint64_t>(1, units);
    const uint64_t blocks = (warps + (kMsBlock / 32) - 1) / (kMsBlock / 32);
    return (uint32_t)std::min<uint64_t>(blocks, 152ull * 8);
}

}  // namespace gxp
