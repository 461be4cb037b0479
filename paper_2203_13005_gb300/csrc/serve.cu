// Kernels of the query server: 64 query slots share every pass over the
// edges (continuous batching). A slot's arithmetic reads only its own column,
// in an order fixed by the edge order, so a query's result is bit-identical
// whether it runs alone or among others.
//
//  * SSSP slots use the batched Bellman-Ford superstep of msssp.cu (its
//    per-slot improvement flags tell the server when a query has converged).
//  * Personalized PageRank slots iterate
//        r_{t+1} = d * A^T D^-1 r_t + ((1 - d) + d * D_t) e_s
//    (Jacobi; D_t = rank mass on dangling vertices, returned to the source s
//    together with the teleport), with fp32 messages c = r * (1 / outdeg)
//    and exact fixed-point dangling sums per slot. A lane holds four slots
//    (128-bit loads), so LG lanes hold a row: 16 for 64 slots, fewer when
//    only the first slots hold queries; a warp works on 32 / LG units at once,
//    each summed in its own edge order, so a slot's result does not depend
//    on LG.
//      k_ppr_units   LG lanes per work unit (<= 256 in-edges of one vertex):
//                    sums the sources' message rows in edge order; a vertex
//                    held by one unit is applied at once, a vertex split
//                    over several units leaves one partial row per unit;
//      k_ppr_split   adds a split vertex's partials in unit order, applies.
//    Apply adds the source term, writes the next messages, and writes the
//    ranks only in a slot's last superstep (the result).
//  * Slot management: batched column initialisation and a row-tile transpose
//    that copies finished columns out as contiguous result vectors.
#include <algorithm>

#include "gxp_internal.hpp"

namespace gxp {
namespace {

constexpr int kSvBlock = 256;
constexpr int kSvWarps = kSvBlock / 32;
constexpr int kSvUnroll = 4;   // message rows in flight per lane
constexpr int kSvDeep = 8;     // and where few warps share the chip
// The lines between them, from bursts of n R-MAT vertices, 12 n edges:
//  * up to kDeepWarps warps a superstep, 8 rows in flight and the next ids read
//    ahead (3 CTAs an SM): 32 queries, n = 2^16, 17 K warps 3,152 us against
//    3,310, n = 2^17, 35 K warps 3,860 / 3,897, n = 2^18 5,114 / 4,659.
//  * lane groups are widened until a superstep has kFullWarps warps (16 an SM):
//    a query alone, n = 2^14: 754 us against 840; 32 an SM 738, 64 an SM 733,
//    but 32 queries, n = 2^15, 2,795 / 2,956 / 3,100 us.
constexpr uint64_t kDeepWarps = 152ull * 160;
constexpr uint64_t kFullWarps = 152ull * 16;
constexpr int kTileRows = 64;   // rows per transpose tile

uint32_t grid_for(uint64_t items, uint64_t per_block) {
    const uint64_t b = (items + per_block - 1) / per_block;
    return (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(b, 152ull * 8));
}

}  // namespace

// Grid of a serving superstep kernel: one warp per item up to 16 waves of
// 8 blocks per SM, so each block lives a fraction of the kernel and the
// block scheduler can interleave lanes of other graphs (higher-priority
// streams) at block boundaries instead of after the whole superstep.
uint32_t serve_grid(uint64_t items) {
    const uint64_t b = (items + kSvWarps - 1) / kSvWarps;
    return (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(b, 152ull * 8 * 16));
}

namespace {

// Per-slot constants of a PPR superstep, kept in shared memory so the
// gather loop keeps its registers for rows in flight: damping, source
// (kInf for an idle slot) and (1 - d) + d * D_t, D_t from the exact
// fixed-point sum of the slot's dangling mass.
struct PprSlots {
    float4 d[16], add[16];
    uint4 src[16];
    unsigned long long dang[64];   // this block's dangling mass of r_{t+1}
    uint32_t warps_done;

    __device__ void init(const PprArgs& a) {
        const int s = threadIdx.x;
        if (s < 64) {
            const bool busy = (a.active_mask >> s) & 1ull;
            const float d_s = a.slot_damping[s];
            reinterpret_cast<float*>(d)[s] = d_s;
            reinterpret_cast<float*>(add)[s] =
                busy ? (float)((1.0 - (double)d_s) + (double)d_s * fx_to_double(a.dang_cur[s])) : 0.0f;
            reinterpret_cast<uint32_t*>(src)[s] = busy ? a.slot_source[s] : kInf;
            dang[s] = 0ull;
        }
        if (threadIdx.x == 0) warps_done = 0u;
        __syncthreads();
    }

    // MSGApply of vertex v (1 / out-degree inv, 0 if dangling) for lane l's
    // slots with merged sum: r = d * sum, plus the source term at the slot's
    // source; message r * inv; ranks only in a slot's last superstep. Rounded
    // operation by operation, so that every lane grouping gives the same bits.
    __device__ void apply(const PprArgs& a, uint32_t v, float inv, float4 sum, uint32_t l) {
        const float4 dl = d[l];
        const uint4 sl = src[l];
        float4 r = make_float4(__fmul_rn(dl.x, sum.x), __fmul_rn(dl.y, sum.y), __fmul_rn(dl.z, sum.z),
                               __fmul_rn(dl.w, sum.w));
        if (v == sl.x || v == sl.y || v == sl.z || v == sl.w) {
            const float4 al = add[l];
            if (v == sl.x) r.x = __fadd_rn(r.x, al.x);
            if (v == sl.y) r.y = __fadd_rn(r.y, al.y);
            if (v == sl.z) r.z = __fadd_rn(r.z, al.z);
            if (v == sl.w) r.w = __fadd_rn(r.w, al.w);
        }
        reinterpret_cast<float4*>(a.msg_nxt)[(uint64_t)v * 16u + l] =
            make_float4(r.x * inv, r.y * inv, r.z * inv, r.w * inv);
        if ((a.finish_mask >> (4 * l)) & 15ull) reinterpret_cast<float4*>(a.rank)[(uint64_t)v * 16u + l] = r;
        if (inv == 0.0f) {
            if (r.x != 0.0f) atomicAdd(&dang[4 * l], fx_of(r.x));
            if (r.y != 0.0f) atomicAdd(&dang[4 * l + 1], fx_of(r.y));
            if (r.z != 0.0f) atomicAdd(&dang[4 * l + 2], fx_of(r.z));
            if (r.w != 0.0f) atomicAdd(&dang[4 * l + 3], fx_of(r.w));
        }
    }

    // the block's dangling sums -> one global atomic per slot, issued by the
    // block's last warp to finish (no barrier: early warps leave at once)
    __device__ void flush(unsigned long long* out) {
        __syncwarp();
        const int lane = threadIdx.x & 31;
        uint32_t last = 0u;
        if (lane == 0) {
            __threadfence_block();
            last = atomicAdd(&warps_done, 1u) == (blockDim.x >> 5) - 1u ? 1u : 0u;
        }
        if (!__shfl_sync(0xFFFFFFFFu, last, 0)) return;
        __threadfence_block();
        for (int i = lane; i < 64; i += 32) {
            const unsigned long long v = atomicAdd(&dang[i], 0ull);
            if (v) atomicAdd(&out[i], v);
        }
    }
};

// LG lanes per work unit, 32 / LG units per warp (neighbours in the units'
// order, which have about the same length); lanes without a busy slot skip
// every load and store. U source ids are read at a time (a broadcast load
// within the lane group), then their message rows are in flight together; the
// sum runs in edge order. What bounds it: the L2 bandwidth of the rows with all
// slots in use; on small graphs the chain of a unit's 256 edges (a query alone
// on 2^14 vertices: 33 us a launch with a unit a warp and 8 rows in flight,
// 64 us with 4 rows and 32 units a warp). 32 queries on
// each of three graphs (8.4, 2.1 and 0.5 M edges, ~22 supersteps each): 10.9 ms
// in this kernel with a unit per warp and two slots a lane whatever the slots
// in use, 4.8 ms so (4 rows in flight and 6 CTAs an SM; 8 rows and 3 / 4 CTAs
// 5.2 / 4.5 ms, 4 rows and 8 CTAs 5.5 ms, the whole burst 13.8 / 13.9 / 12.6
// against 12.8 ms).
template <int LG, int U, int kCtas>
__global__ void __launch_bounds__(kSvBlock, kCtas) k_ppr_units(const PprArgs a) {
    constexpr uint32_t kPer = 32 / LG;
    __shared__ PprSlots sl;
    sl.init(a);
    const uint32_t lane = threadIdx.x & 31u, l = lane % LG, sub = lane / LG;
    const bool live = (a.active_mask >> (4 * l)) & 15ull;
    const float4* msg = reinterpret_cast<const float4*>(a.msg_cur);
    // With up to four slots a warp holds many units and the longest are few
    // warps: those go to a CTA each (a query alone, n = 2^19 R-MAT vertices:
    // 3,100 us against 3,516). With more slots neighbouring units stay together
    // (32 queries there: 6,437 us against 7,692).
    const uint32_t warp = threadIdx.x >> 5;
    const uint64_t warp0 = a.active_mask >> 4 ? (uint64_t)blockIdx.x * kSvWarps + warp
                                              : (uint64_t)warp * gridDim.x + blockIdx.x;
    const uint64_t n_warps = ((uint64_t)gridDim.x * kSvBlock) >> 5;
    for (uint64_t k0 = warp0 * kPer; k0 < a.n_units; k0 += n_warps * kPer) {
        const bool has = k0 + sub < a.n_units;
        const uint4 un = has ? a.units[k0 + sub] : make_uint4(0u, 0u, 0u, 0u);   // dst, first edge, edges, partial + 1 | 0
        const float inv = __ldg(a.inv_outdeg + un.x);
        const uint32_t* e = a.src + un.y;
        float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        uint32_t u[U], next[U];
#pragma unroll
        for (int q = 0; q < U; ++q) u[q] = q < un.z ? __ldg(e + q) : kInf;
        for (uint32_t i = 0; i < un.z; i += U) {
            if (U > kSvUnroll) {   // the next ids on their way with these rows
#pragma unroll
                for (int q = 0; q < U; ++q) next[q] = i + U + q < un.z ? __ldg(e + i + U + q) : kInf;
            }
            float4 m[U];
#pragma unroll
            for (int q = 0; q < U; ++q)
                m[q] = (u[q] != kInf && live) ? msg[(uint64_t)u[q] * 16u + l] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
            for (int q = 0; q < U; ++q) {   // (an absent edge adds zero)
                acc.x += m[q].x;
                acc.y += m[q].y;
                acc.z += m[q].z;
                acc.w += m[q].w;
            }
#pragma unroll
            for (int q = 0; q < U; ++q)
                u[q] = U > kSvUnroll ? next[q] : (i + U + q < un.z ? __ldg(e + i + U + q) : kInf);
        }
        if (!live || !has) continue;
        if (un.w) reinterpret_cast<float4*>(a.partial)[(uint64_t)(un.w - 1u) * 16u + l] = acc;
        else sl.apply(a, un.x, inv, acc, l);
    }
    sl.flush(a.dang_next);
}

// LG lanes per vertex split over several units: its partial rows added in
// unit order (eight in flight), applied.
template <int LG>
__global__ void __launch_bounds__(kSvBlock, 4) k_ppr_split(const PprArgs a) {
    constexpr uint32_t kPer = 32 / LG;
    __shared__ PprSlots sl;
    sl.init(a);
    const uint32_t lane = threadIdx.x & 31u, l = lane % LG, sub = lane / LG;
    const bool live = (a.active_mask >> (4 * l)) & 15ull;
    const float4* part = reinterpret_cast<const float4*>(a.partial);
    const uint32_t warp0 = (blockIdx.x * kSvBlock + threadIdx.x) >> 5;
    const uint32_t n_warps = (gridDim.x * kSvBlock) >> 5;
    for (uint64_t r = (uint64_t)warp0 * kPer + sub; r < a.n_split_rows && live; r += (uint64_t)n_warps * kPer) {
        const uint2 sr = a.split_rows[r];   // {vertex, first partial}
        const uint32_t end = a.split_rows[r + 1].y;
        float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        for (uint32_t p = sr.y; p < end; p += 8u) {   // unit order
            float4 x[8];
#pragma unroll
            for (uint32_t q = 0; q < 8; ++q)
                x[q] = p + q < end ? part[(uint64_t)(p + q) * 16u + l] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
            for (uint32_t q = 0; q < 8; ++q) {
                acc.x += x[q].x;
                acc.y += x[q].y;
                acc.z += x[q].z;
                acc.w += x[q].w;
            }
        }
        sl.apply(a, sr.x, __ldg(a.inv_outdeg + sr.x), acc, l);
    }
    sl.flush(a.dang_next);
}

// thread (v, l): slots 2l and 2l+1 of row v, where they are in `mask`:
// messages of r_0 = e_src (the ranks are written by the slot's last superstep)
__global__ void k_ppr_slots_init(float* msg_cur, const float* inv_outdeg, uint64_t n, uint64_t mask,
                                 const uint32_t* slot_source, unsigned long long* dang_cur) {
    const uint64_t total = n * 32u;
    if (blockIdx.x == 0 && threadIdx.x < 64 && ((mask >> threadIdx.x) & 1ull)) {
        const uint32_t src = slot_source[threadIdx.x];
        dang_cur[threadIdx.x] = inv_outdeg[src] == 0.0f ? fx_of(1.0f) : 0ull;
    }
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t v = i >> 5;
        const uint32_t l = (uint32_t)(i & 31u);
        const uint32_t pair = (uint32_t)(mask >> (2u * l)) & 3u;
        if (!pair) continue;
        const float inv = __ldg(inv_outdeg + v);
#pragma unroll
        for (uint32_t b = 0; b < 2; ++b)
            if ((pair >> b) & 1u) msg_cur[v * 64u + 2u * l + b] = v == slot_source[2u * l + b] ? inv : 0.0f;
    }
}

__global__ void k_sssp_slots_init(uint32_t* dist, uint64_t n, uint64_t mask, const uint32_t* slot_source,
                                  uint32_t* frontier) {
    const uint64_t total = n * 32u;
    if (blockIdx.x == 0 && threadIdx.x < 64 && ((mask >> threadIdx.x) & 1ull)) {
        const uint32_t src = slot_source[threadIdx.x];
        atomicOr(&frontier[src >> 5], 1u << (src & 31u));
    }
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t v = i >> 5;
        const uint32_t l = (uint32_t)(i & 31u);
        const uint32_t pair = (uint32_t)(mask >> (2u * l)) & 3u;
        if (!pair) continue;
#pragma unroll
        for (uint32_t b = 0; b < 2; ++b)
            if ((pair >> b) & 1u) dist[v * 64u + 2u * l + b] = v == slot_source[2u * l + b] ? 0u : kInf;
    }
}

// 64-row tiles of mat[V][64] through shared memory: coalesced row reads,
// then one coalesced 256-byte run per listed column
__global__ void __launch_bounds__(kSvBlock) k_gather_columns(const uint32_t* mat, uint64_t n, GatherList list) {
    __shared__ uint32_t tile[kTileRows][65];
    __shared__ uint32_t s_slot[64];
    __shared__ uint32_t* s_out[64];
    if (threadIdx.x < list.n) {
        s_slot[threadIdx.x] = list.slot[threadIdx.x];
        s_out[threadIdx.x] = list.out[threadIdx.x];
    }
    const uint64_t n_tiles = (n + kTileRows - 1) / kTileRows;
    for (uint64_t t = blockIdx.x; t < n_tiles; t += gridDim.x) {
        const uint64_t v0 = t * kTileRows;
        const uint32_t rows = n - v0 < (uint64_t)kTileRows ? (uint32_t)(n - v0) : (uint32_t)kTileRows;
        __syncthreads();   // previous tile fully written out
        for (uint32_t i = threadIdx.x; i < rows * 64u; i += kSvBlock) tile[i >> 6][i & 63u] = mat[v0 * 64u + i];
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < list.n * (uint32_t)kTileRows; i += kSvBlock) {
            const uint32_t j = i / kTileRows, r = i % kTileRows;
            if (r < rows) s_out[j][v0 + r] = tile[r][s_slot[j]];
        }
    }
}

}  // namespace

cudaError_t launch_ppr_superstep(const PprArgs& a, cudaStream_t s) {
    uint64_t lanes_mask = a.active_mask;   // (LG lanes for the highest set slot)
    for (uint32_t lg = 1; lg < 16u; lg *= 2)
        if (a.n_units * lg < 32u * kFullWarps) lanes_mask |= 1ull << (4u * lg);
    return with_slot_lanes(lanes_mask, [&](auto lanes) {
        constexpr int LG = decltype(lanes)::value;
        constexpr uint64_t kPer = 32 / LG;
        const uint64_t warps = (a.n_units + kPer - 1) / kPer;
        if (warps <= kDeepWarps) k_ppr_units<LG, kSvDeep, 3><<<serve_grid(warps), kSvBlock, 0, s>>>(a);
        else k_ppr_units<LG, kSvUnroll, 6><<<serve_grid(warps), kSvBlock, 0, s>>>(a);
        if (a.n_split_rows)
            k_ppr_split<LG><<<serve_grid((a.n_split_rows + kPer - 1) / kPer), kSvBlock, 0, s>>>(a);
        return cudaGetLastError();
    });
}

cudaError_t launch_ppr_slots_init(float* msg_cur, const float* inv_outdeg, uint64_t n, uint64_t mask,
                                  const uint32_t* slot_source, unsigned long long* dang_cur, cudaStream_t s) {
    if (!mask) return cudaSuccess;
    k_ppr_slots_init<<<grid_for(n * 32u, kSvBlock), kSvBlock, 0, s>>>(msg_cur, inv_outdeg, n, mask, slot_source,
                                                                      dang_cur);
    return cudaGetLastError();
}

cudaError_t launch_sssp_slots_init(uint32_t* dist, uint64_t n, uint64_t mask, const uint32_t* slot_source,
                                   uint32_t* frontier, cudaStream_t s) {
    if (!mask) return cudaSuccess;
    k_sssp_slots_init<<<grid_for(n * 32u, kSvBlock), kSvBlock, 0, s>>>(dist, n, mask, slot_source, frontier);
    return cudaGetLastError();
}

cudaError_t launch_gather_columns(const uint32_t* mat, uint64_t n, const GatherList& list, cudaStream_t s) {
    if (list.n == 0 || n == 0) return cudaSuccess;
    k_gather_columns<<<grid_for((n + kTileRows - 1) / kTileRows, 1), kSvBlock, 0, s>>>(mat, n, list);
    return cudaGetLastError();
}

}  // namespace gxp
