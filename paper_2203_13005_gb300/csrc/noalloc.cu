// gxp_superstep_min_noalloc: one SSSP or CC superstep over a CSC held in the
// caller's device memory, using no device allocation at all.
//
// Who needs it: callers that cannot call cudaMalloc — e.g. code whose device
// memory is entirely owned by another allocator (a framework's caching pool
// that has reserved the GPU), or latency-sensitive callers that cannot accept
// cudaMalloc's implicit device-wide synchronisation. The regular path
// (gxp_init / gxp_load_partition) allocates its own buffers; this entry point
// instead takes every input and output from the caller and keeps its
// internal scratch (edge-block descriptors, hub partials and counters, the
// changed counts and the error words) in one fixed-size file-scope
// __device__ array.
//
// The array is a property of the loaded library: every GPU that loads it
// holds kNoAllocScratchBytes of device memory until the process exits. All
// calls on a device share the array and it keeps the last call's contents;
// the regions that must start at zero are cleared on every call. Calls that
// overlap on the GPU (e.g. issued to different streams without ordering) race
// on the array and must not be made.
#include <algorithm>
#include <mutex>

#include "fault.hpp"
#include "gxp_internal.hpp"

namespace gxp {
namespace {

// Merge items (4 per vertex end, 1 per edge) of an edge block, a warp's work
// unit: 2048 on large inputs, fewer on small ones so that the blocks spread
// over ~32 warps an SM (R-MAT 12, 82 K items: 40 blocks of 2048 kept 40 warps of
// the chip busy). Rows of more than a quarter of that are split.
constexpr uint32_t kNoAllocMaxItems = 2048, kNoAllocMinItems = 64;
constexpr uint64_t kNoAllocMaxTiles = 131072;   // 4 * n_vertices + n_edges <= 2^28
constexpr uint64_t kHeaderBytes = 4096;
constexpr uint64_t kNoAllocScratchBytes =
    kHeaderBytes + kNoAllocMaxTiles * (4 + 4 + 4 + sizeof(Tile));

// Header: [kStatLanes] changed counts, then two error words. A call uses one
// and zeroes the other for the call after it, so no operation has to clear
// the error word before the checks run.
struct NoAllocHeader {
    unsigned long long changed[kStatLanes];
    uint32_t err[2];
};
static_assert(sizeof(NoAllocHeader) <= kHeaderBytes, "header too small");

// The scratch. Host code must not take its address directly (that would be a
// host-side stand-in); it asks the runtime for the device address once per
// device.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

std::mutex g_mu;
constexpr int kMaxDevices = 64;
struct Device {
    unsigned char* scratch = nullptr;
    uint32_t sms = 0;
    uint32_t turn = 0;   // which error word the next call uses
};
Device g_device[kMaxDevices];

struct Layout {
    NoAllocHeader* head;
    uint32_t* hub_cnt;
    uint32_t* part_head;
    uint32_t* part_tail;
    Tile* tiles;
};

Layout layout_of(unsigned char* base) {
    Layout L;
    L.head = reinterpret_cast<NoAllocHeader*>(base);
    unsigned char* p = base + kHeaderBytes;
    L.hub_cnt = reinterpret_cast<uint32_t*>(p);
    p += 4 * kNoAllocMaxTiles;
    L.part_head = reinterpret_cast<uint32_t*>(p);
    p += 4 * kNoAllocMaxTiles;
    L.part_tail = reinterpret_cast<uint32_t*>(p);
    p += 4 * kNoAllocMaxTiles;
    L.tiles = reinterpret_cast<Tile*>(p);
    return L;
}

// The current device's entry, its scratch address and SM count looked up on
// first use.
gxp_status current_device(Device** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return GXP_E_CUDA;
    std::lock_guard<std::mutex> lk(g_mu);
    Device& d = g_device[dev];
    if (!d.scratch) {
        void* ptr = nullptr;
        int sms = 0;
        if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || ptr == nullptr ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
            cudaGetLastError();
            return GXP_E_CUDA;
        }
        d.sms = (uint32_t)sms;
        d.scratch = static_cast<unsigned char*>(ptr);
    }
    *out = &d;
    return GXP_OK;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

bool overlap(const void* a, const void* b, size_t bytes) {
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return x < y + bytes && y < x + bytes;
}

// ------------------------------------------------------------ preparation

// Merge-path cut k: the number of vertex ends and edges among the first k T
// weighted items (a vertex end weighs kVertexCost, an edge one), moved back to
// before the end of the vertex it falls in, and to that vertex's start unless
// it is a hub (in-degree > H). 16 lanes search together (a 16-ary search: 3 to
// 6 dependent loads where halving takes 12 to 24); `lane` is in 0..15, `mask`
// those 16 lanes. Any offsets keep every access inside col_ptr[0..n].
__device__ __forceinline__ void merge_cut(const uint32_t* __restrict__ col_ptr, uint32_t n, uint32_t n_edges,
                                          uint64_t D, uint32_t H, uint32_t lane, unsigned mask, uint32_t& vi,
                                          uint32_t& ej) {
    // largest i in [0, n] with i * cost + col_ptr[i] <= D
    uint32_t lo = 0, hi = n;
    while (lo < hi) {
        const uint32_t step = (hi - lo + 15u) / 16u;
        const uint64_t at = (uint64_t)lo + (uint64_t)(lane + 1u) * step;   // probes in (lo, hi]
        const uint32_t p = (uint32_t)min(at, (uint64_t)hi);
        const bool le = (uint64_t)p * kVertexCost + __ldg(col_ptr + p) <= D;
        const unsigned b = __ballot_sync(mask, le) & mask;
        const unsigned r = mask == 0xFFFFu ? b : b >> 16;
        const uint32_t c = (uint32_t)__popc(r);   // probes at or below D (offsets that decrease are refused)
        const uint64_t nlo = (uint64_t)lo + (uint64_t)c * step;
        const uint64_t nhi = (uint64_t)lo + (uint64_t)(c + 1u) * step - 1u;
        hi = c == 16u ? hi : (uint32_t)min(nhi, (uint64_t)hi);
        lo = (uint32_t)min(nlo, (uint64_t)hi);
        if (c == 16u) lo = hi;
    }
    uint64_t j = D - (uint64_t)lo * kVertexCost;
    if (lo < n) {
        const uint32_t c0 = __ldg(col_ptr + lo), c1 = __ldg(col_ptr + lo + 1);
        if (j > c1) j = c1;   // inside the vertex's end item: cut before it
        if (j > c0 && c1 - c0 <= H) j = c0;
    }
    vi = lo;
    ej = (uint32_t)min(j, (uint64_t)n_edges);
}

// One pass before the superstep: the CSC checked (offsets from 0 to n_edges
// without decreasing: kErrInput; sources below n: kErrBounds), the edge
// blocks cut (a warp per block, its two cuts by half a warp each), the
// arrival counters and the counts zeroed. A block's cuts follow from its
// number alone, so no array of cuts is written and searched. The superstep
// kernel, next in the stream, does nothing when the error word is set.
__global__ void __launch_bounds__(256) k_prepare(const uint32_t* __restrict__ col_ptr, uint32_t n,
                                                 const uint32_t* __restrict__ src, uint32_t n_edges, uint32_t T,
                                                 uint32_t H, uint32_t nt, Tile* __restrict__ tiles,
                                                 uint32_t* __restrict__ hub_cnt, NoAllocHeader* head, uint32_t turn) {
    const uint32_t t0 = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
    if (blockIdx.x == 0) {
        if (threadIdx.x < kStatLanes) head->changed[threadIdx.x] = 0ull;
        if (threadIdx.x == 0) head->err[turn ^ 1u] = 0u;
    }
    uint32_t bad = 0;
    if (t0 == 0 && (col_ptr[0] != 0u || col_ptr[n] != n_edges)) bad |= kErrInput;
    for (uint64_t v = t0; v < n; v += stride)
        if (col_ptr[v] > col_ptr[v + 1]) bad |= kErrInput;
    const uint4* src4 = reinterpret_cast<const uint4*>(src);   // 16-byte aligned (checked by the host)
    for (uint64_t e = t0; e < n_edges / 4u; e += stride) {
        const uint4 u = __ldg(src4 + e);
        if (u.x >= n || u.y >= n || u.z >= n || u.w >= n) bad |= kErrBounds;
    }
    for (uint64_t e = (n_edges & ~3u) + (uint64_t)t0; e < n_edges; e += stride)
        if (__ldg(src + e) >= n) bad |= kErrBounds;
    bad = __reduce_or_sync(0xFFFFFFFFu, bad);
    const uint32_t lane = threadIdx.x & 31u;
    if (bad && lane == 0) atomicOr(&head->err[turn], bad);

    const uint64_t total = (uint64_t)n * kVertexCost + n_edges;
    for (uint32_t k = t0 >> 5; k < nt; k += stride >> 5) {
        const uint32_t half = lane >> 4;   // lanes 0..15: cut k, lanes 16..31: cut k + 1
        uint32_t vi, ej;
        merge_cut(col_ptr, n, n_edges, min((uint64_t)(k + half) * T, total), H, lane & 15u,
                  half ? 0xFFFF0000u : 0xFFFFu, vi, ej);
        __syncwarp();
        const uint32_t i0 = __shfl_sync(0xFFFFFFFFu, vi, 0), j0 = __shfl_sync(0xFFFFFFFFu, ej, 0);
        const uint32_t i1 = __shfl_sync(0xFFFFFFFFu, vi, 16), j1 = __shfl_sync(0xFFFFFFFFu, ej, 16);
        if (lane != 0) continue;
        const bool is_head = i0 < n && j0 > col_ptr[i0];
        const bool is_tail = i1 < n && j1 > col_ptr[i1];
        Tile t;
        t.v0 = i0;
        t.nv = i1 - i0 + (is_tail ? 1u : 0u);
        t.e0 = j0;
        t.ne = j1 - j0;
        t.part = 0u;
        t.flags = (is_head ? kHeadOpen : 0u) | (is_tail ? kTailOpen : 0u);
        t.hub_t0 = kInf;
        t.nparts = 0;
        if (t.nv == 0u && t.ne == 0u) t.flags = 0u;
        // A hub's cuts are not moved back to its start: the block where it
        // starts is the one its first item falls in, and its last part ends at
        // the first cut past its end item.
        if (is_head) t.hub_t0 = (uint32_t)(((uint64_t)i0 * kVertexCost + col_ptr[i0]) / T);
        if (is_tail && !(is_head && t.nv == 1u)) {
            const uint64_t past = (uint64_t)(i1 + 1u) * kVertexCost + col_ptr[i1 + 1];
            t.nparts = (uint32_t)((past + T - 1) / T) - 1u - k + 1u;
        }
        tiles[k] = t;
        hub_cnt[k] = 0u;
    }
}

}  // namespace
}  // namespace gxp

extern "C" GXP_API gxp_status gxp_superstep_min_noalloc(gxp_algo algo, uint32_t n_vertices, uint64_t n_edges,
                                                        const uint32_t* d_col_ptr, const uint32_t* d_src,
                                                        const uint32_t* d_w, const uint32_t* d_cur,
                                                        uint32_t* d_next, uint64_t* n_changed, void* stream) {
    using namespace gxp;
    if (algo != GXP_ALGO_SSSP && algo != GXP_ALGO_CC) return GXP_E_UNSUPPORTED;
    if (n_vertices == 0 || n_vertices >= 0xFFFFFFFFu || n_edges > 0xFFFFFFFFull) return GXP_E_INVAL;
    if (!d_col_ptr || !d_cur || !d_next || (n_edges && !d_src) || (algo == GXP_ALGO_SSSP && n_edges && !d_w))
        return GXP_E_INVAL;
    if (!aligned16(d_col_ptr) || !aligned16(d_cur) || (d_src && !aligned16(d_src)) || (d_w && !aligned16(d_w)))
        return GXP_E_INVAL;
    if (overlap(d_cur, d_next, 4ull * n_vertices)) return GXP_E_INVAL;   // Jacobi: two distinct buffers
    const uint64_t items = (uint64_t)n_vertices * kVertexCost + n_edges;
    if ((items + kNoAllocMaxItems - 1) / kNoAllocMaxItems > kNoAllocMaxTiles)
        return GXP_E_INVAL;   // beyond the scratch's fixed size
    Device* dev = nullptr;
    const gxp_status st = current_device(&dev);
    if (st != GXP_OK) return st;
    uint32_t T = kNoAllocMinItems;
    while (T < kNoAllocMaxItems && (uint64_t)T * 32 * dev->sms < items) T *= 2;
    const uint32_t n_tiles = (uint32_t)((items + T - 1) / T);
    if ((uint64_t)n_tiles > kNoAllocMaxTiles) return GXP_E_INVAL;
    const Layout L = layout_of(dev->scratch);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const Algo a = algo == GXP_ALGO_SSSP ? Algo::SSSP : Algo::CC;

    // The tiles are cut from the offsets and the superstep kernel stages them
    // with bulk copies sized from those cuts: it runs only on a CSC that
    // passed k_prepare's checks.
    const uint64_t warps = std::max<uint64_t>(n_tiles, std::max<uint64_t>(n_edges / 4, n_vertices) / 32);
    const uint32_t grid = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>((warps + 7) / 8, 8ull * dev->sms));
    uint32_t turn;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        turn = dev->turn;
        k_prepare<<<grid, 256, 0, s>>>(d_col_ptr, n_vertices, d_src, (uint32_t)n_edges, T, T / 4, n_tiles, L.tiles,
                                       L.hub_cnt, L.head, turn);
        if (cudaGetLastError() != cudaSuccess) return GXP_E_CUDA;
        dev->turn ^= 1u;   // the launch zeroes the other error word
    }
    SuperstepArgs args{};
    args.tiles = L.tiles;
    args.part = PartDev{d_col_ptr, d_src, algo == GXP_ALGO_SSSP ? d_w : nullptr, n_vertices, 0u, 0u, 0u, n_edges};
    args.n_tiles = n_tiles;
    args.own_cur = d_cur;
    args.own_nxt = d_next;
    args.part_head = L.part_head;
    args.part_tail = L.part_tail;
    args.hub_cnt = L.hub_cnt;
    args.changed = L.head->changed;
    args.err = &L.head->err[turn];
    args.timeout_ns = 2000000000ull;
    args.force_timeout = fault_plan_from_env().timeout ? 1u : 0u;
    args.max_items = T + T / 4;
    if (launch_superstep(a, args, dev->sms, s) != cudaSuccess) return GXP_E_CUDA;

    NoAllocHeader host;
    if (cudaMemcpyAsync(&host, L.head, sizeof(host), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return GXP_E_CUDA;
    const uint32_t err = host.err[turn];
    if (err & kErrInput) return GXP_E_INVAL;
    if (err & (kErrTimeout | kErrDrain)) return GXP_E_TIMEOUT;
    if (err & kErrBounds) return GXP_E_BOUNDS;
    if (n_changed) {
        unsigned long long c = 0;
        for (int i = 0; i < kStatLanes; ++i) c += host.changed[i];
        *n_changed = c;
    }
    return GXP_OK;
}
