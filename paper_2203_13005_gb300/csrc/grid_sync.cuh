// Grid-wide barrier with a bounded wait, of launches all of whose CTAs are on
// the device: a cooperative one (msssp.cu), or one whose CTAs have met at it
// before anything was done (sweep.cu).
#pragma once

#include "gxp_internal.hpp"

namespace gxp {

__device__ __forceinline__ unsigned long long ld_relaxed_gpu(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_gpu(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void fence_acq_rel_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Barrier of all CTAs of a grid: an arrival counter that only grows. `arrived`
// is the caller's count of the arrivals there are once every CTA has passed
// the barriers before: 0 at first in a launch whose counter was zeroed
// (msssp.cu), the counter's value where it is carried from launch to launch
// (sweep.cu). A CTA's arrival is a fire-and-forget add
// and every CTA polls the counter itself, so a barrier costs a fence, the
// add's and the last poll's way to L2: with a generation word to read,
// release and poll, and an error word to read after it, a barrier and the
// superstep's other fixed costs took 10 us (20 supersteps of no work items,
// 152 CTAs). A wait that runs past timeout_ns (or any wait when
// `force`, an injected fault) sets kErrTimeout and the counter's top bit and
// gives up. Returns false when this CTA gave up or saw that another one had;
// the caller then returns.
// kMeet: a barrier before which nothing was done. A wait gives up only while an
// arrival is missing, so that either every CTA passes or none, and it is no
// error (but for an injected one).
constexpr unsigned long long kBarGaveUp = 1ull << 63;
template <bool kMeet = false>
__device__ inline bool grid_barrier(GridBar* b, uint32_t n_ctas, uint64_t& arrived, uint64_t timeout_ns, bool force,
                                    uint32_t* err) {
    __shared__ uint32_t s_ok;
    arrived += n_ctas;
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned long long all = arrived;
        fence_acq_rel_gpu();
        atomicAdd(&b->count, 1ull);   // result unused: a reduction
        unsigned long long c = ld_relaxed_gpu(&b->count);
        if (c < all) {
            const uint64_t t0 = global_ns();
            while ((c = ld_relaxed_gpu(&b->count)) < all) {   // the top bit ends every wait
                if (force || global_ns() - t0 > timeout_ns) {
                    if (kMeet && atomicCAS(&b->count, c, c | kBarGaveUp) != c) continue;   // another arrival
                    if (!kMeet || force) atomicOr(err, kErrTimeout);
                    c = kBarGaveUp;
                    if (!kMeet) atomicOr(&b->count, kBarGaveUp);
                    break;
                }
            }
        }
        fence_acq_rel_gpu();
        s_ok = (c & kBarGaveUp) ? 0u : 1u;
    }
    __syncthreads();
    return s_ok != 0u;
}

}  // namespace gxp
