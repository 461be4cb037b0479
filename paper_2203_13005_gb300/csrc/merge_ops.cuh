// The algorithm template's operators (Section IV-A1: MSGGen, MSGMerge) and
// the warp helpers shared by the superstep kernels (sweep.cu: one partition,
// sell.cu: several, superstep.cu: a CSC in the caller's memory).
#pragma once

#include "gxp_internal.hpp"

namespace gxp {

template <Algo A> struct Ops;

template <> struct Ops<Algo::SSSP> {
    using T = uint32_t;
    static constexpr bool kWeighted = true;
    __device__ static T ident() { return kInf; }
    __device__ static T combine(T a, T b) { return min(a, b); }
    __device__ static T from_bits(uint32_t x) { return x; }
    __device__ static uint32_t to_bits(T x) { return x; }
    // MSGGen: relax; unreachable sources send nothing.
    __device__ static T gen(uint32_t du, uint32_t w) {
        if (du == kInf) return kInf;
        uint32_t s = du + w;
        if (s < du || s == kInf) s = kInf - 1u;   // saturate below INF
        return s;
    }
};

template <> struct Ops<Algo::CC> {
    using T = uint32_t;
    static constexpr bool kWeighted = false;
    __device__ static T ident() { return kInf; }
    __device__ static T combine(T a, T b) { return min(a, b); }
    __device__ static T from_bits(uint32_t x) { return x; }
    __device__ static uint32_t to_bits(T x) { return x; }
    __device__ static T gen(uint32_t lu, uint32_t) { return lu; }
};

template <> struct Ops<Algo::PR> {
    using T = float;
    static constexpr bool kWeighted = false;
    __device__ static T ident() { return 0.0f; }
    __device__ static T combine(T a, T b) { return a + b; }
    __device__ static T from_bits(uint32_t x) { return __uint_as_float(x); }
    __device__ static uint32_t to_bits(T x) { return __float_as_uint(x); }
    // The message array already holds r[u] / outdeg(u) (written by Apply).
    __device__ static T gen(uint32_t cu, uint32_t) { return __uint_as_float(cu); }
};

// Loads of the edge stream (source ids, weights): each word is read once per
// superstep, so evict-first.
__device__ __forceinline__ uint32_t ld_stream(const uint32_t* p) { return __ldcs(p); }
__device__ __forceinline__ uint4 ld_stream4(const uint4* p) { return __ldcs(p); }

// acq_rel arrival: orders this thread's earlier writes before the count
// becomes visible, and makes earlier arrivals' writes visible to the last.
__device__ __forceinline__ uint32_t arrive_acq_rel(uint32_t* ctr) {
    uint32_t old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(ctr) : "memory");
    return old;
}

template <class Op>
__device__ __forceinline__ typename Op::T warp_all(typename Op::T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = Op::combine(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}

// Exact warp sum of 64-bit values below 2^62 (the fixed-point sums and
// counts): three 27-bit limbs, each summed by one warp reduction.
__device__ __forceinline__ unsigned long long warp_sum_u62(unsigned long long x) {
    const uint32_t a0 = (uint32_t)(x & 0x7FFFFFFull), a1 = (uint32_t)((x >> 27) & 0x7FFFFFFull),
                   a2 = (uint32_t)(x >> 54);
    return (unsigned long long)__reduce_add_sync(0xFFFFFFFFu, a0) +
           ((unsigned long long)__reduce_add_sync(0xFFFFFFFFu, a1) << 27) +
           ((unsigned long long)__reduce_add_sync(0xFFFFFFFFu, a2) << 54);
}

}  // namespace gxp
