// Device primitives for the ACRL kernels (sm_103a): streaming 16-byte loads
// and stores with cache hints, bf16 unpacking, the hardware base-2
// exponential, and deterministic warp/CTA reductions.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "acrl.h"

namespace acrl {

constexpr float kLog2e = 1.4426950408889634f;   // 1 / ln 2
constexpr float kLn2 = 0.6931471805599453f;

// The first thing every kernel of the path does (see `launch`): wait until all
// work before this kernel has completed and its writes are visible, then let the
// stream's next kernel start, which waits in turn.  Nothing that earlier work
// may still read or write is touched before this returns.  The order matters:
// letting the next kernel start before the wait starts the one after it too, and
// a grid placed while another still holds most SMs piles up on the few that are
// free (a micro-batch step: 110 us that way round, 88 this way).
__device__ __forceinline__ void grid_begin() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---------------------------------------------------------------------------
// memory
// ---------------------------------------------------------------------------

// 16-byte read of data that is used once: not kept in L1, L2 asked to fetch
// the surrounding 256 bytes (the rest of the row segment follows immediately).
__device__ __forceinline__ uint4 ld_stream(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::256B.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

// L2 cache policies for loads: keep a line (the first of two sweeps over a
// row) or let it go first (the last read of a line).
__device__ __forceinline__ uint64_t policy_evict_last() {
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// 16-byte non-allocating read with an explicit L2 policy.
__device__ __forceinline__ uint4 ld_policy(const uint4* p, uint64_t pol) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p), "l"(pol));
    return v;
}

// 16-byte write of data that is not read back soon (evict-first).
__device__ __forceinline__ void st_stream(uint4* p, const uint4& v) {
    asm volatile("st.global.cs.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z),
                 "r"(v.w)
                 : "memory");
}

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
__device__ __forceinline__ float bf16_to_float(acrl_bf16 h) { return __uint_as_float(uint32_t(h) << 16); }

// Two floats to a bf16x2 word, round to nearest even; `lo` lands in the low half.
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// 2^x on the SFU (flushes subnormal results to zero).
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ void raise_flag(int32_t* flags, int32_t bit) {
    if (flags) atomicOr(flags, bit);
}

// ---------------------------------------------------------------------------
// online log-sum-exp state in base 2
//   u = z * log2(e),  U = running max of u,
//   s0 = sum 2^(u - U),  s1 = sum 2^(u - U) (u - U)
// so that lse = ln2 (U + log2 s0) and entropy = ln2 (log2 s0 - s1 / s0).
// ---------------------------------------------------------------------------

struct LseAcc {
    float U;
    float s0;
    float s1;
};

__device__ __forceinline__ LseAcc lse_empty() { return LseAcc{-INFINITY, 0.f, 0.f}; }

// Merge two partial states.  An empty side (s0 == 0) contributes nothing; the
// selects keep -inf * 0 out of the arithmetic.
__device__ __forceinline__ LseAcc lse_merge(const LseAcc& a, const LseAcc& b) {
    const float U = fmaxf(a.U, b.U);
    LseAcc r;
    r.U = U;
    const float da = a.U - U, db = b.U - U;
    const float fa = a.s0 > 0.f ? ex2(da) : 0.f;
    const float fb = b.s0 > 0.f ? ex2(db) : 0.f;
    r.s0 = fa * a.s0 + fb * b.s0;
    const float ta = a.s0 > 0.f ? fa * fmaf(da, a.s0, a.s1) : 0.f;
    const float tb = b.s0 > 0.f ? fb * fmaf(db, b.s0, b.s1) : 0.f;
    r.s1 = ta + tb;
    return r;
}

// A state's sums against another exponent, at least as large.  Where several states
// become one, merging them level by level takes an exponential at each; brought to
// their common maximum, each takes one, and the rest are plain sums.
__device__ __forceinline__ LseAcc lse_at(const LseAcc& a, float U) {
    const float da = a.U - U, f = a.s0 > 0.f ? ex2(da) : 0.f;   // an empty state contributes nothing
    return LseAcc{U, f * a.s0, a.s0 > 0.f ? f * fmaf(da, a.s0, a.s1) : 0.f};
}

__device__ __forceinline__ LseAcc shfl_xor(const LseAcc& a, int m) {
    return LseAcc{__shfl_xor_sync(0xffffffffu, a.U, m), __shfl_xor_sync(0xffffffffu, a.s0, m),
                  __shfl_xor_sync(0xffffffffu, a.s1, m)};
}

// Butterfly over the warp: every lane ends with the same value, and the
// combination order is fixed, so the result is deterministic.
__device__ __forceinline__ LseAcc warp_lse(LseAcc a) {
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) a = lse_merge(a, shfl_xor(a, m));
    return a;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
    return v;
}

template <typename T>
__device__ __forceinline__ T warp_max(T v) {
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, m));
    return v;
}

// ---------------------------------------------------------------------------
// fp64 sums over a warp.  The part's fp64 pipe takes two lanes a cycle per SM,
// so a warp-wide fp64 add costs 16 cycles of it, and a butterfly that repeats
// every sum in every lane is the wrong shape: these halve the values a lane
// carries at each level where there is more than one (6 adds per warp for four
// sums, 5 for two, against 20 and 10).  The order is fixed.
// ---------------------------------------------------------------------------

__device__ __forceinline__ double shfl_xor_f64(double v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }

// Reciprocal, quotient and square root in fp64 with short dependent chains: from
// one fp64 operation to the next that needs it takes some 80 cycles here, and the
// compiler's division and root are a dozen of them.  Newton-Raphson from the fp32
// approximation (23 bits): one step on the reciprocal (46 bits), then the
// residual of the quotient, which brings the error down to the rounding of the
// last operation; likewise for the root.  `recip64` and `quot64` want
// 2^-100 <= |b| < 2^100, so that the approximation and every product stay normal
// (counts always are); `div64` and `sqrt64` take other operands to the ordinary
// operation.
__device__ __forceinline__ bool exp_within(double v, int lim) {  // 2^-lim <= |v| < 2^lim
    const int e = ((__double2hiint(v) >> 20) & 0x7ff) - 1023;
    return e >= -lim && e < lim;
}

__device__ __forceinline__ double recip64(double b) {
    float x;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(x) : "f"(float(b)));
    const double r = double(x);
    return fma(fma(-b, r, 1.0), r, r);
}

// a / b, r = recip64(b).
__device__ __forceinline__ double quot64(double a, double b, double r) {
    const double q = a * r;
    const double c = fma(fma(-b, q, a), r, q);
    return (__double2hiint(q) & 0x7ff00000) == 0x7ff00000 ? q : c;  // an infinite a has no residual
}

__device__ __forceinline__ double div64(double a, double b) {
    return exp_within(b, 100) ? quot64(a, b, recip64(b)) : a / b;
}

__device__ __forceinline__ double sqrt64(double v) {
    if (!exp_within(v, 100) || v < 0.0) return sqrt(v);
    const double r = double(rsqrtf(float(v)));
    double g = v * r, h = 0.5 * r;
    const double e = fma(-h, g, 0.5);
    g = fma(g, e, g);
    h = fma(h, e, h);
    return fma(fma(-g, g, v), h, g);
}

// Sum of 32 non-negative counts below 2^31.
__device__ __forceinline__ long long warp_count(int n) {
    const unsigned lo = __reduce_add_sync(0xffffffffu, unsigned(n) & 0xffffu);
    const unsigned hi = __reduce_add_sync(0xffffffffu, unsigned(n) >> 16);
    return (long long)(lo) + ((long long)(hi) << 16);
}

// Four sums: lane l ends with the total of value l / 8.
__device__ __forceinline__ double warp_sum4(double a0, double a1, double a2, double a3) {
    const int lane = threadIdx.x & 31;
    const bool hi = lane & 16, odd = lane & 8;
    const double k0 = (hi ? a2 : a0) + shfl_xor_f64(hi ? a0 : a2, 16);
    const double k1 = (hi ? a3 : a1) + shfl_xor_f64(hi ? a1 : a3, 16);
    double k = (odd ? k1 : k0) + shfl_xor_f64(odd ? k0 : k1, 8);
#pragma unroll
    for (int m = 4; m >= 1; m >>= 1) k += shfl_xor_f64(k, m);
    return k;
}

// Two sums: lane l ends with the total of value l / 16.
__device__ __forceinline__ double warp_sum2(double a0, double a1) {
    const bool hi = threadIdx.x & 16;
    double k = (hi ? a1 : a0) + shfl_xor_f64(hi ? a0 : a1, 16);
#pragma unroll
    for (int m = 8; m >= 1; m >>= 1) k += shfl_xor_f64(k, m);
    return k;
}

// Maximum of non-negative floats (their bit patterns order as unsigned integers).
__device__ __forceinline__ float warp_max_nonneg(float v) {
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}

// ---------------------------------------------------------------------------
// thread-block clusters
// ---------------------------------------------------------------------------

__device__ __forceinline__ uint32_t cluster_size() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// All threads of the cluster's CTAs.  The barrier is the .aligned form, which a warp
// executes as one: a caller may come from a block that one lane took.
__device__ __forceinline__ void cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Address of the same shared-memory location in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(r)
                 : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(rank));
    return r;
}

__device__ __forceinline__ double ld_peer_f64(const double* p, uint32_t rank) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(peer_addr(p, rank)) : "memory");
    return v;
}

__device__ __forceinline__ uint32_t ld_peer_u32(const void* p, uint32_t rank) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(peer_addr(p, rank)) : "memory");
    return v;
}

}  // namespace acrl
