// Per-row online log-sum-exp over bf16 logits, shared by the statistics
// kernel, the gradient kernel's recompute sweep and the LM-head epilogue.
#pragma once

#include "acrl_device.cuh"

namespace acrl {

// Element-wise maximum of two bf16 pairs (a NaN gives way to a number, as in fmaxf).
__device__ __forceinline__ uint32_t max_bf16x2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// A running maximum's exponent.  BOUNDED: the products of numbers near the type's
// lowest stay finite, so that a thread which has met nothing else, or (with a state
// that starts at kLowestU) only infinities, holds an empty sum.
constexpr float kLowestU = -3.402823466e38f;

template <bool BOUNDED>
__device__ __forceinline__ float max_exponent(float m) {
    return BOUNDED ? fmaxf(m * kLog2e, kLowestU) : m * kLog2e;
}

// Fold UNROLL 8-element vectors into the thread's running state.
template <int UNROLL, bool BOUNDED = false>
__device__ __forceinline__ void fold_vectors(LseAcc& acc, float& mx, const uint4 (&v)[UNROLL]) {
    float f[UNROLL][8];
#pragma unroll
    for (int k = 0; k < UNROLL; ++k) {
        f[k][0] = bf16_lo(v[k].x); f[k][1] = bf16_hi(v[k].x);
        f[k][2] = bf16_lo(v[k].y); f[k][3] = bf16_hi(v[k].y);
        f[k][4] = bf16_lo(v[k].z); f[k][5] = bf16_hi(v[k].z);
        f[k][6] = bf16_lo(v[k].w); f[k][7] = bf16_hi(v[k].w);
    }
    // the maximum in bf16 pairs: half the instructions of 32-bit maxima, the same value
    uint32_t pm = max_bf16x2(max_bf16x2(v[0].x, v[0].y), max_bf16x2(v[0].z, v[0].w));
#pragma unroll
    for (int k = 1; k < UNROLL; ++k)
        pm = max_bf16x2(pm, max_bf16x2(max_bf16x2(v[k].x, v[k].y), max_bf16x2(v[k].z, v[k].w)));
    const float vm = fmaxf(bf16_lo(pm), bf16_hi(pm));
    if (vm > mx) {  // new running maximum: rescale the partial sums
        const float Un = max_exponent<BOUNDED>(vm);
        if (acc.s0 > 0.f) {
            const float dl = acc.U - Un;
            const float s = ex2(dl);
            acc.s1 = s * fmaf(dl, acc.s0, acc.s1);
            acc.s0 *= s;
        }
        acc.U = Un;
        mx = vm;
    }
    const float U = acc.U;
    float s0a = 0.f, s0b = 0.f, s1a = 0.f, s1b = 0.f;
#pragma unroll
    for (int k = 0; k < UNROLL; ++k)
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
            const float y0 = fmaf(f[k][j], kLog2e, -U);
            const float y1 = fmaf(f[k][j + 1], kLog2e, -U);
            const float e0 = ex2(y0), e1 = ex2(y1);
            s0a += e0;
            s0b += e1;
            s1a = fmaf(e0, y0, s1a);
            s1b = fmaf(e1, y1, s1b);
        }
    acc.s0 += s0a + s0b;
    acc.s1 += s1a + s1b;
}

template <bool BOUNDED = false>
__device__ __forceinline__ void fold_scalar(LseAcc& acc, float& mx, float z) {
    if (z > mx) {
        const float Un = max_exponent<BOUNDED>(z);
        if (acc.s0 > 0.f) {
            const float dl = acc.U - Un;
            const float s = ex2(dl);
            acc.s1 = s * fmaf(dl, acc.s0, acc.s1);
            acc.s0 *= s;
        }
        acc.U = Un;
        mx = z;
    }
    const float y = fmaf(z, kLog2e, -acc.U);
    const float e = ex2(y);
    acc.s0 += e;
    acc.s1 = fmaf(e, y, acc.s1);
}

// The ragged last step of a sweep: vectors v, v + TEAM, ... below n, the next one
// loaded before one is used (two loads in flight, and few registers).
template <int TEAM, typename Load, typename Use>
__device__ __forceinline__ void rest_of_row(int v, int n, Load load, Use use) {
    if (v >= n) return;
    uint4 cur = load(v);
#pragma unroll 1
    for (;;) {
        const int w = v + TEAM;
        uint4 next = cur;
        if (w < n) next = load(w);
        use(cur, v);
        if (w >= n) return;
        cur = next;
        v = w;
    }
}

// The thread's partial state over its share of one row (lane `tid` of a team of TEAM threads).
template <int TEAM, int UNROLL>
__device__ __forceinline__ LseAcc row_partial(const acrl_bf16* __restrict__ row, int V, int tid, float& mx) {
    LseAcc acc = lse_empty();
    mx = -INFINITY;
    const int nvec = V >> 3;
    const uint4* vrow = reinterpret_cast<const uint4*>(row);
    int v = tid;
    for (; v + (UNROLL - 1) * TEAM < nvec; v += UNROLL * TEAM) {
        uint4 buf[UNROLL];
#pragma unroll
        for (int k = 0; k < UNROLL; ++k) buf[k] = ld_stream(vrow + v + k * TEAM);
        fold_vectors<UNROLL>(acc, mx, buf);
    }
    for (; v < nvec; v += TEAM) {
        uint4 buf[1] = {ld_stream(vrow + v)};
        fold_vectors<1>(acc, mx, buf);
    }
    for (int j = (nvec << 3) + tid; j < V; j += TEAM) fold_scalar(acc, mx, bf16_to_float(row[j]));
    return acc;
}

// 16-byte copy from global to shared memory, asynchronous, past L1.
__device__ __forceinline__ void cp_async16(uint4* dst, const uint4* src) {
    asm volatile("cp.async.cg.shared.global.L2::256B [%0], [%1], 16;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// row_partial with DEPTH steps of loads in flight instead of one: each thread
// copies its own vectors into its own slots of shared memory (slot k of step i
// at ring[((i mod DEPTH) UNROLL + k) THREADS]), so nothing is shared and no
// thread waits for another.  The vectors are folded in row_partial's order, so
// the result is the same to the last bit.
template <int TEAM, int UNROLL, int THREADS, int DEPTH>
__device__ __forceinline__ LseAcc row_partial_ring(const acrl_bf16* __restrict__ row, int V, int tid, float& mx,
                                                   uint4* ring) {
    constexpr int STEP = TEAM * UNROLL;
    LseAcc acc = lse_empty();
    mx = -INFINITY;
    const int nvec = V >> 3;
    const uint4* vrow = reinterpret_cast<const uint4*>(row);
    const int rem = nvec - tid - (UNROLL - 1) * TEAM;
    const int full = rem > 0 ? (rem + STEP - 1) / STEP : 0;   // steps in which all of this thread's vectors exist
    auto issue = [&](int i, int slot) {
        const int v = tid + i * STEP;
#pragma unroll
        for (int k = 0; k < UNROLL; ++k)
            if (i <= full && v + k * TEAM < nvec) cp_async16(ring + (slot * UNROLL + k) * THREADS, vrow + v + k * TEAM);
        cp_async_commit();
    };
#pragma unroll
    for (int i = 0; i < DEPTH; ++i) issue(i, i);
    int slot = 0;
    for (int i = 0; i < full; ++i) {
        cp_async_wait<DEPTH - 1>();
        uint4 buf[UNROLL];
#pragma unroll
        for (int k = 0; k < UNROLL; ++k) buf[k] = ring[(slot * UNROLL + k) * THREADS];
        fold_vectors<UNROLL>(acc, mx, buf);
        issue(i + DEPTH, slot);
        slot = slot + 1 == DEPTH ? 0 : slot + 1;
    }
    cp_async_wait<0>();
    int v = tid + full * STEP;
    for (int k = 0; v < nvec; v += TEAM, ++k) {
        uint4 buf[1] = {ring[(slot * UNROLL + k) * THREADS]};
        fold_vectors<1>(acc, mx, buf);
    }
    for (int j = (nvec << 3) + tid; j < V; j += TEAM) fold_scalar(acc, mx, bf16_to_float(row[j]));
    return acc;
}

// The sampled token of a row and its logit, loaded while the row streams.
struct RowTarget {
    float z;
    bool ok;   // the id is inside the vocabulary
};

__device__ __forceinline__ RowTarget row_target(const acrl_bf16* row, int V, int a) {
    const bool ok = a >= 0 && a < V;
    return RowTarget{ok ? bf16_to_float(row[a]) : 0.f, ok};
}

// Outputs of one row from its merged state; mx is the row maximum (natural units).
__device__ __forceinline__ void row_outputs(const LseAcc& acc, float mx, const RowTarget& tgt, float* lse, float* logp,
                                            float* ent, int64_t t, int32_t* flags) {
    const float l2s0 = log2f(acc.s0);
    // acc.U is mx*log2(e) rounded; c is that rounding error, exact through the FMA
    const float c = fmaf(mx, kLog2e, -acc.U);
    const float lse_v = fmaf(kLn2, l2s0 - c, mx);
    const float H = kLn2 * (l2s0 - acc.s1 / acc.s0);
    if (!tgt.ok) raise_flag(flags, ACRL_FLAG_BAD_ID);
    const float lp = tgt.ok ? (tgt.z - mx) - kLn2 * (l2s0 - c) : 0.f;
    if (!isfinite(lse_v) || !isfinite(H)) {
        raise_flag(flags, ACRL_FLAG_NONFINITE);
        lse[t] = logp[t] = ent[t] = __int_as_float(0x7fc00000);
        return;
    }
    lse[t] = lse_v;
    logp[t] = lp;
    ent[t] = H;
}

}  // namespace acrl
