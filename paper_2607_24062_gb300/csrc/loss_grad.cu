// acrl_loss_grad_logits: the loss of Eq. ACRL and its gradient with respect
// to pi's logits, written in bf16 without ever storing the probabilities.
//
//     grad[t, j] = coef_t g_t r_t (p_tj - 1[j = a_t]),  p_tj = exp(z_tj - lse_t)
//
// One streaming pass per live row: read 2 bytes and write 2 bytes per element.
// The row's factor is folded into the exponent, |c| p = 2^(z log2e - (lse log2e
// - log2|c|)), so each element costs one FMA and one SFU exp2; the sign is
// applied to the packed bf16 pair with one XOR.  The target column is written
// as c * expm1(logp) so that p_a - 1 keeps its accuracy when p_a is near 1.
// With an entropy bonus e_t the element becomes p (c + e (z - lse + H)): one
// more FMA and a multiply.  Rows that carry no gradient (masked, zero
// coefficient and no bonus, clipped) are written as zeros without reading
// their logits.  With lse == NULL the row's log-sum-exp is first recomputed
// by a sweep over the same row; the first 16-byte vectors of the row (up to
// 14, 40, 72 or 96 KB, by the CTA's size) stay in the CTA's shared memory and, for
// rows of 65,536 columns or more, the next up to kTmemVecs (128 KB) in its
// tensor memory between the two sweeps, so that only the rest of the row is
// read again, from L2.  The shared-memory part arrives by one bulk copy
// started when the row starts, while the threads load the rest.
#include "acrl_device.cuh"
#include "acrl_host.h"
#include "mbarrier.cuh"
#include "row_lse.cuh"

namespace acrl {
namespace {

constexpr uint32_t kSignPair = 0x80008000u;

// CTA kernel: four 16-byte vectors per thread and step.  The recompute path of
// long rows takes 512 threads and keeps kKeepVecs vectors of a row in shared memory
// between the sweeps (96 KB, three whole sweep chunks; two 512-thread CTAs per SM).
constexpr int kCtaThreads = 512, kCtaUnroll = 4;
// The streaming path (lse given) takes a CTA per row, of the most threads that the
// row keeps busy for one whole step (the smallest for a row of 2,048 columns is 64
// threads; 512 from 16,384 columns), and below that a warp per row.  Fewer threads
// leave the row's later steps to wait for memory one after the other, more leave
// threads idle or the last step ragged.  Kernel with its loss sum, us, warp per row
// (what rows of up to 16,384 columns took before) and now: 1,000 x 2,048 5.3 / 5.0;
// 8,000 x 2,600 21.1 / 19.2; 8,000 x 4,096 27.9 / 24.5; 1,000 x 5,003 11.7 / 8.4;
// 8,000 x 5,003 38.1 / 30.7; 300 x 8,192 8.8 / 4.6; 30,000 x 8,192 150.8 / 144.7;
// 8,000 x 10,007 68.3 / 52.1; 20,000 x 14,001 179.4 / 168.5; 600 x 16,384 18.4 /
// 10.2; 20,000 x 16,384 208 / 189 (a copy of the bytes: 196).  With many short rows
// there is enough in flight whatever the split, and the ragged steps and the CTAs'
// ends weigh more: from kManyRows rows a warp each up to 4,095 columns (40,000 x
// 3,333: 88 against 95 with 64 threads; 12,000: 31.7 against 33.4) and 64 threads up
// to 8,191 (40,000 x 7,000: 169 against 177 with 128; 20,000 x 5,003: 66.7 against
// 68.2).
constexpr int64_t kManyRows = 12000;
constexpr int kStreamStep = 8 * kCtaUnroll;   // columns of one thread's step
// Rows of more than 65,536 columns are split between CTAs of 256 threads, two whole
// steps and a little more for each (nine for 151,936 columns): more of the row is in
// flight when rows are few, the chip stays even when they are many, and a ragged
// last step is short.  A CTA of 768 threads per row / split: 40 x 151,936 12.7 / 9.2
// us, 408 x 151,936 42.4 / 41.2, 700 x 151,936 69.7 / 65.9, 3,000 x 151,936 268 / 262,
// 3,000 x 65,544 123.5 / 117.8, 3,000 x 200,000 355 / 343; with 6 to 8 shares of
// 151,936 columns 66.7, with 11 to 14 68.  Lengths that make wider shares: 3,000 x
// 80,000 (2.4 steps) 148 / 143, 20,000 919 / 917; 3,000 x 128,256 (2.2) 232 / 224, 8,000
// 597 / 585; 300 x 72,000 (2.2) 22.7 / 18.0.
constexpr int kShareThreads = 256, kShareVecs = 2 * kShareThreads * kCtaUnroll;
constexpr int64_t kShareRowMinV = 65537;
// A call of so many rows that the shares would not fit a grid takes a CTA per row.
constexpr int kWideThreads = 768;
constexpr int kChunk = kCtaThreads * kCtaUnroll;   // vectors one sweep step of the CTA covers
constexpr int kKeepVecs = 3 * kChunk;
static_assert(kKeepVecs * 16 <= 100 * 1024, "two CTAs per SM must fit");
// The next chunks of the row (whole chunks only, so that every warp takes part
// in each tensor-memory access) go to tensor memory: each of the two CTAs on an
// SM allocates 256 of its 512 columns, 128 lanes x 256 columns x 4 bytes =
// 128 KB = 4 chunks.  Thread t of warp w keeps its k-th vector of chunk c in
// lane 32 (w mod 4) + t, columns 64 (w / 4) + 16 c + 4 k .. + 3.
constexpr uint32_t kTmemCols = 256;
constexpr int kTmemChunks = 4;
constexpr int kTmemVecs = kTmemChunks * kChunk;
static_assert(kTmemVecs * 16 == 128 * kTmemCols * 4, "tensor-memory share of a CTA");
static_assert(kCtaThreads == 512 && kCtaUnroll == 4, "column layout: 16 warps, 4 vectors per step");
// Tensor memory holds whole chunks only, so rows of fewer than kKeepVecs +
// kChunk vectors (V < 65,536) keep nothing there; they take a kernel instance
// without any tcgen05 code (TM = false).  A resident CTA of a kernel that may
// allocate tensor memory keeps the SM from starting another CTA of that kernel
// until it has given up its allocation permit: measured with ncu, 15.6 warps
// resident per SM against 30.7 for the same work without tcgen05 code.
constexpr int kTmemMinVecs = kKeepVecs + kChunk;
// Shorter rows take smaller CTAs, so that several fit on an SM with what they keep:
//   from kRecomputeCtaMinV columns  64 threads,  up to 14 KB: V <= 7,168
//   up to kTinyKeepVecs vectors    128 threads,  up to 40 KB: V <= 20,487
//   up to kSmallMaxVecs vectors    256 threads,  up to 72 KB: V <= 40,967 (of a row
//                                  longer than 72 KB the rest, at most 8 KB, is read
//                                  again from L2)
// and those below a warp each, which reads its row again from L2.  Us, the call with
// its loss sum: 30,000 x 5,003 126 with a warp, 102 with 64 threads, 131 with 128;
// 8,000 x 6,200 45 / 37 / 44; 1,000 x 8,192 15.5 / 12.5 / 11.8; 16,000 x 14,001
// 199 with 64, 137 with 128, 174 with 256; 10,000 x 24,000 219 with 128 (whose rest
// of the row is a ragged step in each sweep), 151 with 256, 215 with 512; 2,000 x
// 44,000 79 with 256, 68 with 512; 30,000 x 3,333 77 with a warp (in CTAs of two; 83
// in CTAs of eight), 84 with 64 threads.
constexpr int kRecomputeCtaMinV = 4096;
constexpr int kLeastMaxV = 7168;
constexpr int kLeastThreads = 64, kLeastKeepVecs = kLeastMaxV / 8;
constexpr int kTinyThreads = 128, kTinyKeepVecs = 2560;
constexpr int kSmallThreads = 256, kSmallKeepVecs = 4608;
constexpr int kSmallMaxVecs = 5120;

// Vectors of a row that a recompute CTA of THREADS threads keeps in shared memory.
template <int THREADS>
constexpr int kKeepOf = THREADS == kLeastThreads   ? kLeastKeepVecs
                        : THREADS == kTinyThreads  ? kTinyKeepVecs
                        : THREADS == kSmallThreads ? kSmallKeepVecs
                                                   : kKeepVecs;

// Where the vectors of a row live between the two sweeps of the recompute
// path: [0, s) in `smem` (filled by a bulk copy that completes on `bar`),
// [s, s + tm_chunks kChunk) in tensor memory from the thread's column base
// `tbase`, the rest in L2.
struct RowKeep {
    uint4* smem;
    int s;
    uint32_t tbase;
    int tm_chunks;
    uint64_t* bar;
};

// Bulk copy of `bytes` (a multiple of 16; both addresses 16-byte aligned) from
// global to this CTA's shared memory, completing on `bar`, with an L2 policy.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar, uint64_t pol) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::
            "r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol)
        : "memory");
}

__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint4& v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(v.x), "r"(v.y),
                 "r"(v.z), "r"(v.w)
                 : "memory");
}
__device__ __forceinline__ uint4 tmem_ld4(uint32_t taddr) {
    uint4 v;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(taddr));
    return v;
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// The vectors [begin, end) of a row that a CTA handles: all of them, or one of the
// shares of a row that several CTAs split; the first share's CTA also writes what
// there is one of per row.
struct RowShare {
    int begin, end;
};

// Per-row constants of the streaming pass.
struct RowPlan {
    float B;        // policy term only: lse log2e - log2|c|
    uint32_t sgn;   // policy term only: kSignPair when c < 0
    float L2;       // with entropy: lse log2e
    float e;        // with entropy: e_t
    float c2;       // with entropy: c - e (lse - H)
    float target;   // gradient at the sampled column
    int a;          // sampled column
};

template <bool ENT>
__device__ __forceinline__ float grad_elem(float z, const RowPlan& rp) {
    if (ENT) {
        const float p = ex2(fmaf(z, kLog2e, -rp.L2));
        return p * fmaf(rp.e, z, rp.c2);
    }
    return ex2(fmaf(z, kLog2e, -rp.B));  // magnitude; sign applied by the caller
}

template <bool ENT>
__device__ __forceinline__ uint4 grad_vec(const uint4 v, const RowPlan& rp, int rel) {
    float e[8];
    e[0] = grad_elem<ENT>(bf16_lo(v.x), rp);
    e[1] = grad_elem<ENT>(bf16_hi(v.x), rp);
    e[2] = grad_elem<ENT>(bf16_lo(v.y), rp);
    e[3] = grad_elem<ENT>(bf16_hi(v.y), rp);
    e[4] = grad_elem<ENT>(bf16_lo(v.z), rp);
    e[5] = grad_elem<ENT>(bf16_hi(v.z), rp);
    e[6] = grad_elem<ENT>(bf16_lo(v.w), rp);
    e[7] = grad_elem<ENT>(bf16_hi(v.w), rp);
    const uint32_t sgn = ENT ? 0u : rp.sgn;
    uint4 o;
    if (static_cast<unsigned>(rel) < 8u) {  // the vector holding the sampled column
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float val = sgn ? -e[j] : e[j];
            e[j] = (j == rel) ? rp.target : val;
        }
        o.x = pack_bf16x2(e[0], e[1]);
        o.y = pack_bf16x2(e[2], e[3]);
        o.z = pack_bf16x2(e[4], e[5]);
        o.w = pack_bf16x2(e[6], e[7]);
        return o;
    }
    o.x = pack_bf16x2(e[0], e[1]) ^ sgn;
    o.y = pack_bf16x2(e[2], e[3]) ^ sgn;
    o.z = pack_bf16x2(e[4], e[5]) ^ sgn;
    o.w = pack_bf16x2(e[6], e[7]) ^ sgn;
    return o;
}

// First sweep of the recompute path: the thread's partial state over its share
// of the row.  Vectors below `kp.s` (read once from HBM, L2 evict-first: they
// are not read from L2 again) come into shared memory by the bulk copy that
// thread 0 started on `kp.bar` (phase parity `parity`) and are folded last,
// once it has landed; those of the next kp.tm_chunks whole chunks are copied
// to tensor memory; the rest are loaded with the L2 evict-last policy, since
// the second sweep reads them again.  The tensor-memory stores are complete
// when the caller has waited for them (tmem_wait_st).  A copy that has not
// landed after the bounded wait raises ACRL_FLAG_TIMEOUT.
template <int TEAM, int UNROLL, bool TM>
__device__ __forceinline__ LseAcc recompute_partial(const acrl_bf16* __restrict__ row, int V, int tid, float& mx,
                                                    const RowKeep& kp, uint32_t parity, int32_t* flags) {
    LseAcc acc{kLowestU, 0.f, 0.f};   // columns at -infinity add nothing, whichever the thread meets first
    mx = -INFINITY;
    const int nvec = V >> 3;
    const uint4* vrow = reinterpret_cast<const uint4*>(row);
    const uint64_t pol = policy_evict_last(), once = policy_evict_first();
    const int s = kp.s;
    int v = s + tid;
    // whole chunks (s is a multiple of the chunk whenever kp.tm_chunks > 0): every thread takes part
    if constexpr (TM) {
        for (int ch = 0; ch < kp.tm_chunks; ++ch, v += UNROLL * TEAM) {
            uint4 buf[UNROLL];
#pragma unroll
            for (int k = 0; k < UNROLL; ++k) buf[k] = ld_policy(vrow + v + k * TEAM, once);
#pragma unroll
            for (int k = 0; k < UNROLL; ++k) tmem_st4(kp.tbase + uint32_t(16 * ch + 4 * k), buf[k]);
            fold_vectors<UNROLL, true>(acc, mx, buf);
        }
    }
    for (; v + (UNROLL - 1) * TEAM < nvec; v += UNROLL * TEAM) {
        uint4 buf[UNROLL];
#pragma unroll
        for (int k = 0; k < UNROLL; ++k) buf[k] = ld_policy(vrow + v + k * TEAM, pol);
        fold_vectors<UNROLL, true>(acc, mx, buf);
    }
    const int j = (nvec << 3) + tid;   // at most one column per thread beyond the whole vectors
    const float last = j < V ? bf16_to_float(row[j]) : 0.f;
    rest_of_row<TEAM>(
        v, nvec, [&](int i) { return ld_policy(vrow + i, pol); },
        [&](const uint4& x, int) {
            const uint4 buf[1] = {x};
            fold_vectors<1, true>(acc, mx, buf);
        });
    if (j < V) fold_scalar<true>(acc, mx, last);
    if (s > 0) {
        if (!wait_phase(kp.bar, parity, nullptr)) raise_flag(flags, ACRL_FLAG_TIMEOUT);
        for (v = tid; v + (UNROLL - 1) * TEAM < s; v += UNROLL * TEAM) {
            uint4 buf[UNROLL];
#pragma unroll
            for (int k = 0; k < UNROLL; ++k) buf[k] = kp.smem[v + k * TEAM];
            fold_vectors<UNROLL, true>(acc, mx, buf);
        }
        for (; v < s; v += TEAM) {
            uint4 buf[1] = {kp.smem[v]};
            fold_vectors<1, true>(acc, mx, buf);
        }
    }
    return acc;
}

// LAST: this is the second sweep over a row after recompute_partial, and the
// last read of its lines (L2 evict-first policy).  It reads the part that
// comes from L2 in the order the first sweep loaded it, so that every line
// waits about as long in L2 as any other, then the chunks in tensor memory,
// then the vectors in shared memory.
template <int TEAM, int UNROLL, bool ENT, bool LAST = false, bool TM = false>
__device__ __forceinline__ void stream_grad_row(const acrl_bf16* __restrict__ row, acrl_bf16* __restrict__ grow, int V,
                                                int tid, const RowPlan& rp, const RowKeep& kp, const RowShare& sh) {
    const int nvec = LAST ? V >> 3 : sh.end;
    const uint4* src = reinterpret_cast<const uint4*>(row);
    uint4* dst = reinterpret_cast<uint4*>(grow);
    if (LAST) {
        const uint64_t pol = policy_evict_first();
        const int te = kp.s + kp.tm_chunks * UNROLL * TEAM;   // first vector read from L2
        int v = te + tid;
        for (; v + (UNROLL - 1) * TEAM < nvec; v += UNROLL * TEAM) {
            uint4 buf[UNROLL];
#pragma unroll
            for (int k = 0; k < UNROLL; ++k) buf[k] = ld_policy(src + v + k * TEAM, pol);
#pragma unroll
            for (int k = 0; k < UNROLL; ++k) {
                const int vi = v + k * TEAM;
                st_stream(dst + vi, grad_vec<ENT>(buf[k], rp, rp.a - (vi << 3)));
            }
        }
        rest_of_row<TEAM>(
            v, nvec, [&](int i) { return ld_policy(src + i, pol); },
            [&](const uint4& x, int i) { st_stream(dst + i, grad_vec<ENT>(x, rp, rp.a - (i << 3))); });
        for (int ch = 0; TM && ch < kp.tm_chunks; ++ch) {
            uint4 buf[UNROLL];
#pragma unroll
            for (int k = 0; k < UNROLL; ++k) buf[k] = tmem_ld4(kp.tbase + uint32_t(16 * ch + 4 * k));
            tmem_wait_ld();
            const int v0 = kp.s + ch * UNROLL * TEAM + tid;
#pragma unroll
            for (int k = 0; k < UNROLL; ++k) {
                const int vi = v0 + k * TEAM;
                st_stream(dst + vi, grad_vec<ENT>(buf[k], rp, rp.a - (vi << 3)));
            }
        }
        for (int vi = tid; vi < kp.s; vi += TEAM) st_stream(dst + vi, grad_vec<ENT>(kp.smem[vi], rp, rp.a - (vi << 3)));
    } else {
        int v = sh.begin + tid;
        for (; v + (UNROLL - 1) * TEAM < nvec; v += UNROLL * TEAM) {
            uint4 buf[UNROLL];
#pragma unroll
            for (int k = 0; k < UNROLL; ++k) buf[k] = ld_stream(src + v + k * TEAM);
#pragma unroll
            for (int k = 0; k < UNROLL; ++k) {
                const int vi = v + k * TEAM;
                st_stream(dst + vi, grad_vec<ENT>(buf[k], rp, rp.a - (vi << 3)));
            }
        }
        for (; v < nvec; v += TEAM) st_stream(dst + v, grad_vec<ENT>(ld_stream(src + v), rp, rp.a - (v << 3)));
    }
    if (nvec != V >> 3) return;   // the columns beyond the whole vectors are the last share's
    for (int j = (nvec << 3) + tid; j < V; j += TEAM) {
        float val = grad_elem<ENT>(bf16_to_float(row[j]), rp);
        if (!ENT && rp.sgn) val = -val;
        if (j == rp.a) val = rp.target;
        grow[j] = static_cast<acrl_bf16>(pack_bf16x2(val, 0.f) & 0xffffu);
    }
}

// A gradient row of one value (`pair` holds it twice, as a bf16x2 word), written
// without reading the logits: 0 for rows that carry no gradient, NaN for rows
// whose surrogate is undefined.
constexpr uint32_t kZeroPair = 0u, kNaNPair = 0x7FC07FC0u;

template <int TEAM>
__device__ __forceinline__ void fill_row(acrl_bf16* __restrict__ grow, int V, int tid, uint32_t pair, const RowShare& sh) {
    const int nvec = sh.end;
    uint4* dst = reinterpret_cast<uint4*>(grow);
    const uint4 z = make_uint4(pair, pair, pair, pair);
    for (int v = sh.begin + tid; v < nvec; v += TEAM) st_stream(dst + v, z);
    if (nvec != V >> 3) return;
    for (int j = (nvec << 3) + tid; j < V; j += TEAM) grow[j] = static_cast<acrl_bf16>(pair & 0xffffu);
}

struct RowCoef {
    float c;       // coef_t g_t r_t
    float loss;    // token loss (policy term)
};

// Scalar part of a live row: r, the clip gate, the coefficient and the loss.
__device__ __forceinline__ RowCoef row_coef(float c0, float lp, const float* old_logp, int64_t t, float eps) {
    float r = 1.f;
    if (old_logp) r = expf(lp - old_logp[t]);
    const float rc = fminf(fmaxf(r, 1.f - eps), 1.f + eps);
    const bool gate = c0 >= 0.f ? (r <= 1.f + eps) : (r >= 1.f - eps);
    RowCoef out;
    out.c = gate ? c0 * r : 0.f;
    out.loss = c0 == 0.f ? 0.f : -c0 * (c0 >= 0.f ? fminf(r, rc) : fmaxf(r, rc));
    return out;
}

template <bool ENT>
__device__ __forceinline__ RowPlan make_plan(float c, float e, float L, float H, float za, float lp, int a) {
    RowPlan rp;
    rp.a = a;
    if (ENT) {
        rp.L2 = L * kLog2e;
        rp.e = e;
        rp.c2 = fmaf(-e, L - H, c);
        rp.B = 0.f;
        rp.sgn = 0u;
        // c (p_a - 1) + e p_a (z_a - lse + H)
        rp.target = fmaf(e * expf(lp), za - L + H, c * expm1f(lp));
    } else {
        rp.B = fmaf(L, kLog2e, -log2f(fabsf(c)));
        rp.sgn = c < 0.f ? kSignPair : 0u;
        rp.L2 = rp.e = rp.c2 = 0.f;
        rp.target = c * expm1f(lp);
    }
    return rp;
}

// The online state without the entropy's sum: a sum of exponentials s0 against the
// exponent U (a maximum times log2(e), rounded, as the folds keep it).  An empty
// state contributes nothing.
struct LseSum {
    float U, s0;
};

__device__ __forceinline__ float lse_exponent(float m) { return __fmul_rn(m, kLog2e); }

// A state's sum against another exponent.
__device__ __forceinline__ float sum_at(const LseSum& a, float U) { return (a.s0 > 0.f ? ex2(a.U - U) : 0.f) * a.s0; }

// lse_merge's.
__device__ __forceinline__ LseSum sum_exp_merge(const LseSum& a, const LseSum& b) {
    const float U = fmaxf(a.U, b.U);
    const float fa = a.s0 > 0.f ? ex2(a.U - U) : 0.f;
    const float fb = b.s0 > 0.f ? ex2(b.U - U) : 0.f;
    return LseSum{U, fa * a.s0 + fb * b.s0};
}

__device__ __forceinline__ LseSum shfl_xor(const LseSum& a, int m) {
    return LseSum{__shfl_xor_sync(0xffffffffu, a.U, m), __shfl_xor_sync(0xffffffffu, a.s0, m)};
}

// The states of 2 FIRST lanes as one, in each of them; U is their common maximum's
// exponent.  MEET: each sum is brought there once and the rest are plain additions;
// otherwise they merge level by level, with an exponential at each.  Two and eight
// warps meet: they took the rows of one and of four, and the level more had left the
// log-prob of those 0.5-1.1 % further from float64 (rms); meeting, it is 5-9 % closer
// (V = 4,096: 3.68e-7 with a warp, 3.71e-7 merged, 3.51e-7; V = 24,583: 4.19e-7 with
// four warps, 4.23e-7, 3.82e-7), at the same speed.
template <bool MEET, int FIRST>
__device__ __forceinline__ LseSum lanes_sum_exp(LseSum a, float U) {
    if constexpr (MEET) a = LseSum{U, sum_at(a, U)};
#pragma unroll
    for (int m = FIRST; m >= 1; m >>= 1) {
        if constexpr (MEET)
            a.s0 += __shfl_xor_sync(0xffffffffu, a.s0, m);
        else
            a = sum_exp_merge(a, shfl_xor(a, m));
    }
    return a;
}

// lse and logp = z_a - lse of a row from its sum and maximum, in the
// same form as the statistics kernel (the rounding of max*log2(e) corrected
// exactly through an FMA).
__device__ __forceinline__ void lse_logp(float sum, float mx, float za, float& L, float& lp) {
    const float l2s0 = log2f(sum);
    const float c = fmaf(mx, kLog2e, -lse_exponent(mx));
    L = fmaf(kLn2, l2s0 - c, mx);
    lp = (za - mx) - kLn2 * (l2s0 - c);
}

// One row handled by a team (a whole CTA, or one warp).  `part`/`part_mx` are
// the CTA's shared scratch for the recompute sweep, two buffers of one slot
// per warp used in turn (`par`, flipped at every row that uses them; unused by
// warp teams); `kp` says where the recompute path keeps the row between its
// two sweeps (nothing on chip for warp teams).  The bulk copy of the row's
// shared-memory part is started by thread 0 once the row is known to be live,
// and completes the phase of kp.bar whose parity is `par`: both flip at every
// live row of a CTA team.
template <int TEAM, int UNROLL, bool RECOMPUTE, bool ENT, bool TM>
__device__ __forceinline__ void grad_row(const acrl_bf16* __restrict__ logits, int64_t t, int V, int64_t ld,
                                         const int32_t* __restrict__ ids, const uint8_t* __restrict__ mask,
                                         const float* __restrict__ lse, const float* __restrict__ old_logp,
                                         const float* __restrict__ coef, const float* __restrict__ entropy,
                                         const float* __restrict__ ent_coef, float eps, acrl_bf16* __restrict__ grad,
                                         float* __restrict__ token_loss, int32_t* flags, int tid, LseSum* part,
                                         float* part_mx, int& par, const RowKeep& kp, const RowShare& sh) {
    const acrl_bf16* row = logits + t * ld;
    acrl_bf16* grow = grad + t * ld;
    const bool m = mask ? mask[t] != 0 : true;
    const float c0 = coef[t];
    const float e = ENT ? ent_coef[t] : 0.f;
    const int a = ids[t];
    const bool bad_id = a < 0 || a >= V;
    const bool lead = tid == 0 && sh.begin == 0;
    if (m && bad_id && lead) raise_flag(flags, ACRL_FLAG_BAD_ID);
    const bool live = m && !bad_id && (c0 != 0.f || e != 0.f);
    float c = 0.f, loss = 0.f, L = 0.f, H = 0.f, za = 0.f, lp = 0.f;
    bool undefined = false;
    if (live) {
        if (RECOMPUTE && TEAM > 32 && kp.s > 0 && tid == 0) {
            // the threads' reads of the last row's part (before the CTA barrier) come before the copy's writes
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_expect_tx(kp.bar, uint32_t(kp.s) * 16u);
            bulk_load(kp.smem, row, uint32_t(kp.s) * 16u, kp.bar, policy_evict_first());
        }
        za = bf16_to_float(row[a]);
        if (RECOMPUTE) {
            constexpr bool MEET = TEAM == 64 || TEAM == 256;
            float mx;
            const LseAcc mine = recompute_partial<TEAM, UNROLL, TM>(row, V, tid, mx, kp, uint32_t(par), flags);
            mx = warp_max(mx);
            // the entropy's sum is not wanted: the compiler drops it
            LseSum acc = lanes_sum_exp<MEET, 16>(LseSum{mine.U, mine.s0}, lse_exponent(mx));
            if (TM && kp.tm_chunks > 0)
                tmem_wait_st();   // before the barrier: the row's tensor-memory part is written
            if (TEAM > 32) {
                // Every warp combines the warps' states with the same butterfly, so all threads hold the same
                // result with one barrier.  The next write to this buffer comes two rows later, after the next
                // row's barrier, which every warp reaches only once it has read this one.
                constexpr int NW = TEAM / 32;
                static_assert(!RECOMPUTE || (NW <= 32 && (NW & (NW - 1)) == 0), "warps per team");
                const int lane = tid & 31;
                LseSum* pp = part + par * NW;
                float* pm = part_mx + par * NW;
                if (lane == 0) {
                    pp[tid >> 5] = acc;
                    pm[tid >> 5] = mx;
                }
                __syncthreads();
                acc = lane < NW ? pp[lane] : LseSum{-INFINITY, 0.f};
                mx = lane < NW ? pm[lane] : -INFINITY;
#pragma unroll
                for (int o = NW / 2; o >= 1; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                acc = lanes_sum_exp<MEET, NW / 2>(acc, lse_exponent(mx));
                acc.s0 = __shfl_sync(0xffffffffu, acc.s0, 0);
                mx = __shfl_sync(0xffffffffu, mx, 0);
                par ^= 1;
            }
            lse_logp(acc.s0, mx, za, L, lp);
        } else {
            L = lse[t];
            lp = za - L;
        }
        // a row whose lse or log-prob is not finite (a NaN or an infinity among its logits), or whose old
        // log-prob is NaN, has no defined surrogate: NaN token loss and gradient row, and the flag
        undefined = !isfinite(L) || !isfinite(lp) || (old_logp != nullptr && isnan(old_logp[t]));
        if (undefined && lead) raise_flag(flags, ACRL_FLAG_NONFINITE);
        const RowCoef rc = row_coef(c0, lp, old_logp, t, eps);
        c = rc.c;
        loss = rc.loss;
        if (ENT) {
            H = entropy[t];
            loss -= e * H;
        }
    }
    if (lead) token_loss[t] = undefined ? __int_as_float(0x7fc00000) : loss;
    if (undefined) {
        fill_row<TEAM>(grow, V, tid, kNaNPair, sh);
    } else if (c == 0.f && e == 0.f) {
        fill_row<TEAM>(grow, V, tid, kZeroPair, sh);
    } else {
        stream_grad_row<TEAM, UNROLL, ENT, RECOMPUTE, TM>(row, grow, V, tid, make_plan<ENT>(c, e, L, H, za, lp, a),
                                                          kp, sh);
    }
}

// TM: the recompute instance whose CTAs keep whole chunks of a row in tensor
// memory (512 threads, rows of at least kTmemMinVecs vectors).  SHARED_ROW: `shares`
// CTAs per row, T x shares of them.
template <int THREADS, int UNROLL, bool RECOMPUTE, bool ENT, bool TM = false, bool SHARED_ROW = false>
__global__ void __launch_bounds__(THREADS) loss_grad_cta(
    const acrl_bf16* __restrict__ logits, int64_t T, int V, int64_t ld, const int32_t* __restrict__ ids,
    const uint8_t* __restrict__ mask, const float* __restrict__ lse, const float* __restrict__ old_logp,
    const float* __restrict__ coef, const float* __restrict__ entropy, const float* __restrict__ ent_coef, float eps,
    acrl_bf16* __restrict__ grad, float* __restrict__ token_loss, int32_t* flags, int shares) {
    __shared__ LseSum part[2 * (THREADS / 32)];
    __shared__ float part_mx[2 * (THREADS / 32)];
    __shared__ uint32_t tmem_base;
    __shared__ __align__(8) uint64_t keep_bar;
    extern __shared__ uint4 keep[];  // recompute path: min(kKeepOf<THREADS>, V / 8) vectors (dynamic size)
    const int warp = threadIdx.x >> 5;
    static_assert(!TM || (RECOMPUTE && THREADS == kCtaThreads && UNROLL == kCtaUnroll), "tensor-memory layout");
    RowKeep kp{keep, 0, 0u, 0, &keep_bar};
    grid_begin();
    if (RECOMPUTE) {
        const int nvec = V >> 3;
        kp.s = min(kKeepOf<THREADS>, nvec);
        kp.tm_chunks = TM && nvec > kKeepVecs ? min(kTmemChunks, (nvec - kKeepVecs) / kChunk) : 0;
        if (threadIdx.x == 0) {
            mbar_init(&keep_bar, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        if constexpr (TM) {
            if (warp == 0) {   // kp.tm_chunks is the same for every CTA of the launch
                if (kp.tm_chunks > 0)
                    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                                     static_cast<uint32_t>(__cvta_generic_to_shared(&tmem_base))),
                                 "r"(kTmemCols)
                                 : "memory");
                // at once, allocation or not: the SM may then start the kernel's next CTA
                asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        }
        __syncthreads();
        if constexpr (TM) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (kp.tm_chunks > 0)
                kp.tbase = tmem_base + (uint32_t((warp & 3) * 32) << 16) + uint32_t((warp >> 2) * 64);
        }
    }
    int par = 0;
    for (int64_t i = blockIdx.x; i < (SHARED_ROW ? T * shares : T); i += gridDim.x) {
        // a CTA with a further row refills its shared-memory part only once every thread has read the last one
        if (RECOMPUTE && i != blockIdx.x) __syncthreads();
        int64_t t = i;
        RowShare sh{0, V >> 3};
        if (SHARED_ROW) {   // few rows: T x shares fits an int
            t = int(i) / shares;
            const int share = int(i) - int(t) * shares;
            const int per = (((V >> 3) + shares - 1) / shares + 7) & ~7;   // shares begin on 128-byte lines of the row
            sh.begin = min(sh.end, share * per);
            sh.end = share == shares - 1 ? sh.end : min(sh.end, share * per + per);
        }
        grad_row<THREADS, UNROLL, RECOMPUTE, ENT, TM>(logits, t, V, ld, ids, mask, lse, old_logp, coef, entropy,
                                                      ent_coef, eps, grad, token_loss, flags, threadIdx.x, part, part_mx,
                                                      par, kp, sh);
    }
    if constexpr (TM) {
        if (kp.tm_chunks > 0) {   // every tensor-memory read has completed (tmem_wait_ld)
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncthreads();
            if (warp == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                             "r"(kTmemCols)
                             : "memory");
            }
        }
    }
}

template <int THREADS, int UNROLL, bool RECOMPUTE, bool ENT>
__global__ void __launch_bounds__(THREADS) loss_grad_warp(
    const acrl_bf16* __restrict__ logits, int64_t T, int V, int64_t ld, const int32_t* __restrict__ ids,
    const uint8_t* __restrict__ mask, const float* __restrict__ lse, const float* __restrict__ old_logp,
    const float* __restrict__ coef, const float* __restrict__ entropy, const float* __restrict__ ent_coef, float eps,
    acrl_bf16* __restrict__ grad, float* __restrict__ token_loss, int32_t* flags, int) {
    constexpr int NW = THREADS / 32;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int par = 0;
    grid_begin();
    for (int64_t t = int64_t(blockIdx.x) * NW + wid; t < T; t += int64_t(gridDim.x) * NW)
        grad_row<32, UNROLL, RECOMPUTE, ENT, false>(logits, t, V, ld, ids, mask, lse, old_logp, coef, entropy, ent_coef, eps,
                                             grad, token_loss, flags, lane, nullptr, nullptr, par,
                                             RowKeep{nullptr, 0, 0u, 0, nullptr}, RowShare{0, V >> 3});
}

// Scalar loss: sum of token losses in a fixed order, by one cluster of CTAs
// (no scratch memory: the partial sums meet in distributed shared memory).
// CTA c sums its contiguous block of the token losses: each thread adds float4
// groups (four values in fp32) into two alternating fp64 accumulators, so the
// loads pipeline and the fp64 adds are a quarter of the values; then a fixed
// CTA tree in fp64; CTA 0 adds the CTAs' sums in rank order.  The sum is bound
// by latency and by the fp64 pipe (two lanes a cycle per SM), which every warp
// pays five adds of the tree for, so the CTAs have as few warps as keep the
// loads in flight (1,024 losses: 5.4 us with 32 warps per CTA, 2.5 with 8).
constexpr int kSumCtas = 8;
constexpr int kSumThreads = 256;
constexpr int64_t kSumOneCta = 4096;  // up to this many losses are summed by one CTA

__global__ void __launch_bounds__(kSumThreads) loss_sum_kernel(const float* __restrict__ tl, int64_t T,
                                                               float* __restrict__ loss) {
    constexpr int THREADS = kSumThreads, NW = THREADS / 32;
    __shared__ double sh[NW];
    __shared__ double cta_sum;
    const int64_t c = blockIdx.x, ctas = gridDim.x;   // the launch is one cluster: the block index is the rank
    double s0 = 0.0, s1 = 0.0;
    grid_begin();
    if ((reinterpret_cast<uintptr_t>(tl) & 15u) == 0) {
        const int64_t n4 = T / 4;
        const int64_t per = (n4 + ctas - 1) / ctas;
        const int64_t lo = min(n4, c * per), hi = min(n4, lo + per);
        const float4* v = reinterpret_cast<const float4*>(tl);
        int64_t i = lo + threadIdx.x;
#pragma unroll 4
        for (; i + THREADS < hi; i += 2 * THREADS) {
            const float4 a = v[i], b = v[i + THREADS];
            s0 += double((a.x + a.y) + (a.z + a.w));
            s1 += double((b.x + b.y) + (b.z + b.w));
        }
        for (; i < hi; i += THREADS) {
            const float4 a = v[i];
            s0 += double((a.x + a.y) + (a.z + a.w));
        }
        if (c == ctas - 1)
            for (int64_t j = 4 * n4 + threadIdx.x; j < T; j += THREADS) s1 += tl[j];
    } else {
        const int64_t per = (T + ctas - 1) / ctas;
        const int64_t lo = min(T, c * per), hi = min(T, lo + per);
        for (int64_t j = lo + threadIdx.x; j < hi; j += THREADS) s0 += tl[j];
    }
    const double ws = warp_sum(s0 + s1);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = ws;
    __syncthreads();
    double total = 0.0;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int w = 0; w < NW; ++w) total += sh[w];
        cta_sum = total;
    }
    if (ctas > 1) {
        cluster_sync();   // every CTA's sum is in its shared memory
        if (c == 0 && threadIdx.x == 0)
            for (uint32_t k = 1; k < uint32_t(ctas); ++k) total += ld_peer_f64(&cta_sum, k);
    }
    if (c == 0 && threadIdx.x == 0) *loss = float(total);
    if (ctas > 1) cluster_sync();   // no CTA leaves while CTA 0 may still read its shared memory
}

acrl_status launch_loss_sum(const float* token_loss, int64_t T, float* loss, cudaStream_t s) {
    const int ctas = T <= kSumOneCta ? 1 : kSumCtas;
    return launch(loss_sum_kernel, ctas, kSumThreads, 0, ctas, s, token_loss, T, loss);
}

// out = bf16(grad * bf16(*scale)) over the rows' 16-byte vectors: the backward of
// a loss that something else scaled.  Bound by HBM (2 bytes in, 2 out per
// element).  A thread takes kScaleUnroll vectors a block's width apart, all
// loaded before the first is stored, and finds its row once by a division; a
// row of any length then costs no idle lanes.  4,992 rows of 20,011 columns: 58 us
// (6.9 TB/s, a plain copy of the buffer 59; an elementwise product of the
// strided view 208).
constexpr int kScaleThreads = 256, kScaleUnroll = 4;

__device__ __forceinline__ uint32_t scale_pair(uint32_t w, float s) {
    return pack_bf16x2(bf16_lo(w) * s, bf16_hi(w) * s);
}

__global__ void __launch_bounds__(kScaleThreads)
    scale_grad_kernel(const acrl_bf16* __restrict__ grad, int64_t T, int nvec, int64_t ld, const float* __restrict__ scale,
                      acrl_bf16* __restrict__ out, int64_t ldo) {
    grid_begin();
    const float f = *scale;
    if (f == 1.f) return;  // the caller keeps `grad`
    const float s = bf16_lo(pack_bf16x2(f, 0.f));
    const int64_t total = T * nvec, step = int64_t(gridDim.x) * kScaleThreads * kScaleUnroll;
    for (int64_t i = int64_t(blockIdx.x) * kScaleThreads * kScaleUnroll + threadIdx.x; i < total; i += step) {
        int64_t row = i / nvec;
        int64_t col = i - row * nvec;
        uint4 v[kScaleUnroll];
        uint4* dst[kScaleUnroll];
#pragma unroll
        for (int k = 0; k < kScaleUnroll; ++k) {
            dst[k] = nullptr;
            if (row < T) {
                v[k] = ld_stream(reinterpret_cast<const uint4*>(grad + row * ld) + col);
                dst[k] = reinterpret_cast<uint4*>(out + row * ldo) + col;
            }
            for (col += kScaleThreads; col >= nvec && row < T; col -= nvec) ++row;
        }
#pragma unroll
        for (int k = 0; k < kScaleUnroll; ++k)
            if (dst[k])
                st_stream(dst[k], make_uint4(scale_pair(v[k].x, s), scale_pair(v[k].y, s), scale_pair(v[k].z, s),
                                             scale_pair(v[k].w, s)));
    }
}

// Elements m .. m + 7 of the 16 in (lo, hi), m < 8.
__device__ __forceinline__ uint4 shift_elems(const uint4& lo, const uint4& hi, int m) {
    const uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
    uint32_t y[6], z[5];
#pragma unroll
    for (int i = 0; i < 6; ++i) y[i] = m & 4 ? w[i + 2] : w[i];
#pragma unroll
    for (int i = 0; i < 5; ++i) z[i] = m & 2 ? y[i + 1] : y[i];
    const int half = (m & 1) * 16;
    return make_uint4(__funnelshift_r(z[0], z[1], half), __funnelshift_r(z[1], z[2], half),
                      __funnelshift_r(z[2], z[3], half), __funnelshift_r(z[3], z[4], half));
}

// bf16 products of two pairs (one rounding each, as the fp32 product's).
__device__ __forceinline__ uint32_t mul_bf16x2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// The same product into rows without a gap whose length is no multiple of eight (the
// contiguous [T, V] tensor that a framework's own product is).  A lane makes the
// 16-byte vectors of the output as it lies in memory, so that a warp writes whole
// lines; one inside a row is shifted together from the vector of `grad` that holds its
// first column and the next one, which the next lane holds; one that holds a row's end,
// or the output's, goes element by element.  4,992 rows of 20,011 columns: 70 us (the
// next vector loaded again, through L1: 87; a row's vectors from its own start, so that
// warps share 32-byte sectors of the output: 81; a row end's elements all at once, whose
// registers cost residency: 86; a plain copy of the buffer 62; an elementwise product of
// the strided view 216).
constexpr int kDenseUnroll = 2;

__global__ void __launch_bounds__(kScaleThreads)
    scale_grad_dense_kernel(const acrl_bf16* __restrict__ grad, int64_t T, int V, int64_t ld,
                            const float* __restrict__ scale, acrl_bf16* __restrict__ out) {
    constexpr int U = kDenseUnroll, kApart = 8 * kScaleThreads;   // columns between two vectors of a thread
    const int lane = threadIdx.x & 31;
    grid_begin();
    const float f = *scale;
    if (f == 1.f) return;  // the caller keeps `grad`
    const uint32_t s = pack_bf16x2(f, f);
    const int64_t total = T * V, nvec = (total + 7) >> 3, step = int64_t(gridDim.x) * kScaleThreads * U;
    // a warp's lanes stay together, those beyond the end with row >= T
    for (int64_t i = int64_t(blockIdx.x) * kScaleThreads * U + threadIdx.x; i - lane < nvec; i += step) {
        int64_t row = i * 8 / V;
        int col = int(i * 8 - row * V);
        uint4 lo[U];
        int64_t rows[U];
        int cols[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            rows[k] = row;
            cols[k] = col;
            lo[k] = make_uint4(0u, 0u, 0u, 0u);
            if (row < T) lo[k] = ld_stream(reinterpret_cast<const uint4*>(grad + row * ld) + (col >> 3));
            col += kApart;
            const int over = col < V ? 0 : V >= kApart ? 1 : col / V;
            row += over;
            col -= over * V;
        }
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int64_t v = i + k * kScaleThreads;
            const acrl_bf16* src = grad + rows[k] * ld;
            const int c = cols[k], m = c & 7;
            const bool whole = rows[k] < T && c + 8 <= V;
            uint4 hi = make_uint4(__shfl_down_sync(0xffffffffu, lo[k].x, 1), __shfl_down_sync(0xffffffffu, lo[k].y, 1),
                                  __shfl_down_sync(0xffffffffu, lo[k].z, 1), __shfl_down_sync(0xffffffffu, lo[k].w, 1));
            // no next lane, or one that begins the next row; the vector holds column c + 7 at the latest
            if (whole && m && (lane == 31 || c + 8 == V)) hi = ld_stream(reinterpret_cast<const uint4*>(src) + (c >> 3) + 1);
            if (whole) {
                const uint4 x = shift_elems(lo[k], hi, m);
                st_stream(reinterpret_cast<uint4*>(out) + v, make_uint4(mul_bf16x2(x.x, s), mul_bf16x2(x.y, s),
                                                                        mul_bf16x2(x.z, s), mul_bf16x2(x.w, s)));
            } else if (v < nvec) {
                int at = c;
#pragma unroll 1
                for (int64_t j = v * 8; j < min(total, v * 8 + 8); ++j) {
                    out[j] = acrl_bf16(mul_bf16x2(src[at], s) & 0xffffu);
                    if (++at == V) {
                        at = 0;
                        src += ld;
                    }
                }
            }
        }
    }
}

template <bool RECOMPUTE, bool ENT>
acrl_status launch_loss_grad(const acrl_bf16* logits, int64_t T, int V, int64_t ld, const int32_t* ids,
                             const uint8_t* mask, const float* lse, const float* old_logp, const float* coef,
                             const float* entropy, const float* ent_coef, float eps, acrl_bf16* grad,
                             float* token_loss, int32_t* flags, cudaStream_t s) {
    auto run = [&](auto kernel, int64_t rows_per_cta, int threads, int keep_vecs, int shares = 1) {
        const int smem = 16 * min(V >> 3, keep_vecs);
        // the limit belongs to the kernel, not to the call: always its largest, so that threads with different V agree
        if (keep_vecs > 0 &&
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 16 * keep_vecs) != cudaSuccess)
            return ACRL_ERR_CUDA;
        return launch(kernel, grid_for(rows_per_cta, T * shares), threads, size_t(smem), 0, s, logits, T, V, ld, ids, mask,
                      lse, old_logp, coef, entropy, ent_coef, eps, grad, token_loss, flags, shares);
    };
    constexpr int U = kCtaUnroll;
    if constexpr (RECOMPUTE) {
        const int nvec = V >> 3;
        if (V < kRecomputeCtaMinV) return run(loss_grad_warp<64, U, true, ENT>, 2, 64, 0);
        if (V <= kLeastMaxV) return run(loss_grad_cta<kLeastThreads, U, true, ENT>, 1, kLeastThreads, kLeastKeepVecs);
        if (nvec <= kTinyKeepVecs) return run(loss_grad_cta<kTinyThreads, U, true, ENT>, 1, kTinyThreads, kTinyKeepVecs);
        if (nvec <= kSmallMaxVecs)
            return run(loss_grad_cta<kSmallThreads, U, true, ENT>, 1, kSmallThreads, kSmallKeepVecs);
        if (nvec >= kTmemMinVecs) return run(loss_grad_cta<kCtaThreads, U, true, ENT, true>, 1, kCtaThreads, kKeepVecs);
        return run(loss_grad_cta<kCtaThreads, U, true, ENT>, 1, kCtaThreads, kKeepVecs);
    } else {
        if (V >= kShareRowMinV) {
            const int shares = (V >> 3) / kShareVecs;
            if (T <= kMaxGrid / shares)
                return run(loss_grad_cta<kShareThreads, U, false, ENT, false, true>, 1, kShareThreads, 0, shares);
            return run(loss_grad_cta<kWideThreads, U, false, ENT>, 1, kWideThreads, 0);
        }
        if (V >= 512 * kStreamStep) return run(loss_grad_cta<512, U, false, ENT>, 1, 512, 0);
        if (V >= 384 * kStreamStep) return run(loss_grad_cta<384, U, false, ENT>, 1, 384, 0);
        if (V >= 256 * kStreamStep) return run(loss_grad_cta<256, U, false, ENT>, 1, 256, 0);
        const bool many = T >= kManyRows;
        if (V >= 128 * kStreamStep && !many) return run(loss_grad_cta<128, U, false, ENT>, 1, 128, 0);
        if (V >= (many ? 128 : 64) * kStreamStep) return run(loss_grad_cta<64, U, false, ENT>, 1, 64, 0);
        return run(loss_grad_warp<64, U, false, ENT>, 2, 64, 0);
    }
}

}  // namespace
}  // namespace acrl

using namespace acrl;

extern "C" acrl_status acrl_loss_grad_logits(const acrl_bf16* logits, int64_t T, int64_t V, int64_t ld,
                                             const int32_t* ids, const uint8_t* mask, const float* lse,
                                             const float* old_logp, const float* coef, const float* entropy,
                                             const float* ent_coef, float clip_eps, acrl_bf16* grad,
                                             float* token_loss, float* loss, int32_t* dev_flags, acrl_stream stream) {
    if (T < 0 || V < 1 || V > kMaxVocab || ld < V || (ld & 7) != 0) return ACRL_ERR_INVALID_ARG;
    if (!(clip_eps >= 0.f && clip_eps < 1.f)) return ACRL_ERR_INVALID_ARG;
    if (!loss || !dev_flags) return ACRL_ERR_INVALID_ARG;
    if ((entropy == nullptr) != (ent_coef == nullptr)) return ACRL_ERR_INVALID_ARG;
    if (T > 0 && (!logits || !ids || !coef || !grad || !token_loss)) return ACRL_ERR_INVALID_ARG;
    if (T > 0 && (!aligned16(logits) || !aligned16(grad))) return ACRL_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (T > 0) {
        const int v = int(V);
        const bool ent = ent_coef != nullptr;
        acrl_status st;
        if (lse && !ent)
            st = launch_loss_grad<false, false>(logits, T, v, ld, ids, mask, lse, old_logp, coef, entropy, ent_coef,
                                                clip_eps, grad, token_loss, dev_flags, s);
        else if (lse && ent)
            st = launch_loss_grad<false, true>(logits, T, v, ld, ids, mask, lse, old_logp, coef, entropy, ent_coef,
                                               clip_eps, grad, token_loss, dev_flags, s);
        else if (!ent)
            st = launch_loss_grad<true, false>(logits, T, v, ld, ids, mask, lse, old_logp, coef, entropy, ent_coef,
                                               clip_eps, grad, token_loss, dev_flags, s);
        else
            st = launch_loss_grad<true, true>(logits, T, v, ld, ids, mask, lse, old_logp, coef, entropy, ent_coef,
                                              clip_eps, grad, token_loss, dev_flags, s);
        if (st != ACRL_OK) return st;
    }
    return launch_loss_sum(token_loss, T, loss, s);
}

extern "C" acrl_status acrl_reduce_loss(const float* token_loss, int64_t T, float* loss, acrl_stream stream) {
    if (T < 0 || !loss || (T > 0 && !token_loss)) return ACRL_ERR_INVALID_ARG;
    return launch_loss_sum(token_loss, T, loss, reinterpret_cast<cudaStream_t>(stream));
}

extern "C" acrl_status acrl_scale_grad(const acrl_bf16* grad, int64_t T, int64_t V, int64_t ld, const float* scale,
                                       acrl_bf16* out, int64_t ldo, acrl_stream stream) {
    if (T < 0 || V < 1 || V > kMaxVocab || ld < V || (ld & 7) != 0 || ldo < V || (ldo != V && (ldo & 7) != 0))
        return ACRL_ERR_INVALID_ARG;
    if (T == 0) return ACRL_OK;
    if (!grad || !scale || !out || !aligned16(grad) || !aligned16(out)) return ACRL_ERR_INVALID_ARG;
    const int nvec = int((V + 7) >> 3);
    // at most kMaxGrid CTAs: the kernel loops
    const int64_t per_cta = kScaleThreads * kScaleUnroll;
    const int64_t rows = T < kMaxGrid ? T : kMaxGrid;
    if ((ldo & 7) != 0)
        return launch(scale_grad_dense_kernel, grid_for(kScaleThreads * kDenseUnroll, rows * nvec), kScaleThreads, 0, 0,
                      reinterpret_cast<cudaStream_t>(stream), grad, T, int(V), ld, scale, out);
    return launch(scale_grad_kernel, grid_for(per_cta, rows * nvec), kScaleThreads, 0, 0,
                  reinterpret_cast<cudaStream_t>(stream), grad, T, nvec, ld, scale, out, ldo);
}
