// acrl_token_stats: one streaming pass over pi's bf16 logits per token row
// giving the log-sum-exp, the sampled token's log-prob and the entropy.
//
// Each row is read exactly once from HBM in 16-byte loads that L1 does not keep.
// A team of threads (eight or sixteen lanes for the shortest rows, a warp for
// other short rows, the whole CTA for vocabulary-size rows) owns a row; every
// thread keeps an online base-2 state (max, sum 2^(u-U), sum 2^(u-U)(u-U))
// over its strided share of the row, and the team merges the states with a
// fixed butterfly/tree order, so results are bit-reproducible run to run.
//
// A thread's loads go straight into registers (one step of four in flight) or
// through a ring of kDepth steps in its own slots of shared memory; the fold is
// the same, so which one a call takes does not show in its results.
#include "acrl_device.cuh"
#include "acrl_host.h"
#include "row_lse.cuh"

namespace acrl {
namespace {

// A thread's share of its team's row: straight into registers (DEPTH = 0), or
// through a ring of DEPTH steps.
template <int TEAM, int UNROLL, int THREADS, int DEPTH>
__device__ __forceinline__ LseAcc team_partial(const acrl_bf16* row, int V, int tid, float& mx, uint4* ring) {
    if constexpr (DEPTH == 0)
        return row_partial<TEAM, UNROLL>(row, V, tid, mx);
    else
        return row_partial_ring<TEAM, UNROLL, THREADS, DEPTH>(row, V, tid, mx, ring + threadIdx.x);
}

// The register path lives on residency: 48 registers, 1,280 threads per SM.
template <int THREADS, int DEPTH>
constexpr int kMinCtas = DEPTH == 0 && THREADS <= 128 ? 1280 / THREADS : 1;

// A team's states as one, brought to the common maximum (lse_at).
// The lengths of rows whose team has a level more than eight lanes or two warps have
// meet so (sixteen lanes, and four warps up to kMeetMaxV columns): merged, they came out
// further from float64 (rms) than with the smaller team, meeting they are closer.
// Entropy of normal logits (sd 2), V = 4,096: eight lanes 3.74e-7, sixteen merged
// 3.79e-7, meeting 3.49e-7; V = 57,344: two warps 5.10e-7, four merged 5.28e-7, meeting
// 4.77e-7; at the same speed.
template <int LANES>
__device__ __forceinline__ LseAcc lanes_meet(LseAcc a) {
    float U = a.U;
#pragma unroll
    for (int m = LANES / 2; m >= 1; m >>= 1) U = fmaxf(U, __shfl_xor_sync(0xffffffffu, U, m));
    a = lse_at(a, U);
#pragma unroll
    for (int m = LANES / 2; m >= 1; m >>= 1) {
        a.s0 += __shfl_xor_sync(0xffffffffu, a.s0, m);
        a.s1 += __shfl_xor_sync(0xffffffffu, a.s1, m);
    }
    return a;
}

// A whole CTA per row (vocabulary-size rows).
template <int THREADS, int UNROLL, int DEPTH, bool MEET>
__global__ void __launch_bounds__(THREADS, kMinCtas<THREADS, DEPTH>)
    token_stats_cta(const acrl_bf16* __restrict__ logits, int64_t T, int V, int64_t ld,
                    const int32_t* __restrict__ ids, const uint8_t* __restrict__ mask, float* __restrict__ lse,
                    float* __restrict__ logp, float* __restrict__ ent, int32_t* flags) {
    constexpr int NW = THREADS / 32;
    __shared__ LseAcc part[NW];
    __shared__ float pmax[NW];
    extern __shared__ uint4 ring[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    grid_begin();
    for (int64_t t = blockIdx.x; t < T; t += gridDim.x) {
        if (mask && mask[t] == 0) {
            if (threadIdx.x == 0) lse[t] = logp[t] = ent[t] = 0.f;
            continue;
        }
        const acrl_bf16* row = logits + t * ld;
        RowTarget tgt{0.f, false};
        if (threadIdx.x == 0) tgt = row_target(row, V, ids[t]);
        float mx;
        LseAcc acc = team_partial<THREADS, UNROLL, THREADS, DEPTH>(row, V, threadIdx.x, mx, ring);
        acc = MEET ? lanes_meet<32>(acc) : warp_lse(acc);
        mx = warp_max(mx);
        if (lane == 0) {
            part[wid] = acc;
            pmax[wid] = mx;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            LseAcc r = part[0];
            float m = pmax[0];
            if (MEET) {
#pragma unroll
                for (int w = 1; w < NW; ++w) r.U = fmaxf(r.U, part[w].U);
                r = lse_at(part[0], r.U);
            }
#pragma unroll
            for (int w = 1; w < NW; ++w) {
                if (MEET) {
                    const LseAcc a = lse_at(part[w], r.U);
                    r.s0 += a.s0;
                    r.s1 += a.s1;
                } else {
                    r = lse_merge(r, part[w]);
                }
                m = fmaxf(m, pmax[w]);
            }
            row_outputs(r, m, tgt, lse, logp, ent, t, flags);
        }
        __syncthreads();
    }
}

// One warp per row (short rows); THREADS/32 rows per CTA.
template <int THREADS, int UNROLL, int DEPTH>
__global__ void __launch_bounds__(THREADS) token_stats_warp(const acrl_bf16* __restrict__ logits, int64_t T, int V,
                                                            int64_t ld, const int32_t* __restrict__ ids,
                                                            const uint8_t* __restrict__ mask, float* __restrict__ lse,
                                                            float* __restrict__ logp, float* __restrict__ ent,
                                                            int32_t* flags) {
    constexpr int NW = THREADS / 32;
    extern __shared__ uint4 ring[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    grid_begin();
    for (int64_t t = int64_t(blockIdx.x) * NW + wid; t < T; t += int64_t(gridDim.x) * NW) {
        if (mask && mask[t] == 0) {
            if (lane == 0) lse[t] = logp[t] = ent[t] = 0.f;
            continue;
        }
        const acrl_bf16* row = logits + t * ld;
        RowTarget tgt{0.f, false};
        if (lane == 0) tgt = row_target(row, V, ids[t]);
        float mx;
        LseAcc acc = team_partial<32, UNROLL, THREADS, DEPTH>(row, V, lane, mx, ring);
        acc = warp_lse(acc);
        mx = warp_max(mx);
        if (lane == 0) row_outputs(acc, mx, tgt, lse, logp, ent, t, flags);
    }
}

// The shortest rows: LANES lanes per row, 32 / LANES rows per warp at a time.
// The team merges its states over log2(LANES) shuffle levels instead of five,
// which matters where the merges' exponentials are a large share of the row's
// (V = 2,048: 0.75 -> 0.94 of the copy rate with 8 lanes).  Every lane takes part
// in the shuffles, whether its row is masked or not.
template <int LANES>
__device__ __forceinline__ LseAcc team_lse(LseAcc a) {
    if constexpr (LANES == 16) return lanes_meet<LANES>(a);
#pragma unroll
    for (int m = LANES / 2; m >= 1; m >>= 1) a = lse_merge(a, shfl_xor(a, m));
    return a;
}

template <int LANES>
__device__ __forceinline__ float team_max(float v) {
#pragma unroll
    for (int m = LANES / 2; m >= 1; m >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, m));
    return v;
}

template <int THREADS, int UNROLL, int LANES, int DEPTH>
__global__ void __launch_bounds__(THREADS) token_stats_team(const acrl_bf16* __restrict__ logits, int64_t T, int V,
                                                            int64_t ld, const int32_t* __restrict__ ids,
                                                            const uint8_t* __restrict__ mask, float* __restrict__ lse,
                                                            float* __restrict__ logp, float* __restrict__ ent,
                                                            int32_t* flags) {
    constexpr int NW = THREADS / 32, RPW = 32 / LANES;
    extern __shared__ uint4 ring[];
    static_assert(LANES >= 2 && LANES <= 32 && (LANES & (LANES - 1)) == 0, "lanes per row");
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, tl = lane % LANES;
    grid_begin();
    for (int64_t base = (int64_t(blockIdx.x) * NW + wid) * RPW; base < T; base += int64_t(gridDim.x) * NW * RPW) {
        const int64_t t = base + lane / LANES;
        const bool in = t < T;
        const bool live = in && !(mask && mask[t] == 0);
        const acrl_bf16* row = logits + (in ? t : 0) * ld;
        RowTarget tgt{0.f, false};
        if (tl == 0 && live) tgt = row_target(row, V, ids[t]);
        LseAcc acc = lse_empty();
        float mx = -INFINITY;
        if (live) acc = team_partial<LANES, UNROLL, THREADS, DEPTH>(row, V, tl, mx, ring);
        acc = team_lse<LANES>(acc);
        mx = team_max<LANES>(mx);
        if (tl == 0 && in) {
            if (live)
                row_outputs(acc, mx, tgt, lse, logp, ent, t, flags);
            else
                lse[t] = logp[t] = ent[t] = 0.f;
        }
    }
}

// Rows up to kTeamRowMaxV columns are shared by eight lanes each, up to
// kTeam16RowMaxV by sixteen, up to kWarpRowMaxV by a warp, up to kMidRowMaxV
// (80 KB) by two warps, longer ones by four: many independent rows in flight per SM
// and a short end-of-row merge (measured best of teams of 8 to 1,024 threads).  The
// line depends on V alone, so that a row's result does not depend on the batch it
// is in.  Where they lie, us: V = 4,096, T = 1,024 / 8,000 / 30,000: eight lanes
// 6.0 / 14.2 / 43.1, sixteen 3.9 / 14.1 / 40.8, a warp 3.3 / 15.3 / 43.8; V = 3,333:
// eight 5.9 / 12.9 / 35.7, sixteen 3.9 / 13.9 / 36.4; V = 5,003: sixteen 5.2 / 18.9 /
// 51.9, a warp 4.4 / 19.3 / 56.9.  V = 49,152, T = 300 / 1,340 / 4,000 / 16,000: two
// warps 10.2 / 24.7 / 63.8 / 225, four 8.3 / 22.0 / 60.3 / 219; V = 40,000, T = 400 /
// 3,000 / 10,000: two 10.8 / 39.3 / 123, four 8.9 / 40.8 / 119.
constexpr int64_t kTeamRowMaxV = 3584, kTeam16RowMaxV = 4608, kMidRowMaxV = 40960, kMeetMaxV = 65536;
constexpr int kUnroll = 4;

// Steps of the ring: with few rows per SM, one step of loads per thread leaves
// the memory system idle between steps (V = 151,936, T = 64: 30 us in
// registers, 19 / 14.4 / 13.8 us with rings of 2 / 3 / 4 steps; T = 408: 34
// against 26 / 23 / 23; V = 4,096, T = 1,024: 15 against 6.6 / 6.5 / 6.3).
constexpr int kDepth = 3;

// Ring or registers?  The line is drawn in 128-thread teams per SM (q: tenths).
// - Few teams per SM: the ring, up to 2.3 x (above).
// - 5.2 to 10.4 per SM: all of them fit in one wave of the register path (48
//   registers), not in one of the ring's (80); V = 151,936, T = 1,216: 58 us in
//   registers against 67, T = 1,600 (past the wave): 92 against 77; V = 49,152,
//   T = 1,000: 17.4 against 22.8; a warp per row, V = 16,384, T = 6,000: 34.1
//   against 37.9.
// - Many: the ring for rows of a warp or less (V = 16,384, T = 65,536: 296 us
//   against 317; V = 8,192: 153 against 162; V = 4,096: 82 against 88).  Two warps
//   a row: registers where the row's last step is a large part of it (V = 20,011: a
//   step of 12,000 rows 254 us against 257, of 40,000 750 against 762) and up to
//   some 2.5 waves (V = 32,000, 5,000 rows: 174 against 181), except just past one
//   wave (V = 32,000, T = 3,500: 45 against 40); else the ring (V = 32,000, steps of
//   16,000 and 38,000 rows: 485 and 1,084 against 480 and 1,072).  Four warps a row:
//   the ring (V = 72,000, T = 8,000: 181 us in registers, 170; V = 151,936, T =
//   8,000: 361 / 351), except in the last third of the register path's second wave
//   (T = 3,000: V = 128,256 115.5 in registers, 121.4 with the ring; V = 262,144 223
//   / 236; T = 2,400: 188 / 186; T = 3,100, past that wave: 258 / 234) and for the
//   shorter of many rows that do not begin on 128-byte lines (T = 40,000: V = 40,968
//   465 / 475, V = 45,064 509 / 523, but V = 45,184 511 / 510; T = 12,000 and V =
//   43,008: 146 / 141).
bool use_ring(int64_t T, int team, int V, int64_t ld) {
    constexpr int64_t kSms = 152;
    const int64_t q = T >= (int64_t(1) << 40) ? INT64_MAX : T * team * 10 / (128 * kSms);
    if (team <= 16) return true;
    if (q < 52) return true;
    if (team == 64) return V >= 28672 ? q > 400 || (q > 104 && q < 140) : q > 104 && q < 140;
    if (team == 128 && ((q > 168 && q <= 200) || (ld % 64 != 0 && V < 57344 && q > 1400))) return false;
    return q > 104;
}

}  // namespace

}  // namespace acrl

using namespace acrl;

extern "C" acrl_status acrl_token_stats(const acrl_bf16* logits, int64_t T, int64_t V, int64_t ld,
                                        const int32_t* ids, const uint8_t* mask, float* lse, float* logp,
                                        float* entropy, int32_t* dev_flags, acrl_stream stream) {
    if (T < 0 || V < 1 || V > kMaxVocab || ld < V || (ld & 7) != 0) return ACRL_ERR_INVALID_ARG;
    if (T == 0) return ACRL_OK;
    if (!logits || !ids || !lse || !logp || !entropy || !dev_flags) return ACRL_ERR_INVALID_ARG;
    if (!aligned16(logits)) return ACRL_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int v = int(V);
    // `depth` steps of kUnroll 16-byte slots per thread of dynamic shared memory (at most 24 KB)
    auto run = [&](auto kernel, int threads, int depth, int64_t rows_per_cta) {
        return launch(kernel, grid_for(rows_per_cta, T), threads, size_t(threads) * kUnroll * depth * 16, 0, s, logits, T,
                      v, ld, ids, mask, lse, logp, entropy, dev_flags);
    };
    const int team = V <= kTeamRowMaxV     ? 8
                     : V <= kTeam16RowMaxV ? 16
                     : V <= kWarpRowMaxV   ? 32
                     : V <= kMidRowMaxV    ? 64
                                           : 128;
    const bool ring = use_ring(T, team, v, ld);
    if (team == 8) return run(token_stats_team<64, kUnroll, 8, kDepth>, 64, kDepth, 8);
    if (team == 16) return run(token_stats_team<64, kUnroll, 16, kDepth>, 64, kDepth, 4);
    if (team == 32)
        return ring ? run(token_stats_warp<64, kUnroll, kDepth>, 64, kDepth, 2)
                    : run(token_stats_warp<256, kUnroll, 0>, 256, 0, 8);
    if (team == 64)
        return ring ? run(token_stats_cta<64, kUnroll, kDepth, false>, 64, kDepth, 1)
                    : run(token_stats_cta<64, kUnroll, 0, false>, 64, 0, 1);
    if (V <= kMeetMaxV)
        return ring ? run(token_stats_cta<128, kUnroll, kDepth, true>, 128, kDepth, 1)
                    : run(token_stats_cta<128, kUnroll, 0, true>, 128, 0, 1);
    return ring ? run(token_stats_cta<128, kUnroll, kDepth, false>, 128, kDepth, 1)
                : run(token_stats_cta<128, kUnroll, 0, false>, 128, 0, 1);
}
