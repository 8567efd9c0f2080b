// The O(T) part of the path: per-token log-ratio and distance, masked
// per-response / per-prompt / batch aggregates, GRPO advantages and the
// adaptive controller with its importance weights.
//
// One CTA (or a small cluster of CTAs) per response does the segmented
// reductions; single-CTA kernels finalise prompts and the batch.  Every
// reduction has a fixed order (strided per-thread partials, then a fixed warp
// tree and warp-order sum) and no floating-point atomics, so the results are
// bit-reproducible.
//
// What bounds these kernels is latency and the fp64 pipe (two lanes a cycle
// per SM), not their ~25 bytes per token: counts and maxima therefore travel
// as integers, sums share one warp tree, scalar fp64 divisions run once per
// CTA with a different quotient in each lane, and warps without data skip
// their trees.
#include <cmath>

#include "acrl_device.cuh"
#include "acrl_host.h"

namespace acrl {
namespace {

constexpr int kSeqThreads = 256;
constexpr int kSeqUnroll = 4;    // tokens per thread in flight
constexpr int kFinThreads = 512;
constexpr int kSeqCtas = 304, kSeqTokens = 256;  // see ctas_per_response
constexpr int kGrpoThreads = 128;
constexpr int kGrpoTeamPrompts = 1024;  // up to this many prompts are shared by eight lanes each
constexpr int kFinSeqs = 2048;   // responses whose mean distance the batch kernel keeps in shared memory

__device__ __forceinline__ bool seq_range(const int64_t* so, int i, int64_t T, int64_t& lo, int64_t& hi) {
    lo = so[i];
    hi = so[i + 1];
    return lo >= 0 && lo <= hi && hi <= T;
}

// Index g with goff[g] <= i < goff[g+1], or -1; the whole warp searches, 32
// probes at a time (one step for up to 32 prompts, two for up to 1,024).
__device__ __forceinline__ int group_of(const int32_t* goff, int Gn, int i) {
    if (Gn <= 0) return -1;
    const int lane = threadIdx.x & 31;
    int lo = 0, n = Gn;  // invariant: answer in [lo, lo + n)
    while (n > 1) {
        const int step = (n + 31) >> 5;
        const int64_t at = int64_t(lane) * step;
        const unsigned le = __ballot_sync(0xffffffffu, at < n && goff[lo + (at < n ? int(at) : 0)] <= i);
        const int k = le ? 31 - __clz(le) : 0;   // the last probe at or before i
        lo += k * step;
        n = min(step, n - k * step);
    }
    return (goff[lo] <= i && i < goff[lo + 1]) ? lo : -1;
}

// |exp(a) - exp(b)| without cancellation when a and b are close.
__device__ __forceinline__ float prob_distance(float a, float b) {
    const float l = a - b;
    return fabsf(l) < 0.5f ? expf(b) * fabsf(expm1f(l)) : fabsf(expf(a) - expf(b));
}

// One CTA's part of a response's sums.
struct SeqPart {
    double sum[4];  // d, d^2, lr, H
    int n;
    uint32_t max_d; // bits of a non-negative float
};

// The tokens of one thread in its part of a response (t0, t0 + stride, ... below
// hi): lr and d, and the sums of its warp, which land in sum[0..3], *cnt and
// *max_d.  l0 and m0 receive lr and the mask of the thread's first kSeqUnroll
// tokens.  Returns whether a log-prob was NaN.
__device__ __forceinline__ bool stats_tokens(const float* logp_pi, const float* logp_mu, const uint8_t* mask,
                                             const float* entropy, float* lr, float* d, int64_t t0, int64_t hi,
                                             int64_t stride, float (&l0)[kSeqUnroll], bool (&m0)[kSeqUnroll], double* sum,
                                             int* cnt, uint32_t* max_d) {
    constexpr int U = kSeqUnroll;
    const int lane = threadIdx.x & 31;
    int n = 0;
    double sd = 0.0, sd2 = 0.0, slr = 0.0, sH = 0.0;
    float mxd = 0.f;
    bool nan_lr = false, first = true;
#pragma unroll
    for (int k = 0; k < U; ++k) {
        l0[k] = 0.f;
        m0[k] = false;
    }
    for (; t0 < hi; t0 += U * stride) {
        float a[U], b[U], h[U];
        bool m[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int64_t t = t0 + k * stride;
            const bool in = t < hi;
            m[k] = in && (mask ? mask[t] != 0 : true);
            a[k] = in ? logp_pi[t] : 0.f;
            b[k] = in ? logp_mu[t] : 0.f;
            h[k] = in && entropy ? entropy[t] : 0.f;
        }
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int64_t t = t0 + k * stride;
            if (t >= hi) break;
            float l = 0.f, dd = 0.f;
            if (m[k]) {
                l = a[k] - b[k];
                nan_lr |= isnan(l);  // a NaN log-prob on either side
                dd = prob_distance(a[k], b[k]);
                ++n;
                const double dd64 = dd;
                sd += dd64;
                sd2 += dd64 * dd64;
                slr += l;
                if (entropy) sH += h[k];
                mxd = fmaxf(mxd, dd);
            }
            lr[t] = l;
            d[t] = dd;
            if (first) {
                l0[k] = l;
                m0[k] = m[k];
            }
        }
        first = false;
    }
    const double s = warp_sum4(sd, sd2, slr, sH);
    n = __reduce_add_sync(0xffffffffu, n);
    mxd = warp_max_nonneg(mxd);
    if ((lane & 7) == 0) sum[lane >> 3] = s;
    if (lane == 0) {
        *cnt = n;
        *max_d = __float_as_uint(mxd);
    }
    return nan_lr;
}

// A part's sums from its warps' (one warp): value k in lane k, in warp order.
template <int NW>
__device__ __forceinline__ void part_sums(const double* sh, const int* sh_n, const uint32_t* sh_max, double* sum, int& n,
                                          uint32_t& max_d) {
    const int lane = threadIdx.x & 31;
    double s = 0.0;
    if (lane < 4)
#pragma unroll
        for (int w = 0; w < NW; ++w) s += sh[w * 4 + lane];
    const int cnt = __reduce_add_sync(0xffffffffu, lane < NW ? sh_n[lane] : 0);
    const uint32_t mx = __reduce_max_sync(0xffffffffu, lane < NW ? sh_max[lane] : 0u);
    if (lane < 4) sum[lane] = s;
    if (lane == 0) {
        n = cnt;
        max_d = mx;
    }
}

// K2a: per-token lr and d, per-response sums.  A cluster of CTAs per response
// (one CTA where there are enough responses to fill the chip); CTA r takes
// tokens r kSeqThreads + tid of every round of the cluster's threads, and rank
// 0 adds the CTAs' sums in rank order.  A ninth warp finds the response's
// prompt meanwhile.
__global__ void __launch_bounds__(kSeqThreads + 32) seq_stats_kernel(
    const float* __restrict__ logp_pi, const float* __restrict__ logp_mu, const uint8_t* __restrict__ mask,
    int64_t T, const int64_t* __restrict__ so, int S, const int32_t* __restrict__ goff, int Gn,
    const float* __restrict__ entropy, float* __restrict__ lr, float* __restrict__ d, acrl_seq_stats* seq,
    int32_t* flags) {
    constexpr int NW = kSeqThreads / 32, U = kSeqUnroll;
    __shared__ double sh[NW * 4];
    __shared__ int sh_n[NW];
    __shared__ uint32_t sh_max[NW];
    __shared__ int sh_group;
    __shared__ SeqPart part;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nct = int(cluster_size()), rank = int(cluster_rank());
    const int i = int(blockIdx.x) / nct;
    grid_begin();
    if (wid == NW) {
        if (rank == 0) {
            const int g = group_of(goff, Gn, i);
            if (lane == 0) sh_group = g;
        }
    } else {
        int64_t lo, hi;
        if (!seq_range(so, i, T, lo, hi)) {
            if (rank == 0 && threadIdx.x == 0) raise_flag(flags, ACRL_FLAG_BAD_OFFSETS);
            lo = hi = 0;
        }
        float l0[U];
        bool m0[U];
        const bool nan_lr = stats_tokens(logp_pi, logp_mu, mask, entropy, lr, d, lo + rank * kSeqThreads + threadIdx.x, hi,
                                         int64_t(nct) * kSeqThreads, l0, m0, sh + wid * 4, sh_n + wid, sh_max + wid);
        if (nan_lr) raise_flag(flags, ACRL_FLAG_NONFINITE);
    }
    __syncthreads();
    if (wid == 0) {
        part_sums<NW>(sh, sh_n, sh_max, part.sum, part.n, part.max_d);
        __syncwarp();
    }
    if (nct > 1) cluster_sync();  // every CTA's part is in its shared memory
    if (rank == 0 && wid == 0) {
        double s = lane < 4 ? part.sum[lane] : 0.0;
        int n = lane == 0 ? part.n : 0;
        uint32_t mx = lane == 0 ? part.max_d : 0u;
        if (nct > 1) {
            if (lane < 4)
                for (int r = 1; r < nct; ++r) s += ld_peer_f64(&part.sum[lane], uint32_t(r));
            if (lane > 0 && lane < nct) {
                n = int(ld_peer_u32(&part.n, uint32_t(lane)));
                mx = ld_peer_u32(&part.max_d, uint32_t(lane));
            }
            n = __reduce_add_sync(0xffffffffu, n);
            mx = __reduce_max_sync(0xffffffffu, mx);
        }
        const double sd2 = __shfl_sync(0xffffffffu, s, 1), slr = __shfl_sync(0xffffffffu, s, 2),
                     sH = __shfl_sync(0xffffffffu, s, 3);
        if (lane == 0) {
            acrl_seq_stats o;
            o.n = n;
            o.group = sh_group;
            o.mean_d = n ? float(div64(s, n)) : 0.f;
            o.max_d = __uint_as_float(mx);
            o.sum_d = s;
            o.sum_d2 = sd2;
            o.sum_lr = slr;
            o.sum_H = sH;
            o.sum_w = 0.0;
            o.n_trunc = 0;
            o.alpha = 0.f;
            seq[i] = o;
        }
    }
    if (nct > 1) cluster_sync();  // no CTA leaves while rank 0 may still read its shared memory
}

// The batch statistics from the sums over responses and prompts (value k of d,
// d^2, H, lr and Y_g in lane k); one warp.
__device__ __forceinline__ void write_batch(double s, long long N, int sv, int qv, float dmax, acrl_batch_stats* batch) {
    const int lane = threadIdx.x & 31;
    // 1 / N in lane 0, Y_mean in lane 4
    const double den = lane == 4 ? double(qv) : double(N);
    const double q = den > 0.0 ? div64(lane == 4 ? s : 1.0, den) : 0.0;
    const double inv = __shfl_sync(0xffffffffu, q, 0), ymean = __shfl_sync(0xffffffffu, q, 4);
    const double mean = s * inv;  // lanes 0..3: the token means
    const double d_mean = __shfl_sync(0xffffffffu, mean, 0), d2_mean = __shfl_sync(0xffffffffu, mean, 1),
                 H_mean = __shfl_sync(0xffffffffu, mean, 2), lr_mean = __shfl_sync(0xffffffffu, mean, 3);
    const double ysum = __shfl_sync(0xffffffffu, s, 4);
    if (lane == 0) {
        acrl_batch_stats b;
        b.n_tokens = N;
        b.n_seqs_valid = sv;
        b.n_groups_valid = qv;
        b.d_mean = d_mean;
        b.d_max = double(dmax);
        const double var = fma(-d_mean, d_mean, d2_mean);
        b.d_std = var > 0.0 ? sqrt64(var) : 0.0;
        b.Y_sum = ysum;
        b.Y_mean = ymean;
        b.H_mean = H_mean;
        b.lr_mean = lr_mean;
        b.X = b.trunc_frac = b.w_mean = b.alpha_mean = 0.0;
        *batch = b;
    }
}

// K2b: prompt statistics and batch statistics; also checks the offsets.  One CTA.
__device__ __forceinline__ void finalize_seqs(int64_t T, const int64_t* __restrict__ so, int S,
                                              const int32_t* __restrict__ goff, int Gn,
                                              const acrl_seq_stats* __restrict__ seq, acrl_group_stats* grp,
                                              acrl_batch_stats* batch, int32_t* flags) {
    constexpr int NW = kFinThreads / 32;
    __shared__ double sh_D[kFinSeqs];  // D_i, and the valid tokens of response i
    __shared__ int sh_n[kFinSeqs];
    __shared__ double sh[NW * 5];
    __shared__ long long sh_N[NW];
    __shared__ int sh_sv[NW], sh_qv[NW];
    __shared__ float sh_max[NW];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const bool keep = S <= kFinSeqs;
    bool bad = false;
    long long N = 0;
    int sv = 0;
    double sd = 0.0, sd2 = 0.0, sH = 0.0, slr = 0.0;
    float dmax = 0.f;
    for (int i = threadIdx.x; i < S; i += kFinThreads) {
        bad |= so[i] > so[i + 1];
        const int n = seq[i].n;
        const double s = seq[i].sum_d;
        N += n;
        sv += n > 0;
        sd += s;
        sd2 += seq[i].sum_d2;
        sH += seq[i].sum_H;
        slr += seq[i].sum_lr;
        dmax = fmaxf(dmax, seq[i].max_d);
        if (keep) {
            sh_n[i] = n;
            sh_D[i] = n > 0 ? div64(s, n) : 0.0;
        }
    }
    for (int g = threadIdx.x; g < Gn; g += kFinThreads) bad |= goff[g] > goff[g + 1];
    if (threadIdx.x == 0) bad |= so[0] != 0 || so[S] != T || (Gn > 0 ? (goff[0] != 0 || goff[Gn] != S) : S != 0);
    if (bad) raise_flag(flags, ACRL_FLAG_BAD_OFFSETS);
    __syncthreads();

    int qv = 0;
    double ysum = 0.0;
    for (int g = threadIdx.x; g < Gn; g += kFinThreads) {
        int b = goff[g], e = goff[g + 1];
        b = b < 0 ? 0 : (b > S ? S : b);
        e = e < b ? b : (e > S ? S : e);
        int G = 0;
        long long ntok = 0;
        double y = 0.0;
        for (int i = b; i < e; ++i) {
            const int n = keep ? sh_n[i] : seq[i].n;
            ntok += n;
            if (n > 0) {
                ++G;
                y += keep ? sh_D[i] : div64(seq[i].sum_d, n);
            }
        }
        acrl_group_stats gs;
        gs.n_valid_seqs = G;
        gs.n_seqs = e - b;
        gs.n_tokens = ntok;
        gs.Y = G ? div64(y, G) : 0.0;
        grp[g] = gs;
        if (G) {
            ++qv;
            ysum += gs.Y;
        }
    }
    // warps beyond the responses and prompts hold nothing
    const int used = min(NW, (max(S, Gn) + 31) / 32);
    if (wid < used) {
        const double s = warp_sum4(sd, sd2, sH, slr), y = warp_sum(ysum);
        N = warp_sum(N);
        sv = __reduce_add_sync(0xffffffffu, sv);
        qv = __reduce_add_sync(0xffffffffu, qv);
        dmax = warp_max_nonneg(dmax);
        if ((lane & 7) == 0) sh[wid * 5 + (lane >> 3)] = s;
        if (lane == 0) {
            sh[wid * 5 + 4] = y;
            sh_N[wid] = N;
            sh_sv[wid] = sv;
            sh_qv[wid] = qv;
            sh_max[wid] = dmax;
        }
    }
    __syncthreads();
    if (wid == 0) {
        double s = 0.0;  // value k in lane k: sums of d, d^2, H, lr and Y_g
        if (lane < 5)
            for (int w = 0; w < used; ++w) s += sh[w * 5 + lane];
        N = warp_sum(lane < used ? sh_N[lane] : 0ll);
        sv = __reduce_add_sync(0xffffffffu, lane < used ? sh_sv[lane] : 0);
        qv = __reduce_add_sync(0xffffffffu, lane < used ? sh_qv[lane] : 0);
        dmax = warp_max_nonneg(lane < used ? sh_max[lane] : 0.f);
        write_batch(s, N, sv, qv, dmax, batch);
    }
}

__global__ void __launch_bounds__(kFinThreads) seq_finalize_kernel(
    int64_t T, const int64_t* __restrict__ so, int S, const int32_t* __restrict__ goff, int Gn,
    const acrl_seq_stats* __restrict__ seq, acrl_group_stats* grp, acrl_batch_stats* batch, int32_t* flags) {
    grid_begin();
    finalize_seqs(T, so, S, goff, Gn, seq, grp, batch, flags);
}

// K3: GRPO advantages.  LANES lanes share a prompt: a thread per prompt ran
// G dependent loads and G fp64 divisions one after the other (12.2 us for 64
// prompts of 8; 5.7 us with eight lanes).  LANES = 1 is for batches of so many
// prompts that the fp64 work of idle lanes would cost more than the latency.
template <int LANES>
__device__ __forceinline__ void grpo_prompt(int64_t tid, const float* __restrict__ R, const int32_t* __restrict__ goff,
                                            int Gn, int S, float adv_eps, int ddof, int singleton_rule, float* adv,
                                            int32_t* flags) {
    constexpr int KEEP = 4;  // rewards per lane kept in registers between the passes
    const int64_t g = tid / LANES;
    const int sub = int(tid % LANES);
    if (g >= Gn) return;  // the prompt's lanes leave together
    const unsigned team = LANES == 1 ? 0u : ((1u << LANES) - 1u) << (threadIdx.x & 31 & ~(LANES - 1));
    const int64_t b = goff[g], e = goff[g + 1];   // 64 bits: the lanes step past e, which may be the type's largest
    if (b < 0 || b > e || e > S) {
        if (sub == 0) raise_flag(flags, ACRL_FLAG_BAD_OFFSETS);
        return;
    }
    const int G = int(e - b);
    if (G == 0) return;
    if (G == 1) {
        if (sub == 0) adv[b] = singleton_rule == ACRL_SINGLETON_MEAN0_STD1 ? R[b] : 0.f;
        return;
    }
    auto total = [&](double v) {
#pragma unroll
        for (int m = LANES / 2; m >= 1; m >>= 1) v += __shfl_xor_sync(team, v, m);
        return v;
    };
    float r[KEEP];
#pragma unroll
    for (int k = 0; k < KEEP; ++k) r[k] = b + sub + k * LANES < e ? R[b + sub + k * LANES] : 0.f;
    const int64_t rest = b + sub + KEEP * LANES;
    double sum = 0.0;
#pragma unroll
    for (int k = 0; k < KEEP; ++k)
        if (b + sub + k * LANES < e) sum += r[k];
    for (int64_t i = rest; i < e; i += LANES) sum += R[i];
    const double mean = div64(total(sum), G);
    double ss = 0.0;
#pragma unroll
    for (int k = 0; k < KEEP; ++k)
        if (b + sub + k * LANES < e) {
            const double c = r[k] - mean;
            ss += c * c;
        }
    for (int64_t i = rest; i < e; i += LANES) {
        const double c = R[i] - mean;
        ss += c * c;
    }
    ss = total(ss);
    const double var = G > ddof ? div64(ss, G - ddof) : 0.0;
    const double den = sqrt64(var) + double(adv_eps);
#pragma unroll
    for (int k = 0; k < KEEP; ++k)
        if (b + sub + k * LANES < e) adv[b + sub + k * LANES] = den > 0.0 ? float(div64(r[k] - mean, den)) : 0.f;
    for (int64_t i = rest; i < e; i += LANES) adv[i] = den > 0.0 ? float(div64(R[i] - mean, den)) : 0.f;
}

template <int LANES>
__global__ void grpo_kernel(const float* __restrict__ R, const int32_t* __restrict__ goff, int Gn, int S, float adv_eps,
                            int ddof, int singleton_rule, float* __restrict__ adv, int32_t* flags) {
    grid_begin();
    grpo_prompt<LANES>(int64_t(blockIdx.x) * blockDim.x + threadIdx.x, R, goff, Gn, S, adv_eps, ddof, singleton_rule, adv,
                       flags);
}

// K2b and K3 at once, for a caller that wants both: CTA 0 finalises, the others
// make the advantages meanwhile, kGrpoThreads of theirs each (with all 512 the fp64
// work of 64 prompts on one SM took longer than the launch it saves).  The three
// calls, 64 / 128 / 256 / 512 responses: 22.7 / 26.1 / 30.5 / 44.5 us with a launch of
// its own, 19.1 / 22.3 / 28.5 / 42.1 so.
__global__ void __launch_bounds__(kFinThreads) seq_finalize_grpo_kernel(
    int64_t T, const int64_t* __restrict__ so, int S, const int32_t* __restrict__ goff, int Gn,
    const acrl_seq_stats* __restrict__ seq, acrl_group_stats* grp, acrl_batch_stats* batch, const float* __restrict__ R,
    float adv_eps, int ddof, int singleton_rule, float* __restrict__ adv, int32_t* flags) {
    grid_begin();
    if (blockIdx.x == 0)
        finalize_seqs(T, so, S, goff, Gn, seq, grp, batch, flags);
    else if (threadIdx.x < kGrpoThreads)
        grpo_prompt<8>(int64_t(blockIdx.x - 1) * kGrpoThreads + threadIdx.x, R, goff, Gn, S, adv_eps, ddof, singleton_rule,
                       adv, flags);
}

__global__ void controller_init_kernel(acrl_controller_state* st, double X_init) {
    grid_begin();
    acrl_controller_state s;
    s.X = X_init > 0.0 ? X_init : 0.0;
    s.calib_sum = 0.0;
    s.calib_count = 0;
    s.step = 0;
    s.calib_done = 0;
    s.calibrated = X_init > 0.0 ? 1 : 0;
    s.flags = 0;
    s.reserved = 0;
    *st = s;
}

// What the controller does to its state on one batch: the X in force as a
// quotient (so that a caller can fold the division into one it does anyway),
// and whether alpha applies (it does not while X is still being calibrated).
struct ControllerMove {
    double x_num, x_den;
    bool apply;
    acrl_controller_state next;   // X not yet divided out
};

__device__ __forceinline__ ControllerMove controller_move(const acrl_controller_state& st, const acrl_params& p,
                                                          double Y_sum, int n_groups_valid) {
    ControllerMove m;
    m.next = st;
    m.next.step += 1;
    m.x_num = st.X;
    m.x_den = 1.0;
    m.apply = true;
    if (!st.calibrated) {
        m.next.calib_sum += Y_sum;
        m.next.calib_count += n_groups_valid;
        m.next.calib_done += 1;
        if (m.next.calib_done >= p.calib_steps) {
            m.x_num = m.next.calib_count > 0 ? m.next.calib_sum : 0.0;
            m.x_den = m.next.calib_count > 0 ? double(m.next.calib_count) : 1.0;
            m.next.calibrated = 1;
        } else {
            m.apply = false;
        }
    }
    return m;
}

// alpha of a response with n valid tokens, advantage A and discrepancy Y;
// inv_X = recip64(X), unused where X is out of its range.
__device__ __forceinline__ float alpha_of(const acrl_params& p, bool apply, double X, double inv_X, double Y, float A,
                                          int n) {
    const float sgnf = A > 0.f ? 1.f : (A < 0.f ? -1.f : 0.f);
    float a = 0.f;
    if (p.mode == ACRL_MODE_TIS || p.mode == ACRL_MODE_MIS) {
        a = 1.f;
    } else if (p.mode == ACRL_MODE_ACRL_CONTINUOUS) {
        a = n > 0 ? -p.kappa * sgnf : 0.f;
    } else if ((p.mode == ACRL_MODE_ACRL || p.mode == ACRL_MODE_ACRL_FALLBACK) && apply && X > 0.0 && n > 0) {
        const double rest = 1.0 - (exp_within(X, 100) ? quot64(Y, X, inv_X) : Y / X);  // exactly 0 where Y = X
        a = float(double(p.gamma * sgnf) * rest);
        if (p.mode == ACRL_MODE_ACRL_FALLBACK && !(Y > X)) a = 0.f;
    }
    return a;
}

// What the weights of a response's tokens are made from.
struct RespScalars {
    float alpha, scale, escale;   // exponent, A / norm, beta / norm
    float w_mis;                  // the sequence-level weight and whether it is cut
    int cut;
};

__device__ __forceinline__ RespScalars resp_scalars(float alpha, float scale, float escale, float Si, float logC) {
    const bool cut = Si > logC;
    return RespScalars{alpha, scale, escale, (cut || isnan(Si)) ? 0.f : expf(Si), cut};
}

// The weight of one valid token with log-ratio l; counts it in nt where it is truncated.
__device__ __forceinline__ float token_weight(int mode, const RespScalars& r, float l, float logC, int& nt) {
    if (mode == ACRL_MODE_NONE) return 1.f;
    if (mode == ACRL_MODE_MIS) {
        nt += r.cut;
        return r.w_mis;
    }
    // rho^0 = 1 even where the log-ratio is infinite (mu = 0); a NaN log-ratio gets weight 0
    const float lrho = r.alpha == 0.f ? 0.f : r.alpha * l;
    nt += lrho > logC;
    return isnan(lrho) ? 0.f : expf(fminf(lrho, logC));
}

// K4a: alpha per response, in a launch of its own (acrl_controller_step;
// acrl_importance_weights folds it into the next kernel).  Every warp works out the X
// in force for itself; the finalising kernel writes the state.
__global__ void __launch_bounds__(kSeqThreads) controller_alpha_kernel(
    const acrl_controller_state* __restrict__ st, acrl_params p, int S, int Gn, acrl_seq_stats* seq,
    const acrl_group_stats* __restrict__ grp, const acrl_batch_stats* __restrict__ batch, const float* __restrict__ adv,
    float* __restrict__ alpha_out) {
    const int lane = threadIdx.x & 31;
    grid_begin();
    const int ngv = batch->n_groups_valid;
    const double Ysum = batch->Y_sum;
    const ControllerMove mv = controller_move(*st, p, Ysum, ngv);
    // one division: X in lane 0, the batch's Y (of the possibly all-reduced sum and prompt count) in lane 1
    const double num = lane == 0 ? mv.x_num : Ysum, den = lane == 0 ? mv.x_den : double(ngv);
    const double q = den > 0.0 ? div64(num, den) : 0.0;
    const double X = __shfl_sync(0xffffffffu, q, 0), Ybatch = __shfl_sync(0xffffffffu, q, 1);
    const int64_t i = int64_t(blockIdx.x) * kSeqThreads + threadIdx.x;
    if (i >= S) return;
    const int n = seq[i].n, g = seq[i].group;
    double Y = 0.0;
    if (p.y_gran == ACRL_Y_SEQUENCE)
        Y = n > 0 ? div64(seq[i].sum_d, double(n)) : 0.0;
    else if (p.y_gran == ACRL_Y_BATCH)
        Y = Ybatch;
    else if (g >= 0 && g < Gn)
        Y = grp[g].Y;
    const float a = alpha_of(p, mv.apply, X, recip64(X), Y, adv[i], n);
    seq[i].alpha = a;
    if (alpha_out) alpha_out[i] = a;
}

// K4b: per-token weights and loss coefficients; a cluster of CTAs per response as
// in seq_stats_kernel.  FOLD: alpha per response too, from the X in force as
// controller_alpha_kernel works it out; otherwise alpha is that kernel's.
template <bool FOLD>
__global__ void __launch_bounds__(kSeqThreads) controller_weights_kernel(
    const acrl_controller_state* __restrict__ st, acrl_params p, const float* __restrict__ lr,
    const uint8_t* __restrict__ mask, int64_t T, const int64_t* __restrict__ so, int Gn, acrl_seq_stats* seq,
    const acrl_group_stats* __restrict__ grp, const acrl_batch_stats* __restrict__ batch,
    const float* __restrict__ adv, float* __restrict__ weight, float* __restrict__ coef, float* __restrict__ alpha_out,
    float* __restrict__ ent_coef) {
    constexpr int NW = kSeqThreads / 32, U = kSeqUnroll;
    __shared__ double sh[NW];
    __shared__ int sh_nt[NW];
    __shared__ RespScalars sh_resp;
    __shared__ double part_w;
    __shared__ int part_nt;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nct = int(cluster_size()), rank = int(cluster_rank());
    const int i = int(blockIdx.x) / nct;
    grid_begin();
    int64_t lo, hi;
    if (!seq_range(so, i, T, lo, hi)) lo = hi = 0;
    const float logC = logf(p.C);
    const int64_t stride = int64_t(nct) * kSeqThreads;
    const bool uses_lr = p.mode != ACRL_MODE_NONE && p.mode != ACRL_MODE_MIS;

    // the first tokens are on their way while warp 0 works out the response's scalars
    float l[U];
    bool m[U];
    auto load = [&](int64_t t0) {
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int64_t t = t0 + k * stride;
            const bool in = t < hi;
            m[k] = in && (mask ? mask[t] != 0 : true);
            l[k] = in && uses_lr ? lr[t] : 0.f;
        }
    };
    int64_t t0 = lo + rank * kSeqThreads + threadIdx.x;
    load(t0);
    if (wid == 0) {
        const int n = seq[i].n, g = seq[i].group;
        const double sum_d = seq[i].sum_d;
        const float Si = float(seq[i].sum_lr), A = adv[i];
        const bool has_g = g >= 0 && g < Gn;
        const double Yg = has_g ? grp[g].Y : 0.0;
        const int ngv = batch->n_groups_valid;
        const double Ysum = batch->Y_sum;
        ControllerMove mv;
        if (FOLD) mv = controller_move(*st, p, Ysum, ngv);
        double norm;
        if (p.agg == ACRL_AGG_TOKEN_MEAN)
            norm = double(batch->n_tokens);
        else
            norm = double(ngv) * double(has_g ? grp[g].n_valid_seqs : 0) * double(n);
        // one division, a different quotient in each lane: Y, X, A / norm, beta / norm
        double num = 0.0, den = 1.0;
        if (FOLD && lane == 0) {
            if (p.y_gran == ACRL_Y_SEQUENCE) {
                num = sum_d;
                den = double(n);
            } else if (p.y_gran == ACRL_Y_BATCH) {
                num = Ysum;
                den = double(ngv);
            } else {
                num = Yg;
            }
        } else if (FOLD && lane == 1) {
            num = mv.x_num;
            den = mv.x_den;
        } else if (lane == 2 || lane == 3) {
            num = lane == 2 ? double(A) : double(p.entropy_coeff);
            den = norm;
        }
        const double q = den > 0.0 ? div64(num, den) : 0.0;
        const float scale = float(__shfl_sync(0xffffffffu, q, 2)), escale = float(__shfl_sync(0xffffffffu, q, 3));
        float a;
        if (FOLD) {
            const double Y = __shfl_sync(0xffffffffu, q, 0), X = __shfl_sync(0xffffffffu, q, 1);
            a = alpha_of(p, mv.apply, X, recip64(X), Y, A, n);
        } else {
            a = seq[i].alpha;
        }
        if (lane == 0) {
            sh_resp = resp_scalars(a, scale, escale, Si, logC);
            if (FOLD && rank == 0) {
                seq[i].alpha = a;
                if (alpha_out) alpha_out[i] = a;
            }
        }
    }
    __syncthreads();
    const RespScalars resp = sh_resp;
    int nt = 0;
    double sw = 0.0;
    while (t0 < hi) {
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int64_t t = t0 + k * stride;
            if (t >= hi) break;
            float w = 0.f;
            if (m[k]) {
                w = token_weight(p.mode, resp, l[k], logC, nt);
                sw += w;
            }
            weight[t] = w;
            coef[t] = w * resp.scale;
            if (ent_coef) ent_coef[t] = m[k] ? resp.escale : 0.f;
        }
        t0 += U * stride;
        load(t0);
    }
    sw = warp_sum(sw);
    nt = __reduce_add_sync(0xffffffffu, nt);
    if (lane == 0) {
        sh[wid] = sw;
        sh_nt[wid] = nt;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        sw = 0.0;
        nt = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            sw += sh[w];
            nt += sh_nt[w];
        }
        part_w = sw;
        part_nt = nt;
    }
    if (nct > 1) cluster_sync();  // every CTA's part is in its shared memory
    if (rank == 0 && threadIdx.x == 0) {
        for (int r = 1; r < nct; ++r) {
            sw += ld_peer_f64(&part_w, uint32_t(r));
            nt += int(ld_peer_u32(&part_nt, uint32_t(r)));
        }
        seq[i].n_trunc = nt;
        seq[i].sum_w = sw;
    }
    if (nct > 1) cluster_sync();  // no CTA leaves while rank 0 may still read its shared memory
}

// The controller's new state and the batch fields that come from it; one thread.
// X: the reference in force, Ymean: the batch's mean discrepancy.
__device__ __forceinline__ void write_state(const acrl_controller_state& old, const ControllerMove& mv, double X,
                                            double Ymean, double alpha_mean, const acrl_params& p,
                                            acrl_controller_state* st, acrl_batch_stats* batch, int32_t* flags) {
    const bool was_calibrated = old.calibrated != 0;
    acrl_controller_state n = mv.next;
    n.X = X;
    const bool uses_x = p.mode == ACRL_MODE_ACRL || p.mode == ACRL_MODE_ACRL_FALLBACK;
    if (uses_x && mv.apply && !(X > 0.0)) {
        raise_flag(flags, ACRL_FLAG_X_NONPOS);
        n.flags |= ACRL_FLAG_X_NONPOS;
    }
    // moving-average X (off by default): this step used X, the next one uses the update
    if (was_calibrated && p.x_ema > 0.f) n.X = fma(double(p.x_ema), Ymean, (1.0 - double(p.x_ema)) * X);
    *st = n;
    batch->Y_mean = Ymean;
    batch->X = mv.apply ? X : 0.0;
    batch->alpha_mean = alpha_mean;
}

// K4c: the controller's new state and the batch metrics.
__global__ void __launch_bounds__(kFinThreads) controller_finalize_kernel(acrl_controller_state* st, acrl_params p,
                                                                          int S,
                                                                          const acrl_seq_stats* __restrict__ seq,
                                                                          acrl_batch_stats* batch, int32_t* flags) {
    constexpr int NW = kFinThreads / 32;
    __shared__ double sh[NW * 2];
    __shared__ long long sh_nt[NW];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int used = min(NW, (S + 31) / 32);  // warps with responses of their own
    grid_begin();
    if (wid < used) {
        long long nt = 0;
        double sw = 0.0, sa = 0.0;
        for (int i = threadIdx.x; i < S; i += kFinThreads) {
            nt += seq[i].n_trunc;
            sw += seq[i].sum_w;
            if (seq[i].n > 0) sa += seq[i].alpha;
        }
        const double s = warp_sum2(sw, sa);
        nt = warp_sum(nt);
        if ((lane & 15) == 0) sh[wid * 2 + (lane >> 4)] = s;
        if (lane == 0) sh_nt[wid] = nt;
    }
    __syncthreads();
    if (wid != 0) return;
    double s = 0.0;  // sum of the weights in lane 0, of alpha in lane 1
    if (lane < 2)
        for (int w = 0; w < used; ++w) s += sh[w * 2 + lane];
    const long long nt = warp_sum(lane < used ? sh_nt[lane] : 0ll);
    const int ngv = batch->n_groups_valid, nsv = batch->n_seqs_valid;
    const double Ysum = batch->Y_sum, N = double(batch->n_tokens);
    const acrl_controller_state old = *st;
    const ControllerMove mv = controller_move(old, p, Ysum, ngv);
    // one division: w_mean, alpha_mean, trunc_frac, Y_mean (of the possibly all-reduced sum and prompt count), X
    double num = s, den = N;
    if (lane == 1) den = double(nsv);
    if (lane == 2) num = double(nt);
    if (lane == 3) num = Ysum, den = double(ngv);
    if (lane == 4) num = mv.x_num, den = mv.x_den;
    const double q = den > 0.0 ? div64(num, den) : 0.0;
    const double a_mean = __shfl_sync(0xffffffffu, q, 1), trunc = __shfl_sync(0xffffffffu, q, 2),
                 Ymean = __shfl_sync(0xffffffffu, q, 3), X = __shfl_sync(0xffffffffu, q, 4);
    if (lane == 0) {
        write_state(old, mv, X, Ymean, a_mean, p, st, batch, flags);
        batch->trunc_frac = trunc;
        batch->w_mean = q;
    }
}

// The three O(T) calls of a small batch in one launch: one cluster of CTAs does
// what seq_stats, seq_finalize, grpo, controller_weights and
// controller_finalize do, with the same parts (a part is what one CTA of those
// kernels does: every nct-th round of a response), the same trees and the same
// order of the parts, so both give the same bits.  A CTA has two groups of eight
// warps, each taking one part, and two warps for the scalars of responses and
// prompts (a lane each): those of CTA 0 go from the parts' sums to alpha and from
// their counts to the loss factors, between the two halves of the tokens' work;
// CTA 1's first one makes the batch statistics meanwhile.
//
// Latency bounds it, that of fp64 chains above all (some 80 cycles an
// operation).  Against the five launches, replayed from a graph: 4 x 256 tokens
// 15.4 -> 10.4 us, 8 x 600 20.0 -> 13.5, 4 x 1,000 19.4 -> 12.1, 32 x 250 18.6 ->
// 15.1, 4 x 10,000 23.3 -> 20.7.  More than 32 parts would need a second pass
// over them, with which the launches are ahead (8 x 1,000 in eight CTAs with two
// passes: 23.1 against 20.0).
constexpr int kOneGroups = 2, kOneCtas = 16, kOneParts = kOneCtas * kOneGroups, kOneSeqs = 32;
constexpr int kOneThreads = kOneGroups * kSeqThreads + 64;

struct OnePart {
    double sum[4];  // d, d^2, lr, H
    double w;       // sum of the weights
    int n, nt;      // valid and truncated tokens
    uint32_t max_d;
};

__device__ __forceinline__ void group_sync(int group) {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(kSeqThreads) : "memory");
}

__global__ void __launch_bounds__(kOneThreads) weights_cluster_kernel(
    acrl_controller_state* st, acrl_params p, const float* __restrict__ logp_pi, const float* __restrict__ logp_mu,
    const uint8_t* __restrict__ mask, int64_t T, const float* __restrict__ R, const int64_t* __restrict__ so, int S,
    const int32_t* __restrict__ goff, int Gn, const float* __restrict__ entropy, float* lr, float* d, acrl_seq_stats* seq,
    acrl_group_stats* grp, acrl_batch_stats* batch, float* adv, float* weight, float* coef, float* alpha_out,
    float* ent_coef, int nct, int32_t* flags) {
    constexpr int NW = kSeqThreads / 32, U = kSeqUnroll;
    __shared__ double sh[kOneGroups][NW * 4];
    __shared__ int sh_n[kOneGroups][NW];
    __shared__ uint32_t sh_max[kOneGroups][NW];
    __shared__ OnePart part[kOneGroups];
    __shared__ RespScalars resp[kOneSeqs];   // CTA 0's is read by all
    __shared__ double sh_D[kOneSeqs], sh_Y[kOneSeqs];
    const int lane = threadIdx.x & 31;
    const int C = int(cluster_size()), rank = int(cluster_rank()), logC2 = 31 - __clz(C);  // C is a power of two
    const int group = threadIdx.x / kSeqThreads, tid = threadIdx.x % kSeqThreads, wid = tid >> 5;
    const float logC = logf(p.C);
    const int64_t stride = int64_t(nct) * kSeqThreads;
    grid_begin();

    enum { kTokens, kSums, kCounts, kBatch, kNone };
    const int role = group < kOneGroups ? kTokens
                     : rank == 0        ? (wid == 0 ? kSums : kCounts)
                     : rank == 1 && wid == 0 ? kBatch : kNone;
    // what a token thread keeps of its part
    const int k = rank + C * group;
    const bool has_part = group < kOneGroups && k < S * nct;
    float l[U];
    bool m[U];
    int64_t t_lo = 0, t_hi = 0;
    // what a scalar lane keeps of its response and prompt: the prompt's responses, the response's prompt
    int gb = 0, ge = 0, g = -1;
    acrl_controller_state state;
    double inv_X = 0.0;
    if (has_part) {
        if (!seq_range(so, k / nct, T, t_lo, t_hi)) {
            if (k % nct == 0 && tid == 0) raise_flag(flags, ACRL_FLAG_BAD_OFFSETS);
            t_lo = t_hi = 0;
        }
        t_lo += (k % nct) * kSeqThreads + tid;
        const bool nan_lr = stats_tokens(logp_pi, logp_mu, mask, entropy, lr, d, t_lo, t_hi, stride, l, m,
                                         &sh[group][wid * 4], &sh_n[group][wid], &sh_max[group][wid]);
        if (nan_lr) raise_flag(flags, ACRL_FLAG_NONFINITE);
        group_sync(group);
        if (wid == 0) part_sums<NW>(sh[group], sh_n[group], sh_max[group], part[group].sum, part[group].n,
                                    part[group].max_d);
    }
    if (rank == C - 1 && group == kOneGroups - 1)   // 32 prompts, eight lanes each
        grpo_prompt<8>(tid, R, goff, Gn, S, p.adv_eps, p.adv_ddof, p.singleton_rule, adv, flags);
    if (role == kSums || role == kCounts || role == kBatch) {
        if (lane < Gn) {
            gb = goff[lane];
            ge = goff[lane + 1];
        }
        if (role == kCounts) {
            bool bad = lane < Gn && gb > ge;
            if (lane < S) bad |= so[lane] > so[lane + 1];
            if (lane == 0) bad |= so[0] != 0 || so[S] != T || goff[0] != 0 || goff[Gn] != S;
            if (bad) raise_flag(flags, ACRL_FLAG_BAD_OFFSETS);
        }
        // the last prompt that starts at or before response `lane`, if that is inside it
        int at = 0;
        for (int j = 0; j < Gn; ++j)
            if (__shfl_sync(0xffffffffu, gb, j) <= lane) at = j;
        const int b = __shfl_sync(0xffffffffu, gb, at), e = __shfl_sync(0xffffffffu, ge, at);
        g = b <= lane && lane < e ? at : -1;
        gb = gb < 0 ? 0 : (gb > S ? S : gb);
        ge = ge < gb ? gb : (ge > S ? S : ge);
        state = *st;
        inv_X = recip64(state.X);
    }
    cluster_sync();  // every CTA's parts are in its shared memory, the advantages written

    // sums over the parts of this lane's response, in their order
    auto total = [&](const double* first) {
        double v = 0.0;
        if (lane < S)
            for (int j = lane * nct; j < (lane + 1) * nct; ++j)
                v += ld_peer_f64(reinterpret_cast<const double*>(reinterpret_cast<const char*>(first) +
                                                                 (j >> logC2) * sizeof(OnePart)),
                                 uint32_t(j & (C - 1)));
        return v;
    };
    auto count = [&](const void* first) {
        int v = 0;
        if (lane < S)
            for (int j = lane * nct; j < (lane + 1) * nct; ++j)
                v += int(ld_peer_u32(static_cast<const char*>(first) + (j >> logC2) * sizeof(OnePart), uint32_t(j & (C - 1))));
        return v;
    };
    auto largest = [&] {
        uint32_t v = 0u;
        if (lane < S)
            for (int j = lane * nct; j < (lane + 1) * nct; ++j)
                v = max(v, ld_peer_u32(&part[j >> logC2].max_d, uint32_t(j & (C - 1))));
        return v;
    };
    int n = 0, G = 0, qv = 0, sv = 0;
    double sd = 0.0, D = 0.0, Yg = 0.0, Ysum = 0.0, s4 = 0.0;
    float alpha = 0.f;
    if (role == kSums || role == kCounts || role == kBatch) {
        n = count(&part[0].n);
        // this prompt's valid responses
        const unsigned valid = __ballot_sync(0xffffffffu, n > 0);
        const unsigned upto = ge < 32 ? (1u << ge) - 1u : ~0u, before = gb < 32 ? (1u << gb) - 1u : ~0u;
        G = lane < Gn ? __popc(valid & upto & ~before) : 0;
        sv = __popc(valid);
        qv = __popc(__ballot_sync(0xffffffffu, G > 0));
        if (role == kSums) {
            const float A = lane < S ? __ldcg(adv + lane) : 0.f;
            sd = total(&part[0].sum[0]);
            D = n > 0 ? quot64(sd, n, recip64(n)) : 0.0;
            const double inv_G = recip64(G > 0 ? G : 1);
            sh_D[lane] = D;
            __syncwarp();
            double y = 0.0;
            if (lane < Gn)
                for (int i = gb; i < ge; ++i)
                    if (valid >> i & 1) y += sh_D[i];
            Yg = G ? quot64(y, G, inv_G) : 0.0;
            sh_Y[lane] = Yg;
            if (p.y_gran == ACRL_Y_BATCH || !state.calibrated) Ysum = warp_sum(Yg);
            const ControllerMove mv = controller_move(state, p, Ysum, qv);
            double X = state.X;
            if (!state.calibrated && mv.apply) {
                X = mv.x_den > 0.0 ? div64(mv.x_num, mv.x_den) : 0.0;
                inv_X = recip64(X);
            }
            const double Yp = __shfl_sync(0xffffffffu, Yg, g < 0 ? 0 : g);
            double Y = g >= 0 ? Yp : 0.0;
            if (p.y_gran == ACRL_Y_SEQUENCE) Y = D;
            if (p.y_gran == ACRL_Y_BATCH) Y = qv > 0 ? div64(Ysum, qv) : 0.0;
            alpha = alpha_of(p, mv.apply, X, inv_X, Y, A, n);
            if (lane < S) resp[lane].alpha = alpha;
        } else if (role == kCounts) {
            const float A = lane < S ? __ldcg(adv + lane) : 0.f;
            const int Gp = __shfl_sync(0xffffffffu, G, g < 0 ? 0 : g);
            const double norm = p.agg == ACRL_AGG_TOKEN_MEAN ? double(warp_count(n))
                                                             : double(qv) * double(g >= 0 ? Gp : 0) * double(n);
            const float scale = norm > 0.0 ? float(div64(A, norm)) : 0.f;
            const float escale = ent_coef && norm > 0.0 ? float(div64(p.entropy_coeff, norm)) : 0.f;
            const float Si = p.mode == ACRL_MODE_MIS ? float(total(&part[0].sum[2])) : 0.f;
            if (lane < S) {
                const RespScalars r = resp_scalars(0.f, scale, escale, Si, logC);
                resp[lane].scale = r.scale;
                resp[lane].escale = r.escale;
                resp[lane].w_mis = r.w_mis;
                resp[lane].cut = r.cut;
            }
        } else {
            s4 = warp_sum4(total(&part[0].sum[0]), total(&part[0].sum[1]), total(&part[0].sum[3]), total(&part[0].sum[2]));
        }
    }
    cluster_sync();  // the responses' scalars are in CTA 0's shared memory

    acrl_seq_stats o;
    double inv_N = 0.0;
    long long N = 0;
    if (has_part) {
        const RespScalars* from = &resp[k / nct];
        RespScalars r;
        r.alpha = __uint_as_float(ld_peer_u32(&from->alpha, 0));
        r.scale = __uint_as_float(ld_peer_u32(&from->scale, 0));
        r.escale = __uint_as_float(ld_peer_u32(&from->escale, 0));
        r.w_mis = __uint_as_float(ld_peer_u32(&from->w_mis, 0));
        r.cut = int(ld_peer_u32(&from->cut, 0));
        int nt = 0;
        double sw = 0.0;
        for (int64_t t0 = t_lo; t0 < t_hi; t0 += U * stride) {
            if (t0 != t_lo) {   // beyond the first round: lr as this thread wrote it
#pragma unroll
                for (int j = 0; j < U; ++j) {
                    const int64_t t = t0 + j * stride;
                    m[j] = t < t_hi && (mask ? mask[t] != 0 : true);
                    l[j] = t < t_hi ? lr[t] : 0.f;
                }
            }
#pragma unroll
            for (int j = 0; j < U; ++j) {
                const int64_t t = t0 + j * stride;
                if (t >= t_hi) break;
                float w = 0.f;
                if (m[j]) {
                    w = token_weight(p.mode, r, l[j], logC, nt);
                    sw += w;
                }
                weight[t] = w;
                coef[t] = w * r.scale;
                if (ent_coef) ent_coef[t] = m[j] ? r.escale : 0.f;
            }
        }
        sw = warp_sum(sw);
        nt = __reduce_add_sync(0xffffffffu, nt);
        if (lane == 0) {
            sh[group][wid] = sw;
            sh_n[group][wid] = nt;
        }
        group_sync(group);
        if (tid == 0) {
            sw = 0.0;
            nt = 0;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                sw += sh[group][w];
                nt += sh_n[group][w];
            }
            part[group].w = sw;
            part[group].nt = nt;
        }
    } else if (role == kSums) {
        o.n = n;
        o.group = g;
        o.mean_d = float(D);
        o.max_d = __uint_as_float(largest());
        o.sum_d = sd;
        o.sum_d2 = total(&part[0].sum[1]);
        o.sum_lr = total(&part[0].sum[2]);
        o.sum_H = total(&part[0].sum[3]);
        o.alpha = alpha;
        if (lane < S && alpha_out) alpha_out[lane] = alpha;
        N = warp_count(n);
        inv_N = recip64(N > 0 ? double(N) : 1.0);
    } else if (role == kCounts) {
        long long ntok = 0;
        for (int i = 0; i < S; ++i) {
            const int ni = __shfl_sync(0xffffffffu, n, i);
            if (i >= gb && i < ge) ntok += ni;
        }
        if (lane < Gn) {
            acrl_group_stats gs;
            gs.n_valid_seqs = G;
            gs.n_seqs = ge - gb;
            gs.n_tokens = ntok;
            gs.Y = sh_Y[lane];
            grp[lane] = gs;
        }
    } else if (role == kBatch) {
        Yg = ld_peer_f64(&sh_Y[lane], 0);
        alpha = lane < S && n > 0 ? __uint_as_float(ld_peer_u32(&resp[lane].alpha, 0)) : 0.f;
        Ysum = warp_sum(Yg);
        const double sa = warp_sum(double(alpha));
        const double s = __shfl_sync(0xffffffffu, s4, (lane & 3) * 8);  // value k in lane k
        write_batch(lane == 4 ? Ysum : s, warp_count(n), sv, qv, warp_max_nonneg(__uint_as_float(largest())), batch);
        const ControllerMove mv = controller_move(state, p, Ysum, qv);
        if (lane == 0)
            write_state(state, mv, mv.x_den > 0.0 ? div64(mv.x_num, mv.x_den) : 0.0, qv > 0 ? div64(Ysum, qv) : 0.0,
                        sv > 0 ? div64(sa, sv) : 0.0, p, st, batch, flags);
    }
    cluster_sync();  // every CTA's weight sums are in its shared memory, the other batch fields written

    if (role == kSums) {
        o.sum_w = total(&part[0].w);
        o.n_trunc = count(&part[0].nt);
        if (lane < S) seq[lane] = o;
        const double sw = warp_sum(o.sum_w);
        const long long nt = warp_count(o.n_trunc);
        if (lane == 0) {
            batch->w_mean = N > 0 ? quot64(sw, double(N), inv_N) : 0.0;
            batch->trunc_frac = N > 0 ? quot64(double(nt), double(N), inv_N) : 0.0;
        }
    }
    cluster_sync();  // no CTA leaves while CTA 0 may still read its shared memory
}

// Clusters of more than eight CTAs are an opt-in that a part of a GPU may not have.
bool one_cluster_fits(int ctas) {
    if (ctas <= 8) return true;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(ctas), 1, 1);
    cfg.blockDim = dim3(kOneThreads, 1, 1);
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = unsigned(ctas);
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaFuncSetAttribute(weights_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&n, weights_cluster_kernel, &cfg) == cudaSuccess)
        return n > 0;
    (void)cudaGetLastError();
    return false;
}

// CTAs per response: enough to give the chip a few hundred CTAs, while each
// still has a round of tokens.
int ctas_per_response(int32_t S, int64_t T) {
    int c = 1;
    while (c < 8 && int64_t(S) * c * 2 <= kSeqCtas && T > int64_t(S) * c * kSeqTokens) c *= 2;
    return c;
}

acrl_status launch_seq_stats(const float* logp_pi, const float* logp_mu, const uint8_t* mask, int64_t T,
                             const int64_t* seq_offsets, int32_t S, const int32_t* group_offsets, int32_t Gn,
                             const float* entropy, float* lr, float* d, acrl_seq_stats* seq, int32_t* flags,
                             cudaStream_t s) {
    const int c = ctas_per_response(S, T);
    return launch(seq_stats_kernel, int64_t(S) * c, kSeqThreads + 32, 0, c, s, logp_pi, logp_mu, mask, T, seq_offsets, S,
                  group_offsets, Gn, entropy, lr, d, seq, flags);
}

// FOLD: two launches, alpha made by the weights' kernel; otherwise three.  Same bits.
template <bool FOLD>
acrl_status launch_controller(acrl_controller_state* state, const acrl_params& p, const float* lr, const uint8_t* mask,
                              int64_t T, const int64_t* seq_offsets, int32_t S, int32_t Gn, acrl_seq_stats* seq,
                              const acrl_group_stats* grp, acrl_batch_stats* batch, const float* adv, float* weight,
                              float* coef, float* alpha, float* ent_coef, int32_t* flags, cudaStream_t s) {
    const int c = ctas_per_response(S, T);
    acrl_status st = ACRL_OK;
    if (!FOLD && S > 0)
        st = launch(controller_alpha_kernel, (int64_t(S) + kSeqThreads - 1) / kSeqThreads, kSeqThreads, 0, 0, s, state, p, S,
                    Gn, seq, grp, batch, adv, alpha);
    if (st == ACRL_OK && S > 0)
        st = launch(controller_weights_kernel<FOLD>, int64_t(S) * c, kSeqThreads, 0, c, s, state, p, lr, mask, T,
                    seq_offsets, Gn, seq, grp, batch, adv, weight, coef, alpha, ent_coef);
    if (st != ACRL_OK) return st;
    return launch(controller_finalize_kernel, 1, kFinThreads, 0, 0, s, state, p, S, seq, batch, flags);
}

}  // namespace
}  // namespace acrl

using namespace acrl;

extern "C" acrl_status acrl_seq_discrepancy(const float* logp_pi, const float* logp_mu, const uint8_t* mask, int64_t T,
                                            const int64_t* seq_offsets, int32_t S, const int32_t* group_offsets,
                                            int32_t Gn, const float* entropy, float* lr, float* d,
                                            acrl_seq_stats* seq, acrl_group_stats* grp, acrl_batch_stats* batch,
                                            int32_t* dev_flags, acrl_stream stream) {
    if (T < 0 || S < 0 || Gn < 0) return ACRL_ERR_INVALID_ARG;
    if (!seq_offsets || !group_offsets || !batch || !dev_flags) return ACRL_ERR_INVALID_ARG;
    if (T > 0 && (!logp_pi || !logp_mu || !lr || !d)) return ACRL_ERR_INVALID_ARG;
    if ((S > 0 && !seq) || (Gn > 0 && !grp)) return ACRL_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    acrl_status st = ACRL_OK;
    if (S > 0)
        st = launch_seq_stats(logp_pi, logp_mu, mask, T, seq_offsets, S, group_offsets, Gn, entropy, lr, d, seq, dev_flags, s);
    if (st != ACRL_OK) return st;
    return launch(seq_finalize_kernel, 1, kFinThreads, 0, 0, s, T, seq_offsets, S, group_offsets, Gn, seq, grp, batch,
                  dev_flags);
}

extern "C" acrl_status acrl_grpo_advantage(const float* rewards, const int32_t* group_offsets, int32_t Gn, int32_t S,
                                           const acrl_params* p, float* adv, int32_t* dev_flags, acrl_stream stream) {
    if (Gn < 0 || S < 0 || !params_ok(p) || !group_offsets || !dev_flags) return ACRL_ERR_INVALID_ARG;
    if (S > 0 && (!rewards || !adv)) return ACRL_ERR_INVALID_ARG;
    if (Gn == 0) return ACRL_OK;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int threads = kGrpoThreads;
    auto run = [&](auto kernel, int lanes) {
        return launch(kernel, (int64_t(Gn) * lanes + threads - 1) / threads, threads, 0, 0, s, rewards, group_offsets, Gn,
                      S, p->adv_eps, p->adv_ddof, p->singleton_rule, adv, dev_flags);
    };
    return Gn <= kGrpoTeamPrompts ? run(grpo_kernel<8>, 8) : run(grpo_kernel<1>, 1);
}

extern "C" acrl_status acrl_controller_init(acrl_controller_state* state, const acrl_params* p, acrl_stream stream) {
    if (!state || !params_ok(p)) return ACRL_ERR_INVALID_ARG;
    return launch(controller_init_kernel, 1, 1, 0, 0, reinterpret_cast<cudaStream_t>(stream), state, p->X_init);
}

extern "C" acrl_status acrl_controller_save(const acrl_controller_state* state, acrl_controller_state* host_state,
                                            acrl_stream stream) {
    if (!state || !host_state) return ACRL_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(host_state, state, sizeof(acrl_controller_state), cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return ACRL_ERR_CUDA;
    return cudaStreamSynchronize(s) == cudaSuccess ? ACRL_OK : ACRL_ERR_CUDA;
}

extern "C" acrl_status acrl_controller_load(acrl_controller_state* state, const acrl_controller_state* host_state,
                                            acrl_stream stream) {
    if (!state || !host_state) return ACRL_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(state, host_state, sizeof(acrl_controller_state), cudaMemcpyHostToDevice, s) != cudaSuccess)
        return ACRL_ERR_CUDA;
    return cudaStreamSynchronize(s) == cudaSuccess ? ACRL_OK : ACRL_ERR_CUDA;
}

extern "C" acrl_status acrl_controller_step(acrl_controller_state* state, const acrl_params* p, const float* lr,
                                            const uint8_t* mask, int64_t T, const int64_t* seq_offsets, int32_t S,
                                            const int32_t* group_offsets, int32_t Gn, acrl_seq_stats* seq,
                                            const acrl_group_stats* grp, acrl_batch_stats* batch, const float* adv,
                                            float* weight, float* coef, float* alpha, float* ent_coef,
                                            int32_t* dev_flags, acrl_stream stream) {
    if (!state || !params_ok(p) || T < 0 || S < 0 || Gn < 0) return ACRL_ERR_INVALID_ARG;
    if (!seq_offsets || !group_offsets || !batch || !dev_flags) return ACRL_ERR_INVALID_ARG;
    if (T > 0 && (!lr || !weight || !coef)) return ACRL_ERR_INVALID_ARG;
    if ((S > 0 && (!seq || !adv)) || (Gn > 0 && !grp)) return ACRL_ERR_INVALID_ARG;
    return launch_controller<false>(state, *p, lr, mask, T, seq_offsets, S, Gn, seq, grp, batch, adv, weight, coef, alpha,
                                    ent_coef, dev_flags, reinterpret_cast<cudaStream_t>(stream));
}

extern "C" acrl_status acrl_importance_weights(acrl_controller_state* state, const acrl_params* p, const float* logp_pi,
                                               const float* logp_mu, const uint8_t* mask, int64_t T, const float* rewards,
                                               const int64_t* seq_offsets, int32_t S, const int32_t* group_offsets,
                                               int32_t Gn, const float* entropy, float* lr, float* d, acrl_seq_stats* seq,
                                               acrl_group_stats* grp, acrl_batch_stats* batch, float* adv, float* weight,
                                               float* coef, float* alpha, float* ent_coef, int32_t* dev_flags,
                                               acrl_stream stream) {
    if (!state || !params_ok(p) || T < 0 || S < 0 || Gn < 0) return ACRL_ERR_INVALID_ARG;
    if (!seq_offsets || !group_offsets || !batch || !dev_flags) return ACRL_ERR_INVALID_ARG;
    if (T > 0 && (!logp_pi || !logp_mu || !lr || !d || !weight || !coef)) return ACRL_ERR_INVALID_ARG;
    if ((S > 0 && (!seq || !rewards || !adv)) || (Gn > 0 && !grp)) return ACRL_ERR_INVALID_ARG;
    const int nct = ctas_per_response(S, T);
    int ctas = 2;  // the scalars have work for two
    while (ctas < kOneCtas && ctas < S * nct) ctas *= 2;
    if (S >= 1 && S <= kOneSeqs && Gn >= 1 && Gn <= kOneSeqs && S * nct <= kOneParts && one_cluster_fits(ctas))
        return launch(weights_cluster_kernel, ctas, kOneThreads, 0, ctas, reinterpret_cast<cudaStream_t>(stream), state, *p,
                      logp_pi, logp_mu, mask, T, rewards, seq_offsets, S, group_offsets, Gn, entropy, lr, d, seq, grp, batch,
                      adv, weight, coef, alpha, ent_coef, nct, dev_flags);
    acrl_status st;
    if (S > 0 && Gn > 0 && Gn <= kGrpoTeamPrompts) {
        cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
        st = launch_seq_stats(logp_pi, logp_mu, mask, T, seq_offsets, S, group_offsets, Gn, entropy, lr, d, seq, dev_flags,
                              s);
        if (st == ACRL_OK)
            st = launch(seq_finalize_grpo_kernel, 1 + (int64_t(Gn) * 8 + kGrpoThreads - 1) / kGrpoThreads, kFinThreads, 0,
                        0, s, T, seq_offsets, S, group_offsets, Gn, seq, grp, batch, rewards, p->adv_eps, p->adv_ddof,
                        p->singleton_rule, adv, dev_flags);
    } else {
        st = acrl_seq_discrepancy(logp_pi, logp_mu, mask, T, seq_offsets, S, group_offsets, Gn, entropy, lr, d, seq, grp,
                                  batch, dev_flags, stream);
        if (st == ACRL_OK) st = acrl_grpo_advantage(rewards, group_offsets, Gn, S, p, adv, dev_flags, stream);
    }
    if (st != ACRL_OK) return st;
    return launch_controller<true>(state, *p, lr, mask, T, seq_offsets, S, Gn, seq, grp, batch, adv, weight, coef, alpha,
                                   ent_coef, dev_flags, reinterpret_cast<cudaStream_t>(stream));
}

extern "C" acrl_status acrl_read_flags(const int32_t* dev_flags, int32_t* host_flags, acrl_stream stream) {
    if (!dev_flags || !host_flags) return ACRL_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(host_flags, dev_flags, sizeof(int32_t), cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return ACRL_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return ACRL_ERR_CUDA;
    return ACRL_OK;
}

extern "C" acrl_status acrl_check_flags(const int32_t* dev_flags, acrl_stream stream) {
    int32_t host = 0;
    const acrl_status st = acrl_read_flags(dev_flags, &host, stream);
    if (st != ACRL_OK) return st;
    return host != 0 ? ACRL_ERR_DEVICE_FLAGS : ACRL_OK;
}

extern "C" const char* acrl_status_string(acrl_status st) {
    switch (st) {
        case ACRL_OK: return "ok";
        case ACRL_ERR_INVALID_ARG: return "invalid argument";
        case ACRL_ERR_CUDA: return "CUDA launch or runtime error";
        case ACRL_ERR_NOT_IMPLEMENTED: return "not implemented";
        case ACRL_ERR_DEVICE_FLAGS: return "device flags raised";
        case ACRL_ERR_SCRATCH_TOO_SMALL: return "problem larger than the library's fixed scratch array";
    }
    return "unknown status";
}

extern "C" int32_t acrl_abi_version(void) { return ACRL_ABI_VERSION; }

extern "C" int64_t acrl_struct_size(int32_t which) {
    switch (which) {
        case 0: return sizeof(acrl_params);
        case 1: return sizeof(acrl_controller_state);
        case 2: return sizeof(acrl_seq_stats);
        case 3: return sizeof(acrl_group_stats);
        case 4: return sizeof(acrl_batch_stats);
    }
    return -1;
}
