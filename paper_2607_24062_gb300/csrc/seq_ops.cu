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
        int n = 0;
        double sd = 0.0, sd2 = 0.0, slr = 0.0, sH = 0.0;
        float mxd = 0.f;
        bool nan_lr = false;
        const int64_t stride = int64_t(nct) * kSeqThreads;
        for (int64_t t0 = lo + rank * kSeqThreads + threadIdx.x; t0 < hi; t0 += U * stride) {
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
            }
        }
        if (nan_lr) raise_flag(flags, ACRL_FLAG_NONFINITE);
        const double s = warp_sum4(sd, sd2, slr, sH);
        n = __reduce_add_sync(0xffffffffu, n);
        mxd = warp_max_nonneg(mxd);
        if ((lane & 7) == 0) sh[wid * 4 + (lane >> 3)] = s;
        if (lane == 0) {
            sh_n[wid] = n;
            sh_max[wid] = __float_as_uint(mxd);
        }
    }
    __syncthreads();
    if (wid == 0) {  // the warps' sums in order, value k in lane k
        double s = 0.0;
        if (lane < 4)
#pragma unroll
            for (int w = 0; w < NW; ++w) s += sh[w * 4 + lane];
        const int n = __reduce_add_sync(0xffffffffu, lane < NW ? sh_n[lane] : 0);
        const uint32_t mx = __reduce_max_sync(0xffffffffu, lane < NW ? sh_max[lane] : 0u);
        if (lane < 4) part.sum[lane] = s;
        if (lane == 0) {
            part.n = n;
            part.max_d = mx;
        }
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
            o.mean_d = n ? float(s / n) : 0.f;
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

// K2b: prompt statistics and batch statistics; also checks the offsets.
__global__ void __launch_bounds__(kFinThreads) seq_finalize_kernel(
    int64_t T, const int64_t* __restrict__ so, int S, const int32_t* __restrict__ goff, int Gn,
    const acrl_seq_stats* __restrict__ seq, acrl_group_stats* grp, acrl_batch_stats* batch, int32_t* flags) {
    constexpr int NW = kFinThreads / 32;
    __shared__ double sh_D[kFinSeqs];  // D_i, and the valid tokens of response i
    __shared__ int sh_n[kFinSeqs];
    __shared__ double sh[NW * 5];
    __shared__ long long sh_N[NW];
    __shared__ int sh_sv[NW], sh_qv[NW];
    __shared__ float sh_max[NW];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const bool keep = S <= kFinSeqs;
    grid_begin();
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
            sh_D[i] = n > 0 ? s / n : 0.0;
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
                y += keep ? sh_D[i] : seq[i].sum_d / n;
            }
        }
        acrl_group_stats gs;
        gs.n_valid_seqs = G;
        gs.n_seqs = e - b;
        gs.n_tokens = ntok;
        gs.Y = G ? y / G : 0.0;
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
        // 1 / N in lane 0, Y_mean in lane 4
        const double den = lane == 4 ? double(qv) : double(N);
        const double q = den > 0.0 ? (lane == 4 ? s : 1.0) / den : 0.0;
        const double inv = __shfl_sync(0xffffffffu, q, 0), ymean = __shfl_sync(0xffffffffu, q, 4);
        const double mean = s * inv;  // lanes 0..3: the token means
        const double d_mean = __shfl_sync(0xffffffffu, mean, 0), d2_mean = __shfl_sync(0xffffffffu, mean, 1),
                     H_mean = __shfl_sync(0xffffffffu, mean, 2), lr_mean = __shfl_sync(0xffffffffu, mean, 3);
        ysum = __shfl_sync(0xffffffffu, s, 4);
        if (lane == 0) {
            acrl_batch_stats b;
            b.n_tokens = N;
            b.n_seqs_valid = sv;
            b.n_groups_valid = qv;
            b.d_mean = d_mean;
            b.d_max = double(dmax);
            const double var = d2_mean - d_mean * d_mean;
            b.d_std = var > 0.0 ? sqrt(var) : 0.0;
            b.Y_sum = ysum;
            b.Y_mean = ymean;
            b.H_mean = H_mean;
            b.lr_mean = lr_mean;
            b.X = 0.0;
            b.trunc_frac = 0.0;
            b.w_mean = 0.0;
            b.alpha_mean = 0.0;
            *batch = b;
        }
    }
}

// K3: GRPO advantages.  LANES lanes share a prompt: a thread per prompt ran
// G dependent loads and G fp64 divisions one after the other (12.2 us for 64
// prompts of 8; 5.7 us with eight lanes).  LANES = 1 is for batches of so many
// prompts that the fp64 work of idle lanes would cost more than the latency.
template <int LANES>
__global__ void grpo_kernel(const float* __restrict__ R, const int32_t* __restrict__ goff, int Gn, int S, float adv_eps,
                            int ddof, int singleton_rule, float* __restrict__ adv, int32_t* flags) {
    constexpr int KEEP = 4;  // rewards per lane kept in registers between the passes
    const int64_t tid = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t g = tid / LANES;
    const int sub = int(tid % LANES);
    grid_begin();
    if (g >= Gn) return;  // the prompt's lanes leave together
    const unsigned team = LANES == 1 ? 0u : ((1u << LANES) - 1u) << (threadIdx.x & 31 & ~(LANES - 1));
    const int b = goff[g], e = goff[g + 1];
    if (b < 0 || b > e || e > S) {
        if (sub == 0) raise_flag(flags, ACRL_FLAG_BAD_OFFSETS);
        return;
    }
    const int G = e - b;
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
    const int rest = b + sub + KEEP * LANES;
    double sum = 0.0;
#pragma unroll
    for (int k = 0; k < KEEP; ++k)
        if (b + sub + k * LANES < e) sum += r[k];
    for (int64_t i = rest; i < e; i += LANES) sum += R[i];
    const double mean = total(sum) / G;
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
    const double var = G > ddof ? ss / (G - ddof) : 0.0;
    const double den = sqrt(var) + double(adv_eps);
#pragma unroll
    for (int k = 0; k < KEEP; ++k)
        if (b + sub + k * LANES < e) adv[b + sub + k * LANES] = den > 0.0 ? float((r[k] - mean) / den) : 0.f;
    for (int64_t i = rest; i < e; i += LANES) adv[i] = den > 0.0 ? float((R[i] - mean) / den) : 0.f;
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

// K4a: alpha per response, per-token weights and loss coefficients; a cluster
// of CTAs per response as in seq_stats_kernel.  The controller state is only
// read here (every CTA works out the X in force for itself); the finalising
// kernel writes it.
__global__ void __launch_bounds__(kSeqThreads) controller_weights_kernel(
    const acrl_controller_state* __restrict__ st, acrl_params p, const float* __restrict__ lr,
    const uint8_t* __restrict__ mask, int64_t T, const int64_t* __restrict__ so, int Gn, acrl_seq_stats* seq,
    const acrl_group_stats* __restrict__ grp, const acrl_batch_stats* __restrict__ batch,
    const float* __restrict__ adv, float* __restrict__ weight, float* __restrict__ coef, float* __restrict__ alpha_out,
    float* __restrict__ ent_coef) {
    constexpr int NW = kSeqThreads / 32, U = kSeqUnroll;
    __shared__ double sh[NW];
    __shared__ int sh_nt[NW];
    __shared__ float sh_alpha, sh_scale, sh_escale, sh_wmis;
    __shared__ int sh_cut;
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
        const ControllerMove mv = controller_move(*st, p, Ysum, ngv);
        double norm;
        if (p.agg == ACRL_AGG_TOKEN_MEAN)
            norm = double(batch->n_tokens);
        else
            norm = double(ngv) * double(has_g ? grp[g].n_valid_seqs : 0) * double(n);
        // one division, a different quotient in each lane: Y, X, A / norm, beta / norm
        double num = 0.0, den = 1.0;
        if (lane == 0) {
            if (p.y_gran == ACRL_Y_SEQUENCE) {
                num = sum_d;
                den = double(n);
            } else if (p.y_gran == ACRL_Y_BATCH) {
                num = Ysum;
                den = double(ngv);
            } else {
                num = Yg;
            }
        } else if (lane == 1) {
            num = mv.x_num;
            den = mv.x_den;
        } else if (lane == 2 || lane == 3) {
            num = lane == 2 ? double(A) : double(p.entropy_coeff);
            den = norm;
        }
        const double q = den > 0.0 ? num / den : 0.0;
        const double Y = __shfl_sync(0xffffffffu, q, 0), X = __shfl_sync(0xffffffffu, q, 1);
        const float scale = float(__shfl_sync(0xffffffffu, q, 2)), escale = float(__shfl_sync(0xffffffffu, q, 3));
        const float sgnf = A > 0.f ? 1.f : (A < 0.f ? -1.f : 0.f);
        float a = 0.f;
        if (p.mode == ACRL_MODE_TIS || p.mode == ACRL_MODE_MIS) {
            a = 1.f;
        } else if (p.mode == ACRL_MODE_ACRL_CONTINUOUS) {
            a = n > 0 ? -p.kappa * sgnf : 0.f;
        } else if ((p.mode == ACRL_MODE_ACRL || p.mode == ACRL_MODE_ACRL_FALLBACK) && mv.apply && X > 0.0 && n > 0) {
            a = float(double(p.gamma) * double(sgnf) * (1.0 - Y / X));
            if (p.mode == ACRL_MODE_ACRL_FALLBACK && !(Y > X)) a = 0.f;
        }
        if (lane == 0) {
            const bool cut = Si > logC;
            sh_alpha = a;
            sh_scale = scale;
            sh_escale = escale;
            sh_cut = cut;
            sh_wmis = (cut || isnan(Si)) ? 0.f : expf(Si);
            if (rank == 0) {
                seq[i].alpha = a;
                if (alpha_out) alpha_out[i] = a;
            }
        }
    }
    __syncthreads();
    const float alpha = sh_alpha, scale = sh_scale, escale = sh_escale, w_mis = sh_wmis;
    const bool mis_cut = sh_cut != 0;
    int nt = 0;
    double sw = 0.0;
    while (t0 < hi) {
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int64_t t = t0 + k * stride;
            if (t >= hi) break;
            float w = 0.f;
            if (m[k]) {
                if (p.mode == ACRL_MODE_NONE) {
                    w = 1.f;
                } else if (p.mode == ACRL_MODE_MIS) {
                    w = w_mis;
                    nt += mis_cut;
                } else {
                    // rho^0 = 1 even where the log-ratio is infinite (mu = 0); a NaN log-ratio gets weight 0
                    const float lrho = alpha == 0.f ? 0.f : alpha * l[k];
                    w = isnan(lrho) ? 0.f : expf(fminf(lrho, logC));
                    nt += lrho > logC;
                }
                sw += w;
            }
            weight[t] = w;
            coef[t] = w * scale;
            if (ent_coef) ent_coef[t] = m[k] ? escale : 0.f;
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

// K4b: the controller's new state and the batch metrics.
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
    ControllerMove mv = controller_move(*st, p, Ysum, ngv);
    // one division: w_mean, alpha_mean, trunc_frac, Y_mean (of the possibly all-reduced sum and prompt count), X
    double num = s, den = N;
    if (lane == 1) den = double(nsv);
    if (lane == 2) num = double(nt);
    if (lane == 3) num = Ysum, den = double(ngv);
    if (lane == 4) num = mv.x_num, den = mv.x_den;
    const double q = den > 0.0 ? num / den : 0.0;
    const double a_mean = __shfl_sync(0xffffffffu, q, 1), trunc = __shfl_sync(0xffffffffu, q, 2),
                 Ymean = __shfl_sync(0xffffffffu, q, 3), X = __shfl_sync(0xffffffffu, q, 4);
    if (lane == 0) {
        const bool was_calibrated = st->calibrated != 0;
        acrl_controller_state n = mv.next;
        n.X = X;
        const bool uses_x = p.mode == ACRL_MODE_ACRL || p.mode == ACRL_MODE_ACRL_FALLBACK;
        if (uses_x && mv.apply && !(X > 0.0)) {
            raise_flag(flags, ACRL_FLAG_X_NONPOS);
            n.flags |= ACRL_FLAG_X_NONPOS;
        }
        // moving-average X (off by default): this step used X, the next one uses the update
        if (was_calibrated && p.x_ema > 0.f) n.X = (1.0 - double(p.x_ema)) * X + double(p.x_ema) * Ymean;
        *st = n;
        batch->Y_mean = Ymean;
        batch->X = mv.apply ? X : 0.0;
        batch->trunc_frac = trunc;
        batch->w_mean = q;
        batch->alpha_mean = a_mean;
    }
}

// CTAs per response: enough to give the chip a few hundred CTAs, while each
// still has a round of tokens.
int ctas_per_response(int32_t S, int64_t T) {
    int c = 1;
    while (c < 8 && int64_t(S) * c * 2 <= kSeqCtas && T > int64_t(S) * c * kSeqTokens) c *= 2;
    return c;
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
    const int c = ctas_per_response(S, T);
    acrl_status st = ACRL_OK;
    if (S > 0)
        st = launch(seq_stats_kernel, int64_t(S) * c, kSeqThreads + 32, 0, c, s, logp_pi, logp_mu, mask, T, seq_offsets, S,
                    group_offsets, Gn, entropy, lr, d, seq, dev_flags);
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
    const int threads = 128;
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
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int c = ctas_per_response(S, T);
    acrl_status st = ACRL_OK;
    if (S > 0)
        st = launch(controller_weights_kernel, int64_t(S) * c, kSeqThreads, 0, c, s, state, *p, lr, mask, T, seq_offsets, Gn,
                    seq, grp, batch, adv, weight, coef, alpha, ent_coef);
    if (st != ACRL_OK) return st;
    return launch(controller_finalize_kernel, 1, kFinThreads, 0, 0, s, state, *p, S, seq, batch, dev_flags);
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
