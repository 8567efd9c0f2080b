// acrl_step: the whole on-policy pass in one call.  Host code only: with a small
// batch the device waits for the host, and one call with every pointer costs less
// than half of the five (a step of 4 x 256 tokens at V = 4,096 called from Python:
// 82 us as five calls and nine launches, 35 as one call and four).
#include "acrl_host.h"

using namespace acrl;

extern "C" acrl_status acrl_step(acrl_controller_state* state, const acrl_params* p, const acrl_bf16* logits, int64_t T,
                                 int64_t V, int64_t ld, const int32_t* ids, const uint8_t* mask, const float* logp_mu,
                                 const float* rewards, const int64_t* seq_offsets, int32_t S, const int32_t* group_offsets,
                                 int32_t Gn, float* lse, float* logp, float* entropy, float* lr, float* d,
                                 acrl_seq_stats* seq, acrl_group_stats* grp, acrl_batch_stats* batch, float* adv,
                                 float* weight, float* coef, float* alpha, float* ent_coef, acrl_bf16* grad,
                                 float* token_loss, float* loss, int32_t* dev_flags, acrl_stream stream) {
    // what the later calls would refuse, before the first one launches anything
    if (!state || !params_ok(p) || T < 0 || S < 0 || Gn < 0) return ACRL_ERR_INVALID_ARG;
    if (!seq_offsets || !group_offsets || !batch || !loss || !dev_flags) return ACRL_ERR_INVALID_ARG;
    if (T > 0 && (!logp_mu || !lr || !d || !weight || !coef || !grad || !token_loss || !aligned16(grad)))
        return ACRL_ERR_INVALID_ARG;
    if ((S > 0 && (!seq || !rewards || !adv)) || (Gn > 0 && !grp)) return ACRL_ERR_INVALID_ARG;
    acrl_status st = acrl_token_stats(logits, T, V, ld, ids, mask, lse, logp, entropy, dev_flags, stream);
    if (st == ACRL_OK)
        st = acrl_importance_weights(state, p, logp, logp_mu, mask, T, rewards, seq_offsets, S, group_offsets, Gn, entropy,
                                     lr, d, seq, grp, batch, adv, weight, coef, alpha, ent_coef, dev_flags, stream);
    if (st == ACRL_OK)
        st = acrl_loss_grad_logits(logits, T, V, ld, ids, mask, lse, nullptr, coef, ent_coef ? entropy : nullptr, ent_coef,
                                   p->clip_eps, grad, token_loss, loss, dev_flags, stream);
    return st;
}
