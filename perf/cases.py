"""The work that this library is timed on: whole passes through its public entry points, as a training program
calls them, over the range of sizes such programs have.

A case is a dict of plain values; `kind` says which call it is:

  step        AcrlStep.run: the on-policy pass of one optimiser step, called eagerly (statistics, discrepancy,
              advantages, controller, then the loss and dL/dlogits);
  graph       the same pass captured once by AcrlStep.capture and replayed (fixed-shape training loops);
  autograd    acrl_loss and its backward, the way a model's own loss is used, the loss scaled as gradient
              accumulation scales it;
  cached_old  loss_grad_logits on the logits of a later update over the same rollout: the old policy's log-probs are
              cached, the log-sum-exp is recomputed in the call, ratios are clipped;
  weights     importance_weights: the weights alone from cached per-token log-probs;
  lmhead      lmhead_logits_stats + lmhead_merge: the LM head on the tensor cores, statistics in its epilogue;
  lmhead_noalloc  the same in one call for callers that cannot allocate (rollout scoring, plugins).

HostPipeline is left out: it runs the kernels of `step` behind copies at the host link's rate, which the host
decides.  Sizes are those of the repository's workloads (4 x 256 tokens at V = 4,096; 8 x 8 responses at V = 32,000
right-padded; 8 responses a prompt at V = 151,936; 64 x 8 responses of up to 2,048 tokens) and generic ones
between them.  Response lengths, masks and rewards follow from the case alone, so that shapes and work do not change
with the seed; every other value is drawn from the seed."""

import math
import random
from types import SimpleNamespace

import torch

import paper_2607_24062_gb300 as acrl
from paper_2607_24062_gb300 import api

DEV = "cuda"
E4M3_MAX = 448.0
CHUNK_ELEMS = 1 << 28        # elements of fp32 work at a time while making inputs
EXACT_ELEMS = 1 << 27        # the same in 64 bits
MAX_ELEMS = 5_600_000_000    # logits of the largest step
MAX_OLD_ELEMS = 2_500_000_000
CLIP_EPS = 0.2
X_INIT = 0.004               # the reference discrepancy of a run under way, fixed before this batch


# ---------------------------------------------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------------------------------------------

def _rows(kind, prompts, group, lo, hi, V, **more):
    """A case over responses: `prompts` x `group` responses of lo..hi tokens, each padded to a multiple of `pad`."""
    c = {"kind": kind, "prompts": prompts, "group": group, "lo": lo, "hi": hi, "V": V, "pad": 0, "dist": "normal",
         "scale": 2.0, "entropy_coeff": 0.0}
    c.update(more)
    return c


def listed():
    return [
        # the smallest whole step: four short responses, a small vocabulary; called eagerly, launches and host work count
        dict(_rows("step", 4, 1, 256, 256, 4096), name="tiny_step"),
        # the same step replayed from a CUDA graph: the latency of its chain of kernels
        dict(_rows("graph", 4, 1, 256, 256, 4096), name="tiny_graph"),
        # one micro-batch of a large-vocabulary model: a few short responses, with the entropy bonus
        dict(_rows("step", 1, 4, 32, 256, 151936, dist="t4", entropy_coeff=0.001), name="micro_step"),
        # a GRPO batch of 64 right-padded responses, mid-size vocabulary
        dict(_rows("step", 8, 8, 64, 1024, 32000, pad=64, dist="boost", scale=3.0), name="grpo_step"),
        # a large-vocabulary batch, ~37 k tokens: the logits fill HBM many times over L2
        dict(_rows("step", 4, 8, 256, 2048, 151936, dist="t4"), name="qwen_step"),
        # the loss as an autograd node of the model, one of four accumulated micro-batches, a vocabulary that is no
        # multiple of eight
        dict(_rows("autograd", 2, 4, 64, 1024, 20011, pad=16, dist="boost", scale=3.0, loss_scale=0.25),
             name="autograd_step"),
        # the second update on a rollout: lse recomputed, PPO ratio against cached log-probs
        dict(_rows("cached_old", 2, 8, 256, 1024, 151936, dist="t4"), name="cached_old_large"),
        # the same on one micro-batch at a middle vocabulary
        dict(_rows("cached_old", 1, 4, 64, 512, 49152), name="cached_old_micro"),
        # the weights of the paper's overhead measurement: 64 x 8 responses, lengths up to 2,048, log-probs only
        dict(_rows("weights", 64, 8, 1, 2048, 0), name="weights"),
        # the LM head of a large-vocabulary model over one micro-batch of 4,096 tokens
        {"kind": "lmhead", "M": 4096, "K": 4096, "N": 151936, "name": "lmhead_large"},
        # ragged rows and columns, mid-size vocabulary, a small hidden size
        {"kind": "lmhead", "M": 1003, "K": 2048, "N": 32001, "name": "lmhead_mid"},
        # scoring a handful of tokens: the weight's own bytes bound it
        {"kind": "lmhead_noalloc", "M": 48, "K": 4096, "N": 151936, "name": "lmhead_decode"},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "graph", "autograd", "cached_old", "cached_old", "weights", "lmhead",
                       "lmhead", "lmhead_noalloc"])
    if kind == "weights":
        prompts, group = _log_int(rng, 1, 64), rng.choice([1, 2, 4, 8])
        hi = _log_int(rng, 16, 2048)
        return _rows(kind, prompts, group, rng.randint(1, hi), hi, 0, mode=rng.choice([acrl.MODE_ACRL, acrl.MODE_TIS, acrl.MODE_MIS]))
    if kind == "lmhead":
        return {"kind": kind, "M": _log_int(rng, 16, 4096), "K": 8 * _log_int(rng, 64, 512), "N": _log_int(rng, 4096, 151936)}
    if kind == "lmhead_noalloc":
        N = _log_int(rng, 4096, 151936)
        most = (16 << 20) // (16 * ((N + 255) // 256))
        return {"kind": kind, "M": _log_int(rng, 1, min(1024, most)), "K": 8 * _log_int(rng, 64, 512), "N": N}
    V = _log_int(rng, 2048, 151936)
    if rng.random() < 0.5:
        V = V // 8 * 8
    most = {"graph": 4096, "cached_old": min(16384, MAX_OLD_ELEMS // V)}.get(kind, min(40000, MAX_ELEMS // V))
    group = rng.choice([1, 2, 4, 8])
    rows = _log_int(rng, 128, most)
    prompts = _log_int(rng, 1, max(1, min(16, rows // (8 * group))))
    hi = max(8, rows // (prompts * group))
    c = _rows(kind, prompts, group, rng.randint(max(1, hi // 8), hi), hi, V, pad=rng.choice([0, 0, 8]) if hi >= 64 else 0,
              dist=rng.choice(["normal", "t4", "boost"]), scale=rng.choice([2.0, 3.0]),
              entropy_coeff=rng.choice([0.0, 0.0, 0.001]))
    if kind == "autograd":
        c["loss_scale"] = rng.choice([1.0, 0.5, 0.25])
        c["entropy_coeff"] = 0.0
    if kind == "cached_old":
        c["entropy_coeff"] = 0.0
    return c


# ---------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------

def _structure(case):
    """Lengths, offsets, mask and binary rewards: from the case's sizes alone."""
    r = random.Random("%(prompts)d %(group)d %(lo)d %(hi)d %(pad)d" % case)
    S, pad = case["prompts"] * case["group"], max(1, case["pad"])
    lengths = [r.randint(case["lo"], case["hi"]) for _ in range(S)]
    rewards = [1.0 if r.random() < 0.3 else 0.0 for _ in range(S)]
    rewards[0] = 1.0
    offsets, mask = [0], bytearray()
    for n in lengths:
        rows = (n + pad - 1) // pad * pad
        mask += b"\x01" * n + b"\x00" * (rows - n)
        offsets.append(offsets[-1] + rows)
    G = case["group"]
    live = 0    # rows that carry a policy gradient: valid, and the response's advantage is not zero
    for i, n in enumerate(lengths):
        R = rewards[i // G * G: i // G * G + G]
        if (G == 1 and R[0] != 0.0) or (G > 1 and len(set(R)) > 1):
            live += n
    return SimpleNamespace(S=S, Gn=case["prompts"], T=offsets[-1], valid=sum(lengths), live=live, offsets=offsets, mask=mask,
                           rewards=rewards, groups=[g * G for g in range(case["prompts"] + 1)])


def _device_structure(st):
    return SimpleNamespace(
        S=st.S, Gn=st.Gn, T=st.T,
        mask=torch.frombuffer(st.mask, dtype=torch.uint8).to(DEV),
        rewards=torch.tensor(st.rewards, dtype=torch.float32, device=DEV),
        seq_offsets=torch.tensor(st.offsets, dtype=torch.int64, device=DEV),
        group_offsets=torch.tensor(st.groups, dtype=torch.int32, device=DEV))


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _fill_logits(out, V, dist, scale, gen):
    """Rows of normal values, of Student-t values (4 degrees of freedom, heavy tails), or of normal values of which one
    in a hundred is raised by 8 (a peaked policy)."""
    T = out.shape[0]
    step = max(1, CHUNK_ELEMS // V)
    for r0 in range(0, T, step):
        n = min(step, T - r0)
        z = torch.randn((n, V), generator=gen, device=DEV).mul_(scale)
        if dist == "t4":     # chi2 with 4 degrees of freedom is -2 ln(u v)
            u = torch.rand((n, V), generator=gen, device=DEV)
            u.mul_(torch.rand((n, V), generator=gen, device=DEV)).clamp_(min=1e-30).log_().mul_(-0.5)
            z.mul_(u.rsqrt_())
        elif dist == "boost":
            z.add_(torch.rand((n, V), generator=gen, device=DEV).lt_(0.01).mul_(8.0))
        out[r0:r0 + n, :V] = z
        del z


def _sampled(logits, V, gen):
    """Token ids drawn from softmax(logits), and the log-probs that an engine with FP8 (E4M3, per-row scale) logits
    gives them."""
    T = logits.shape[0]
    ids = torch.empty(T, dtype=torch.int32, device=DEV)
    logp_mu = torch.empty(T, dtype=torch.float32, device=DEV)
    step = max(1, CHUNK_ELEMS // V)
    for r0 in range(0, T, step):
        r1 = min(T, r0 + step)
        z = logits[r0:r1, :V].float()
        u = torch.empty_like(z).exponential_(generator=gen).log_().neg_().add_(z)     # Gumbel-max
        a = u.argmax(dim=1)
        del u
        s = (z.abs().amax(dim=1, keepdim=True) / E4M3_MAX).clamp_(min=1e-30)
        q = (z / s).clamp_(-E4M3_MAX, E4M3_MAX).to(torch.float8_e4m3fn).float().mul_(s)
        ids[r0:r1] = a.to(torch.int32)
        logp_mu[r0:r1] = (q.gather(1, a.view(-1, 1)) - q.logsumexp(dim=1, keepdim=True)).view(-1)
        del z, q
    return ids, logp_mu


def _inputs(case, seed):
    """What the rollout and the model hand over, on the GPU."""
    gen = _gen(seed)
    if case["kind"] in ("lmhead", "lmhead_noalloc"):
        M, K, N = case["M"], case["K"], case["N"]
        hidden = torch.randn((M, K), generator=gen, device=DEV).to(torch.bfloat16)
        weight = torch.empty((N, K), dtype=torch.bfloat16, device=DEV)
        for r0 in range(0, N, 16384):
            n = min(16384, N - r0)
            weight[r0:r0 + n] = torch.randn((n, K), generator=gen, device=DEV).mul_(1.25 / math.sqrt(K))
        ids = torch.randint(0, N, (M,), generator=gen, device=DEV, dtype=torch.int32)
        return SimpleNamespace(hidden=hidden, weight=weight, ids=ids)
    st = _structure(case)
    x = _device_structure(st)
    if case["kind"] == "weights":    # log-probs only; one response in ten is off by more than the quantisation
        x.logp_old = torch.empty(x.T, device=DEV).exponential_(generator=gen).mul_(-2.0)
        noise = torch.randn(x.T, generator=gen, device=DEV)
        rows = torch.tensor([b - a for a, b in zip(st.offsets, st.offsets[1:])], device=DEV)
        off = torch.rand(x.S, generator=gen, device=DEV).lt(0.1).float().mul_(0.3).add_(0.02)
        x.logp_mu = (x.logp_old + noise * torch.repeat_interleave(off, rows)).clamp_(max=0.0)
        return x
    V = case["V"]
    ld = (V + 7) // 8 * 8
    x.full = torch.zeros((x.T, ld), dtype=torch.bfloat16, device=DEV)
    _fill_logits(x.full, V, case["dist"], case["scale"], gen)
    x.ids, x.logp_mu = _sampled(x.full, V, gen)
    x.logp_mu.add_(torch.randn(x.T, generator=gen, device=DEV).mul_(0.02)).clamp_(max=0.0)
    if case["kind"] == "cached_old":
        # the old policy is a few updates back: its log-probs differ by ~0.1, so some ratios leave the clip range
        x.old_logp = (x.logp_mu + torch.randn(x.T, generator=gen, device=DEV).mul_(0.1)).clamp_(max=0.0)
        rows = torch.tensor([b - a for a, b in zip(st.offsets, st.offsets[1:])], device=DEV)
        adv = _advantages(x.rewards.double(), case["group"])
        w = torch.randn(x.T, generator=gen, device=DEV).mul_(0.05).exp_()
        x.coef = (w * x.mask * torch.repeat_interleave(adv / rows / x.S, rows).float())
    return x


# ---------------------------------------------------------------------------------------------------------------
# the passes
# ---------------------------------------------------------------------------------------------------------------

def _figures(batch):
    """The statistics of the batch struct (its eleven doubles) as a tensor over the struct's own bytes."""
    return batch[16:].view(torch.float64)


def prepare(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    x.kind = kind
    if kind in ("lmhead", "lmhead_noalloc"):
        M, N = case["M"], case["N"]
        x.N = N
        x.logits = torch.empty((M, (N + 7) // 8 * 8), dtype=torch.bfloat16, device=DEV)
        x.lse, x.logp, x.entropy = (torch.empty(M, device=DEV) for _ in range(3))
        x.flags = api.new_flags(DEV)
        if kind == "lmhead":
            x.partials = torch.empty(api.lmhead_workspace_bytes(M, N) // 4, device=DEV)
        x.out = {"logits": x.logits[:, :N], "lse": x.lse, "logp": x.logp, "entropy": x.entropy}
        return x
    if kind == "weights":
        x.params = acrl.Params(mode=case.get("mode", acrl.MODE_ACRL))
        x.state = acrl.controller_init(x.params, device=DEV)
        return x
    V, ld = case["V"], x.full.stride(0)
    if kind == "cached_old":
        x.grad = torch.empty_like(x.full)
        x.token_loss, x.loss = torch.empty(x.T, device=DEV), torch.empty(1, device=DEV)
        x.flags = api.new_flags(DEV)
        x.V = V
        x.out = {"grad": x.grad[:, :V], "token_loss": x.token_loss, "loss": x.loss}
        return x
    params = acrl.Params(entropy_coeff=case["entropy_coeff"], X_init=X_INIT)
    step = x.step = acrl.AcrlStep(x.T, V, ld, x.S, x.Gn, params, device=DEV)
    x.args = (x.ids, x.mask, x.logp_mu, x.rewards, x.seq_offsets, x.group_offsets)
    x.out = {"lse": step.lse, "logp": step.logp, "entropy": step.entropy, "lr": step.disc.lr, "d": step.disc.d,
             "adv": step.adv, "alpha": step.alpha, "weight": step.weight, "coef": step.coef,
             "batch": _figures(step.disc.batch), "token_loss": step.token_loss}
    if kind == "autograd":
        x.logits = x.full[:, :V].detach().requires_grad_(True)
        x.loss_scale = case["loss_scale"]
        return x
    x.out.update(grad=step.grad[:, :V], loss=step.loss)
    if kind == "graph":
        x.logits = x.full
        x.graph = step.capture(x)
    return x


def run(x):
    if x.kind == "step":
        x.step.run(x.full, *x.args)
        return x.out
    if x.kind == "graph":
        x.graph.replay()
        return x.out
    if x.kind == "autograd":
        loss = acrl.acrl_loss(x.step, x.logits, *x.args)
        grad, = torch.autograd.grad(loss * x.loss_scale, x.logits)
        return dict(x.out, grad=grad, loss=loss.detach())
    if x.kind == "cached_old":
        acrl.loss_grad_logits(x.full, x.ids, x.mask, None, x.old_logp, x.coef, CLIP_EPS, V=x.V, grad=x.grad,
                              token_loss=x.token_loss, loss=x.loss, flags=x.flags)
        return x.out
    if x.kind == "weights":
        w = acrl.importance_weights(x.state, x.params, x.logp_old, x.logp_mu, x.mask, x.rewards, x.seq_offsets,
                                    x.group_offsets)
        return {"weight": w.weight, "coef": w.coef, "adv": w.adv, "alpha": w.alpha, "lr": w.disc.lr, "d": w.disc.d,
                "batch": _figures(w.disc.batch)}
    if x.kind == "lmhead":
        api.lmhead_logits_stats(x.hidden, x.weight, N=x.N, logits=x.logits, partials=x.partials, flags=x.flags)
        api.lmhead_merge(x.partials, x.logits, x.ids, None, N=x.N, lse=x.lse, logp=x.logp, entropy=x.entropy, flags=x.flags)
        return x.out
    api.lmhead_stats_noalloc(x.hidden, x.weight, x.ids, None, N=x.N, logits=x.logits, lse=x.lse, logp=x.logp,
                             entropy=x.entropy, flags=x.flags)
    return x.out


def work(case):
    """Inputs read once, outputs written once.  A step's logits count once, although the weights of a prompt need all of
    its rows before the gradient can start, so that a batch larger than L2 reads them twice."""
    kind = case["kind"]
    if kind in ("lmhead", "lmhead_noalloc"):
        M, K, N = case["M"], case["K"], case["N"]
        return {"bytes": 2 * (M * K + N * K + M * N) + 16 * M, "flops": 2 * M * N * K}
    st = _structure(case)
    if kind == "weights":    # reads pi, mu (4 B each) and the mask; writes lr, d, weight, coef
        return {"bytes": 25 * st.T + 100 * st.S, "flops": 0}
    V, T = case["V"], st.T
    if kind == "cached_old":
        return {"bytes": 2 * V * (st.live + T) + 21 * T, "flops": 0}
    if kind == "autograd" and case["loss_scale"] != 1.0:
        return {"bytes": 2 * V * (st.valid + T) + 57 * T, "flops": V * T}
    return {"bytes": 2 * V * (st.valid + T) + 57 * T, "flops": 0}


def tolerance(case):
    """Measured against `exact`: bf16 gradients and logits are 1.4e-3 to 1.9e-3 off (their rounding); the fp32 vectors
    of `weights` 1e-8 to 4e-6 (a distance of two close probabilities, an exponent 1 - Y / X)."""
    return {"rel": 1e-5} if case["kind"] == "weights" else {"rel": 7e-3}


# ---------------------------------------------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------------------------------------------

def _advantages(R, G):
    R = R.view(-1, G)
    if G == 1:
        return R.reshape(-1).clone()
    c = R - R.mean(dim=1, keepdim=True)
    std = (c.square().sum(dim=1, keepdim=True) / (G - 1)).sqrt()
    return torch.where((c == 0).all(dim=1, keepdim=True), torch.zeros_like(c), c / (std + float(torch.tensor(1e-6)))).reshape(-1)


def _exact_weights(case, x, logp, logp_mu, entropy, mode, entropy_coeff, X_init):
    """Discrepancy, advantages, controller (X calibrated on this batch where X_init is 0) and loss coefficients."""
    f = lambda v: float(torch.tensor(v, dtype=torch.float32))  # noqa: E731  parameters are 32-bit in the call
    gamma, C, G = f(0.65), f(3.0), case["group"]
    m = x.mask.double()
    rows = x.seq_offsets[1:] - x.seq_offsets[:-1]
    seg = torch.repeat_interleave(torch.arange(x.S, device=DEV), rows)
    total = lambda v: torch.zeros(x.S, dtype=torch.float64, device=DEV).index_add_(0, seg, v)  # noqa: E731
    lr = (logp - logp_mu) * m
    d = (logp.exp() - logp_mu.exp()).abs() * m
    n = total(m)
    D = total(d) / n
    Y = D.view(-1, G).mean(dim=1)
    X = torch.full_like(Y[0], X_init) if X_init > 0 else Y.mean()
    adv = _advantages(x.rewards.double(), G)
    alpha = gamma * adv.sign() * (1 - Y.repeat_interleave(G) / X)
    if mode in (acrl.MODE_TIS, acrl.MODE_MIS):
        alpha = torch.ones_like(adv)
    if mode == acrl.MODE_MIS:
        Si = total(lr)
        cut = Si > math.log(C)
        w = torch.where(cut, torch.zeros_like(Si), Si.exp())[seg] * m
        trunc = (cut[seg] * m).sum()
    else:
        e = alpha[seg] * lr
        w = e.clamp(max=math.log(C)).exp() * m
        trunc = ((e > math.log(C)) * m).sum()
    norm = x.Gn * G * n
    coef = w * (adv / norm)[seg]
    ent_coef = m * (f(entropy_coeff) / norm)[seg]
    N = m.sum()
    mean = d.sum() / N
    batch = torch.stack([mean, d.max(), (d.square().sum() / N - mean * mean).clamp(min=0).sqrt(), Y.sum(), Y.mean(),
                         (entropy * m).sum() / N, lr.sum() / N, X, trunc / N, w.sum() / N, alpha.mean()])
    return SimpleNamespace(lr=lr, d=d, adv=adv, alpha=alpha, weight=w, coef=coef, ent_coef=ent_coef, batch=batch)


def _exact_rows(x, V):
    """lse, log-prob of the sampled token and entropy of every valid row."""
    lse, logp, ent = (torch.zeros(x.T, dtype=torch.float64, device=DEV) for _ in range(3))
    step = max(1, EXACT_ELEMS // V)
    for r0 in range(0, x.T, step):
        s = slice(r0, min(x.T, r0 + step))
        z = x.full[s, :V].double()
        lse[s] = z.logsumexp(dim=1)
        za = z.gather(1, x.ids[s].long().view(-1, 1)).view(-1)
        logp[s] = za - lse[s]
        z -= lse[s, None]
        ent[s] = -(z.exp() * z).sum(dim=1)
    m = x.mask.double()
    return lse * m, logp * m, ent * m


def _exact_grad(x, V, lse, c, e, H):
    grad = torch.zeros((x.T, V), dtype=torch.float64, device=DEV)
    step = max(1, EXACT_ELEMS // V)
    for r0 in range(0, x.T, step):
        s = slice(r0, min(x.T, r0 + step))
        lp = x.full[s, :V].double() - lse[s, None]
        p = lp.exp()
        g = p * c[s, None]
        if e is not None:
            g += e[s, None] * p * (lp + H[s, None])
        g.scatter_add_(1, x.ids[s].long().view(-1, 1), -c[s, None])
        live = (c[s] != 0) if e is None else (c[s] != 0) | (e[s] != 0)
        grad[s] = torch.where(live[:, None], g, torch.zeros_like(g))
    return grad


def exact(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    if kind in ("lmhead", "lmhead_noalloc"):
        N, logits = case["N"], []
        h = x.hidden.double()
        for r0 in range(0, N, 16384):
            logits.append(h @ x.weight[r0:r0 + 16384].double().T)
        z = torch.cat(logits, dim=1)
        del logits
        x.full, x.T, x.mask = z.to(torch.bfloat16), case["M"], torch.ones(case["M"], dtype=torch.uint8, device=DEV)
        lse, logp, ent = _exact_rows(x, N)     # the statistics are those of the stored (rounded) logits
        return {"logits": z, "lse": lse, "logp": logp, "entropy": ent}
    if kind == "weights":
        mode = case.get("mode", acrl.MODE_ACRL)
        w = _exact_weights(case, x, x.logp_old.double(), x.logp_mu.double(), torch.zeros(x.T, dtype=torch.float64, device=DEV), mode, 0.0, 0.0)
        return {k: getattr(w, k) for k in ("weight", "coef", "adv", "alpha", "lr", "d", "batch")}
    V = case["V"]
    lse, logp, ent = _exact_rows(x, V)
    if kind == "cached_old":
        c0 = x.coef.double()
        r = (logp - x.old_logp.double()).exp()
        lo, hi = 1.0 - CLIP_EPS, 1.0 + CLIP_EPS
        up = c0 >= 0
        gate = torch.where(up, r <= hi, r >= lo)
        rc = r.clamp(lo, hi)
        token_loss = -c0 * torch.where(up, torch.minimum(r, rc), torch.maximum(r, rc))
        token_loss = torch.where(c0 == 0, torch.zeros_like(c0), token_loss)
        return {"grad": _exact_grad(x, V, lse, torch.where(gate, c0 * r, torch.zeros_like(c0)), None, None),
                "token_loss": token_loss, "loss": token_loss.sum().view(1)}
    w = _exact_weights(case, x, logp, x.logp_mu.double(), ent, acrl.MODE_ACRL, case["entropy_coeff"], X_INIT)
    bonus = case["entropy_coeff"] > 0
    token_loss = -w.coef - (w.ent_coef * ent if bonus else 0.0)
    out = {"lse": lse, "logp": logp, "entropy": ent, "lr": w.lr, "d": w.d, "adv": w.adv, "alpha": w.alpha,
           "weight": w.weight, "coef": w.coef, "batch": w.batch, "token_loss": token_loss,
           "grad": _exact_grad(x, V, lse, w.coef, w.ent_coef if bonus else None, ent),
           "loss": None}    # advantages sum to zero in a prompt: the sum cancels, its rounding is not its terms'
    if kind == "autograd":
        out["grad"] *= case["loss_scale"]
    return out
