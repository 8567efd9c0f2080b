"""The O(T) calls where their kernels change shape: one CTA per response or a
cluster of two, four or eight; responses shorter than a round of threads and
empty ones; more responses than the batch kernel keeps in shared memory; one,
two and three steps of the prompt search; prompts of one, of a few and of more
responses than lanes; losses summed by one CTA and by the cluster.  Against
the float64 oracle, with the bars of the parity tests."""

import numpy as np
import pytest
import torch

import oracle as O
from parity import assert_close_abs, assert_close_rel, compare_batch, compare_grp, compare_seq, host, oracle_params

pytestmark = pytest.mark.gpu

import paper_2607_24062_gb300 as acrl  # noqa: E402
from paper_2607_24062_gb300 import _abi, api  # noqa: E402

DEV = "cuda"

# prompts x responses, lengths lo..hi
_SHAPES = [(1, 1, 1, 1), (1, 1, 255, 255), (1, 1, 257, 257), (1, 1, 2049, 2049), (1, 3, 0, 1600), (2, 2, 500, 700),
           (4, 8, 200, 2048), (19, 8, 500, 600), (20, 8, 1, 300), (33, 2, 0, 40), (1025, 2, 0, 9), (1, 70, 1, 30),
           (5, 33, 1, 20)]


def _tokens(Q, G, lo, hi, seed):
    rng = np.random.default_rng(seed)
    lengths = rng.integers(lo, hi + 1, size=Q * G)
    so = np.concatenate([[0], np.cumsum(lengths)])
    T = int(so[-1])
    pi = -2.0 * rng.exponential(size=T)
    mu = np.minimum(pi + 0.05 * rng.normal(size=T), 0.0)
    mask = (rng.random(T) < 0.9).astype(np.uint8)
    R = (rng.random(Q * G) < 0.4).astype(np.float32) + rng.integers(0, 3, size=Q * G) / 8.0
    go = (np.arange(Q + 1) * G).astype(np.int32)
    f = lambda x, dt: torch.tensor(np.asarray(x), dtype=dt, device=DEV)  # noqa: E731
    return (f(pi, torch.float32), f(mu, torch.float32), f(mask, torch.uint8), f(so, torch.int64), f(go, torch.int32),
            f(R, torch.float32), f(rng.random(T), torch.float32))


@pytest.mark.parametrize("Q,G,lo,hi", _SHAPES)
@pytest.mark.parametrize("mode,y_gran", [(acrl.MODE_ACRL, acrl.Y_GROUP), (acrl.MODE_ACRL, acrl.Y_SEQUENCE),
                                         (acrl.MODE_MIS, acrl.Y_GROUP)])
def test_shapes_match_oracle(Q, G, lo, hi, mode, y_gran):
    pi, mu, mask, so, go, R, H = _tokens(Q, G, lo, hi, seed=Q * 1000 + G)
    p = acrl.Params(mode=mode, y_gran=y_gran, C=1.1)
    op = oracle_params(p)
    state, flags = api.controller_init(p), api.new_flags()
    disc = api.seq_discrepancy(pi, mu, mask, so, go, H, flags=flags)
    adv = api.grpo_advantage(R, go, p, flags=flags)
    w, coef, alpha = api.controller_step(state, p, disc, mask, so, go, adv, flags=flags)
    lr, d, seq, grp, batch, f0 = O.seq_discrepancy(host(pi).astype(np.float64), host(mu).astype(np.float64), host(mask),
                                                   host(so), host(go), host(H).astype(np.float64))
    oadv = O.grpo_advantage(host(R).astype(np.float64), host(go), op)
    ow, oalpha, ost, info, f1 = O.controller_step(O.controller_init(op), op, lr, host(mask), host(so), host(go), seq,
                                                  grp, batch, oadv)
    assert api.read_flags(flags) == f0 | f1
    compare_seq(disc.seq_host(), seq)
    compare_grp(disc.grp_host(), grp)
    gb = disc.batch_host()
    compare_batch(gb, batch)
    assert_close_rel(host(adv), oadv, floor=1e-6, what="adv")
    assert_close_rel(host(w), ow, floor=1e-7, what="weight")
    assert_close_rel(host(alpha), oalpha, floor=1e-6, what="alpha")
    ocoef = O.loss_coefficients(ow, oadv, host(mask), host(so), seq, grp, batch, op)
    assert_close_rel(host(coef), ocoef, floor=1e-9, what="coef")
    gs = disc.seq_host()
    assert_close_rel(gs["sum_w"], np.array([ow[a:b].sum() for a, b in zip(host(so), host(so)[1:])]), floor=1e-6,
                     what="sum_w")
    st = api.read_state(state)
    assert int(st["step"]) == 1
    assert_close_rel(st["X"], ost.X, floor=1e-12, what="X")
    N = max(1, int(host(mask).sum()))
    assert_close_rel(gb["w_mean"], ow.sum() / N, floor=1e-9, what="w_mean")
    assert_close_abs(gb["trunc_frac"], info["trunc_frac"], 2.0 / N, what="trunc_frac")   # ties at ln C


@pytest.mark.parametrize("T", [0, 1, 3, 255, 1024, 4097, 32768, 32769, 100003, 262147])
def test_loss_sum_sizes(T):
    """Sums of T values, from a 16-byte-aligned start and from one that is not."""
    gen = torch.Generator(device=DEV).manual_seed(T)
    v = torch.randn(T + 1, generator=gen, device=DEV)
    for off in (0, 1):
        x = v[off:off + T]
        want = float(x.double().sum())
        # fp32 sums of four values, then fp64: 2 roundings of 2^-24 on a group's partial sums
        bound = 4 * 2.0 ** -24 * float(x.double().abs().sum()) + 1e-30
        assert abs(float(api.reduce_loss(x)) - want) <= bound
        assert torch.equal(api.reduce_loss(x), api.reduce_loss(x))


def _three_calls_and_one(p, steps, pi, mu, mask, so, go, R, H, ent):
    """Every output byte of the three calls and of the one that does all, after `steps` steps of one controller."""
    outs = []
    for one in (False, True):
        T, S, Gn = pi.numel(), so.numel() - 1, go.numel() - 1
        state, flags = api.controller_init(p), api.new_flags()
        f = lambda n: torch.full((n,), 7.0, device=DEV)  # noqa: E731
        disc = api.Discrepancy(f(T), f(T), api.struct_buffer(_abi.SEQ_DTYPE, S), api.struct_buffer(_abi.GRP_DTYPE, Gn),
                               api.struct_buffer(_abi.BATCH_DTYPE, 1), S, Gn)
        adv, w, coef, alpha, ec = f(S), f(T), f(T), f(S), (f(T) if ent else None)
        for _ in range(steps):
            if one:
                api.importance_weights(state, p, pi, mu, mask, R, so, go, H, out=disc, adv=adv, weight=w, coef=coef,
                                       alpha=alpha, ent_coef=ec, flags=flags)
            else:
                api.seq_discrepancy(pi, mu, mask, so, go, H, out=disc, flags=flags)
                api.grpo_advantage(R, go, p, adv=adv, flags=flags)
                api.controller_step(state, p, disc, mask, so, go, adv, weight=w, coef=coef, alpha=alpha, ent_coef=ec,
                                    flags=flags)
        outs.append([host(x.view(torch.uint8)) for x in
                     (state, flags, disc.lr, disc.d, disc.seq, disc.grp, disc.batch, adv, w, coef, alpha) +
                     ((ec,) if ent else ())])
    return outs


def _assert_same_bytes(a, b):
    names = "state flags lr d seq grp batch adv weight coef alpha ent_coef".split()
    assert not [(nm, np.flatnonzero(x != y)[:8].tolist()) for nm, x, y in zip(names, a, b) if not np.array_equal(x, y)]


# one part and one prompt; two, four and eight parts a response; parts that fill one group and both groups of the
# cluster's CTAs; more than a round of tokens a thread; empty responses; the largest counts it takes and the next
_ONE_SHAPES = [(1, 1, 1, 1), (1, 1, 9000, 9000), (4, 1, 256, 256), (2, 4, 64, 1100), (1, 9, 0, 700), (4, 4, 100, 520),
               (8, 4, 0, 260), (32, 1, 1, 200), (33, 1, 1, 9), (1, 33, 1, 9), (3, 1, 300, 12000),
               # beyond it: advantages beside the batch statistics, in one, in several and (too many prompts) in no CTAs there
               (17, 3, 0, 40), (64, 8, 0, 30), (1024, 1, 0, 3), (1025, 1, 0, 3)]


@pytest.mark.parametrize("Q,G,lo,hi", _ONE_SHAPES)
@pytest.mark.parametrize("kw", [dict(), dict(y_gran=acrl.Y_BATCH, agg=acrl.AGG_TOKEN_MEAN, calib_steps=2),
                                dict(mode=acrl.MODE_MIS, C=1.1), dict(mode=acrl.MODE_ACRL_FALLBACK, X_init=0.01, x_ema=0.3),
                                dict(y_gran=acrl.Y_SEQUENCE, entropy_coeff=0.01, adv_ddof=0)])
def test_one_call_has_the_bits_of_the_three(Q, G, lo, hi, kw):
    pi, mu, mask, so, go, R, H = _tokens(Q, G, lo, hi, seed=Q * 77 + G)
    p = acrl.Params(**kw)
    ent = p.entropy_coeff > 0
    a, b = _three_calls_and_one(p, 3, pi, mu, mask, so, go, R, H if ent else None, ent)
    _assert_same_bytes(a, b)
    a, b = _three_calls_and_one(p, 1, pi, mu, None, so, go, R, H, ent)
    _assert_same_bytes(a, b)


def test_one_call_on_uneven_prompts_and_bad_offsets():
    pi, mu, mask, so, go, R, H = _tokens(6, 2, 1, 300, seed=5)
    p = acrl.Params()
    uneven = torch.tensor([0, 0, 1, 1, 5, 12, 12], dtype=torch.int32, device=DEV)   # empty prompts, one of one
    broken_go = torch.tensor([0, 3, 2, 7, 9, 11, 13], dtype=torch.int32, device=DEV)
    broken_so = so.clone()
    broken_so[4] = so[-1] + 5
    nan = pi.clone()
    nan[3] = float("nan")
    for args in ((pi, so, uneven), (pi, so, broken_go), (pi, broken_so, go), (nan, so, go)):
        a, b = _three_calls_and_one(p, 2, args[0], mu, mask, args[1], args[2], R, H, False)
        _assert_same_bytes(a, b)


def test_fp64_quotients_and_roots_are_rounded_ones():
    """The kernels' own fp64 quotient and square root (Newton-Raphson with a final residual) against IEEE division and
    root: one ulp on D_i = sum_d / n as it comes out as Y of a prompt with one response, for many n and magnitudes; on
    the token means; and on the standard deviation, whose argument is a difference of two of them."""
    S = 1500
    rng = np.random.default_rng(3)
    n = rng.integers(1, 700, size=S)
    so = np.concatenate([[0], np.cumsum(n)])
    T = int(so[-1])
    pi = (-rng.exponential(size=T) * np.repeat(10.0 ** rng.uniform(-6, 1.2, size=S), n)).astype(np.float32)
    mu = np.minimum(pi + (0.3 * rng.normal(size=T)).astype(np.float32), 0.0)
    f = lambda x, dt: torch.tensor(np.asarray(x), dtype=dt, device=DEV)  # noqa: E731
    disc = api.seq_discrepancy(f(pi, torch.float32), f(mu, torch.float32), None, f(so, torch.int64),
                               f(np.arange(S + 1), torch.int32))
    seq, grp, b = disc.seq_host(), disc.grp_host(), disc.batch_host()
    want = seq["sum_d"] / n
    assert np.all(seq["n"] == n) and np.all(np.abs(grp["Y"] - want) <= 2.0 ** -52 * want)
    assert float(seq["sum_d"].max() / seq["sum_d"].min()) > 1e3
    # a mean is sum * (1 / N): two roundings, and the sums' own order
    for got, v in ((b["d_mean"], seq["sum_d"]), (b["lr_mean"], seq["sum_lr"])):
        assert abs(float(got) - float(v.sum()) / T) <= 1e-14 * float(np.abs(v).sum()) / T
    var = float(seq["sum_d2"].sum()) / T - (float(seq["sum_d"].sum()) / T) ** 2
    assert abs(float(b["d_std"]) - np.sqrt(var)) <= 1e-13 * float(seq["sum_d2"].sum()) / T / np.sqrt(var)
