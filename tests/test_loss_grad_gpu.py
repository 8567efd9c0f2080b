"""acrl_loss_grad_logits where the CTA that a row gets changes size, with the lse
given and recomputed: rows one column short of, at and past the lines, rows
shorter than a step, with one to seven columns beyond whole vectors and with a
ragged rest beyond what the CTA keeps on chip, against float64."""

import ctypes
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu

import paper_2607_24062_gb300 as acrl  # noqa: E402
import workloads as W  # noqa: E402
from paper_2607_24062_gb300 import _abi, api  # noqa: E402

DEV = "cuda"


@pytest.mark.parametrize("V", [1, 7, 257, 2047, 2048, 2049, 3333, 4095, 4096, 4097, 6145, 8191, 8192, 8193, 12287, 12288, 12289,
                               16383, 16384, 16385, 20011, 65536, 65537, 65543, 65544, 81921, 100003, 151936, 200001])
@pytest.mark.parametrize("bonus", [False, True])
def test_streaming_gradient_by_row_length(V, bonus):
    _check(V, bonus, recompute=False)


@pytest.mark.parametrize("V", [2049, 4095, 4096, 8191])
def test_many_short_rows_agree_with_few(V):
    """The split of a row between threads does not show in its gradient."""
    gen = torch.Generator(device=DEV).manual_seed(V)
    T, few, ld = 12001, 5, (V + 7) // 8 * 8
    x = torch.randn((T, ld), generator=gen, device=DEV).to(torch.bfloat16)
    ids = torch.randint(0, V, (T,), generator=gen, device=DEV, dtype=torch.int32)
    coef = torch.randn(T, generator=gen, device=DEV)
    lse = x[:, :V].float().logsumexp(dim=1)
    a, tl, _ = api.loss_grad_logits(x, ids, None, lse, None, coef, 0.2, V=V)
    b, tl2, _ = api.loss_grad_logits(x[-few:], ids[-few:], None, lse[-few:], None, coef[-few:], 0.2, V=V)
    assert torch.equal(a[-few:, :V].view(torch.int16), b[:, :V].view(torch.int16))
    assert torch.equal(tl[-few:], tl2)


@pytest.mark.parametrize("V", [1, 7, 1025, 4095, 4096, 4097, 7168, 7169, 10240, 10243, 20480, 20487, 20488, 24007, 36864, 40001,
                               40967, 40968, 49155, 61003, 65535, 65536, 70001])
@pytest.mark.parametrize("bonus", [False, True])
def test_recomputed_gradient_by_row_length(V, bonus):
    _check(V, bonus, recompute=True)


def _check(V, bonus, recompute):
    gen = torch.Generator(device=DEV).manual_seed(V)
    T, ld = 37, (V + 7) // 8 * 8
    x = torch.full((T, ld), float("nan"), dtype=torch.bfloat16, device=DEV)   # columns past V are never used
    x[:, :V] = torch.randn((T, V), generator=gen, device=DEV) * 2
    ids = torch.randint(0, V, (T,), generator=gen, device=DEV, dtype=torch.int32)
    mask = (torch.arange(T, device=DEV) % 5 != 1).to(torch.uint8)
    coef = torch.randn(T, generator=gen, device=DEV) * 1e-2
    coef[3] = 0.0
    z = x[:, :V].double()
    lse = z.logsumexp(dim=1)
    lp = z - lse[:, None]
    H = -(lp.exp() * lp).sum(dim=1)
    e = mask * 1e-3 if bonus else None
    flags = api.new_flags()
    grad = torch.full((T, ld), 5.0, dtype=torch.bfloat16, device=DEV)
    g, tl, loss = api.loss_grad_logits(x, ids, mask, None if recompute else lse.float(), None, coef * mask, 0.2, V=V, grad=grad, flags=flags,
                                       entropy=H.float() if bonus else None, ent_coef=e)
    assert api.read_flags(flags) == 0
    c = (coef * mask).double()
    p = lp.exp()
    want = p * c[:, None]
    want.scatter_add_(1, ids.long()[:, None], -c[:, None])
    if bonus:
        want += e.double()[:, None] * p * (lp + H[:, None])
    # bf16 rounding of the result, and the fp32 rounding of lse and of the exponent (2^-24 of some 30) on its terms
    size = p * (c.abs()[:, None] + (e.double()[:, None] * (lp.abs() + H[:, None]) if bonus else 0.0))
    size.scatter_add_(1, ids.long()[:, None], c.abs()[:, None])
    assert bool(((g[:, :V].double() - want).abs() <= 2.0 ** -8 * want.abs() + 2.0 ** -17 * size + 1e-38).all())
    assert bool((g[:, V:] == 5.0).all())
    want_tl = -c - (e.double() * H if bonus else 0.0)
    assert bool(((tl.double() - want_tl).abs() <= 2.0 ** -22 * (c.abs() + (e.double() * H if bonus else 0.0)) + 1e-30).all())
    whole = tl.double().sum()
    assert abs(float(loss) - float(whole)) <= 2.0 ** -21 * float(tl.double().abs().sum()) + 1e-30


@pytest.mark.parametrize("short,long", [(41000, 65000), (20488, 36864), (7200, 20480), (4096, 7168), (70000, 151936)])
def test_threads_with_rows_of_one_class(short, long):
    """Two host threads whose rows take the same kernel with different amounts of shared memory: neither's call fails
    for what the other sets in between."""
    fn = _abi.lib().acrl_loss_grad_logits
    start, bad = threading.Barrier(2), []

    def work(V):
        T, ld = 2, (V + 7) // 8 * 8
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            x = torch.randn((T, ld), device=DEV).to(torch.bfloat16)
            ids = torch.zeros(T, dtype=torch.int32, device=DEV)
            coef, tl, loss, flags = torch.ones(T, device=DEV), torch.empty(T, device=DEV), torch.empty(1, device=DEV), api.new_flags()
            grad = torch.empty_like(x)
        p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
        args = (p(x), T, V, ld, p(ids), None, None, None, p(coef), None, None, 0.2, p(grad), p(tl), p(loss), p(flags),
                ctypes.c_void_p(stream.cuda_stream))
        start.wait()
        for _ in range(4000):
            st = fn(*args)
            if st != 0:
                bad.append((V, st))
        stream.synchronize()
        if api.read_flags(flags) != 0 or not bool(torch.isfinite(grad[:, :V]).all()):
            bad.append((V, "result"))

    threads = [threading.Thread(target=work, args=(V,)) for V in (short, long)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, (len(bad), bad[:4])


# vectors of the output that hold one row's end, several rows, the output's end; rows shorter and longer than the
# 2,048 columns between two vectors of a thread; every shift of a row against its vectors
@pytest.mark.parametrize("T,V,ld", [(1, 1, 8), (1, 3, 8), (9, 1, 8), (300, 7, 8), (5, 9, 16), (131, 15, 24), (40, 2047, 2048),
                                    (17, 2049, 2056), (3, 6143, 6144), (1, 4099, 4104), (131, 20011, 20016), (9, 100003, 100008)])
def test_scaled_gradient_without_gaps(T, V, ld):
    """acrl_scale_grad into rows of V columns against torch's bf16 product, bit for bit, with nothing written beyond."""
    gen = torch.Generator(device=DEV).manual_seed(T + V)
    g = torch.full((T, ld), float("nan"), dtype=torch.bfloat16, device=DEV)   # columns past V are never used
    g[:, :V] = torch.randn((T, V), generator=gen, device=DEV)
    for f in (0.25, -3.7, 0.0):
        s = torch.tensor(f, device=DEV)
        whole = torch.full((T * V + 64,), 5.0, dtype=torch.bfloat16, device=DEV)
        out = whole[: T * V].view(T, V)
        assert api.scale_grad(g, s, V=V, out=out) is out
        assert torch.equal(out.view(torch.int16), (g[:, :V] * s.to(torch.bfloat16)).view(torch.int16))
        assert bool((whole[T * V:] == 5.0).all())
    before = out.clone()
    api.scale_grad(g, torch.ones((), device=DEV), V=V, out=out)
    assert torch.equal(out.view(torch.int16), before.view(torch.int16))
    with pytest.raises(acrl.AcrlError):   # neither V nor a multiple of eight
        api.scale_grad(g, s, V=V, out=torch.empty((T, (V + 7) // 8 * 8 + 1), dtype=torch.bfloat16, device=DEV))


@pytest.mark.parametrize("V", [1000, 1003])
def test_gradient_of_a_scaled_loss_is_contiguous(V):
    """As the product of the gradient with the scale is: a hook may flatten it."""
    b = W.generate(W.small_variant(W.GRPO, name="contiguous", n_prompts=2, group_size=4, len_lo=5, len_hi=20, V=V), seed=6,
                   device=DEV)
    step = acrl.AcrlStep.for_batch(b, acrl.Params())
    x = b.logits[:, :V].detach().requires_grad_(True)
    seen = []
    x.register_hook(lambda g: seen.append(g.view(-1)))
    loss = acrl.acrl_loss(step, x, b.ids, b.mask, b.logp_mu, b.rewards, b.seq_offsets, b.group_offsets)
    (loss * 0.25).backward()
    assert torch.equal(seen[0].view(x.shape).view(torch.int16), (step.grad[:, :V] * 0.25).view(torch.int16))


@pytest.mark.parametrize("V,rms", [(4096, 3.70e-7), (6144, 3.78e-7), (24583, 4.20e-7)])
def test_recomputed_log_prob_is_as_close_as_with_fewer_warps(V, rms):
    """Rms error of the recomputed log-prob against float64, read from the token loss (coefficient -1 and a ratio
    within the clip: the loss is the ratio), over normal logits (sd 2): no larger than with a warp a row (3.68e-7 and
    3.77e-7 at V = 4,096 and 6,144) and four warps a row (4.19e-7 at V = 24,583)."""
    sq, rows, ld = 0.0, 0, (V + 7) // 8 * 8
    for seed in range(8):
        gen = torch.Generator(device=DEV).manual_seed(7919 * seed + V)
        T = min(4096, 40_000_000 // V)
        x = (torch.randn((T, ld), generator=gen, device=DEV) * 2).to(torch.bfloat16)
        ids = torch.randint(0, V, (T,), generator=gen, device=DEV, dtype=torch.int32)
        z = x[:, :V].double()
        lp = z.gather(1, ids.long()[:, None])[:, 0] - z.logsumexp(dim=1)
        old = (lp - 0.001).float()
        _, tl, _ = api.loss_grad_logits(x, ids, None, None, old, -torch.ones(T, device=DEV), 0.2, V=V)
        sq += float((tl.double().log() + old.double() - lp).square().sum())
        rows += T
    assert (sq / rows) ** 0.5 <= rms, (sq / rows) ** 0.5


@pytest.mark.parametrize("V", [7, 1001, 4097, 5003, 6143, 6145, 7168, 7170, 20011, 22001, 24583, 36870, 40967, 49155, 61003, 70001,
                               151937])
@pytest.mark.parametrize("mask_value", [float("-inf"), -3.3895313892515355e38])
def test_recomputed_gradient_of_masked_columns(V, mask_value):
    """Columns at -infinity or at bf16's lowest number have probability 0 wherever in the row they are: the ragged last
    column, the last vectors, the first half, all but a few; the lse of the others is finite, and so is the gradient."""
    gen = torch.Generator(device=DEV).manual_seed(V)
    ld = (V + 7) // 8 * 8
    few = torch.randperm(V, generator=gen, device=DEV)[:5]
    off = torch.zeros((5, V), dtype=torch.bool, device=DEV)
    off[0, V - 1:] = True
    off[1, max(1, V - 27):] = True
    off[2, : V // 2] = True
    off[3, :] = True
    off[3, few] = False
    x = torch.full((5, ld), float("nan"), dtype=torch.bfloat16, device=DEV)
    x[:, :V] = (torch.randn((5, V), generator=gen, device=DEV) * 2).masked_fill(off, mask_value)
    ids = (~off).to(torch.uint8).argmax(dim=1).to(torch.int32)
    coef = torch.tensor([0.5, -0.25, 1.0, -1.0, 0.125], device=DEV)
    z = x[:, :V].double()
    lp = z - z.logsumexp(dim=1)[:, None]
    old = lp.gather(1, ids.long()[:, None])[:, 0].float()
    flags = api.new_flags()
    g, tl, _ = api.loss_grad_logits(x, ids, None, None, old, coef, 0.2, V=V, flags=flags)
    assert api.read_flags(flags) == 0
    c, p = coef.double(), lp.exp()
    want = p * c[:, None]
    want.scatter_add_(1, ids.long()[:, None], -c[:, None])
    # as in _check, the ratio's rounding of 2^-22 besides
    size = (p * c.abs()[:, None]).scatter_add_(1, ids.long()[:, None], c.abs()[:, None])
    assert bool(((g[:, :V].double() - want).abs() <= 2.0 ** -8 * want.abs() + 2.0 ** -16 * size + 1e-38).all())
    assert bool((g[:, :V][off] == 0).all())
    assert bool(((tl.double() + c).abs() <= 2.0 ** -18 * c.abs()).all())
