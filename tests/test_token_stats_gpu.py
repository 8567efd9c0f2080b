"""acrl_token_stats where its load path or its row team changes: a call of few
rows (ring of loads in shared memory) and a call of many rows that takes the
register path (from 4,609 columns; shorter rows have the ring alone) give the
same rows the same bits, at row lengths around a whole step of the team's
loads, around whole rings and around whole vectors; and both agree with a
float64 log-softmax."""

import pytest
import torch

pytestmark = pytest.mark.gpu

from paper_2607_24062_gb300 import api  # noqa: E402

DEV = "cuda"

# team of 8: steps of 256 columns; 16: 512; 32: 1,024; 64: 2,048; 128: 4,096
_WIDTHS = [1, 8, 63, 64, 255, 256, 257, 767, 768, 769, 1024, 4095, 4096, 4097, 5119, 5120, 5121, 3584, 3585, 4608, 4609, 7168, 16383, 16384, 16385,
           18431, 18432, 18441, 20011, 32000, 40960, 40961, 65535, 65536, 65537, 65544, 69632, 69640, 100003, 151936]


def _many(V):
    """Rows that put the call on the register path (between 5.2 and 10.4 teams of 128 threads per SM); up to 4,608
    columns, where eight or sixteen lanes a row have the ring alone, more rows than are resident at once."""
    team = 8 if V <= 4608 else 32 if V <= 16384 else 64 if V <= 40960 else 128
    return 6 * 128 * 152 // team if team > 8 else 4096


@pytest.mark.parametrize("V", _WIDTHS)
def test_few_and_many_rows_agree(V):
    gen = torch.Generator(device=DEV).manual_seed(V)
    R, ld = 5, (V + 7) // 8 * 8
    base = torch.full((R, ld), float("nan"), dtype=torch.bfloat16, device=DEV)   # columns past V are never read
    base[:, :V] = torch.randn((R, V), generator=gen, device=DEV) * 3
    base[1, V // 2] = 40.0
    base[2, :V] = -3.0
    ids = torch.randint(0, V, (R,), generator=gen, device=DEV, dtype=torch.int32)
    mask = torch.tensor([1, 1, 1, 0, 1], dtype=torch.uint8, device=DEV)
    flags = api.new_flags()
    few = api.token_stats(base, ids, mask, V=V, flags=flags)
    T = _many(V)
    pick = torch.arange(T, device=DEV) % R
    many = api.token_stats(base[pick], ids[pick], mask[pick], V=V, flags=flags)
    assert api.read_flags(flags) == 0
    for a, b in zip(few, many):
        assert torch.equal(a[pick].view(torch.int32), b.view(torch.int32))
    z = base[:, :V].double()
    lse = z.logsumexp(dim=1)
    lp = z - lse[:, None]
    want = (lse, lp.gather(1, ids.long()[:, None])[:, 0], -(lp.exp() * lp).sum(dim=1))
    live = mask.bool()
    for got, ref in zip(few, want):
        assert float((got.double() - ref)[live].abs().max()) <= 2e-5 * max(1.0, float(ref[live].abs().max()))
        assert float(got[3]) == 0.0


@pytest.mark.parametrize("V", [256, 5000, 20011, 100003])
def test_undefined_rows_and_bad_ids(V):
    """NaN and infinities anywhere in the row, ids outside the vocabulary, on the ring path."""
    ld = (V + 7) // 8 * 8
    spots = [0, V // 3, V - 1]
    rows = torch.zeros((3 * len(spots) + 2, ld), dtype=torch.bfloat16, device=DEV)
    for k, bad in enumerate((float("nan"), float("inf"), float("-inf"))):
        for j, c in enumerate(spots):
            rows[k * len(spots) + j, c] = bad
    T = rows.shape[0]
    ids = torch.zeros(T, dtype=torch.int32, device=DEV)
    ids[-2], ids[-1] = V, -1
    flags = api.new_flags()
    lse, logp, ent = api.token_stats(rows, ids, None, V=V, flags=flags)
    assert api.read_flags(flags) == 0x3       # BAD_ID and NONFINITE
    for x in (lse, logp, ent):
        assert bool(x[:-2].isnan().all()) and not bool(x[-2:].isnan().any())
    assert float(logp[-2]) == 0.0 and float(logp[-1]) == 0.0


@pytest.mark.parametrize("V,ld,T", [(40968, 40968, 2553), (40968, 40968, 2600), (40968, 40968, 3040), (40968, 40968, 3041),
                                    (40968, 40968, 21300), (40968, 41024, 21300), (65537, 65544, 2700), (262144, 262144, 2600)])
def test_many_rows_of_four_warps_agree_with_few(V, ld, T):
    """On both sides of the lines between ring and registers for rows of four warps, by rows and by row stride."""
    gen = torch.Generator(device=DEV).manual_seed(V)
    R = 7
    base = torch.full((R, ld), float("nan"), dtype=torch.bfloat16, device=DEV)
    base[:, :V] = torch.randn((R, V), generator=gen, device=DEV) * 3
    ids = torch.randint(0, V, (R,), generator=gen, device=DEV, dtype=torch.int32)
    flags = api.new_flags()
    few = api.token_stats(base, ids, None, V=V, flags=flags)
    pick = torch.arange(T, device=DEV) % R
    many = api.token_stats(base[pick], ids[pick], None, V=V, flags=flags)
    assert api.read_flags(flags) == 0
    for a, b in zip(few, many):
        assert torch.equal(a[pick].view(torch.int32), b.view(torch.int32))


@pytest.mark.parametrize("V,rows,lse_rms,ent_rms", [(3592, 65536, 3.14e-7, 3.71e-7), (4096, 65536, 3.155e-7, 3.755e-7),
                                                    (40968, 12288, 3.45e-7, 5.10e-7), (57344, 12288, 3.53e-7, 5.13e-7)])
def test_larger_teams_are_as_close_as_smaller_ones(V, rows, lse_rms, ent_rms):
    """Rms errors against float64 over normal logits (sd 2), no larger than those of the teams with a level of merges
    less: eight lanes a row (3.13e-7 and 3.69e-7 at V = 3,592, 3.15e-7 and 3.74e-7 at V = 4,096), two warps a row
    (3.43e-7 and 5.08e-7 at V = 40,968, 3.51e-7 and 5.10e-7 at V = 57,344)."""
    sq, T = torch.zeros(2, dtype=torch.float64, device=DEV), 4096 if V < 10000 else 1024
    for seed in range(rows // T):
        gen = torch.Generator(device=DEV).manual_seed(7919 * seed + V)
        x = (torch.randn((T, V), generator=gen, device=DEV) * 2).to(torch.bfloat16)
        lse, _, ent = api.token_stats(x, torch.zeros(T, dtype=torch.int32, device=DEV))
        z = x.double()
        want = z.logsumexp(dim=1)
        lp = z - want[:, None]
        sq += torch.stack([(lse.double() - want).square().sum(), (ent.double() + (lp.exp() * lp).sum(dim=1)).square().sum()])
    got = (sq / rows).sqrt()
    assert float(got[0]) <= lse_rms and float(got[1]) <= ent_rms, got
