"""The tensor-core prefill's units: value blocks per unit, the order of a ragged chunk's rows and what it costs."""
import pytest
import torch

import paper_2608_27513_gb300 as damp
from tests.test_gpu_prefill import _built  # noqa: F401  (module fixture)
from tests.timing import assert_at_most

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _operands(kind, B, T, H, seed, fmt=0, k_hi=16, g_shift=-3.0):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    n = lambda *s: torch.randn(*s, generator=gen, device=DEV)
    unit = lambda x: (x / x.norm(dim=-1, keepdim=True)).bfloat16()
    ops = dict(q=unit(n(B, T, H, 128)), k=unit(n(B, T, H, 128)), v=n(B, T, H, 128).bfloat16(),
               g=-torch.nn.functional.softplus(n(B, T, H) if kind == "gdn" else n(B, T, H, 128) + g_shift),
               beta=torch.sigmoid(n(B, T, H)))
    L = damp.Layout(H, H, 128, 128, k_hi, fmt)
    perm = torch.stack([torch.randperm(128, generator=gen, device=DEV) for _ in range(H)]).to(torch.uint8)
    pool = damp.new_state(L, B, DEV)
    damp.quantize_state(L, 0.1 * n(B, H, 128, 128), perm, pool)
    return L, perm, pool, ops, gen


def _chunk(kind):
    return damp.kda_prefill_chunk if kind == "kda" else damp.gdn_prefill_chunk


@pytest.mark.parametrize("kind", ["gdn", "kda"])
@pytest.mark.parametrize("B", [3, 129, 255, 256, 257])
def test_any_lengths_name_every_row_once(kind, B):
    """Lengths below zero, above T, equal and distinct ones, up to and past the rows that are ordered:
    every row runs its clamped length, as in calls of its own."""
    H, T = 2, 33
    L, perm, pool, ops, gen = _operands(kind, B, T, H, 60 + B)
    lengths = torch.randint(-5, T + 6, (B,), generator=gen, device=DEV, dtype=torch.int32)
    lengths[0], lengths[B // 2], lengths[B - 1] = -2 ** 31, 2 ** 31 - 1, T
    alone = pool.clone()
    o = _chunk(kind)(L, pool, perm, lengths=lengths, **ops)
    for b in range(B):
        ob = _chunk(kind)(L, alone[b:b + 1], perm, lengths=lengths[b:b + 1].clone(),
                          **{n: t[b:b + 1] for n, t in ops.items()})
        assert torch.equal(o[b:b + 1], ob), b
    assert torch.equal(pool, alone)


@pytest.mark.parametrize("B", [256, 512])
def test_lengths_cost_little_where_all_rows_are_whole(B):
    """A chunk with every length given as T against the same chunk without lengths, two heads: at most
    5 % longer (12 % where every CTA compares 512 lengths from global memory)."""
    H, T = 2, 64
    L, perm, pool, ops, _ = _operands("gdn", B, T, H, 7)
    o = torch.empty(B, T, H, 128, device=DEV)
    lengths = torch.full((B,), T, dtype=torch.int32, device=DEV)
    call = lambda n: (lambda: damp.gdn_prefill_chunk(L, pool, perm, o=o, lengths=n, **ops))
    assert_at_most(call(lengths), call(None), 1.05, f"{B} rows")


@pytest.mark.parametrize("kind", ["gdn", "kda"])
def test_one_longer_row_shares_no_cta_of_the_last_round(kind):
    """Ten rows of 32 heads are two units for every CTA and a third for a few.  One row with a token in a
    second piece costs at most 12 % (20 % and more where the CTAs with its units get the third ones)."""
    B, H, T = 10, 32, 65
    L, perm, pool, ops, _ = _operands(kind, B, T, H, 9)
    o = torch.empty(B, T, H, 128, device=DEV)
    even = torch.full((B,), 60, dtype=torch.int32, device=DEV)
    one = even.clone()
    one[5] = T
    call = lambda n: (lambda: _chunk(kind)(L, pool, perm, o=o, lengths=n, **ops))
    assert_at_most(call(one), call(even), 1.12, kind)


@pytest.mark.parametrize("kind,what", [("gdn", "plain"), ("gdn", "head map"), ("kda", "plain"), ("kda", "head map"),
                                       ("kda", "strong decay")])
@pytest.mark.parametrize("fmt,k_hi", [(0, 40), (1, 16), (3, 10), (4, 0)])
@pytest.mark.parametrize("B", [8, 40])
def test_heads_in_two_and_in_four_blocks_equal_heads_in_one(kind, fmt, k_hi, B, what):
    """A head's value blocks go one, two or four to a unit by the number of (row, head) pairs: 8 pairs
    (a row of its own: one block, the case that the oracle tests pin), 64 and 320.  Rows of a batch get
    what they get alone, bit for bit, in every format; for held heads that are a subset of the layer's in
    another order, and for KDA decays that cut the pieces short."""
    H, T = 8, 70
    L, perm, pool, ops, gen = _operands(kind, B, T, H, 80 + B + fmt, fmt, k_hi)
    if what == "strong decay":
        ops["g"] *= torch.where(torch.rand(B, 1, H, 1, generator=gen, device=DEV) < 0.5, 60.0, 8.0)
    rest = slice(0, 0)
    if what == "head map":
        Hm = 12
        L, _, _, ops, _ = _operands(kind, B, T, Hm, 81 + B, fmt, k_hi)
        held = torch.randperm(Hm, generator=gen, device=DEV)[:H].to(torch.int32)
        rest = [m for m in range(Hm) if m not in held.tolist()]
        L = damp.Layout(H, Hm, 128, 128, k_hi, fmt, model_heads=Hm, head_map=held)
    lengths = torch.randint(1, T + 1, (B,), generator=gen, device=DEV, dtype=torch.int32)
    lengths[B // 2] = T
    idx = torch.randperm(B, generator=gen, device=DEV).to(torch.int32)
    alone = pool.clone()
    o = _chunk(kind)(L, pool, perm, lengths=lengths, slot_idx=idx, **ops)
    assert bool(torch.isfinite(o).all())
    for b in range(B):
        ob = _chunk(kind)(L, alone, perm, lengths=lengths[b:b + 1].clone(), slot_idx=idx[b:b + 1].clone(),
                          **{n: t[b:b + 1] for n, t in ops.items()})
        assert torch.equal(o[b:b + 1], ob), b
    assert not o[:, :, rest].any()
    assert torch.equal(pool, alone)
