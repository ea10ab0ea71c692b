"""GPU parity of the prefill chunk on the tensor cores (chunkwise closed form of Sec. 3.1
Eq. delta_update, App. A.5 "Prefill path") against the oracle's per-token chunk: GDN and
KDA, d_k = d_v = 128, bf16 q/k/v, chunks of at least 32 tokens (one or more pieces of up
to 64 tokens, ragged rows masked); the UINT8 and UINT4 low tiers.  KDA pieces are cut
short where a channel's decay would leave FP32 on either side of the reference token."""
import pytest
import torch

import paper_2608_27513_gb300 as damp
import workloads as wl
from tests.test_gpu_prefill import _built, _run  # noqa: F401  (module fixture and runner)

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _gdn(name, batch, heads, qk_heads, k_hi, fmt=0, seed=31):
    return wl.Workload(name, "gdn", batch, heads, qk_heads, 128, 128, k_hi, 4, 24, "bf16", seed, fmt)


def test_one_piece_gqa():
    """64 tokens (one full piece), GQA (two value heads per q/k head), K_hi = 8."""
    _run(_gdn("tc_gqa_k8", 2, 4, 2, 8), 64)


def test_two_pieces_two_chunks():
    """128 tokens (two pieces in one launch), two chunks in a row."""
    _run(_gdn("tc_two_pieces", 1, 2, 2, 10, seed=32), 128, chunks=2)


def test_ragged_rows_and_slot_indirection():
    """Rows of 40, 17 and 0 tokens in a 40-token chunk (a partial piece: masked tokens),
    scattered over a larger pool; the zero-length row's slot stays as it was."""
    _run(_gdn("tc_ragged", 3, 2, 2, 6, seed=33), 40, lengths=[40, 17, 0], slot_of={0: 4, 1: 1, 2: 0}, pool=5)


@pytest.mark.parametrize("k_hi,fmt", [(0, 0), (16, 1), (40, 0), (127, 1), (10, 3), (16, 4), (0, 3)])
def test_tiers(k_hi, fmt):
    """No FP16 rows, FP16 rows in one warp or over two, all but one row FP16; the UINT8 and
    UINT4 tiers with and without H_32."""
    _run(_gdn(f"tc_k{k_hi}_f{fmt}", 1, 2, 1, k_hi, fmt, seed=34 + k_hi), 64)


def test_full_piece_and_a_partial_one():
    """97 tokens: a full piece and a partial one of 33."""
    _run(_gdn("tc_97", 1, 2, 2, 12, seed=35), 97)


def _kda(name, batch, heads, qk_heads, k_hi, fmt=0, seed=41):
    return wl.Workload(name, "kda", batch, heads, qk_heads, 128, 128, k_hi, 4, 24, "bf16", seed, fmt)


def test_kda_one_piece_gqa():
    """KDA, 64 tokens (one full piece), GQA, K_hi = 10."""
    _run(_kda("tck_gqa_k10", 2, 4, 2, 10), 64)


def test_kda_two_pieces_two_chunks():
    _run(_kda("tck_two_pieces", 1, 2, 2, 16, seed=42), 128, chunks=2)


def test_kda_ragged_rows_and_slot_indirection():
    _run(_kda("tck_ragged", 3, 2, 2, 6, seed=43), 40, lengths=[40, 17, 0], slot_of={0: 4, 1: 1, 2: 0}, pool=5)


@pytest.mark.parametrize("k_hi,fmt", [(0, 0), (16, 1), (40, 0), (127, 1), (10, 3), (16, 4)])
def test_kda_tiers(k_hi, fmt):
    _run(_kda(f"tck_k{k_hi}_f{fmt}", 1, 2, 1, k_hi, fmt, seed=44 + k_hi), 64)


@pytest.mark.parametrize("g_scale", [8.0, 60.0])
def test_kda_strong_decay_shortens_the_pieces(g_scale):
    """Log-decays 8x and 60x the workload's (down to about -8 and -60 per token and
    channel): the pieces are cut to 32 tokens or fewer, down to single tokens, and the
    chunk still matches the per-token recurrence."""
    _run(_kda(f"tck_decay{int(g_scale)}", 1, 2, 2, 12, seed=45), 64, g_scale=g_scale)


# (Rows are ordered up to 256 of them, and GDN heads go in one, two or four parts as KDA heads do:
# test_gpu_prefill_tc_units.py has the edges of both.)
@pytest.mark.parametrize("kind", ["gdn", "kda"])
@pytest.mark.parametrize("B,T", [(1, 40), (8, 70), (40, 130), (512, 32), (513, 33)])
def test_ragged_batches_equal_their_rows_alone(kind, B, T):
    """The units of a ragged chunk are taken by falling length (up to 512 rows), in rounds from both
    ends of the order, KDA heads in one, two or four value parts by the number of pairs: every row, empty, full and equally long ones among them, gets what a call of
    its own gives it, bit for bit, and rows past a length stay zero."""
    H = 8
    gen = torch.Generator(device=DEV)
    gen.manual_seed(B)
    n = lambda *s: torch.randn(*s, generator=gen, device=DEV)
    unit = lambda x: (x / x.norm(dim=-1, keepdim=True)).bfloat16()
    q, k, v = unit(n(B, T, H, 128)), unit(n(B, T, H, 128)), n(B, T, H, 128).bfloat16()
    g = -torch.nn.functional.softplus(n(B, T, H) if kind == "gdn" else n(B, T, H, 128) - 3.0)
    beta = torch.sigmoid(n(B, T, H))
    lengths = torch.randint(0, T + 1, (B,), generator=gen, device=DEV, dtype=torch.int32)
    lengths[B // 2] = T
    lengths[: B // 4] = T // 2
    L = damp.Layout(H, H, 128, 128, 16, 0)
    perm = torch.stack([torch.randperm(128, generator=gen, device=DEV) for _ in range(H)]).to(torch.uint8)
    pool = damp.new_state(L, B, DEV)
    damp.quantize_state(L, 0.1 * n(B, H, 128, 128), perm, pool)
    alone = pool.clone()
    chunk = damp.kda_prefill_chunk if kind == "kda" else damp.gdn_prefill_chunk
    o = chunk(L, pool, perm, q, k, v, g, beta, lengths=lengths)
    for b in range(B):
        ob = chunk(L, alone[b:b + 1], perm, q[b:b + 1], k[b:b + 1], v[b:b + 1], g[b:b + 1], beta[b:b + 1],
                   lengths=lengths[b:b + 1].clone())
        assert torch.equal(o[b:b + 1], ob)
        assert not o[b, int(lengths[b]):].any()
    assert torch.equal(pool, alone)
    assert damp.device_status() == 0
