"""The FP32-state step over its shapes: calls large enough that a CTA or warp takes several units
one after the other, on both kernels (the pipelined one and one warp per tile), and no shape far
behind the others at the same bytes."""
import numpy as np
import pytest
import torch

import paper_2608_27513_gb300 as damp
import workloads as wl
from oracle import core, runs
from tests import parity as P
from tests.timing import assert_at_most

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2608_27513_gb300 import build
    build.build()
    torch.cuda.init()
    yield
    assert damp.device_status() == 0


def _workload(kind, dk, dv, batch, dtype="bf16", heads=32, qk_heads=16):
    return wl.Workload(f"fp32_{kind}_{dk}x{dv}", kind, batch, heads, qk_heads, dk, dv, 0, 1, 1, dtype, 51)


# 1280 units and more: above four per resident CTA of the pipelined kernel, several tiles per warp
@pytest.mark.parametrize("kind,dk,dv,dtype,batch", [
    ("gdn", 128, 128, "bf16", 40), ("kda", 128, 128, "fp32", 40), ("gdn", 128, 96, "bf16", 40),
    ("kda", 128, 256, "bf16", 40), ("kda", 64, 128, "bf16", 130), ("gdn", 64, 96, "fp32", 170),
    ("gdn", 128, 160, "bf16", 40), ("kda", 128, 64, "bf16", 40), ("gdn", 64, 64, "bf16", 40),
    ("kda", 32, 32, "fp32", 80), ("gdn", 32, 288, "bf16", 40),
    # a part-full wave of the pipelined kernel's CTAs: a warp per tile, rows alone pipelined
    ("gdn", 128, 128, "bf16", 14), ("kda", 128, 256, "bf16", 8), ("gdn", 128, 384, "fp32", 7)])
def test_rows_of_a_large_step_equal_their_own_call(kind, dk, dv, dtype, batch):
    """Every row of a large step over scattered slots gets what a call of its own gives it, bit for
    bit, and three rows what the oracle gives them; rows whose slot is outside the pool are left
    out (flagged, outputs untouched) and no other slot changes."""
    w = _workload(kind, dk, dv, batch, dtype)
    H = w.heads
    L = damp.Layout(H, w.qk_heads, dk, dv, 0, 0)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(52)
    slots = batch + 3
    S = 0.3 * torch.randn(slots, H, dk, dv, generator=gen, device=DEV)
    alone, before = S.clone(), S.clone()
    idx = torch.randperm(slots, generator=gen, device=DEV)[:batch].to(torch.int32)
    bad = [batch // 2, batch // 2 + 1, batch - 1]
    idx[bad[0]], idx[bad[1]], idx[bad[2]] = slots, -1, slots + 7
    rows = [0, batch // 2 - 1, batch - 2]
    inp = wl.step_inputs(w, 0, rows=list(range(batch)))
    d = P.inputs_to_dev(w, inp, DEV)
    step = damp.fp32_kda_decode_step if kind == "kda" else damp.fp32_gdn_decode_step
    o = torch.full((batch, H, dv), 7.0, device=DEV)
    step(L, S, d["q"], d["k"], d["v"], d["g"], d["beta"], o=o, slot_idx=idx)
    assert damp.device_status() == damp.DEV_BAD_SLOT
    for b in range(batch):
        if b in bad:
            assert bool((o[b] == 7.0).all())
            continue
        ob = step(L, alone, *(d[n][b:b + 1] for n in ("q", "k", "v", "g", "beta")), slot_idx=idx[b:b + 1].clone())
        assert torch.equal(o[b:b + 1], ob), b
    assert torch.equal(S, alone)
    used = [int(idx[b]) for b in range(batch) if b not in bad]
    for s in set(range(slots)) - set(used):
        assert torch.equal(S[s], before[s])
    u = runs.unit_operands(w, {n: v[rows] for n, v in inp.items()})
    at = idx[rows].long()
    Sr = before[at].cpu().numpy().reshape(-1, dk, dv).copy()
    o_ref = core.delta_step_heads(Sr, u["q"], u["k"], u["v"], u["g"], u["beta"], kind)
    P.compare_o(o[rows].cpu().numpy().reshape(-1, dv), o_ref, "large FP32 step")
    got = S[at].cpu().numpy().reshape(Sr.shape)
    assert np.all(np.abs(got - Sr) <= P.ATOL + P.RTOL * np.abs(Sr))


@pytest.mark.parametrize("dk,dv,batch,square_batch", [(32, 32, 256, 16), (64, 32, 256, 32), (64, 160, 64, 40)])
def test_narrow_states_keep_pace_with_square_ones(dk, dv, batch, square_batch):
    """A step on narrow states takes at most twice as long as one on 128 x 128 states of the same
    total size (1.2 to 1.4 times with a warp per tile; 3 to 4 times where CTAs of one or two warps
    are held to two per SM)."""
    def call(k, v, b):
        w = _workload("gdn", k, v, b, heads=32, qk_heads=32)
        L = damp.Layout(32, 32, k, v, 0, 0)
        d = wl.torch_step_inputs(w, 1, DEV)[0]
        S = torch.zeros(b, 32, k, v, device=DEV)
        o = torch.empty(b, 32, v, device=DEV)
        return lambda: damp.fp32_gdn_decode_step(L, S, d["q"], d["k"], d["v"], d["g"], d["beta"], o=o)
    assert batch * dk * dv == square_batch * 128 * 128
    assert_at_most(call(dk, dv, batch), call(128, 128, square_batch), 2.0, f"{dk} x {dv}")


@pytest.mark.parametrize("kind", ["gdn", "kda"])
def test_a_part_full_wave_costs_little(kind):
    """320 units of 128 x 256 states (two CTAs per SM and a few units more) take at most 2.05 times
    as long as 128 x 128 states of the same bytes: 1.85 with a warp per tile, 2.2 where the last few
    units cost the pipelined kernel as much as a whole wave."""
    def call(v, b):
        w = _workload(kind, 128, v, b, heads=16, qk_heads=16)
        L = damp.Layout(16, 16, 128, v, 0, 0)
        d = wl.torch_step_inputs(w, 1, DEV)[0]
        S = torch.zeros(b, 16, 128, v, device=DEV)
        o = torch.empty(b, 16, v, device=DEV)
        step = damp.fp32_kda_decode_step if kind == "kda" else damp.fp32_gdn_decode_step
        return lambda: step(L, S, d["q"], d["k"], d["v"], d["g"], d["beta"], o=o)
    assert_at_most(call(256, 10), call(128, 20), 2.05, kind)


@pytest.mark.parametrize("kind,dk,dv,T,every", [("kda", 128, 128, 21, 8), ("gdn", 128, 160, 17, 8), ("gdn", 64, 96, 7, 2),
                                                ("kda", 64, 256, 9, 4), ("gdn", 32, 64, 11, 5), ("kda", 32, 32, 5, 1)])
def test_documents_of_a_calibration_run_equal_their_own_run(kind, dk, dv, T, every):
    """A run over 12 documents (384 units and more: several per CTA, each over all tokens between two
    samples, and single steps where a run is short) leaves every document the states that a run of
    its own gives it, bit for bit."""
    docs = 12
    w = _workload(kind, dk, dv, docs)
    L = damp.Layout(w.heads, w.qk_heads, dk, dv, 0, 0)
    inputs = wl.torch_step_inputs(w, T, DEV)
    st = {n: torch.stack([d[n] for d in inputs]) for n in ("q", "k", "v", "g", "beta")}
    gen = torch.Generator(device=DEV)
    gen.manual_seed(53)
    S = 0.3 * torch.randn(docs, w.heads, dk, dv, generator=gen, device=DEV)
    alone = S.clone()

    def run(s, sl):
        E, G = (torch.zeros((w.heads, dk), device=DEV) for _ in range(2))
        damp.calib_accumulate(L, kind, s, *(st[n][:, sl].contiguous() for n in ("q", "k", "v", "g", "beta")), E, G, every)
    run(S, slice(0, docs))
    for b in range(docs):
        run(alone[b:b + 1], slice(b, b + 1))
    assert torch.equal(S, alone)


@pytest.mark.parametrize("dk,dv", [(32, 32), (64, 64)])
def test_a_sample_every_token_costs_no_more_than_single_steps(dk, dv):
    """calib_accumulate with every = 1 takes at most 1.2 times its steps and error passes called one
    by one (which write outputs as well); 1.3 to 1.6 times where one token starts a whole run."""
    docs, T = 32, 12
    w = _workload("gdn", dk, dv, docs, qk_heads=32)
    L = damp.Layout(w.heads, w.qk_heads, dk, dv, 0, 0)
    inputs = wl.torch_step_inputs(w, T, DEV)
    st = {n: torch.stack([d[n] for d in inputs]) for n in ("q", "k", "v", "g", "beta")}
    S = damp.new_fp32_state(L, docs, DEV)
    o = torch.empty(docs, w.heads, dv, device=DEV)
    E, G = (torch.zeros((w.heads, dk), device=DEV) for _ in range(2))

    def single():
        for d in inputs:
            damp.fp32_gdn_decode_step(L, S, d["q"], d["k"], d["v"], d["g"], d["beta"], o=o)
            damp.calib_error_energy(L, S, E)
        damp.calib_log_decay(L, st["g"].flatten(0, 1), G)

    def one_call():
        damp.calib_accumulate(L, "gdn", S, st["q"], st["k"], st["v"], st["g"], st["beta"], E, G, 1)
    assert_at_most(one_call, single, 1.2, f"{dk} x {dv}")
