"""The binding's quick checks (_fits_*) stand alone before a call: where they accept, the per-tensor
checks are not run.  These tests reach them on the host, with CPU tensors of a class that says it is
on a GPU and a library stand-in that records the compute calls."""
import pytest
import torch

import paper_2608_27513_gb300 as damp
from paper_2608_27513_gb300 import _lib, build
from tests.test_binding_shapes import B, DK, DV, H, HQK, K, T, _layout, _NoCompute, _ops, _perm, _pool


class _OnGpu(torch.Tensor):
    is_cuda = property(lambda self: True)


def _dev(x):
    if isinstance(x, torch.Tensor):
        return x.as_subclass(_OnGpu)
    if isinstance(x, dict):
        return {k: _dev(v) for k, v in x.items()}
    return x


class _Stream:
    cuda_stream = 0


class _Recorder(_NoCompute):
    def __getattr__(self, name):
        if name in self.SIZE_CALLS:
            return getattr(self.real, name)

        def call(*a):
            self.calls.append(name)
            return 0
        return call


@pytest.fixture()
def calls(monkeypatch):
    build.build()
    f = _Recorder(_lib.lib())
    monkeypatch.setattr(damp, "lib", lambda: f)
    return f.calls


def test_sizes_that_are_no_integers_stay_refused(calls):
    """A layout's struct is kept by its values: 4.0 equals 4 as a key, but is no size."""
    good = _layout()
    args = dict(_dev(_ops("kda")), stream=_Stream())
    damp.kda_decode_step(good, _dev(_pool(good)), _dev(_perm()), **args)
    S = _dev(torch.zeros((B, H, DK, DV)))
    damp.fp32_kda_decode_step(good, S, **args)
    assert len(calls) == 2
    for bad in (damp.Layout(float(H), HQK, DK, DV, K), damp.Layout(H, HQK, DK, DV, float(K))):
        with pytest.raises(TypeError):
            damp.kda_decode_step(bad, _dev(_pool(good)), _dev(_perm()), **args)
        with pytest.raises(TypeError):
            damp.fp32_kda_decode_step(bad, S, **args)
    assert len(calls) == 2


def test_a_size_tensor_is_read_at_each_call(calls):
    """An integer tensor is a size by its value at the call, not by its identity."""
    k_hi = torch.tensor(K)
    L = damp.Layout(H, HQK, DK, DV, k_hi)
    assert damp._cptr(L).contents.k_hi == K
    k_hi += 2
    assert damp._cptr(L).contents.k_hi == K + 2


def test_a_layout_looks_up_its_sizes_at_its_first_call(calls):
    """Making a layout does no more than store its fields; equal layouts stay equal afterwards."""
    L = _layout()
    assert "_sizes" not in vars(L)
    damp.kda_decode_step(L, _dev(_pool(L)), _dev(_perm()), **dict(_dev(_ops("kda")), stream=_Stream()))
    assert "_sizes" in vars(L)
    assert L == _layout() and hash(L) == hash(_layout())


def test_outputs_are_plain_tensors_whatever_class_v_has(calls):
    L = _layout()
    args = dict(stream=_Stream())
    step, chunk = _dev(_ops("gdn")), _dev(_ops("gdn", (B, T)))
    heads = _dev(torch.arange(H, dtype=torch.int32))
    M = damp.Layout(H, HQK, DK, DV, K, model_heads=H, head_map=heads)
    state, perm = _dev(_pool(L)), _dev(_perm())
    outs = [damp.gdn_decode_step(L, state, perm, **step, **args), damp.gdn_decode_step(M, state, perm, **step, **args),
            damp.gdn_decode_step_groups([(M, state, perm)], **step, **args),
            damp.gdn_prefill_chunk(L, state, perm, **chunk, **args),
            damp.gdn_prefill_chunk(L, state, perm, lengths=_dev(torch.zeros(B, dtype=torch.int32)), **chunk, **args)]
    assert len(calls) == len(outs)
    for o in outs:
        assert type(o) is torch.Tensor and o.dtype is torch.float32


def _fp32_state():
    return torch.zeros((B, H, DK, DV))


def _entries():
    """(name, call of the keyword arguments, good arguments) of every entry point with quick checks."""
    L = _layout()
    heads = _dev(torch.arange(H, dtype=torch.int32))
    M = damp.Layout(H, HQK, DK, DV, K, model_heads=H, head_map=heads)
    idx = torch.arange(B, dtype=torch.int32)
    out = []
    for kind in ("gdn", "kda"):
        step, chunk = _ops(kind), _ops(kind, (B, T))
        fn = lambda name: getattr(damp, name.format(kind))
        packed = dict(state=_pool(L), perm=_perm(), slot_idx=idx, num_slots=8)
        out += [
            (f"{kind} step", lambda state, perm, f=fn("{}_decode_step"), **a: f(L, state, perm, **a),
             dict(step, o=torch.zeros((B, H, DV)), **packed)),
            (f"{kind} fp32 step", lambda state, f=fn("fp32_{}_decode_step"), **a: f(L, state, **a),
             dict(step, state=_fp32_state(), o=torch.zeros((B, H, DV)), slot_idx=idx, num_slots=B)),
            (f"{kind} chunk", lambda state, perm, f=fn("{}_prefill_chunk"), **a: f(L, state, perm, **a),
             dict(chunk, o=torch.zeros((B, T, H, DV)), lengths=torch.zeros(B, dtype=torch.int32), **packed)),
            (f"{kind} group step", lambda state, perm, f=fn("{}_decode_step_groups"), **a: f([(M, state, perm)], **a),
             dict(step, o=torch.zeros((B, H, DV)), state=_pool(L), perm=_perm(), slot_idx=idx))]
    out.append(("quantize", lambda S, state, perm, **a: damp.quantize_state(L, S, perm, state, **a),
                dict(S=_fp32_state(), state=_pool(L), perm=_perm(), slot_idx=idx, num_slots=8)))
    return out


def _wrong(name, t):
    """The argument with one thing wrong: each dimension one longer and one shorter, a dimension more and
    one less, another type, not contiguous, not on the GPU."""
    for d in range(t.dim()):
        if name == "state" and d == 0:
            continue  # any number of slots
        for step in (1, -1):
            shape = list(t.shape)
            shape[d] += step
            yield f"dim {d} {step:+d}", _dev(torch.zeros(shape, dtype=t.dtype))
    yield "a dimension more", _dev(t[None])
    yield "a dimension less", _dev(t[0].contiguous())
    other = {torch.uint8: torch.int8, torch.int32: torch.int64, torch.float32: torch.float64, torch.bfloat16: torch.float16}
    yield "type", _dev(t.to(other[t.dtype]))
    if t.dim() > 1:
        yield "not contiguous", _dev(t.transpose(0, 1).contiguous().transpose(0, 1))
    yield "on the host", t


@pytest.mark.parametrize("i", range(9))
def test_quick_checks_refuse_one_wrong_argument_at_a_time(calls, monkeypatch, i):
    """Well-formed arguments pass the quick checks alone (the per-tensor checks are taken out for that
    call); with any single one wrong the call raises and nothing is launched."""
    name, call, good = _entries()[i]
    good = dict(_dev(good), stream=_Stream())
    with monkeypatch.context() as m:
        for check in ("_want", "_want_pool", "_want_batch", "_want_operands", "_cuda_contig"):
            m.setattr(damp, check, lambda *a, **k: pytest.fail(f"{name}: good arguments reached the per-tensor checks"))
        call(**good)
        call(**{k: None if k in ("slot_idx", "num_slots", "o", "lengths") else v for k, v in good.items()})
    assert len(calls) == 2
    for arg, t in good.items():
        if not isinstance(t, torch.Tensor):
            continue
        for what, bad in _wrong(arg, t.as_subclass(torch.Tensor)):
            with pytest.raises((ValueError, TypeError)):
                call(**dict(good, **{arg: bad}))
            assert len(calls) == 2, (name, arg, what)
        if arg not in ("slot_idx", "o", "lengths", "perm"):
            with pytest.raises((ValueError, TypeError, AttributeError)):
                call(**dict(good, **{arg: None}))
            assert len(calls) == 2, (name, arg, "missing")
    slots = good["state"].shape[0]
    few = dict(good, slot_idx=None, state=_dev(good["state"].as_subclass(torch.Tensor)[:B - 1].clone()))
    pools = [few] if "num_slots" not in good else [
        dict(good, num_slots=slots + 1), dict(good, num_slots=-1), dict(good, slot_idx=None, num_slots=B - 1), dict(few, num_slots=None)]
    for args in pools:
        with pytest.raises(ValueError):
            call(**args)
        assert len(calls) == 2, name


def test_operands_of_one_wrong_type_and_groups_without_a_map_are_refused(calls):
    L = _layout()
    state, perm, args = _dev(_pool(L)), _dev(_perm()), dict(stream=_Stream())
    with pytest.raises(TypeError):
        damp.kda_decode_step(L, state, perm, **_dev(_ops("kda", dt=torch.float16)), **args)
    with pytest.raises(ValueError, match="head map"):
        damp.kda_decode_step_groups([(L, state, perm)], **_dev(_ops("kda")), **args)
    assert calls == []
