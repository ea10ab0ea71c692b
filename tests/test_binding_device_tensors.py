"""The binding's quick checks (_fits_*) stand alone before a call: where they accept, the per-tensor
checks are not run.  These tests reach them on the host, with CPU tensors of a class that says it is
on a GPU and a library stand-in that records the compute calls."""
import pytest
import torch

import paper_2608_27513_gb300 as damp
from paper_2608_27513_gb300 import _lib, build
from tests.test_binding_shapes import B, DK, DV, H, HQK, K, T, _NoCompute, _bad_ops, _layout, _ops, _perm, _pool


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
