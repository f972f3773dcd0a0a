"""The extension module behind the codec calls: a changed parameter is seen by the next call, wrong arguments raise."""
import copy
import ctypes
import importlib.util
import pickle
import sys
import types

import pytest
import torch

from paper_2506_01352_b200 import binding as T


def test_a_changed_field_reaches_the_next_call():
    p = T.Params(tokens=128, hidden=256, group_tokens=64)
    assert T.tahq_encode(p, 4096, 8192, 16, 12288, 1 << 30, 0) == 3      # packed buffer too small
    q = copy.copy(p)
    p.tile = 48
    assert T.tahq_encode(p, 4096, 8192, 16, 12288, 1 << 30, 0) == 1 and p.raw() == bytes(p.c())
    assert q.raw() == bytes(q.c()) and T.tahq_encode(q, 4096, 8192, 16, 12288, 1 << 30, 0) == 3
    g = T.QNaiveParams(tokens=4, hidden=64)
    assert T.tahq_qnaive_encode(g, 4096, 8192, 16, 12288, 1 << 30, 0) == 3
    g.bits = 17
    assert T.tahq_qnaive_encode(g, 4096, 8192, 16, 12288, 1 << 30, 0) == 1
    assert p == T.Params(tokens=128, hidden=256, group_tokens=64, tile=48)   # what is kept is no field


def test_wrong_arguments_raise():
    p = T.Params(tokens=128, hidden=256, group_tokens=64)
    for args in [(p.raw(),), (b"short", 0, 0, 0, 0, 0, 0), (p.raw(), "x", 0, 0, 0, 0, 0), (p.c(), 0, 0, 0, 0, 0, 0)]:
        with pytest.raises(TypeError):
            T.call().encode(*args)
    assert T.call().encode(p.raw(), None, 0, 0, None, 0, None) == 1


def test_tensors_that_are_not_on_a_gpu_are_refused_before_the_call(monkeypatch):
    """Their addresses mean nothing to the kernels; the four calls are replaced, so nothing is launched here either way."""
    class Recorder:
        def __getattr__(self, name):
            return lambda *args: reached.append(name) or 0

    reached = []
    monkeypatch.setattr(T, "_call", Recorder())
    monkeypatch.setattr(T, "_raw_stream", lambda device: 0)
    monkeypatch.setattr(T, "_device", lambda: 0)
    x, ws = torch.zeros(4, 64), torch.zeros(256, dtype=torch.uint8)
    g = T.QNaiveParams(tokens=4, hidden=64)
    packed = torch.zeros(T.qnaive_packed_bound(g), dtype=torch.uint8)
    with pytest.raises(ValueError, match="cuda"):
        T.qnaive_encode(g, x, packed=packed, ws=ws)
    with pytest.raises(ValueError, match="cuda"):
        T.qnaive_decode(g, packed, out=x, ws=ws)
    with pytest.raises(ValueError, match="CUDA"):
        T.encode(T.params_for(x), x, packed=packed, ws=ws)
    assert reached == []


def test_a_field_that_changes_while_the_structure_is_laid_out_is_not_missed(monkeypatch):
    """Another thread's change, at the worst moment: between reading the fields and keeping the bytes."""
    p = T.Params(tokens=128, hidden=256, group_tokens=64)
    c = T.Params.c

    def interrupted(self):
        laid_out = c(self)
        self.tile = 32
        return laid_out

    monkeypatch.setattr(T.Params, "c", interrupted)
    p.raw()
    monkeypatch.setattr(T.Params, "c", c)
    assert p.raw() == bytes(p.c()) and p.c().tile == 32


def test_parameters_travel_as_their_fields_alone():
    p = T.Params(tokens=128, hidden=256, group_tokens=64)
    g = T.QNaiveParams(tokens=4, hidden=64)
    p.raw(), g.raw()
    assert T.Params(**vars(p)) == p and T.QNaiveParams(**vars(g)) == g
    for q in (pickle.loads(pickle.dumps(p)), copy.copy(p), copy.deepcopy(p)):
        assert q == p and T.tahq_encode(q, 4096, 8192, 16, 12288, 1 << 30, 0) == 3
        q.tile = 48
        assert T.tahq_encode(q, 4096, 8192, 16, 12288, 1 << 30, 0) == 1 and T.tahq_encode(p, 4096, 8192, 16, 12288, 1 << 30, 0) == 3
    assert p.__reduce_ex__(4)[2] == {k: getattr(p, k) for k in T.Params.__dataclass_fields__}   # what a file holds of it


def test_a_torch_without_the_private_stream_functions(monkeypatch):
    for name in ("_cuda_getDevice", "_cuda_getCurrentRawStream"):
        monkeypatch.delattr(torch._C, name, raising=False)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 1)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device: types.SimpleNamespace(cuda_stream=40 + device))
    spec = importlib.util.spec_from_file_location("paper_2506_01352_b200._binding_again", T.__file__)
    again = importlib.util.module_from_spec(spec)
    monkeypatch.setitem(sys.modules, spec.name, again)   # (dataclasses look their module up)
    spec.loader.exec_module(again)
    assert again._raw_stream(again._device()) == 41


@pytest.mark.parametrize("form", [int, ctypes.c_void_p, lambda v: types.SimpleNamespace(_as_parameter_=v),
                                  lambda v: types.SimpleNamespace(_as_parameter_=ctypes.c_void_p(v)), lambda v: v - (1 << 64)])
def test_the_forms_of_an_address(form):
    """As ctypes takes them, addresses in the upper half as negative numbers among them: what is wrong with the call is its
    alignment (4), not its arguments."""
    p = T.Params(tokens=128, hidden=256, group_tokens=64)
    odd, even = form(0x9000000000000008), form(0x9000000000000010)
    assert T.tahq_encode(p, odd, even, 1 << 40, even, ctypes.c_size_t(1 << 40), even) == 4
    assert T.tahq_decode(p, even, 1 << 40, odd, even, 1 << 40, form(0)) == 4
    g = T.QNaiveParams(tokens=4, hidden=64)
    assert T.tahq_qnaive_encode(g, even, odd, 1 << 40, even, 1 << 40, None) == 4
    for wrong in ("x", b"x", 1.5, [1], types.SimpleNamespace(value="x")):
        with pytest.raises(TypeError):
            T.tahq_encode(p, wrong, 0, 0, 0, 0, 0)


def test_a_field_that_is_deleted_has_its_default_again():
    p = T.Params(tokens=128, hidden=256, group_tokens=64, tile=48)
    assert T.tahq_encode(p, 4096, 8192, 16, 12288, 1 << 30, 0) == 1
    del p.tile
    assert p.raw() == bytes(p.c()) and T.tahq_encode(p, 4096, 8192, 16, 12288, 1 << 30, 0) == 3
