"""The extension module behind the codec calls: a changed parameter is seen by the next call, wrong arguments raise."""
import copy

import pytest

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
