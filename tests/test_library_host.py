"""Host-only checks of the C-ABI library (no GPU needed): it builds, loads, exports every symbol the
header declares, and its size/layout functions agree with the oracle's independent arithmetic."""
import ctypes as C
import os
import re

import pytest

import oracle as O
from paper_2506_01352_b200 import binding as T
from paper_2506_01352_b200 import build as B

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def test_every_declared_symbol_is_exported():
    lib = C.CDLL(B.LIB)
    declared = {}
    for h in ("tahq.h", "tahq_testing.h"):
        hdr = open(os.path.join(ROOT, "include", h)).read()
        hdr = re.sub(r"/\*.*?\*/", "", hdr, flags=re.S)
        declared[h] = set(re.findall(r"\b(tahq_[a-z0-9_]+)\s*\(", hdr))
        for name in sorted(declared[h]):
            assert hasattr(lib, name), f"{name} is declared in include/{h} but not exported"
    assert {"tahq_encode", "tahq_decode", "tahq_packed_bound", "tahq_workspace_bound"} <= declared["tahq.h"]
    # the codec's header holds the codec, Q_Naive and the workspace-free encode only
    assert not {n for n in declared["tahq.h"] if "profile" in n or "selftest" in n or "launch_count" in n}
    assert declared["tahq.h"] | declared["tahq_testing.h"] == set(T.EXPORTS)


CASES = [
    dict(tokens=128, hidden=256, group_tokens=64, tile=64, budget_millibits=3800),
    dict(tokens=128, hidden=256, group_tokens=64, tile=32, budget_millibits=4000),
    dict(tokens=8192, hidden=768, group_tokens=1024, tile=64, budget_millibits=3000),
    dict(tokens=8192, hidden=4096, dtype=1, group_tokens=2048, tile=64, budget_millibits=3500),
    dict(tokens=16384, hidden=5120, group_tokens=2048, tile=128, budget_millibits=3000),
    dict(tokens=65536, hidden=8192, dtype=1, group_tokens=4096, tile=64, budget_millibits=2200),
    dict(tokens=77, hidden=96, group_tokens=11, tile=32, budget_millibits=7999),
    dict(tokens=5, hidden=128, group_tokens=0, tile=128, budget_millibits=8000),
]


@pytest.mark.parametrize("kw", CASES)
def test_layout_agrees_with_the_oracle(kw):
    lt = T.packed_layout(T.Params(**kw))
    lo = O.layout(O.Params(**kw))
    assert lt == lo
    assert T.packed_bound(T.Params(**kw)) == O.packed_bound(O.Params(**kw)) == lt["total_bytes"]
    assert T.workspace_bound(T.Params(**kw)) >= 256


def test_invalid_and_unsupported_parameters():
    base = dict(tokens=128, hidden=256, group_tokens=64, tile=64, budget_millibits=3800)
    for kw in [dict(tile=48), dict(hidden=100), dict(group_tokens=5), dict(budget_millibits=1999),
               dict(budget_millibits=8001), dict(tile=256), dict(dtype=2), dict(tokens=0), dict(tau=-1.0),
               dict(tile=4), dict(rounding=2), dict(alloc_tile=96), dict(hidden=32768, tile=128, alloc_tile=16384)]:
        p = T.Params(**{**base, **kw})
        assert T.packed_bound(p) == 0 and T.workspace_bound(p) == 0
        with pytest.raises(T.TahqError):
            T.packed_layout(p)
    # host-detectable errors come back before anything touches CUDA
    p = T.Params(**base)
    assert T.tahq_encode(p, 0, 0, 0, 0, 0, 0) == 1                       # null pointers
    assert T.tahq_encode(p, 4096, 8192, 16, 12288, 1 << 30, 0) == 3      # packed buffer too small
    assert T.tahq_encode(p, 4096, 8192, 1 << 30, 12288, 16, 0) == 3      # workspace too small
    assert T.tahq_encode(p, 4100, 8192, 1 << 30, 12288, 1 << 30, 0) == 4  # misaligned input
    assert T.tahq_decode(p, 8192, 1 << 30, 4104, 12288, 1 << 30, 0) == 4
    bad = p.c(); bad.struct_size = 8
    assert T.lib().tahq_packed_bound(C.byref(bad)) == 0
    assert T.status_string(0) == "ok" and "small" in T.status_string(3)


def test_no_shuffle_takes_whoever_happens_to_be_there():
    """__activemask() names the lanes that run together at that moment, which need not be all that take the branch: votes that
    only choose between two ways to the same result may use it, an exchange between lanes may not."""
    for f in sorted(os.listdir(os.path.join(ROOT, "paper_2506_01352_b200", "csrc"))):
        if f.endswith((".cu", ".cuh")):
            src = open(os.path.join(ROOT, "paper_2506_01352_b200", "csrc", f)).read()
            assert not re.search(r"__(shfl|reduce|match)\w*_sync\(\s*__activemask", src), f


@pytest.mark.parametrize("tokens,M,G,m", [(9018, 214, 128, 1), (14572, 138, 64, 1), (16257, 244, 128, 2), (25921, 300, 128, 4),
                                          (736428, 77, 64, 77), (669310, 3, 8, 1), (1023, 1024, 64, 1), (65535, 16, 64, 1)])
def test_the_workspace_free_encode_takes_what_it_always_took(tokens, M, G, m):
    """Scores (4 bytes a ranked tile) and look-back flags fit the built-in scratch; the offset prefixes have room of their own.
    (Accepted is: refused for the packed buffer's size, or, without a GPU, for the lack of one.)"""
    p = T.Params(tokens=tokens, hidden=M * G, group_tokens=4 if m == M else 0, tile=G, budget_millibits=3800, alloc_tile=m * G)
    assert T.packed_bound(p) > 0 and 4 * tokens * M // m + 8 * 2048 + 512 <= T.NOALLOC_SCRATCH_BYTES
    assert T.tahq_encode_noalloc(p, 4096, 8192, 16, 0) in (3, 5)
