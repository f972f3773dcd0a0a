"""Every width of the fixed-point compressor at rows that end inside a lane's 32 elements, inside a warp's 1024 and past
a CTA's 8192, with few and many rows, and on tensors that start 16 bytes off a 32-byte boundary."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2506_01352_b200 import binding as T
from paper_2506_01352_b200 import synth
from tests.guards import Guarded
from tests.test_gpu_qnaive import _check

pytestmark = pytest.mark.gpu


def rows(tokens, hidden, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(tokens, hidden, generator=g, device="cuda") * torch.randn(tokens, 1, generator=g, device="cuda").exp()
    return (x * 1e-3).to(dtype)


@pytest.mark.parametrize("bits", range(2, 17))
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("shape", [(700, 8), (261, 72), (37, 520), (19, 1024), (5, 1048), (3, 5160), (2, 16408)])
def test_every_width_at_ragged_rows(shape, dtype, bits):
    _check(rows(*shape, dtype, bits), bits, bits % 2, 1000.0 if bits % 3 else 1024.0)


@pytest.mark.parametrize("bits", [6, 7, 8])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_tensors_off_a_32_byte_boundary(dtype, bits):
    x = rows(33, 1056, dtype, bits)
    dt = T.F32 if dtype == torch.float32 else T.BF16
    p = T.QNaiveParams(tokens=33, hidden=1056, dtype=dt, bits=bits)
    po = O.QNaiveParams(tokens=33, hidden=1056, dtype=dt, bits=bits)
    nb = x.numel() * x.element_size()
    gin, gout = Guarded(nb + 16, "cuda"), Guarded(nb + 16, "cuda")
    src, dst = gin.view[16:].view(dtype).view(33, 1056), gout.view[16:].view(dtype).view(33, 1056)
    src.copy_(x)
    packed, _ = T.qnaive_encode(p, src)
    T.qnaive_decode(p, packed, out=dst)
    torch.cuda.synchronize()
    gout.check("output tensor")
    want = O.qnaive_encode(po, synth.to_host_array(x))
    assert np.array_equal(packed.cpu().numpy(), want)
    assert np.array_equal(synth.to_host_array(dst), O.qnaive_decode(po, want))


@pytest.mark.parametrize("c", [3.0, 1000.0, 0.1, 8191.0, 1.0000001, 1.9999999, 3e-12, 7e13])
@pytest.mark.parametrize("bits", [8, 13, 16])
def test_division_by_pre_scales_that_are_no_power_of_two(bits, c):
    """Scales from far below to far above the range in which the quotient is formed from the reciprocal."""
    x = rows(64, 2048, torch.float32, bits) * torch.logspace(-18, 18, 64, device="cuda")[:, None]
    x[5] = 0
    _check(x.contiguous(), bits, 0, c)


@pytest.mark.parametrize("dtype,n", [(torch.float32, 1025), (torch.bfloat16, 2049)])
def test_a_row_beyond_four_gibibytes(dtype, n):
    """The tensor as a single row and as rows of 2^20 elements, with one scale: the same codes, the same values."""
    dt = T.F32 if dtype == torch.float32 else T.BF16
    x = torch.empty(n, 1 << 20, dtype=dtype, device="cuda")
    for r in range(0, n, 205):
        x[r:r + 205] = rows(min(205, n - r), 1 << 20, dtype, r)
    short = T.QNaiveParams(tokens=n, hidden=1 << 20, dtype=dt, bits=2, per_tensor=1)
    long = T.QNaiveParams(tokens=1, hidden=n << 20, dtype=dt, bits=2, per_tensor=1)
    a, ws = T.qnaive_encode(short, x)
    b, _ = T.qnaive_encode(long, x.view(1, -1), ws=ws)
    assert T.device_status(ws) == 0 and torch.equal(a[128:], b[128:])
    want, _ = T.qnaive_decode(short, a, ws=ws)
    got, _ = T.qnaive_decode(long, b, out=x.view(1, -1).fill_(float("nan")), ws=ws)
    assert T.device_status(ws) == 0 and torch.equal(got.view(n, -1), want)


@pytest.mark.parametrize("bits", range(2, 17))
@pytest.mark.parametrize("per_tensor", [0, 1])
@pytest.mark.parametrize("dtype,shape", [(torch.float32, (9, 2056)), (torch.bfloat16, (9, 1024)), (torch.bfloat16, (3, 8392))])
def test_rows_whose_scaled_gradients_overflow(dtype, shape, per_tensor, bits):
    """Finite gradients, and c g beyond the largest number in every third element of every second row: the scale is infinite
    and each code that of zero."""
    x = rows(*shape, dtype, bits)
    x[::2, ::3] = 3e37
    dt = T.F32 if dtype == torch.float32 else T.BF16
    kw = dict(tokens=shape[0], hidden=shape[1], dtype=dt, bits=bits, per_tensor=per_tensor, prescale=1024.0)
    packed, _ = T.qnaive_encode(T.QNaiveParams(**kw), x)
    assert np.array_equal(packed.cpu().numpy(), O.qnaive_encode(O.QNaiveParams(**kw), synth.to_host_array(x)))
