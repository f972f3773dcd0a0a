"""Edges of the lane-shared tile kernels against the oracle: numbers of tiles around a round and around a bit-map word,
every pair of widths, every tile transformed, tensors that start 16 bytes off a 32-byte boundary, a corrupt bit map."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2506_01352_b200 import binding as T
from paper_2506_01352_b200 import synth
from tests.guards import Guarded
from tests.test_gpu_parity import check_decode, check_encode, oparams

pytestmark = pytest.mark.gpu


def tensor(tokens, hidden, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(tokens, hidden, generator=g, device="cuda") * torch.randn(tokens, 1, generator=g, device="cuda").exp()
    x[:, ::37] *= 25
    return x.to(dtype)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("G", [32, 64, 128])
@pytest.mark.parametrize("tokens,M", [(1, 1), (1, 3), (1, 31), (1, 33), (7, 9), (129, 37), (1, 4743), (593, 32)])
def test_tile_counts_around_rounds_and_words(tokens, M, G, dtype):
    x = tensor(tokens, M * G, dtype, tokens * 1000 + M)
    for beta, tau in ((3800, 2.0), (2500, 0.0)):
        p = T.params_for(x, tile=G, budget_millibits=beta, tau=tau)
        packed, want, ws = check_encode(p, x)
        check_decode(p, packed, want, ws)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("G", [32, 64, 128])
@pytest.mark.parametrize("beta", [2000, 2500, 3000, 3500, 4000, 4500, 5000, 5500, 6000, 6500, 7000, 7500, 8000])
def test_every_pair_of_widths(beta, G, dtype):
    x = tensor(40, 3 * G, dtype, beta)
    p = T.params_for(x, tile=G, group_tokens=20, budget_millibits=beta)
    packed, want, ws = check_encode(p, x)
    check_decode(p, packed, want, ws)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("beta", [3800, 6500])
def test_tensors_off_a_32_byte_boundary(beta, dtype):
    x = tensor(100, 192, dtype, 5)
    p = T.params_for(x, budget_millibits=beta)
    nb = x.numel() * x.element_size()
    want = O.encode(oparams(p), synth.to_host_array(x))
    gin, gout = Guarded(nb + 16, "cuda"), Guarded(nb + 16, "cuda")
    src, dst = gin.view[16:].view(dtype).view(100, 192), gout.view[16:].view(dtype).view(100, 192)
    src.copy_(x)
    packed = T.encode(p, src)
    T.decode(p, packed, out=dst)
    torch.cuda.synchronize()
    gout.check("output tensor")
    assert np.array_equal(packed.cpu().numpy(), want)
    back = synth.to_host_array(dst)
    assert np.array_equal(back, O.decode(oparams(p), want))


@pytest.mark.parametrize("fill", [0x00, 0xFF, 0x5A])
def test_a_corrupt_bit_map_is_reported_and_stays_inside_the_buffers(fill):
    x = tensor(600, 640, torch.bfloat16, 9)
    p = T.params_for(x, budget_millibits=3800)
    L = T.packed_layout(p)
    gpk = Guarded(T.packed_bound(p), "cuda")
    gout = Guarded(x.numel() * 2, "cuda")
    ws = T.alloc_workspace(p)
    T.encode(p, x, packed=gpk.view, ws=ws)
    gpk.view[L["off_bitmap"]:L["off_scale_zero"]] = fill
    T.decode(p, gpk.view, out=gout.typed(torch.bfloat16, (600, 640)), ws=ws)
    torch.cuda.synchronize()
    assert T.device_status(ws) == T.DEV_BAD_BITMAP
    gout.check("output tensor")
