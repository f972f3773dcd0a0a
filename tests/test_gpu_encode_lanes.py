"""The quantiser's reciprocal and division against the correctly rounded ones, over every scale and every width (one tile
per scale whose range makes the scale); bf16 on both sides of the size where the tile kernel changes."""
import numpy as np
import pytest
import torch

from paper_2506_01352_b200 import binding as T
from tests.test_gpu_parity import check_decode, check_encode

pytestmark = pytest.mark.gpu


def check(x, **kw):
    p = T.params_for(x, **kw)
    packed, want, ws = check_encode(p, x)
    check_decode(p, packed, want, ws)


@pytest.mark.parametrize("bits", [2, 3, 4, 5, 6, 7, 8])
def test_every_binary16_scale(bits):
    """Tile j holds 32 values between 0 and scale j times 2^bits - 1 (as far as binary16 goes), some of them on and around
    the midpoints between codes, where a reciprocal that is one unit off gives another code."""
    s = np.arange(1, 0x7C00, dtype=np.uint16).view(np.float16).astype(np.float64)
    q = 2 ** bits - 1
    s = s[s * q < 60000]
    x = (s[:, None] * (np.arange(32) % q + 0.5)[None, :]).astype(np.float32)
    x[:, 0] = 0
    x[:, 1] = (s * q).astype(np.float32)
    x[:, 2::3] = np.nextafter(x[:, 2::3], np.float32(0))
    x[:, 3::3] = np.nextafter(x[:, 3::3], np.float32(1e9))
    n = len(x) // 8 * 8
    check(torch.from_numpy(x[:n].reshape(n // 8, 256)).cuda(), tile=32, budget_millibits=bits * 1000, tau=float("inf"))


@pytest.mark.parametrize("bits", [2, 3, 4, 5, 6, 7, 8])
def test_ranges_that_round_both_ways(bits):
    g = torch.Generator(device="cuda").manual_seed(bits)
    x = torch.randn(3000, 256, generator=g, device="cuda") * torch.randn(3000, 1, generator=g, device="cuda").mul(9).exp()
    check(x, tile=32, budget_millibits=bits * 1000)


@pytest.mark.parametrize("G,tokens", [(32, 2959), (32, 2961), (64, 2959), (64, 2961), (128, 1479), (128, 1481)])
@pytest.mark.parametrize("rounding", [0, 1])
def test_bf16_around_two_rounds_per_warp(G, tokens, rounding):
    """148 SMs x 20 warps x 2 rounds of 32, 16 or 8 tiles: 64, 32 or 32 tiles to a token put the line at 2960, 2960, 1480."""
    g = torch.Generator(device="cuda").manual_seed(G)
    x = torch.randn(tokens, G * (64 if G == 32 else 32), generator=g, device="cuda")
    x[:, ::41] *= 30
    check(x.bfloat16(), tile=G, budget_millibits=3600, rounding=rounding, seed=5)


@pytest.mark.parametrize("tokens", [1479, 1480, 1481])
@pytest.mark.parametrize("budget", [3600, 4000, 4600])
def test_bf16_around_one_round_per_warp(tokens, budget):
    """148 SMs x 20 warps x 16 tiles of 64, the line where no width is above 4 bits: 1480 tokens of 32 tiles."""
    g = torch.Generator(device="cuda").manual_seed(tokens)
    x = torch.randn(tokens, 2048, generator=g, device="cuda")
    x[:, ::41] *= 30
    check(x.bfloat16(), tile=64, budget_millibits=budget)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("G", [8, 16, 32, 64, 128])
@pytest.mark.parametrize("budget,rounding", [(3500, 0), (6500, 0), (8000, 1)])
def test_transformed_tiles_whose_sums_overflow(budget, rounding, G, dtype):
    """One or two magnitudes near the largest number in a tile: finite input whose transform (Eq. 4) is not."""
    x = torch.zeros(60, 4 * G, device="cuda")
    x[:, ::G] = 3e38
    x[:, 3::G] = torch.linspace(0, 1.4e38, 60, device="cuda")[:, None]
    x[1::2] *= -1
    check(x.to(dtype), tile=G, budget_millibits=budget, rounding=rounding, seed=3)


@pytest.mark.parametrize("bits", [2, 3, 4, 5, 6, 7, 8])
def test_scales_up_to_the_largest_and_beyond(bits):
    """As test_every_binary16_scale, for the scales that it leaves out, up to 65504, and ranges of up to 2^40 whose scale is that."""
    s = np.arange(1, 0x7C00, dtype=np.uint16).view(np.float16).astype(np.float64)
    q = 2 ** bits - 1
    s = np.concatenate([s[s * q > 50000], 65504 * 2.0 ** (np.arange(1, 49) / 2)])
    s = np.concatenate([s, s[-1:].repeat(-len(s) % 8)])
    x = (s[:, None] * (np.arange(32) % q + 0.5)[None, :]).astype(np.float32)
    x[:, 0] = 0
    x[:, 1] = (s * q).astype(np.float32)
    x[:, 2::3] = np.nextafter(x[:, 2::3], np.float32(0))
    x[:, 3::3] = np.nextafter(x[:, 3::3], np.float32(1e30))
    check(torch.from_numpy(x.reshape(-1, 256)).cuda(), tile=32, budget_millibits=bits * 1000, tau=float("inf"))
