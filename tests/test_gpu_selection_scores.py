"""Scores outside the usual range -- tiles whose entropy, as Eq. 2 evaluates it with its varsigma, is below zero -- against
the oracle: such a tile ranks behind the others, and exactly k_hi tiles get the higher width all the same."""
import pytest
import torch

from paper_2506_01352_b200 import binding as T
from tests.test_gpu_parity import check_decode, check_encode

pytestmark = pytest.mark.gpu


def check(x, **kw):
    p = T.params_for(x, **kw)
    packed, want, ws = check_encode(p, x)
    check_decode(p, packed, want, ws)


def one_hot(tokens, hidden, dtype, step, dense=0.0):
    """One element in `step` is not zero; `dense`: share of the tokens that are filled."""
    g = torch.Generator(device="cuda").manual_seed(tokens + step)
    x = torch.randn(tokens, hidden, generator=g, device="cuda")
    keep = torch.zeros(hidden, dtype=torch.bool, device="cuda")
    keep[::step] = True
    rows = torch.rand(tokens, generator=g, device="cuda") >= dense
    x[rows[:, None] & ~keep[None, :]] = 0
    return x.to(dtype)


# groups of whole words of the bit map and others, tiles above and below the width of a lane, allocation tiles
FORMS = [dict(tile=64, group_tokens=64), dict(tile=64, group_tokens=37), dict(tile=32, group_tokens=148), dict(tile=128, group_tokens=37),
         dict(tile=8, group_tokens=74), dict(tile=64, alloc_tile=256, group_tokens=37), dict(tile=32, alloc_tile=512, group_tokens=64)]


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("dense", [0.0, 0.1])
@pytest.mark.parametrize("eps_log", [1e-6, 1e-4])
def test_scores_just_below_zero(eps_log, dense, form, dtype):
    tokens = form["group_tokens"] * 3
    check(one_hot(tokens, 512, dtype, 64, dense), budget_millibits=3500, eps_log=eps_log, **form)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("dense", [0.0, 1.0])
@pytest.mark.parametrize("eps_log", [1.0, 4.0, 1e30])
def test_scores_far_below_zero(eps_log, dense, form, dtype):
    tokens = form["group_tokens"] * 3
    check(one_hot(tokens, 512, dtype, 64, dense), budget_millibits=3500, eps_log=eps_log, **form)
