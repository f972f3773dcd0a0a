"""Scores outside the usual range against the oracle: tiles whose entropy, as Eq. 2 evaluates it with its varsigma, is below
zero, magnitudes and epsilons near the ends of binary32.  Exactly k_hi tiles get the higher width, and the right ones."""
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


# groups whose scores a kernel of their own forms, or the selection (a few whole words of a small tensor)
LONG = [dict(tile=32, group_tokens=300), dict(tile=64, group_tokens=512), dict(tile=128, group_tokens=300), dict(tile=8, group_tokens=150),
        dict(tile=16, group_tokens=512)]


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("form", FORMS[:5] + LONG)
@pytest.mark.parametrize("low,high", [(-37, -20), (-25, 37), (20, 36), (35.5, 38.3)])
@pytest.mark.parametrize("eps_l1", [1e-30, 1e-8, 1e20])
def test_magnitudes_near_the_ends_of_binary32(eps_l1, low, high, form, dtype):
    """Tokens from 10^low to 10^high; the largest sums of magnitudes overflow, which Eq. 1 gives a score of zero."""
    tokens = form["group_tokens"] * 2
    g = torch.Generator(device="cuda").manual_seed(tokens)
    x = torch.randn(tokens, 1024, generator=g, device="cuda").clamp_(-1.5, 1.5).to(torch.float64)
    x *= 10.0 ** (low + (high - low) * torch.rand(tokens, 1, generator=g, device="cuda", dtype=torch.float64))
    x[torch.rand(tokens, generator=g, device="cuda") < 0.1] = 0
    check(x.to(dtype), budget_millibits=3500, eps_l1=eps_l1, tau=float("inf"), **form)


@pytest.mark.parametrize("form", [FORMS[0], FORMS[1], FORMS[6], LONG[1], LONG[3]])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("eps_l1", [3e38, float("inf")])
def test_an_epsilon_that_leaves_no_score(eps_l1, dtype, form):
    """Every score is next to or exactly zero: the first tiles of a group get the higher width."""
    check(one_hot(form["group_tokens"] * 2, 512, dtype, 64, 0.5), budget_millibits=3500, eps_l1=eps_l1, **form)


@pytest.mark.parametrize("form", [FORMS[0], FORMS[1], FORMS[5], LONG[1], LONG[3]])
def test_tiles_of_zeroes_without_epsilon(form):
    """p = 0/0, which leaves the rank of such a tile open, but not the number of tiles of either width."""
    x = one_hot(form["group_tokens"] * 2, 512, torch.float32, 64, 0.5)
    x[::3] = 0
    p = T.params_for(x, budget_millibits=3500, eps_l1=0.0, **form)
    ws = T.alloc_workspace(p)
    packed = T.encode(p, x, ws=ws)
    assert T.device_status(ws) == 0
    out = T.decode(p, packed, ws=ws)
    assert T.device_status(ws) == 0
    assert (out[::3] == 0).all() and ((out - x).abs().amax(1) <= 0.2 * x.abs().amax(1)).all()
