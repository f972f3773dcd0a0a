"""The cluster selection against the oracle at the lengths where its paths change: groups around a word, a thread's
scores in registers, a cluster, slices whose words leave shared memory; groups that share words of the bit map;
allocation tiles; more equal scores than the key list holds, in all of these."""
import pytest
import torch

from paper_2506_01352_b200 import binding as T
from tests.test_gpu_parity import check_decode, check_encode

pytestmark = pytest.mark.gpu


def tensor(tokens, hidden, dtype, seed, equal=0.0):
    """`equal`: share of the tokens whose tiles are all the same, so that their scores tie."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(tokens, hidden, generator=g, device="cuda") * torch.randn(tokens, 1, generator=g, device="cuda").exp()
    x[:, ::37] *= 25
    n = int(tokens * equal)
    if n:
        x[torch.randperm(tokens, generator=g, device="cuda")[:n]] = torch.linspace(-1, 1, 8, device="cuda").repeat(hidden // 8)
    return x.to(dtype)


def check(x, **kw):
    p = T.params_for(x, **kw)
    packed, want, ws = check_encode(p, x)
    check_decode(p, packed, want, ws)


@pytest.mark.parametrize("groups,tiles", [(1, 1), (3, 5), (5, 31), (4, 33), (2, 4096), (3, 4099), (1, 65536), (2, 65537), (300, 7),
                                          (40, 4097), (1, 70003)])
@pytest.mark.parametrize("equal", [0.0, 0.9])
def test_group_lengths(groups, tiles, equal):
    """A group of `tiles` tokens of one tile each."""
    check(tensor(groups * tiles, 32, torch.bfloat16, tiles, equal), tile=32, group_tokens=tiles, budget_millibits=3700)


@pytest.mark.parametrize("tokens,equal", [(131101, 0.0), (131101, 0.5), (131072, 0.0)])
def test_slices_beyond_shared_memory(tokens, equal):
    check(tensor(tokens, 72, torch.bfloat16, 1, equal), tile=8, budget_millibits=2600)


@pytest.mark.parametrize("S,G,A", [(37, 32, 96), (100, 32, 32 * 45), (5, 64, 64 * 3), (1000, 8, 40), (3, 32, 32 * 9)])
@pytest.mark.parametrize("equal", [0.0, 0.9])
def test_allocation_tiles_in_groups_that_share_words(S, G, A, equal):
    check(tensor(7 * S, 32 * 45 if A % 45 == 0 else A * 3, torch.float32, S, equal), tile=G, group_tokens=S, alloc_tile=A,
          budget_millibits=3300)


def test_one_group_of_thousands_of_equal_allocation_tiles():
    check(tensor(9001, 192, torch.bfloat16, 2, 0.95), tile=32, alloc_tile=96, group_tokens=9001, budget_millibits=3500)


@pytest.mark.parametrize("groups,tiles,G,dtype", [
    (1, 32, 32, torch.bfloat16), (74, 32, 64, torch.float32), (75, 32, 64, torch.float32),   # half the SMs' worth of CTAs
    (3, 544, 32, torch.bfloat16), (2, 96, 128, torch.float32), (9, 288, 64, torch.bfloat16),
    (2, 8192, 32, torch.float32), (2, 8224, 32, torch.float32),     # 16384 elements in each of 16 CTAs
    (4, 4096, 64, torch.bfloat16), (4, 4128, 64, torch.bfloat16), (1, 2048, 128, torch.bfloat16), (1, 2080, 128, torch.bfloat16)])
@pytest.mark.parametrize("equal", [0.0, 0.9])
def test_scores_formed_in_the_selection(groups, tiles, G, dtype, equal):
    check(tensor(groups * tiles, G, dtype, tiles, equal), tile=G, group_tokens=tiles, budget_millibits=3300)
