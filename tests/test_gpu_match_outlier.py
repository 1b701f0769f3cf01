"""Greedy matching in phases where the rows' best values crowd: more of them in
the first of the 256 ranges than rows can be listed."""
import numpy as np
import pytest
import torch

from test_gpu_large_match import greedy, near_rank_one, pack
from test_gpu_match_ties import took

pytestmark = pytest.mark.gpu
api = pytest.importorskip("paper_1707_02423_gb300.api")
DEV = "cuda"


def crowded(na, nb, how):
    """Rows whose best values agree to 1 in 2**how, and one far below."""
    g = torch.Generator(device=DEV).manual_seed(3)
    x = 1 + 2.0 ** -how * torch.rand(na, nb, generator=g, device=DEV)
    x[na // 2] *= -1 if how % 2 else 1e-6
    return x


@pytest.mark.parametrize("na,nb", [(900, 700), (170, 200), (5200, 90)])
@pytest.mark.parametrize("how", [2, 9, 16, 21, 23])
def test_matchings(na, nb, how):
    x = crowded(na, nb, how)
    pk = pack((na, nb))
    r = api.match(pk, pk, [(0, 1)], x.flatten())
    assert np.array_equal(r.match.cpu().numpy(), greedy(x.cpu().numpy()))


def test_no_cliff():
    """One row far below the others puts them all into one range."""
    g = torch.Generator(device=DEV).manual_seed(8)
    pk = pack((1500, 1500))
    near = took(pk, [(0, 1)], near_rank_one(g, 1500, 1500).flatten())
    far = took(pk, [(0, 1)], crowded(1500, 1500, 6).flatten())
    print(f"\n  1,500 x 1,500: near rank one {1e3 * near:.2f} ms, one row far below {1e3 * far:.2f} ms")
    assert far <= 4 * near
