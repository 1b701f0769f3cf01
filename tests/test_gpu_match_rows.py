"""Greedy matching in phases of matrices with short rows, whose best values a warp
finds several rows at a time: up to two chunks of 32 columns, and beyond."""
import numpy as np
import pytest
import torch

from test_gpu_large_match import greedy, near_rank_one, pack
from test_gpu_match_ties import took

pytestmark = pytest.mark.gpu
api = pytest.importorskip("paper_1707_02423_gb300.api")
DEV = "cuda"


@pytest.mark.parametrize("nb", [3, 31, 32, 33, 64, 65, 96, 97, 129, 161, 193, 225, 256, 257])
@pytest.mark.parametrize("na", [6000 // 3, 5300])
def test_matchings(na, nb):
    g = torch.Generator(device=DEV).manual_seed(nb)
    x = near_rank_one(g, na if nb > 3 else 3 * na, nb)
    x[5, :] = float("-inf")  # a row that is never taken
    pk = pack(tuple(x.shape))
    r = api.match(pk, pk, [(0, 1)], x.flatten())
    assert np.array_equal(r.match.cpu().numpy(), greedy(x.cpu().numpy()))


def test_short_rows():
    """13 steps a matrix, whichever way round."""
    g = torch.Generator(device=DEV).manual_seed(8)
    t = []
    for s in ((5000, 13), (13, 5000)):
        t.append(took(pack(s), np.tile([(0, 1)], (304, 1)), near_rank_one(g, *s).flatten().repeat(304)))
    print(f"\n  304 matrices of 5,000 x 13: {1e3 * t[0]:.2f} ms, of 13 x 5,000: {1e3 * t[1]:.2f} ms")
    assert t[0] <= 12 * t[1]
