"""Matching of a batch of large given matrices: side by side, a CTA each, as many
as there are CTAs."""
import numpy as np
import pytest
import torch

from test_gpu_large_match import greedy, near_rank_one, pack
from test_gpu_match_ties import took

pytestmark = pytest.mark.gpu
api = pytest.importorskip("paper_1707_02423_gb300.api")
DEV = "cuda"


def test_side_by_side():
    g = torch.Generator(device=DEV).manual_seed(8)
    P = torch.cuda.get_device_properties(0).multi_processor_count
    pk, x = pack((2000, 2000)), near_rank_one(g, 2000, 2000).flatten()
    one = took(pk, [(0, 1)], x)
    X, pairs = x.repeat(P), np.tile([(0, 1)], (P, 1))
    all_ = took(pk, pairs, X)
    print(f"\n  2,000 x 2,000: one {1e3 * one:.2f} ms, {P} {1e3 * all_:.2f} ms")
    assert all_ <= 10 * one
    m = api.match(pk, pk, pairs, X).match.cpu().numpy().reshape(P, 2000)
    assert (m == greedy(x.view(2000, 2000).cpu().numpy())).all()
