"""The default configuration by the number of pairs: batches on either side of
each of its lines (one, four and eight pairs per SM) against a fixed tune, with
pairs of every size up to a global-class one, and a plan used again."""
import numpy as np
import pytest
import torch

from gen.cfg_grammar import structured_cfg
from _helpers import valid_matching

pytestmark = pytest.mark.gpu
api = pytest.importorskip("paper_1707_02423_gb300.api")
B = pytest.importorskip("paper_1707_02423_gb300._binding")
DEV = "cuda"


@pytest.mark.parametrize("per_sm,more", [(0, 1), (1, 0), (1, 1), (4, 0), (4, 1), (8, 0), (8, 1)])
def test_lines(per_sm, more):
    rng = np.random.default_rng(per_sm)
    P = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + more
    sizes = [1, 2, 7, 20, 33, 34, 47, 64, 70, 95, 96, 120, 137, 140, 300]
    cfgs = [structured_cfg(rng, n, 5, 7) for n in sizes]
    pairs = rng.integers(0, len(cfgs) - 3, (P, 2)).astype(np.int32)
    pairs[-1] = (P % len(cfgs), len(cfgs) - 1)
    pk = api.Pack(cfgs, 8, device=DEV)
    om = torch.linspace(0.5, 1.5, 8, device=DEV)
    ref = api.similarity(pk, pk, pairs, om, want_x=True, want_match=True, tune=1)
    ws = api.Workspace(DEV)
    for flags in (0, B.CF_FLAG_REUSE_PLAN):
        r = api.similarity(pk, pk, pairs, om, want_x=True, want_match=True, ws=ws, flags=flags)
        # either side is within 1e-5 of the exact X
        assert (r.X - ref.X).abs().max().item() <= 2e-5
        mt = r.match.cpu().numpy()
        for p in range(0, P, max(1, P // 40)):
            assert valid_matching(mt[r.m_off[p]:r.m_off[p + 1]], sizes[pairs[p][0]], sizes[pairs[p][1]])
        X = r.X.cpu().numpy()
        sc = r.scores.cpu().numpy()
        for p in range(0, P, max(1, P // 40)):  # the score is the matching's, in the call's own X
            x = X[r.x_off[p]:r.x_off[p + 1]].reshape(sizes[pairs[p][0]], -1).astype(np.float64)
            m = mt[r.m_off[p]:r.m_off[p + 1]]
            k = np.flatnonzero(m >= 0)
            assert abs(sc[p] - x[k, m[k]].sum()) <= 1e-5


@pytest.mark.parametrize("lo,hi", [(4, 12), (20, 45)])
def test_large_batch_defers_with_the_same_bits(lo, hi):
    """32 pairs per SM and more: the steps in the second kernel (pairs large
    enough, room in the workspace) or in place, with the bits of tune 1."""
    rng = np.random.default_rng(lo)
    P = 32 * torch.cuda.get_device_properties(0).multi_processor_count + 5
    sizes = [int(n) for n in rng.integers(lo, hi, 30)] + [300]
    cfgs = [structured_cfg(rng, n, 5, 7) for n in sizes]
    pairs = rng.integers(0, 30, (P, 2)).astype(np.int32)
    pairs[7] = (30, 3)
    pairs[8] = (30, 30)
    pk = api.Pack(cfgs, 8, device=DEV)
    om = torch.linspace(0.5, 1.5, 8, device=DEV)
    ref = api.similarity(pk, pk, pairs, om, want_match=True, tune=1)
    small = api.ws_size(pk, pk, pairs, B.params(tune=1))
    full = api.ws_size(pk, pk, pairs, B.params())
    assert (full > small) == (lo == 20)
    ws = api.Workspace(DEV)
    for size, flags in ((full, 0), (full, B.CF_FLAG_REUSE_PLAN), (small, 0)):
        r = api.similarity(pk, pk, pairs, om, want_match=True, ws=ws, ws_bytes=size, flags=flags)
        assert torch.equal(r.scores, ref.scores) and torch.equal(r.match, ref.match)
