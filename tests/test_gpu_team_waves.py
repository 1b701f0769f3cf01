"""Batches of global-class pairs of one size, fewer than CTAs but more than teams
of two: a CTA each, in one wave."""
import time

import numpy as np
import pytest
import torch

from gen.cfg_grammar import structured_cfg

pytestmark = pytest.mark.gpu
api = pytest.importorskip("paper_1707_02423_gb300.api")
DEV = "cuda"


@pytest.mark.parametrize("na,nb", [(40, 600), (150, 150)])
def test_one_wave(na, nb):
    rng = np.random.default_rng(3)
    n = torch.cuda.get_device_properties(0).multi_processor_count
    pk = api.Pack([structured_cfg(rng, k, 6, 12) for k in (na, nb)], 13, device=DEV)
    om, took, res = torch.ones(13, device=DEV), [], []
    for P in (2 * n // 3, n):
        ws, pairs, best = api.Workspace(DEV), np.tile([(0, 1)], (P, 1)), 1e9
        for _ in range(5):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            r = api.similarity(pk, pk, pairs, om, ws=ws, want_match=True)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        took.append(best)
        res.append((r.scores[0], r.match[:na]))
        assert (r.scores == r.scores[0]).all()
    assert torch.equal(res[0][1], res[1][1]) and abs(res[0][0] - res[1][0]) <= 1e-5
    print(f"\n  {na} x {nb}: {2 * n // 3} pairs {1e3 * took[0]:.2f} ms, {n} {1e3 * took[1]:.2f} ms")
    assert took[0] <= 1.2 * took[1]
