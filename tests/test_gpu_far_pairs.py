"""Pairs whose rows are too long for a ring in shared memory (about 3,800 columns
and more): the sweep that reads both graphs' lists and the rows from memory."""
import time

import numpy as np
import pytest
import torch

import oracle
from gen.cfg_grammar import CFG, structured_cfg

pytestmark = pytest.mark.gpu
api = pytest.importorskip("paper_1707_02423_gb300.api")
DEV = "cuda"


def graph(rng, n, hubs=()):
    """A structured graph with blocks of the given in-degrees (a STOP block
    collects an edge from every early return) and as many branches."""
    c = structured_cfg(rng, n, 6, 12)
    src, dst, w = [c.src], [c.dst], [c.w]
    for k in hubs:
        h = int(rng.integers(0, n))
        other = rng.choice(n, min(k, n), replace=False).astype(np.int32)
        for s, d in ((other, np.full_like(other, h)), (np.full(3, (h + 1) % n, np.int32), other[:3])):
            src.append(s)
            dst.append(d)
            w.append(rng.random(len(s)).astype(np.float32))
    return CFG(n, np.concatenate(src), np.concatenate(dst), np.concatenate(w), c.attr)


# lists on both sides of a lane's (16) and of a warp's width, in rows, columns and both
@pytest.mark.parametrize("na,nb,ha,hb", [(130, 4100, (), ()), (130, 4100, (16, 17, 40), (16, 17, 33)),
                                         (61, 4097, (50,), (200, 200)), (200, 3999, (5, 18), ()),
                                         (4100, 4100, (17, 90), (130,)), (1, 4500, (), (40,))])
@pytest.mark.parametrize("K", [1, 6])
def test_against_the_oracle(na, nb, ha, hb, K):
    rng = np.random.default_rng([na, nb, K])
    a, b = graph(rng, na, ha), graph(rng, nb, hb)
    pk = api.Pack([a, b], 13, device=DEV)
    om = torch.linspace(0.5, 1.5, 13, device=DEV)
    r = api.similarity(pk, pk, [(0, 1)], om, 0.8, K, want_x=True, want_scores=False)
    ref = oracle.similarity(a, b, om.cpu().numpy(), 0.8, K)["X"]
    assert np.abs(r.X.cpu().numpy().reshape(ref.shape) - ref).max() <= 1e-5


def chain(rng, n, hub=0):
    src, dst = np.arange(n - 1), np.arange(n - 1) + 1
    src, dst = np.append(src, rng.choice(n - 2, hub, replace=False)), np.append(dst, np.full(hub, n - 1))
    return CFG(n, src.astype(np.int32), dst.astype(np.int32), rng.random(len(src)).astype(np.float32),
               rng.integers(0, 20, (n, 13)).astype(np.float32))


def test_long_lists_do_not_hold_the_sweep_up():
    """STOP blocks of 240 neighbours on both sides add 1.1 M terms to the 8.4 M
    entries, 57,600 of them at one entry: not one warp's or one thread's work
    while the others wait."""
    rng = np.random.default_rng(1)
    pk = api.Pack([chain(rng, n, hub) for hub in (0, 240) for n in (2000, 4200)], 13, device=DEV)
    om = torch.ones(13, device=DEV)

    def took(pair):
        best = 1e9
        for _ in range(4):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            api.similarity(pk, pk, [pair], om, want_x=True, want_scores=False)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        return best

    assert took((2, 3)) <= 8 * took((0, 1))
