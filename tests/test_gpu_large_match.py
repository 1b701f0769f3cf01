"""Greedy matching of matrices on either side of the sizes up to which the team
tier keeps the rows' best values in registers (5,120 rows) and the columns'
numbers in shared memory (10,616 columns)."""
import time

import numpy as np
import pytest
import torch

from gen.cfg_grammar import CFG

pytestmark = pytest.mark.gpu
api = pytest.importorskip("paper_1707_02423_gb300.api")
DEV = "cuda"


def pack(sizes):
    z = np.zeros(0, np.int32)
    return api.Pack([CFG(n, z, z, z.astype(np.float32), np.ones((n, 4), np.float32)) for n in sizes], 4, device=DEV)


def greedy(x):
    """Largest entry first (ties: smaller row, then smaller column), by sorting."""
    na, nb = x.shape
    order = np.argsort(-x.ravel(), kind="stable")
    row, col = np.zeros(na, bool), np.zeros(nb, bool)
    m, left, at, step = np.full(na, -1, np.int32), min(na, nb), 0, 1 << 12
    while left:
        q = order[at:at + step]
        at += step
        while left:
            q = q[~row[q // nb] & ~col[q % nb]]
            if not len(q):
                break
            i, j = divmod(int(q[0]), nb)
            row[i] = col[j] = True
            m[i] = j
            left -= 1
    return m


def near_rank_one(g, na, nb):
    u, v = torch.rand(na, 1, generator=g, device=DEV), torch.rand(1, nb, generator=g, device=DEV)
    return (u + 0.05) * (v + 0.05) * (1 + 0.01 * torch.rand(na, nb, generator=g, device=DEV))


@pytest.mark.parametrize("sizes", [[(5120, 400), (5121, 400)], [(60, 10616), (60, 10617)], [(8, 32000), (2, 16000)],
                                   [(5200, 10700)]])
@pytest.mark.parametrize("kind", ["rank one", "ties"])
def test_matchings(sizes, kind):
    g = torch.Generator(device=DEV).manual_seed(7)
    xs = [near_rank_one(g, *s) for s in sizes]
    if kind == "ties":
        xs = [torch.floor(16 * x) for x in xs]
    pk = pack([n for s in sizes for n in s])
    pairs = np.arange(2 * len(sizes), dtype=np.int32).reshape(-1, 2)
    r = api.match(pk, pk, pairs, torch.cat([x.flatten() for x in xs]))
    mt, sc = r.match.cpu().numpy(), r.scores.cpu().numpy()
    for p, x in enumerate(xs):
        x = x.cpu().numpy()
        m = greedy(x)
        assert np.array_equal(mt[r.m_off[p]:r.m_off[p + 1]], m)
        k = np.flatnonzero(m >= 0)
        s = x[k, m[k]].astype(np.float64).sum()
        # a term passes at most 64 additions (32,000 rows by 512 threads, the warp, the CTA, the team)
        assert abs(float(sc[p]) - s) <= 80 * 2.0 ** -24 * s


@pytest.mark.parametrize("below,above", [((5000, 5200), (5200, 5200)), ((100, 10600), (100, 10700))])
def test_no_cliff(below, above):
    """The team goes on with the matching past those sizes, and no CTA waits for
    another one's whole matching."""
    g = torch.Generator(device=DEV).manual_seed(8)
    took = []
    for s in (below, above):
        pk, x, best = pack(s), near_rank_one(g, *s).flatten(), 1e9
        for _ in range(3):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            api.match(pk, pk, [(0, 1)], x)
            best = min(best, time.perf_counter() - t0)
        took.append(best)
    print(f"\n  {below}: {1e3 * took[0]:.2f} ms, {above}: {1e3 * took[1]:.2f} ms")
    assert took[1] <= 3 * took[0]
