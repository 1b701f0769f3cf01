"""The team tier: pairs beyond one CTA's shared memory on several CTAs, against
the FP64 oracle, at the sizes where its pieces meet: column chunks of 32 and
the warps that share them, row slabs and ring steps, team sizes by batch,
busy rows and columns, graphs too large to stage, ties in the matching."""
import numpy as np
import pytest
import torch

import oracle
from gen.cfg_grammar import CFG, structured_cfg
from _helpers import eps_greedy, greedy_margin, valid_matching

pytestmark = pytest.mark.gpu
api = pytest.importorskip("paper_1707_02423_gb300.api")
B = pytest.importorskip("paper_1707_02423_gb300._binding")
DEV = "cuda"
ATOL, TIE = 1e-5, 1e-6


def graph(rng, n, hubs=0):
    c = structured_cfg(rng, n, 6, 12)
    if not hubs:
        return c
    src, dst, w = [c.src], [c.dst], [c.w]
    for h in rng.choice(n, hubs, replace=False):
        k = min(n, 40)
        src.append(rng.choice(n, k, replace=False).astype(np.int32))
        dst.append(np.full(k, h, np.int32))
        w.append(rng.random(k).astype(np.float32))
    return CFG(n, np.concatenate(src), np.concatenate(dst), np.concatenate(w), c.attr)


def check(cfgs, pairs, sample=None, alpha=0.8, K=40, norm=None):
    pairs = np.asarray(pairs, np.int32)
    pk = api.Pack(cfgs, 13, device=DEV)
    om = torch.linspace(0.5, 1.5, 13, device=DEV)
    kw = {} if norm is None else {"norm_mode": norm}
    r = api.similarity(pk, pk, pairs, om, alpha, K, want_x=True, want_match=True, **kw)
    X, sc, mt = r.X.cpu().numpy(), r.scores.cpu().numpy(), r.match.cpu().numpy()
    for p in range(len(pairs)) if sample is None else sample:
        a, b = cfgs[pairs[p][0]], cfgs[pairs[p][1]]
        ref = oracle.similarity(a, b, om.cpu().numpy(), alpha, K, normalize=norm is None)["X"]
        got = X[r.x_off[p]:r.x_off[p + 1]].reshape(ref.shape)
        assert np.abs(got - ref).max() <= ATOL, (a.n, b.n, np.abs(got - ref).max())
        m = mt[r.m_off[p]:r.m_off[p + 1]]
        assert valid_matching(m, *ref.shape)
        if greedy_margin(ref) > TIE:
            m_ref, s_ref = oracle.greedy_match(ref)
            assert np.array_equal(m, m_ref)
            assert abs(float(sc[p]) - s_ref) <= ATOL
        else:
            assert eps_greedy(got, ref, m, 2 * ATOL)


# one column short of a chunk, on it and past it; one warp per row up to all of
# them; more columns than the consumer warps own at four chunks each; slabs of
# few and of many rows
@pytest.mark.parametrize("na,nb", [(700, 31), (640, 33), (500, 64), (333, 97), (150, 150), (130, 257), (60, 513),
                                   (33, 1025), (19, 2049), (9, 4000), (2600, 17), (137, 140)])
def test_shapes(na, nb):
    rng = np.random.default_rng([na, nb])
    check([graph(rng, na), graph(rng, nb)], [(0, 1)])


@pytest.mark.parametrize("ha,hb", [(3, 0), (0, 3), (2, 40), (40, 2)])
def test_busy_rows_and_columns(ha, hb):
    rng = np.random.default_rng([ha, hb])
    check([graph(rng, 210, ha), graph(rng, 190, hb)], [(0, 1), (1, 0)])


@pytest.mark.parametrize("n", [2, 7, 40, 170])
def test_batches(n):
    """As many pairs as teams of half the grid down to single CTAs."""
    rng = np.random.default_rng(n)
    cfgs = [graph(rng, int(k)) for k in rng.integers(140, 230, 6)]
    pairs = [(i % 6, (i * 5 + 1) % 6) for i in range(n)]
    check(cfgs, pairs, sample=sorted({0, 1, n // 2, n - 1}))


@pytest.mark.parametrize("K,norm", [(0, None), (1, None), (2, None), (5, 1), (70, None)])
def test_iterations(K, norm):
    rng = np.random.default_rng(K)
    check([graph(rng, 180), graph(rng, 161)], [(0, 1)], K=K, norm=norm)


@pytest.mark.parametrize("na,nb", [(300, 260), (260, 300), (1200, 30)])
def test_all_entries_tied(na, nb):
    """No edges, equal attributes: every entry is equal, and greedy's order
    (row, then column) pairs block i with block i."""
    z = np.zeros(0, np.int32)
    cfgs = [CFG(n, z, z, np.zeros(0, np.float32), np.ones((n, 13), np.float32)) for n in (na, nb)]
    pk = api.Pack(cfgs, 13, device=DEV)
    r = api.similarity(pk, pk, [(0, 1)], torch.ones(13, device=DEV), want_match=True)
    m = r.match.cpu().numpy()
    want = np.where(np.arange(na) < nb, np.arange(na), -1)
    assert np.array_equal(m, want)
    assert abs(float(r.scores[0]) - min(na, nb) / np.sqrt(na * nb)) <= ATOL * min(na, nb)


def test_replay_under_a_graph():
    """The cooperative kernel in a captured graph: replays give the same bits."""
    rng = np.random.default_rng(5)
    cfgs = [graph(rng, n) for n in (200, 180, 20, 30)]
    pairs = np.array([(0, 1), (1, 0), (2, 3), (0, 3)], np.int32)
    pk = api.Pack(cfgs, 13, device=DEV)
    om = torch.ones(13, device=DEV)
    first = api.similarity(pk, pk, pairs, om, want_match=True)
    ws, dp = api.Workspace(DEV), torch.from_numpy(pairs).to(DEV)
    nbytes = api.ws_size(pk, pk, pairs, B.params())
    ws.get(nbytes)
    out = {"scores": torch.zeros(4, device=DEV), "match": torch.zeros_like(first.match)}
    g = api.Graph()
    with g.capture():
        api.similarity(pk, pk, pairs, om, want_match=True, d_pairs=dp, out=out, ws=ws, ws_bytes=nbytes,
                       check_status=False)
    for _ in range(3):
        out["scores"].zero_()
        g.launch()
        torch.cuda.synchronize()
        assert torch.equal(out["scores"], first.scores) and torch.equal(out["match"], first.match)
