"""Long, thin pairs: with the longer side at 513 to 1,024 they fit a CTA of 1,024
threads (one column per thread) but none of 512, where they are global-class and
need a scratch slot -- in the workspace the library asks for, under the tunes of
512 threads and under the default configuration of small batches."""
import ctypes as C

import numpy as np
import pytest

from gen.cfg_grammar import CFG

B = pytest.importorskip("paper_1707_02423_gb300._binding")
api = pytest.importorskip("paper_1707_02423_gb300.api")
torch = pytest.importorskip("torch")

THIN = [(13, 994), (19, 755), (25, 684), (994, 13)]


def graph(rng, n):
    """A chain with a branch over one block at 15 % of the blocks."""
    skip = np.arange(0, max(n - 2, 0) * 15 // 100) * 6
    src = np.concatenate([np.arange(n - 1), skip]).astype(np.int32)
    dst = np.concatenate([np.arange(n - 1) + 1, skip + 2]).astype(np.int32)
    return CFG(n, src, dst, rng.random(len(src)).astype(np.float32), rng.integers(0, 20, (n, 13)).astype(np.float32))


def graphs(na, nb):
    rng = np.random.default_rng([na, nb])
    return [graph(rng, n) for n in (na, nb, 400, 1)]


def sized(pk, pairs, tune):
    return api.ws_size(pk, pk, np.ascontiguousarray(pairs, np.int32), B.params(tune=tune))


@pytest.mark.parametrize("na,nb", THIN)
def test_workspace_has_their_slots(na, nb):
    pk = api.Pack(graphs(na, nb), 13, device=None)
    slot = 4 * 3 * na * nb  # three matrices, and more
    for P in (1, 7, 300):
        fixed = sized(pk, [(3, 3)] * P, 1)
        assert sized(pk, [(0, 1)] * P, 1) == fixed  # 1,024 threads: one CTA holds them
        for tune in (0, 2, 182):
            assert sized(pk, [(0, 1)] * P, tune) >= fixed + min(P, 152) * slot, (P, tune)
    # sized without parameters: enough for the default call
    n = C.c_size_t(0)
    one = np.array([[0, 1]], np.int32)
    B.check(B.lib().cf_similarity_ws_size(pk.host_ptr, pk.host_ptr, one.ctypes.data, 1, None, C.byref(n)))
    assert n.value >= sized(pk, [(0, 1)], 0)


@pytest.mark.gpu
@pytest.mark.parametrize("tune", [0, 2])
@pytest.mark.parametrize("na,nb", THIN)
def test_calls(na, nb, tune):
    """Alone and beside a larger pair, in a workspace of the size asked for."""
    pk = api.Pack(graphs(na, nb), 13, device="cuda")
    om = torch.linspace(0.5, 1.5, 13, device="cuda")
    for pairs in ([(0, 1)], [(0, 1)] * 40 + [(2, 2), (1, 2), (2, 0)] + [(0, 1)] * 3):
        pairs = np.array(pairs, np.int32)
        ref = api.similarity(pk, pk, pairs, om, want_x=True, tune=1)
        for _ in range(2):
            r = api.similarity(pk, pk, pairs, om, want_x=True, tune=tune, ws=api.Workspace("cuda"))
            # either side is within 1e-5 of the exact X
            assert (r.X - ref.X).abs().max().item() <= 2e-5
    t, _ = api.autotune(pk, pk, pairs, om)  # every candidate finds its room
    assert 1 <= t <= 240
