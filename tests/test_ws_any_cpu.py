"""cf_similarity_ws_size_any bounds cf_similarity_ws_size for every pair list, the
default configuration's room for deferred steps (from 32 pairs per SM on)
included."""
import numpy as np
import pytest

from gen.cfg_grammar import structured_cfg

api = pytest.importorskip("paper_1707_02423_gb300.api")
B = pytest.importorskip("paper_1707_02423_gb300._binding")


@pytest.mark.parametrize("flags", [0, B.CF_FLAG_PER_PAIR_LAUNCH])
@pytest.mark.parametrize("tune", [0, 1, 2, 181, 182])
@pytest.mark.parametrize("P", [1, 152, 1217, 4863, 4864, 4865, 60000])
def test_bound(P, tune, flags):
    rng = np.random.default_rng(P)
    for sizes in ([4, 9, 20], [5, 40, 90], [30, 130, 400], [700, 994, 13]):
        pk = api.Pack([structured_cfg(rng, n, 4, 4) for n in sizes], 5, device=None)
        prm = B.params(tune=tune, flags=flags)
        bound = api.ws_size_any(pk, pk, P, prm)
        for pairs in (rng.integers(0, 3, (P, 2)), np.full((P, 2), int(np.argmax(sizes))), np.tile([[1, 2]], (P, 1))):
            assert api.ws_size(pk, pk, np.ascontiguousarray(pairs, dtype=np.int32), prm) <= bound
