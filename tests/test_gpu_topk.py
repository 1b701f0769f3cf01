"""cf_topk against a stable sort: the forms of its selection (groups of a warp
down to one thread, too few groups, too many candidates), ties, rows of few
and of many columns, infinities and NaN."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
api = pytest.importorskip("paper_1707_02423_gb300.api")
DEV = "cuda"


def order_key(v):
    """Unsigned order of the float's bits: -NaN < -inf < ... < inf < NaN."""
    u = v.view(np.uint32).astype(np.int64)
    return np.where(u & 0x80000000, 0xffffffff - u, u + 0x80000000)


def check(s, k):
    top, idx = api.topk(torch.from_numpy(s).to(DEV), k)
    top, idx = top.cpu().numpy(), idx.cpu().numpy()
    for q in range(len(s)):
        ref = np.lexsort((np.arange(s.shape[1]), -order_key(s[q])))[:k]
        assert np.array_equal(idx[q], ref)
        assert np.array_equal(top[q].view(np.uint32), s[q][ref].view(np.uint32))


@pytest.mark.parametrize("C", [1, 7, 255, 256, 613, 2048, 2049, 8193, 40000])
@pytest.mark.parametrize("k", [1, 5, 6, 16, 21, 22, 64, 170, 171, 600, 1024])
def test_values(C, k):
    if k > C:
        pytest.skip("k > C")
    rng = np.random.default_rng(C * 2000 + k)
    check(rng.standard_normal((3, C)).astype(np.float32), k)
    check(rng.integers(0, 5, (2, C)).astype(np.float32), k)


@pytest.mark.parametrize("C", [613, 5000, 40000])
@pytest.mark.parametrize("k", [16, 40])
def test_crowded_rows(C, k):
    # the best elements in one thread's columns, one warp's, ascending, all equal
    n = 256 if C <= 2048 else 1024
    c = np.arange(C)
    rows = [np.where(c % n == 3, 2.0, 1.0) + c * 1e-6, np.where(c % n < 32, 2.0, 1.0) - c * 1e-6, c * 1.0, c * 0.0]
    check(np.stack(rows).astype(np.float32), k)


def test_not_finite():
    rng = np.random.default_rng(3)
    s = rng.standard_normal((2, 3000)).astype(np.float32)
    s[0, ::7] = np.nan
    s[0, 1::7] = -np.nan
    s[0, 2::7] = np.inf
    s[1] = -np.inf
    s[1, 5] = -0.0
    s[1, 9] = 0.0
    check(s, 500)
