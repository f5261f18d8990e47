"""Errors and traces over leaf counts at the edges of the sum's tiles (4096 leaves): whole
numbers, so the sums are exact in any order, and leaves that only one of the two
matrices has."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1906_08148_gb300 import spamm
    return spamm


@pytest.mark.parametrize("nx,ny,common", [(1, 1, 1), (1, 1, 0), (3, 0, 0), (0, 3, 0), (4095, 17, 17), (4096, 4097, 4000),
                                          (4097, 4096, 1), (8192, 8193, 100), (20000, 12289, 5000)])
def test_error_of_partly_shared_leaves(S, nx, ny, common):
    ctx = S.Context(0)
    bs, nb = 32, 200
    rng = np.random.default_rng(nx + ny)
    at = rng.choice(nb * nb, nx + ny - common, replace=False)
    sets, vals = (at[:nx], np.concatenate([at[:common], at[nx:]])), []
    mats = []
    for a in sets:
        v = rng.integers(1, 100, len(a)).astype(np.float64)
        pay = np.zeros((len(a), bs, bs))
        pay[:, 7, 7] = v
        vals.append(dict(zip(a.tolist(), v)))
        mats.append(S.spamm_from_blocks(ctx, nb * bs, bs, (a // nb).astype(np.int32), (a % nb).astype(np.int32), pay))
    want = sum((vals[0].get(k, 0.0) - vals[1].get(k, 0.0)) ** 2 for k in set(vals[0]) | set(vals[1]))
    for _ in range(2):  # the counters are left as they were
        assert S.spamm_error(ctx, *mats) == np.sqrt(want)
        for M, v in zip(mats, vals):
            assert S.spamm_trace(ctx, M) == sum(x for k, x in v.items() if k // nb == k % nb)
