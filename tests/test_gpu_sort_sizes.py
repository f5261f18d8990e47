"""The key sort at the edges of its forms (one block with four or sixteen rounds of 1024
pairs, tiles above): leaves in random order come back in Morton order with their own
payload, and the error-controlled rule, which sorts 64-bit norms, drops exactly the
smallest leaves."""
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


@pytest.mark.parametrize("count,nb", [(2, 2), (33, 9), (4095, 100), (4096, 2000), (4097, 64 + 1), (8193, 3000), (16383, 900), (16384, 130), (16385, 5000),
                                      (30000, 200), (65535, 300), (65536, 2500), (65537, 260)])
def test_sorted_leaves_and_smallest_dropped(S, count, nb):
    ctx = S.Context(0)
    bs = 32
    rng = np.random.default_rng(count)
    at = rng.permutation(rng.choice(nb * nb, count, replace=False))
    r, c = (at // nb).astype(np.int32), (at % nb).astype(np.int32)
    # squared norms: distinct whole numbers times 2^-40, so every partial sum is exact
    val = (rng.permutation(count) + 1).astype(np.float64) * 2.0 ** -20
    pay = np.zeros((count, bs, bs))
    pay[:, 0, 0] = val
    M = S.spamm_from_blocks(ctx, nb * bs, bs, r, c, pay)
    gr, gc, gp, _ = S.spamm_to_blocks(ctx, M)
    code = np.zeros(count, np.int64)
    for b in range(16):
        code |= (((gr.astype(np.int64) >> b) & 1) << (2 * b + 1)) | (((gc.astype(np.int64) >> b) & 1) << (2 * b))
    assert np.all(np.diff(code) > 0)
    value = dict(zip(at.tolist(), val))
    assert all(value[int(i) * nb + int(j)] == v for i, j, v in zip(gr, gc, gp[:, 0, 0]))
    order = np.sort(val)
    total = np.cumsum((order * 2.0 ** 20) ** 2)  # whole numbers below 2^53
    for drop in (1, count // 3, count - 1):
        tau = float(np.sqrt(total[drop - 1] + 0.5) * 2.0 ** -20) if drop else 0.0
        T = S.spamm_truncate(ctx, M, tau, "error")
        assert T.info()["nleaves"] == count - drop
        kept = S.spamm_to_blocks(ctx, T)[2][:, 0, 0]
        assert np.array_equal(np.sort(kept), order[drop:])
