"""The FP64 leaf products on both sides of the rule that picks the tile (quarter tiles
for launches with few units per SM): every element is the same sum in the same order,
so a product of many leaves equals the products of its parts bit for bit, and the
stored leaf norms are those of the finished leaves."""
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


# three products per output leaf; many x many output leaves take the large tile
@pytest.mark.parametrize("bs,many", [(32, 70), (64, 70), (128, 34), (256, 20)])
def test_tile_does_not_change_results(S, bs, many):
    ctx = S.Context(0)
    rng = np.random.default_rng(bs)
    k = 3
    A = rng.uniform(-1, 1, (many, k, bs, bs))
    B = rng.uniform(-1, 1, (k, many, bs, bs))
    n = many * bs

    def product(rows, cols):
        ar, ak = np.meshgrid(rows, range(k), indexing="ij")
        bk, bc = np.meshgrid(range(k), cols, indexing="ij")
        GA = S.spamm_from_blocks(ctx, n, bs, ar.ravel().astype(np.int32), ak.ravel().astype(np.int32),
                                 A[rows].reshape(-1, bs, bs))
        GB = S.spamm_from_blocks(ctx, n, bs, bk.ravel().astype(np.int32), bc.ravel().astype(np.int32),
                                 B[:, cols].reshape(-1, bs, bs))
        return S.spamm_to_blocks(ctx, S.spamm_multiply(ctx, GA, GB, 0.0, "spamm"))

    whole = product(np.arange(many), np.arange(many))
    at = {(int(r), int(c)): q for q, (r, c) in enumerate(zip(whole[0], whole[1]))}
    assert len(at) == many * many
    for rows, cols in ((np.array([0, many - 1]), np.array([1])), (np.arange(5), np.arange(3, 9))):
        for r, c, p, s in zip(*product(rows, cols)):
            q = at[(int(r), int(c))]
            assert np.array_equal(p, whole[2][q]) and s == whole[3][q]
    again = S.spamm_to_blocks(ctx, S.spamm_from_blocks(ctx, n, bs, whole[0], whole[1], whole[2]))
    assert np.array_equal(again[3], whole[3])
    assert np.allclose(whole[2][at[(0, 1)]], sum(A[0, j] @ B[j, 1] for j in range(k)), rtol=1e-12, atol=1e-12)
