"""Scattered leaf sets at the edges of what the tree kernels take at a time (groups of 32
nodes, pieces of one block, tiles): many levels, most parents with one child.  Codes and norms of
every level; the child links by a product with the identity, whose descent reaches
every leaf once."""
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


def _codes(r, c):
    m = np.zeros(len(r), np.int64)
    for b in range(16):
        m |= (((r >> b) & 1) << (2 * b + 1)) | (((c >> b) & 1) << (2 * b))
    return m


@pytest.mark.parametrize("count,nb", [(1, 1), (1, 700), (2, 2), (31, 6), (32, 40), (33, 1000), (1023, 32), (1024, 2000),
                                      (1025, 90), (4095, 64), (4096, 64), (4096, 3000), (4097, 65), (9000, 700),
                                      (32767, 1000), (32768, 3000), (32769, 400)])
def test_levels_of_scattered_leaves(S, count, nb):
    ctx = S.Context(0)
    bs, n = 32, 32 * nb
    rng = np.random.default_rng(count + nb)
    at = rng.choice(nb * nb, count, replace=False)
    r, c = at // nb, at % nb
    val = 10.0 ** rng.uniform(-4, 0, count)
    pay = np.zeros((count, bs, bs))
    pay[:, 3, 5] = val
    M = S.spamm_from_blocks(ctx, n, bs, r.astype(np.int32), c.astype(np.int32), pay)

    def check(M, r, c, sq):
        code = _codes(r, c)
        o = np.argsort(code)
        code, sq = code[o], sq[o]
        for t in range(M.info()["levels"], -1, -1):
            got, norm = S.spamm_level_norms(ctx, M, t)
            assert np.array_equal(got.astype(np.int64), code), t
            assert np.allclose(norm, sq, rtol=1e-14, atol=0.0), t
            code, up = np.unique(code >> 2, return_inverse=True)
            sq = np.bincount(up, weights=sq, minlength=len(code))
        kept = S.spamm_kept_tasks(ctx, M, S.spamm_identity(ctx, n, bs), 0.0, "spamm")
        assert len(kept) == len(r) and np.all(kept[:, 1] == kept[:, 2])
        assert np.array_equal(np.sort(kept[:, 0] * nb + kept[:, 2]), np.sort(r * nb + c))

    check(M, r, c, val ** 2)
    keep = ~(np.sqrt(val ** 2) < 0.01)
    if keep.any():
        check(S.spamm_truncate(ctx, M, 0.01), r[keep], c[keep], val[keep] ** 2)
