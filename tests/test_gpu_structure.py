"""Quadtree structure and task lists at the edges of the kernels that build them:
the one-block form (up to 32768 items) and the tiled form (2048 per tile), the
one-block steps of the descent (five levels) and the tiled ones (64 groups per
tile).  Leaf sets, codes, child counts and kept sets are compared exactly with the
oracle, norms with its sums (1e-14 relative, as for every stored norm)."""
import numpy as np
import pytest

import oracle

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


@pytest.fixture(scope="module")
def ctx(S):
    return S.Context(0)


def _band(nb, width, seed, fill=1.0, bs=32):
    """Leaves within `width` of the diagonal of an nb x nb grid, in random order, norms over four decades."""
    rng = np.random.default_rng(seed)
    bi, bj = np.nonzero(np.abs(np.arange(nb)[:, None] - np.arange(nb)[None, :]) <= width)
    if fill < 1.0:
        at = rng.random(len(bi)) < fill
        bi, bj = bi[at], bj[at]
    p = rng.permutation(len(bi))
    bi, bj = bi[p].astype(np.int32), bj[p].astype(np.int32)
    pay = np.zeros((len(bi), bs, bs))
    pay[:, 0, 0] = rng.choice([-1.0, 1.0], len(bi)) * 10.0 ** rng.uniform(-4, 0, len(bi))
    pay[:, bs - 1, 1] = rng.uniform(-1, 1, len(bi)) * pay[:, 0, 0]
    return bi, bj, pay


def _code(r, c):
    r, c = r.astype(np.uint64), c.astype(np.uint64)
    m = np.zeros_like(r)
    for b in range(16):
        m |= (((r >> np.uint64(b)) & np.uint64(1)) << np.uint64(2 * b + 1)) | (((c >> np.uint64(b)) & np.uint64(1))
                                                                              << np.uint64(2 * b))
    return m


def _check_levels(S, ctx, M, bi, bj, sq):
    """Every level of M against the codes and sums of its leaves."""
    L = M.info()["levels"]
    code = _code(bi, bj)
    o = np.argsort(code)
    code, sq = code[o], sq[o]
    for t in range(L, -1, -1):
        got_code, got_sq = S.spamm_level_norms(ctx, M, t)
        assert np.array_equal(got_code.astype(np.uint64), code), t
        assert np.allclose(got_sq, sq, rtol=1e-14, atol=0.0), t
        up = code >> np.uint64(2)
        code, at = np.unique(up, return_inverse=True)
        sq = np.bincount(at, weights=sq, minlength=len(code))


# leaves: 1, a full tile of the one-block form and one more, its largest size and one more, several tiles
@pytest.mark.parametrize("nb,width,fill", [(1, 0, 1.0), (2, 1, 1.0), (3, 2, 1.0), (64, 63, 1.0), (64, 63, 0.5),
                                           (65, 64, 1.0), (181, 180, 1.0), (182, 181, 1.0), (300, 299, 0.7),
                                           (3000, 6, 1.0)])
def test_levels_of_built_and_truncated_matrices(S, ctx, nb, width, fill):
    bi, bj, pay = _band(nb, width, 3, fill)
    M = S.spamm_from_blocks(ctx, nb * 32, 32, bi, bj, pay)
    sq = (pay ** 2).sum((1, 2))
    _check_levels(S, ctx, M, bi, bj, sq)
    for tau in (1e-3, 0.3, 10.0):
        T = S.spamm_truncate(ctx, M, tau)
        keep = ~(np.sqrt(sq) < tau)
        assert T.info()["nleaves"] == keep.sum()
        if keep.any():
            _check_levels(S, ctx, T, bi[keep], bj[keep], sq[keep])


# leaf grids of 2^0 .. 2^9 per side: no step, one-block steps only, and one to four tiled ones; full and banded
@pytest.mark.parametrize("nb,width", [(1, 0), (2, 1), (5, 4), (16, 15), (32, 31), (33, 32), (64, 20), (128, 6), (300, 4),
                                      (512, 2)])
@pytest.mark.parametrize("mode", ["spamm", "combined", "truncate"])
def test_kept_sets_at_every_depth(S, ctx, nb, width, mode):
    a, b = _band(nb, width, 5, 0.8 if nb > 2 else 1.0), _band(nb, width, 6, 0.9 if nb > 2 else 1.0)
    n = nb * 32
    GA, GB = S.spamm_from_blocks(ctx, n, 32, *a), S.spamm_from_blocks(ctx, n, 32, *b)
    MA, MB = oracle.from_leaves(n, 32, *a), oracle.from_leaves(n, 32, *b)
    for tau in (1e-5, 1e-2, 100.0):
        got = S.spamm_kept_tasks(ctx, GA, GB, tau, mode)
        At, Bt = (MA, MB) if mode == "spamm" else (oracle.truncate_block(MA, tau), oracle.truncate_block(MB, tau))
        want = np.asarray(oracle.kept_flat(At, Bt, tau, oracle.MODES[mode]), np.int32).reshape(-1, 3)
        key = lambda x: x[np.lexsort((x[:, 1], x[:, 2], x[:, 0]))]
        assert np.array_equal(key(got), key(want)), (tau, len(got), len(want))
        c = _code(got[:, 0], got[:, 2])
        assert np.all(np.diff(c.astype(np.int64)) >= 0)  # grouped by output leaf in Morton order
        same = np.diff(c.astype(np.int64)) == 0
        assert np.all(np.diff(got[:, 1])[same] > 0)  # k ascending within a group


# quad steps (written with the list) drive the tensor forms: integer inputs are exact
@pytest.mark.parametrize("nb,width", [(1, 0), (2, 1), (3, 2), (9, 3), (33, 2), (66, 1)])
@pytest.mark.parametrize("same", [False, True])
def test_quad_steps_at_every_depth(S, ctx, nb, width, same):
    def ints(seed):
        bi, bj, _ = _band(nb, width, seed, 0.8, 64)
        return bi, bj, np.random.default_rng(seed).integers(-15, 16, (len(bi), 64, 64)).astype(np.float64)
    a, b = ints(7), ints(8)
    n = nb * 64
    if len(a[0]) == 0 or len(b[0]) == 0:
        a = b = (np.zeros(1, np.int32), np.zeros(1, np.int32), np.ones((1, 64, 64)))
    if same:  # a symmetric X times itself: one set of terms serves both roles
        D = np.zeros((n, n))
        for r, c, p in zip(*a):
            D[r * 64:r * 64 + 64, c * 64:c * 64 + 64] = p
        D = np.tril(D) + np.tril(D, -1).T
        GA = S.spamm_from_dense(ctx, D, 64)
        GA.set_symmetric()
        C = S.spamm_to_dense(ctx, S.spamm_multiply(ctx, GA, GA, 0.0, "spamm", "bf16_split4"))
        assert np.array_equal(C, D @ D)
        return
    A, B = np.zeros((n, n)), np.zeros((n, n))
    for D, x in ((A, a), (B, b)):
        for r, c, p in zip(*x):
            D[r * 64:r * 64 + 64, c * 64:c * 64 + 64] = p
    GA, GB = S.spamm_from_blocks(ctx, n, 64, *a), S.spamm_from_blocks(ctx, n, 64, *b)
    C = S.spamm_to_dense(ctx, S.spamm_multiply(ctx, GA, GB, 0.0, "spamm", "bf16_split4"))
    assert np.array_equal(C, A @ B)
