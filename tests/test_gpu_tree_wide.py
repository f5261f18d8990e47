"""Trees of more than 1,048,576 candidates or nodes, whose tile counts are scanned (up to there
every tile of 1024 adds up the counts before it): codes and norms of every level."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _codes(r, c):
    m = np.zeros(len(r), np.int64)
    for b in range(16):
        m |= (((r >> b) & 1) << (2 * b + 1)) | (((c >> b) & 1) << (2 * b))
    return m


def _check(S, ctx, M, r, c, sq):
    code = _codes(r, c)
    o = np.argsort(code)
    code, sq = code[o], sq[o]
    for t in range(M.info()["levels"], -1, -1):
        got, norm = S.spamm_level_norms(ctx, M, t)
        assert np.array_equal(got.astype(np.int64), code), t
        assert np.allclose(norm, sq, rtol=1e-13, atol=0.0), t  # up to a million terms a node, pairwise
        code, up = np.unique(code >> 2, return_inverse=True)
        sq = np.bincount(up, weights=sq, minlength=len(code))


# leaf grids of 1024 and 2048 per side: 2^20 candidates (1024 tiles) and 2^22
@pytest.mark.parametrize("nb", [1024, 1025])
def test_many_candidates(S, nb):
    ctx = S.Context(0)
    bs, n = 32, 32 * nb - 7
    p = synth.DecayParams(n=n, kind=synth.KIND_1D, alpha=2.0, seed=5)
    M = S.spamm_generate(ctx, p, bs)
    r, c = np.nonzero(np.abs(np.arange(nb)[:, None] - np.arange(nb)[None, :]) <= 1)
    # exp(-2 d) >= 1e-16 up to d = 18: a diagonal leaf and its neighbours
    want = (synth.leaves(p, bs, r, c) ** 2).sum((1, 2))
    assert np.all(want > 0.0)
    _check(S, ctx, M, r, c, want)
    kept = S.spamm_kept_tasks(ctx, M, S.spamm_identity(ctx, n, bs), 0.0, "spamm")
    assert np.array_equal(np.sort(_codes(kept[:, 0].astype(np.int64), kept[:, 2].astype(np.int64))), np.sort(_codes(r, c)))


# 1,050,625 leaves: the levels above them in scanned tiles too, and the block rule over them
def test_many_leaves(S):
    import torch
    ctx = S.Context(0)
    bs, nb = 32, 1025
    rng = np.random.default_rng(2)
    r, c = np.divmod(np.arange(nb * nb), nb)
    val = 10.0 ** rng.uniform(-4, 0, nb * nb)
    pay = torch.zeros((nb * nb, bs, bs), dtype=torch.float64, device="cuda")
    pay[:, 3, 5] = torch.from_numpy(val).cuda()
    M = S.spamm_from_blocks(ctx, nb * bs, bs, torch.from_numpy(r.astype(np.int32)).cuda(),
                            torch.from_numpy(c.astype(np.int32)).cuda(), pay)
    del pay
    _check(S, ctx, M, r, c, val ** 2)
    for tau in (0.00011, 0.1):
        keep = ~(np.sqrt(val ** 2) < tau)
        _check(S, ctx, S.spamm_truncate(ctx, M, tau), r[keep], c[keep], val[keep] ** 2)
    torch.cuda.empty_cache()
    M.close()
    S.spamm_trim(ctx)
