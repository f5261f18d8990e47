"""The leaf norms of FP64 outputs: one launch for a batch, whatever its size, and for every
leaf the bits that a matrix built from the finished leaves stores."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _diagonal(S, ctx, nb, bs, rng):
    at = np.arange(nb, dtype=np.int32)
    return S.spamm_from_blocks(ctx, nb * bs, bs, at, at, rng.uniform(-1, 1, (nb, bs, bs)))


def test_launches_do_not_grow_with_the_batch(S):
    ctx = S.Context(0)
    rng = np.random.default_rng(1)
    plans = []
    for _ in range(9):
        A, B = _diagonal(S, ctx, 3, 32, rng), _diagonal(S, ctx, 3, 32, rng)
        plans.append(S.spamm_plan_create(ctx, A, B, 0.0, "spamm", "fp64"))
    few = S.spamm_execute(ctx, plans[:2], stats=True)[1][0]["n_launches"]
    assert S.spamm_execute(ctx, plans, stats=True)[1][0]["n_launches"] == few


# one leaf, a few, more than the GPU holds at once; 0: no leaves
@pytest.mark.parametrize("bs,counts", [(32, (1,)), (32, (0, 607)), (32, (600, 0, 9)), (32, (2000, 1, 3000)),
                                       (64, (3, 1)), (64, (700, 5)), (128, (2, 1)), (128, (300, 309)), (256, (1, 3)),
                                       (256, (100,))])
@pytest.mark.parametrize("graph", [0, 1])
def test_norms_of_every_output(S, bs, counts, graph):
    ctx = S.Context(0)
    S._check(ctx.handle, S.load().spamm_set_exec_graph(ctx.handle, graph))
    rng = np.random.default_rng(bs)
    plans = []
    for nb in counts:
        if nb:
            A, B = _diagonal(S, ctx, nb, bs, rng), _diagonal(S, ctx, nb, bs, rng)
        else:  # operands that do not meet
            one = rng.uniform(-1, 1, (1, bs, bs))
            A = S.spamm_from_blocks(ctx, 2 * bs, bs, np.zeros(1, np.int32), np.ones(1, np.int32), one)
            B = S.spamm_from_blocks(ctx, 2 * bs, bs, np.zeros(1, np.int32), np.zeros(1, np.int32), one)
        plans.append(S.spamm_plan_create(ctx, A, B, 0.0, "spamm", "fp64"))
    for C, nb in zip(S.spamm_execute(ctx, plans), counts):
        bi, bj, pay, sq = S.spamm_to_blocks(ctx, C)
        assert np.array_equal(bi, np.arange(nb)) and np.array_equal(bj, np.arange(nb))
        if nb:
            again = S.spamm_from_blocks(ctx, nb * bs, bs, bi, bj, pay)
            assert np.array_equal(S.spamm_to_blocks(ctx, again)[3], sq)
            for t in range(C.info()["levels"] + 1):
                assert all(np.array_equal(x, y)
                           for x, y in zip(S.spamm_level_norms(ctx, C, t), S.spamm_level_norms(ctx, again, t)))
