"""Batches whose outputs are finished together: outputs of one leaf, of some hundred, and
without leaves (first, between others, last) equal the same products run alone, leaves
and norms bit for bit."""
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


@pytest.mark.parametrize("prec", ["fp16_scaled", "bf16_split", "bf16_split4", "fp64"])
@pytest.mark.parametrize("sides", [(1,), (0,), (0, 3), (3, 0, 9, 1, 0), (7, 1, 0, 0, 12, 2, 5, 1)])
def test_outputs_finished_together(S, prec, sides):
    ctx = S.Context(0)
    bs = 64
    rng = np.random.default_rng(len(sides))
    pairs = []
    for nb in sides:  # 0: operands that do not meet
        grid = max(nb, 2)
        mats = []
        for role in range(2):
            r, c = np.nonzero(np.ones((nb, nb))) if nb else (np.array([0]), np.array([role]))
            if nb == 0 and role == 1:
                r, c = np.array([0]), np.array([0])
            mats.append(S.spamm_from_blocks(ctx, grid * bs, bs, r.astype(np.int32),
                                            c.astype(np.int32) + (1 if nb == 0 and role == 0 else 0),
                                            rng.uniform(-1, 1, (len(r), bs, bs))))
        pairs.append(mats)
    plans = [S.spamm_plan_create(ctx, A, B, 0.0, "spamm", prec) for A, B in pairs]
    for C, (A, B), nb in zip(S.spamm_execute(ctx, plans), pairs, sides):
        alone = S.spamm_to_blocks(ctx, S.spamm_multiply(ctx, A, B, 0.0, "spamm", prec))
        got = S.spamm_to_blocks(ctx, C)
        assert len(got[0]) == nb * nb
        assert all(np.array_equal(x, y) for x, y in zip(got, alone))
