"""n_steps and executed_flops of a product from its kept set: 64 x 64 leaves take one step per quad
of output leaves and k, half as wide in the BF16 forms where the kept products lie in one
column of the quad; 128 x 128 leaves two whole steps per kept product; FP64 what is kept."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TERMS = {"bf16_split": 3, "bf16_split4": 4, "fp16_scaled": 2}


def _matrix(S, ctx, nb, bs, fill, seed):
    rng = np.random.default_rng(seed)
    r, c = np.nonzero(rng.random((nb, nb)) < fill)
    if len(r) == 0:
        r, c = np.zeros(1, np.int64), np.zeros(1, np.int64)
    pay = rng.uniform(-1, 1, (len(r), bs, bs)) * 10.0 ** rng.uniform(-4, 0, (len(r), 1, 1))
    return S.spamm_from_blocks(ctx, nb * bs, bs, r.astype(np.int32), c.astype(np.int32), pay)


@pytest.mark.parametrize("prec", ["fp64", "bf16_split", "bf16_split4", "fp16_scaled"])
@pytest.mark.parametrize("bs,nb,fill", [(64, 1, 1.0), (64, 2, 1.0), (64, 3, 0.7), (64, 5, 1.0), (64, 39, 0.3), (64, 80, 0.1),
                                        (128, 1, 1.0), (128, 6, 0.5)])
@pytest.mark.parametrize("tau", [0.0, 1.0])
def test_executed_flops(S, prec, bs, nb, fill, tau):
    ctx = S.Context(0)
    A, B = _matrix(S, ctx, nb, bs, fill, 1), _matrix(S, ctx, nb, bs, fill, 2)
    kept = S.spamm_kept_tasks(ctx, A, B, tau, "spamm")
    st = S.spamm_multiply(ctx, A, B, tau, "spamm", prec, stats=True)[1]
    assert st["n_kept"] == len(kept)
    if prec == "fp64":
        assert (st["n_steps"], st["executed_flops"]) == (len(kept), 2.0 * bs ** 3 * len(kept))
        return
    t = TERMS[prec]
    whole = t * (t + 1) // 2 * 2.0 * 128 * 128 * 64
    if bs == 128:
        assert (st["n_steps"], st["executed_flops"]) == (2 * len(kept), 2 * len(kept) * whole)
        return
    cols = {}
    for i, k, j in kept.tolist():
        cols.setdefault((i // 2, j // 2, k), set()).add(j % 2)
    half = 0 if prec == "fp16_scaled" else sum(len(x) == 1 for x in cols.values())
    assert (st["n_steps"], st["executed_flops"]) == (len(cols), (len(cols) - 0.5 * half) * whole)
