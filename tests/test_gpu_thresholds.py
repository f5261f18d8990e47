"""A threshold of -0.0 (finite and >= 0, so accepted) means what 0 means: by every rule of
the truncation, in every builder and in every method of the product."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _same(S, ctx, X, Y):
    for x, y in zip(S.spamm_to_blocks(ctx, X), S.spamm_to_blocks(ctx, Y)):
        assert np.array_equal(x.view(np.uint64) if x.dtype == np.float64 else x,
                              y.view(np.uint64) if y.dtype == np.float64 else y)


def _input(bs):
    rng = np.random.default_rng(bs)
    r, c = np.nonzero(np.ones((5, 5)))
    pay = rng.uniform(-1, 1, (25, bs, bs)) * 10.0 ** rng.uniform(-300, 0, (25, 1, 1))  # squares underflow in some
    pay[rng.random(pay.shape) < 0.3] = 0.0
    pay[rng.random(pay.shape) < 0.1] = -0.0
    return 5 * bs, r.astype(np.int32), c.astype(np.int32), pay


@pytest.mark.parametrize("rule", ["block", "element", "error"])
@pytest.mark.parametrize("bs", [32, 64])
def test_truncations(S, rule, bs):
    ctx = S.Context(0)
    n, r, c, pay = _input(bs)
    A = S.spamm_from_blocks(ctx, n, bs, r, c, pay)
    T = S.spamm_truncate(ctx, A, -0.0, rule)
    _same(S, ctx, T, S.spamm_truncate(ctx, A, 0.0, rule))
    if rule != "error":  # nothing lies below 0 (the error rule drops leaves whose norm is 0)
        _same(S, ctx, T, A)


@pytest.mark.parametrize("rule", ["block", "element", "error"])
def test_builders(S, rule):
    import torch
    ctx = S.Context(0)
    n, r, c, pay = _input(32)
    dense = pay.reshape(5, 5, 32, 32).transpose(0, 2, 1, 3).reshape(n, n).copy()
    i, j = np.nonzero(dense)
    dev = [torch.from_numpy(x).cuda() for x in (r, c, pay)]
    p = synth.DecayParams(n=300, kind=synth.KIND_1D, alpha=0.5, seed=3)
    for build in (lambda t: S.spamm_from_blocks(ctx, n, 32, r, c, pay, t, rule),
                  lambda t: S.spamm_from_blocks(ctx, n, 32, *dev, t, rule),
                  lambda t: S.spamm_from_dense(ctx, dense, 32, t, rule),
                  lambda t: S.spamm_from_coo(ctx, n, i, j, dense[i, j], 32, t, rule),
                  lambda t: S.spamm_generate(ctx, p, 32, t, rule)):
        _same(S, ctx, build(-0.0), build(0.0))


@pytest.mark.parametrize("mode", ["spamm", "combined", "truncate"])
def test_products(S, mode):
    ctx = S.Context(0)
    n, r, c, pay = _input(64)
    A = S.spamm_from_blocks(ctx, n, 64, r, c, pay)
    assert np.array_equal(S.spamm_kept_tasks(ctx, A, A, -0.0, mode), S.spamm_kept_tasks(ctx, A, A, 0.0, mode))
    for prec in ("fp64", "bf16_split4"):
        _same(S, ctx, S.spamm_multiply(ctx, A, A, -0.0, mode, prec), S.spamm_multiply(ctx, A, A, 0.0, mode, prec))
