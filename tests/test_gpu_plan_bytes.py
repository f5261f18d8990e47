"""spamm_plan_info's plan_bytes against the device memory that the context's allocator
hands out for the plan: requests are admitted by it."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture
def counted(S):
    """A context on an allocator that counts, and its live bytes by address."""
    import torch
    live = {}

    def alloc(nbytes, _user):
        p = torch.cuda.caching_allocator_alloc(int(nbytes), 0)
        live[p] = int(nbytes)
        return p

    def free(p, _user):
        del live[p]
        torch.cuda.caching_allocator_delete(p)

    ctx = S.Context(0)
    ctx._callbacks = (S._ALLOC_T(alloc), S._FREE_T(free))
    S._check(ctx.handle, S.load().spamm_set_allocator(ctx.handle, *ctx._callbacks, ctypes.c_void_p(0)))
    return ctx, live


def _band(S, ctx, nb, width, bs, seed):
    rng = np.random.default_rng(seed)
    r, c = np.nonzero(np.abs(np.arange(nb)[:, None] - np.arange(nb)[None, :]) <= width)
    pay = np.zeros((len(r), bs, bs))
    pay[:, 1, 2] = 10.0 ** rng.uniform(-3, 0, len(r))
    return S.spamm_from_blocks(ctx, nb * bs, bs, r.astype(np.int32), c.astype(np.int32), pay)


# 33,000 candidates: the exact leaf count is waited for; else the tree has room for every candidate
@pytest.mark.parametrize("prec,bs,nb,width", [("fp64", 32, 1, 0), ("fp64", 32, 300, 20), ("fp64", 32, 1100, 15),
                                              ("fp64", 128, 12, 4), ("fp64", 256, 5, 1), ("fp16_scaled", 64, 60, 9),
                                              ("bf16_split", 128, 9, 3), ("bf16_split4", 64, 30, 29)])
@pytest.mark.parametrize("same", [False, True])
def test_plan_bytes_are_what_the_plan_holds(S, counted, prec, bs, nb, width, same):
    ctx, live = counted
    A = _band(S, ctx, nb, width, bs, 1)
    B = A if same else _band(S, ctx, nb, width, bs, 2)
    before = sum(live.values())
    plan = S.spamm_plan_create(ctx, A, B, 0.03, "combined", prec)
    assert plan.info()["plan_bytes"] == sum(live.values()) - before
    plan.close()
    assert sum(live.values()) == before
