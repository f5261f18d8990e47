"""Allocators of the caller: addresses at 16-byte boundaries, between the 32-byte ones."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _context(S, alloc, free, stream=None):
    ctx = S.Context(0, stream=stream)
    ctx._callbacks = (S._ALLOC_T(alloc), S._FREE_T(free))
    S._check(ctx.handle, S.load().spamm_set_allocator(ctx.handle, *ctx._callbacks, ctypes.c_void_p(0)))
    return ctx


def _operands(S, ctx, nb, bs):
    rng = np.random.default_rng(nb)
    out = []
    for _ in range(2):
        r, c = np.nonzero(rng.random((nb, nb)) < 0.6)
        pay = rng.uniform(-1, 1, (len(r), bs, bs)) * 10.0 ** rng.uniform(-3, 0, (len(r), 1, 1))
        out.append(S.spamm_from_blocks(ctx, nb * bs, bs, r.astype(np.int32), c.astype(np.int32), pay))
    return out


@pytest.mark.parametrize("prec", ["fp64", "bf16_split", "bf16_split4", "fp16_scaled"])
@pytest.mark.parametrize("bs,nb", [(64, 2), (64, 21), (128, 7)])
def test_addresses_between_sectors(S, prec, bs, nb):
    import torch

    def alloc(nbytes, _user):
        p = torch.cuda.caching_allocator_alloc(int(nbytes) + 16, 0)
        assert p % 32 == 0
        return p + 16

    def free(p, _user):
        torch.cuda.caching_allocator_delete(p - 16)

    got = []
    for ctx in (S.Context(0), _context(S, alloc, free)):
        A, B = _operands(S, ctx, nb, bs)
        C = S.spamm_multiply(ctx, A, B, 1e-4, "combined", prec)
        plan = S.spamm_plan_create(ctx, B, A, 1e-4, "spamm", prec)
        job = S.spamm_job_begin(ctx, plan)
        while job.info()["units_done"] < job.info()["units"]:
            S.spamm_run(ctx, [job], 3.0)
        D = S.spamm_job_finish(ctx, job)
        E = S.spamm_truncate(ctx, S.spamm_add(ctx, 2.0, C, -0.3, D), 1e-2, "error")
        got.append([S.spamm_to_blocks(ctx, M) for M in (A, C, D, E)] + [S.spamm_error(ctx, C, D), S.spamm_trace(ctx, C)])
    for x, y in zip(*got):
        assert np.all([np.array_equal(u, v) for u, v in zip(x, y)]) if isinstance(x, tuple) else x == y
