"""Allocators of the caller: addresses at 16-byte boundaries, between the 32-byte ones, and
allocations that fail at every point of a call."""
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


# operands of another context on another stream: their owner may release them as soon as the call has returned
@pytest.mark.parametrize("call", ["multiply", "plan", "execute", "add", "truncate"])
def test_a_failed_call_leaves_nothing_in_flight(S, call):
    import torch
    count, limit = [0], [1 << 30]

    def alloc(nbytes, _user):
        count[0] += 1
        if count[0] > limit[0]:
            return None
        return torch.cuda.caching_allocator_alloc(int(nbytes), 0)

    def free(p, _user):
        torch.cuda.caching_allocator_delete(p)

    owner, stream = S.Context(0), torch.cuda.Stream()
    ctx = _context(S, alloc, free, stream)
    nb, bs = 40, 128
    rng = np.random.default_rng(1)
    r, c = np.nonzero(np.ones((nb, nb)))
    A = S.spamm_from_blocks(owner, nb * bs, bs, r.astype(np.int32), c.astype(np.int32),
                            rng.uniform(-1, 1, (nb * nb, bs, bs)))
    mine = S.spamm_from_blocks(ctx, nb * bs, bs, r[:9].astype(np.int32), c[:9].astype(np.int32),
                               rng.uniform(-1, 1, (9, bs, bs)))
    plan = S.spamm_plan_create(ctx, A, A, 0.0, "combined", "bf16_split4")
    run = {"multiply": lambda: S.spamm_multiply(ctx, A, A, 0.0, "combined", "bf16_split4"),
           "plan": lambda: S.spamm_plan_create(ctx, A, A, 0.0, "combined", "bf16_split4"),
           "execute": lambda: S.spamm_execute(ctx, [plan, plan]),
           "add": lambda: S.spamm_add(ctx, 2.0, A, -0.3, A),
           "truncate": lambda: S.spamm_truncate(ctx, mine, 1.0, "element")}[call]
    done = None
    for k in range(200):
        count[0], limit[0] = 0, k
        try:
            done = run()
            break
        except S.SpammError as e:
            assert stream.query()  # nothing of the call is left on its stream
            assert e.status == S.E_OOM
    assert done is not None and k > 3


def test_failed_calls_give_everything_back(S):
    """Every builder, truncation and product, with each of its allocations failing in turn, and inputs refused for
    what they hold: what the allocator handed out during the call has come back."""
    import torch
    import synth
    count, limit, live = [0], [1 << 30], set()

    def alloc(nbytes, _user):
        count[0] += 1
        if count[0] > limit[0]:
            return None
        p = torch.cuda.caching_allocator_alloc(int(nbytes), 0)
        live.add(p)
        return p

    def free(p, _user):
        live.remove(p)
        torch.cuda.caching_allocator_delete(p)

    ctx = _context(S, alloc, free)
    n, bs = 640, 64
    A, B = _operands(S, ctx, 10, bs)
    r, c, pay, _ = S.spamm_to_blocks(ctx, A)
    dense = S.spamm_to_dense(ctx, A)
    i, j = (x[:500] for x in np.nonzero(dense))
    bad = pay.copy()
    bad[3, 5, 7] = np.nan
    bad_dense = dense.copy()
    bad_dense[9, 9] = np.inf
    gen = synth.DecayParams(n=n, kind=synth.KIND_1D, alpha=0.5, seed=3)
    calls = [lambda: S.spamm_from_blocks(ctx, n, bs, r, c, pay, 1e-3, "error"),
             lambda: S.spamm_from_dense(ctx, dense, bs),
             lambda: S.spamm_from_coo(ctx, n, i, j, dense[i, j], bs, 1e-6, "block"),
             lambda: S.spamm_generate(ctx, gen, bs),
             lambda: S.spamm_identity(ctx, n, bs),
             lambda: S.spamm_add(ctx, 2.0, A, -1.0, B),
             lambda: S.spamm_kept_tasks(ctx, A, B, 1e-3, "combined")]
    calls += [lambda rule=rule: S.spamm_truncate(ctx, A, 0.1, rule) for rule in S.RULES]
    calls += [lambda prec=prec: S.spamm_multiply(ctx, A, B, 1e-3, "combined", prec) for prec in S.PRECS]
    refused = [lambda: S.spamm_from_blocks(ctx, n, bs, r, c, bad), lambda: S.spamm_from_dense(ctx, bad_dense, bs),
               lambda: S.spamm_from_blocks(ctx, n, bs, np.append(r, r[0]), np.append(c, c[0]), pay[[*range(len(r)), 0]]),
               lambda: S.spamm_from_blocks(ctx, n, bs, r + 1, c, pay),
               lambda: S.spamm_from_coo(ctx, n, i, j, np.full(len(i), np.nan), bs),
               lambda: S.spamm_add(ctx, 1e200, S.spamm_add(ctx, 1e200, A, 0.0, B), 1.0, B)]
    before = set(live)
    for call in calls:
        for k in range(300):
            count[0], limit[0] = 0, k
            try:
                call()
                break
            except S.SpammError as e:
                assert e.status == S.E_OOM
                assert live == before
        assert k > 0 and live == before  # the result has been released
    limit[0] = 1 << 30
    for call in refused:
        with pytest.raises(S.SpammError) as e:
            call()
        assert e.value.status in (S.E_NONFINITE, S.E_INVALID_ARG)
        del e
        assert live == before
