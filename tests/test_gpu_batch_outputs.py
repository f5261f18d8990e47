"""Batches whose outputs are finished together: outputs of one leaf, of some hundred, and
without leaves (first, between others, last) equal the same products run alone, leaves
and norms bit for bit."""
import ctypes

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


# to the host a product's leaves go straight from its pool, a truncated one's (fewer leaves, shared pool) are gathered
@pytest.mark.parametrize("bs", [32, 64])
def test_exports_to_host_and_device_agree(S, bs):
    import torch
    ctx = S.Context(0)
    nb = 9
    rng = np.random.default_rng(bs)
    r, c = np.nonzero(np.ones((nb, nb)))
    pay = rng.uniform(-1, 1, (len(r), bs, bs)) * 10.0 ** rng.uniform(-4, 0, (len(r), 1, 1))
    A = S.spamm_from_blocks(ctx, nb * bs, bs, r.astype(np.int32), c.astype(np.int32), pay)
    C = S.spamm_multiply(ctx, A, A, 0.0, "spamm")
    norms = np.sort(S.spamm_to_blocks(ctx, C)[3])
    for M in (A, C, S.spamm_truncate(ctx, C, float(np.sqrt(norms[len(norms) // 2]))), S.spamm_add(ctx, 1.0, C, 1.0, A)):
        n = M.info()["nleaves"]
        dev = [torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda"),
               torch.zeros(n, bs, bs, dtype=torch.float64, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda")]
        ptr = [ctypes.c_void_p(t.data_ptr()) for t in dev]
        assert S.load().spamm_to_blocks(ctx.handle, M.handle, *ptr, n, 1) == S.OK
        host = S.spamm_to_blocks(ctx, M)
        for x, y in zip(host, dev):
            assert np.array_equal(x, y.cpu().numpy())
        # norms to an address of four bytes' alignment
        raw = torch.zeros(8 * n + 8, dtype=torch.uint8, device="cuda")
        ptr[3] = ctypes.c_void_p(raw.data_ptr() + 4)
        assert S.load().spamm_to_blocks(ctx.handle, M.handle, *ptr, n, 1) == S.OK
        assert np.array_equal(raw.cpu().numpy()[4:4 + 8 * n].copy().view(np.float64), host[3])
