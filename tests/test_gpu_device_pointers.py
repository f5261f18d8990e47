"""Device pointers at any byte: spamm_from_blocks copied its arrays and so never asked for
more than memory that a copy can read."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _at(a, offset):
    """The bytes of `a` in device memory, `offset` bytes past a 256-byte boundary."""
    import torch
    raw = torch.zeros(a.nbytes + offset + 16, dtype=torch.uint8, device="cuda")
    raw[offset:offset + a.nbytes] = torch.from_numpy(a.reshape(-1).view(np.uint8).copy())
    assert raw.data_ptr() % 256 == 0
    return raw, ctypes.c_void_p(raw.data_ptr() + offset)


@pytest.mark.parametrize("offsets", [(0, 0, 0), (1, 0, 0), (0, 2, 0), (3, 1, 0), (4, 8, 8), (0, 0, 4), (2, 3, 1)])
@pytest.mark.parametrize("rule,tau", [("block", 0.0), ("element", 0.5)])
def test_from_blocks(S, offsets, rule, tau):
    ctx = S.Context(0)
    bs, nb = 32, 6
    rng = np.random.default_rng(3)
    p = rng.permutation(nb * nb)
    bi, bj = (p // nb).astype(np.int32), (p % nb).astype(np.int32)
    pay = rng.uniform(-1, 1, (nb * nb, bs, bs))
    kept = [_at(a, o) for a, o in zip((bi, bj, pay), offsets)]
    out = ctypes.c_void_p()
    S._check(ctx.handle, S.load().spamm_from_blocks(ctx.handle, nb * bs, bs, nb * nb, kept[0][1], kept[1][1], kept[2][1],
                                                    1, tau, S.RULES[rule], ctypes.byref(out)))
    want = S.spamm_from_blocks(ctx, nb * bs, bs, bi, bj, pay, tau, rule)
    for x, y in zip(S.spamm_to_blocks(ctx, S.Matrix(ctx, out)), S.spamm_to_blocks(ctx, want)):
        assert np.array_equal(x, y)
