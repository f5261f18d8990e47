"""Operands of one context in a call on another, whose stream is not ordered with theirs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["spamm", "combined", "truncate"])
@pytest.mark.parametrize("nb", [1, 2, 30])
def test_kept_tasks_while_the_owners_stream_is_busy(S, mode, nb):
    import torch
    owner_stream, stream = torch.cuda.Stream(), torch.cuda.Stream()
    owner, ctx = S.Context(0, stream=owner_stream), S.Context(0, stream=stream)
    rng = np.random.default_rng(nb)
    r, c = np.nonzero(np.ones((nb, nb)))
    A, B = (S.spamm_from_blocks(owner, nb * 32, 32, r.astype(np.int32), c.astype(np.int32),
                                rng.uniform(0.5, 1, (nb * nb, 32, 32)) * 10.0 ** rng.uniform(-3, 0, (nb * nb, 1, 1)))
            for _ in range(2))
    want = S.spamm_kept_tasks(owner, A, B, 0.1, mode)
    assert len(want) > 0
    with torch.cuda.stream(owner_stream):
        torch.cuda._sleep(100_000_000)  # some 50 ms
    assert np.array_equal(S.spamm_kept_tasks(ctx, A, B, 0.1, mode), want)
    owner_stream.synchronize()
