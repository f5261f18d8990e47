"""The tensor-core products at the edges of what their kernels batch: operand tiles
beside a whole number of tiles per thread block, and output quads of 1 to 20 steps, so
that a block's queue of steps and scales is cut at every place.  Whole numbers small
enough for every form: the results are exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TC = ["bf16_split", "bf16_split4", "fp16_scaled"]


@pytest.fixture(scope="module")
def S():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1906_08148_gb300 import spamm
    return spamm


def _leaves(S, ctx, n, M, bs, keep=None):
    """The leaves of M (all, or those of the boolean grid keep) as a quadtree."""
    R, K = M.shape[0] // bs, M.shape[1] // bs
    r, k = np.nonzero(np.ones((R, K), bool) if keep is None else keep)
    pay = M.reshape(R, bs, K, bs).transpose(0, 2, 1, 3)[r, k]
    return S.spamm_from_blocks(ctx, n, bs, r.astype(np.int32), k.astype(np.int32), np.ascontiguousarray(pay))


def _dense(S, ctx, C, bs, shape):
    out = np.zeros(shape)
    for r, c, p in zip(*S.spamm_to_blocks(ctx, C)[:3]):
        out[r * bs:(r + 1) * bs, c * bs:(c + 1) * bs] = p
    return out


# 64: two blocks per multiprocessor, both operands' tiles in one launch; 128: four tiles per leaf
@pytest.mark.parametrize("prec", TC)
@pytest.mark.parametrize("bs,count", [(64, 1), (64, 303), (64, 304), (64, 305), (64, 609), (64, 913), (128, 1),
                                      (128, 113), (128, 114), (128, 115), (128, 229), (128, 343)])
def test_operand_tiles_per_block(S, prec, bs, count):
    ctx = S.Context(0)
    rng = np.random.default_rng(count)
    A = rng.integers(-4, 5, (bs, bs * count)).astype(np.float64)
    B = rng.integers(-4, 5, (bs * count, bs)).astype(np.float64)
    n = bs * count
    C = S.spamm_multiply(ctx, _leaves(S, ctx, n, A, bs), _leaves(S, ctx, n, B, bs), 0.0, "spamm", prec)
    # |sum| <= 16 n < 2^24: exact in FP32, and so is every step on the way
    assert np.array_equal(_dense(S, ctx, C, bs, (bs, bs)), A @ B)


@pytest.mark.parametrize("prec", TC)
def test_quads_of_1_to_20_steps(S, prec):
    ctx = S.Context(0)
    bs, K = 64, 20
    rng = np.random.default_rng(20)
    keep = np.arange(K)[None, :] <= np.arange(2 * K)[:, None] // 2  # leaf rows 2 l, 2 l + 1: l + 1 leaves
    A = rng.integers(-4, 5, (2 * K * bs, K * bs)) * np.kron(keep, np.ones((bs, bs), int)).astype(np.float64)
    B = rng.integers(-4, 5, (K * bs, 39 * bs)).astype(np.float64)  # the last quads have one column of leaves
    n = 2 * K * bs
    C = S.spamm_multiply(ctx, _leaves(S, ctx, n, A, bs, keep), _leaves(S, ctx, n, B, bs), 0.0, "spamm", prec)
    assert np.array_equal(_dense(S, ctx, C, bs, (n, 39 * bs)), A @ B)
