"""The passes that make leaves with their norms (alpha X + beta Y, copies of device
leaves, the element rule) and the radix sort behind the builders and the
error-controlled truncation, at the edges of their forms.  Everything is compared bit
for bit: the sums are one rounded operation after the other in a fixed order."""
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


@pytest.fixture(scope="module")
def ctx(S):
    return S.Context(0)


def _values(rng, shape):
    """Doubles over the whole range an exact factor may shift, with zeros of both signs and subnormals."""
    v = rng.uniform(-1, 1, shape) * 2.0 ** rng.integers(-1060, 900, shape)
    v[rng.random(shape) < 0.2] = 0.0
    v[rng.random(shape) < 0.1] = -0.0
    return v


@pytest.mark.parametrize("alpha,beta", [(2.0, -1.0), (-4.0, 1.0), (1.0, 1.0), (-1.0, -1.0), (2.0, 0.3), (0.3, -2.0),
                                        (0.3, 1.0), (-1.0, 8.0), (0.5, -0.25), (0.7, 0.9), (0.0, 2.0), (2.0, 0.0)])
@pytest.mark.parametrize("bs", [32, 128])
def test_add_rounds_each_operation(S, ctx, alpha, beta, bs):
    rng = np.random.default_rng(11)
    where = {"both": (0, 0), "x": (0, 1), "y": (1, 0)}
    X, Y = _values(rng, (2, bs, bs)), _values(rng, (2, bs, bs))
    GX = S.spamm_from_blocks(ctx, 2 * bs, bs, [0, 0], [0, 1], X)
    GY = S.spamm_from_blocks(ctx, 2 * bs, bs, [0, 1], [0, 0], Y)
    C = S.spamm_add(ctx, alpha, GX, beta, GY)
    bi, bj, pay, sq = S.spamm_to_blocks(ctx, C)
    got = {(int(r), int(c)): (p, s) for r, c, p, s in zip(bi, bj, pay, sq)}
    zero = np.zeros((bs, bs))
    want = {where["both"]: alpha * X[0] + beta * Y[0], where["x"]: alpha * X[1] + zero, where["y"]: zero + beta * Y[1]}
    for at, w in want.items():
        if not np.any(w):
            assert at not in got
            continue
        assert np.array_equal(got[at][0].view(np.uint64), w.view(np.uint64)), at
    # the stored norms are those of the finished leaves built anew
    again = S.spamm_from_blocks(ctx, 2 * bs, bs, bi, bj, pay)
    assert np.array_equal(S.spamm_to_blocks(ctx, again)[3], sq)


@pytest.mark.parametrize("alpha,beta", [(2.0, -1.0), (1.0, -4.0), (0.7, 2.0)])
def test_add_refuses_overflow_of_one_product(S, ctx, alpha, beta):
    """The product overflows although the sum would not."""
    exact_x = alpha in (2.0, 4.0)
    X, Y = np.zeros((1, 32, 32)), np.zeros((1, 32, 32))
    big = 2.0 ** 1023 * 1.5
    if exact_x:
        X[0, 3, 5], Y[0, 3, 5] = big, big
    else:
        X[0, 3, 5], Y[0, 3, 5] = big * (1 if beta < 0 else -1), big
    # squares overflow in the norms of X and Y themselves, which is allowed: only elements must be finite
    GX, GY = S.spamm_from_blocks(ctx, 32, 32, [0], [0], X), S.spamm_from_blocks(ctx, 32, 32, [0], [0], Y)
    with np.errstate(over="ignore", invalid="ignore"):
        assert not np.isfinite((alpha * X + beta * Y)[0, 3, 5])
    with pytest.raises(S.SpammError) as e:
        S.spamm_add(ctx, alpha, GX, beta, GY)
    assert e.value.status == S.E_NONFINITE


@pytest.mark.parametrize("rule,tau", [("block", 0.0), ("element", 0.25)])
@pytest.mark.parametrize("offset", [0, 1])
def test_device_leaves_equal_host_leaves(S, ctx, rule, tau, offset):
    """Leaves on the device (copied in the norm pass; an address between 16-byte pairs takes the copy first)."""
    import torch
    rng = np.random.default_rng(5)
    nb, bs = 9, 64
    p = rng.permutation(nb * nb)
    bi, bj = (p // nb).astype(np.int32), (p % nb).astype(np.int32)
    pay = rng.uniform(-1, 1, (nb * nb, bs, bs))
    pay[4] = 0.0
    pay[5, 0, 0] = -0.0
    flat = torch.zeros(pay.size + 2, dtype=torch.float64, device="cuda")
    flat[offset:offset + pay.size] = torch.from_numpy(pay.ravel())
    dev = flat[offset:offset + pay.size].view(pay.shape)
    A = S.spamm_from_blocks(ctx, nb * bs, bs, bi, bj, pay, tau, rule)
    B = S.spamm_from_blocks(ctx, nb * bs, bs, torch.from_numpy(bi).cuda(), torch.from_numpy(bj).cuda(), dev, tau, rule)
    for x, y in zip(S.spamm_to_blocks(ctx, A), S.spamm_to_blocks(ctx, B)):
        assert np.array_equal(x.view(np.uint64) if x.dtype == np.float64 else x,
                              y.view(np.uint64) if y.dtype == np.float64 else y)


# one round of one warp, one item more, the largest one-block sort, one more, several tiles
@pytest.mark.parametrize("nnz", [1, 32, 33, 1024, 4096, 4097, 16384, 16385, 50000])
def test_coo_sums_duplicates_in_input_order(S, ctx, nnz):
    rng = np.random.default_rng(nnz)
    n, bs = 5000, 32
    row = rng.integers(0, 40, nnz) * 125
    col = np.minimum(row + rng.integers(0, 6, nnz), n - 1)
    val = rng.uniform(-1, 1, nnz) * 10.0 ** rng.integers(-8, 8, nnz)  # the order of a sum shows in its bits
    M = S.spamm_from_coo(ctx, n, row, col, val, bs)
    bi, bj, pay, _ = S.spamm_to_blocks(ctx, M)
    want = {}
    for r, c, v in zip(row, col, val):
        want[(r, c)] = want.get((r, c), 0.0) + v
    got = {}
    for r, c, p in zip(bi, bj, pay):
        for i, j in zip(*np.nonzero(p)):
            got[(r * bs + i, c * bs + j)] = p[i, j]
    assert got == {k: v for k, v in want.items() if v != 0.0}


@pytest.mark.parametrize("nb,width", [(1, 0), (20, 19), (128, 127), (129, 128), (2000, 12)])
def test_error_controlled_truncation_drops_the_smallest(S, ctx, nb, width):
    rng = np.random.default_rng(nb)
    bi, bj = np.nonzero(np.abs(np.arange(nb)[:, None] - np.arange(nb)[None, :]) <= width)
    pay = np.zeros((len(bi), 32, 32))
    pay[:, 1, 1] = 2.0 ** rng.integers(-20, 20, len(bi))  # squares and their sums are exact, ties are common
    code = np.zeros(len(bi), np.int64)
    for b in range(12):
        code |= (((bi >> b) & 1) << (2 * b + 1)) | (((bj >> b) & 1) << (2 * b))
    M = S.spamm_from_blocks(ctx, nb * 32, 32, bi.astype(np.int32), bj.astype(np.int32), pay)
    sq = pay[:, 1, 1] ** 2
    o = np.lexsort((code, sq))  # ascending, ties in Morton order
    csum = np.cumsum(sq[o])
    for tau in (0.0, 1e-5, 3.0, 1e4, 1e30):
        T = S.spamm_truncate(ctx, M, tau, "error")
        keep = np.ones(len(bi), bool)
        keep[o[csum <= tau * tau]] = False
        ti, tj, _, _ = S.spamm_to_blocks(ctx, T, payload=False)
        got = set(zip(ti.tolist(), tj.tolist()))
        assert got == set(zip(bi[keep].tolist(), bj[keep].tolist())), tau
