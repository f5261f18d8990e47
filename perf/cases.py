"""The measured workloads of this library, each through its public entry points.

Matrices have exponential decay, a_ij = u_ij exp(-alpha d(i, j)), u_ij uniform in
[-1, 1), |a_ij| < 1e-16 taken as 0: on the index line (kind "1d", the paper's model
problem) or on a 3-D unit lattice in Morton order (kind "3d"); leaves whose Frobenius
norm lies below `store` are not part of the input, as when a matrix is built with the
block rule.  Every case is a dict of plain values with an "op":

  multiply  one spamm_multiply of resident operands
  batch     plans for several requests of different sizes, one spamm_execute for all
  host      leaves in pinned host memory: build both operands, multiply, read C back
  purify    one step of a purification chain: X X, 2 X - X^2, traces, the idempotency
            error and an error-controlled truncation of the new state
  blocks    spamm_from_blocks from unordered leaves in device memory
  coo       spamm_from_coo from unordered triplets in device memory
"""
import ctypes
import functools
import math

import torch

from paper_1906_08148_gb300 import spamm as S

DEV = "cuda"
CUTOFF = 1e-16
MULTIPLY = dict(op="multiply", kind="3d", n=4096, alpha=1.0, bs=64, tau=1e-6, store=1e-8, mode="combined",
                prec="fp64", same=False)


def listed():
    m = MULTIPLY
    return [
        # the smallest request: a ragged handful of 32-leaves, where only latency counts
        dict(m, name="line300_fp64", kind="1d", n=300, alpha=0.05, bs=32, tau=1e-6, store=0.0, mode="spamm"),
        # the single-request configuration: the paper's 1-D model problem at n = 2048, A = B
        dict(m, name="line2048_fp64", kind="1d", n=2048, alpha=0.05, bs=32, tau=1e-8, store=0.0, mode="spamm",
             same=True),
        # the small end of the served stream, in the form the autotuner picks there
        dict(m, name="lattice4096_fp16", n=4096, tau=1e-4, store=1e-6, prec="fp16_scaled"),
        # plain double precision with large leaves, n not a multiple of the leaf size, Truncmul
        dict(m, name="line10000_fp64_bs128", kind="1d", n=10000, alpha=0.05, bs=128, tau=1e-8, store=1e-10,
             mode="truncate"),
        # the middle of the range, each split form at the tau it is chosen for
        dict(m, name="lattice16384_split3", n=16384, prec="bf16_split"),
        # 128-leaves on the tensor cores, ragged, the widest decay of the served range
        dict(m, name="lattice20000_fp16_bs128", n=20000, alpha=0.8, bs=128, tau=1e-4, store=1e-6,
             prec="fp16_scaled"),
        # the benchmark lattice in the benchmark's form: the largest multiply
        dict(m, name="lattice65536_split4", n=65536, prec="bf16_split4"),
        # continuous arrivals: requests of a served stream planned one by one, executed together
        dict(op="batch", name="batch8_fp16", count=8, nmin=1000, nmax=5000, alpha=0.9, bs=64, tau=1e-4, store=1e-6,
             mode="combined", prec="fp16_scaled"),
        # data that lives on the host, in and out
        dict(m, op="host", name="host8000_split4", n=8000, tau=1e-8, store=1e-10, prec="bf16_split4"),
        # the application of the paper: one step of density-matrix purification
        dict(op="purify", name="purify8192_split4", n=8192, alpha=1.0, bs=64, tau=1e-6, store=1e-8,
             prec="bf16_split4"),
        # building a matrix from leaves a program already has on the device
        dict(op="blocks", name="blocks16384", kind="3d", n=16384, alpha=0.8, bs=64, store=1e-8),
        # assembling a matrix from triplets, with repeated coordinates
        dict(op="coo", name="coo20000", n=20000, nnz=2000000, width=40.0, bs=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    m = MULTIPLY
    op = rng.choice(["line", "fp64", "tensor", "tensor", "tensor", "batch", "host", "purify", "blocks", "coo"])
    tau = rng.choice([1e-4, 1e-6, 1e-8])
    alpha = round(rng.uniform(0.7, 1.2), 3)
    mode = rng.choice(["combined", "combined", "spamm", "truncate"])
    prec = rng.choice(["fp16_scaled", "bf16_split", "bf16_split4"])
    if op == "line":
        return dict(m, kind="1d", n=_log(rng, 64, 12000), alpha=round(rng.uniform(0.04, 0.2), 4),
                    bs=rng.choice([32, 64, 128, 256]), tau=tau, store=tau / 100, mode=mode, same=rng.random() < 0.5)
    if op == "fp64":
        return dict(m, n=_log(rng, 200, 4096), alpha=alpha, bs=rng.choice([32, 64, 128]), tau=tau, store=tau / 100,
                    mode=mode)
    if op == "tensor":
        return dict(m, n=_log(rng, 500, 24000), alpha=alpha, bs=rng.choice([64, 64, 128]), tau=max(tau, 1e-6),
                    store=max(tau, 1e-6) / 100, mode=rng.choice(["combined", "spamm"]), prec=prec)
    if op == "batch":
        lo = _log(rng, 200, 2000)
        return dict(op="batch", count=rng.randint(2, 10), nmin=lo, nmax=rng.randint(2 * lo, 6000), alpha=alpha, bs=64,
                    tau=tau, store=tau / 100, mode="combined", prec=prec)
    if op == "host":
        return dict(m, op="host", n=_log(rng, 1000, 9000), alpha=alpha, bs=64, tau=tau, store=tau / 100, mode="combined",
                    prec=prec)
    if op == "purify":
        return dict(op="purify", n=_log(rng, 1000, 10000), alpha=alpha, bs=rng.choice([64, 128]), tau=tau,
                    store=tau / 100, prec=rng.choice(["fp16_scaled", "bf16_split4"]))
    if op == "blocks":
        return dict(op="blocks", kind=rng.choice(["1d", "3d"]), n=_log(rng, 500, 20000), alpha=alpha,
                    bs=rng.choice([32, 64, 128, 256]), store=1e-7)
    return dict(op="coo", n=_log(rng, 500, 40000), nnz=_log(rng, 5000, 2000000), width=round(rng.uniform(10.0, 80.0), 1),
                bs=rng.choice([32, 64, 128]))


# ------------------------------------------------------------------ inputs
def _points(n):
    """Lattice points of the indices 0 .. n - 1: bit b of x, y, z is bit 3b, 3b + 1, 3b + 2 of the index."""
    i = torch.arange(n, device=DEV)
    xyz = []
    for a in range(3):
        c = torch.zeros_like(i)
        for b in range(7):
            c |= ((i >> (3 * b + a)) & 1) << b
        xyz.append(c.to(torch.float32))
    return xyz


def _axes(kind, n):
    return [torch.arange(n, device=DEV, dtype=torch.float32)] if kind == "1d" else _points(n)


def _decay(ax, r, c, alpha):
    """exp(-alpha d) over the leaves (r, c)."""
    d2 = 0.0
    for x in ax:
        d2 = d2 + (x[r][:, :, None] - x[c][:, None, :]).square()
    return torch.exp_(d2.double().sqrt_().mul_(-alpha))


@functools.lru_cache(maxsize=32)
def _limits(kind, n, alpha, bs, store):
    """Largest norm a leaf of such a matrix can have (|u| = 1), 0 where it cannot be stored: a block grid on the host."""
    nb = -(-n // bs)
    ax = [x.view(nb, bs) for x in _axes(kind, nb * bs)]
    gap = torch.zeros(nb, nb, device=DEV, dtype=torch.float64)
    for x in ax:  # distance between the bounding boxes of two runs of bs indices
        lo, hi = x.amin(1).double(), x.amax(1).double()
        gap += torch.clamp(torch.maximum(lo[None, :] - hi[:, None], lo[:, None] - hi[None, :]), min=0.0).square()
    bound = torch.exp(-alpha * gap.sqrt())
    bi, bj = ((bound >= CUTOFF) & (bound * bs >= store)).nonzero(as_tuple=True)
    top = torch.zeros_like(gap)
    step = max(1, (1 << 25) // (bs * bs))
    for q in range(0, len(bi), step):
        r, c = bi[q:q + step], bj[q:q + step]
        top[r, c] = _decay(ax, r, c, alpha).square_().sum((1, 2)).sqrt() * (1 + 1e-9)
    return torch.where(top >= store, top, 0.0).cpu()


def _leaves(kind, n, alpha, bs, store, seed, symmetric=False):
    """(bi, bj, payload, norm) of the stored leaves in row order, on the device."""
    g = torch.Generator(DEV).manual_seed(seed)
    nb = -(-n // bs)
    ax = [x.view(nb, bs) for x in _axes(kind, nb * bs)]
    want = _limits(kind, n, alpha, bs, store).to(DEV) > 0.0
    if symmetric:
        want = torch.triu(want)
    bi, bj = want.nonzero(as_tuple=True)
    inside = (torch.arange(nb * bs, device=DEV) < n).view(nb, bs).double()
    keep_i, keep_j, keep_p, keep_s = [], [], [], []
    step = max(1, (1 << 25) // (bs * bs))
    for q in range(0, len(bi), step):
        r, c = bi[q:q + step], bj[q:q + step]
        a = _decay(ax, r, c, alpha)
        a *= torch.rand(a.shape, generator=g, device=DEV, dtype=torch.float64).mul_(2.0).sub_(1.0)
        a *= inside[r][:, :, None]
        a *= inside[c][:, None, :]
        a[a.abs() < CUTOFF] = 0.0
        if symmetric:
            at = r == c
            a[at] = torch.triu(a[at]) + torch.triu(a[at], 1).transpose(1, 2)
        s = a.square().sum((1, 2)).sqrt()
        ok = (s > 0.0) & (s >= store)
        keep_i.append(r[ok]), keep_j.append(c[ok]), keep_p.append(a[ok]), keep_s.append(s[ok])
    bi, bj, pay, s = torch.cat(keep_i), torch.cat(keep_j), torch.cat(keep_p), torch.cat(keep_s)
    if symmetric:
        off = bi != bj
        bi, bj, pay, s = (torch.cat([bi, bj[off]]), torch.cat([bj, bi[off]]),
                          torch.cat([pay, pay[off].transpose(1, 2)]), torch.cat([s, s[off]]))
    return bi, bj, pay.contiguous(), s


def _operands(case, seed):
    a = _leaves(case["kind"], case["n"], case["alpha"], case["bs"], case["store"], 2 * seed + 1)
    if case["same"]:
        return a, a
    return a, _leaves(case["kind"], case["n"], case["alpha"], case["bs"], case["store"], 2 * seed + 2)


def _requests(case, seed):
    """The batch's requests: sizes spread over [nmin, nmax], each with its own pair of operands."""
    k = case["count"]
    for r in range(k):
        n = int(case["nmin"] * (case["nmax"] / case["nmin"]) ** (r / max(1, k - 1)))
        sub = dict(case, kind="3d", n=n, same=False)
        yield sub, seed * 64 + r


def _state(case, seed):
    """A purification state X = (b - F) / (2 b), F = V + D: V the decay matrix, D = -+6 by sublattice, b >= |F|."""
    n, bs = case["n"], case["bs"]
    bi, bj, pay, _ = _leaves("3d", n, case["alpha"], bs, case["store"], 2 * seed + 1, symmetric=True)
    b = 32.0
    pay *= -0.5 / b
    nb = -(-n // bs)
    x, y, z = _points(nb * bs)
    site = torch.where((x + y + z) % 2 == 0, -6.0, 6.0).double()
    site = torch.where(torch.arange(nb * bs, device=DEV) < n, 0.5 - 0.5 * site / b, 0.0).view(nb, bs)
    on = (bi == bj).nonzero()[:, 0]
    pay[on] += torch.diag_embed(site[bi[on]])
    return bi, bj, pay, pay.square().sum((1, 2)).sqrt()


def _triplets(case, seed):
    g = torch.Generator(DEV).manual_seed(seed)
    n, nnz, w = case["n"], case["nnz"], case["width"]
    row = torch.randint(0, n, (nnz,), generator=g, device=DEV)
    u = torch.rand(nnz, generator=g, device=DEV, dtype=torch.float64).clamp_(min=1e-12)
    off = torch.floor(-w * torch.log(u)).long()
    sign = torch.randint(0, 2, (nnz,), generator=g, device=DEV) * 2 - 1
    col = (row + sign * off).clamp_(0, n - 1)
    val = (torch.rand(nnz, generator=g, device=DEV, dtype=torch.float64) * 2 - 1) * torch.exp(-(row - col).abs() / w)
    return row, col, val


# ------------------------------------------------------------ the workloads
_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = S.Context(0)
    return _ctx


def _matrix(n, bs, leaves):
    bi, bj, pay = leaves[:3]
    return S.spamm_from_blocks(_context(), n, bs, bi.int(), bj.int(), pay)


def _room(case):
    """Leaves a result can have, whatever the values drawn: the size of the program's output buffers (a list, one per
    output matrix)."""
    op = case["op"]
    if op == "batch":
        return [r for c, _ in _requests(case, 0) for r in _room(dict(c, op="multiply"))]
    nb = -(-case["n"] // case["bs"])
    if op == "coo":  # |row - col| is at most w ln 1e12
        far = int(case["width"] * math.log(1e12)) + 2
        d = torch.arange(nb)
        return [int(((d[:, None] - d[None, :]).abs() <= (far + case["bs"] - 1) // case["bs"]).sum())]
    if op == "purify":
        top = _limits("3d", case["n"], case["alpha"], case["bs"], case["store"]).to(DEV) / 64.0
        top += torch.eye(nb, device=DEV) * math.sqrt(case["bs"])
        can = _can(top, top, case["tau"], "combined")
        both = int((can | (top > 0.0)).sum())
        return [int(can.sum()), both, both]
    top = _limits(case["kind"], case["n"], case["alpha"], case["bs"], case["store"]).to(DEV)
    return [int((top > 0.0).sum()) if op == "blocks" else int(_can(top, top, case["tau"], case["mode"]).sum())]


def _can(a, b, tau, mode):
    """Output blocks that a product of leaves of at most these norms can reach."""
    if mode != "spamm":
        a, b = a * (a >= tau), b * (b >= tau)
    out = torch.zeros_like(a, dtype=torch.bool)
    for k in range(a.shape[0]):
        p = a[:, k, None] * b[None, k, :]
        out |= p > 0.0 if mode == "truncate" else (p >= tau) & (p > 0.0)
    return out


def _buffers(case):
    bs = case["bs"]
    return [[torch.full((m,), -1, dtype=torch.int32, device=DEV), torch.full((m,), -1, dtype=torch.int32, device=DEV),
             torch.zeros((m, bs, bs), dtype=torch.float64, device=DEV),
             torch.zeros(m, dtype=torch.float64, device=DEV)] for m in _room_of(tuple(sorted(case.items())))]


@functools.lru_cache(maxsize=32)
def _room_of(items):
    return _room(dict(items))


def prepare(case, seed):
    op = case["op"]
    state = {"case": case, "out": _buffers(case)}
    if op == "multiply":
        a, b = _operands(case, seed)
        state["A"] = _matrix(case["n"], case["bs"], a)
        state["B"] = state["A"] if case["same"] else _matrix(case["n"], case["bs"], b)
    elif op == "batch":
        state["pairs"] = [tuple(_matrix(c["n"], c["bs"], x) for x in _operands(c, s)) for c, s in _requests(case, seed)]
    elif op == "host":
        state["host"] = [[x.int().cpu().numpy(), y.int().cpu().numpy(), p.cpu().pin_memory().numpy()]
                         for x, y, p, _ in _operands(case, seed)]
        state["out"] = [x.cpu().pin_memory().numpy() for x in state["out"][0]]
    elif op == "purify":
        state["X"] = _matrix(case["n"], case["bs"], _state(case, seed))
        state["X"].set_symmetric()
    elif op == "blocks":
        bi, bj, pay, _ = _leaves(case["kind"], case["n"], case["alpha"], case["bs"], case["store"], 2 * seed + 1)
        p = torch.randperm(len(bi), generator=torch.Generator(DEV).manual_seed(seed), device=DEV)
        state["leaves"] = (bi[p].int(), bj[p].int(), pay[p])
    else:
        state["coo"] = _triplets(case, seed)
    return state


def _out(M, out):
    """A matrix's leaves into device memory: block coordinates, payload, squared norms (Morton order)."""
    ctx = _context()
    st = S.load().spamm_to_blocks(ctx.handle, M.handle, *(ctypes.c_void_p(t.data_ptr()) for t in out), len(out[0]), 1)
    if st != S.OK:
        raise S.SpammError(st, "spamm_to_blocks")
    return out


def run(state):
    case, out, ctx = state["case"], state["out"], _context()
    op = case["op"]
    if op == "multiply":
        return _out(S.spamm_multiply(ctx, state["A"], state["B"], case["tau"], case["mode"], case["prec"]), out[0])
    if op == "batch":
        plans = [S.spamm_plan_create(ctx, A, B, case["tau"], case["mode"], case["prec"]) for A, B in state["pairs"]]
        return [_out(C, o) for C, o in zip(S.spamm_execute(ctx, plans), out)]
    if op == "host":
        A, B = (S.spamm_from_blocks(ctx, case["n"], case["bs"], *h) for h in state["host"])
        C = S.spamm_multiply(ctx, A, B, case["tau"], case["mode"], case["prec"])
        return list(S.spamm_to_blocks(ctx, C, out=out))
    if op == "purify":
        X = state["X"]
        X2 = S.spamm_multiply(ctx, X, X, case["tau"], "combined", case["prec"])
        Y = S.spamm_add(ctx, 2.0, X, -1.0, X2)
        Z = S.spamm_truncate(ctx, Y, case["tau"], "error")
        return [_out(X2, out[0]), _out(Y, out[1]), _out(Z, out[2]),
                [S.spamm_trace(ctx, X), S.spamm_trace(ctx, X2), S.spamm_error(ctx, X, X2)]]
    if op == "blocks":
        M = S.spamm_from_blocks(ctx, case["n"], case["bs"], *state["leaves"])
    else:
        M = S.spamm_from_coo(ctx, case["n"], *state["coo"], case["bs"])
    return [_out(M, out[0]), S.spamm_frob_norm(ctx, M)]


# --------------------------------------------------- what the path must do
def _grid(n, bs, leaves, value):
    nb = -(-n // bs)
    x = torch.zeros((nb, nb), device=DEV, dtype=value.dtype)
    x[leaves[0], leaves[1]] = value
    return x


def _kept(case, a, b):
    """For each k the (i, j) of the kept products."""
    n, bs, tau, mode = case["n"], case["bs"], case["tau"], case["mode"]
    na, nb = _grid(n, bs, a, a[3]), _grid(n, bs, b, b[3])
    if mode != "spamm":
        na, nb = na * (na >= tau), nb * (nb >= tau)
    for k in range(na.shape[0]):
        p = na[:, k, None] * nb[None, k, :]
        yield p > 0.0 if mode == "truncate" else (p >= tau) & (p > 0.0)


def _multiply_work(case, a, b):
    bs = case["bs"]
    kept, out = 0, None
    for p in _kept(case, a, b):
        kept = kept + p.sum()
        out = p if out is None else out | p
    leaves = len(a[0]) + (0 if b is a else len(b[0])) + int(out.sum())
    return {"bytes": 8.0 * bs * bs * leaves, "flops": 2.0 * bs ** 3 * int(kept)}


def work(case):
    op = case["op"]
    if op in ("multiply", "host"):
        return _multiply_work(case, *_operands(case, 0))
    if op == "batch":
        w = [_multiply_work(c, *_operands(c, s)) for c, s in _requests(case, 0)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    e = 8.0 * case["bs"] ** 2
    if op == "purify":
        x = _state(case, 0)
        w = _multiply_work(dict(case, mode="combined"), x, x)
        out = w["bytes"] / e - len(x[0])
        # X read, X^2, 2 X - X^2 and its truncation written
        return {"bytes": e * (len(x[0]) + 3 * out), "flops": w["flops"] + out * case["bs"] ** 2 * 8.0}
    if op == "blocks":
        m = len(_leaves(case["kind"], case["n"], case["alpha"], case["bs"], case["store"], 1)[0])
        return {"bytes": 2 * e * m, "flops": 2.0 * case["bs"] ** 2 * m}
    row, col, _ = _triplets(case, 0)
    m = len(torch.unique((row // case["bs"]) * (1 << 32) + col // case["bs"]))
    return {"bytes": 24.0 * case["nnz"] + e * m, "flops": float(case["nnz"] + 2 * case["bs"] ** 2 * m)}


# ------------------------------------------------------ values in 64 bits
def _code(bi, bj):
    c = torch.zeros_like(bi)
    for b in range(16):
        c |= (((bi >> b) & 1) << (2 * b + 1)) | (((bj >> b) & 1) << (2 * b))
    return c


def _padded(pay, room):
    """What the output buffers hold: the leaves, then zeros."""
    full = torch.zeros((room,) + pay.shape[1:], dtype=torch.float64, device=DEV)
    full[:len(pay)] = pay
    return [None, None, full, full.square().sum((1, 2))]


def _sorted(bi, bj, pay, room):
    return _padded(pay[torch.argsort(_code(bi, bj))], room)


def _product(case, a, b):
    """(bi, bj, payload) of the method's product, from batched matrix products in 64 bits."""
    n, bs = case["n"], case["bs"]
    ia = _grid(n, bs, a, torch.arange(len(a[0]), device=DEV))
    ib = _grid(n, bs, b, torch.arange(len(b[0]), device=DEV))
    out = None
    for p in _kept(case, a, b):
        out = p if out is None else out | p
    bi, bj = out.nonzero(as_tuple=True)
    ic = _grid(n, bs, (bi, bj), torch.arange(len(bi), device=DEV))
    pay = torch.zeros((len(bi), bs, bs), device=DEV, dtype=torch.float64)
    step = max(1, (1 << 27) // (bs * bs))
    for k, p in enumerate(_kept(case, a, b)):
        i, j = p.nonzero(as_tuple=True)
        for q in range(0, len(i), step):
            x, y = i[q:q + step], j[q:q + step]
            pay.index_add_(0, ic[x, y], torch.bmm(a[2][ia[x, k]], b[2][ib[k, y]]))
    return bi, bj, pay


def exact(case, seed):
    op = case["op"]
    if op in ("multiply", "host") and case["n"] > 24000:  # tens of seconds of 64-bit products
        return None
    room = _room(case)
    if op in ("multiply", "host"):
        return _sorted(*_product(case, *_operands(case, seed)), room[0])
    if op == "batch":
        return [_sorted(*_product(c, *_operands(c, s)), r) for (c, s), r in zip(_requests(case, seed), room)]
    if op == "purify":
        x = _state(case, seed)
        n, bs = case["n"], case["bs"]
        bi, bj, pay = _product(dict(case, mode="combined"), x, x)
        both = torch.cat([_code(x[0], x[1]), _code(bi, bj)])
        codes, at = torch.unique(both, return_inverse=True)
        y = torch.zeros((len(codes), bs, bs), device=DEV, dtype=torch.float64)
        m = len(x[0])
        y[at[:m]] += 2.0 * x[2]
        y[at[m:]] -= pay
        d = torch.zeros_like(y)
        d[at[:m]] += x[2]
        d[at[m:]] -= pay

        def trace(i, j, p):
            return float(p[i == j].diagonal(dim1=1, dim2=2).sum())

        return [_sorted(bi, bj, pay, room[0]), _padded(y, room[1]), [None, None, None, None],
                [trace(*x[:3]), trace(bi, bj, pay), float(d.square().sum().sqrt())]]
    if op == "blocks":
        bi, bj, pay, _ = _leaves(case["kind"], case["n"], case["alpha"], case["bs"], case["store"], 2 * seed + 1)
        return [_sorted(bi, bj, pay, room[0]), float(pay.square().sum().sqrt())]
    row, col, val = _triplets(case, seed)
    bs = case["bs"]
    codes, at = torch.unique(_code(row // bs, col // bs), return_inverse=True)
    pay = torch.zeros(len(codes) * bs * bs, device=DEV, dtype=torch.float64)
    pay.index_add_(0, at * (bs * bs) + (row % bs) * bs + col % bs, val)
    pay = pay.view(-1, bs, bs)
    return [_padded(pay, room[0]), float(pay.square().sum().sqrt())]
