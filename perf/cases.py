"""Workloads of the block-tridiagonal HPD solver, as a user's program runs them.

A case is a dict of plain values; its "kind" is the call that the program makes:

  solve    crs.solve on device tensors: one system, one call, breakdown checked
  plan     a kept plan: factor a new matrix and solve (one step of a Newton or
           implicit time integration)
  resolve  a kept factorisation, a new right-hand side
  grad     CRSolveFn forward and backward (a solver layer in a training step)
  batch    many systems of uneven N, m and k in one launch
  mixed    FP32 levels refined to FP64 accuracy
  host     a kept plan with pinned host buffers in and out

and its "system" says how the matrix is made:

  random     the recipe of synthetic.gen_system (block diagonally dominant),
             drawn on the device; sqrt(||B||_1 ||B||_inf) stands for ||B||_2
  diffusion  one implicit step of a variable-coefficient heat equation on an
             N x m grid: A_j tridiagonal, B_j diagonal, condition number of
             the order of 8 * "lam"
"""
import math

import numpy as np
import torch

import paper_1807_00370_gb300 as crs

DEVICE = "cuda"
BATCH_N = (16, 4096)
BATCH_M = (4, 8, 16, 32)
BATCH_K = (1, 16)


def _case(name, kind, N, m, k, system="random", **more):
    c = {"name": name, "kind": kind, "N": N, "m": m, "k": k, "system": system}
    c.update(more)
    return c


def listed():
    return [
        # the smallest call in use: a short system solved once, plan and check included
        _case("solve_small", "solve", 64, 4, 1),
        # a short system re-factored in a loop: launches and the coarse levels
        _case("plan_short", "plan", 1024, 8, 4),
        # the benchmark's plain workload: a long chain of small blocks
        _case("plan_long", "plan", 1 << 20, 8, 4),
        # sizes that are no multiple of anything
        _case("plan_odd", "plan", 100003, 5, 3),
        # a grid line of 24 points per block, a few right-hand sides
        _case("plan_grid24", "plan", 5001, 24, 7, system="diffusion", lam=25.0),
        # the widest block class in FP64
        _case("plan_wide", "plan", 1 << 12, 64, 32),
        # time stepping with a constant matrix: factor once, one vector per step
        _case("resolve_step", "resolve", 1 << 16, 16, 1, system="diffusion", lam=100.0),
        # the benchmark's adjoint workload: forward and backward of a solver layer
        _case("grad_layer", "grad", 1 << 16, 16, 8),
        # the same layer on a short sequence (smoothing of a 12-state signal)
        _case("grad_short", "grad", 1024, 12, 2),
        # the benchmark's batch with fewer systems
        _case("batch_uneven", "batch", 512, 0, 0, shapes=3003),
        # the benchmark's mixed-precision workload
        _case("mixed_wide", "mixed", 1 << 14, 64, 32),
        # data that live on the host, copied in and out in every call
        _case("host_call", "host", 1 << 18, 8, 4),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["solve", "plan", "plan", "plan", "resolve", "resolve", "grad", "grad", "batch", "mixed", "host"])
    if kind == "batch":
        return {"kind": kind, "N": _log_int(rng, 24, 512), "m": 0, "k": 0, "system": "random",
                "shapes": rng.randrange(1 << 30)}
    m = rng.randint(33, 64) if kind == "mixed" else _log_int(rng, 2, 64)
    k = _log_int(rng, 1, 32)
    per_row = 40.0 * m * m * k + (0.0 if kind == "resolve" else 25.33 * m ** 3)
    most = {"solve": 1 << 14, "grad": 1 << 17, "host": 1 << 18, "mixed": 1 << 13}.get(kind, 1 << 20)
    # at most a quarter of the plain workload's factor and solve
    most = max(64, min(most, int(6e9 / per_row)))
    c = {"kind": kind, "N": _log_int(rng, 16, most), "m": m, "k": k}
    if kind != "mixed" and rng.random() < 0.3:
        c.update(system="diffusion", lam=round(10.0 ** rng.uniform(0.0, 2.5), 3))
    else:
        c.update(system="random")
    return c


def _batch_shapes(case):
    r = np.random.default_rng(case["shapes"])
    n = case["N"]
    Ns = r.integers(BATCH_N[0], BATCH_N[1] + 1, size=n).astype(np.int64)
    ms = r.choice(np.asarray(BATCH_M), size=n).astype(np.int32)
    ks = r.integers(BATCH_K[0], BATCH_K[1] + 1, size=n).astype(np.int32)
    return Ns, ms, ks


def _cn(gen, *shape):
    z = torch.randn(tuple(shape) + (2,), generator=gen, device=DEVICE, dtype=torch.float64)
    return torch.view_as_complex(z.mul_(math.sqrt(0.5)))


def _random_system(gen, N, m, cuts=None):
    """A [N, m, m], B [N-1, m, m]; B is zero after the blocks in `cuts`."""
    B = _cn(gen, max(N - 1, 0), m, m).mul_(0.5 / math.sqrt(m))
    if cuts is not None and len(cuts):
        B[torch.as_tensor(cuts, device=DEVICE)] = 0
    G = _cn(gen, N, m, m)
    A = torch.matmul(G, G.mH)
    del G
    A.mul_(1.0 / m)
    shift = torch.ones(N, device=DEVICE, dtype=torch.float64)
    if N > 1:
        a = B.abs()
        nb = torch.sqrt(a.sum(1).amax(1) * a.sum(2).amax(1))
        del a
        shift[1:] += nb
        shift[:-1] += nb
    d = torch.diagonal(A, dim1=1, dim2=2)
    d += shift[:, None]
    A = A.add(A.mH).mul_(0.5)
    torch.diagonal(torch.view_as_real(A)[..., 1], dim1=1, dim2=2).zero_()
    return A, B


def _diffusion_system(gen, N, m, lam):
    def conductances(*shape):
        return lam * (0.5 + torch.rand(shape, generator=gen, device=DEVICE, dtype=torch.float64))
    across, along = conductances(N, m + 1), conductances(N + 1, m)
    A = torch.zeros(N, m, m, device=DEVICE, dtype=torch.float64)
    torch.diagonal(A, dim1=1, dim2=2).copy_(1.0 + across[:, :-1] + across[:, 1:] + along[:-1] + along[1:])
    if m > 1:
        torch.diagonal(A, offset=-1, dim1=1, dim2=2).copy_(-across[:, 1:-1])
        torch.diagonal(A, offset=1, dim1=1, dim2=2).copy_(-across[:, 1:-1])
    B = torch.diag_embed(-along[1:-1])
    return A.to(torch.complex128), B.to(torch.complex128)


def _inputs(case, seed):
    """A, B, y and (grad) the cotangent, on the device."""
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(int(seed))
    N, m, k = case["N"], case["m"], case["k"]
    if case["system"] == "diffusion":
        A, B = _diffusion_system(gen, N, m, case["lam"])
    else:
        A, B = _random_system(gen, N, m)
    y = _cn(gen, N, m, k)
    gx = _cn(gen, N, m, k) if case["kind"] == "grad" else None
    return A, B, y, gx


def _batch_groups(case, seed):
    """Per block size m: (systems, their blocks laid end to end as one chain
    with no coupling between systems, their right-hand sides)."""
    Ns, ms, ks = _batch_shapes(case)
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(int(seed))
    for m in sorted(set(ms.tolist())):
        sel = np.flatnonzero(ms == m)
        ends = np.cumsum(Ns[sel])
        A, B = _random_system(gen, int(ends[-1]), m, cuts=ends[:-1] - 1)
        yield m, sel, ends, A, B, [_cn(gen, int(Ns[i]), m, int(ks[i])) for i in sel]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        Ns, ms, ks = _batch_shapes(case)
        b = crs.Batch(Ns, ms, ks)
        A = torch.empty(b.nA, dtype=torch.complex128, device=DEVICE)
        B = torch.empty(b.nB, dtype=torch.complex128, device=DEVICE)
        y = torch.empty(b.nY, dtype=torch.complex128, device=DEVICE)
        for _, sel, ends, Am, Bm, ys in _batch_groups(case, seed):
            for i, end, yi in zip(sel, ends, ys):
                first = int(end - Ns[i])
                a, bb, v = b.system_view(i, A, B, y)
                a.copy_(Am[first:int(end)])
                bb.copy_(Bm[first:int(end) - 1])
                v.copy_(yi)
        return {"kind": kind, "batch": b, "A": A, "B": B, "y": y}
    A, B, y, gx = _inputs(case, seed)
    state = {"kind": kind, "A": A, "B": B, "y": y}
    N, m, k = case["N"], case["m"], case["k"]
    if kind == "grad":
        state.update(A=A.requires_grad_(), B=B.requires_grad_(), y=y.requires_grad_(), gx=gx)
    elif kind == "plan":
        state["plan"] = crs.Plan(N, m, k)
    elif kind == "resolve":
        state["plan"] = crs.Plan(N, m, k)
        crs.crsolve_factor(state["plan"], A, B)
    elif kind == "mixed":
        state["plan"] = crs.Plan(N, m, k, precision=1)
    elif kind == "host":
        state["plan"] = crs.Plan(N, m, k, flags=1)
        for name in ("A", "B", "y"):
            state[name] = torch.empty(state[name].shape, dtype=torch.complex128, pin_memory=True).copy_(state[name])
    return state


def run(state):
    kind, A, B, y = state["kind"], state["A"], state["B"], state["y"]
    if kind == "solve":
        return crs.solve(A, B, y)
    if kind in ("plan", "mixed"):
        crs.crsolve_factor(state["plan"], A, B)
        return crs.crsolve_solve(state["plan"], y)
    if kind == "resolve":
        return crs.crsolve_solve(state["plan"], y)
    if kind == "grad":
        x = crs.CRSolveFn.apply(A, B, y)
        gA, gB, gy = torch.autograd.grad(x, (A, B, y), state["gx"])
        return [x.detach(), gA, gB, gy]
    if kind == "batch":
        return crs.crsolve_batch_solve(state["batch"], A, B, y)
    x, _ = crs.crsolve_solve_host(state["plan"], A, B, y)
    return x


def work(case):
    """Inputs read once, outputs written once; the block operations of classic
    cyclic reduction in leading order (8 per complex multiply-add)."""
    if case["kind"] == "batch":
        Ns, ms, ks = (v.astype(np.float64) for v in _batch_shapes(case))
        return {"bytes": float((16 * ((2 * Ns - 1) * ms * ms + 2 * Ns * ms * ks)).sum()),
                "flops": float((Ns * (25.33 * ms ** 3 + 40 * ms * ms * ks)).sum())}
    kind, N, m, k = case["kind"], case["N"], case["m"], case["k"]
    mat, vec = 16.0 * (2 * N - 1) * m * m, 16.0 * N * m * k
    factor, solve = N * 25.33 * m ** 3, N * 40.0 * m * m * k
    if kind == "resolve":
        # the kept factors (L, P and Q of every block) are its inputs
        return {"bytes": 16.0 * N * (m * (m + 1) / 2 + 2 * m * m) + 2 * vec, "flops": solve}
    if kind == "grad":
        return {"bytes": 2 * mat + 4 * vec, "flops": factor + 2 * solve + N * 8.0 * (1.5 * m * m + 0.5 * m) * 2 * k}
    return {"bytes": mat + 2 * vec, "flops": factor + solve}


# ------------------------------------------------------- 64-bit values
# Block elimination of every second block by torch's own factorisations, then
# corrections with a residual whose products and sums keep their rounding
# errors (two-term arithmetic), so that the result is good to the last bits.

def _chunks(n, size=1 << 15):
    return [(i, min(i + size, n)) for i in range(0, max(n, 1), size)]


def _chol(A):
    return torch.cat([torch.linalg.cholesky(A[a:b]) for a, b in _chunks(len(A))])


def _tri(L, R, adjoint=False):
    if adjoint:
        return torch.cat([torch.linalg.solve_triangular(L[a:b].mH, R[a:b], upper=True) for a, b in _chunks(len(L))])
    return torch.cat([torch.linalg.solve_triangular(L[a:b], R[a:b], upper=False) for a, b in _chunks(len(L))])


def _eliminate(A, B):
    levels = []
    while True:
        L = _chol(A[0::2].contiguous())
        n, e = len(L), len(A) // 2
        if not e:
            levels.append((L, None, None))
            return levels
        Q = _tri(L[:e], B[0::2].mH.contiguous())                      # odd block t and its right neighbour
        P = _tri(L[1:], B[1::2].contiguous())                         # odd block t + 1 and its left neighbour
        levels.append((L, P, Q))
        S = A[1::2] - Q.mH @ Q
        S[:n - 1] -= P.mH @ P
        B = -(Q[1:].mH @ P[:e - 1])
        A = S


def _substitute(levels, y):
    kept = []
    for L, P, Q in levels:
        r = _tri(L, y[0::2].contiguous())
        kept.append(r)
        if Q is None:
            break
        v = y[1::2] - Q.mH @ r[:len(Q)]
        v[:len(P)] -= P.mH @ r[1:]
        y = v
    x = None
    for (L, P, Q), r in zip(reversed(levels), reversed(kept)):
        if Q is None:
            x = _tri(L, r, adjoint=True)
            continue
        r[:len(Q)] -= Q @ x
        r[1:] -= P @ x[:len(P)]
        full = torch.empty((len(L) + len(Q),) + tuple(r.shape[1:]), dtype=r.dtype, device=r.device)
        full[0::2] = _tri(L, r, adjoint=True)
        full[1::2] = x
        x = full
    return x


def _halves(a):
    c = 134217729.0 * a
    hi = c - (c - a)
    return hi, a - hi


class _TwoTerm:
    """A sum of products a * b kept as value + error (Dekker, Knuth)."""

    def __init__(self, start):
        self.s, self.e = start.clone(), torch.zeros_like(start)

    def sub(self, a, b):
        (a, ah, al), (b, bh, bl) = a, b
        p = a * b
        err = ((ah * bh - p) + ah * bl + al * bh) + al * bl
        t = self.s - p
        z = t - self.s
        self.e += (self.s - (t - z)) - (p + z)
        self.e -= err
        self.s = t


def _residual(A, B, x, y):
    N, m = A.shape[0], A.shape[1]
    re, im = _TwoTerm(y.real.contiguous()), _TwoTerm(y.imag.contiguous())
    zero = torch.zeros_like(x[:1])
    left, right = torch.cat([zero, x[:-1]]), torch.cat([x[1:], zero])
    empty = torch.zeros(1, m, m, dtype=A.dtype, device=A.device)
    Bl = torch.cat([empty, B])
    Bu = torch.cat([B.mH, empty])
    for M, v in ((Bl, left), (A, x), (Bu, right)):
        for s in range(m):
            def parts(t):
                t = t.contiguous()
                return (t,) + _halves(t)
            ar, ai = parts(M.real[:, :, s:s + 1]), parts(M.imag[:, :, s:s + 1])
            xr, xi = parts(v.real[:, s:s + 1]), parts(v.imag[:, s:s + 1])
            neg = tuple(-t for t in ai)
            re.sub(ar, xr)
            re.sub(neg, xi)
            im.sub(ar, xi)
            im.sub(ai, xr)
    return torch.complex(re.s + re.e, im.s + im.e)


def _exact_solve(A, B, *rhs):
    levels = _eliminate(A, B)
    out = []
    for y in rhs:
        x = _substitute(levels, y)
        for _ in range(2):
            x = x + _substitute(levels, _residual(A, B, x, y))
        out.append(x)
    return out


def exact(case, seed):
    kind = case["kind"]
    with torch.no_grad():
        if kind == "batch":
            Ns, ms, ks = _batch_shapes(case)
            xs = [None] * len(Ns)
            for m, sel, ends, A, B, ys in _batch_groups(case, seed):
                y = torch.zeros(len(A), m, BATCH_K[1], dtype=torch.complex128, device=DEVICE)
                for i, end, yi in zip(sel, ends, ys):
                    y[int(end - Ns[i]):int(end), :, :int(ks[i])] = yi
                x, = _exact_solve(A, B, y)
                for i, end in zip(sel, ends):
                    xs[i] = x[int(end - Ns[i]):int(end), :, :int(ks[i])].reshape(-1)
            return torch.cat(xs)
        A, B, y, gx = _inputs(case, seed)
        if kind != "grad":
            x, = _exact_solve(A, B, y)
            return x.cpu() if kind == "host" else x
        x, gy = _exact_solve(A, B, y, gx)
        gA = gy @ x.mH
        gA = (gA + gA.mH).mul_(-0.5)
        gB = -(gy[1:] @ x[:-1].mH + x[1:] @ gy[:-1].mH)
        return [x, gA, gB, gy]
