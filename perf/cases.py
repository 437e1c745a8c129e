"""What this solver's users have it do, as cases that can be timed and checked.

A case is one call sequence through the public binding (paper_1505_06864_gb300.dm) on one system or one
batch: factor and solve a new system, or solve a new right-hand side on resident factors.  `listed()` holds
fixed sizes, `draw()` others of the same ranges.  Inputs are drawn on the GPU from the seed alone, with the
distributions of the library's workloads (paper_1505_06864_gb300/workloads.py).

Fields of a case:
  op         "step": dm_factor + dm_solve; "solve": dm_solve on resident factors; "complex": the same step
             on a complex system; "batch": dm_factor + dm_solve of a batch plan
  gen        "dominant", "pde" (banded blocks stored dense), "conditioned" (cond(B_i) = `cond`), "laplace"
  N, m, r    block rows, block size, right-hand-side columns (batch: `count` systems, shapes from `shapes`)
  P, levels  decomposition (0: the library's choice)
  prec       "fp64", "fp32", "tf32", "bf16x3" (the last three: refinement to float64 accuracy)
"""
import math
import random

import torch

from paper_1505_06864_gb300 import dm

BATCH_M = (32, 64, 96, 128)


def listed():
    return [
        # the smallest plan: a quick check or an inner solve of another method; launches and latency
        dict(name="small_fp64_m16", op="step", gen="dominant", N=64, m=16, r=1, P=4, levels=1, prec="fp64"),
        # a mid-size dense system, a few right-hand sides, the library's own decomposition
        dict(name="dense_fp64_m64", op="step", gen="dominant", N=500, m=64, r=4, P=0, levels=0, prec="fp64"),
        # the headline workload: finite differences x cubic splines, banded blocks stored dense
        dict(name="pde_fp64_m256", op="step", gen="pde", N=2048, m=256, r=1, P=64, levels=3, prec="fp64"),
        # dense nonsymmetric blocks with cond 1e4, several right-hand sides, in plain float64 ...
        dict(name="cond_fp64_m128", op="step", gen="conditioned", N=4096, m=128, r=8, P=0, levels=0, prec="fp64",
             cond=1e4),
        # ... and with split-bf16 factors refined to float64
        dict(name="cond_bf16x3_m128", op="step", gen="conditioned", N=4096, m=128, r=8, P=0, levels=0,
             prec="bf16x3", cond=1e4),
        # TF32 factors, a block size and a length that fill no tile evenly
        dict(name="ragged_tf32_m88", op="step", gen="dominant", N=777, m=88, r=3, P=0, levels=0, prec="tf32"),
        # a parameter sweep: systems of uneven N, m and nrhs in one plan, inputs used in place
        dict(name="batch_bf16x3_48", op="batch", gen="dominant", count=48, shapes=4, prec="bf16x3"),
        # the paper's validation shapes (Laplace blocks with small random fill): block sizes that are no
        # multiple of 8 ...
        dict(name="laplace_fp64_m100", op="step", gen="laplace", N=3071, m=100, r=1, P=32, levels=1, prec="fp64"),
        # ... and the large one, on a shorter system
        dict(name="laplace_fp64_m400", op="step", gen="laplace", N=511, m=400, r=1, P=16, levels=1, prec="fp64"),
        # a repeat right-hand side on resident factors: one column on float64 factors ...
        dict(name="resolve_fp64_m256", op="solve", gen="pde", N=2048, m=256, r=1, P=64, levels=3, prec="fp64"),
        # ... and several on split-bf16 factors with refinement (what a server runs)
        dict(name="resolve_bf16x3_m128", op="solve", gen="conditioned", N=4096, m=128, r=8, P=0, levels=0,
             prec="bf16x3", cond=1e4),
        # complex boundary conditions: a complex system through its real embedding
        dict(name="complex_fp64_m64", op="complex", gen="dominant", N=512, m=64, r=2, P=0, levels=0, prec="fp64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["step", "step", "step", "step", "batch", "solve", "complex"])
    if op == "batch":
        return dict(op="batch", gen="dominant", count=rng.randint(2, 32), shapes=rng.randint(100, 10**6),
                    prec=rng.choice(["bf16x3", "tf32", "fp64"]))
    prec = "fp64" if op == "complex" else rng.choice(["fp64", "fp64", "fp32", "tf32", "bf16x3"])
    # block sizes up to 400 (256 on the tensor-core precisions), multiples of 8 and others
    m = _log_int(rng, 8, 100 if op == "complex" else 400 if prec == "fp64" else 256)
    if rng.random() < 0.6:
        m = max(8, 8 * (m // 8))
    N = _log_int(rng, 24, 4096)
    while N > 24 and N * float(m) ** 3 > 1.0e10:
        N = max(24, int(N * 0.8))
    gen = rng.choice(["dominant", "pde", "laplace", "conditioned"] if prec == "fp64" and op != "complex" else
                     ["dominant", "pde"])
    case = dict(op=op, gen=gen, N=N, m=m, r=rng.choice([1, 1, 2, 3, 5, 8, 16]), P=0, levels=0, prec=prec)
    if rng.random() < 0.3:
        case.update(P=rng.randint(1, max(1, min(96, N // 8))), levels=rng.randint(1, 2))
        if case["P"] < 8:  # a short chain of block rows keeps such a case no longer than the listed ones
            case["N"] = min(N, 512)
            case["P"] = max(1, min(case["P"], case["N"] // 8))
    if gen == "conditioned":
        case["cond"] = rng.choice([1e2, 1e3, 1e4])
    return case


# ---------------------------------------------------------------- inputs
def _shapes(case):
    rng = random.Random(case["shapes"])
    return [(rng.randint(32, 2048), rng.choice(BATCH_M), rng.randint(1, 16)) for _ in range(case["count"])]


class _Draw:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def uniform(self, shape, lo, hi):
        return torch.rand(shape, generator=self.g, device="cuda", dtype=torch.float64).mul_(hi - lo).add_(lo)

    def normal(self, shape):
        return torch.randn(shape, generator=self.g, device="cuda", dtype=torch.float64)

    def orthogonal(self, n, m):
        """[n, m, m] products of three random reflections."""
        q = torch.eye(m, device="cuda", dtype=torch.float64).expand(n, m, m).clone()
        for _ in range(3):
            v = self.normal((n, m, 1))
            v /= v.norm(dim=1, keepdim=True)
            q.baddbmm_(torch.bmm(q, v), v.transpose(1, 2), alpha=-2.0)
        return q


def _blocks(d, gen, N, m, cond):
    if gen == "dominant":
        A, B, C = (d.uniform((N, m, m), -1.0, 1.0) for _ in range(3))
    elif gen == "pde":
        k = torch.arange(m, device="cuda")
        near = (k[:, None] - k[None, :]).abs() <= 3
        A, B, C = (d.uniform((N, m, m), 0.5, 2.0) * near for _ in range(3))
        A, C = -A, -C
    elif gen == "laplace":
        A, B, C = (d.uniform((N, m, m), -1e-2, 1e-2) for _ in range(3))
        for M, v in ((A, -1.0), (B, 4.0), (C, -1.0)):
            M.diagonal(dim1=1, dim2=2).fill_(v)
        for off in (-1, 1):
            B.diagonal(offset=off, dim1=1, dim2=2).fill_(-1.0)
    else:
        sigma = torch.logspace(math.log10(cond), 0.0, m, device="cuda", dtype=torch.float64)
        U, V = d.orthogonal(N, m), d.orthogonal(N, m)
        B = torch.bmm(U * sigma, V.transpose(1, 2))
        A, C = (d.uniform((N, m, m), -1.0, 1.0) for _ in range(2))
        for M in (A, C):
            M *= 0.25 / M.norm(dim=(1, 2), keepdim=True)
    A[0] = 0.0
    C[N - 1] = 0.0
    return A, B, C


def _shift(A, B, C):
    """Strict diagonal dominance with margin 1, in every point row."""
    s = A.abs().sum(dim=2) + B.abs().sum(dim=2) + C.abs().sum(dim=2) + 1.0
    B.diagonal(dim1=1, dim2=2).add_(s)


def _times(A, B, C, x):
    b = torch.bmm(B, x)
    b[1:] += torch.bmm(A[1:], x[:-1])
    b[:-1] += torch.bmm(C[:-1], x[1:])
    return b


def _system(d, gen, N, m, r, cond=1.0, is_complex=False):
    A, B, C = _blocks(d, gen, N, m, cond)
    if is_complex:
        A, B, C = (torch.complex(X, Y) for X, Y in zip((A, B, C), _blocks(d, gen, N, m, cond)))
    if gen in ("dominant", "pde"):
        _shift(A, B, C)
    x = d.normal((N, m, r))
    if is_complex:
        x = torch.complex(x, d.normal((N, m, r)))
    return A, B, C, _times(A, B, C, x)


def _inputs(case, seed):
    """The systems of a case, one (A, B, C, b) each."""
    d = _Draw(seed)
    if case["op"] == "batch":
        return [_system(d, case["gen"], N, m, r) for N, m, r in _shapes(case)]
    return [_system(d, case["gen"], case["N"], case["m"], case["r"], case.get("cond", 1.0),
                    case["op"] == "complex")]


# ---------------------------------------------------------------- the calls
class _State:
    """A plan and the arrays of one user."""

    def __init__(self, case):
        self.op, self.plan = case["op"], None

    def __del__(self):
        if self.plan is not None:
            dm.dm_destroy(self.plan)
            self.plan = None


def prepare(case, seed):
    s = _State(case)
    systems = _inputs(case, seed)
    if case["op"] == "batch":
        s.A, s.B, s.C, s.b = (torch.cat([sy[i].reshape(-1) for sy in systems]) for i in range(4))
        Ns, ms, rs = zip(*_shapes(case))
        s.count = len(Ns)
        s.plan = dm.dm_plan_batch(Ns, ms, rs, case["prec"])
        dm.dm_set_borrow_inputs(s.plan)
    else:
        s.A, s.B, s.C, s.b = systems[0]
        make = dm.dm_plan_complex if case["op"] == "complex" else dm.dm_plan
        s.plan = make(case["N"], case["m"], case["r"], case["P"], case["levels"], case["prec"])
    s.x = torch.empty_like(s.b)
    torch.cuda.synchronize()  # the plan works on a stream of its own
    if case["op"] == "solve":
        dm.dm_factor(s.plan, s.A, s.B, s.C)
    return s


def run(s):
    if s.op == "complex":
        dm.dm_factor_complex(s.plan, s.A, s.B, s.C)
        dm.dm_solve_complex(s.plan, s.b, s.x)
    elif s.op == "batch":
        dm.dm_factor(s.plan, s.A, s.B, s.C)
        dm.dm_solve(s.plan, s.b, s.x, count=s.count)
    else:
        if s.op == "step":
            dm.dm_factor(s.plan, s.A, s.B, s.C)
        dm.dm_solve(s.plan, s.b, s.x)
    return s.x


def work(case):
    """Block elimination of a tridiagonal block matrix: per row one LU (2/3 m^3), one solve with m columns
    (2 m^3) and one product (2 m^3), then three m x m products with the r columns; a complex multiply-add
    counts as four.  A solve on resident factors reads three blocks per row of its factors' type, and with
    refinement the float64 blocks besides."""
    bytes_ = flops = 0.0
    shapes = _shapes(case) if case["op"] == "batch" else [(case["N"], case["m"], case["r"])]
    for N, m, r in shapes:
        e = 16.0 if case["op"] == "complex" else 8.0
        f = 4.0 if case["op"] == "complex" else 1.0
        bytes_ += 2 * e * N * m * r
        flops += f * 6.0 * N * m * m * r
        if case["op"] == "solve":
            bytes_ += 3.0 * N * m * m * (8.0 if case["prec"] == "fp64" else 4.0 + 8.0)
        else:
            bytes_ += 3.0 * e * N * m * m
            flops += f * 14.0 / 3.0 * N * float(m) ** 3
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------- the exact solutions
class _Reduction:
    """Block cyclic reduction of (A, B, C): the even rows are eliminated, level by level."""

    def __init__(self, A, B, C):
        N = B.shape[0]
        self.N, self.A, self.C = N, A, C
        self.G = torch.linalg.inv(B[0::2])
        self.next = None
        if N > 1:
            Ao, Bo, Co = A[1::2], B[1::2].clone(), C[1::2]
            n = Ao.shape[0]
            L = torch.bmm(Ao, self.G[:n])  # A_i B_{i-1}^{-1}
            nu = self.G.shape[0] - 1
            U = torch.bmm(Co[:nu], self.G[1:])  # C_i B_{i+1}^{-1}, where row i + 1 is there
            self.L, self.U = L, U
            An = -torch.bmm(L, A[0::2][:n])
            Bo -= torch.bmm(L, C[0::2][:n])
            Bo[:nu] -= torch.bmm(U, A[2::2])
            Cn = torch.zeros_like(An)
            Cn[:nu] = -torch.bmm(U, C[2::2])
            self.next = _Reduction(An, Bo, Cn)

    def solve(self, b):
        x = torch.empty_like(b)
        if self.next is None:
            x[0::2] = torch.bmm(self.G, b[0::2])
            return x
        be, n, nu = b[0::2], self.L.shape[0], self.U.shape[0]
        bo = b[1::2] - torch.bmm(self.L, be[:n])
        bo[:nu] -= torch.bmm(self.U, be[1:])
        xo = self.next.solve(bo)
        t = be.clone()
        t[1:] -= torch.bmm(self.A[2::2], xo[:nu])
        t[:n] -= torch.bmm(self.C[0::2][:n], xo)
        x[0::2] = torch.bmm(self.G, t)
        x[1::2] = xo
        return x


def _pieces(v, dim):
    """v as a sum of three terms, the first two of at most 18 bits below the largest value along `dim`."""
    top = torch.frexp(v.abs().amax(dim=dim, keepdim=True)).exponent
    out = []
    for k in (1, 2):
        c = torch.exp2((top - 18 * k).double()) * (1.5 * 2.0 ** 52)
        p = (v + c) - c
        out.append(p)
        v = v - p
    return out + [v]


def _residual(A, B, C, x, b):
    """b - T x with the products of the leading pieces exact and the sums in two float64 words."""
    hi, lo = b.clone(), torch.zeros_like(b)

    def subtract(p, sl):
        s = hi[sl] - p
        z = s - hi[sl]
        lo[sl] += (hi[sl] - (s - z)) + (-p - z)
        hi[sl] = s

    xs = _pieces(x, 1)
    pairs = [(i, j) for d in range(5) for i in range(3) for j in range(3) if i + j == d]
    for M, sl, xl in ((B, slice(None), slice(None)), (A, slice(1, None), slice(None, -1)),
                      (C, slice(None, -1), slice(1, None))):
        Ms = _pieces(M, 2)
        for i, j in pairs:
            subtract(torch.bmm(Ms[i][sl], xs[j][xl]), sl)
    return hi + lo


def _solution(A, B, C, b):
    if A.is_complex():
        emb = lambda X: torch.cat([torch.cat([X.real, -X.imag], 2), torch.cat([X.imag, X.real], 2)], 1)  # noqa: E731
        m = A.shape[1]
        x = _solution(emb(A), emb(B), emb(C), torch.cat([b.real, b.imag], 1))
        return torch.complex(x[:, :m].contiguous(), x[:, m:].contiguous())
    R = _Reduction(A, B, C)
    x = R.solve(b)
    for _ in range(3):
        x = x + R.solve(_residual(A, B, C, x, b))
    return x


def exact(case, seed):
    """The solution to the last bits: block cyclic reduction in float64, refined on residuals in about
    twice that precision."""
    xs = [_solution(*sy) for sy in _inputs(case, seed)]
    return torch.cat([x.reshape(-1) for x in xs]) if case["op"] == "batch" else xs[0]
