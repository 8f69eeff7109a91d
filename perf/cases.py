"""What this library is timed on: the work its users have it do.

Each case is one call (or one small group of calls) through the public
binding on systems of the paper's randsvd kind: A = Q1 diag(sigma) Q2^T with
sigma_i = kappa^(-(i-1)/(n-1)) and b = A x_true, x_true ~ N(0, 1).  Q1 and Q2
are products of Hartley transforms, random signs and random permutations
(orthogonal, dense and unstructured for this purpose, and made in n^2 log n
operations on the device, where a QR of a random matrix would take seconds at
n = 8192).

Kinds of work ("kind"):
  solve     Context.solve: one system, 1 to 16 right-hand sides
  batch     Context.solve_batched: many small systems at once
  factor    Context.factor and one application of the new factors: what a
            program pays that brings its own iteration and a new matrix
  apply     Factors.apply on factors a program keeps: the preconditioner of
            its own iteration, fp32 / fp64 / double-double arithmetic
  residual  Context.residual of an approximate solution
  serve     Server: a burst of host-buffer requests of mixed sizes and
            precisions, submitted together and polled until all are done

Solutions are returned in the working precision of their system: the library
writes them as doubles that hold fp32 values when u = fp32, so the
conversion changes no value.
"""

import math
import time

import numpy as np
import torch

import paper_2107_06200_gb300 as M

DEV = "cuda:0"
HALF, BRAIN, SINGLE = "fp16,fp32,fp64", "bf16,fp32,fp64", "fp32,fp64,dd"

_kept = {}


def _context():
    """The context of the process: a program creates one and keeps it."""
    if "ctx" not in _kept:
        _kept["ctx"] = M.Context(0)
    return _kept["ctx"]


def _server():
    if "srv" not in _kept:
        _kept["srv_ctx"] = M.Context(0)
        _kept["srv"] = M.Server(_kept["srv_ctx"], hbm_budget_bytes=64 << 30, max_slots=8)
    return _kept["srv"]


# ------------------------------------------------------------------ cases

def listed():
    return [
        # the paper's own size (randsvd experiments, n = 100): one small system, latency
        dict(name="solve_100_half", kind="solve", n=100, kappa=1e2, triple=HALF, nrhs=1),
        # an odd size between the small systems and the sweep, bf16 factors, a few right-hand sides
        dict(name="solve_777_bf16_3rhs", kind="solve", n=777, kappa=1e2, triple=BRAIN, nrhs=3),
        # the n = 2000 sweep: fp16 factors that need GMRES, and fp32 factors with a double-double residual
        dict(name="solve_2000_half", kind="solve", n=2000, kappa=1e4, triple=HALF, nrhs=1),
        dict(name="solve_2000_single", kind="solve", n=2000, kappa=1e8, triple=SINGLE, nrhs=1),
        # the large configuration: the benchmark's three precision triples at n = 8192
        dict(name="solve_8192_half", kind="solve", n=8192, kappa=1e3, triple=HALF, nrhs=1),
        dict(name="solve_8192_bf16", kind="solve", n=8192, kappa=1e3, triple=BRAIN, nrhs=1),
        dict(name="solve_8192_single", kind="solve", n=8192, kappa=1e3, triple=SINGLE, nrhs=1),
        # several right-hand sides sharing one factorisation, at a ragged size
        dict(name="solve_4133_half_16rhs", kind="solve", n=4133, kappa=1e3, triple=HALF, nrhs=16),
        # the batched workload: n uniform in [32, 512], kappa log-uniform in [1e1, 1e6]
        dict(name="batch_600_half", kind="batch", count=600, n_lo=32, n_hi=512, sizes=0, triple=HALF),
        # a new matrix factored in fp32 and applied once, and kept fp16 factors applied to 4 vectors in fp64
        dict(name="factor_3000_fp32", kind="factor", n=3000, kappa=1e4, u="fp64", uf="fp32", arith="fp32", nrhs=1),
        dict(name="apply_5000_fp64", kind="apply", n=5000, kappa=1e3, u="fp32", uf="fp16", arith="fp64", nrhs=4),
        # a serving burst: sizes log-uniform in [256, 2048], kappa log-uniform in [1e2, 1e5], the three triples
        dict(name="serve_16", kind="serve", count=16, n_lo=256, n_hi=2048, sizes=0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "batch", "factor", "apply", "residual"])
    if kind == "solve":
        triple = rng.choice([HALF, BRAIN, SINGLE])
        n = int(round(_log(rng, 64, 8192)))
        nrhs = rng.choice([1, 1, 1, rng.randint(2, 16)])
        # hard systems (GMRES stages, refactorisations) stay small enough to cost no more than the largest case
        most = {HALF: 1e4, BRAIN: 1e2, SINGLE: 1e7}[triple]
        if n > 3000:
            most = {HALF: 1e3, BRAIN: 30.0, SINGLE: 1e5}[triple]
        return dict(kind="solve", n=n, kappa=float("%.3g" % _log(rng, 10, most)), triple=triple, nrhs=nrhs)
    if kind == "batch":
        lo = rng.randint(16, 200)
        return dict(kind="batch", count=int(round(_log(rng, 8, 600))), n_lo=lo, n_hi=rng.randint(lo, 512),
                    sizes=rng.randint(1, 10 ** 6), triple=rng.choice([HALF, BRAIN, SINGLE]))
    n = int(round(_log(rng, 64, 8192)))
    if kind == "residual":
        u = rng.choice(["fp32", "fp64"])
        return dict(kind="residual", n=n, kappa=float("%.3g" % _log(rng, 10, 1e4)), u=u)
    uf = rng.choice(["fp16", "bf16", "fp32"])
    arith = rng.choice(["fp32", "fp64", "dd"]) if kind == "apply" else "fp32"
    return dict(kind=kind, n=n, kappa=float("%.3g" % _log(rng, 10, 1e3)), u="fp64" if uf == "fp32" else "fp32",
                uf=uf, arith=arith, nrhs=rng.randint(1, 8))


# ----------------------------------------------------------------- inputs

def _hartley(X):
    """The orthonormal discrete Hartley transform of the rows of X."""
    F = torch.fft.fft(X, dim=1)
    return (F.real - F.imag) / math.sqrt(X.shape[1])


def _mix(X, g):
    """X Q^T with a random orthogonal Q: three rounds of random signs, a
    random permutation and a Hartley transform along the rows."""
    n = X.shape[1]
    for _ in range(3):
        s = (torch.randint(0, 2, (n,), generator=g, device=X.device) * 2 - 1).to(X.dtype)
        X = _hartley(X[:, torch.randperm(n, generator=g, device=X.device)] * s)
    return X


def _system(n, kappa, g, nrhs=1):
    """A (n x n), B (n x nrhs), X (n x nrhs) in fp64 on the device."""
    e = -torch.arange(n, dtype=torch.float64, device=DEV) / max(n - 1, 1)
    A = torch.diag(torch.pow(torch.tensor(float(kappa), dtype=torch.float64, device=DEV), e))
    A = _mix(_mix(A, g).t().contiguous(), g)
    X = torch.randn((n, nrhs), generator=g, dtype=torch.float64, device=DEV)
    return A, A @ X, X


def _sizes(case):
    """Sizes, condition numbers and triples of a batch or a burst: fixed by
    the case, so that every seed is the same work on other numbers."""
    rng = np.random.default_rng(case["sizes"])
    c = case["count"]
    if case["kind"] == "batch":
        ns = rng.integers(case["n_lo"], case["n_hi"] + 1, size=c)
        ks = 10.0 ** rng.uniform(1.0, 6.0, size=c)
        return [(int(n), float(k), case["triple"]) for n, k in zip(ns, ks)]
    ns = np.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), size=c))
    ks = 10.0 ** rng.uniform(2.0, 5.0, size=c)
    # bf16 factors take the better-conditioned requests
    return [(int(round(n)), float(k), HALF if k > 10 ** 3.5 and j % 3 == 1 else (HALF, BRAIN, SINGLE)[j % 3])
            for j, (n, k) in enumerate(zip(ns, ks))]


def _code(name):
    return M.PREC_CODES[name]


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def prepare(case, seed):
    g, kind = _gen(seed), case["kind"]
    if kind == "solve":
        A, B, _ = _system(case["n"], case["kappa"], g, case["nrhs"])
        return dict(case=case, ctx=_context(), A=A, B=B[:, 0].contiguous() if case["nrhs"] == 1 else B)
    if kind == "batch":
        made = [_system(n, k, g) for n, k, _ in _sizes(case)]
        return dict(case=case, ctx=_context(), As=[m[0] for m in made], bs=[m[1][:, 0].contiguous() for m in made])
    if kind == "serve":
        made = [_system(n, k, g) for n, k, _ in _sizes(case)]
        # host buffers, column-major as the library takes them
        return dict(case=case, srv=_server(), specs=[t for _, _, t in _sizes(case)],
                    As=[m[0].t().contiguous().cpu().numpy().T for m in made],
                    bs=[m[1][:, 0].cpu().numpy() for m in made])
    if kind == "residual":
        A, B, X = _system(case["n"], case["kappa"], g)
        x = X[:, 0] * (1 + 1e-7 * torch.randn(case["n"], generator=g, dtype=torch.float64, device=DEV))
        if case["u"] == "fp32":
            x = x.float().double()
        return dict(case=case, ctx=_context(), A=A, x=x, b=B[:, 0].contiguous())
    A, _, _ = _system(case["n"], case["kappa"], g)
    B = torch.randn((case["n"], case["nrhs"]), generator=g, dtype=torch.float64, device=DEV)
    state = dict(case=case, ctx=_context(), A=A, B=B)
    if kind == "apply":
        state["factors"] = state["ctx"].factor(A, _code(case["u"]), _code(case["uf"]))
        del state["A"]
    return state


# -------------------------------------------------------------------- run

def _working(x, triple):
    """A solution in the working precision of its system."""
    return x if triple == SINGLE else (x.float() if torch.is_tensor(x) else x.astype(np.float32))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        X, reports, status = state["ctx"].solve(state["A"], state["B"], case["triple"])
        return dict(x=_working(X, case["triple"]), status=status)
    if kind == "batch":
        xs, reports, status = state["ctx"].solve_batched(state["As"], state["bs"], case["triple"])
        return dict(x=_working(torch.cat(xs), case["triple"]), status=status)
    if kind == "serve":
        srv, specs = state["srv"], state["specs"]
        tickets = [srv.submit(A, b, spec) for A, b, spec in zip(state["As"], state["bs"], specs)]
        xs, left = [None] * len(tickets), set(range(len(tickets)))
        while left:
            for i in sorted(left):
                done, x, report, latency = srv.poll(tickets[i], state["bs"][i].shape[0])
                if done == 2:
                    xs[i] = _working(x, specs[i])
                    left.discard(i)
            if left:
                time.sleep(0.0002)
        return dict(x32=np.concatenate([x for x, t in zip(xs, specs) if t != SINGLE]),
                    x64=np.concatenate([x for x, t in zip(xs, specs) if t == SINGLE] or [np.zeros(1)]))
    if kind == "residual":
        u0, ur = _code(case["u"]), _code("dd" if case["u"] == "fp64" else "fp64")
        r, s = state["ctx"].residual(state["A"], state["x"], state["b"], u0, ur)
        return dict(r=r, s=s)
    arith = _code(case["arith"])
    if kind == "factor":
        f = state["ctx"].factor(state["A"], _code(case["u"]), _code(case["uf"]))
        X = f.apply(state["B"], arith, arith)
        f.close()
    else:
        X = state["factors"].apply(state["B"], arith, arith if case["arith"] != "dd" else M.FP64)
    return X.float() if case["arith"] == "fp32" else X.contiguous()


# ------------------------------------------------------------------- work

def work(case):
    """Bytes: every matrix and right-hand side read once in fp64, every
    output written once.  Operations: 2/3 n^3 for each factorisation asked
    for and 2 n^2 per solved or multiplied vector."""
    kind = case["kind"]
    if kind in ("batch", "serve"):
        ns = [n for n, _, _ in _sizes(case)]
        return dict(bytes=sum(8.0 * n * n + 16.0 * n for n in ns), flops=sum(2 / 3 * n ** 3 + 2.0 * n * n for n in ns))
    n, r = float(case["n"]), case.get("nrhs", 1)
    if kind == "residual":
        return dict(bytes=8 * n * n + 24 * n, flops=2 * n * n)
    if kind == "apply":
        size = {"fp16": 2, "bf16": 2, "fp32": 4, "fp64": 8}[case["uf"]]
        return dict(bytes=size * n * n + 16 * n * r, flops=2 * n * n * r)
    return dict(bytes=8 * n * n + 16 * n * r, flops=2 / 3 * n ** 3 + 2 * n * n * r)


# ------------------------------------------------------------------ exact

def _exact_x(A, B, triple):
    """The solution of the system that the library solves: A and b rounded to
    the working precision."""
    if triple != SINGLE:
        A, B = A.float().double(), B.float().double()
    return torch.linalg.solve(A, B)


def _two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def _exact_residual(A, x, b):
    """b - A x as an unevaluated pair, from exact products (Dekker's
    splitting) and error-free additions in a tree; rows in chunks."""
    def split(v):
        c = v * 134217729.0
        h = c - (c - v)
        return h, v - h
    out_h, out_l = [], []
    xh, xl = split(x)
    for i in range(0, A.shape[0], 1024):
        a = A[i:i + 1024]
        ah, al = split(a)
        p = a * x
        e = ((ah * xh - p) + ah * xl + al * xh) + al * xl
        p = torch.cat([b[i:i + 1024, None], -p], 1)
        e = -e.sum(1)
        while p.shape[1] > 1:
            if p.shape[1] % 2:
                p = torch.cat([p, torch.zeros_like(p[:, :1])], 1)
            p, d = _two_sum(p[:, 0::2], p[:, 1::2])
            e = e + d.sum(1)
        h, l = _two_sum(p[:, 0], e)
        out_h.append(h)
        out_l.append(l)
    return torch.cat(out_h), torch.cat(out_l)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("apply", "factor"):
        return None  # the result is that of the rounded factors, which no other code has
    s = prepare(case, seed)
    if kind == "solve":
        return dict(x=_exact_x(s["A"], s["B"], case["triple"]), status=None)
    if kind == "batch":
        return dict(x=torch.cat([_exact_x(A, b, case["triple"]) for A, b in zip(s["As"], s["bs"])]), status=None)
    if kind == "serve":
        xs = [_exact_x(torch.from_numpy(np.ascontiguousarray(A)).to(DEV), torch.from_numpy(b).to(DEV), t).cpu()
              for A, b, t in zip(s["As"], s["bs"], s["specs"])]
        return dict(x32=torch.cat([x for x, t in zip(xs, s["specs"]) if t != SINGLE]),
                    x64=torch.cat([x for x, t in zip(xs, s["specs"]) if t == SINGLE]))
    A, x, b = s["A"], s["x"], s["b"]
    if case["u"] == "fp32":
        A, b = A.float().double(), b.float().double()
    h, l = _exact_residual(A, x, b)
    if case["u"] == "fp32":
        return dict(r=h, s=float(h.abs().max()))
    return dict(r=torch.cat([h, l]), s=float(h.abs().max()))
