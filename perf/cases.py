"""The work that is timed: what a symbolic-regression program has the library do, over the sizes it meets.

Every case goes through the public binding.  Populations are random valid postfix programs, or the same
after some generations of selection and crossover (what every evaluation after the first one sees);
targets are a closed formula of the variables with 1 % noise.  Inputs come from the seed alone.
"""
import math

import torch

from paper_2603_12292_gb300 import binding as sr

DEV = "cuda"
MSE, CORR, BOTH = sr.SR_MSE, sr.SR_CORR, sr.SR_MSE_CORR
FLT_LIMIT = 2.0 ** 128 - 2.0 ** 103  # an FP32 result at or beyond this is infinite


def _case(name, path, P, Lmin, Lmax, nvars, K, N, kind=0, ops=6, xlo=1.0, xhi=10.0, gens=0, nprob=1, graph=False):
    c = dict(path=path, P=P, Lmin=Lmin, Lmax=Lmax, nvars=nvars, K=K, N=N, kind=kind, ops=ops, xlo=xlo, xhi=xhi,
             gens=gens, nprob=nprob, graph=graph)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a quick look at a handful of formulas on a few measurements: launches and latency only
        _case("eval-32x512", "eval", 32, 1, 24, 2, 2, 512, MSE, xhi=5.0),
        # the plain generation of a small interactive run, captured once and replayed
        _case("generation-256x1k-graph", "generation", 256, 1, 32, 3, 4, 1000, MSE, xhi=5.0, gens=4, graph=True),
        # the ordinary generation: 4,096 programs, 100,000 cases, both fitness kinds, a population under way
        _case("generation-4096x100k", "generation", 4096, 8, 128, 10, 4, 100_000, BOTH, gens=8),
        # the first generation of such a run, on a number of cases that no tile divides
        _case("eval-1500x100003", "eval", 1500, 8, 128, 10, 4, 100_003, BOTH),
        # a large population of long programs, 1 - r^2, variables of both signs
        _case("eval-8192x131072-long", "eval", 8192, 4, 256, 10, 4, 131_072, CORR, xlo=-3.0, xhi=3.0),
        # Eq. 2 scores over all of Table 1's operators, with invalid targets
        _case("score-r4-table1", "score", 2048, 8, 128, 10, 4, 50_001, sr.SR_SCORE_R4, ops=12),
        # Eq. 3 point-to-point scores, with invalid targets
        _case("score-p2p", "score", 4096, 8, 128, 10, 4, 40_000, sr.SR_SCORE_P2P),
        # the outputs of the best programs on a validation set
        _case("predict-512x30011", "predict", 512, 4, 128, 7, 4, 30_011, gens=4),
        # many small problems at once (316 to 10,000 cases, 64 to 1,024 programs each)
        _case("batch-64-small", "batch", 1024, 4, 64, 10, 4, 10_000, nprob=64),
        # constant gradients of a population over many cases
        _case("grad-2048x65536", "grad", 2048, 4, 96, 5, 8, 65_536, xhi=5.0),
        # a few Adam steps on the constants of many small problems
        _case("constants-24-small", "constants", 512, 4, 64, 8, 4, 6_000, nprob=24, xhi=5.0),
        # selection and variation of a large population of long programs
        _case("vary-262144", "vary", 262_144, 4, 256, 10, 4, 64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["eval", "eval", "generation", "generation", "score", "predict", "batch", "grad", "constants",
                       "vary"])
    nvars, K = rng.randint(1, 12), rng.choice([0, 2, 4, 8])
    Lmax = rng.choice([16, 24, 32, 57, 64, 96, 128, 200, 256])
    Lmin, ops, gens = rng.randint(1, 8), rng.choice([6, 6, 12]), rng.choice([0, 4, 8])
    xlo, xhi = rng.choice([(1.0, 10.0), (1.0, 5.0), (-3.0, 3.0)])
    nodes = 2.0e10  # programs x mean length x cases, at most
    if path == "vary":
        return _case("", path, _log(rng, 256, 262_144), Lmin, Lmax, nvars, K, 64, ops=ops)
    if path in ("batch", "constants"):
        n = rng.randint(4, 64 if path == "batch" else 24)
        return _case("", path, _log(rng, 64, 1024), Lmin, min(Lmax, 64), nvars, max(K, 2), _log(rng, 400, 10_000),
                     ops=ops, xlo=xlo, xhi=xhi, nprob=n)
    P = _log(rng, 32, 8192)
    N = max(257, min(_log(rng, 400, 200_000), int(nodes / (P * 0.5 * Lmax))))
    if path == "grad":
        return _case("", path, min(P, 2048), Lmin, min(Lmax, 128), nvars, max(K, 2), min(N, 65_536), ops=ops, xlo=xlo,
                     xhi=xhi)
    if path == "predict":
        return _case("", path, min(P, 1024), Lmin, Lmax, nvars, K, min(N, 50_000), ops=ops, xlo=xlo, xhi=xhi,
                     gens=gens)
    kind = rng.choice([0, 1]) if path == "score" else rng.choice([MSE, CORR, BOTH])
    return _case("", path, P, Lmin, Lmax, nvars, K, N, kind, ops=ops, xlo=xlo, xhi=xhi, gens=gens)


# ---------------------------------------------------------------- populations
def _rand_int(g, n, size):
    return (torch.rand(size, generator=g, device=DEV) * n).long().clamp_(max=max(n - 1, 0))


def _random_programs(g, P, Lmin, Lmax, nvars, K, ops):
    """Random walks on the stack depth: a class uniform over those allowed, a token uniform inside it."""
    L = Lmin + _rand_int(g, Lmax - Lmin + 1, P)
    prog = torch.zeros((P, Lmax), dtype=torch.uint8, device=DEV)
    d = torch.zeros(P, dtype=torch.long, device=DEV)
    for t in range(Lmax):
        r = L - t
        allowed = torch.stack([d <= r - 1, (d >= 1) & (d <= r), (d >= 2) & (d <= r + 1)], 1)
        cls = torch.rand((P, 3), generator=g, device=DEV).masked_fill_(~allowed, -1.0).argmax(1)
        q = _rand_int(g, nvars + K, P)
        term = torch.where(q < nvars, 16 + q, 32 + q - nvars)
        tok = torch.where(cls == 0, term, torch.where(cls == 1, 4 + _rand_int(g, ops, P), _rand_int(g, 4, P)))
        prog[:, t] = torch.where(r > 0, tok, 0).to(torch.uint8)
        d += torch.where(r > 0, 1 - cls, 0)
    return prog, L


def _effects(prog, L):
    t = torch.arange(prog.shape[1], device=DEV)
    e = (prog >= 16).int() - (prog < 4).int()
    return torch.where(t < L[:, None], e, 0)


def _values(prog, L, c, X):
    """Outputs of every program on a few cases, all programs in step."""
    P, Lmax = prog.shape
    stack = torch.zeros((P, Lmax // 2 + 3, X.shape[1]), device=DEV)
    rows, d = torch.arange(P, device=DEV), torch.zeros(P, dtype=torch.long, device=DEV)
    eff = _effects(prog, L).long()
    for t in range(Lmax):
        v = prog[:, t].long()
        live = t < L
        b, a = stack[rows, (d - 1).clamp(min=0)], stack[rows, (d - 2).clamp(min=0)]
        term = torch.where((v >= 32)[:, None], c.gather(1, (v - 32).clamp(0, c.shape[1] - 1)[:, None]),
                           X[(v - 16).clamp(0, X.shape[0] - 1)])
        out = torch.where((v >= 16)[:, None], term, b)
        for tok, f in _FUNCTIONS.items():
            m = (v == tok)[:, None]
            out = torch.where(m, f(a, b) if tok < 4 else f(b), out)
        d = d + torch.where(live, eff[:, t], 0)
        at = (d - 1).clamp(min=0)
        stack[rows, at] = torch.where(live[:, None], out, stack[rows, at])
    return stack[:, 0]


def _divide(a, b):
    near = b.abs() <= 1e-3
    return torch.where(near, 1.0, a / torch.where(near, 1.0, b))


def _logarithm(x):
    near = x.abs() <= 1e-3
    return torch.where(near, 0.0, torch.where(near, 1.0, x).abs().log())


_FUNCTIONS = {
    0: torch.add, 1: torch.sub, 2: torch.mul, 3: _divide, 4: torch.sin, 5: torch.cos,
    6: lambda x: x.clamp(-80.0, 80.0).exp(), 7: _logarithm, 8: lambda x: x.abs().sqrt(), 9: torch.square,
    10: lambda x: _divide(torch.ones_like(x), x), 11: torch.tan, 12: torch.asin, 13: torch.acos, 14: torch.atan,
    15: torch.tanh}


def _breed(g, prog, L, c, X, y):
    """One generation: tournaments of four on 1 - r^2 over the cases given, subtree crossover of nine in ten, a new
    constant now and then."""
    P, Lmax = prog.shape
    v = _values(prog, L, c, X).double()
    dv, dy = v - v.mean(1, True), (y - y.mean()).double()
    r2 = (dv @ dy) ** 2 / ((dv * dv).sum(1) * (dy * dy).sum())
    fit = torch.where(torch.isfinite(r2), 1.0 - r2, 1.0)
    pick = []
    for _ in range(2):
        cand = _rand_int(g, P, (P, 4))
        pick.append(cand.gather(1, fit[cand].argmin(1, True))[:, 0])
    A, B = pick
    eff = _effects(prog, L)
    after = eff.cumsum(1)
    before = after - eff

    def span(par, point):  # first token of the subtree that ends at `point`
        root = after[par].gather(1, point[:, None]) - 1
        t = torch.arange(Lmax, device=DEV)
        return torch.where((before[par] == root) & (t <= point[:, None]), t, -1).amax(1)

    a = (torch.rand(P, generator=g, device=DEV) * L[A]).long().clamp(max=Lmax - 1)
    b = (torch.rand(P, generator=g, device=DEV) * L[B]).long().clamp(max=Lmax - 1)
    sa, sb = span(A, a), span(B, b)
    n = L[A] - (a - sa + 1) + (b - sb + 1)
    cross = (torch.rand(P, generator=g, device=DEV) < 0.9) & (n <= Lmax)
    q = torch.arange(Lmax, device=DEV)[None, :]
    nb = (b - sb + 1)[:, None]
    from_b = (q >= sa[:, None]) & (q < sa[:, None] + nb)
    at_a = torch.where(q < sa[:, None], q, q - nb + (a - sa + 1)[:, None]).clamp(0, Lmax - 1)
    at_b = (q - sa[:, None] + sb[:, None]).clamp(0, Lmax - 1)
    child = torch.where(from_b, prog[B].gather(1, at_b), prog[A].gather(1, at_a))
    child = torch.where(cross[:, None], child, prog[A])
    length = torch.where(cross, n, L[A])
    child = torch.where(q < length[:, None], child, 0).to(torch.uint8)
    new_c = c[A].clone()
    if c.shape[1]:
        k = _rand_int(g, c.shape[1], (P, 1))
        move = (torch.rand((P, 1), generator=g, device=DEV) - 0.5) * (torch.rand((P, 1), generator=g, device=DEV) < 0.1)
        new_c.scatter_add_(1, k, move)
    return child, length, new_c


def _problem(g, P, Lmin, Lmax, nvars, K, N, ops, xlo, xhi, gens):
    ldx = (N + 3) // 4 * 4
    X = torch.rand((nvars, ldx), generator=g, device=DEV) * (xhi - xlo) + xlo
    w = torch.rand(4, generator=g, device=DEV) * 4.0 - 2.0
    x = [X[j % nvars, :N] for j in range(4)]
    y = w[0] * x[0] * x[1] + w[1] * torch.sin(x[2]) + w[2] * x[3] / (1.0 + x[1] * x[1]) + w[3]
    y = (y + 0.01 * y.std() * torch.randn(N, generator=g, device=DEV)).contiguous()
    prog, L = _random_programs(g, P, min(Lmin, Lmax), Lmax, nvars, K, ops)
    c = torch.rand((P, K), generator=g, device=DEV) * 10.0 - 5.0
    for _ in range(gens):
        prog, L, c = _breed(g, prog, L, c if K else torch.zeros((P, 1), device=DEV), X[:, :48], y[:48])
        c = c[:, :K]
    return dict(prog=prog.contiguous(), len=L.int(), c=c.contiguous(), X=X, y=y, N=N, nvars=nvars)


def _inputs(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 13)
    a = [case[k] for k in ("P", "Lmin", "Lmax", "nvars", "K", "N", "ops", "xlo", "xhi", "gens")]
    if case["nprob"] == 1:
        p = _problem(g, *a)
        if case["path"] == "score":  # one invalid target in a hundred
            bad = torch.rand(case["N"], generator=g, device=DEV) < 0.01
            p["y"] = torch.where(bad, math.nan, p["y"])
        return [p]
    out = []  # sizes spread below the case's own, the same for every seed
    for i in range(case["nprob"]):
        u, v, w = ((i * s) % 1.0 for s in (0.618034, 0.754878, 0.569840))
        out.append(_problem(g, max(64, int(case["P"] ** (0.6 + 0.4 * u))), case["Lmin"],
                            max(4, int(case["Lmax"] * (0.1 + 0.9 * v))), 1 + int(w * case["nvars"]), case["K"],
                            max(316, int(case["N"] ** (0.63 + 0.37 * v * u + 0.2 * (1 - v) * w))), *a[6:9], 0))
    return out


# ---------------------------------------------------------------- the calls
def prepare(case, seed):
    probs = _inputs(case, seed)
    p, path = probs[0], case["path"]
    s = dict(case=case, p=p, probs=probs, ctx=sr.Context(0), seed=seed)
    empty = lambda shape, dt: torch.empty(shape, dtype=dt, device=DEV)  # noqa: E731
    P, K = case["P"], case["K"]
    if path in ("generation", "vary"):
        s["var"] = sr.var_cfg(max_subtree=min(8, case["Lmax"]), unary_ops=case["ops"])
        s["fit"] = empty((2, P) if path == "generation" and case["kind"] == BOTH else (P,), torch.float64)
        s["parents"] = empty((P, 2), torch.int32)
        s["next"] = (empty((P, case["Lmax"]), torch.uint8), empty(P, torch.int32),
                     empty((P, K), torch.float32) if K else None)
        if path == "vary":
            g = torch.Generator(device=DEV)
            g.manual_seed(int(seed) + 1)
            s["fit"].copy_(torch.rand(P, generator=g, device=DEV, dtype=torch.float64))
    elif path in ("eval", "score"):
        s["fit"] = empty((2, P) if path == "eval" and case["kind"] == BOTH else (P,), torch.float64)
        s["counts"] = empty((P, 2), torch.int32)
        s["flags"] = empty(P, torch.int32)
    elif path == "predict":
        s["yhat"] = empty((P, case["N"]), torch.float32)
    elif path == "grad":
        s["mse"], s["dconst"] = empty(P, torch.float64), empty((P, K), torch.float64)
    elif path in ("batch", "constants"):
        rows = sum(q["prog"].shape[0] for q in probs)
        s["fit"] = empty(2 * rows if path == "batch" else rows, torch.float64)
        s["c"], s["dc"] = empty((rows, K), torch.float32), empty((rows, K), torch.float64)
        s["m"], s["v"] = torch.zeros_like(s["dc"]), torch.zeros_like(s["dc"])
        s["c0"] = torch.cat([q["c"] for q in probs])
        s["list"], s["tables"], at, out = [], [], 0, 0
        for i, q in enumerate(probs):
            n = q["prog"].shape[0]
            c = s["c"][at:at + n]
            if path == "batch":
                kind = (MSE, CORR, BOTH)[i % 3]
                f = s["fit"][out:out + (2 if kind == BOTH else 1) * n]
                out += f.numel()
                s["list"].append(sr.make_problem(q["prog"], q["len"], q["c"], q["X"], q["y"], q["N"], kind, fitness=f))
            else:
                dc = s["dc"][at:at + n]
                s["list"].append(sr.make_grad_problem(q["prog"], q["len"], c, q["X"], q["y"], q["N"],
                                                      mse=s["fit"][at:at + n], dconst=dc))
                s["tables"].append((c, dc, s["m"][at:at + n], s["v"][at:at + n]))
            at += n
        if path == "batch":
            s["fit"] = s["fit"][:out]
        s["adam"] = sr.adam_cfg()
    if case["graph"]:  # what a long run of small generations does: one capture, many replays
        run(s)
        torch.cuda.synchronize()
        stream = torch.cuda.Stream()
        s["ctx"].set_stream(stream)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            s["out"] = run(s)
        s["graph"] = graph
    return s


def run(s):
    if "graph" in s:
        s["graph"].replay()
        return s["out"]
    case, p, ctx = s["case"], s["p"], s["ctx"]
    path = case["path"]
    c = p["c"] if case["K"] else None
    if path in ("eval", "generation"):
        sr.sr_eval(ctx, p["prog"], p["len"], c, p["X"], p["y"], p["N"], case["kind"], fitness=s["fit"],
                   prog_flags=s.get("flags"))
        if path == "eval":
            return [s["fit"][0], s["fit"][1], s["flags"]] if case["kind"] == BOTH else [s["fit"], s["flags"]]
    if path in ("generation", "vary"):
        row = s["fit"][1] if path == "generation" and case["kind"] == BOTH else s["fit"]
        sr.sr_select_tournament(ctx, row, 4, 20260312, 3, parents=s["parents"])
        sr.sr_vary(ctx, p["prog"], p["len"], c, s["parents"], p["nvars"], s["var"], 20260312, 3, out=s["next"])
        kids = [t for t in (s["parents"],) + s["next"] if t is not None]
        return kids if path == "vary" else kids + [s["fit"]]
    if path == "score":
        sr.sr_eval_score(ctx, p["prog"], p["len"], c, p["X"], p["y"], p["N"], case["kind"], 1000, score=s["fit"],
                         pair_counts=s["counts"], prog_flags=s["flags"])
        return [s["fit"], s["counts"], s["flags"]]
    if path == "predict":
        return sr.sr_predict(ctx, p["prog"], p["len"], c, p["X"], p["N"], yhat=s["yhat"])
    if path == "batch":
        sr.sr_eval_batched(ctx, s["list"])
        return s["fit"]
    if path == "grad":
        return sr.sr_eval_grad(ctx, p["prog"], p["len"], c, p["X"], p["y"], p["N"], mse=s["mse"], dconst=s["dconst"])
    s["c"].copy_(s["c0"])  # constants: three Adam steps from where the generation left them
    s["m"].zero_()
    s["v"].zero_()
    for t in (1, 2, 3):
        sr.sr_eval_grad_batched(ctx, s["list"])
        sr.sr_adam_step_batched(ctx, s["tables"], t, s["adam"])
    return [s["c"], s["fit"], s["dc"], s["m"], s["v"]]


def work(case):
    """One operation a token and case (three with the gradient); inputs read once, outputs written once."""
    mean = 0.5 * (case["Lmin"] + case["Lmax"])
    P, K, N, n = case["P"], case["K"], case["N"], case["nprob"]
    if n > 1:  # sizes spread below the case's own
        P, N, mean = n * 0.35 * P, 0.25 * N, 0.55 * mean
    pop = P * (mean + 4 + 4 * K)
    data = 4.0 * N * (case["nvars"] + 1) * n
    path = case["path"]
    if path == "vary":
        return {"bytes": 3 * pop + 24 * P, "flops": 8 * P * mean}
    out = 4.0 * P * N if path == "predict" else 16.0 * P + (pop if path == "generation" else 0)
    out += 8.0 * P * K if path in ("grad", "constants") else 0
    passes = 3 if path == "grad" else 9 if path == "constants" else 1
    return {"bytes": pop + data + out, "flops": passes * P * mean * N}


# ---------------------------------------------------------------- the same in 64 bits
def _outputs64(tokens, c, X):
    """One program on every case in FP64; a value that FP32 cannot hold is infinite, as the library documents."""
    st = []
    for v in tokens:
        if v >= 32:
            st.append(c[v - 32])
            continue
        if v >= 16:
            st.append(X[v - 16])
            continue
        b = st.pop()
        r = _FUNCTIONS[v](st.pop(), b) if v < 4 else _FUNCTIONS[v](b)
        if v in (0, 1, 2, 3, 6, 9):
            r = torch.where(r.abs() < FLT_LIMIT, r, r.sign() * math.inf)
        st.append(r)
    return st[0]


def _score64(v, y, kind, M=1000.0):
    """Eq. 2 or Eq. 3 of one program, and its pair counts."""
    vh, vy = torch.isfinite(v), torch.isfinite(y)
    c1, c2 = (vh != vy).sum(), (~vh & ~vy).sum()
    both = vh & vy
    if kind == sr.SR_SCORE_P2P:
        a, b = v.abs(), y.abs()
        top = torch.maximum(a, b)
        q = M * torch.minimum(a, b) / torch.where(top > 0, top, 1.0) - torch.where(v * y < 0, M / 11.0, 0.0)
        return torch.where(both, torch.where(top > 0, q.round(), M), torch.where(vh | vy, -M, M)).sum(), c1, c2
    v, y = v[both], y[both]
    dv, dy = v - v.mean(), y - y.mean()
    r2 = (dv @ dy) ** 2 / ((dv @ dv) * (dy @ dy))
    r2 = torch.where(torch.isfinite(r2), r2.clamp(0.0, 1.0), 0.0)
    return M * r2 * r2 * both.sum() - M * (c1 - c2), c1, c2


def exact(case, seed):
    path, grad = case["path"], case["path"] == "grad"
    tokens = case["P"] * 0.5 * (case["Lmin"] + case["Lmax"]) * (2.5 if grad else 1)
    if path in ("vary", "batch", "constants") or tokens > 290_000 or tokens * case["N"] > 3e10:
        return None
    p = _inputs(case, seed)[0]
    X, y, N = p["X"][:, :case["N"]].double(), p["y"].double(), case["N"]
    mse, corr, dconst, score, yhat = [], [], [], [], []
    dy = y - y.mean()
    for i, (tok, n) in enumerate(zip(p["prog"].tolist(), p["len"].tolist())):
        c = p["c"][i].double()
        v = _outputs64(tok[:n], c.requires_grad_() if grad else c, X)
        v = v.expand(N) if v.dim() == 0 else v
        if path == "predict":
            yhat.append(v)
            continue
        if path == "score":
            score.append(torch.stack([t.double() for t in _score64(v, y, case["kind"])]))
            continue
        m = ((v - y) ** 2).mean()
        if grad:
            d = torch.autograd.grad(m, c, allow_unused=True)[0] if m.requires_grad else None
            dconst.append(torch.zeros_like(c) if d is None else d)
        m = m.detach()
        mse.append(torch.where(m * N < FLT_LIMIT, m, math.inf))
        if not grad:
            dv = v - v.mean()
            r2 = (dv @ dy) ** 2 / ((dv @ dv) * (dy @ dy))
            corr.append(torch.where(torch.isfinite(r2), (1.0 - r2).clamp(0.0, 1.0), 1.0))
    if path == "predict":
        return torch.stack(yhat)
    if path == "score":
        return [torch.stack(score)[:, 0], None, None]
    mse = torch.stack(mse)
    if grad:
        return [mse, torch.stack(dconst)]
    fit = [mse, torch.stack(corr)]
    fit = fit if case["kind"] == BOTH else [fit[1]] if case["kind"] == CORR else [fit[0]]
    if path == "generation":
        return [None] * (4 if case["K"] else 3) + [torch.stack(fit) if case["kind"] == BOTH else fit[0]]
    return fit + [None]
