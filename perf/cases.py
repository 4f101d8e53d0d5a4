"""Timing cases of the engine: what programs have it do, through its public entry points.

Kinds of case
  step      a batch of searches with built-in objectives: `gens` generations of
            `cmaes_step_batch`, then the state of every search read back (a
            driver that looks at its searches every few generations, or
            checkpoints them). With `resume` the pass starts by loading the
            checkpoint, so every pass does the same generation: a scheduler
            that swaps long searches in and out.
  asktell   an external objective: `cmaes_ask`, the caller's function on the
            host, `cmaes_tell`, then the state.
  dgemm     `cmaes_ozaki_dgemm` on device matrices.
  evaluate  `cmaes_evaluate_noalloc` on a device panel of points.

Searches start from a mid-run state: nonzero paths, a moderate step size and a
covariance matrix with a spread, distinct spectrum (the eigenvectors of nearly
equal eigenvalues are arbitrary, so a state that has them has no one answer).
"""
import ctypes
import math

import numpy as np
import torch

import paper_2409_11765_gb300 as eng
from paper_2409_11765_gb300 import workloads as W

PRECISIONS = ("fp64", "tf32", "bf16")
KINDS = {"ellipsoid": W.ELLIPSOID, "rastrigin": W.RASTRIGIN, "sphere": W.SPHERE}
GEN0 = 59  # generations behind a search when it is taken up
STATE = ("m", "ps", "pc", "D", "best_x", "C", "B")


def listed():
    return [
        # the smallest search that is run in earnest: plain CMA-ES on the n = 10
        # ellipsoid, looked at every 20 generations; launches and latency
        dict(name="n10-fp64", kind="step", shape="levels", n=10, lam=10, levels=1, objective="ellipsoid",
             precision="fp64", gens=20, resume=False),
        # K-Distributed at the size of the strategy comparison (n = 40, lambda
        # 12 .. 384), looked at every 10 generations
        dict(name="kdist-n40-tf32", kind="step", shape="levels", n=40, lam=12, levels=6, objective="rastrigin",
             precision="tf32", gens=10, resume=False),
        # the n = 100 benchmark: ten levels, lambda 17 .. 8704, in one batch
        dict(name="kdist-n100-tf32", kind="step", shape="levels", n=100, lam=17, levels=10, objective="rastrigin",
             precision="tf32", gens=10, resume=False),
        # the same batch in plain FP64
        dict(name="kdist-n100-fp64", kind="step", shape="levels", n=100, lam=17, levels=10, objective="rastrigin",
             precision="fp64", gens=4, resume=False),
        # one medium search in FP64
        dict(name="n500-fp64", kind="step", shape="levels", n=500, lam=704, levels=1, objective="rastrigin",
             precision="fp64", gens=1, resume=True),
        # odd sizes, a population that is no multiple of any tile
        dict(name="n333-lam1001-bf16", kind="step", shape="levels", n=333, lam=1001, levels=1, objective="ellipsoid",
             precision="bf16", gens=1, resume=True),
        # the single large search of the configurations
        dict(name="n1000-tf32", kind="step", shape="levels", n=1000, lam=1024, levels=1, objective="ellipsoid",
             precision="tf32", gens=1, resume=True),
        # the large-scale search
        dict(name="n4096-bf16", kind="step", shape="levels", n=4096, lam=8192, levels=1, objective="ellipsoid",
             precision="bf16", gens=1, resume=True),
        # concurrent restarts over uneven searches (n 50 .. 2000, lambda 15 ..
        # 6656): the first 64 shapes of the 256-search benchmark
        dict(name="batch64-tf32", kind="step", shape="uneven", count=64, batch=W.SEED, precision="tf32", gens=1,
             resume=True),
        # a costly external function: one search asked and told from the host
        dict(name="asktell-n200-fp64", kind="asktell", n=200, lam=304, precision="fp64"),
        # the FP64-accurate product on its own
        dict(name="dgemm-1000x1024x2000", kind="dgemm", M=1000, N=1024, K=2000, beta=0.0),
        # points of another component's memory, at the largest population of the n = 100 levels
        dict(name="evaluate-n100", kind="evaluate", n=100, lam=8704, pad=4, objective="rastrigin"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["levels"] * 5 + ["uneven", "uneven", "asktell", "dgemm", "evaluate"])
    precision = rng.choice(PRECISIONS)
    objective = rng.choice(["ellipsoid", "rastrigin", "sphere"])
    if kind == "levels":
        n = _log(rng, 2, 2200)
        if n > 160:  # one search
            return dict(kind="step", shape="levels", n=n, lam=W.default_lambda(n) + _log(rng, 1, 3000), levels=1,
                        objective=objective, precision=precision, gens=1, resume=True)
        return dict(kind="step", shape="levels", n=n, lam=W.default_lambda(n) + rng.randint(0, 5),
                    levels=rng.randint(1, 9), objective=objective, precision=precision, gens=rng.randint(2, 10),
                    resume=False)
    if kind == "uneven":
        return dict(kind="step", shape="uneven", count=rng.randint(6, 48), batch=rng.randrange(1, 1 << 20),
                    precision=rng.choice(("tf32", "bf16", "fp64")), gens=1, resume=True)
    if kind == "asktell":
        return dict(kind="asktell", n=_log(rng, 5, 400), lam=_log(rng, 8, 1500), precision=precision)
    if kind == "dgemm":
        return dict(kind="dgemm", M=_log(rng, 16, 3000), N=_log(rng, 16, 3000), K=_log(rng, 16, 3000),
                    beta=rng.choice([0.0, 0.5]))
    n = _log(rng, 3, 1000)
    pad = rng.randint(0, 5)
    return dict(kind="evaluate", n=n, lam=_log(rng, 8, (1 << 20) // (n + pad)), pad=pad, objective=objective)


def _searches(case):
    """(n, lambda, objective) of every search of a step or asktell case."""
    if case["kind"] == "asktell":
        return [(case["n"], case["lam"], W.SPHERE)]
    if case["shape"] == "uneven":
        return W.batch256_shapes(case["batch"], case["count"])
    return [(case["n"], case["lam"] << k, KINDS[case["objective"]]) for k in range(case["levels"])]


def _cond(n):
    """Condition number of the starting covariance matrix."""
    return 1000.0 if n <= 32 else (30.0 if n <= 400 else 10.0)


def _gen(seed, *stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(np.random.SeedSequence([seed, *stream]).generate_state(1, np.uint64)[0] >> 1))
    return g


def _rotation(n, g):
    q, r = torch.linalg.qr(torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g))
    return q * torch.sign(torch.diagonal(r))


def _inputs(case, seed):
    """Problem and starting state of every search, on the GPU. The searches of
    one dimension share their two rotations; the rest is each one's own."""
    turns, out = {}, []
    for s, (n, lam, obj) in enumerate(_searches(case)):
        if n not in turns:
            g = _gen(seed, 1, n)
            turns[n] = (_rotation(n, g), _rotation(n, g))
        Q, B = turns[n]
        g = _gen(seed, 2, s)

        def rand(k):
            return torch.rand(k, dtype=torch.float64, device="cuda", generator=g)

        def randn(k):
            return torch.randn(k, dtype=torch.float64, device="cuda", generator=g)

        # eigenvalues 1 .. cond on a jittered geometric grid, ascending
        t = (torch.arange(n, dtype=torch.float64, device="cuda") + 0.4 * rand(n)) / n
        d2 = _cond(n) ** t
        # columns in the engine's canonical sign: the largest entry positive
        big = torch.gather(B, 0, B.abs().argmax(0, keepdim=True))
        B = B * torch.sign(big)
        C = (B * d2) @ B.T
        C = 0.5 * (C + C.T)
        lamdiag = 1e6 ** (torch.arange(n, dtype=torch.float64, device="cuda") / max(1, n - 1))
        out.append(dict(n=n, lam=lam, obj=obj, Q=Q, B=B, C=C, D=torch.sqrt(d2), lamdiag=lamdiag,
                        xstar=8.0 * rand(n) - 4.0, m=4.0 * rand(n) - 2.0, ps=0.5 * randn(n), pc=0.1 * randn(n),
                        sigma=0.1 + 0.3 * float(rand(1)), sigma0=2.0))
    return out


def _pinned(x):
    return torch.empty(x.shape, dtype=x.dtype, pin_memory=True).copy_(x)


class _Searches:
    """A handle, its checkpoint and the pinned buffers that its state is read into."""

    def __init__(self, case, seed):
        self.case, self.h = case, None
        inp = _inputs(case, seed)
        self.ns = [x["n"] for x in inp]
        opt = eng.cmaes_default_options(precision=PRECISIONS.index(case["precision"]), max_restarts=255, ipop_double=0)
        self.h = eng.cmaes_create_batch(self.ns, [x["lam"] for x in inp], [x["m"].cpu().numpy() for x in inp],
                                        [x["sigma0"] for x in inp], seed, opt)
        hosts = {}  # one host copy of what searches share
        self.saved = []
        for s, x in enumerate(inp):
            if case["kind"] == "step":
                if x["n"] not in hosts:
                    hosts[x["n"]] = x["Q"].T.contiguous().cpu().numpy().T
                eng.cmaes_set_problem(self.h, s, x["obj"], hosts[x["n"]] if x["obj"] != W.SPHERE else None,
                                      x["lamdiag"].cpu().numpy(), x["xstar"].cpu().numpy())
            d = dict(n=x["n"], lam=x["lam"], sigma=x["sigma"], gen=GEN0)
            d.update({k: _pinned(x[k]).numpy() for k in ("m", "ps", "pc", "D")})
            d["C"] = _pinned(x["C"]).numpy().T
            d["B"] = _pinned(x["B"].T.contiguous()).numpy().T  # column-major, as the engine keeps it
            eng.cmaes_set_state(self.h, s, d)
            if case.get("resume"):
                self.saved.append(d)
        size = {k: [n * n if k in "CB" else n for n in self.ns] for k in STATE}
        self.out = {k: torch.zeros(sum(v), dtype=torch.float64, pin_memory=True) for k, v in size.items()}
        self.out["sigma"] = torch.zeros(len(self.ns), dtype=torch.float64)
        self.out["best_f"] = torch.zeros(len(self.ns), dtype=torch.float64)
        self.read = []
        at = {k: 0 for k in STATE}
        for s, n in enumerate(self.ns):
            st = eng.cmaes_state()
            for k in STATE:
                setattr(st, k, ctypes.cast(self.out[k].data_ptr() + 8 * at[k], ctypes.POINTER(ctypes.c_double)))
                at[k] += size[k][s]
            self.read.append(st)

    def state(self):
        """Every search's state: each quantity of all searches one after the other, matrices column-major."""
        for s, st in enumerate(self.read):
            if eng.lib().cmaes_get_state(self.h, s, ctypes.byref(st)):
                raise RuntimeError(eng.cmaes_last_error(self.h))
            self.out["sigma"][s] = st.sigma
            self.out["best_f"][s] = st.best_f
        return dict(self.out)

    def __del__(self):
        if self.h:
            eng.cmaes_destroy(self.h)
            self.h = None


def _host_function(n):
    """The caller's function: a shifted quartic sum."""
    shift = np.linspace(-1.0, 1.0, n)[:, None]

    def f(X):
        r = X - shift
        r *= r
        return r.sum(axis=0) + 0.1 * np.einsum("ij,ij->j", r, r)

    return f


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("step", "asktell"):
        return _Searches(case, seed)
    g = _gen(seed, 3)
    if kind == "dgemm":
        # rows of uneven scale, as the engine's own operands have them; column-major
        def matrix(r, c):
            scale = torch.exp(2.0 * torch.randn(r, dtype=torch.float64, device="cuda", generator=g))
            return torch.randn(c, r, dtype=torch.float64, device="cuda", generator=g) * scale

        return dict(case=case, A=matrix(case["M"], case["K"]), B=matrix(case["K"], case["N"]),
                    C=matrix(case["M"], case["N"]))
    n, ld = case["n"], case["n"] + case["pad"]
    X = 4.0 * torch.randn(case["lam"], ld, dtype=torch.float64, device="cuda", generator=g)
    return dict(case=case, X=X, Q=_rotation(n, g).T.contiguous(),
                lamdiag=1e6 ** (torch.arange(n, dtype=torch.float64, device="cuda") / max(1, n - 1)),
                xstar=8.0 * torch.rand(n, dtype=torch.float64, device="cuda", generator=g) - 4.0,
                f=torch.zeros(case["lam"], dtype=torch.float64, device="cuda"))


def run(state):
    case = state.case if isinstance(state, _Searches) else state["case"]
    kind = case["kind"]
    if kind == "step":
        for s, d in enumerate(state.saved):
            eng.cmaes_set_state(state.h, s, d)
        eng.cmaes_step_batch(state.h, case["gens"])
        return state.state()
    if kind == "asktell":
        n = case["n"]
        X = eng.cmaes_ask(state.h, 0, n)
        f = _host_function(n)(X)
        eng.cmaes_tell(state.h, 0, f)
        return dict(state.state(), X=X.T, f=f, best_f=None)
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "dgemm":
        M, N, K = case["M"], case["N"], case["K"]
        eng.cmaes_ozaki_dgemm(M, N, K, 1.0, state["A"].data_ptr(), M, state["B"].data_ptr(), K, case["beta"],
                              state["C"].data_ptr(), M, stream)
        return state["C"]
    n, ld = case["n"], case["n"] + case["pad"]
    eng.cmaes_evaluate_noalloc(KINDS[case["objective"]], n, case["lam"], state["X"].data_ptr(), ld,
                               state["Q"].data_ptr(), n, state["lamdiag"].data_ptr(), state["xstar"].data_ptr(),
                               state["f"].data_ptr(), stream)
    return state["f"]


def work(case):
    """Flops: the sampling and objective products, the rank-mu sum, 10/3 n^3 per
    decomposition. Bytes: the state once in and once out, the instance once."""
    kind = case["kind"]
    if kind == "dgemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 8 * (M * K + K * N + M * N * (2 if case["beta"] else 1)), "flops": 2 * M * N * K}
    if kind == "evaluate":
        n, lam = case["n"], case["lam"]
        turned = case["objective"] != "sphere"
        return {"bytes": 8 * (n * lam + lam + (n * n if turned else 0)), "flops": (2 * n * n if turned else 3 * n) * lam}
    gens = case.get("gens", 1)
    flops = bytes_ = 0
    for n, lam, obj in _searches(case):
        turned = obj != W.SPHERE
        flops += gens * (2 * n * n * lam * (2 if turned else 1) + (lam // 2) * n * (n + 1))
        flops += sum(10 * n ** 3 // 3 for g in range(gens) if (GEN0 + g + 1) % _constants(n, lam)["g_eig"] == 0)
        bytes_ += 8 * (4 * n * n + (n * n if turned else 0) + 10 * n)
        if kind == "asktell":
            bytes_ += 8 * lam * (n + 1)
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------------------
# The same results in 64 bits, from torch alone.
# ---------------------------------------------------------------------------
def _constants(n, lam):
    """Hansen's tutorial defaults (arXiv:1604.00772), positive weights."""
    mu = lam // 2
    w = math.log((lam + 1) / 2.0) - np.log(np.arange(1, mu + 1, dtype=np.float64))
    w = w / w.sum()
    mueff = 1.0 / float(np.sum(w * w))
    c1 = 2.0 / ((n + 1.3) ** 2 + mueff)
    cmu = min(1.0 - c1, 2.0 * (mueff - 2.0 + 1.0 / mueff) / ((n + 2.0) ** 2 + mueff))
    cs = (mueff + 2.0) / (n + mueff + 5.0)
    return dict(mu=mu, w=w, mueff=mueff, c1=c1, cmu=cmu, cs=cs, cc=(4.0 + mueff / n) / (n + 4.0 + 2.0 * mueff / n),
                ds=1.0 + 2.0 * max(0.0, math.sqrt((mueff - 1.0) / (n + 1.0)) - 1.0) + cs,
                chin=math.sqrt(n) * (1.0 - 1.0 / (4.0 * n) + 1.0 / (21.0 * n * n)),
                g_eig=max(1, math.floor(1.0 / ((c1 + cmu) * n * 10.0))))


def _normals(seed, search, gen, n, lam):
    """n x lam normals: Philox4x32-10 (Salmon et al., SC'11) at counter (i >> 1,
    k, gen, search << 8), key = seed, and Box-Muller on 52-bit uniforms."""
    mask = 0xFFFFFFFF
    p = torch.arange((n + 1) // 2, dtype=torch.int64, device="cuda")[:, None]
    k = torch.arange(lam, dtype=torch.int64, device="cuda")[None, :]
    c = [p.expand(-1, lam), k.expand(p.shape[0], -1), torch.full_like(p * k, gen), torch.full_like(p * k, search << 8)]
    k0, k1 = seed & mask, (seed >> 32) & mask
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # modulo 2^64
        c = [((b >> 32) & mask) ^ c[1] ^ k0, b & mask, ((a >> 32) & mask) ^ c[3] ^ k1, a & mask]

    def uniform(a, b):
        return ((((a << 20) | (b >> 12)) & ((1 << 52) - 1)).double() + 0.5) * 2.0 ** -52

    radius = torch.sqrt(-2.0 * torch.log(uniform(c[0], c[1])))
    angle = (2.0 * math.pi) * uniform(c[2], c[3])
    return torch.stack([radius * torch.cos(angle), radius * torch.sin(angle)], 1).reshape(-1, lam)[:n]


def _value(kind, X, Q, lamdiag, xstar):
    R = X - xstar[:, None]
    if kind == W.SPHERE:
        return (R * R).sum(0)
    U = Q @ R
    if kind == W.ELLIPSOID:
        return (lamdiag[:, None] * U * U).sum(0)
    return 10.0 * X.shape[0] + (U * U - 10.0 * torch.cos(2.0 * math.pi * U)).sum(0)


def _generation(x, seed, search, f_of):
    """One generation of search state x, in place; returns its points and values."""
    n, lam = x["n"], x["lam"]
    p = _constants(n, lam)
    Z = _normals(seed, search, x["gen"], n, lam)
    Y = x["B"] @ (x["D"][:, None] * Z)
    X = x["m"][:, None] + x["sigma"] * Y
    f = f_of(X)
    sel = torch.sort(f, stable=True).indices[: p["mu"]]
    if float(f[sel[0]]) < x["best_f"]:
        x["best_f"], x["best_x"] = float(f[sel[0]]), X[:, sel[0]].clone()
    w = torch.from_numpy(p["w"]).cuda()
    Ys = Y[:, sel]
    yw, zw = Ys @ w, Z[:, sel] @ w
    x["m"] = x["m"] + x["sigma"] * yw
    x["ps"] = (1.0 - p["cs"]) * x["ps"] + math.sqrt(p["cs"] * (2.0 - p["cs"]) * p["mueff"]) * (x["B"] @ zw)
    psn = float(torch.linalg.norm(x["ps"]))
    left = psn / math.sqrt(1.0 - (1.0 - p["cs"]) ** (2 * (x["gen"] + 1)))
    hs = 1.0 if left < (1.4 + 2.0 / (n + 1.0)) * p["chin"] else 0.0
    x["pc"] = (1.0 - p["cc"]) * x["pc"] + hs * math.sqrt(p["cc"] * (2.0 - p["cc"]) * p["mueff"]) * yw
    keep = 1.0 - p["c1"] - p["cmu"] + p["c1"] * (1.0 - hs) * p["cc"] * (2.0 - p["cc"])
    C = keep * x["C"] + p["c1"] * torch.outer(x["pc"], x["pc"]) + p["cmu"] * ((Ys * w) @ Ys.T)
    x["C"] = 0.5 * (C + C.T)
    x["sigma"] *= math.exp((p["cs"] / p["ds"]) * (psn / p["chin"] - 1.0))
    x["gen"] += 1
    if x["gen"] % p["g_eig"] == 0:
        e, B = torch.linalg.eigh(x["C"])
        x["B"], x["D"] = B * torch.sign(torch.gather(B, 0, B.abs().argmax(0, keepdim=True))), torch.sqrt(e)
    return X, f


def exact(case, seed):
    kind = case["kind"]
    if kind == "dgemm":
        s = prepare(case, seed)
        return s["B"] @ s["A"] + case["beta"] * s["C"]  # transposed: column-major
    if kind == "evaluate":
        s = prepare(case, seed)
        return _value(KINDS[case["objective"]], s["X"][:, : case["n"]].T, s["Q"].T, s["lamdiag"], s["xstar"])
    mixed = case["precision"] != "fp64"
    if kind == "step" and (case["shape"] == "uneven" or mixed and case["gens"] > 1):
        return None  # too long; and the ranks of many generations in 16 or 19 bits are not those of 64
    inp = _inputs(case, seed)
    for s, x in enumerate(inp):
        x.update(gen=GEN0, best_f=math.inf, best_x=None)
        if kind == "asktell":
            host = _host_function(x["n"])
            X, f = _generation(x, seed, s, lambda X: torch.from_numpy(host(X.cpu().numpy())).cuda())
        else:
            for _ in range(case["gens"]):
                _generation(x, seed, s, lambda X: _value(x["obj"], X, x["Q"], x["lamdiag"], x["xstar"]))
    out = {k: torch.cat([(x[k].T if k in "CB" else x[k]).reshape(-1) for x in inp]) for k in STATE}
    out["sigma"] = torch.tensor([x["sigma"] for x in inp], dtype=torch.float64)
    out["best_f"] = torch.tensor([x["best_f"] for x in inp], dtype=torch.float64)
    if mixed:  # what the choice among near-equal candidates decides has no one value
        out.update(B=None, best_x=None, best_f=None, ps=None, pc=None)
    if kind == "asktell":
        out.update(best_f=None, X=X.T if not mixed else None, f=f if not mixed else None)
    return out
