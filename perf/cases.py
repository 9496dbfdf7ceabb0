"""The work that a program using this package has it do, as cases that can be timed.

Each case is one pass through the public entry points of ``paper_2201_06958_gb300.tdb`` on
the synthetic streams of ``paper_2201_06958_gb300.synth`` (the shapes of the paper's
workloads and the ranges around them):

* ``step``      a saved state is loaded and a window of the stream pushed: every push is one
                step of the compressor (difference, projection, update, error), and the
                compressed form (core and bases) is read back at the end, as an in-situ
                consumer stores it.  The window runs forth and back in time over a ring of
                six input buffers, so that it ends on the snapshot it began with.
* ``reinit``    the truncated HOSVD of a new snapshot (the rank rule's re-initialisation and
                the start of every stream), and the field it stands for.
* ``reconstruct``  the field of a compressed state, written out.
* ``batch``     many small tensors of uneven sizes and ranks, stepped together.
* ``estimator`` one training iteration of the learned error estimator.
"""

import functools
import math

import numpy as np
import torch

from paper_2201_06958_gb300 import synth, tdb

RING = (0, 1, 2, 3, 2, 1)        # times of the ring's buffers, in steps of the stream
DEV = "cuda"


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the paper's stochastic stream at its size: the largest three-mode step, error every step
        {"name": "step_stochastic", "kind": "step", "field": "stochastic",
         "stream": 1003, "n1": 256, "n2": 128, "n3": 512,
         "cap": 20, "precision": "bf16", "error_mode": "exact", "integrator": "euler", "rounds": 2},
        # the channel flow: four modes, an odd second mode, error on a schedule
        {"name": "step_channel", "kind": "step", "field": "channel",
         "stream": 1004, "n1": 192, "n2": 129, "n3": 192,
         "cap": 30, "precision": "bf16", "error_mode": "every_k", "integrator": "euler", "rounds": 2},
        # the reactive flow: an ordinary step, few species
        {"name": "step_reactive", "kind": "step", "field": "reactive",
         "stream": 1002, "n1": 512, "n2": 256, "n3": 12,
         "cap": 16, "precision": "bf16", "error_mode": "exact", "integrator": "euler", "rounds": 2},
        # the same stream as the first without reduced precision anywhere
        {"name": "step_stochastic_fp32", "kind": "step", "field": "stochastic",
         "stream": 1003, "n1": 256, "n2": 128, "n3": 512,
         "cap": 20, "precision": "fp32", "error_mode": "exact", "integrator": "euler", "rounds": 1},
        # the Runge function of the paper's first example, double precision throughout
        {"name": "step_runge_fp64", "kind": "step", "field": "runge",
         "stream": 1005, "n1": 126, "n2": 126, "n3": 126,
         "cap": 8, "precision": "fp64", "error_mode": "exact", "integrator": "euler", "rounds": 1},
        # the smallest calls: two grouped modes, 6144 points, the learned estimator gating the error
        {"name": "step_dbo", "kind": "step", "field": "dbo", "stream": 1006, "n1": 32, "n2": 16, "n3": 12,
         "cap": 8, "precision": "bf16", "error_mode": "mlp", "integrator": "euler", "rounds": 2},
        # a second-order integrator in double precision on a small cube
        {"name": "step_analytic_heun", "kind": "step", "field": "analytic",
         "stream": 1001, "n1": 64, "n2": 64, "n3": 64,
         "cap": 4, "precision": "fp64", "error_mode": "exact", "integrator": "heun", "rounds": 1},
        # re-initialisation of the large stream: three long modes
        {"name": "reinit_stochastic", "kind": "reinit", "field": "stochastic",
         "stream": 1003, "n1": 256, "n2": 128, "n3": 512,
         "cap": 20, "precision": "bf16"},
        # re-initialisation in double precision
        {"name": "reinit_runge_fp64", "kind": "reinit", "field": "runge",
         "stream": 1005, "n1": 126, "n2": 126, "n3": 126,
         "cap": 8, "precision": "fp64"},
        # decompression of a four-mode field
        {"name": "reconstruct_channel", "kind": "reconstruct", "field": "channel",
         "stream": 1004, "n1": 192, "n2": 129, "n3": 192,
         "cap": 30, "precision": "fp32"},
        # many tensors at once, uneven sizes 32..128 and ranks 4..24
        {"name": "batch_64", "kind": "batch", "members": 64, "sizes": 1005, "low": 32, "high": 128,
         "precision": "bf16", "pushes": 8},
        # training of the estimator on a full trace
        {"name": "estimator_8192", "kind": "estimator", "rows": 8192},
    ]


def _spread(rng, lo, hi):
    """A whole number, spread over the logarithm of lo..hi."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_field(rng, fields):
    f = rng.choice(fields)
    n = {"stochastic": lambda: (_spread(rng, 32, 256), _spread(rng, 24, 128), _spread(rng, 24, 512)),
         "channel": lambda: (_spread(rng, 32, 192), _spread(rng, 17, 129), _spread(rng, 24, 192)),
         "reactive": lambda: (_spread(rng, 48, 512), _spread(rng, 32, 256), rng.randint(8, 16)),
         "dbo": lambda: (_spread(rng, 24, 251), _spread(rng, 12, 76), rng.randint(10, 23)),
         "runge": lambda: (_spread(rng, 24, 126),) * 3,
         "analytic": lambda: (_spread(rng, 16, 80),) * 3}[f]()
    cap = {"stochastic": rng.randint(8, 20), "channel": rng.randint(8, 30), "reactive": rng.randint(6, 16),
           "dbo": rng.randint(4, 8), "runge": rng.randint(4, 8), "analytic": 4}[f]
    prec = "fp64" if f in ("runge", "analytic") else rng.choice(("bf16", "bf16", "bf16", "fp32"))
    return {"field": f, "stream": rng.randint(1, 9999), "n1": n[0], "n2": n[1], "n3": n[2], "cap": cap,
            "precision": prec}


def draw(rng):
    kind = rng.choice(("step", "step", "step", "step", "reinit", "reinit", "reconstruct", "batch", "estimator"))
    if kind == "step":
        c = _draw_field(rng, ("stochastic", "channel", "reactive", "dbo", "runge", "analytic"))
        modes = ("exact", "every_k", "none") + (() if c["precision"] == "fp64" else ("mlp",))
        return {"kind": kind, **c, "error_mode": rng.choice(modes),
                "integrator": rng.choice(("euler", "euler", "euler", "heun")), "rounds": 1}
    if kind == "reinit":
        return {"kind": kind, **_draw_field(rng, ("stochastic", "channel", "reactive", "dbo", "runge"))}
    if kind == "reconstruct":
        return {"kind": kind, **_draw_field(rng, ("stochastic", "channel", "reactive", "dbo", "runge"))}
    if kind == "batch":
        return {"kind": kind, "members": _spread(rng, 2, 32), "sizes": rng.randint(0, 9999),
                "low": rng.randint(24, 48), "high": rng.randint(64, 128),
                "precision": rng.choice(("bf16", "fp32")), "pushes": 4}
    return {"kind": kind, "rows": _spread(rng, 64, 8192)}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

@functools.lru_cache(maxsize=64)
def _stream(f, n, stream, cap):
    """A stream and the ranks it is compressed at: those that keep gamma_th of its first
    snapshot's energy in every mode, within the cap."""
    size = {"stochastic": dict(nx=n[0], ny=n[1], ns=n[2]), "channel": dict(nx=n[0], ny=n[1], nz=n[2]),
            "reactive": dict(nx=n[0], ny=n[1], ns=n[2]), "dbo": dict(nx=n[0], ny=n[1], ns=n[2]),
            "runge": dict(n=n[0]), "analytic": dict(n=n[0])}[f]
    wl = synth.make_workload("reactive_dbo" if f == "dbo" else f, seed=stream, **size)
    X, r = _weighted(wl.snapshot(0, device=DEV, dtype=torch.float64), wl.weights), []
    for m in range(X.ndim):
        lam, _ = _spectrum(X, m)
        r.append(min(cap, wl.dims[m], int((lam.cumsum(0) < wl.gamma_th / 100 * lam.sum()).sum()) + 1))
    for _ in r:
        r = [min(x, int(np.prod(r[:m] + r[m + 1:]))) for m, x in enumerate(r)]
    return wl, r


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _snapshots(case, seed, times):
    """The stream, its ranks and snapshots from the time on that the seed gives."""
    wl, r = _stream(case["field"], (case["n1"], case["n2"], case["n3"]), case["stream"], case["cap"])
    k0 = 250.0 * (seed % 1000003) / 1000003
    return wl, r, [wl.snapshot(k0 + t, device=DEV, dtype=_dtype(case)) for t in times]


class _Member:
    """One tensor of a batch: more smooth separable terms than the rank kept, advected."""

    def __init__(self, sizes, rng, low, high):
        self.dims = [int(v) for v in sizes.integers(low, high + 1, size=3)]
        self.rank = [min(int(sizes.integers(4, 25)), min(self.dims) - 4)] * 3
        J = self.rank[0] + 4
        self.k = [rng.permutation(J) + 1 for _ in range(3)]
        self.ph, self.vel = rng.uniform(0, 2 * np.pi, (3, J)), rng.uniform(-1, 1, (3, J))
        self.amp = 10.0 ** (-2.0 * np.arange(J) / J)
        self.weights = [synth.uniform_unit(d) for d in self.dims]

    def snapshot(self, t):
        f = [torch.cos(torch.as_tensor(np.pi * self.k[m][:, None] * np.linspace(0, 1, self.dims[m])[None, :]
                                       + (self.ph[m] + self.vel[m] * t)[:, None], device=DEV)) for m in range(3)]
        a = torch.as_tensor(self.amp, device=DEV)
        return torch.einsum("j,jc,jb,ja->cba", a, f[2], f[1], f[0]).to(torch.float32).contiguous()


def _members(case, seed):
    sizes, rng = np.random.default_rng(case["sizes"]), np.random.default_rng(seed)
    return [_Member(sizes, rng, case["low"], case["high"]) for _ in range(case["members"])]


def _estimator_params(seed):
    """A fitted estimator as a program installs it: small weights, wide feature ranges."""
    n = tdb.load().tdb_mlp_param_count()
    rng = np.random.default_rng(seed)
    p = np.empty(n + 18, dtype=np.float32)
    p[:n] = 0.05 * rng.standard_normal(n)
    p[n:n + 8], p[n + 8:n + 16], p[n + 16], p[n + 17] = -3.0, 4.0, 0.0, 0.01
    return p


def prepare(case, seed):
    kind = case["kind"]
    if kind == "estimator":
        g = torch.Generator(device=DEV).manual_seed(seed)
        n = tdb.load().tdb_mlp_param_count()
        X = torch.randn(case["rows"], 8, generator=g, device=DEV)
        t = torch.tanh(X[:, 0] - 0.5 * X[:, 2]) + 0.1 * torch.randn(case["rows"], generator=g, device=DEV)
        return {"kind": kind, "step": 10, "X": X, "t": t.contiguous(),
                "params": 0.15 * torch.randn(n, generator=g, device=DEV),
                "m": 1e-3 * torch.randn(n, generator=g, device=DEV),
                "v": 1e-5 * (0.1 + torch.rand(n, generator=g, device=DEV))}
    if kind == "batch":
        ctx, blobs, slots = [], [], []
        for mb in _members(case, seed):
            V = [mb.snapshot(1e-3 * k) for k in range(2)]
            core, U = _hosvd(V[0].double(), mb.weights, mb.rank)
            c = tdb.TDB(mb.dims, mb.rank, mb.rank, weights=mb.weights, precision=case["precision"], error_mode="exact")
            c.init_from_factors(_host(core), [_host(u) for u in U], V[0])
            c.set_input_slots(V[0], V[1])
            ctx.append(c)
            blobs.append(c.save_state())
            slots.append(V)
        return {"kind": kind, "ctx": ctx, "blobs": blobs, "slots": slots, "batch": tdb.Batch(ctx),
                "pushes": case["pushes"]}
    ring = RING if kind == "step" else (0, 3)
    wl, r, V = _snapshots(case, seed, ring)
    core, U = _hosvd(V[0].double(), wl.weights, r)
    mlp = case.get("error_mode") == "mlp"
    c = tdb.TDB(wl.dims, r, r, weights=wl.weights, eps_th=1e3 if mlp else 0.0, gamma_th=100.0,
                precision=case["precision"], error_mode=case.get("error_mode", "exact"),
                error_every={"every_k": 4, "mlp": 20}.get(case.get("error_mode"), 1),
                integrator=case.get("integrator", "euler"))
    if kind == "reinit":
        c.init(V[0])
        return {"kind": kind, "c": c, "V": V, "out": torch.empty_like(V[0])}
    c.init_from_factors(_host(core), [_host(u) for u in U], V[0])
    if kind == "reconstruct":
        return {"kind": kind, "c": c, "V": V, "out": torch.empty_like(V[0])}
    if mlp:
        c.estimator_params(_estimator_params(seed), gate=0.9)
    return {"kind": kind, "c": c, "V": V, "blob": c.save_state(), "rounds": case["rounds"]}


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def run(state):
    kind = state["kind"]
    if kind == "step":
        c, V = state["c"], state["V"]
        c.load_state(state["blob"], V[0])
        eps, dv = [], []
        for _ in range(state["rounds"]):
            for k in range(1, len(V) + 1):
                info = c.push(V[k % len(V)])
                eps.append(info["eps"])
                dv.append(info["dv_norm"])
        core, U = c.factors()
        kept = np.float64 if c.precision == "fp64" else np.float32     # stored as wide as the stream
        return {"core": core.astype(kept), "U": [u.astype(kept) for u in U], "eps": np.array(eps, kept),
                "dv": np.array(dv, kept)}
    if kind == "reinit":
        state["c"].reinit(state["V"][1])
        return state["c"].reconstruct(state["out"])
    if kind == "reconstruct":
        return state["c"].reconstruct(state["out"])
    if kind == "batch":
        for c, blob, V in zip(state["ctx"], state["blobs"], state["slots"]):
            c.load_state(blob, V[0])
        eps = []
        for k in range(state["pushes"]):
            eps.append([info["eps"] for info in state["batch"].push((k + 1) % 2)])
        f = [c.factors() for c in state["ctx"]]
        return {"core": np.concatenate([x[0].ravel() for x in f]).astype(np.float32),
                "U": np.concatenate([u.ravel() for x in f for u in x[1]]).astype(np.float32),
                "eps": np.array(eps, np.float32)}
    state["step"] += 1
    loss, grad = tdb.mlp_loss_grad(state["params"], state["X"], state["t"])
    tdb.mlp_adam_step(state["params"], grad, state["m"], state["v"], state["step"], 1e-3)
    return {"loss": loss, "grad": grad, "params": state["params"], "m": state["m"], "v": state["v"]}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def _dims(case):
    n = [case["n1"], case["n2"], case["n3"]]
    return [n[0] * n[1], n[2]] if case["field"] == "dbo" else n + [3] if case["field"] == "channel" else n


def work(case):
    kind = case["kind"]
    if kind == "estimator":
        # X and t read; parameters, moments and gradient read or written; three products per layer
        n = 8 * 64 + 64 + 64 * 64 + 64 + 64 + 1
        return {"bytes": 4 * (9 * case["rows"] + 7 * n), "flops": 6 * n * case["rows"]}
    if kind == "batch":
        mean = (case["low"] + case["high"]) / 2
        s = case["members"] * mean ** 3
        return {"bytes": case["pushes"] * 8 * s, "flops": case["pushes"] * s * 2 * 14 * 3}
    dims = _dims(case)
    s = 1
    for d in dims:
        s *= d
    esz = 8 if case["precision"] == "fp64" else 4
    r = [min(case["cap"], d) for d in dims]
    if kind == "step":
        # both snapshots once a stage; the first contractions of modes 1 and 2, and U_1 in the exact error
        pushes, stages = case["rounds"] * len(RING), 2 if case["integrator"] == "heun" else 1
        evals = {"exact": pushes, "every_k": pushes // 4}.get(case["error_mode"], 0)
        return {"bytes": pushes * 2 * esz * s * stages,
                "flops": pushes * stages * 2 * s * (r[0] + r[1]) + evals * 2 * s * r[0]}
    if kind == "reinit":
        # the snapshot in, the field out; the symmetric Grams, the core and the field
        return {"bytes": 2 * esz * s, "flops": s * sum(min(d, s // d) for d in dims) + 2 * 2 * s * r[0]}
    return {"bytes": esz * s, "flops": 2 * s * r[-1]}


# ---------------------------------------------------------------------------
# The same results in 64 bits
# ---------------------------------------------------------------------------

def _host(x):
    return x.cpu().numpy()


def _logical(V):
    return V.permute(*reversed(range(V.ndim)))


def _unfold(X, n):
    return X.movedim(n, 0).reshape(X.shape[n], -1)


def _mode(X, M, n):
    """X x_n M^T, M of shape (size of mode n, new size)."""
    return torch.tensordot(X, M, dims=([n], [0])).movedim(-1, n)


def _weighted(V, weights):
    X = _logical(V)
    for n, w in enumerate(weights):
        X = X * torch.as_tensor(w, device=V.device).sqrt().reshape([-1 if m == n else 1 for m in range(X.ndim)])
    return X


def _spectrum(X, n):
    """Eigenvalues (descending) and eigenvectors of the mode-n Gram, from its shorter side."""
    B = _unfold(X, n)
    short = B.shape[0] <= B.shape[1] or B.shape[0] <= 1024
    lam, q = torch.linalg.eigh(B @ B.T if short else B.T @ B)
    lam, q = lam.flip(0).clamp(min=0), q.flip(1)
    if not short:
        q = (B @ q) / lam.sqrt().clamp(min=1e-300)
    return lam, q * torch.sign(q.gather(0, q.abs().argmax(0, keepdim=True)))


def _hosvd(V, weights, ranks):
    X, U = _weighted(V, weights), []
    for n in range(X.ndim):
        U.append(_spectrum(X, n)[1][:, :ranks[n]] / torch.as_tensor(weights[n], device=V.device).sqrt()[:, None])
    core = _logical(V)
    for n, u in enumerate(U):
        core = _mode(core, torch.as_tensor(weights[n], device=V.device)[:, None] * u, n)
    return core.contiguous(), [u.contiguous() for u in U]


def _field(core, U):
    for n, u in enumerate(U):
        core = _mode(core, u.T, n)
    return core


def _increment(T, U, W, dV):
    A = [w[:, None] * u for w, u in zip(W, U)]
    dU = []
    for n in range(dV.ndim):
        Y = dV
        for m in sorted((m for m in range(dV.ndim) if m != n), key=lambda m: U[m].shape[1] / U[m].shape[0]):
            Y = _mode(Y, A[m], m)
        if n == 0:
            dS = _mode(Y, A[0], 0)
        Tn = _unfold(T, n)
        X = torch.linalg.solve(Tn @ Tn.T, (_unfold(Y, n) @ Tn.T).T).T
        dU.append(X - U[n] @ (A[n].T @ X))
    return dS, dU


def _step(T, U, W, Vp, Vn, integrator):
    dS, dU = _increment(T, U, W, Vn - Vp)
    if integrator == "heun":
        dS2, dU2 = _increment(T + dS, [u + d for u, d in zip(U, dU)], W, Vn - Vp)
        dS, dU = (dS + dS2) / 2, [(a + b) / 2 for a, b in zip(dU, dU2)]
    T, U = T + dS, [u + d for u, d in zip(U, dU)]
    for n, u in enumerate(U):
        L = torch.linalg.cholesky(u.T @ (W[n][:, None] * u))
        U[n] = torch.linalg.solve_triangular(L, u.T, upper=False).T
        T = _mode(T, L, n)
    return T, U


def _wnorm(X, W):
    X = X * X
    for n, w in enumerate(W):
        X = X * w.reshape([-1 if m == n else 1 for m in range(X.ndim)])
    return float(X.sum().sqrt())


def _window(V, weights, ranks, pushes, integrator):
    """The steps of a window over the ring V (storage order): core, bases, errors, norms."""
    W = [torch.as_tensor(w, device=V[0].device) for w in weights]
    T, U = _hosvd(V[0].double(), weights, ranks)
    eps, dv, Vp = [], [], _logical(V[0]).double()
    for k in range(1, pushes + 1):
        Vn = _logical(V[k % len(V)]).double()
        T, U = _step(T, U, W, Vp, Vn, integrator)
        eps.append(_wnorm(Vn - _field(T, U), W))
        dv.append(_wnorm(Vn - Vp, W))
        Vp = Vn
    return T, U, eps, dv


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        wl, r, V = _snapshots(case, seed, RING)
        T, U, eps, dv = _window(V, wl.weights, r, case["rounds"] * len(RING), case["integrator"])
        return {"core": T.contiguous(), "U": [u.contiguous() for u in U],
                "eps": np.array(eps) if case["error_mode"] == "exact" else None, "dv": np.array(dv)}
    if kind in ("reinit", "reconstruct"):
        wl, r, V = _snapshots(case, seed, (0, 3))
        core, U = _hosvd(V[1 if kind == "reinit" else 0].double(), wl.weights, r)
        return _logical(_field(core, U)).contiguous()
    if kind == "batch":
        got = []
        for mb in _members(case, seed):
            V = [mb.snapshot(1e-3 * k) for k in range(2)]
            got.append(_window(V, mb.weights, mb.rank, case["pushes"], "euler"))
        return {"core": np.concatenate([_host(g[0].contiguous()).ravel() for g in got]),
                "U": np.concatenate([_host(u.contiguous()).ravel() for g in got for u in g[1]]),
                "eps": np.array([g[2] for g in got]).T.copy()}
    s = prepare(case, seed)
    P, X, t = s["params"].double().requires_grad_(True), s["X"].double(), s["t"].double()
    H = 64
    o = np.cumsum([0, H * 8, H, H * H, H, H, 1])
    W1, b1, W2, b2, w3, b3 = (P[o[i]:o[i + 1]] for i in range(6))
    h = torch.tanh(X @ W1.reshape(H, 8).T + b1)
    h = torch.tanh(h @ W2.reshape(H, H).T + b2)
    loss = ((h @ w3 + b3 - t) ** 2).mean()
    (g,) = torch.autograd.grad(loss, P)
    k = s["step"] + 1
    m, v = 0.9 * s["m"].double() + 0.1 * g, 0.999 * s["v"].double() + 0.001 * g * g
    new = P.detach() - 1e-3 * (m / (1 - 0.9 ** k)) / ((v / (1 - 0.999 ** k)).sqrt() + 1e-8)
    return {"loss": loss.detach().reshape(1), "grad": g, "params": new, "m": m, "v": v}
