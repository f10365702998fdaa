"""Performance cases: the work that users of this library have it do.

Every case goes through the public entry points (`Solver`, `MPCGSolve`,
`SQP`) on seeded synthetic LQ subproblems with the shapes of the repository's
own configurations: the Kuka arm (nx = 14, nu = 7, 32..512 knots), the
large-state robot (nx = 36, nu = 12, 64..256 knots), float32 and float64,
diagonal and dense cost blocks, one instance and ragged batches.

Solves are warm-started as in a receding-horizon controller: lambda0 is the
solution of the same subproblem with 1 % noise on each entry.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2309_08079_gb300.autograd import MPCGSolve
from paper_2309_08079_gb300.nmpc import SQP
from paper_2309_08079_gb300.solver import LQTensors, Solver, make_opts

DEV = "cuda"
KUKA = dict(nx=14, nu=7, dt=0.01, q_lo=1.0, q_hi=10.0)      # the arm of the measured workloads
LARGE = dict(nx=36, nu=12, dt=0.005, q_lo=0.1, q_hi=100.0)  # the large-state robot: needs refinement


def listed():
    return [
        # one short-horizon control step, the whole call: launches and latency
        dict(name="solve_n32", kind="solve", **KUKA, B=1, N_lo=32, N_hi=32, dtype="float32", tol=1e-6, refine=1),
        # the library's headline workload: formation and PCG of one long horizon, real time
        dict(name="pcg_n512", kind="pcg", **KUKA, B=1, N_lo=512, N_hi=512, dtype="float32", tol=1e-6, refine=0),
        # a double-precision reference solve of an odd horizon
        dict(name="pcg_f64_n101", kind="pcg", **KUKA, B=1, N_lo=101, N_hi=101, dtype="float64", tol=1e-12, refine=0),
        # one control step of the large-state robot, refined once
        dict(name="pcg_nx36_n64", kind="pcg", **LARGE, B=1, N_lo=64, N_hi=64, dtype="float32", tol=1e-6, refine=1),
        # many independent arms or sampled scenarios at once, ragged horizons
        dict(name="batch_256", kind="pcg", **KUKA, B=256, N_lo=32, N_hi=512, dtype="float32", tol=1e-6, refine=0),
        # the large-state batch, refined once
        dict(name="batch_nx36_160", kind="pcg", **LARGE, B=160, N_lo=64, N_hi=256, dtype="float32", tol=1e-6, refine=1),
        # differentiable solve in a training step: forward and adjoint
        dict(name="train_64x128", kind="train", **KUKA, B=64, N_lo=128, N_hi=128, dtype="float32", tol=1e-6, refine=1),
        # the layers around the PCG alone: S+, gamma, Phi^-1 and dz ...
        dict(name="condense_256", kind="condense", **KUKA, B=256, N_lo=32, N_hi=512, dtype="float32", dense=False),
        # ... of the large-state robot (its packed blocks included) ...
        dict(name="condense_nx36_256", kind="condense", **LARGE, B=256, N_lo=64, N_hi=256, dtype="float32", dense=False),
        # ... with general SPD cost blocks
        dict(name="condense_dense_32", kind="condense", **KUKA, B=32, N_lo=32, N_hi=256, dtype="float32", dense=True),
        # ... and of the outer loop: linearisation and line search of a batch of arms
        dict(name="nlp_64x128", kind="nlp", nx=14, nu=7, B=64, N=128),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "pcg", "pcg36", "pcg64", "batch", "batch36", "train", "condense", "condense36", "dense", "nlp"])
    if kind in ("solve", "pcg"):
        n = _log(rng, 20, 512)
        return dict(kind=kind, **KUKA, B=1, N_lo=n, N_hi=n, dtype="float32", tol=1e-6, refine=int(kind == "solve"))
    if kind == "pcg36":
        n = _log(rng, 16, 128)
        return dict(kind="pcg", **LARGE, B=1, N_lo=n, N_hi=n, dtype="float32", tol=1e-6, refine=1)
    if kind == "pcg64":
        n = _log(rng, 20, 160)
        return dict(kind="pcg", **KUKA, B=1, N_lo=n, N_hi=n, dtype="float64", tol=1e-12, refine=0)
    if kind == "batch":
        lo = _log(rng, 16, 128)
        return dict(kind="pcg", **KUKA, B=_log(rng, 5, 256), N_lo=lo, N_hi=_log(rng, lo + 1, 512), dtype="float32", tol=1e-6, refine=0)
    if kind == "batch36":
        lo = rng.randint(40, 100)
        return dict(kind="pcg", **LARGE, B=_log(rng, 24, 160), N_lo=lo, N_hi=rng.randint(lo + 1, 256), dtype="float32", tol=1e-6, refine=1)
    if kind == "train":
        n = _log(rng, 24, 200)
        return dict(kind="train", **KUKA, B=_log(rng, 4, 64), N_lo=n, N_hi=n + rng.randint(0, 40), dtype="float32", tol=1e-6, refine=1)
    if kind == "nlp":
        return dict(kind="nlp", nx=14, nu=7, B=_log(rng, 2, 128), N=_log(rng, 24, 300))
    lo = _log(rng, 16, 128)
    shape = LARGE if kind == "condense36" else KUKA
    b = _log(rng, 1, 32) if kind == "dense" else _log(rng, 1, 256)
    return dict(kind="condense", **shape, B=b, N_lo=lo, N_hi=lo + rng.randint(1, 128), dtype="float32", dense=kind == "dense")


# --------------------------------------------------------------------------
# Inputs.  A concatenated ragged batch in the library's layouts; knot `prev[j]`
# and `prev[j] + 1` are the ends of control j.
# --------------------------------------------------------------------------
def _horizons(case):
    """The same for every seed, so that a case's work does not change with it."""
    rng = np.random.default_rng([case["B"], case["N_lo"], case["N_hi"]])
    return rng.integers(case["N_lo"], case["N_hi"] + 1, size=case["B"]).astype(np.int64)


def _layout(Ns):
    ko = np.zeros(len(Ns) + 1, dtype=np.int64)
    ko[1:] = np.cumsum(Ns)
    keep = np.ones(int(ko[-1]), dtype=bool)
    keep[ko[1:] - 1] = False
    return ko, torch.as_tensor(np.nonzero(keep)[0], device=DEV)


def _lq(case, seed):
    """Kuka-shaped LQ data on the GPU, rounded to the case's type."""
    nx, nu, dt, h = case["nx"], case["nu"], case["dt"], case["nx"] // 2
    Ns = _horizons(case)
    ko, prev = _layout(Ns)
    K, J = int(ko[-1]), int(ko[-1]) - len(Ns)
    g = torch.Generator(device=DEV).manual_seed(seed)
    n = lambda *s: torch.randn(*s, generator=g, device=DEV, dtype=torch.float64)  # noqa: E731
    u = lambda lo, hi, *s: lo + (hi - lo) * torch.rand(*s, generator=g, device=DEV, dtype=torch.float64)  # noqa: E731
    A = torch.eye(nx, device=DEV, dtype=torch.float64).repeat(J, 1, 1)
    A[:, :h, h:] = dt * torch.eye(h, device=DEV, dtype=torch.float64)
    A[:, h:, :h] = 0.5 * dt * n(J, h, h)
    A[:, h:, h:] += 0.5 * dt * n(J, h, h)
    L = n(J, h, h)
    B = torch.zeros(J, nx, nu, device=DEV, dtype=torch.float64)
    B[:, h:] = dt * (L @ L.mT + 0.1 * torch.eye(h, device=DEV, dtype=torch.float64))[:, :, :nu]
    d = dict(A=A, B=B, Qd=u(case["q_lo"], case["q_hi"], K, nx), Rd=u(0.01, 0.1, J, nu), q=n(K, nx), r=n(J, nu), c=n(K, nx))
    if case.get("dense"):
        W, V = n(K, nx, nx), n(J, nu, nu)
        d["Q"] = (0.5 / nx) * W @ W.mT + torch.diag_embed(d["Qd"])
        d["R"] = (0.01 / nu) * V @ V.mT + torch.diag_embed(d["Rd"])
        d["Qd"], d["Rd"] = (torch.diagonal(d[f], dim1=1, dim2=2) for f in ("Q", "R"))
    t = torch.float64 if case.get("dtype") == "float64" else torch.float32
    d = {f: v.to(t).contiguous() for f, v in d.items()}
    return d, Ns, ko, prev, g


# --------------------------------------------------------------------------
# The same quantities in plain 64-bit torch.
# --------------------------------------------------------------------------
def _mv(M, x):
    return (M @ x.unsqueeze(-1)).squeeze(-1)


def _ginv(d):
    """x -> Q^-1 x, u -> R^-1 u and the inverse blocks."""
    if "Q" in d:
        Qi, Ri = torch.linalg.inv_ex(d["Q"])[0], torch.linalg.inv_ex(d["R"])[0]
    else:
        Qi, Ri = torch.diag_embed(1 / d["Qd"]), torch.diag_embed(1 / d["Rd"])
    return Qi, Ri


def _schur(d, prev):
    Qi, Ri = _ginv(d)
    A, B = d["A"], d["B"]
    Sd = Qi.clone()
    AQ = A @ Qi[prev]
    Sd[prev + 1] += AQ @ A.mT + B @ Ri @ B.mT
    gamma = d["c"] - _mv(Qi, d["q"])
    gamma[prev + 1] += _mv(A, _mv(Qi, d["q"])[prev]) + _mv(B, _mv(Ri, d["r"]))
    return Sd, -AQ, gamma


def _ctv(d, prev, v):
    """C^T v as (state part, control part)."""
    x = v.clone()
    x[prev] -= _mv(d["A"].mT, v[prev + 1])
    return x, -_mv(d["B"].mT, v[prev + 1])


def _c(d, prev, x, u):
    """C (x, u)."""
    y = x.clone()
    y[prev + 1] -= _mv(d["A"], x[prev]) + _mv(d["B"], u)
    return y


def _recover(d, prev, lam, q, r):
    x, u = _ctv(d, prev, lam)
    if "Q" in d:
        Qi, Ri = _ginv(d)
        return _mv(Qi, x - q), _mv(Ri, u - r)
    return (x - q) / d["Qd"], (u - r) / d["Rd"]


def _direct(Sd, So, rhs, Ns, ko):
    """Block-tridiagonal Cholesky-like elimination, all instances at once."""
    B, N, nx = len(Ns), int(max(Ns)), Sd.shape[-1]
    k = torch.arange(N, device=DEV)
    n = torch.as_tensor(Ns, device=DEV)[:, None]
    at = torch.as_tensor(ko[:-1], device=DEV)[:, None] + k
    on, oc = k < n, k < n - 1
    eye = torch.eye(nx, device=DEV, dtype=torch.float64)
    D = torch.where(on[..., None, None], Sd[at.clamp(max=len(Sd) - 1)], eye)
    b = torch.where(on[..., None], rhs[at.clamp(max=len(Sd) - 1)], 0.0)
    at_c = (at - torch.arange(B, device=DEV)[:, None]).clamp(max=max(len(So) - 1, 0))
    O = torch.where(oc[..., None, None], So[at_c], 0.0) if len(So) else torch.zeros_like(D)
    inv, y = [], []
    for i in range(N):
        M, v = D[:, i], b[:, i]
        if i:
            F = O[:, i - 1] @ inv[-1]
            M, v = M - F @ O[:, i - 1].mT, v - _mv(F, y[-1])
        inv.append(torch.linalg.inv_ex(M)[0])
        y.append(v)
    x = [None] * N
    for i in reversed(range(N)):
        x[i] = _mv(inv[i], y[i] if i == N - 1 else y[i] - _mv(O[:, i].mT, x[i + 1]))
    return torch.stack(x, 1)[on]


def _exact_solution(d, Ns, ko, prev):
    d = {f: v.double() for f, v in d.items()}
    Sd, So, gamma = _schur(d, prev)
    lam = _direct(Sd, So, -gamma, Ns, ko)
    return (d, Sd, So, lam) + _recover(d, prev, lam, d["q"], d["r"])


# --------------------------------------------------------------------------
# The synthetic arm of the SQP loop.
# --------------------------------------------------------------------------
def _tracking(case, seed):
    """Model, tracking problems at their straight-line guess, and a step (dX,
    dU, lambda) of the size that the first iterations take."""
    nx, nu, N, B, h = case["nx"], case["nu"], case["N"], case["B"], case["nx"] // 2
    rng = np.random.default_rng(seed)
    f = lambda a: np.ascontiguousarray(a, dtype=np.float32)  # noqa: E731
    L = rng.normal(size=(h, h))
    wq = rng.uniform(1.0, 10.0, nx)
    model = SimpleNamespace(nx=nx, nu=nu, dt=0.01, P=f((L @ L.T + 0.1 * np.eye(h))[:, :nu]), damp=f(rng.uniform(0.1, 1.0, h)),
                            stiff=f(rng.uniform(1.0, 10.0, h)), wq=f(wq), wr=f(rng.uniform(0.01, 0.1, nu)), wf=f(10.0 * wq))
    trks, steps = [], []
    for _ in range(B):
        xs = rng.normal(0.0, 0.5, nx)
        a, w, ph = rng.uniform(0.2, 1.0, h), rng.uniform(0.5, 3.0, h), rng.uniform(0.0, 2 * np.pi, h)
        t = np.arange(N)[:, None] * model.dt
        xref = np.concatenate([a * np.sin(w * t + ph), a * w * np.cos(w * t + ph)], axis=1)
        X = xs + np.linspace(0.0, 1.0, N)[:, None] * (xref[-1] - xs)
        trks.append(SimpleNamespace(N=N, xs=f(xs), xref=f(xref), X=f(X), U=f(rng.normal(0.0, 0.5, (N - 1, nu)))))
        steps.append((0.5 * (xref - X), rng.normal(0.0, 0.5, (N - 1, nu)), 20.0 * rng.normal(size=(N, nx))))
    return model, trks, [f(np.concatenate(v)) for v in zip(*steps)]


# --------------------------------------------------------------------------
# prepare, run
# --------------------------------------------------------------------------
def _opts(case):
    # a correction only has to shrink an error at the float32 floor of S+, which is ten times higher for the large state
    return make_opts(tol=case["tol"], refine_tol=(1e-4 if case["nx"] == LARGE["nx"] else 1e-3) if case["refine"] else 0.0)


def prepare(case, seed):
    s = Solver(DEV)
    st = SimpleNamespace(case=dict(case), s=s)
    if case["kind"] == "nlp":
        model, trks, steps = _tracking(case, seed)
        st.sqp = SQP(s, model, trks)
        st.start = [t.clone() for t in (st.sqp.X, st.sqp.U)]
        for t, v in zip((st.sqp.dx, st.sqp.du, st.sqp.lam), steps):
            t.copy_(torch.as_tensor(v))
        return st
    d, Ns, ko, prev, g = _lq(case, seed)
    K, nx, nu, t = int(ko[-1]), case["nx"], case["nu"], d["A"].dtype
    batched = case["B"] > 1
    st.lq = LQTensors(nx, nu, int(max(Ns)), **d, knot_off=torch.as_tensor(ko.astype(np.int32), device=DEV) if batched else None,
                      nb=len(Ns), total=K, Ns=Ns if batched else None)
    st.schur = s.alloc_schur(st.lq)
    if case["kind"] == "condense":
        # multipliers that change slowly from knot to knot, as A ~ I makes them
        st.lam = torch.cumsum(torch.randn(K, nx, generator=g, device=DEV, dtype=t), 0)
        st.dx, st.du = torch.empty(K, nx, dtype=t, device=DEV), torch.empty(max(K - len(Ns), 1), nu, dtype=t, device=DEV)
        return st
    lam = _exact_solution(d, Ns, ko, prev)[3]
    st.lam0 = (lam * (1 + 0.01 * torch.randn(K, nx, generator=g, device=DEV, dtype=torch.float64))).to(t)
    st.opts = _opts(case)
    st.lam, st.ws = torch.empty_like(st.lam0), s.alloc_workspace(st.lq)
    st.stats, st.rstats = s.alloc_stats(len(Ns)), s.alloc_stats(len(Ns))
    if case["kind"] == "train":
        st.w = torch.randn(K, nx, generator=g, device=DEV, dtype=t)
        st.leaves = [getattr(st.lq, f).requires_grad_(True) for f in LQTensors.FIELDS]
        st.cfg = dict(solver=s, nx=nx, nu=nu, N=st.lq.N, knot_off=st.lq.knot_off, nb=len(Ns), total=K, opts=st.opts,
                      workspace=st.ws, refine=case["refine"])
    return st


def run(st):
    s, kind = st.s, st.case["kind"]
    if kind == "nlp":
        for t, t0 in zip((st.sqp.X, st.sqp.U), st.start):
            t.copy_(t0)
        st.sqp.linearize()
        st.sqp.line_search()
        return dict(X=st.sqp.X, U=st.sqp.U, alpha=st.sqp.alpha_index, **{f: getattr(st.sqp.lq, f) for f in LQTensors.FIELDS})
    if kind == "condense":
        s.form(st.lq, st.schur)
        s.recover_step(st.lq, st.lam, st.dx, st.du)
        sc = st.schur
        return dict(Sd=sc.Sd, So=sc.So, Pd=sc.Pd, Po=sc.Po, gamma=sc.gamma, info=sc.info, dx=st.dx, du=st.du)
    if kind == "train":
        lam, dx, du, _ = MPCGSolve.apply(*st.leaves, st.lam0, st.cfg)
        loss = (dx * dx).sum() + (du * du).sum() + (st.w * lam).sum()
        grads = torch.autograd.grad(loss, st.leaves)
        return dict(lam=lam, dx=dx, du=du, **{"g" + f: x for f, x in zip(LQTensors.FIELDS, grads)})
    status = st.stats.view(torch.int32).view(st.lq.nb, -1)[:, 1]
    if kind == "solve":
        lam, dx, du, _, _ = s.solve(st.lq, st.lam0.clone(), st.opts, st.schur, st.stats, st.ws, refine=st.case["refine"])
        return dict(lam=lam, dx=dx, du=du, status=status)
    st.lam.copy_(st.lam0)
    s.form(st.lq, st.schur)
    s.pcg_solve(st.lq, st.schur, st.lam, st.opts, st.stats, st.ws)
    for _ in range(st.case["refine"]):
        s.refine_step(st.lq, st.schur, st.lam, st.opts, st.rstats, st.ws)
    return dict(lam=st.lam, status=status)


# --------------------------------------------------------------------------
# work, exact
# --------------------------------------------------------------------------
def _iters(case, n):
    """PCG iterations that such a solve takes, roughly (the longest horizon's
    share counts: one instance's 1e-6 solve takes about 30 sqrt(N))."""
    return 30.0 * math.sqrt(n) * math.log10(1 / case["tol"]) / 6.0


def work(case):
    nx, nu = case["nx"], case["nu"]
    Ns = np.full(case["B"], case["N"]) if case["kind"] == "nlp" else _horizons(case)
    K = float(Ns.sum())
    J = K - len(Ns)
    e = 8 if case.get("dtype") == "float64" else 4
    lq = J * (nx * nx + nx * nu + 2 * nu) + K * 3 * nx
    if case.get("dense"):
        lq += K * (nx * nx - nx) + J * (nu * nu - nu)
    blocks = 2 * (K + J) * nx * nx + K * nx           # Sd, So, Pd, Po, gamma
    form = J * (2 * nx * nx * (nx + nu) + 4 * nx ** 3) + K * 2 * nx ** 3
    dz = K * nx + J * nu
    prod = lambda n: (6 * n - 4) * nx * nx * 2.0      # one S+ and one Phi^-1 product  # noqa: E731
    if case["kind"] == "condense":
        return dict(bytes=e * (lq + blocks + K * nx + dz), flops=form + J * 2 * nx * (nx + nu))
    if case["kind"] == "nlp":
        return dict(bytes=e * (lq + 5 * K * nx + 3 * J * nu), flops=9 * J * (nx * nu + 10 * nx))
    pcg = sum(_iters(case, n) * prod(n) for n in Ns)
    out = K * nx * 2 + (0 if case["kind"] == "pcg" else dz)
    if case["kind"] == "train":
        return dict(bytes=e * (2 * lq + out + K * nx), flops=form + 2 * pcg)
    return dict(bytes=e * (lq + out), flops=form + pcg * (1.4 if case["refine"] else 1.0))


def _exact_nlp(case, seed):
    model, trks, (dX, dU, lam) = _tracking(case, seed)
    f = lambda a: torch.as_tensor(a, dtype=torch.float64, device=DEV)  # noqa: E731
    P, damp, stiff, wq, wr, wf = (f(getattr(model, n)) for n in ("P", "damp", "stiff", "wq", "wr", "wf"))
    nx, nu, N, B, h, dt = case["nx"], case["nu"], case["N"], case["B"], case["nx"] // 2, model.dt
    X, U, xref, xs = (torch.stack([f(getattr(t, n)) for t in trks]) for n in ("X", "U", "xref", "xs"))
    dX, dU, lam = f(dX).view(B, N, nx), f(dU).view(B, N - 1, nu), f(lam).view(B, -1)
    w = torch.cat([wq.expand(N - 1, nx), wf[None]])

    def defects(x, u):
        p, v = x[:, :-1, :h], x[:, :-1, h:]
        vn = v + dt * (u @ P.mT - damp * v - stiff * torch.sin(p))
        return torch.cat([x[:, :1] - xs[:, None], x[:, 1:] - torch.cat([p + dt * vn, vn], -1)], 1)

    def merit(x, u, mu):
        cost = 0.5 * (w * (x - xref) ** 2).sum((1, 2)) + 0.5 * (wr * u * u).sum((1, 2))
        return cost + mu * defects(x, u).abs().sum((1, 2))

    p = X[:, :-1, :h].reshape(-1, h)
    eye = torch.eye(h, dtype=torch.float64, device=DEV)
    vp, vv = torch.diag_embed(-dt * stiff * torch.cos(p)), (eye - dt * torch.diag(damp)).expand(len(p), h, h)
    A = torch.cat([torch.cat([eye + dt * vp, dt * vv], 2), torch.cat([vp, vv], 2)], 1)
    lq = dict(A=A, B=torch.cat([dt * dt * P, dt * P]).repeat(len(p), 1, 1), Qd=w.repeat(B, 1), Rd=wr.repeat(len(p), 1),
              q=(w * (X - xref)).reshape(-1, nx), r=(wr * U).reshape(-1, nu), c=defects(X, U).reshape(-1, nx))
    mu = 1.1 * lam.abs().amax(1).clamp(min=1.0)
    m = torch.stack([merit(X + 0.5 ** a * dX, U + 0.5 ** a * dU, mu) for a in range(9)])
    al = (0.5 ** m.argmin(0).double())[:, None, None]
    return dict(X=(X + al * dX).reshape(-1, nx), U=(U + al * dU).reshape(-1, nu), alpha=None, **lq)


def exact(case, seed):
    if case["kind"] == "nlp":
        return _exact_nlp(case, seed)
    d, Ns, ko, prev, g = _lq(case, seed)
    K, nx, t = int(ko[-1]), case["nx"], d["A"].dtype
    if case["kind"] == "condense":
        lam = torch.cumsum(torch.randn(K, nx, generator=g, device=DEV, dtype=t), 0).double()
        d = {f: v.double() for f, v in d.items()}
        Sd, So, gamma = _schur(d, prev)
        Pd = torch.linalg.inv_ex(Sd)[0]
        dx, du = _recover(d, prev, lam, d["q"], d["r"])
        return dict(Sd=Sd, So=So, Pd=Pd, Po=-Pd[prev + 1] @ So @ Pd[prev], gamma=gamma, info=None, dx=dx, du=du)
    d, Sd, So, lam, dx, du = _exact_solution(d, Ns, ko, prev)
    if case["kind"] == "pcg":
        return dict(lam=lam, status=None)
    if case["kind"] == "solve":
        return dict(lam=lam, dx=dx, du=du, status=None)
    torch.randn(K, nx, generator=g, device=DEV, dtype=torch.float64)  # lambda0's noise
    w = torch.randn(K, nx, generator=g, device=DEV, dtype=t).double()
    bx, bu = 2 * dx, 2 * du  # gradients of the loss by dx and du
    mu = _direct(Sd, So, w + _c(d, prev, bx / d["Qd"], bu / d["Rd"]), Ns, ko)
    gx, gu = _recover(d, prev, mu, bx, bu)
    o = lambda a, b: a.unsqueeze(-1) * b.unsqueeze(-2)  # noqa: E731
    gA = o(mu[prev + 1], dx[prev]) + o(lam[prev + 1], gx[prev])
    gB = o(mu[prev + 1], du) + o(lam[prev + 1], gu)
    return dict(lam=lam, dx=dx, du=du, gA=gA, gB=gB, gQd=gx * dx, gRd=gu * du, gq=gx, gr=gu, gc=-mu)
