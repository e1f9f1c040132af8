"""Cases of the semi-implicit RBF-FD path: what users of the package have it
do, through its public entry points, over the range of sizes, degrees and
solver options of the repository's own configurations and tests.

A case is a dict of plain values.  ``kind`` says which call it is:

* ``apply``: gradient and Laplacian of a field with a problem's packed
  operators (post-processing of a solution; the smallest calls).
* ``clouds``: S1, the clouds of a tagged point set.
* ``weights``: S2, the d/dx, d/dy and Laplacian weights of given clouds.
* ``iterate``: one outer iteration (the two Krylov solves and the row
  kernels) of a problem whose clouds, weights and hierarchy exist, from a
  given state: the inner call of every march.
* ``step``: rebuild for new points and the first BDF2 time step (the
  benchmark's default step).
* ``batch``: one outer iteration of many problems, one launch per solve.
* ``serve``: requests through the request server, a few time steps each.

Point clouds come from ``paper_2106_07616_gb300.clouds`` (inputs only:
coordinates, tags, normals, boundary values) with the seed's own jitter; the
fields are closed forms where the flow has one, plus smooth seeded modes
that vanish on the boundary; steps, batches and requests start from rest.

Every Krylov solve stops on its FP64 relative residual: 1e-12 (the default)
where the p' solver is BiCGSTAB, 1e-10 with flexible GMRES, whose FP64
iterate has its floor near 1e-12 on some of these clouds.
"""
import math

import numpy as np
import torch

from paper_2106_07616_gb300 import clouds, rbffd

DEV = "cuda:0"
PRECISION = {"fp64": rbffd.PREC_FP64, "mixed": rbffd.PREC_MIXED, "ff": rbffd.PREC_MIXED_FF}
PRECOND = {"jacobi": rbffd.PRECOND_JACOBI, "amg": rbffd.PRECOND_AMG,
           "fgmres": rbffd.PRECOND_AMG_FGMRES}
ALPHA = (1.5, -2.0, 0.5)
DENSE_ROWS = 10500  # largest system that exact() solves densely in 64 bits


def listed():
    return [
        # a derived field (vorticity, pressure gradient) of a small solution:
        # latency of the shortest calls
        dict(name="apply_kov50", kind="apply", flow="kovasznay", side=50, degree=3, q=20, re=40, cfl=10),
        # clouds of the largest configuration's points (graded, four tags)
        dict(name="clouds_cyl150k", kind="clouds", flow="cylinder", n=150000, h0=0.02, hmax=0.2,
             degree=3, q=20, re=100, cfl=10),
        # low-degree weights of a mid-sized odd lattice: small local systems
        dict(name="weights_kov101_k2", kind="weights", flow="kovasznay", side=101, degree=2, q=12, re=40, cfl=10),
        # the weights of the benchmark's default workload
        dict(name="weights_cav200_k4", kind="weights", flow="cavity", side=200, degree=4, q=30, re=1000, cfl=10),
        # an outer iteration of the smallest configuration, default solvers
        dict(name="iterate_kov50", kind="iterate", flow="kovasznay", side=50, degree=3, q=20,
             re=40, cfl=10, precision="mixed", precond="fgmres"),
        # of the benchmark's default workload: the inner call of its march
        dict(name="iterate_cav200", kind="iterate", flow="cavity", side=200, degree=4, q=30,
             re=1000, cfl=10, precision="mixed", precond="fgmres"),
        # of the largest configuration: outlet, symmetry lines, graded cloud
        dict(name="iterate_cyl150k", kind="iterate", flow="cylinder", n=150000, h0=0.02, hmax=0.2,
             degree=3, q=20, re=100, cfl=10, precision="mixed", precond="fgmres"),
        # FP64 throughout with the multigrid preconditioner, odd size
        dict(name="iterate_cav99_amg64", kind="iterate", flow="cavity", side=99, degree=3, q=20,
             re=400, cfl=1, precision="fp64", precond="amg"),
        # the binding's defaults, the paper's own solver: FP64 and Jacobi
        dict(name="iterate_kov30_jac64", kind="iterate", flow="kovasznay", side=30, degree=3, q=20,
             re=40, cfl=5, precision="fp64", precond="jacobi"),
        # new points: clouds, weights, operators, hierarchy, first time step
        dict(name="step_cav200", kind="step", flow="cavity", side=200, degree=4, q=30,
             re=1000, cfl=10, precision="mixed", precond="fgmres"),
        # the batched workload's recipe (mixed sizes and degrees) at 16 members
        dict(name="batch16", kind="batch", count=16, n_lo=1000, n_hi=64000, mix=4),
        # requests of the serving workload's lower sizes through the server
        dict(name="serve4", kind="serve", count=4, n_lo=5000, n_hi=10000, steps=2, mix=5),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _flow_case(rng, n_lo, n_hi, degrees):
    """Flow, size and cloud size of a drawn single problem."""
    flow = rng.choice(["kovasznay", "cavity", "cylinder"])
    k = rng.choice(degrees)
    c = dict(flow=flow, degree=k, q=rng.choice([(k + 1) * (k + 2), (k + 1) * (k + 2)]
                                               + ([30] if k == 4 else [])))
    n = _log(rng, max(n_lo, 5000) if flow == "cylinder" else n_lo, n_hi)
    if flow == "cylinder":
        c.update(n=int(n), h0=round(0.1 * math.sqrt(5000.0 / n), 6), hmax=0.5, re=100)
        if n > 50000:
            c.update(n=int(max(n, 120000)), h0=0.02, hmax=0.2)
    else:
        c.update(side=max(int(math.ceil(math.sqrt(n))), 24))
    # a Courant number and a Reynolds number at which the lattice's Jacobi
    # momentum solves converge for any jitter
    c["cfl"] = round(_log(rng, 0.8, 5.0), 2)
    if flow == "kovasznay":
        c["re"] = rng.choice([40, 60])
        c["cfl"] = min(c["cfl"], 2.0)
    if flow == "cavity":
        c["re"] = 1000 if c["side"] >= 130 else 100
        if c["side"] < 130:
            c["cfl"] = round(_log(rng, 0.5, 1.5), 2)
    return c


def draw(rng):
    kind = rng.choice(["apply", "clouds", "weights", "iterate", "iterate", "iterate", "iterate",
                       "step", "batch", "serve"])
    if kind == "apply":
        return dict(kind=kind, **_flow_case(rng, 900, 64000, [2, 3, 4, 5]))
    if kind == "clouds":
        return dict(kind=kind, **_flow_case(rng, 900, 150000, [2, 3, 4, 5]))
    if kind == "weights":
        c = _flow_case(rng, 900, 64000, [2, 3, 4, 5])
        return dict(kind=kind, **c)
    if kind == "iterate":
        how = rng.choice(["default", "default", "amg64", "ff", "jac64"])
        if how == "jac64":
            return dict(kind=kind, flow="kovasznay", side=rng.randint(20, 40), degree=3, q=20,
                        re=40, cfl=round(_log(rng, 1.0, 10.0), 2), precision="fp64",
                        precond="jacobi")
        c = _flow_case(rng, 900, 50000 if how == "default" else 20000, [3, 4])
        c.update(precision={"default": "mixed", "amg64": "fp64", "ff": "ff"}[how],
                 precond={"default": "fgmres", "amg64": "amg", "ff": "fgmres"}[how])
        return dict(kind=kind, **c)
    if kind == "step":
        k = rng.choice([3, 4])
        side = rng.randint(40, 180)
        c = dict(kind=kind, flow=rng.choice(["kovasznay", "cavity"]), side=side, degree=k,
                 q=(k + 1) * (k + 2), cfl=10, precision="mixed", precond="fgmres")
        c["re"] = 40 if c["flow"] == "kovasznay" else 1000 if side >= 130 else 100
        return c
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(3, 14), n_lo=1000,
                    n_hi=int(_log(rng, 4000, 50000)), mix=rng.randint(0, 1 << 20))
    return dict(kind=kind, count=rng.randint(2, 4), n_lo=2000, n_hi=int(_log(rng, 3000, 9000)),
                steps=rng.randint(1, 3), mix=rng.randint(0, 1 << 20))


# ---------------------------------------------------------------- inputs


def _flow(c, seed):
    """The points and boundary data of a case (host arrays)."""
    s = 1 + int(seed) % 1000003
    kw = dict(seed=s, degree=c["degree"], q=c["q"], re=float(c["re"]))
    if c["flow"] == "cylinder":
        # one graded cloud (the number of points depends on its seed), its
        # interior points moved by the case's seed
        fp = clouds.cylinder(c["n"], h0=c["h0"], hmax=c["hmax"], dt=c["cfl"] * c["h0"],
                             **dict(kw, seed=3))
        r = np.random.Generator(np.random.PCG64(s))
        move = np.where(fp.tag == clouds.TAG_INTERIOR, 0.1 * c["h0"], 0.0)
        fp.x = fp.x + move * r.uniform(-1, 1, fp.n)
        fp.y = fp.y + move * r.uniform(-1, 1, fp.n)
        return fp
    if c["flow"] == "cavity":
        return clouds.cavity(c["side"], dt=c["cfl"] / (c["side"] - 1), **kw)
    return clouds.kovasznay(c["side"], dt=2.0 * c["cfl"] / (c["side"] - 1), **kw)


def _members(c, seed):
    """A batch's or server's problems: sizes, degrees and flows by ``mix``
    (the same for every seed), the points' jitter by the seed."""
    r = np.random.Generator(np.random.PCG64(c["mix"]))
    out = []
    for i in range(c["count"]):
        side = int(math.ceil(math.sqrt(math.exp(r.uniform(math.log(c["n_lo"]),
                                                          math.log(c["n_hi"]))))))
        k = int(r.integers(3, 5)) if c["kind"] == "serve" else int(r.integers(2, 6))
        flow = "kovasznay" if r.uniform() < 0.5 else "cavity"
        re = 40 if flow == "kovasznay" else 100 if c["kind"] == "serve" else 1000
        m = dict(flow=flow, side=side, degree=k, q=(k + 1) * (k + 2), re=re, cfl=10)
        out.append((m, int(seed) + 7919 * (i + 1)))
    return out


def _rest(fp):
    """The state a build leaves: the boundary velocity, rest inside."""
    u, v = (np.where(fp.tag == clouds.TAG_INTERIOR, 0.0, b) for b in (fp.ubc, fp.vbc))
    return dict(u=u, un=u, unm1=u, v=v, vn=v, vnm1=v, p=np.zeros(fp.n))


def _tol(c):
    return 1e-10 if c["precond"] == "fgmres" else 1e-12


def _fields(fp, c, seed):
    """A developed-looking state: the flow's closed form or a boundary-layer
    profile plus smooth seeded modes that vanish on the boundary."""
    r = np.random.Generator(np.random.PCG64([int(seed), 77]))
    X = (fp.x - fp.x.min()) / np.ptp(fp.x)
    Y = (fp.y - fp.y.min()) / np.ptp(fp.y)
    bub = 16.0 * X * (1 - X) * Y * (1 - Y)
    if c["flow"] == "cylinder":
        d = np.hypot(fp.x, fp.y) - 0.5
        bub = bub * (1.0 - np.exp(-np.maximum(d, 0.0) ** 2 / 0.25))
    bub[fp.tag != clouds.TAG_INTERIOR] = 0.0

    def modes():
        s = np.zeros(fp.n)
        for _ in range(4):
            kx, ky = r.integers(0, 3, 2)
            s += r.uniform(-1, 1) * np.sin(2 * math.pi * (kx * X + ky * Y) + r.uniform(0, 6.28))
        return s * bub

    if fp.exact is not None:
        u, v, p = fp.exact["u"], fp.exact["v"], fp.exact["p"]
    elif c["flow"] == "cavity":
        u = np.where(fp.tag == 0, Y ** 8 * (1 - (2 * X - 1) ** 8), fp.ubc)
        v, p = fp.vbc, np.zeros(fp.n)
    else:
        u, v, p = fp.initial["u"], fp.vbc, np.zeros(fp.n)
    f = {}
    for name, base in (("u", u), ("v", v)):
        now, rate = modes(), modes()
        f[name] = base + 0.05 * now
        f[name + "n"] = base + 0.05 * (now - 0.1 * rate)
        f[name + "nm1"] = base + 0.05 * (now - 0.2 * rate)
    f["p"] = p + 0.05 * modes()
    return {k: np.ascontiguousarray(a) for k, a in f.items()}


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


_CTX = None


def _ctx():
    """The context a program keeps for all its problems."""
    global _CTX
    if _CTX is None:
        _CTX = rbffd.Context(0)
    return _CTX


def _problem(fp, c, f):
    """A problem as a march has it: built, its state set, one outer iteration
    behind it."""
    P = rbffd.Problem(_ctx(), fp, PRECISION[c["precision"]], precond=PRECOND[c["precond"]])
    for k, a in f.items():
        P.set(k, a)
    P.simple_iterate(fp.dt, krylov_tol=_tol(c))
    return P, {k: _dev(f[k]) for k in ("u", "v", "p")}


def prepare(c, seed):
    kind = c["kind"]
    if kind == "batch":
        ms = [(m, s, _flow(m, s)) for m, s in _members(c, seed)]
        probs, start = [], []
        for m, s, fp in ms:
            P, f = _problem(fp, dict(m, precision="fp64", precond="amg"), _rest(fp))
            probs.append(P)
            start.append(f)
        B = rbffd.Batch(_ctx(), probs)
        B.set_autotune(False)  # the planned team sizes: the same sums on every run
        s = dict(kind=kind, B=B, probs=probs, start=start, dt=np.array([f.dt for *_, f in ms]),
                 out=[{k: torch.empty_like(f[k]) for k in f} for f in start])
        torch.cuda.synchronize()
        run(s)  # a march's iterations are captured from the second on
        return s
    if kind == "serve":
        ctx = rbffd.Context(0)  # a server owns its context's stream
        return dict(kind=kind, S=rbffd.Server(ctx), steps=c["steps"],
                    fps=[_flow(m, s) for m, s in _members(c, seed)])
    fp = _flow(c, seed)
    if kind == "iterate":
        P, f = _problem(fp, c, _fields(fp, c, seed))
        s = dict(kind=kind, P=P, start=f, dt=fp.dt, tol=_tol(c), out={k: torch.empty_like(f[k]) for k in f})
    elif kind == "step":
        d = {k: _dev(getattr(fp, k)) for k in ("x", "y", "tag", "nx", "ny", "ubc", "vbc")}
        desc = rbffd.desc_from_pointers(fp.n, fp.q, fp.degree, fp.pin, fp.rho, fp.mu,
                                        PRECISION[c["precision"]], d["x"], d["y"], d["tag"],
                                        d["nx"], d["ny"], d["ubc"], d["vbc"],
                                        PRECOND[c["precond"]])
        P = rbffd.Problem(_ctx(), desc=desc)
        s = dict(kind=kind, P=P, keep=d, desc=desc, dt=fp.dt, tol=_tol(c),
                 out={k: torch.empty_like(d["x"]) for k in ("u", "v", "p")})
    elif kind == "apply":
        P = rbffd.Problem(_ctx(), fp)
        f = _fields(fp, c, seed)
        s = dict(kind=kind, P=P, f=_dev(f["u"]),
                 out=[torch.empty(fp.n, dtype=torch.float64, device=DEV) for _ in range(3)])
    else:
        x, y, tag = _dev(fp.x), _dev(fp.y), _dev(fp.tag)
        idx = torch.empty((fp.n, fp.q), dtype=torch.int32, device=DEV)
        s = dict(kind=kind, x=x, y=y, tag=tag, q=fp.q, degree=fp.degree, idx=idx)
        if kind == "weights":
            torch.cuda.synchronize()
            rbffd.rbffd_build_stencils(_ctx(), x, y, tag, fp.q, idx)
            s["out"] = [torch.empty((fp.n, fp.q), dtype=torch.float64, device=DEV)
                        for _ in range(3)]
    torch.cuda.synchronize()
    return s


# ------------------------------------------------------------------- run


def run(s):
    kind = s["kind"]
    if kind == "apply":
        for op, y in zip((rbffd.OP_DX, rbffd.OP_DY, rbffd.OP_LAP), s["out"]):
            s["P"].apply(op, s["f"], y)
        return s["out"]
    if kind == "clouds":
        rbffd.rbffd_build_stencils(_ctx(), s["x"], s["y"], s["tag"], s["q"], s["idx"])
        return s["idx"]
    if kind == "weights":
        bad = rbffd.rbffd_weights(_ctx(), s["x"], s["y"], s["q"], s["idx"], s["degree"], *s["out"])
        return [*s["out"], bad]
    if kind == "iterate":
        P = s["P"]
        for k, a in s["start"].items():
            P.set(k, a)
        delta, _ = P.simple_iterate(s["dt"], krylov_tol=s["tol"])
        for k, a in s["out"].items():
            P.get(k, a)
        return {**s["out"], "delta": delta}
    if kind == "step":
        P = s["P"]
        P.reload(desc=s["desc"])
        P.time_step(s["dt"], 1e-4, max_outer=20, krylov_tol=s["tol"])
        for k, a in s["out"].items():
            P.get(k, a)
        return s["out"]
    if kind == "batch":
        for P, f in zip(s["probs"], s["start"]):
            for k, a in f.items():
                P.set(k, a)
        delta, _, status = s["B"].iterate(s["dt"])
        for P, f in zip(s["probs"], s["out"]):
            for k, a in f.items():
                P.get(k, a)
        return {"fields": s["out"], "delta": delta, "status": status}
    S = s["S"]
    tickets = [S.submit(fp, max_steps=s["steps"], criterion=2, precond=rbffd.PRECOND_AMG)
               for fp in s["fps"]]
    S.drain()
    got = [S.poll(t, fields=True) for t in tickets]
    return [[g["status"], g["steps"], g["u"], g["v"], g["p"]] for g in got]


# ------------------------------------------------------------------ work


def _points(c):
    return c["n"] if c["flow"] == "cylinder" else c["side"] * c["side"]


def _build_work(n, q, k):
    """Clouds and weights from coordinates: (bytes, FP64 flops)."""
    big = q + (k + 1) * (k + 2) // 2
    return n * (17 + q * 28), n * (2.0 * big ** 3 / 3 + 6.0 * big ** 2 + 10.0 * q * q)


def _iterate_work(n, q):
    """One outer iteration's least traffic: the weights and indices, the two
    matrices and the fields once; and the operations of assembling them and
    of applying each once (what the solves repeat is the method's choice)."""
    return n * (q * 28 + 14 * 8 + 3 * 8), n * q * (3 * 2 + 2 * 9 + 3 * 2.0)


def work(c):
    kind = c["kind"]
    if kind in ("batch", "serve"):
        b = f = 0.0
        for m, _ in _members(c, 0):
            n, q = m["side"] ** 2, m["q"]
            wb, wf = _iterate_work(n, q)
            if kind == "serve":
                gb, gf = _build_work(n, q, m["degree"])
                wb, wf = gb + c["steps"] * wb, gf + c["steps"] * wf
            b, f = b + wb, f + wf
        return dict(bytes=b, flops=f)
    n, q = _points(c), c["q"]
    if kind == "apply":
        return dict(bytes=n * (q * 28 + 8 + 24), flops=n * q * 6.0)
    if kind == "clouds":
        return dict(bytes=n * (17 + 4 * q), flops=n * q * 5.0)
    if kind == "weights":
        b, f = _build_work(n, q, c["degree"])
        return dict(bytes=b, flops=f)
    b, f = _iterate_work(n, q)
    if kind == "step":
        gb, gf = _build_work(n, q, c["degree"])
        b, f = b + gb, f + gf
    return dict(bytes=b, flops=f)


# ----------------------------------------------------------------- exact
# The method in plain torch, 64 bits, on the same inputs: brute-force clouds,
# dense local systems by LU, dense global systems by LU.


def _ref_clouds(x, y, tag, q):
    n = x.numel()
    idx = torch.empty((n, q), dtype=torch.int64, device=DEV)
    interior = tag == 0
    for lo in range(0, n, 2048):
        hi = min(n, lo + 2048)
        dx, dy = x[None, :] - x[lo:hi, None], y[None, :] - y[lo:hi, None]
        d2 = dx * dx + dy * dy
        d2 = torch.where(~interior[lo:hi, None] & ~interior[None, :], torch.inf, d2)
        d2[torch.arange(hi - lo, device=DEV), torch.arange(lo, hi, device=DEV)] = -1.0
        idx[lo:hi] = torch.topk(d2, q, dim=1, largest=False, sorted=True).indices
    return idx


def _ref_weights(x, y, idx, degree):
    """(n, q) weights of d/dx, d/dy and the Laplacian."""
    n, q = idx.shape
    exps = [(a, d - a) for d in range(degree + 1) for a in range(d, -1, -1)]
    m = len(exps)
    out = [torch.empty((n, q), dtype=torch.float64, device=DEV) for _ in range(3)]
    for lo in range(0, n, 4096):
        hi = min(n, lo + 4096)
        cl = idx[lo:hi]
        dx, dy = x[cl] - x[lo:hi, None], y[cl] - y[lo:hi, None]
        h = torch.sqrt((dx * dx + dy * dy).amax(1, keepdim=True))
        xi, et = dx / h, dy / h
        r = torch.sqrt((xi[:, :, None] - xi[:, None, :]) ** 2
                       + (et[:, :, None] - et[:, None, :]) ** 2)
        A = torch.zeros((hi - lo, q + m, q + m), dtype=torch.float64, device=DEV)
        R = torch.zeros((hi - lo, q + m, 3), dtype=torch.float64, device=DEV)
        A[:, :q, :q] = r ** 3
        for l, (a, b) in enumerate(exps):
            A[:, :q, q + l] = A[:, q + l, :q] = xi ** a * et ** b
            if (a, b) in ((1, 0), (0, 1)):
                R[:, q + l, 0 if a else 1] = 1.0
            if (a, b) in ((2, 0), (0, 2)):
                R[:, q + l, 2] = 2.0
        rj = torch.sqrt(xi * xi + et * et)
        R[:, :q, 0], R[:, :q, 1], R[:, :q, 2] = -3 * rj * xi, -3 * rj * et, 9 * rj
        S = torch.linalg.solve(A, R)[:, :q]
        for k, scale in enumerate((h, h, h * h)):
            out[k][lo:hi] = S[:, :, k] / scale
    return out


class _Ref:
    """A flow problem in 64 bits: sparse rows (idx, weights), dense solves."""

    def __init__(self, fp):
        self.fp, self.n = fp, fp.n
        self.x, self.y, self.tag = _dev(fp.x), _dev(fp.y), _dev(fp.tag)
        self.nx, self.ny = _dev(fp.nx), _dev(fp.ny)
        self.ubc, self.vbc = _dev(fp.ubc), _dev(fp.vbc)
        self.idx = _ref_clouds(self.x, self.y, self.tag, fp.q)
        self.wx, self.wy, self.wl = _ref_weights(self.x, self.y, self.idx, fp.degree)
        self.inside = self.tag == clouds.TAG_INTERIOR
        self.G = self.nx[:, None] * self.wx + self.ny[:, None] * self.wy
        self.M = torch.where(self.inside[:, None], self.wl, self.G)
        unit = torch.zeros_like(self.wx)
        unit[:, 0] = 1.0  # a cloud's first member is its centre
        self.unit = unit
        fixed = self.tag == clouds.TAG_OUTFLOW
        if fp.pin >= 0:
            fixed = fixed.clone()
            fixed[fp.pin] = True
        self.M = torch.where(fixed[:, None], unit, self.M)
        sym = self.tag == clouds.TAG_SYMMETRY
        along_x = self.nx.abs() > self.ny.abs()
        ident = self.tag == clouds.TAG_DIRICHLET
        self.ident = (ident | (sym & along_x), ident | (sym & ~along_x))
        self.lu_p = None

    def mul(self, w, f):
        return (w * f[self.idx]).sum(1)

    def dense(self, w):
        A = torch.zeros((self.n, self.n), dtype=torch.float64, device=DEV)
        A.scatter_add_(1, self.idx, w)
        return A

    def iterate(self, f, dt):
        fp, (a1, a2, a3) = self.fp, ALPHA
        rho, mu = fp.rho, fp.mu
        old = [(f["u"], f["un"], f["unm1"]), (f["v"], f["vn"], f["vnm1"])]
        grads, bc, tilde, lu, kept = (self.wx, self.wy), (self.ubc, self.vbc), [], None, None
        eq = (rho * f["u"][:, None] * self.wx + rho * f["v"][:, None] * self.wy - mu * self.wl
              + (rho * a1 / dt) * self.unit)
        for c in range(2):
            w = torch.where(self.inside[:, None], eq, self.G)
            w = torch.where(self.ident[c][:, None], self.unit, w)
            b = -rho * (a2 * old[c][1] + a3 * old[c][2]) / dt - self.mul(grads[c], f["p"])
            b = torch.where(self.inside, b, torch.where(self.ident[c], bc[c], 0.0))
            if kept is None or not torch.equal(kept, w):
                lu, kept = torch.linalg.lu_factor(self.dense(w)), w
            tilde.append(torch.linalg.lu_solve(*lu, b[:, None])[:, 0])
        del lu, kept
        ut, vt = tilde
        s = rho * a1 / dt * (self.mul(self.wx, ut) + self.mul(self.wy, vt))
        b = torch.where(self.inside, s, 0.0)
        if self.lu_p is None:
            self.lu_p = torch.linalg.lu_factor(self.dense(self.M))
        one = self.inside.to(torch.float64)
        X = torch.linalg.lu_solve(*self.lu_p, torch.stack([b, one], 1))
        pc = X[:, 0]
        if fp.pin >= 0:  # the compatible source: the pin's Neumann row holds too
            g = (self.G[fp.pin][:, None] * X[self.idx[fp.pin]]).sum(0)
            pc = pc - (g[0] / g[1]) * X[:, 1]
        p = torch.where(self.inside, f["p"] + pc, f["p"])
        F = []
        for t, (_, n0, n1) in zip(tilde, old):
            F.append(-rho * (a1 * t + a2 * n0 + a3 * n1) / dt
                     - rho * (ut * self.mul(self.wx, t) + vt * self.mul(self.wy, t))
                     + mu * self.mul(self.wl, t))
        g = self.G.clone()
        g[:, 0] = 0.0
        pb = (self.nx * F[0] + self.ny * F[1] - self.mul(g, p)) / torch.where(
            self.inside, 1.0, self.G[:, 0])
        p = torch.where(self.inside | (self.tag == clouds.TAG_OUTFLOW), p, pb)
        k = dt / (rho * a1)
        u = torch.where(self.ident[0], ut, ut - k * self.mul(self.wx, pc))
        v = torch.where(self.ident[1], vt, vt - k * self.mul(self.wy, pc))
        delta = (u - f["u"]).abs().mean() + (v - f["v"]).abs().mean()
        return {"u": u, "v": v, "p": p, "delta": float(delta)}


def exact(c, seed):
    kind = c["kind"]
    if kind in ("clouds", "serve"):
        return None
    if kind == "batch":
        fields, delta = [], []
        for m, s in _members(c, seed):
            fp = _flow(m, s)
            if fp.n > DENSE_ROWS // 2:
                fields.append({"u": None, "v": None, "p": None})
                continue
            f = {k: _dev(a) for k, a in _rest(fp).items()}
            g = _Ref(fp).iterate(f, fp.dt)
            fields.append({k: g[k] for k in ("u", "v", "p")})
        return {"fields": fields, "delta": None, "status": None}
    fp = _flow(c, seed)
    if kind in ("apply", "weights"):
        x, y, tag = _dev(fp.x), _dev(fp.y), _dev(fp.tag)
        idx = _ref_clouds(x, y, tag, fp.q)
        w = _ref_weights(x, y, idx, fp.degree)
        if kind == "weights":
            return [*w, None]
        f = _dev(_fields(fp, c, seed)["u"])
        return [(a * f[idx]).sum(1) for a in w]
    if fp.n > DENSE_ROWS or kind == "step":
        return None
    f = {k: _dev(a) for k, a in _fields(fp, c, seed).items()}
    return _Ref(fp).iterate(f, fp.dt)
