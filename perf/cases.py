"""The work that users of this package have it do, as a list of measurable cases.

A case is one public call, or one implicit time step made of the calls that a
time loop makes, on one of the package's flows: the isentropic vortex on quads
or on triangles and the Taylor-Green vortex on hexes.  Operations:

  residual  R(W), FP64 (explicit parts, right-hand sides, monitoring)
  jvp       K v, exact linearisation, FP64 (the outer Krylov product) or FP32
            (the mixed preconditioner's fine-level operator); an FP32 product
            comes back widened to FP64 and is returned in the 32 bits it has
  apply     one application of the mixed p-multigrid preconditioner to a
            residual vector; its 32-bit result likewise
  step      one BDF2 step: preconditioner refresh at W^n, two Newton
            iterations (right-hand side, FGMRES solve, update); W^{n+1}
  serve     a burst of step requests through the serving runtime, host arrays

exact() restates the discretisation in plain FP64 torch, dense and element by
element (affine elements and face pairs; forward-mode derivatives by torch), and
solves the time steps with Newton and unpreconditioned GMRES.
"""
import itertools
import math
import random
import time

import numpy as np
import torch

from paper_1812_04789_gb300 import binding as B
from paper_1812_04789_gb300 import workloads as wl

GAMMA, PR, ROE_DELTA = 1.4, 0.72, 0.1


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: residual of the 16 x 16, p = 2 vortex, all latency and launches
        dict(name="residual_vortex16_p2", op="residual", flow="vortex", n0=16, n1=16, n2=1, p=2, space="P"),
        # the outer Krylov product on the largest mesh of the workloads (13.8 M unknowns)
        dict(name="jvp_tgv32_p6_fp64", op="jvp", flow="tgv", n0=32, n1=32, n2=32, p=6, space="P", mode="fp64"),
        # the paper's tensor-product space on a mesh with three unequal directions
        dict(name="jvp_q3_ragged_fp64", op="jvp", flow="tgv", n0=17, n1=13, n2=11, p=3, space="Q", mode="fp64"),
        # the smoother's fine-level operator on the headline mesh
        dict(name="jvp_tgv16_p4_fp32", op="jvp", flow="tgv", n0=16, n1=16, n2=16, p=4, space="P", mode="fp32"),
        # one application of the mixed preconditioner on the headline mesh
        dict(name="apply_tgv16_p4_mixed", op="apply", flow="tgv", n0=16, n1=16, n2=16, p=4, space="P",
             levels="4,2,1,0", storage="native", dt=0.01),
        # the small 2-D workload in full: one FP64 step with block Jacobi
        dict(name="step_vortex16_p2_bj_fp64", op="step", flow="vortex", n0=16, n1=16, n2=1, p=2, space="P",
             levels="2", precision="fp64", storage="native", dt=0.05),
        # the headline workload in full
        dict(name="step_tgv16_p4_mixed", op="step", flow="tgv", n0=16, n1=16, n2=16, p=4, space="P",
             levels="4,2,1,0", precision="mixed", storage="native", dt=0.01),
        # the high-order, low-Mach workload with BF16 blocks, on an eighth of its elements
        dict(name="step_tgv16_p6_bf16", op="step", flow="tgv", n0=16, n1=16, n2=16, p=6, space="P",
             levels="6,2,1,0", precision="mixed", storage="bf16", dt=0.01),
        # a served FP64 request: 3-D, odd sizes
        dict(name="step_tgv_ragged_p3_fp64", op="step", flow="tgv", n0=9, n1=10, n2=12, p=3, space="P",
             levels="3,2,1,0", precision="fp64", storage="native", dt=0.01),
        # a served mixed request: 2-D, many small elements
        dict(name="step_vortex_ragged_p3_mixed", op="step", flow="vortex", n0=100, n1=75, n2=1, p=3, space="P",
             levels="3,2,1,0", precision="mixed", storage="native", dt=0.05),
        # the paper's triangular grids
        dict(name="step_tri32_p4_mixed", op="step", flow="tri", n0=32, n1=32, n2=1, p=4, space="tri",
             levels="4,2,1,0", precision="mixed", storage="native", dt=0.05),
        # serving: six small requests of different shapes at once
        dict(name="serve_burst6", op="serve", count=6, mix=1812, workers=4),
    ]


def _n_modes(c, p=None):
    p = c["p"] if p is None else p
    if c["space"] == "tri":
        return (p + 1) * (p + 2) // 2
    d = _dim(c)
    return (p + 1) ** d if c["space"] == "Q" else math.comb(p + d, d)


def _dim(c):
    return 3 if c["flow"] == "tgv" else 2


def _n_elem(c):
    return c["n0"] * c["n1"] * (c["n2"] if c["flow"] == "tgv" else 1) * (2 if c["flow"] == "tri" else 1)


def _dofs(c):
    return _n_elem(c) * (_dim(c) + 2) * _n_modes(c)


def _levels(p):
    return ",".join(str(q) for q in [p] + [q for q in (2, 1, 0) if q < p])


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    """One more case of the same ranges: sizes spread over their logarithm,
    directions drawn apart, orders 1 to 6; a size that would cost more than the
    largest listed case of its kind is drawn again."""
    op = rng.choice(["residual", "jvp", "jvp", "apply", "step", "step", "step", "serve"])
    if op == "serve":
        return dict(op="serve", count=rng.randint(3, 6), mix=rng.randint(1, 10**6), workers=rng.choice([2, 3, 4]))
    while True:
        flow = rng.choice(["tgv", "tgv", "vortex"] if op != "step" else ["tgv", "tgv", "vortex", "tri"])
        c = dict(op=op, flow=flow)
        if flow == "tgv":
            n = _log_int(rng, 5, 32)
            c.update(n0=n, n1=max(4, n + rng.randint(-3, 3)), n2=max(4, n + rng.randint(-3, 3)))
        elif flow == "vortex":
            n = _log_int(rng, 16, 256)
            c.update(n0=n, n1=max(12, int(n * rng.uniform(0.6, 1.4))), n2=1)
        else:
            n = _log_int(rng, 8, 40)
            c.update(n0=n, n1=max(6, n + rng.randint(-4, 4)), n2=1)
        c["p"] = rng.randint(1, 5 if flow == "tri" else 6)
        c["space"] = "tri" if flow == "tri" else "P"
        if op in ("residual", "jvp") and c["p"] <= 4 and rng.random() < 0.25:
            c["space"] = "Q"
        if op == "jvp":
            c["mode"] = rng.choice(["fp64", "fp32"])
        if op in ("apply", "step"):
            c.update(levels=_levels(c["p"]), storage="native", dt=0.01 if flow == "tgv" else 0.05)
        if op == "step":
            c["precision"] = rng.choice(["mixed", "mixed", "fp64"])
            if c["precision"] == "mixed" and flow != "tri" and rng.random() < 0.3:
                c["storage"] = "bf16"
            if flow == "vortex" and c["precision"] == "fp64" and rng.random() < 0.3:
                c["levels"] = str(c["p"])
        most = 13.8e6
        if op == "apply":
            most = 1.0e6
        if op == "step":
            most = 1.2e6 if flow != "tri" else 1.6e5
            if c["precision"] == "fp64":
                most = 1.2e5 if flow != "tri" else 4e4
        if _dofs(c) <= most:
            return c


def _requests(c):
    """The requests of a serving case: small 2-D and 3-D steps of different
    orders, FP64 or mixed."""
    rng = random.Random(c["mix"])
    out = []
    for _ in range(c["count"]):
        if rng.random() < 0.5:
            r = dict(flow="vortex", n0=rng.randint(16, 40), n1=rng.randint(16, 40), n2=1, p=rng.randint(1, 4))
        else:
            n = rng.randint(5, 9)
            r = dict(flow="tgv", n0=n, n1=n, n2=n + rng.randint(-1, 1), p=rng.randint(1, 3))
        precision = "mixed" if rng.random() < 0.6 else "fp64"
        r.update(op="step", space="P", levels=_levels(r["p"]), precision=precision, storage="native",
                 dt=0.01 if r["flow"] == "tgv" else 0.05)
        out.append(r)
    return out


# ------------------------------------------------------------------ flows and inputs
def _config(c):
    """The package's description of the case's flow and mesh."""
    if c["flow"] == "tri":
        return wl.tri_config((c["n0"], c["n1"]), c["p"], dt_conv=c.get("dt", 0.05))
    if c["flow"] == "vortex":
        return wl.make_config("vortex", 2, (c["n0"], c["n1"]), c["p"], M=0.5, Re=1000.0, dt_conv=c.get("dt", 0.05),
                              space=c["space"])
    return wl.make_config("tgv", 3, (c["n0"], c["n1"], c["n2"]), c["p"], M=0.05 if c["p"] == 6 else 0.1, Re=1600.0,
                          dt_conv=c.get("dt", 0.01), space=c["space"])


def _uref(c):
    return (0.5 if c["flow"] != "tgv" else 0.05 if c["p"] == 6 else 0.1) * math.sqrt(GAMMA)


def _mu(c):
    return _uref(c) * 10.0 / 1000.0 if c["flow"] != "tgv" else _uref(c) / 1600.0


def _dt(c):
    return c["dt"] * (10.0 if c["flow"] != "tgv" else 1.0) / _uref(c)


def _box(c):
    return ((0.0,) * 3, (2 * math.pi,) * 3) if c["flow"] == "tgv" else ((0.0,) * 2, (10.0,) * 2)


def _modes(c):
    d, p = _dim(c), c["p"]
    deg = max if c["space"] == "Q" else sum
    out = []
    for s in range(p + 1):
        out += sorted((a for a in itertools.product(range(s + 1), repeat=d) if deg(a) == s), reverse=True)
    return out


def _legendre(p, x):
    """Orthonormal Legendre polynomials and their derivatives at x: (n, p + 1) each."""
    L = np.polynomial.legendre
    sc = np.sqrt((2 * np.arange(p + 1) + 1) / 2.0)
    V = L.legvander(x, p) * sc
    D = np.stack([L.legval(x, L.legder(np.eye(p + 1)[i])) if i else 0 * x for i in range(p + 1)], axis=1) * sc
    return V, D


def _flow_at(c, X, rng):
    """The flow's conservative variables at points X (..., d): the closed form
    with a seeded phase and strength, plus two seeded weak long waves."""
    u0 = _uref(c)
    if c["flow"] == "tgv":
        ph, amp = rng.uniform(0, 2 * math.pi, 3), rng.uniform(0.95, 1.05)
        x, y, z = (X[..., k] + float(ph[k]) for k in range(3))
        v0 = u0 * amp
        vel = [v0 * torch.sin(x) * torch.cos(y) * torch.cos(z), -v0 * torch.cos(x) * torch.sin(y) * torch.cos(z), 0 * x]
        pr = 1 + v0 * v0 / 16 * (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2)
        rho = pr.clone()
    else:
        ctr, beta = 5.0 + rng.uniform(-1, 1, 2), rng.uniform(0.018, 0.022)
        dx, dy = (torch.remainder(X[..., k] - float(ctr[k]) + 5.0, 10.0) - 5.0 for k in range(2))
        r2 = (dx * dx + dy * dy) / 0.25
        vel = [u0 * (1 - beta * dy / 0.5 * torch.exp(-r2 / 2)), u0 * beta * dx / 0.5 * torch.exp(-r2 / 2)]
        T = 1 - u0 * u0 * beta * beta * (GAMMA - 1) / (2 * GAMMA) * torch.exp(-r2)
        rho = T ** (1 / (GAMMA - 1))
        pr = rho * T
    lo, hi = _box(c)
    for j in range(len(vel)):
        for _ in range(2):
            k = rng.integers(0, X.shape[-1])
            s = 2 * math.pi / (hi[k] - lo[k]) * int(rng.integers(1, 3))
            vel[j] = vel[j] + 0.02 * u0 * torch.sin(s * X[..., k] + float(rng.uniform(0, 6.28)))
    q2 = sum(v * v for v in vel)
    return [rho] + [rho * v for v in vel] + [pr / (GAMMA - 1) + 0.5 * rho * q2]


def _state(c, seed):
    """Modal coefficients W[e, v, i] of the seeded flow by L2 projection, on the GPU."""
    rng = np.random.default_rng([seed, c["p"], c["n0"], c["n1"], c["n2"]])
    g = _geometry(c, extra=3)
    nq = len(g["wq"])
    E, nm, m = _n_elem(c), _n_modes(c), _dim(c) + 2
    P = g["phi"] * g["wq"][:, None]
    W = torch.empty((E, m, nm), dtype=torch.float64, device="cuda")
    own = rng.bit_generator.state
    for a in range(0, E, max(1, 2**22 // nq)):
        b = min(E, a + max(1, 2**22 // nq))
        rng.bit_generator.state = own
        for v, f in enumerate(_flow_at(c, g["at"](a, b), rng)):
            W[a:b, v] = f @ P
    return W


def _vector(c, W, seed, k):
    """A seeded vector of W's shape with the spectrum of a smooth field's
    coefficients: each degree half as large as the one below it."""
    gen = torch.Generator(device="cuda").manual_seed(1000003 * (seed % 2**40) + k)
    v = torch.randn(W.shape, dtype=torch.float64, device="cuda", generator=gen)
    deg = [i + j for i, j in _tri_modes(c["p"])] if c["space"] == "tri" else [sum(a) for a in _modes(c)]
    return v * torch.tensor([0.5**s for s in deg], dtype=torch.float64, device="cuda")


def _tri_modes(p):
    return [(i, s - i) for s in range(p + 1) for i in range(s, -1, -1)]


# ------------------------------------------------------------------ prepare / run
def _mesh(c):
    cfg = _config(c)
    if c["flow"] == "tri":
        return B.Mesh.from_tri_workload(wl.tri_mesh(cfg), wl.tri_physics(cfg), c["p"])
    return B.Mesh.from_workload(wl.mesh_desc(cfg), wl.physics(cfg))


def _opts(c):
    levels = tuple(int(x) for x in c["levels"].split(","))
    mixed = c["op"] == "apply" or c["precision"] == "mixed"
    return B.pmg_opts(levels, cycle=B.CYCLE_FMG if len(levels) > 1 else B.CYCLE_BJ,
                      precision=B.PREC_MIXED if mixed else B.PREC_FP64,
                      storage=B.STORE_BF16 if c["storage"] == "bf16" else B.STORE_NATIVE)


def prepare(case, seed):
    c = dict(case)
    if c["op"] == "serve":
        reqs = _requests(c)
        s = dict(op="serve", server=B.Server(40 << 30, workers=c["workers"]), reqs=[])
        for k, r in enumerate(reqs):
            cfg = _config(r)
            W = _state(r, seed + k).cpu().numpy()
            s["reqs"].append((wl.mesh_desc(cfg), wl.physics(cfg), _opts(r), W, W.copy(), _dt(r), np.zeros_like(W)))
        return s
    s = dict(op=c["op"], mesh=_mesh(c), W=_state(c, seed))
    s["out"] = torch.empty_like(s["W"])
    if c["op"] == "jvp":
        s["sigma"] = 1.5 / _dt(dict(c, dt=0.01 if c["flow"] == "tgv" else 0.05))
        s["mode"] = B.JVP_EXACT if c["mode"] == "fp64" else B.JVP_EXACT_FP32
        s["v"] = _vector(c, s["W"], seed, 1)
    if c["op"] in ("apply", "step"):
        s["dt"] = _dt(c)
        s["sigma"] = 1.5 / s["dt"]
        s["pmg"] = B.PMG(s["mesh"], s["W"], s["sigma"], _opts(c))
    if c["op"] == "apply":
        s["r"] = _vector(c, s["W"], seed, 2)
    if c["op"] == "step":
        s["b"], s["dW"] = torch.empty_like(s["W"]), torch.empty_like(s["W"])
    return s


def run(s):
    if s["op"] == "serve":
        for k, (desc, phys, opts, W, Wm, dt, out) in enumerate(s["reqs"]):
            s["server"].submit(k, desc, phys, opts, W, Wm, dt, out)
        left = len(s["reqs"])
        while left:
            for done in s["server"].poll(min_done=left):
                if done["status"] != B.DG_OK:
                    raise RuntimeError("request %d ended with status %d" % (done["id"], done["status"]))
                left -= 1
        return [r[-1] for r in s["reqs"]]
    mesh, W, out = s["mesh"], s["W"], s["out"]
    if s["op"] == "residual":
        mesh.residual(W, out)
        return out
    if s["op"] == "jvp":
        mesh.jvp(W, s["v"], out, s["sigma"], mode=s["mode"])
        return out.float() if s["mode"] == B.JVP_EXACT_FP32 else out
    if s["op"] == "apply":
        s["pmg"].apply(s["r"], out)
        return out.float()
    s["pmg"].refresh(W, s["sigma"])
    out.copy_(W)
    for _ in range(2):
        mesh.bdf2_rhs(out, W, W, s["dt"], s["b"])
        s["pmg"].fgmres(out, s["b"], s["dW"], rtol=1e-5, max_restarts=4)
        mesh.axpy(1.0, s["dW"], out)
    return out


# ------------------------------------------------------------------ work
def _work_rhs(c, jvp):
    """Operations of one residual or product: basis contractions by sum
    factorisation (tensor elements; dense ones on triangles) both ways, and
    the pointwise fluxes; bytes: the vectors."""
    d, p, E, nm = _dim(c), c["p"], _n_elem(c), _n_modes(c)
    m, q = d + 2, p + 2
    fields = m * (2 if jvp else 1)
    if c["space"] == "tri":
        vol = 2 * q**2 * nm * (fields + m) * (1 + d) + q**2 * (600 if jvp else 250)
        face = 1.5 * (2 * 2 * q * nm * (fields + m) * (1 + d) + q * (2000 if jvp else 900))
    else:
        def tensor(d):  # one field, one way: contract one index after the other
            return sum(2 * (math.comb(p + d - j, d - j) if c["space"] == "P" else (p + 1) ** (d - j)) * q ** (j + 1)
                       for j in range(d))
        vol = (fields + m) * 0.5 * (1 + d) * tensor(d) + q**d * (600 if jvp else 250)
        face = d * (2 * (fields + m) * (4 * nm + 0.5 * (1 + d) * tensor(d - 1)) + q ** (d - 1) * (2000 if jvp else 900))
    return E * (vol + face)


def work(case):
    c = case
    if c["op"] == "serve":
        ws = [work(r) for r in _requests(c)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    N = _dofs(c)
    if c["op"] == "residual":
        return {"bytes": 16 * N, "flops": _work_rhs(c, False)}
    if c["op"] == "jvp":
        return {"bytes": 24 * N, "flops": _work_rhs(c, True)}
    # preconditioner: a full cycle smooths each level with GMRES (10 + 10, coarsest 30); every iteration is one
    # product and one block-Jacobi apply, whose blocks are read again each time where they exceed the caches
    E, d = _n_elem(c), _dim(c)
    levels = [int(x) for x in c["levels"].split(",")]
    size = (8 if c.get("precision") == "fp64" else 2 if c["storage"] == "bf16" else 4)
    faces = 3 if c["space"] == "tri" else 2 * d
    fl, by = 0.0, 16.0 * N
    for l, p in enumerate(levels):
        nb = (d + 2) * _n_modes(c, p)
        if len(levels) == 1:
            its = 1
        else:
            # the full cycle meets level l once itself and once from each finer one
            its = (l + 1) * (20 if l < len(levels) - 1 else 30)
        blocks = E * nb * nb * (1 + (1 + faces if l else 0))
        fl += its * 2 * blocks + (its * _work_rhs(c, True) if l == 0 and len(levels) > 1 else 0)
        by += (its if blocks * size > 1.2e8 else 1) * blocks * size
    if c["op"] == "apply":
        return {"bytes": by, "flops": fl}
    # step: two right-hand sides, two solves of at least one iteration (product and application), and a refresh:
    # diagonal blocks (contractions of the pointwise Jacobians with both bases) and their inverses
    nb = (d + 2) * _n_modes(c)
    pts = (c["p"] + 2) ** d + faces * (c["p"] + 2) ** (d - 1)
    refresh = E * (2 * nb * nb * pts * (1 + d) / (4 if c["space"] != "tri" else 1) + 2.0 * nb**3)
    return {"bytes": 2 * by + 8 * N + 2.0 * E * nb * nb * size,
            "flops": 2 * (fl + _work_rhs(c, True) + _work_rhs(c, False)) + refresh}


# ------------------------------------------------------------------ exact values
def _geometry(c, extra=0):
    """Reference tables, affine maps, points and face pairs of the case's mesh
    (extra: so many more quadrature points per direction)."""
    return _geometry_tri(c, extra) if c["space"] == "tri" else _geometry_box(c, extra)


def _t(x, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=dtype, device="cuda")


def _geometry_box(c, extra):
    d, p = _dim(c), c["p"]
    q = p + 2 + (extra - 1 if extra else 0)
    n = [c["n0"], c["n1"], c["n2"]][:d]
    lo, hi = _box(c)
    h = [(hi[k] - lo[k]) / n[k] for k in range(d)]
    x, w = np.polynomial.legendre.leggauss(q)
    V, D = _legendre(p, x)
    Ve, De = _legendre(p, np.array([-1.0, 1.0]))
    md = _modes(c)

    def table(vals, pts, der=None):
        """prod_k vals[k][point_k, mode_k] with direction `der` differentiated"""
        out = np.ones((len(pts), len(md)))
        for k in range(d):
            t = vals[k][1 if der == k else 0]
            out *= t[np.array([a[k] for a in pts])][:, [a[k] for a in md]]
        return out

    pts = list(itertools.product(range(q), repeat=d))
    vol = [(V, D)] * d
    wq = np.prod([w[[a[k] for a in pts]] for k in range(d)], axis=0)
    xi = np.stack([x[[a[k] for a in pts]] for k in range(d)], axis=1)
    E = int(np.prod(n))
    e = np.arange(E)
    ijk = [e % n[0], e // n[0] % n[1]] + ([e // (n[0] * n[1])] if d == 3 else [])
    ctr = _t(np.stack([lo[k] + (ijk[k] + 0.5) * h[k] for k in range(d)], axis=1))
    half = _t(np.array(h) / 2)
    g = dict(d=d, E=E, phi=_t(table(vol, pts)), dphi=_t(np.stack([table(vol, pts, k) for k in range(d)])), wq=_t(wq),
             J=torch.diag(2 / half / 2).expand(E, d, d), det=torch.full((E,), float(np.prod(h)) / 2**d,
                                                                       dtype=torch.float64, device="cuda"),
             eta=2.0 * d + 1, faces=[], at=lambda a, b: ctr[a:b, None] + _t(xi)[None] * half)
    if extra:
        return g
    for k in range(d):
        sides = []
        fp = [t[:k] + (0,) + t[k:] for t in itertools.product(range(q), repeat=d - 1)]
        for s in (0, 1):
            tabs = [(V, D)] * d
            tabs[k] = (Ve[s:s + 1], De[s:s + 1])
            sides.append((_t(table(tabs, fp)), _t(np.stack([table(tabs, fp, j) for j in range(d)]))))
        wf = np.prod([w[[a[j] for a in fp]] for j in range(d) if j != k], axis=0)
        j = [i.copy() for i in ijk]
        j[k] = (j[k] + 1) % n[k]
        right = j[0] + n[0] * (j[1] + (n[1] * j[2] if d == 3 else 0))
        nrm = np.zeros((E, d))
        nrm[:, k] = 1.0
        g["faces"].append(dict(L=_t(e, torch.int64), R=_t(right, torch.int64), tL=sides[1], tR=sides[0], wf=_t(wf),
                               n=_t(nrm), JF=_t(np.full(E, np.prod([h[i] / 2 for i in range(d) if i != k])))))
    return g


def _tri_basis(p, r, s):
    """The orthonormal Dubiner polynomials and their (r, s) derivatives at
    points: Gram-Schmidt of Legendre products on the reference triangle, degree
    by degree with the r-degree rising, which is what the closed form spans."""
    x, w = np.polynomial.legendre.leggauss(p + 3)
    a, b = (t.ravel() for t in np.meshgrid(x, x))
    wq = (np.outer(w, w)).ravel() * (1 - b) / 2
    order = sorted(_tri_modes(p), key=lambda t: (t[0] + t[1], t[0]))

    def products(r, s):
        (Vr, Dr), (Vs, Ds) = _legendre(p, np.asarray(r)), _legendre(p, np.asarray(s))
        i, j = [t[0] for t in order], [t[1] for t in order]
        return Vr[:, i] * Vs[:, j], Dr[:, i] * Vs[:, j], Vr[:, i] * Ds[:, j]

    A = products((1 + a) * (1 - b) / 2 - 1, b)[0] * np.sqrt(wq)[:, None]
    T = np.linalg.qr(A, mode="r")
    T = T * np.sign(np.diag(T))[:, None]
    back = [order.index(t) for t in _tri_modes(p)]
    return [np.linalg.solve(T.T, f.T).T[:, back] for f in products(r, s)]


def _geometry_tri(c, extra):
    p = c["p"]
    q = p + 2 + (extra - 1 if extra else 0)
    msh = wl.tri_mesh(_config(c))
    Vx = msh["X"][msh["tri"]] + msh["shift"] * (msh["hi"] - msh["lo"])
    E = len(Vx)
    x, w = np.polynomial.legendre.leggauss(q)
    a, b = np.tile(x, q), np.repeat(x, q)
    wq = np.tile(w, q) * np.repeat(w, q) * (1 - b) / 2
    r, s = (1 + a) * (1 - b) / 2 - 1, b
    f = _tri_basis(p, r, s)
    J = np.stack([Vx[:, 1] - Vx[:, 0], Vx[:, 2] - Vx[:, 0]], axis=2) / 2
    V0, Jt, xi = _t(Vx[:, 0]), _t(J), _t(np.stack([r, s], axis=1) + 1)
    g = dict(d=2, E=E, phi=_t(f[0]), dphi=_t(np.stack(f[1:])), wq=_t(wq), J=_t(np.linalg.inv(J)),
             det=_t(np.linalg.det(J)), eta=4.0, faces=[],
             at=lambda a, b: V0[a:b, None] + torch.einsum("ekl,ql->eqk", Jt[a:b], xi))
    if extra:
        return g
    ref = np.array([[-1.0, -1.0], [1.0, -1.0], [-1.0, 1.0]])
    seen, pairs = {}, {}
    for e in range(E):
        for k in range(3):
            i, j = (int(msh["tri"][e, t]) for t in (k, (k + 1) % 3))
            dl = tuple(int(t) for t in msh["shift"][e, (k + 1) % 3] - msh["shift"][e, k])
            key = min((i, j, dl), (j, i, tuple(-t for t in dl)))
            if key in seen:
                e0, k0 = seen.pop(key)
                pairs.setdefault((k0, k), []).append((e0, e))
            else:
                seen[key] = (e, k)
    tab = []
    for k in range(3):
        A0, B0 = ref[k], ref[(k + 1) % 3]
        pt = A0 + (B0 - A0) * ((1 + x) / 2)[:, None]
        tab.append([_tri_basis(p, *pt.T), _tri_basis(p, *pt[::-1].T)])
    for (kL, kR), es in pairs.items():
        es = np.array(es)
        dv = Vx[es[:, 0], (kL + 1) % 3] - Vx[es[:, 0], kL]
        ln = np.hypot(dv[:, 0], dv[:, 1])
        tL, tR = tab[kL][0], tab[kR][1]
        g["faces"].append(dict(L=_t(es[:, 0], torch.int64), R=_t(es[:, 1], torch.int64), wf=_t(w), JF=_t(ln / 2),
                               tL=(_t(tL[0]), _t(np.stack(tL[1:]))), tR=(_t(tR[0]), _t(np.stack(tR[1:]))),
                               n=_t(np.stack([dv[:, 1], -dv[:, 0]], axis=1) / ln[:, None])))
    return g


def _prim(u):
    d = len(u) - 2
    vel = [u[1 + j] / u[0] for j in range(d)]
    pr = (GAMMA - 1) * (u[-1] - 0.5 * u[0] * sum(v * v for v in vel))
    return vel, pr, (u[-1] + pr) / u[0]


def _inviscid(u, n):
    """F_c(u) . n; n: d numbers or arrays."""
    vel, pr, h0 = _prim(u)
    vn = sum(v * k for v, k in zip(vel, n))
    return [u[0] * vn] + [u[1 + j] * vn + pr * n[j] for j in range(len(vel))] + [u[0] * vn * h0]


def _viscous(u, g, mu):
    """K(u) g as F[v][k] (v >= 1): (tau, v . tau + kappa grad T) for the gradient-shaped g[v][k]."""
    d = len(u) - 2
    vel = _prim(u)[0]
    e0 = u[-1] / u[0]
    gv = [[(g[1 + j][k] - vel[j] * g[0][k]) / u[0] for k in range(d)] for j in range(d)]
    gT = [(GAMMA - 1) * ((g[-1][k] - e0 * g[0][k]) / u[0] - sum(vel[j] * gv[j][k] for j in range(d))) for k in range(d)]
    div = sum(gv[j][j] for j in range(d))
    kap = mu * GAMMA / ((GAMMA - 1) * PR)
    tau = [[mu * (gv[j][k] + gv[k][j]) - (2 / 3 * mu * div if j == k else 0.0) for k in range(d)] for j in range(d)]
    return [None] + tau + [[sum(vel[j] * tau[j][k] for j in range(d)) + kap * gT[k] for k in range(d)]]


def _roe(uL, uR, n):
    d = len(uL) - 2
    (vL, pL, hL), (vR, pR, hR) = _prim(uL), _prim(uR)
    sL, sR = torch.sqrt(uL[0]), torch.sqrt(uR[0])
    rho = sL * sR
    vel = [(sL * vL[j] + sR * vR[j]) / (sL + sR) for j in range(d)]
    h0 = (sL * hL + sR * hR) / (sL + sR)
    q2 = sum(v * v for v in vel)
    c2 = (GAMMA - 1) * (h0 - 0.5 * q2)
    cs = torch.sqrt(c2)
    vn = sum(vel[j] * n[j] for j in range(d))
    dr, dp, dv = uR[0] - uL[0], pR - pL, [vR[j] - vL[j] for j in range(d)]
    dvn = sum(dv[j] * n[j] for j in range(d))

    def speed(lam):
        dl = ROE_DELTA * cs
        return torch.where(lam.abs() < dl, (lam * lam + dl * dl) / (2 * dl), torch.where(lam >= 0, lam, -lam))

    a1 = speed(vn - cs) * (dp - rho * cs * dvn) / (2 * c2)
    a3 = speed(vn + cs) * (dp + rho * cs * dvn) / (2 * c2)
    l2 = speed(vn)
    a2 = l2 * (dr - dp / c2)
    out = [a1 + a3 + a2]
    for j in range(d):
        out.append(a1 * (vel[j] - cs * n[j]) + a3 * (vel[j] + cs * n[j]) + a2 * vel[j] + l2 * rho * (dv[j] - dvn * n[j]))
    vdv = sum(vel[j] * dv[j] for j in range(d))
    out.append(a1 * (h0 - cs * vn) + a3 * (h0 + cs * vn) + a2 * 0.5 * q2 + l2 * rho * (vdv - vn * dvn))
    FL, FR = _inviscid(uL, n), _inviscid(uR, n)
    return [0.5 * (FL[v] + FR[v] - out[v]) for v in range(d + 2)]


def _residual(g, mu, W):
    """R(W), M dW/dt + R(W) = 0: volume term, Roe and BR2 fluxes, dual-consistency term."""
    d = g["d"]
    m = d + 2

    def traces(Wt, tab, J):
        U = Wt @ tab[0].T
        G = [Wt @ t.T for t in tab[1]]
        gr = [sum(J[:, l, k, None, None] * G[l] for l in range(d)) for k in range(d)]
        return [U[:, v] for v in range(m)], [[gr[k][:, v] for k in range(d)] for v in range(m)]

    def tested(F, tab, J):
        """sum_q F[v][k] d_k phi_i, F[v] None for no flux"""
        out = []
        for v in range(m):
            if F[v] is None:
                out.append(torch.zeros_like(W[:1, 0]).expand(len(J), -1))
            else:
                out.append(sum(sum(J[:, l, k, None] * F[v][k] for k in range(d)) @ tab[1][l] for l in range(d)))
        return torch.stack(out, dim=1)

    J, det = g["J"], g["det"]
    u, gr = traces(W, (g["phi"], g["dphi"]), J)
    unit = [[1.0 if j == k else 0.0 for j in range(d)] for k in range(d)]
    Fc = [_inviscid(u, unit[k]) for k in range(d)]
    Kg = _viscous(u, gr, mu)
    F = [[(Fc[k][v] - (Kg[v][k] if v else 0.0)) * g["wq"] for k in range(d)] for v in range(m)]
    R = -det[:, None, None] * tested(F, (g["phi"], g["dphi"]), J)
    del u, gr, Fc, Kg, F
    for f in g["faces"]:
        L, Rr, wf = f["L"], f["R"], f["wf"]
        n = [f["n"][:, k, None] for k in range(d)]
        JL, JR = J[L], J[Rr]
        uL, gL = traces(W[L], f["tL"], JL)
        uR, gR = traces(W[Rr], f["tR"], JR)
        jump = [[(uL[v] - uR[v]) * n[k] for k in range(d)] for v in range(m)]
        XL, XR = _viscous(uL, jump, mu), _viscous(uR, jump, mu)
        KL, KR = _viscous(uL, gL, mu), _viscous(uR, gR, mu)
        flux = _roe(uL, uR, n)
        clL, clR = (f["JF"] / (2 * det[i]) for i in (L, Rr))
        for v in range(1, m):
            nL, nR = (sum(X[v][k] * n[k] for k in range(d)) for X in (XL, XR))
            lift = clL[:, None] * (((nL * wf) @ f["tL"][0]) @ f["tL"][0].T) + \
                clR[:, None] * (((nR * wf) @ f["tR"][0]) @ f["tR"][0].T)
            flux[v] = flux[v] - sum(0.5 * (KL[v][k] + KR[v][k]) * n[k] for k in range(d)) + 0.5 * g["eta"] * lift
        fw = torch.stack([x * wf for x in flux], dim=1)
        half = [[None] + [[0.5 * X[v][k] * wf for k in range(d)] for v in range(1, m)] for X in (XL, XR)]
        JF = f["JF"][:, None, None]
        R = R.index_add(0, L, JF * (fw @ f["tL"][0] - tested(half[0], f["tL"], JL)))
        R = R.index_add(0, Rr, JF * (-(fw @ f["tR"][0]) - tested(half[1], f["tR"], JR)))
    return R


def _product(g, mu, W, v, sigma):
    _, t = torch.func.jvp(lambda x: _residual(g, mu, x), (W,), (v,))
    return t + sigma * g["det"][:, None, None] * v


def _replayed(f, *like):
    """f captured as a CUDA graph on buffers of its own: called with tensors to
    copy into them (None: as they are), it returns the graph's output buffer."""
    own = [x.clone() for x in like]
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        f(*own)
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = f(*own)

    def call(*xs):
        for o, x in zip(own, xs):
            if x is not None:
                o.copy_(x)
        graph.replay()
        return out

    return call


def _gmres(A, b, rtol, most):
    nb = float(b.norm())
    Q, H = b.new_empty((most + 1, b.numel())), np.zeros((most + 1, most))
    Q[0] = b.reshape(-1) / nb
    for j in range(most):
        w = A(Q[j].reshape(b.shape)).reshape(-1)
        V = Q[:j + 1]
        for _ in range(2):
            h = V @ w
            w = w - h @ V
            H[:j + 1, j] += h.cpu().numpy()
        H[j + 1, j] = float(w.norm())
        if j % 8 == 7 or j == most - 1:
            rhs = np.zeros(j + 2)
            rhs[0] = nb
            y, *_ = np.linalg.lstsq(H[:j + 2, :j + 1], rhs, rcond=None)
            if np.linalg.norm(H[:j + 2, :j + 1] @ y - rhs) <= rtol * nb or j == most - 1:
                return (torch.as_tensor(y, device=b.device) @ V).reshape(b.shape)
        Q[j + 1] = w / H[j + 1, j]


def _exact_step(c, seed, limit_s):
    """W^{n+1} of the BDF2 step with W^{n-1} = W^n, solved until Newton stalls; None where time runs out."""
    began = time.monotonic()
    g, mu, Wn, dt = _geometry(c), _mu(c), _state(c, seed), _dt(c)
    det, sigma = g["det"][:, None, None], 1.5 / dt
    W, first = Wn.clone(), None
    product = _replayed(lambda w, v: _product(g, mu, w, v, sigma) / (det * sigma), W, W)
    for _ in range(8):
        f = -(W - Wn) * sigma - _residual(g, mu, W) / det
        if float(f.norm()) <= 1e-13 * sigma * float(W.norm()):
            break
        first = first or float(f.norm())

        def A(v):
            if time.monotonic() - began > limit_s:
                raise TimeoutError
            return product(None, v).clone()

        product(W, W)
        try:
            dW = _gmres(A, f / sigma, 1e-6, 400)
        except TimeoutError:
            return None
        W = W + dW
        if float(dW.norm()) <= 1e-12 * float(W.norm()):
            return W
    return W if float(f.norm()) <= 1e-9 * first else None


def exact(case, seed):
    c = case
    if c["op"] == "apply":
        return None  # the blocks alone take hundreds of products
    if c["op"] == "serve":
        out = [_exact_step(r, seed + k, 12.0 / c["count"]) for k, r in enumerate(_requests(c))]
        return None if all(W is None for W in out) else [None if W is None else W.cpu().numpy() for W in out]
    if c["op"] == "step":
        return _exact_step(c, seed, 12.0)
    g, mu, W = _geometry(c), _mu(c), _state(c, seed)
    if c["op"] == "residual":
        return _residual(g, mu, W)
    sigma = 1.5 / _dt(dict(c, dt=0.01 if c["flow"] == "tgv" else 0.05))
    return _product(g, mu, W, _vector(c, W, seed, 1), sigma)
