"""The work that a user of the p-multigrid DG solver has it do, as cases to time.

A program that steps a flow in time calls, per implicit stage: the residual and the linearisation
(`dg_set_linearization_rhs`), the preconditioner's assembly, the solve (`fgmres_solve`, or a captured
`Plan`) and `dg_stage_update`; around them stand the exact Jacobian action (`dg_jvp`), the multigrid cycle
(`pmg_vcycle`) and the training of the learned coarse correction. Every case goes through the package's
public entry points on a state of the flow the repository works with: the Taylor-Green vortex on a periodic
box, or the laminar profile of the walled channel, each with a seeded smooth divergence-free perturbation,
projected onto the modal basis.

Sizes are the repository's own workloads (4^3 P2, 16^3, 24^3 and 32^3 P4, the 24 x 12 x 12 P3 channel, the
batch of uneven boxes), and ragged stretched boxes between them. Solves run to a tolerance far below the
rounding of the reduced-precision cycle, so that the solution, with its free constant pressure projected out,
does not depend on that rounding.

`exact` evaluates the residual and its linearisation in plain torch, FP64, by dense quadrature.
"""
import math

import numpy as np
import torch

import paper_1809_00866_gb300 as P

TWO_PI = 2.0 * math.pi
NU_BOX = 1.0 / 1600.0  # Taylor-Green vortex at Re = 1600
NU_CHANNEL = 2.0 / 180.0 ** 2  # laminar profile of friction Reynolds number 180
AC_C = 1.0
ETA = 7.0
CFL = 50.0  # acoustic; the smallest box steps more carefully
MODES = 8  # Fourier modes per component of the perturbation's vector potential
LEVELS = {1: (1,), 2: (2, 1), 3: (3, 2, 1), 4: (4, 2, 1)}


def nb_of(k):
    return (k + 1) * (k + 2) * (k + 3) // 6


def listed():
    return [
        # the smallest call: one Jacobian action on the 4^3 P2 box (launch latency)
        box("jv_tiny", "jv", 4, 4, 4, 2),
        # an ordinary one: the outer products of the 16^3 P4 stage
        box("jv_box", "jv", 16, 16, 16, 4),
        # the largest operator application: 4.6 million unknowns
        box("jv_large", "jv", 32, 32, 32, 4),
        # an explicit or host-driven integrator's right-hand side, on an odd, stretched mesh
        box("residual_ragged", "residual", 13, 9, 11, 3, mesh="stretched"),
        # start of every implicit stage (right-hand side and linearisation), and the first product with it
        box("linearize_large", "linearize", 24, 24, 24, 4),
        # one cycle of the paper's preconditioner in FP64 (2/2/2 block-Jacobi sweeps)
        box("vcycle_fp64", "vcycle", 16, 16, 16, 4),
        # a whole stage of the smallest workload with the host-driven solver
        box("stage_tiny", "stage", 4, 4, 4, 2, precision="fp64", solver="fgmres", cfl=10.0),
        # a whole stage in the paper's form: FP64 assembly, FP64 cycle
        box("stage_fp64", "stage", 12, 12, 12, 3, precision="fp64", solver="plan"),
        # the headline: a whole stage at 32^3 P4 with the FP16 tensor-core cycle inside FP64 FGMRES
        box("stage_large", "stage", 32, 32, 32, 4, precision="h16tc", solver="plan"),
        # the same on the no-slip channel
        dict(name="stage_channel", kind="stage", nx=24, ny=12, nz=12, k=3, mesh="channel", precision="h16tc",
             solver="plan"),
        # independent uneven boxes of three degrees in one captured plan
        dict(name="batch_uneven", kind="batch", count=16, nmin=6, nmax=10, boxes=64),
        # one gradient of the coarse network's training over 16384 pairs
        dict(name="train_coarse", kind="train", rows=16384),
    ]


def box(name, kind, nx, ny, nz, k, mesh="uniform", **kw):
    return dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, k=k, mesh=mesh, **kw)


def draw(rng):
    kind = rng.choice(["jv", "jv", "residual", "linearize", "vcycle", "stage", "stage", "channel", "batch", "train"])
    if kind == "train":
        return dict(kind="train", rows=int(round(math.exp(rng.uniform(math.log(300), math.log(16384))))))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(3, 16), nmin=rng.randint(5, 7), nmax=rng.randint(7, 10),
                    boxes=rng.randint(1, 1000))
    if kind == "channel":
        return dict(kind="stage", nx=rng.randint(8, 24), ny=rng.randint(6, 12), nz=rng.randint(6, 12),
                    k=rng.choice([2, 3]), mesh="channel", precision=rng.choice(["h16", "h16tc", "fp32"]),
                    solver="plan")
    k = rng.choice([2, 3, 4, 4] + ([1] if kind in ("jv", "residual") else []))
    top = {"jv": 32000, "residual": 16000, "linearize": 13000, "vcycle": 4000, "stage": 4000}[kind]
    ne = math.exp(rng.uniform(math.log(30), math.log(top)))
    side = ne ** (1.0 / 3.0)
    n = [max(3, int(round(side * math.exp(rng.uniform(-0.35, 0.35))))) for _ in range(3)]
    case = box("", kind, n[0], n[1], n[2], k, mesh=rng.choice(["uniform", "stretched"]))
    del case["name"]
    if kind == "stage":
        case["mesh"] = "uniform"
        m = max(6, int(round(side)))
        case.update(nx=m, ny=m, nz=m, precision=rng.choice(["fp64", "fp32", "h16", "h16tc", "h16tc", "bf16"]))
        case["solver"] = rng.choice(["fgmres", "plan"])
    return case


# ---------------------------------------------------------------- meshes and states


def nodes(case):
    """The case's boxes, each (x, y, z) node coordinates."""
    if case["kind"] == "batch":
        rs = np.random.RandomState(case["boxes"])
        out = {2: [], 3: [], 4: []}
        for q in range(case["count"]):
            n, k = int(rs.randint(case["nmin"], case["nmax"] + 1)), 2 + q % 3
            out[k].append((np.linspace(0.0, TWO_PI, n + 1),) * 3)
        return out
    if case["mesh"] == "channel":
        s = np.linspace(-1.0, 1.0, case["ny"] + 1)
        y = np.tanh(1.3 * s) / np.tanh(1.3)  # cells shrink towards the walls
        return [(np.linspace(0.0, TWO_PI, case["nx"] + 1), y, np.linspace(0.0, math.pi, case["nz"] + 1))]
    xs = []
    for d, key in enumerate(("nx", "ny", "nz")):
        n = case[key]
        h = np.ones(n)
        if case["mesh"] == "stretched":
            h += 0.25 * (2.0 * np.random.RandomState(17 * n + d).rand(n) - 1.0)
        x = np.concatenate([[0.0], np.cumsum(h)])
        xs.append(x * (TWO_PI / x[-1]))
    return [tuple(xs)]


def shift_of(b, k, cfl=CFL):
    """1 / dt of an acoustic CFL number on the box's smallest cell."""
    h = min(float(np.diff(x).min()) for x in b)
    return (2 * k + 1) * (1.0 + math.sqrt(2.0)) / (cfl * h)


class Basis:
    """Orthonormal modal basis of total degree k on [-1, 1]^3: exponents, Gauss rule, tables (numpy)."""

    def __init__(self, k):
        self.k, self.n = k, k + 1
        self.x, self.w = np.polynomial.legendre.leggauss(k + 1)
        self.exps = [(a, b, t - a - b) for t in range(k + 1) for a in range(t, -1, -1) for b in range(t - a, -1, -1)]
        self.nb = len(self.exps)

    def p(self, x, deriv=False):
        """[n, len(x)] values (or derivatives) of the normalised Legendre polynomials."""
        rows = []
        for a in range(self.k + 1):
            c = np.zeros(a + 1)
            c[a] = math.sqrt((2 * a + 1) / 2.0)
            rows.append(np.polynomial.legendre.legval(x, np.polynomial.legendre.legder(c) if deriv else c)
                        * np.ones(len(x)))
        return np.stack(rows)

    def table(self, points, d=None):
        """[q, nb] basis at the tensor points (one 1D array per axis), differentiated along axis d."""
        one = [self.p(x, deriv=(d == a)) for a, x in enumerate(points)]
        t = np.stack([np.einsum("i,j,l->ijl", one[0][a], one[1][b], one[2][c]) for a, b, c in self.exps], axis=-1)
        return t.reshape(-1, self.nb)


def geometry(boxes):
    """Cell sizes and lower corners [ne, 3] of all boxes' cells, one after another, x fastest."""
    hs, los = [], []
    for b in boxes:
        h = np.meshgrid(*[np.diff(x) for x in b], indexing="ij")
        lo = np.meshgrid(*[x[:-1] for x in b], indexing="ij")
        hs.append(np.stack([a.transpose(2, 1, 0).reshape(-1) for a in h], -1))
        los.append(np.stack([a.transpose(2, 1, 0).reshape(-1) for a in lo], -1))
    return np.concatenate(hs), np.concatenate(los)


def field(case, seed, x, y, z):
    """(u, v, w, p) at points: the base flow plus 0.05 times a unit-rms divergence-free perturbation, the
    curl of a vector potential of seeded Fourier modes, which vanishes with its gradient on channel walls."""
    rs = np.random.RandomState((seed * 7919 + 11) % (2 ** 31))
    kk, ph = rs.randint(1, 4, size=(3, MODES, 3)).astype(float), rs.uniform(0.0, TWO_PI, (3, MODES))
    aa = rs.standard_normal((3, MODES))
    wall = case.get("mesh") == "channel"
    if wall:
        kk[..., 2] = 2.0 * rs.randint(1, 3, size=(3, MODES))  # the box is pi wide along z

    def curl(x, y, z):
        g, dg = ((1.0 - y * y) ** 2, -4.0 * y * (1.0 - y * y)) if wall else (1.0, 0.0)
        d = [[0.0] * 3 for _ in range(3)]
        for i in range(3):
            for m in range(MODES):
                t = kk[i, m, 0] * x + kk[i, m, 1] * y + kk[i, m, 2] * z + ph[i, m]
                s, c = torch.sin(t) * aa[i, m], torch.cos(t) * aa[i, m]
                d[i][0] = d[i][0] - kk[i, m, 0] * s * g
                d[i][1] = d[i][1] - kk[i, m, 1] * s * g + c * dg
                d[i][2] = d[i][2] - kk[i, m, 2] * s * g
        return [d[2][1] - d[1][2], d[0][2] - d[2][0], d[1][0] - d[0][1]]

    ax = torch.linspace(0.0, TWO_PI, 17, dtype=torch.float64, device=x.device)[:-1]
    ay = torch.linspace(-1.0, 1.0, 17, dtype=torch.float64, device=x.device) if wall else ax
    gx, gy, gz = torch.meshgrid(ax, ay, ax, indexing="ij")
    rms = math.sqrt(float(sum((t * t).mean() for t in curl(gx, gy, gz))))
    du = [0.05 / rms * t for t in curl(x, y, z)]
    if wall:
        return 1.0 - y * y + du[0], du[1], du[2], 0.0 * x
    return (torch.sin(x) * torch.cos(y) * torch.cos(z) + du[0], -torch.cos(x) * torch.sin(y) * torch.cos(z) + du[1],
            du[2], (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2.0) / 16.0)


def dev(a, device):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=device)


def state(case, seed, boxes, k, device="cuda"):
    """[ne, 4, nb] modal coefficients: the Gauss-rule L2 projection of the field."""
    B = Basis(k)
    h, lo = (dev(a, device) for a in geometry(boxes))
    x1, w1 = dev(B.x, device), B.w
    pts = [(lo[:, d, None] + 0.5 * h[:, d, None] * (x1 + 1.0)) for d in range(3)]
    n = B.n
    full = [pts[0][:, :, None, None].expand(-1, n, n, n), pts[1][:, None, :, None].expand(-1, n, n, n),
            pts[2][:, None, None, :].expand(-1, n, n, n)]
    f = torch.stack([t.expand(h.shape[0], n, n, n).reshape(-1, n ** 3) for t in field(case, seed, *full)], 1)
    tab = dev(B.table([B.x] * 3) * np.einsum("i,j,l->ijl", w1, w1, w1).reshape(-1, 1), device)
    return torch.einsum("evq,qm->evm", f, tab).mul_(h.prod(1).div(8.0).sqrt()[:, None, None]).contiguous()


def direction(shape, k, seed, device="cuda"):
    """Seeded direction: N(0, 1) coefficients over 1 + degree."""
    g = torch.Generator(device="cpu").manual_seed(int(seed) + 1809)
    deg = np.array([sum(e) for e in Basis(k).exps])
    return torch.randn(shape, generator=g, dtype=torch.float64).to(device) / dev(1.0 + deg, device)


def options(case):
    prec = {"fp64": P.DG_PRECOND_FP64, "fp32": P.DG_PRECOND_FP32, "h16": P.DG_PRECOND_FP32_H16,
            "bf16": P.DG_PRECOND_FP32_BF16, "h16tc": P.DG_PRECOND_FP32_H16_TC}[case.get("precision", "h16")]
    if prec == P.DG_PRECOND_FP64:
        return P.solve_opts(rtol=1e-11, maxit=300, omega=0.9, precision=prec)
    return P.solve_opts(rtol=1e-11, maxit=300, omega=0.95, pre_sweeps=5, post_sweeps=5, precision=prec)


def handle(case, boxes, k):
    nu = NU_CHANNEL if case.get("mesh") == "channel" else NU_BOX
    if case["kind"] == "batch":
        return P.DG(None, None, None, LEVELS[k], nu, AC_C, ETA, boxes=boxes)
    return P.DG(*boxes[0], LEVELS[k], nu, AC_C, ETA, walls=case.get("mesh") == "channel")


# ---------------------------------------------------------------- the cases' programs


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        X, T, theta = pairs(case, seed)
        return dict(case=case, X=X, T=T, theta=theta, ws=P.mlp_workspace(case["rows"]),
                    grad=torch.empty_like(theta), loss=torch.empty(1, device="cuda"))
    if kind == "batch":
        parts, opts = [], options(case)
        for k, boxes in nodes(case).items():
            if not boxes:
                continue
            dg = handle(case, boxes, k)
            dg.dg_set_problem_shifts([shift_of(b, k) for b in boxes])
            w = state(case, seed, boxes, k)
            dg.dg_set_linearization(w, 1.0)
            dg.dg_assemble(precision=opts.precision)
            parts.append(dict(dg=dg, w=w, g=dg.empty(), x=dg.empty()))
        plan = P.Plan([p["dg"] for p in parts], [p["g"] for p in parts], [p["x"] for p in parts], opts)
        return dict(case=case, parts=parts, plan=plan, opts=opts)
    k, boxes = case["k"], nodes(case)
    dg = handle(case, boxes, k)
    w = state(case, seed, boxes, k)
    st = dict(case=case, dg=dg, w=w, inv=shift_of(boxes[0], k, case.get("cfl", CFL)), out=dg.empty())
    if kind in ("jv", "linearize", "vcycle"):
        st["v"] = direction(w.shape, k, seed)
    if kind == "jv":
        dg.dg_set_linearization(w, st["inv"])
    elif kind == "linearize":
        st["g"] = dg.empty()
    elif kind == "vcycle":
        dg.dg_set_linearization(w, st["inv"])
        dg.dg_assemble()
        st["opts"] = P.solve_opts(omega=0.9)
    elif kind == "stage":
        # a time-stepping program has its mesh's part of the assembly from its first stage on
        opts = st["opts"] = options(case)
        st.update(g=dg.empty(), x=dg.empty())
        if len(LEVELS[k]) > 1:
            dg.dg_set_stb_rescaling(True)
        dg.dg_set_linearization(w, st["inv"])
        dg.dg_assemble(precision=opts.precision)
        if case["solver"] == "plan":
            st["plan"] = P.Plan([dg], [st["g"]], [st["x"]], opts)
    return st


def run(st):
    kind = st["case"]["kind"]
    if kind == "train":
        P.dg_mlp_grad(st["theta"], st["X"], st["T"], st["case"]["rows"], st["grad"], loss=st["loss"], ws=st["ws"])
        return [st["loss"], st["grad"]]
    if kind == "batch":
        for p in st["parts"]:
            p["dg"].dg_set_linearization_rhs(p["w"], 1.0, p["g"])
            p["dg"].dg_assemble(precision=st["opts"].precision)
        st["plan"].dg_plan_solve()
        return [[p["g"], without_constant(p)] for p in st["parts"]]
    dg = st["dg"]
    if kind == "residual":
        dg.dg_residual(st["w"], st["out"])
        return st["out"]
    if kind == "jv":
        dg.dg_jvp(st["v"], st["out"])
        return st["out"]
    if kind == "linearize":
        dg.dg_set_linearization_rhs(st["w"], st["inv"], st["g"])
        dg.dg_jvp(st["v"], st["out"])
        return [st["g"], st["out"]]
    if kind == "vcycle":
        dg.pmg_vcycle(st["v"], st["out"], st["opts"])
        return st["out"]
    dg.dg_set_linearization_rhs(st["w"], st["inv"], st["g"])
    dg.dg_assemble(precision=st["opts"].precision)
    if "plan" in st:
        st["plan"].dg_plan_solve()
    elif dg.fgmres_solve(st["g"], st["x"], st["opts"])[1] != P.DG_OK:
        raise RuntimeError("the stage's solve did not converge")
    dg.pmg_project_pressure(0, st["x"])  # the constant pressure is free
    st["out"].copy_(st["w"])
    dg.dg_stage_update(st["out"], st["x"])
    return [st["g"], st["x"], st["out"]]


def without_constant(p):
    """The batch's solution with every box's mean pressure taken out: the mean of mode 0 on uniform boxes."""
    for a, b in zip(p["dg"].elem_start[:-1], p["dg"].elem_start[1:]):
        p["x"][a:b, 3, 0] -= p["x"][a:b, 3, 0].mean()
    return p["x"]


def pairs(case, seed):
    """Training pairs of the coarse network (unit feature rows) and a network as training starts it."""
    g = torch.Generator(device="cpu").manual_seed(int(seed) + 112)
    X = torch.randn((case["rows"], P.DG_MLP_IN), generator=g)
    X /= X.norm(dim=1, keepdim=True)
    T = torch.randn((case["rows"], P.DG_MLP_OUT), generator=g) / 4.0
    shapes = [(P.DG_MLP_HIDDEN, P.DG_MLP_IN), (P.DG_MLP_HIDDEN,), (P.DG_MLP_HIDDEN, P.DG_MLP_HIDDEN),
              (P.DG_MLP_HIDDEN,), (P.DG_MLP_OUT, P.DG_MLP_HIDDEN), (P.DG_MLP_OUT,)]
    theta = torch.cat([(torch.randn(s, generator=g) / math.sqrt(s[-1])).reshape(-1) for s in shapes])
    return X.cuda(), T.cuda(), theta.cuda()


# ---------------------------------------------------------------- what a pass cannot do without


def operator_flops(k):
    """FLOP per element of one Jacobian action: modal traces, sum-factorised points and projections."""
    n, nb, n2 = k + 1, nb_of(k), (k + 1) * (k + 2) // 2
    face = 3 * 2 * (14 * nb + 12 * n * (n2 + n * n) + 32 * n * n + 24 * n2)
    vol = 2 * (18 * nb + 9 * (nb * n + n2 * n * n + n ** 4) + 6 * n ** 3 + 30 * nb)
    return float(face + vol)


def work(case):
    if case["kind"] == "train":
        r = case["rows"]
        return {"bytes": 4.0 * (r * (P.DG_MLP_IN + P.DG_MLP_OUT) + 2 * P.DG_MLP_NPARAM),
                "flops": 6.0 * P.DG_MLP_NPARAM * r}
    if case["kind"] == "batch":
        sizes = [(k, sum(int(np.prod([len(x) - 1 for x in b])) for b in bs)) for k, bs in nodes(case).items()]
        each = [work(dict(kind="stage", ne=ne, k=k)) for k, ne in sizes if ne]
        return {key: sum(w[key] for w in each) for key in ("bytes", "flops")}
    k = case["k"]
    ne = case["ne"] if "ne" in case else case["nx"] * case["ny"] * case["nz"]
    op, b = operator_flops(k) * ne, 4 * nb_of(k)
    n = 8.0 * ne * b
    cycle = 4 * op + 4 * 2.0 * b * b * ne  # four sweeps: a product with G and one with the block inverses
    vectors, flops = {"jv": (3, op), "residual": (2, op), "linearize": (4, 2 * op),
                      "vcycle": (2, cycle), "stage": (4, 12 * (cycle + op) + 2.0 * b ** 3 * ne)}[case["kind"]]
    return {"bytes": vectors * n, "flops": flops}


# ---------------------------------------------------------------- the same in plain torch, FP64


def exact(case, seed):
    if case["kind"] == "train":
        return exact_train(case, seed)
    if case["kind"] == "vcycle":
        return None  # its block inverses and coarse operators take minutes to form this way
    dual = torch.autograd.forward_ad
    if case["kind"] == "batch":
        out = []
        for k, boxes in nodes(case).items():
            if boxes:
                out.append([-Plain(case, boxes, k).residual(state(case, seed, boxes, k)), None])
        return out  # the solutions: a linear system too large for a plain solve in seconds
    boxes, k = nodes(case), case["k"]
    op, w = Plain(case, boxes, k), state(case, seed, boxes, k)

    def jvp(op, w, v):
        with dual.dual_level():
            t = dual.unpack_dual(op.residual(dual.make_dual(w, v))).tangent
        t = t.clone()
        t[:, :3] += shift_of(boxes[0], k, case.get("cfl", CFL)) * v[:, :3]
        return t

    if case["kind"] == "residual":
        return op.residual(w)
    if case["kind"] == "jv":
        return jvp(op, w, direction(w.shape, k, seed))
    if case["kind"] == "linearize":
        return [-op.residual(w), jvp(op, w, direction(w.shape, k, seed))]
    g = -op.residual(w)
    n = w.numel()
    if n > 3000:
        return [g, None, None]  # a dense solve would not fit the time
    # all columns of G: copies of the box side by side, one unit direction each
    G = torch.empty((n, n), dtype=torch.float64, device=w.device)
    many = 64
    wide = Plain(case, boxes * many, k)
    for c in range(0, n, many):
        v = torch.zeros((many, n), dtype=torch.float64, device=w.device)
        for j in range(min(many, n - c)):
            v[j, c + j] = 1.0
        t = jvp(wide, w.repeat(many, 1, 1), v.reshape(-1, *w.shape[1:])).reshape(many, n)
        G[:, c:c + many] = t[:n - c].T
    e = torch.zeros_like(w)
    e[:, 3, 0] = op.s * math.sqrt(8.0)
    e = (e / e.norm()).reshape(-1)  # the constant pressure: left and right null vector
    x = torch.linalg.solve(G + torch.outer(e, e) * G.abs().max(), g.reshape(-1))
    x = (x - e * (e @ x)).reshape(w.shape)
    return [g, x, w + x]


def exact_train(case, seed):
    X, T, theta = (t.double() for t in pairs(case, seed))
    shapes = [(128, 112), (128,), (128, 128), (128,), (16, 128), (16,)]
    ps, at = [], 0
    for s in shapes:
        m = math.prod(s)
        ps.append(theta[at:at + m].reshape(s).clone().requires_grad_(True))
        at += m
    h = torch.nn.functional.gelu(X @ ps[0].T + ps[1])
    h = torch.nn.functional.gelu(h @ ps[2].T + ps[3])
    loss = ((h @ ps[4].T + ps[5] - T) ** 2).sum(1).mean()
    loss.backward()
    return [loss.detach().reshape(1), torch.cat([p.grad.reshape(-1) for p in ps])]


class Plain:
    """The residual by dense quadrature: Gauss rule with k + 1 points per axis in the volume and on faces."""

    def __init__(self, case, boxes, k, device="cuda"):
        B = self.B = Basis(k)
        self.k, self.walls = k, case.get("mesh") == "channel"
        self.nu = NU_CHANNEL if self.walls else NU_BOX
        self.h = dev(geometry(boxes)[0], device)
        self.s = self.h.prod(1).div(8.0).sqrt()
        self.J = 2.0 / self.h
        t = lambda a: dev(a, device)  # noqa: E731
        self.vol = t(B.table([B.x] * 3))
        self.dvol = [t(B.table([B.x] * 3, d)) for d in range(3)]
        self.w3 = t(np.einsum("i,j,l->ijl", B.w, B.w, B.w).reshape(-1))
        self.w2 = t(np.einsum("i,j->ij", B.w, B.w).reshape(-1))
        self.face, self.dface, self.pairs = [], [], []
        at = 0
        plus = [[] for _ in range(3)]
        low = []
        for b in boxes:
            n = [len(x) - 1 for x in b]
            ids = at + np.arange(n[0] * n[1] * n[2]).reshape(n[2], n[1], n[0])
            for d in range(3):
                r = np.roll(ids, -1, axis=2 - d)
                if d == 1 and self.walls:
                    r[:, -1, :] = -1
                    low.append(ids[:, 0, :].reshape(-1))
                plus[d].append(r.reshape(-1))
            at += ids.size
        for d in range(3):
            sides = []
            for x in (1.0, -1.0):  # the face seen from its - side element (at xi_d = 1) and its + side one
                pts = [np.array([x]) if a == d else B.x for a in range(3)]
                sides.append((t(B.table(pts)), [t(B.table(pts, a)) for a in range(3)]))
            self.face.append([s[0] for s in sides])
            self.dface.append([s[1] for s in sides])
            p = np.concatenate(plus[d])
            i = lambda a: torch.as_tensor(a, device=device)  # noqa: E731
            inner = np.nonzero(p >= 0)[0]
            self.pairs.append((d, i(inner), i(p[inner]), 0))
            if d == 1 and self.walls:
                upper, lower = i(np.nonzero(p < 0)[0]), i(np.concatenate(low))
                self.pairs += [(d, upper, upper, 1), (d, lower, lower, -1)]

    def side(self, c, e, d, sd):
        """Values [e, 4, q] and velocity gradients [b][e, 3, q] of elements e at their face (d, sd)."""
        is_ = (1.0 / self.s[e])[:, None, None]
        u = torch.einsum("evm,qm->evq", c[e], self.face[d][sd]) * is_
        g = [torch.einsum("evm,qm->evq", c[e][:, :3], self.dface[d][sd][b]) * is_ * self.J[e, b][:, None, None]
             for b in range(3)]
        return u, g

    def residual(self, c):
        lift = [torch.zeros_like(c[:, :3]) for _ in range(3)]
        out = torch.zeros_like(c)
        for d, L, R, wall in self.pairs:
            A4 = 0.25 * self.h[L].prod(1) / self.h[L, d]
            uL, gL = self.side(c, L, d, 0 if wall >= 0 else 1)
            uR, gR = (uL, gL) if wall else self.side(c, R, d, 1)
            mirror = torch.tensor([-1.0, -1.0, -1.0, 1.0], dtype=c.dtype, device=c.device)[None, :, None]
            if wall > 0:
                uR = uL * mirror
            elif wall < 0:
                uL = uL * mirror
            jump = (uL - uR)[:, :3] * (0.5 if wall else 1.0)
            share = 1.0 if wall else 0.5
            sides = [(L, 0)] * (wall >= 0) + [(R, 1)] * (wall <= 0)
            rs = 0.0
            for e, sd in sides:  # local lifting: int r . tau = int [u] {tau} . n
                r = torch.einsum("evq,q,qm->evm", jump, self.w2, self.face[d][sd]) * (share * A4 / self.s[e])[:, None, None]
                lift[d] = lift[d].index_add(0, e, r)
                rs = rs + share * torch.einsum("evm,qm->evq", r, self.face[d][sd]) / self.s[e][:, None, None]
            g = [0.5 * (a + b) for a, b in zip(gL, gR)]
            g[d] = g[d] - ETA * rs
            tr = g[0][:, 0] + g[1][:, 1] + g[2][:, 2]
            fn = riemann(uL, uR, d)
            for i in range(3):
                fn[i] = fn[i] - self.nu * (g[d][:, i] + g[i][:, d] - (2.0 / 3.0 * tr if i == d else 0.0))
            f = torch.stack(fn, 1) * (self.w2 * A4[:, None])[:, None, :]
            for e, sd in sides:
                t = torch.einsum("evq,qm->evm", f, self.face[d][sd]) * ((1.0 - 2.0 * sd) / self.s[e])[:, None, None]
                out = out.index_add(0, e, t)
        is_ = (1.0 / self.s)[:, None, None]
        u = torch.einsum("evm,qm->evq", c, self.vol) * is_
        g = [(torch.einsum("evm,qm->evq", c[:, :3], self.dvol[b]) * self.J[:, b][:, None, None]
              - torch.einsum("evm,qm->evq", lift[b], self.vol)) * is_ for b in range(3)]
        tr = g[0][:, 0] + g[1][:, 1] + g[2][:, 2]
        for p in range(3):
            flux = []
            for i in range(3):
                f = self.nu * (g[p][:, i] + g[i][:, p]) - u[:, p] * u[:, i]
                flux.append(f - 2.0 / 3.0 * self.nu * tr - u[:, 3] if i == p else f)
            flux.append(-u[:, p])
            f = torch.stack(flux, 1) * self.w3 * (self.s * self.J[:, p])[:, None, None]
            out = out + torch.einsum("evq,qm->evm", f, self.dvol[p])
        return out


def riemann(uL, uR, d):
    """[4] interface fluxes (x, y, z momentum; continuity) of the artificial-compressibility problem along
    axis d, at the star state between the two acoustic waves."""
    plain = lambda t: torch.autograd.forward_ad.unpack_dual(t).primal  # noqa: E731
    c2 = AC_C * AC_C
    G = lambda u: 0.5 * (u * u + u * torch.sqrt(u * u + c2) + c2 * torch.asinh(u / AC_C))  # noqa: E731
    H = lambda u: 0.5 * (u * torch.sqrt(u * u + c2) + c2 * torch.asinh(u / AC_C) - u * u)  # noqa: E731

    def speed(u, v, sign):
        t = u + v
        return 0.5 * (t + sign * torch.sqrt(t * t + 4.0 * c2))

    def jump(u, ul, pl, ur, pr):
        p1 = torch.where(u < ul, pl + c2 * (u - ul) / speed(u, ul, -1.0), pl - (G(u) - G(ul)))
        p3 = torch.where(u > ur, pr + c2 * (u - ur) / speed(u, ur, 1.0), pr + H(u) - H(ur))
        return p1, p3

    def slope(u, ul, ur):
        """d(p1 - p3)/du: on a shock c^2 ((1/s) - (u - v) (ds/du) / s^2) with ds/du = |s| / Q."""
        a = torch.sqrt(u * u + c2)
        s1, q1 = speed(u, ul, -1.0), torch.sqrt((u + ul) ** 2 + 4.0 * c2)
        s3, q3 = speed(u, ur, 1.0), torch.sqrt((u + ur) ** 2 + 4.0 * c2)
        d1 = torch.where(u < ul, c2 * (1.0 / s1 + (u - ul) / (q1 * s1)), -(u + a))
        d3 = torch.where(u > ur, c2 * (1.0 / s3 - (u - ur) / (q3 * s3)), a - u)
        return d1 - d3

    ul, ur, pl, pr = uL[:, d], uR[:, d], uL[:, 3], uR[:, 3]
    fl, fr, fpl, fpr = (plain(t) for t in (ul, ur, pl, pr))
    u = 0.5 * (fl + fr)
    lo, hi = torch.full_like(u, -1e6), torch.full_like(u, 1e6)
    for _ in range(60):
        p1, p3 = jump(u, fl, fpl, fr, fpr)
        up = p1 > p3  # the jump falls with u
        lo, hi = torch.where(up, u, lo), torch.where(up, hi, u)
        new = u - (p1 - p3) / slope(u, fl, fr)
        u = torch.where((new > lo) & (new < hi), new, torch.where(p1 == p3, u, 0.5 * (lo + hi)))
    p1, p3 = jump(u, ul, pl, ur, pr)
    u = u - (p1 - p3) / slope(u, fl, fr)  # carries the implicit derivative
    ps, _ = jump(u, ul, pl, ur, pr)
    root = lambda t: torch.sqrt(t * t + c2)  # noqa: E731
    s1, s3 = speed(u, ul, -1.0), speed(u, ur, 1.0)
    tl = torch.where(u < ul, (s1 - ul) / (s1 - u), (ul + root(ul)) / (u + root(u)))
    tr = torch.where(u > ur, (s3 - ur) / (s3 - u), (u + root(u)) / (ur + root(ur)))
    band = 1e-12 * (fl.abs() + fr.abs() + AC_C)
    wl = torch.where(plain(u) > band, 1.0, torch.where(plain(u) < -band, 0.0, 0.5))
    f = [None] * 4
    for i in range(3):
        f[i] = u * u + ps if i == d else u * (wl * tl * uL[:, i] + (1.0 - wl) * tr * uR[:, i])
    f[3] = u
    return f
