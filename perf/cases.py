"""The work that is timed: what a user of this library has it do, through its
public entry points (the Python package over the C ABI), one case per kind of
call and range of sizes.

A case names a call ("step", "operator", "adjoint", "gradient", "setup",
"batch"), a workload of `mhfp_inputs` with its size, and the options that the
program sets.  `prepare` builds what the program holds before the call,
`run` is one call, `exact` is the same result from plain torch in 64 bits
where that is a matter of seconds.

Solves in the FP64 form stop at 1e-8, the benchmark's tolerance; solves whose
preconditioner runs in FP32 stop at 1e-12, the gradient driver's tolerance
(1e-11 on the cantilever), where the solution no longer depends on how the preconditioner rounded.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import mhfp_inputs as mi
from paper_2002_09603_gb300 import Solver, default_options
from paper_2002_09603_gb300.adjoint import MisfitGradient
from paper_2002_09603_gb300.batch import LoadBatch, prepare_batch

F64 = dict(precision=0, restart=50, cheb_degree=2, coarse_max=125, reorth=1, near_kernel=0, formulation=0, tol=1e-8)
FP32 = dict(precision=1, restart=20, cheb_degree=1, coarse_max=512, reorth=0, near_kernel=0, formulation=0, tol=1e-12)
# (the cantilever's float-float operator reaches about 2e-12 at these sizes)
RBM = {**FP32, "near_kernel": 1, "cheb_degree": 2, "restart": 30, "coarse_max": 125, "tol": 1e-11}
OPTIONS = ("precision", "restart", "cheb_degree", "coarse_max", "reorth", "near_kernel", "formulation")


def _box(nx, ny, nz):
    return dict(nx=nx, ny=ny, nz=nz)


def listed():
    return [
        # the smallest model anyone solves (the plain-FP64 consolidation cube),
        # library defaults: launches and latency
        dict(name="step_fp64_cube8", call="step", mesh="terzaghi", **_box(8, 8, 8), **F64),
        # a first heterogeneous model with ragged sides, library defaults
        dict(name="step_fp64_ragged", call="step", mesh="random", **_box(37, 22, 29), **F64),
        # a time step of the 64^3 log-normal benchmark model, its options
        dict(name="step_mixed_64", call="step", mesh="lognormal", **_box(64, 64, 64), **{**FP32, "restart": 12}),
        # a time step of the 128^3 jittered, layered benchmark model: the largest
        dict(name="step_mixed_128", call="step", mesh="layered", **_box(128, 128, 128), **FP32),
        # the cantilever with the rigid-body-mode multigrid, odd size
        dict(name="step_rbm_47", call="step", mesh="cantilever", **_box(47, 47, 47), **RBM),
        # the mixed (flux) formulation that the cantilever study compares against
        dict(name="step_flux_40", call="step", mesh="cantilever", **_box(40, 40, 40),
             **{**F64, "formulation": 1, "restart": 30, "reorth": 0}),
        # a monitor or outer loop that applies the operator (both directions,
        # both arithmetics) and the residual norm to vectors of its own
        dict(name="operator_ragged", call="operator", mesh="random", **_box(83, 64, 71), **FP32),
        # one step of a reverse sweep: misfit, adjoint solve, gradient
        dict(name="adjoint_48", call="adjoint", mesh="lognormal", **_box(48, 48, 48), **{**FP32, "cheb_degree": 2}),
        # one evaluation of the log-permeability gradient (parameter update,
        # forward and reverse sweep), the driver's defaults
        dict(name="gradient_20", call="gradient", mesh="lognormal", **_box(20, 20, 20), steps=2, **{**F64, "tol": 1e-12}),
        # a new model: handle, assembly and preconditioner set-up, library
        # defaults; once per mesh or material
        dict(name="setup_fp64_ragged", call="setup", mesh="random", **_box(45, 52, 39), **F64),
        # the same for a larger model in the benchmark's options
        dict(name="setup_mixed_96", call="setup", mesh="layered", **_box(96, 96, 96), **FP32),
        # many small uneven models times four loads in one launch
        dict(name="batch_6x4", call="batch", mesh="lognormal", count=6, nmin=12, nmax=36, lanes=4, **{**FP32, "restart": 12}),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["step", "step", "step", "step", "operator", "adjoint", "gradient", "setup", "setup", "batch"])
    opt = dict(F64 if rng.random() < 0.4 else FP32)
    if call == "batch":
        nmin = rng.randint(9, 16)
        return dict(call=call, mesh="lognormal", count=rng.randint(3, 7), nmin=nmin, nmax=nmin + rng.randint(6, 26),
                    lanes=rng.choice([1, 2, 4]), **{**FP32, "restart": rng.choice([12, 16, 20])})
    if call == "gradient":
        n = _log_int(rng, 8, 24)
        return dict(call=call, mesh="lognormal", **_box(n, n, n), steps=rng.randint(1, 3),
                    **{**F64, "precision": rng.choice([0, 1]), "tol": 1e-12})
    mesh = rng.choice(["random", "random", "terzaghi", "lognormal", "layered", "cantilever"])
    top = {"step": 56 if opt["precision"] == 0 else 104, "adjoint": 56, "operator": 110, "setup": 96}[call]
    if mesh in ("random", "terzaghi"):
        size = _box(*(_log_int(rng, 6, min(top, 80)) for _ in range(3)))
    else:
        n = _log_int(rng, 9, {"layered": top, "lognormal": min(top, 72), "cantilever": min(top, 56)}[mesh])
        size = _box(n, n, n)
    if call == "operator":
        return dict(call=call, mesh=mesh, **size, **FP32)
    if call == "adjoint":
        opt = dict(FP32)
    if call == "step" and mesh == "cantilever":
        if opt["precision"] == 0 and rng.random() < 0.6:
            opt.update(formulation=1, restart=30, reorth=0)
        else:
            opt.update({k: RBM[k] for k in ("near_kernel", "restart", "cheb_degree", "coarse_max")})
    else:
        opt.update(cheb_degree=rng.choice([1, 2, 3]), restart=rng.choice([12, 20, 30, 50]))
    if mesh == "cantilever" and opt["precision"] == 1:
        opt["tol"] = RBM["tol"]
    return dict(call=call, mesh=mesh, **size, **opt)


# ------------------------------------------------------------------ inputs
def _problem(case, seed):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["mesh"] == "terzaghi":
        return mi.terzaghi_cube(nx=nx, ny=ny, nz=nz)
    if case["mesh"] == "random":
        return mi.random_small(nx, ny, nz, seed=seed, jitter=0.15)
    if case["mesh"] == "lognormal":
        return mi.lognormal_cube(nx, seed=seed)
    if case["mesh"] == "layered":
        return mi.layered_jitter_cube(nx, seed=seed)
    return mi.cantilever_cube(nx)


def _options(case):
    o = default_options()
    for k in OPTIONS:
        setattr(o, k, case[k])
    return o


def _state(prob, seed):
    """A smooth state [u | p | pi] of the size a loaded column has (u of the
    order of load / E, pressures of the order of the load), as FP64 values
    that FP32 holds exactly."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 7919)
    X = torch.as_tensor(prob.coords, device="cuda")
    f = lambda: torch.rand(4, dtype=torch.float64, device="cuda", generator=g)  # noqa: E731

    def modes(P, k=4):
        v = torch.zeros(P.shape[0], dtype=torch.float64, device="cuda")
        for _ in range(k):
            c = f()
            v += (c[3] - 0.5) * torch.cos(math.pi * (3 * c[0] * P[:, 0] + 3 * c[1] * P[:, 1] + 3 * c[2] * P[:, 2]) + 6 * c[3])
        return v

    scale = 1.0 / float(np.median(prob.E))
    u = torch.stack([scale * modes(X) * X[:, 2] for _ in range(3)], 1).reshape(-1)
    idx = torch.arange(prob.n_cells, device="cuda")
    C = torch.stack([(idx % prob.nx + 0.5) / prob.nx, (idx // prob.nx % prob.ny + 0.5) / prob.ny,
                     (idx // (prob.nx * prob.ny) + 0.5) / prob.nz], 1).double()
    p = 0.5 + 0.25 * modes(C)
    pi = 0.5 + 0.1 * torch.randn(prob.n_faces, dtype=torch.float64, device="cuda", generator=g)
    return torch.cat([u, p, pi]).float().double()


def _load(seed):
    return mi.LOAD_SCALES[seed % len(mi.LOAD_SCALES)]


def prepare(case, seed):
    torch.cuda.set_device(0)
    if case["call"] == "batch":
        sizes = np.random.default_rng(case["count"]).integers(case["nmin"], case["nmax"] + 1, size=case["count"])
        probs = [mi.lognormal_cube(int(n), seed=seed + 100 * i, sigma=1.5) for i, n in enumerate(sizes)]
        solvers = prepare_batch(probs, **{k: case[k] for k in OPTIONS})
        lb = LoadBatch(solvers, mi.LOAD_SCALES, tol=case["tol"], lanes=case["lanes"])
        return dict(case=case, batch=lb, solvers=solvers)
    prob = _problem(case, seed)
    st = dict(case=case, prob=prob, options=_options(case), x=_state(prob, seed), load=_load(seed))
    if case["call"] == "setup":
        return st
    if case["call"] == "gradient":
        rng = np.random.default_rng(seed)
        n = case["steps"]
        top = (prob.nx + 1) * (prob.ny + 1)
        uz = [-5e-5 * (1.0 + 0.1 * rng.standard_normal(top)) for _ in range(n)]
        pt = [0.5 + 0.1 * rng.standard_normal(prob.n_cells) for _ in range(n)]
        st["mg"] = MisfitGradient(prob, n, uz, pt, tol=case["tol"], precision=case["precision"], restart=case["restart"])
        st["logk"] = np.log(prob.kappa[:, 0]) + 0.1 * rng.standard_normal(prob.n_cells)
        return st
    s = Solver(prob)
    s.assemble_condense()
    s.setup_precond(st["options"])
    st["solver"] = s
    if case["call"] == "operator":
        st["b"] = s.build_rhs(_state(prob, seed + 1), load_scale=st["load"])
    if case["call"] == "adjoint":
        other = _state(prob, seed + 1)
        nu, np_, _ = s.sizes
        st["uz"] = other[2:nu:3][-s.uz_target_size():].contiguous()
        st["p"] = other[nu:nu + np_].contiguous()
        st["lam"] = _state(prob, seed + 2)
    return st


def run(st):
    call = st["case"]["call"]
    if call == "batch":
        return st["batch"].run()[0]
    if call == "setup":
        s = Solver(st["prob"])
        s.assemble_condense()
        s.setup_precond(st["options"])
        bt, ds = s.scalings()
        z = s.apply_precond(st["x"])  # the preconditioner that was set up, on a vector
        if st["case"]["precision"] == 1:
            z = z.float()  # FP32 V-cycles: the values are FP32 ones, widened
        s.close()
        return [bt, ds, z]
    if call == "gradient":
        J, grad = st["mg"].value_and_grad(st["logk"])
        return [J, grad]
    s = st["solver"]
    if call == "step":
        b = s.build_rhs(st["x"], load_scale=st["load"])
        return s.solve(b, tol=st["case"]["tol"])[0]
    if call == "operator":
        return [s.apply_operator(st["x"]), s.apply_operator_ff(st["x"]), s.apply_operator_t(st["x"]),
                s.residual_norm_noalloc(st["b"], st["x"])]
    # adjoint
    J = torch.zeros(1, dtype=torch.float64, device="cuda")
    g = s.empty()
    s.misfit(st["x"], st["uz"], st["p"], 1.0, 1.0, J, g)
    rhs = s.adjoint_rhs(g, st["lam"])
    lam = s.adjoint_solve(rhs, tol=st["case"]["tol"])[0]
    grad = s.grad_logk(lam, st["x"], torch.zeros(s.sizes[1], dtype=torch.float64, device="cuda"))
    return [J, lam, grad]


# ------------------------------------------------------------------ work
def _counts(nx, ny, nz):
    nN, nT = (nx + 1) * (ny + 1) * (nz + 1), nx * ny * nz
    nF = (nx + 1) * ny * nz + nx * (ny + 1) * nz + nx * ny * (nz + 1)
    return nN, nT, nF, 3 * nN + nT + nF


def _coefficients(nx, ny, nz):
    """Distinct coefficients of the condensed operator: the symmetric half of
    A_uu, A_up, the p block, W_T 1 and the symmetric half of W_T."""
    nN, nT, _, _ = _counts(nx, ny, nz)
    return 126 * nN + (24 + 4 + 6 + 21) * nT


def work(case):
    """Bytes of the inputs and outputs of the call and one pass over the
    operator's distinct coefficients (8 B each) per system that it solves or
    applies; two operations per coefficient of the full operator.  (A solve
    takes tens of such passes; how many is the method's affair.)"""
    if case["call"] == "batch":
        n = (case["nmin"] + case["nmax"]) // 2
        k = case["count"] * len(mi.LOAD_SCALES)
        return dict(bytes=8.0 * (case["count"] * _coefficients(n, n, n) + 2 * k * _counts(n, n, n)[3]),
                    flops=2.0 * k * (243 * _counts(n, n, n)[0] + 100 * n ** 3))
    size = (case["nx"], case["ny"], case["nz"])
    nN, nT, nF, n = _counts(*size)
    a, fl = _coefficients(*size), 243 * nN + (48 + 4 + 12 + 33) * nT
    if case["call"] == "setup":  # mesh and materials in; operator and scalings out
        return dict(bytes=8.0 * (3 * nN + 8 * nT + a + 2 * n), flops=2.0 * 8 * 24 * 25 / 2 * 3 * nT)
    k = {"step": 1, "operator": 4, "adjoint": 1, "gradient": 3 * case.get("steps", 1)}[case["call"]]
    return dict(bytes=8.0 * (a + 2 * k * n), flops=2.0 * k * fl)


# ------------------------------------------------------------------ exact
class _Plain:
    """The hybridized system of a problem from its definition: element
    integrals with 2x2x2 Gauss points, RT0 condensation, macro-element
    stabilization, Dirichlet rows and columns, applied element by element."""

    def __init__(self, prob):
        dev, d = "cuda", torch.float64
        t = lambda v, k=d: torch.as_tensor(np.ascontiguousarray(v), device=dev).to(k)  # noqa: E731
        nx, ny, nz = prob.nx, prob.ny, prob.nz
        self.nN, self.nT, self.nF, self.n = _counts(nx, ny, nz)
        self.dt = float(prob.dt)
        c = torch.arange(self.nT, device=dev)
        i, j, k = c % nx, c // nx % ny, c // (nx * ny)
        self.nodes = torch.stack([(i + (a & 1)) + (nx + 1) * ((j + (a >> 1 & 1)) + (ny + 1) * (k + (a >> 2))) for a in range(8)], 1)
        nfx, nfy = (nx + 1) * ny * nz, nx * (ny + 1) * nz
        self.faces = torch.stack([i + (nx + 1) * (j + ny * k), i + 1 + (nx + 1) * (j + ny * k),
                                  nfx + i + nx * (j + (ny + 1) * k), nfx + i + nx * (j + 1 + (ny + 1) * k),
                                  nfx + nfy + i + nx * (j + ny * k), nfx + nfy + i + nx * (j + ny * (k + 1))], 1)
        E, nu, b, S, mu, kap = (t(v) for v in (prob.E, prob.nu, prob.biot, prob.Seps, prob.mu, prob.kappa))
        lam, G = E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))
        X = t(prob.coords)[self.nodes]  # cell, node, axis
        K = torch.zeros(self.nT, 24, 24, dtype=d, device=dev)
        Aup = torch.zeros(self.nT, 8, 3, dtype=d, device=dev)
        Aww = torch.zeros(self.nT, 6, 6, dtype=d, device=dev)
        vol = torch.zeros(self.nT, dtype=d, device=dev)
        s = t([[1.0 if a >> q & 1 else -1.0 for q in range(3)] for a in range(8)])
        I3 = torch.eye(3, dtype=d, device=dev)
        for xi in s / math.sqrt(3.0):
            f = 1 + s * xi
            ref = 0.125 * torch.stack([s[:, 0] * f[:, 1] * f[:, 2], s[:, 1] * f[:, 0] * f[:, 2], s[:, 2] * f[:, 0] * f[:, 1]], 1)
            J = torch.einsum("tai,aj->tij", X, ref)
            det = torch.linalg.det(J)
            g = torch.einsum("aj,tji->tai", ref, torch.linalg.inv(J))
            gg = torch.einsum("tai,tbj->taibj", g, g)
            blk = lam[:, None, None, None, None] * gg + G[:, None, None, None, None] * (
                gg.permute(0, 1, 4, 3, 2) + torch.einsum("tak,tbk->tab", g, g)[:, :, None, :, None] * I3[None, None, :, None, :])
            K += (det[:, None, None, None, None] * blk).reshape(self.nT, 24, 24)
            Aup -= (b * det)[:, None, None] * g
            vol += det
            M = torch.einsum("tip,tir,ti->tpr", J, J, mu[:, None] / kap) / det[:, None, None]
            v = torch.stack([(1 + xi[q // 2]) / 8 if q & 1 else -(1 - xi[q // 2]) / 8 for q in range(6)])
            ax = torch.tensor([0, 0, 1, 1, 2, 2], device=dev)
            Aww += M[:, ax][:, :, ax] * v[None, :, None] * v[None, None, :]
            del gg, blk
        W = torch.linalg.inv(Aww)
        self.W = 0.5 * (W + W.transpose(1, 2))
        W1 = self.W.sum(2)
        self.K, self.vol, self.S = K, vol, S
        bits = t(prob.node_fix, torch.int64)
        self.free = torch.stack([(bits >> q & 1) == 0 for q in range(3)], 1).reshape(-1).to(d)
        self.udof = (3 * self.nodes[:, :, None] + torch.arange(3, device=dev)).reshape(self.nT, 24)
        self.Aup = Aup.reshape(self.nT, 24) * self.free[self.udof]
        self.open = ((t(prob.face_bc, torch.int64) >> 1 & 1) == 0).to(d)
        self.App = -W1 * self.open[self.faces]
        mx, my = (nx + 1) // 2, (ny + 1) // 2
        macro = i // 2 + mx * (j // 2 + my * (k // 2))
        nm = mx * my * ((nz + 1) // 2)
        total = lambda v: torch.zeros(nm, dtype=d, device=dev).index_add_(0, macro, v * vol)  # noqa: E731
        sv = total(torch.ones_like(vol))
        beta = (3 * total(b) / sv) ** 2 / (32 * (total(lam) / sv + 4 * total(G) / sv)) * sv
        self.partner = torch.stack([torch.where((i ^ 1) < nx, (i ^ 1) + nx * (j + ny * k), c), torch.where((j ^ 1) < ny, i + nx * ((j ^ 1) + ny * k), c),
                                    torch.where((k ^ 1) < nz, i + nx * (j + ny * (k ^ 1)), c)], 1)
        self.stab = beta[macro]
        self.sW = W1.sum(1)
        diag = lambda m, idx, size: torch.zeros(size, dtype=d, device=dev).index_add_(  # noqa: E731
            0, idx.reshape(-1), torch.diagonal(m, dim1=1, dim2=2).reshape(-1))
        self.du, self.dpi = diag(K, self.udof, 3 * self.nN), diag(self.W, self.faces, self.nF)
        sd = self.stab * (self.partner != c[:, None]).sum(1)
        self.bt = S * vol + sd + (self.Aup ** 2 / self.du[self.udof]).sum(1) + self.dt * self.sW
        drop = torch.zeros(self.nF, dtype=d, device=dev).index_add_(0, self.faces.reshape(-1), (self.dt * W1 ** 2 / self.bt[:, None]).reshape(-1))
        self.ds = torch.cat([self.du, self.bt, self.dpi - drop * self.open]).rsqrt()

    def apply(self, x, transpose=False):
        """A x (or A^T x) for the columns of x (n, k)."""
        nU = 3 * self.nN
        xu, xp, xq = x[:nU], x[nU:nU + self.nT], x[nU + self.nT:]
        sgn, cpi, cpp = (-1.0, 1.0, self.dt) if transpose else (1.0, self.dt, 1.0)
        fr, op = self.free[:, None], self.open[:, None]
        yu = torch.zeros_like(xu)
        e = torch.bmm(self.K, (fr * xu)[self.udof])
        yu.index_add_(0, self.udof.reshape(-1), e.reshape(-1, x.shape[1]))
        yu = fr * yu + (1 - fr) * self.du[:, None] * xu
        yu.index_add_(0, self.udof.reshape(-1), (sgn * self.Aup[:, :, None] * xp[:, None, :]).reshape(-1, x.shape[1]))
        yp = -sgn * torch.einsum("te,tek->tk", self.Aup, xu[self.udof]) + (self.S * self.vol + self.dt * self.sW)[:, None] * xp
        for a in range(3):
            yp += self.stab[:, None] * (xp - xp[self.partner[:, a]])
        yp += cpi * torch.einsum("te,tek->tk", self.App, xq[self.faces])
        yq = torch.zeros_like(xq)
        e = torch.bmm(self.W, (op * xq)[self.faces])
        yq.index_add_(0, self.faces.reshape(-1), e.reshape(-1, x.shape[1]))
        yq = op * yq + (1 - op) * self.dpi[:, None] * xq
        yq.index_add_(0, self.faces.reshape(-1), (cpp * self.App[:, :, None] * xp[:, None, :]).reshape(-1, x.shape[1]))
        return torch.cat([yu, yp, yq])

    def rhs(self, prob, x, load):
        """One backward-Euler right-hand side: the traction on the flat top
        faces (nodes share a face's area evenly only on rectangles, so the
        bilinear shape functions are integrated with 2x2 Gauss points)."""
        nU = 3 * self.nN
        fu = torch.zeros(self.nN, dtype=torch.float64, device=x.device)
        hit = (torch.as_tensor(prob.face_bc, device=x.device).long() & 1)[self.faces] == 1
        X = torch.as_tensor(prob.coords, device=x.device)
        for lf in range(6):
            T = torch.nonzero(hit[:, lf])[:, 0]
            if not T.numel():
                continue
            ax = lf // 2
            u, v = (a for a in range(3) if a != ax)
            q = [(lf & 1) << ax | (m & 1) << u | (m >> 1) << v for m in range(4)]
            nd = self.nodes[T][:, q]
            P = X[nd]
            for gs in (-1, 1):
                for gt in (-1, 1):
                    s, r = gs / math.sqrt(3.0), gt / math.sqrt(3.0)
                    sg = [(1 if m & 1 else -1, 1 if m >> 1 else -1) for m in range(4)]
                    N = [0.25 * (1 + a * s) * (1 + b * r) for a, b in sg]
                    ts = sum(0.25 * a * (1 + b * r) * P[:, m] for m, (a, b) in enumerate(sg))
                    tr = sum(0.25 * b * (1 + a * s) * P[:, m] for m, (a, b) in enumerate(sg))
                    area = torch.linalg.norm(torch.linalg.cross(ts, tr), dim=1)
                    for m in range(4):
                        fu.index_add_(0, nd[:, m], N[m] * area)
        tr = torch.as_tensor(np.asarray(prob.traction, float), device=x.device)
        bu = load * (fu[:, None] * tr).reshape(-1) * self.free
        bp = -(self.Aup * x[:nU][self.udof]).sum(1) + self.S * self.vol * x[nU:nU + self.nT]
        return torch.cat([bu, bp, torch.zeros(self.nF, dtype=torch.float64, device=x.device)])


def exact(case, seed):
    if case["call"] in ("batch", "gradient", "adjoint") or case.get("formulation") == 1:
        return None
    n = _counts(case["nx"], case["ny"], case["nz"])[3]
    if case["call"] == "step" and n > 9000:
        return None
    prob = _problem(case, seed)
    x = _state(prob, seed)
    A = _Plain(prob)
    if case["call"] == "step":
        M = A.apply(torch.eye(n, dtype=torch.float64, device="cuda"))
        b = A.rhs(prob, x, _load(seed))
        return (A.ds * torch.linalg.solve(A.ds[:, None] * M * A.ds[None, :], A.ds * b))
    if case["call"] == "setup":
        return [A.bt, A.ds, None]
    y = A.apply(x[:, None])[:, 0]
    b = A.rhs(prob, _state(prob, seed + 1), _load(seed))
    return [y, y, A.apply(x[:, None], True)[:, 0], torch.stack([torch.linalg.norm(A.ds * (b - y)), torch.linalg.norm(A.ds * b)])]
