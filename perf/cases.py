"""The work that a user of the solver has it do, as cases that can be timed and compared.

A case is one pass through the public binding (paper_1810_04289_gb300.fsi) on a context that
the program keeps: a residual, a Jacobian with a product, a product with a Jacobian already
there, a preconditioner apply, a preconditioner rebuilt and applied, a linear solve, a time
step. Meshes are this repository's own: the straight compliant tube, a batch of independent
tubes, the three-generation tree. Sizes run from the 429-node tube of the parity tests to
trees of 174,000 nodes (1.1 M unknowns), in FP64 and in mixed precision.
"""
import functools
import json

import numpy as np
import torch

import vesselmesh as vm
from paper_1810_04289_gb300 import fsi

MAT = dict(rho_f=1.05, mu_f=0.035, rho_s=1.2, E_s=3.0e6, nu_s=0.45, eta_s=0.0)
DT = 1e-3


def listed():
    small = dict(mesh="tube", nz=12, nt=8, nrf=3, nrw=1)         # the tube of the parity tests
    middle = dict(mesh="tube", nz=49, nt=26, nrf=9, nrw=2)       # between the two, odd counts
    bench = dict(mesh="tube", nz=96, nt=32, nrf=12, nrw=3)       # the 289k-unknown tube of the benchmark
    tree = dict(mesh="tree", h=0.10)                             # 174k nodes: larger than L2 in every array
    coarse = dict(mesh="tree", h=0.12)                           # 103k nodes
    batch = dict(mesh="batch", tubes=6, lo=5e3, hi=6e4)          # uneven independent vessels in one context
    return [
        # F(y) of the smallest mesh: what a residual monitor or an outer solver calls many times
        dict(name="residual-small", op="residual", precision=0, np=4, ilu=1, order=1, **small),
        # F(y) of a large mesh: the line search's call
        dict(name="residual-tree", op="residual", precision=0, np=1088, ilu=1, order=1, **tree),
        # a fresh Jacobian and one product with it, FP64: Newton's assembly where the FP64 form is asked for
        dict(name="assemble-fp64-tube", op="assemble", precision=0, np=64, ilu=1, order=1, **middle),
        # the same in the mixed form on a large mesh
        dict(name="assemble-mixed-tree", op="assemble", precision=1, np=640, ilu=1, order=1, **coarse),
        # J x alone, once per Krylov iteration of every solver a user writes around the operator
        dict(name="spmv-fp64-tree", op="spmv", precision=0, np=640, ilu=1, order=1, **coarse),
        dict(name="spmv-mixed-tree", op="spmv", precision=1, np=1088, ilu=1, order=1, tpr=16, **tree),
        # B^-1 r alone: FP64 with the benchmark tube's options, mixed with the tree's subdomain size
        dict(name="apply-fp64-tube", op="apply", precision=0, np=512, ilu=1, order=1, **bench),
        dict(name="apply-mixed-tree", op="apply", precision=1, np=1088, ilu=2, order=1, **tree),
        # Jacobian, ILU(2) factors and one apply of a batch: a Newton iteration's setup (Jacobian lag 1)
        dict(name="refresh-mixed-batch", op="refresh", precision=1, np=256, ilu=2, order=1, **batch),
        # one Newton correction with the default options (64 subdomains, ILU(1), RCM, FP64)
        dict(name="solve-fp64-tube", op="solve", precision=0, np=64, ilu=1, order=1, rtol=1e-3, **middle),
        # a whole step of the smallest tube to tight tolerances, as the parity tests take it
        dict(name="step-fp64-small", op="step", precision=0, np=4, ilu=1, order=1, ntol=1e-10, rtol=1e-6, lag=1, **small),
        # a whole step of the benchmark tube in mixed precision: the benchmark's subdomains and Jacobian lag,
        # the parity tests' tolerances for that form
        dict(name="step-mixed-tube", op="step", precision=1, np=512, ilu=1, order=1, ntol=1e-10, rtol=1e-4, lag=3, **bench),
    ]


def draw(rng):
    op = rng.choice(["residual", "assemble", "spmv", "spmv", "apply", "apply", "apply", "refresh", "solve", "step"])
    c = dict(op=op, precision=rng.randint(0, 1), ilu=rng.choice([1, 1, 2]), order=rng.choice([1, 1, 1, 2]))
    whole = op in ("solve", "step")
    kind = rng.choice(["tube", "tube", "batch"] if whole else ["tube", "batch", "tree"])
    if kind == "tree":
        h = round(0.10 * (0.20 / 0.10) ** rng.random(), 4)
        c.update(mesh="tree", h=h)
        nodes = 174e3 * (0.10 / h) ** 3
    elif kind == "batch":
        tubes, hi = rng.randint(2, 6), round(10 ** rng.uniform(4.0, 4.8))
        c.update(mesh="batch", tubes=tubes, lo=4e3, hi=hi)
        nodes = tubes * hi / 20
    else:
        nrf = round(3 * 4 ** rng.random())
        c.update(mesh="tube", nz=max(8, round(nrf * rng.uniform(4, 8))), nt=2 * round(1.33 * nrf + rng.random()),
                 nrf=nrf, nrw=max(1, round(nrf * 0.25)))
        nodes = (c["nz"] + 1) * (1 + c["nt"] * (nrf + c["nrw"]))
    # subdomains of 90 to 400 owned nodes, as the committed and the default options give
    c["np"] = max(2, round(nodes / (90 * (400 / 90) ** rng.random())))
    if op == "spmv":
        c["tpr"] = rng.choice([16, 32])
    if whole:
        # ILU(2) converges on every tube, thin-walled ones among them
        c.update(ilu=2, order=1, rtol=rng.choice([1e-3, 1e-4]))
    if op == "solve":
        c.update(precision=0)
    if op == "step":
        # the mixed form's linear solves are accurate to FP32: its steps take the parity tests' Newton tolerance
        c.update(ntol=1e-10 if c["precision"] else rng.choice([1e-6, 1e-8]), lag=rng.choice([1, 3]))
    return c


@functools.lru_cache(maxsize=4)
def _mesh(key):
    c = json.loads(key)
    if c["mesh"] == "tube":
        return vm.tube_mesh(c["nz"], c["nt"], c["nrf"], c["nrw"], seed=1810042890)
    if c["mesh"] == "batch":
        return vm.batch_tubes(n_tubes=c["tubes"], unk_lo=c["lo"], unk_hi=c["hi"])
    return vm.tree_config("tree-3gen", h=c["h"])


def mesh_of(case):
    keys = {"tube": ("nz", "nt", "nrf", "nrw"), "batch": ("tubes", "lo", "hi"), "tree": ("h",)}[case["mesh"]]
    return _mesh(json.dumps({k: case[k] for k in ("mesh",) + keys}, sort_keys=True))


def states(case, seed):
    """y, y_n, y_{n-1} and the time t_n: flow at a random instant of the inflow's period, disturbed in every
    field by a tenth of the parity tests' disturbances (whole steps and solves: the undisturbed flow, which is
    what a run starts from)."""
    m = mesh_of(case)
    rng = np.random.default_rng(seed)
    t = float(rng.uniform(0.0, 1.0))
    fluid = ((m.node_tag & vm.FLUID) != 0)[:, None]
    if case["mesh"] == "tree":
        base = np.zeros((m.n_nodes, 7))
        base[:, 2] = 10.0 * (1.0 + 0.5 * np.sin(2 * np.pi * 1.25 * t))
    else:
        base = vm.poiseuille_state(m, t=t)
    out = []
    for _ in range(3):
        y = base.copy()
        if case["op"] not in ("solve", "step"):
            y += rng.normal(size=y.shape) * np.array([0.3, 0.3, 0.3, 1.0, 1e-5, 1e-5, 1e-5])
        y[:, 0:4] *= fluid
        out.append(y)
    return out, t, rng


def prepare(case, seed):
    m = mesh_of(case)
    (y, y1, y2), t, rng = states(case, seed)
    opt = fsi.fsi_default_options(dt=DT, precision=case["precision"], n_subdomains=case["np"], ilu_level=case["ilu"],
                                  ordering=case["order"], threads_per_row=case.get("tpr", 32),
                                  gmres_rtol=case.get("rtol", 1e-3), newton_rtol=case.get("ntol", 1e-6),
                                  jac_lag=case.get("lag", 1))
    S = fsi.Solver(m, MAT, opt)
    s = dict(op=case["op"], S=S, t=t, y=S.vec(y), y1=S.vec(y1), y2=S.vec(y2), a=S.vec(), b=S.vec())
    fsi.fsi_set_state(S.ctx, s["y1"], s["y2"], s["y2"], t)
    if case["op"] in ("assemble", "spmv"):
        s["x"] = S.vec(rng.normal(size=y.shape))                       # a Krylov direction
    if case["op"] in ("apply", "refresh", "solve"):
        s["x"] = S.vec()                                               # the Newton system's right-hand side
        fsi.fsi_residual(S.ctx, s["y"], s["x"])
        s["x"].neg_()
    if case["op"] in ("spmv", "apply", "solve"):
        fsi.fsi_jacobian(S.ctx, s["y"])
    if case["op"] in ("apply", "solve"):
        fsi.fsi_pc_apply(S.ctx, s["x"], s["b"])                        # the factors are there
    return s


def run(s):
    c, op = s["S"].ctx, s["op"]
    if op == "residual":
        fsi.fsi_residual(c, s["y"], s["a"])
    elif op == "assemble":
        fsi.fsi_jacobian(c, s["y"])
        fsi.fsi_spmv(c, s["x"], s["a"])
    elif op == "spmv":
        fsi.fsi_spmv(c, s["x"], s["a"])
    elif op == "apply":
        fsi.fsi_pc_apply(c, s["x"], s["a"])
    elif op == "refresh":
        fsi.fsi_jacobian(c, s["y"])
        fsi.fsi_pc_apply(c, s["x"], s["a"])
    elif op == "solve":
        fsi.fsi_linear_solve(c, s["x"], s["a"], raise_on_divergence=False)
    else:
        fsi.fsi_set_state(c, s["y1"], s["y2"], s["y2"], s["t"])
        fsi.fsi_step(c)
        return {"y": s["a"], "t": fsi.fsi_get_state(c, s["a"])}
    return s["a"]


@functools.lru_cache(maxsize=None)
def _counts(key):
    """Sizes of the discrete problem, and how many iterations one solve or step of it takes."""
    case = json.loads(key)
    s = prepare(case, 1)
    i = s["S"].info()
    n = dict(N=i.n_nodes, T=i.n_tets, Tf=i.n_fluid_tets, nnzb=i.nnzb, fb=i.factor_blocks, fr=i.factor_rows)
    if case["op"] == "solve":
        n["li"] = fsi.fsi_linear_solve(s["S"].ctx, s["x"], s["a"], raise_on_divergence=False).iterations
    if case["op"] == "step":
        q = fsi.fsi_step(s["S"].ctx)
        n.update(li=q.linear_iterations, jac=q.jacobian_evaluations, res=q.residual_evaluations)
    s["S"].close()
    return n


def work(case):
    n = _counts(json.dumps(case, sort_keys=True))
    w = 4 if case["precision"] else 8
    N, T, nnzb, fb, fr = n["N"], n["T"], n["nnzb"], n["fb"], n["fr"]
    # per call: (bytes that have to move once, operations)
    res = (N * (24 + 3 * 56 + 56) + 16 * T, 1000 * n["Tf"] + 500 * (T - n["Tf"]))
    jac = (N * (24 + 3 * 56) + 16 * T + nnzb * 49 * w, 6000 * n["Tf"] + 2500 * (T - n["Tf"]))
    mul = (nnzb * (49 * w + 4) + 8 * N + 2 * 56 * N, 98 * nnzb)
    app = (fb * (49 * w + 4) + 56 * (fr + N), 98 * fb)
    fac = (nnzb * 49 * w + fb * 49 * w, 686 * 3 * fb)
    orth = (15 * 4 * 56 * N, 15 * 8 * 7 * N)          # a mean of 15 basis vectors, two passes
    parts = {"residual": [(1, res)], "assemble": [(1, jac), (1, mul)], "spmv": [(1, mul)], "apply": [(1, app)],
             "refresh": [(1, jac), (1, fac), (1, app)],
             "solve": [(n.get("li", 0), mul), (n.get("li", 0), app), (n.get("li", 0), orth)],
             "step": [(n.get("res", 0), res), (n.get("jac", 0), jac), (n.get("jac", 0), fac), (n.get("li", 0), mul),
                      (n.get("li", 0), app), (n.get("li", 0), orth)]}[case["op"]]
    return {"bytes": sum(k * p[0] for k, p in parts), "flops": sum(k * p[1] for k, p in parts)}


# ---------------------------------------------------------------------------
# the same residual in plain numpy, real or complex (its derivative along x is Im F(y + i e x) / e)
# ---------------------------------------------------------------------------
QA, QB = 0.5854101966249685, 0.1381966011250105


def _gradients(x):
    e = x[:, 1:] - x[:, :1]
    c = np.stack([np.cross(e[:, 1], e[:, 2]), np.cross(e[:, 2], e[:, 0]), np.cross(e[:, 0], e[:, 1])], axis=1)
    det = np.einsum("ti,ti->t", e[:, 0], c[:, 0])
    g = c / det[:, None, None]
    return np.concatenate([-g.sum(axis=1, keepdims=True), g], axis=1), det / 6.0


def _fluid(X, y, y1):
    u, p, d, u1, d1 = y[:, :, 0:3], y[:, :, 3], y[:, :, 4:7], y1[:, :, 0:3], y1[:, :, 4:7]
    rho, mu = MAT["rho_f"], MAT["mu_f"]
    g, vol = _gradients(X + d)
    g0, vol0 = _gradients(X)
    G = np.einsum("tai,taj->tij", u, g)
    gp = np.einsum("ta,tai->ti", p, g)
    div = G[:, 0, 0] + G[:, 1, 1] + G[:, 2, 2]
    adv = u - (d - d1) / DT
    ac = adv.mean(axis=1)
    h = np.cbrt(6.0 * np.sqrt(2.0) * vol0)
    D = np.sqrt((2 * rho / DT) ** 2 + (2 * rho / h) ** 2 * (ac * ac).sum(axis=1) + (4 * mu / h ** 2) ** 2)
    Rm, Rc = np.zeros_like(u), np.zeros_like(p)
    for q in range(4):
        Nq = np.full(4, QB)
        Nq[q] = QA
        aq = np.einsum("a,tai->ti", Nq, adv)
        inert = rho * np.einsum("a,tai->ti", Nq, u - u1) / DT + rho * np.einsum("tij,tj->ti", G, aq)
        rM = inert + gp
        along = np.einsum("ti,tai->ta", aq, g)
        Rm = Rm + 0.25 * vol[:, None, None] * (Nq[None, :, None] * inert[:, None, :]
                                              + (rho / D)[:, None, None] * along[:, :, None] * rM[:, None, :])
        Rc = Rc + 0.25 * vol[:, None] * (Nq[None, :] * div[:, None] + np.einsum("tai,ti->ta", g, rM) / D[:, None])
    stress = mu * (G + G.transpose(0, 2, 1)) + (h * h / 12.0 * D * div - p.mean(axis=1))[:, None, None] * np.eye(3)
    Rm = Rm + vol[:, None, None] * np.einsum("tij,taj->tai", stress, g)
    Rh = np.einsum("tab,tbi->tai", vol0[:, None, None] * np.einsum("tai,tbi->tab", g0, g0), d)
    return Rm, Rc, Rh


def _wall(X, d, d1, d2):
    nu, E = MAT["nu_s"], MAT["E_s"]
    mu, lam = E / (2 * (1 + nu)), E * nu / ((1 + nu) * (1 - 2 * nu))
    g0, vol0 = _gradients(X)
    F = np.einsum("tai,taj->tij", d, g0) + np.eye(3)
    Eg = 0.5 * (np.einsum("tki,tkj->tij", F, F) - np.eye(3))
    S = 2 * mu * Eg + lam * (Eg[:, 0, 0] + Eg[:, 1, 1] + Eg[:, 2, 2])[:, None, None] * np.eye(3)
    P = np.einsum("tik,tkj->tij", F, S)
    acc = MAT["rho_s"] * (d - 2 * d1 + d2) / DT ** 2 + MAT["eta_s"] * (d - d1) / DT
    return vol0[:, None, None] * ((acc.sum(axis=1, keepdims=True) + acc) / 20.0 + np.einsum("tij,taj->tai", P, g0))


def _residual(m, y, y1, y2, t):
    tag = np.asarray(m.node_tag)
    fl, wl, itf = (tag & vm.FLUID) != 0, (tag & vm.WALL) != 0, (tag & vm.INTERFACE) != 0
    inlet = fl & ((tag & vm.INLET) != 0)
    kin = itf & ~inlet
    wall_only = wl & ~fl
    fixed = (tag & (vm.INLET | vm.OUTLET | vm.WALL_END)) != 0
    F = np.zeros_like(y)
    for dom in (0, 1):
        sel = np.nonzero(np.asarray(m.tet_domain) == dom)[0]
        for at in range(0, len(sel), 100_000):
            tv = np.asarray(m.tets)[sel[at:at + 100_000]].astype(np.int64)
            rows = tv.ravel()

            def add(comp, v):
                v = v.reshape(len(rows), -1)
                for k in range(v.shape[1]):
                    s = np.bincount(rows, v[:, k].real, minlength=len(F))
                    F[:, comp + k] += s + 1j * np.bincount(rows, v[:, k].imag, minlength=len(F)) if np.iscomplexobj(F) else s

            if dom == 0:
                Rm, Rc, Rh = _fluid(m.X[tv], y[tv], y1[tv])
                free, on = ~(inlet | kin | wall_only)[tv][:, :, None], itf[tv][:, :, None]
                add(0, Rm * free)
                add(3, Rc)
                add(4, np.where(on, Rm, Rh))
            else:
                add(4, _wall(m.X[tv], y[tv][:, :, 4:7], y1[tv][:, :, 4:7], y2[tv][:, :, 4:7]))
    F[kin, 0:3] = (y[:, 0:3] - (y[:, 4:7] - y1[:, 4:7]) / DT)[kin]
    F[wall_only, 0:4] = y[wall_only, 0:4]
    F[fixed, 4:7] = y[fixed, 4:7]
    for k, b in enumerate(m.inlets):
        on = inlet & (np.asarray(m.node_problem) == k)
        n = np.asarray(b["normal"]) / np.linalg.norm(b["normal"])
        rel = m.X[on] - np.asarray(b["center"])
        r2 = (rel * rel).sum(axis=1) - (rel @ n) ** 2
        U = b["peak"] * (1 + b["amp"] * np.sin(2 * np.pi * b["freq"] * t + b["phase"]))
        F[on, 0:3] = y[on, 0:3] - (U * np.maximum(0.0, 1 - r2 / b["radius"] ** 2))[:, None] * n
    return F


def exact(case, seed):
    """Residuals and products with the Jacobian; an ILU, a Krylov process or a Newton process in plain numpy
    takes minutes at most of these sizes."""
    if case["op"] not in ("residual", "assemble", "spmv"):
        return None
    m = mesh_of(case)
    (y, y1, y2), t, rng = states(case, seed)
    if case["op"] == "residual":
        return _residual(m, y, y1, y2, t + DT)
    x = rng.normal(size=y.shape)
    return _residual(m, y + 1e-30j * x, y1, y2, t + DT).imag / 1e-30
