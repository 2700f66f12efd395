"""The work whose speed is measured: scenario solves of the Henry problem,
MLMC passes, gradients, and the block calls a program builds on, each through
the public entry points of ``paper_2302_07804_gb300``.

A case is a dict of plain values; its ``"kind"`` says which call it is:

  solve       Solver.level_batch_solve: n scenarios of one level, with their
              coarse partners or without (cell- or vertex-centred scheme,
              FP64 or mixed precision, each coefficient model and QoI set)
  pass        one MLMC round as the driver makes it: Philox xi, one uneven
              batch over levels 0..3, the merge into the running sums
  gradient    scenario_qoi and its backward: a solve and its discrete adjoint
  assemble    Solver.assemble: residual and Jacobian blocks of given states
  accumulate  the MLMC sums of a batch whose rows hold many QoIs (the c field)

``steps0`` steps of ``tau0`` seconds at level 0 give the simulated time, T =
steps0 tau0 (the configuration's own is 20 steps of 360 s).
"""
import math

import numpy as np
import torch

from paper_2302_07804_gb300 import henry

_PRECISION = {"fp64": henry.HENRY_FP64, "mixed": henry.HENRY_MIXED}
_MODEL = {"uniform": henry.HENRY_MODEL_UNIFORM3, "kl": henry.HENRY_MODEL_KL, "layers": henry.HENRY_MODEL_TWO_LAYER}
_SCHEME = {"cell": henry.HENRY_SCHEME_CELL, "vertex": henry.HENRY_SCHEME_VERTEX}
_QOI = {"standard": henry.HENRY_QOI_STANDARD, "paper": henry.HENRY_QOI_PAPER, "field": henry.HENRY_QOI_PAPER_FIELD}

#: Cell-steps of one call at most (about half a second of solves).
_MOST = 9.0e7


def _solve(level, n, precision="fp64", model="uniform", scheme="cell", qoi="standard", coarse=False, steps0=20,
           tau0=360.0):
    return {"kind": "solve", "level": level, "n": n, "precision": precision, "model": model, "scheme": scheme,
            "qoi": qoi, "coarse": coarse, "steps0": steps0, "tau0": tau0}


def listed():
    return [
        # The plain single-level workload: 64 Philox samples at 32 x 16 cells.  A
        # small call, where launches and host round trips count.
        dict(_solve(0, 64), name="level0-fp64-64"),
        # Most of an MLMC run's samples are level-0 ones: a large batch of them.
        dict(_solve(0, 8192), name="level0-fp64-8192"),
        # The pilot's level-0 batch in mixed precision.
        dict(_solve(0, 1000, precision="mixed"), name="level0-mixed-1000"),
        # A level's own batch of pairs (fine and coarse) at 128 x 64 cells.
        dict(_solve(2, 33, coarse=True), name="level2-fp64-33"),
        # Residuals and Jacobian blocks of 512 x 256 cells, for a program's own
        # solver or a check of one step.
        {"kind": "assemble", "level": 4, "n": 8, "name": "assemble-level4-8"},
        # Random fields at the widest grid, 1024 x 512 cells, two samples; the
        # first 32 of its 640 steps.
        dict(_solve(5, 2, precision="mixed", model="kl", steps0=1), name="level5-kl-mixed-2"),
        # The paper's variant: two layers, its QoIs, tau = 32 s at level 0.
        dict(_solve(1, 50, model="layers", qoi="paper", steps0=24, tau0=32.0), name="layers-level1-50"),
        # The paper's own discretisation.
        dict(_solve(1, 64, scheme="vertex"), name="vertex-level1-64"),
        # One round of an MLMC run over levels 0..3: the allocation for RMSE
        # 1e-3 divided by ten, FP64.
        {"kind": "pass", "m0": 8168, "m1": 88, "m2": 16, "m3": 3, "precision": "fp64", "name": "mlmc-pass-fp64"},
        # The pilot round of an MLMC run in mixed precision.
        {"kind": "pass", "m0": 1000, "m1": 200, "m2": 50, "m3": 20, "precision": "mixed", "name": "mlmc-pilot-mixed"},
        # dQoI / d(64 KL coefficients, q_in) at 256 x 128 cells: steps of 36 s
        # as in the 200-step workload, checkpoints every 5 of 16 steps.
        {"kind": "gradient", "level": 3, "n": 12, "model": "kl", "steps0": 2, "tau0": 288.0, "every": 5,
         "name": "gradient-kl-level3-12"},
        # Mean and variance fields: the sums of 20000 rows of 15 + 512 QoIs.
        {"kind": "accumulate", "n": 20000, "qoi": "field", "coarse": True, "name": "accumulate-field-20000"},
    ]


def _between(rng, lo, hi):
    """A whole number from lo to hi, spread over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["solve"] * 5 + ["pass"] * 2 + ["gradient"] * 2 + ["assemble", "accumulate"])
    if kind == "solve":
        scheme = rng.choice(["cell", "cell", "cell", "vertex"])
        model = "uniform" if scheme == "vertex" else rng.choice(["uniform", "uniform", "kl", "layers"])
        level = rng.randint(0, 3 if scheme == "vertex" else 5)
        steps0 = {0: 20, 1: 20, 2: rng.randint(5, 20), 3: rng.randint(3, 9), 4: rng.randint(1, 3), 5: 1}[level]
        # the vertex scheme costs about three times as much a cell
        most = int(_MOST / (3 if scheme == "vertex" else 1) / _cell_steps(level, steps0))
        return _solve(level, _between(rng, 1, max(1, min(most, 8000))), precision=rng.choice(["fp64", "mixed"]),
                      model=model, scheme=scheme,
                      qoi="standard" if scheme == "vertex" else rng.choice(["standard", "standard", "paper", "field"]),
                      coarse=level > 0 and rng.random() < 0.5, steps0=steps0, tau0=360.0)
    if kind == "pass":
        return {"kind": "pass", "m0": _between(rng, 100, 6000), "m1": _between(rng, 20, 200),
                "m2": _between(rng, 4, 30), "m3": rng.randint(1, 5), "precision": rng.choice(["fp64", "mixed"])}
    if kind == "gradient":
        level = rng.randint(0, 3)
        steps0 = {0: 20, 1: rng.randint(4, 12), 2: rng.randint(2, 6), 3: rng.randint(1, 2)}[level]
        most = int(1.0e7 / _cell_steps(level, steps0))
        return {"kind": "gradient", "level": level, "n": _between(rng, 1, max(1, most)),
                "model": rng.choice(["uniform", "kl", "layers"]), "steps0": steps0, "tau0": 288.0,
                "every": rng.randint(3, 20)}
    if kind == "assemble":
        level = rng.randint(0, 5)
        return {"kind": "assemble", "level": level, "n": _between(rng, 1, int(4.0e6 / _cells(level)))}
    return {"kind": "accumulate", "n": _between(rng, 50, 20000), "qoi": rng.choice(["paper", "field"]),
            "coarse": rng.random() < 0.7}


def _cells(level):
    return (32 << level) * (16 << level)


def _cell_steps(level, steps0):
    return _cells(level) * (steps0 << level)


def _n_qoi(case):
    return {"standard": 2, "paper": 15, "field": 15 + 512}[case["qoi"]]


def _solver(case):
    """A program's solver: the configuration with the case's settings."""
    kw = {"precision": _PRECISION[case.get("precision", "fp64")], "coef_model": _MODEL[case.get("model", "uniform")],
          "scheme": _SCHEME[case.get("scheme", "cell")], "qoi_set": _QOI[case.get("qoi", "standard")]}
    if "steps0" in case:
        kw.update(steps0=case["steps0"], T=case["steps0"] * case["tau0"])
    return henry.Solver(**kw)


def _inputs(case, gen, n):
    """Random inputs as the models define them: uniform on (-1, 1), and for the
    KL model 64 standard normals and one uniform."""
    if case.get("model") == "kl":
        x = np.concatenate([gen.standard_normal((n, 64)), gen.uniform(-1.0, 1.0, (n, 1))], axis=1)
    else:
        x = gen.uniform(-1.0, 1.0, (n, 3))
    return torch.from_numpy(x).cuda()


def _wedge(gen, n, level):
    """Salt-wedge states: a smooth front of random place and slope, hydrostatic
    p with 20 Pa of smooth perturbation; (n, ny, nx, 2)."""
    ny, nx = 16 << level, 32 << level
    x = ((torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5) * (2.0 / nx))[None, None, :]
    y = ((torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) * (1.0 / ny))[None, :, None]
    u = torch.from_numpy(gen.uniform(-1.0, 1.0, (n, 4))).cuda()[:, :, None, None]
    c = 0.5 * (1.0 + torch.tanh((x - 1.3 - (0.5 + 0.1 * u[:, 0]) * y + 0.2 * u[:, 1]) / 0.15))
    p = 1000.0 * 9.81 * (1.0 - y) * (1.0 + 0.025 * c) + 20.0 * u[:, 2] * torch.cos(math.pi * x + u[:, 3] + 2.0 * y)
    return torch.stack([p, c], dim=-1).contiguous()


def prepare(case, seed):
    gen = np.random.Generator(np.random.PCG64([int(seed), 7]))
    kind = case["kind"]
    state = {"case": case}
    if kind == "solve":
        state.update(solver=_solver(case), xi=_inputs(case, gen, case["n"]))
    elif kind == "pass":
        counts = [case["m%d" % k] for k in range(4)]
        state.update(solver=_solver(case), seed=int(seed), counts=counts,
                     levels=np.repeat(np.arange(4, dtype=np.int32), counts))
    elif kind == "gradient":
        state.update(solver=_solver(case), xi=_inputs(case, gen, case["n"]),
                     weights=torch.from_numpy(gen.uniform(0.5, 1.5, (case["n"], 2)) * np.array([0.01, 1.0])).cuda())
    elif kind == "assemble":
        n, level = case["n"], case["level"]
        state.update(solver=henry.Solver(), xi=_inputs(case, gen, n), new=_wedge(gen, n, level),
                     old=_wedge(gen, n, level))
    else:
        n, nq = case["n"], _n_qoi(case)
        # rows as a solve returns them (the salt mass first, then mass fractions),
        # a coarse partner a little off, now and then a failed sample
        fine = torch.from_numpy(gen.uniform(0.0, 1.0, (n, nq))).cuda()
        fine[:, 0] = 100.0 + 50.0 * fine[:, 0]
        near = fine * (1.0 + 0.01 * torch.from_numpy(gen.standard_normal((n, 1))).cuda())
        status = torch.from_numpy((gen.random(n) < 0.002).astype(np.int32)).cuda()
        first = torch.zeros((2, nq, 3), dtype=torch.float64, device="cuda")
        state.update(fine=fine, near=near if case["coarse"] else None, status=status, first=first)
    return state


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "solve":
        qf, qc, status, _ = state["solver"].level_batch_solve(case["level"], state["xi"], with_coarse=case["coarse"],
                                                              allow_failures=True)
        return {"fine": qf, "coarse": qc, "status": status}
    if kind == "pass":
        solver, counts = state["solver"], state["counts"]
        xi = torch.cat([henry.sample_xi(state["seed"], k, 0, m) for k, m in enumerate(counts)])
        qf, qc, status, _ = solver.batch_solve_mixed(state["levels"], xi, with_coarse=True, allow_failures=True)
        sums, a = [], 0
        for k, m in enumerate(counts):
            s = torch.zeros((2, 2, 3), dtype=torch.float64, device="cuda")
            sums.append(henry.mlmc_accumulate(k, qf[a:a + m], qc[a:a + m] if k > 0 else None, status[a:a + m], s))
            a += m
        return {"xi": xi, "fine": qf, "coarse": qc, "status": status, "sums": sums}
    if kind == "gradient":
        xi = state["xi"].detach().requires_grad_()
        q = henry.scenario_qoi(state["solver"], case["level"], xi, checkpoint_every=case["every"])
        q.backward(state["weights"])
        return {"qoi": q.detach(), "gradient": xi.grad}
    if kind == "assemble":
        F, J = state["solver"].assemble(case["level"], state["xi"], state["new"], state["old"])
        return {"residual": F, "jacobian": J}
    sums = state["first"].clone()
    return henry.mlmc_accumulate(1 if case["coarse"] else 0, state["fine"], state["near"], state["status"], sums)


def work(case):
    """A cell of a step is read and written once (two FP64 unknowns) and needs,
    at the least, one residual and Jacobian (about 200 flops), one V-cycle (about
    230) and the residual test of the result (about 100); twice the couplings on
    the vertex-centred scheme; the adjoint step one assembly, one V-cycle and
    its sensitivities beside the forward step."""
    kind = case["kind"]
    if kind == "assemble":  # states in, residual and five 2 x 2 blocks out
        c = float(case["n"]) * _cells(case["level"])
        return {"bytes": c * (32 + 16 + 160), "flops": c * 200}
    if kind == "accumulate":
        rows = float(case["n"]) * _n_qoi(case) * (2 if case["coarse"] else 1)
        return {"bytes": rows * 8 + 4.0 * case["n"], "flops": rows * 6}
    if kind == "pass":
        cs = sum(float(case["m%d" % k]) * (_cell_steps(k, 20) + (_cell_steps(k - 1, 20) if k else 0))
                 for k in range(4))
        return {"bytes": 32 * cs, "flops": 530 * cs}
    cs = float(case["n"]) * _cell_steps(case["level"], case["steps0"])
    if kind == "gradient":  # the solve, the adjoint's forward and its backward sweep
        return {"bytes": (32 + 32 + 64) * cs, "flops": (2 * 530 + 550) * cs}
    if case["coarse"]:
        cs += float(case["n"]) * _cell_steps(case["level"] - 1, case["steps0"])
    return {"bytes": 32 * cs, "flops": (1000 if case["scheme"] == "vertex" else 530) * cs}


# ---------------------------------------------------------------------------
# The same results in plain 64-bit torch, without the framework.

_PHYS = dict(Lx=2.0, Ly=1.0, rho0=1000.0, drho=25.0, mu=1e-3, g=9.81, Dm=1.886e-5)


def _system(p, c, co, phi, kmu, PD, qin, h, tau):
    """Residual (n, ny, nx, 2) and 2 x 2 blocks (self, W, E, S, N; rows fluid and
    salt mass, columns p and c) of the cell-centred scheme, in units of rho0 h^2
    / tau; p, c, co are (n, ny, nx), the coefficients (n, 1, 1)."""
    rho0, drho, g = _PHYS["rho0"], _PHYS["drho"], _PHYS["g"]
    n, ny, nx = p.shape
    rho, v = rho0 + drho * c, h * h / tau
    F = torch.zeros((n, ny, nx, 2), dtype=torch.float64, device=p.device)
    J = torch.zeros((n, ny, nx, 5, 2, 2), dtype=torch.float64, device=p.device)
    ro = rho0 + drho * co
    F[..., 0] = phi * (rho - ro) * v
    F[..., 1] = phi * (rho * c - ro * co) * v
    J[..., 0, 0, 1] = phi * drho * v
    J[..., 0, 1, 1] = phi * (drho * c + rho) * v

    def faces(L, R, kL, kR, grav):  # slices of the two sides, the block of R in L and of L in R
        rf = 0.5 * (rho[L] + rho[R])
        q = -kmu * ((p[R] - p[L]) / h + grav * rf)
        Fl = rf * q * h
        up = Fl >= 0
        cup = torch.where(up, c[L], c[R])
        dif = PD * (c[R] - c[L])
        G = Fl * cup - rf * dif
        dp = rf * kmu
        dc = 0.5 * drho * h * (q - rf * kmu * grav)
        zero = torch.zeros_like(Fl)
        gL = dc * cup + torch.where(up, Fl, zero) - (0.5 * drho * dif - rf * PD)
        gR = dc * cup + torch.where(up, zero, Fl) - (0.5 * drho * dif + rf * PD)
        F[L + (0,)] += Fl
        F[R + (0,)] -= Fl
        F[L + (1,)] += G
        F[R + (1,)] -= G
        one = ((dp, dc), (dp * cup, gL))     # d(F, G) / d(p, c) of L
        two = ((-dp, dc), (-dp * cup, gR))   # ... of R
        for r in range(2):
            for k in range(2):
                J[L + (0, r, k)] += one[r][k]
                J[L + (kL, r, k)] += two[r][k]
                J[R + (0, r, k)] -= two[r][k]
                J[R + (kR, r, k)] -= one[r][k]

    a = slice(None)
    faces((a, a, slice(0, nx - 1)), (a, a, slice(1, nx)), 2, 1, 0.0)
    faces((a, slice(0, ny - 1), a), (a, slice(1, ny), a), 4, 3, g)
    # land: fresh inflow, c = 0; sea: hydrostatic brine, c = 1
    W, E = (a, a, slice(0, 1)), (a, a, slice(nx - 1, nx))
    Fl = -rho0 * qin * h * torch.ones_like(p[W])
    rb = 0.5 * (rho[W] + rho0)
    up = Fl >= 0
    F[W + (0,)] += Fl
    F[W + (1,)] += torch.where(up, Fl * c[W], torch.zeros_like(Fl)) + 2.0 * rb * PD * c[W]
    J[W + (0, 1, 1)] += torch.where(up, Fl, torch.zeros_like(Fl)) + PD * (drho * c[W] + 2.0 * rb)
    y = ((torch.arange(ny, dtype=torch.float64, device=p.device) + 0.5) * h)[None, :, None]
    pb = (rho0 + drho) * g * (_PHYS["Ly"] - y)
    rb = 0.5 * (rho[E] + rho0 + drho)
    q = -kmu * (pb - p[E]) * (2.0 / h)
    Fr = rb * q * h
    up = Fr >= 0
    cup = torch.where(up, c[E], torch.ones_like(Fr))
    dif = PD * (1.0 - c[E])
    dp, dc = 2.0 * rb * kmu, 0.5 * drho * q * h
    F[E + (0,)] += Fr
    F[E + (1,)] += Fr * cup - 2.0 * rb * dif
    J[E + (0, 0, 0)] += dp
    J[E + (0, 0, 1)] += dc
    J[E + (0, 1, 0)] += dp * cup
    J[E + (0, 1, 1)] += dc * cup + torch.where(up, Fr, torch.zeros_like(Fr)) - (drho * dif - 2.0 * rb * PD)
    s = 1.0 / (rho0 * v)
    return F * s, J * s


def _coefficients(xi):
    phi = 0.35 * (1.0 + 0.2 * xi[:, 0])
    kmu = 1.02e-9 * torch.exp(0.5 * xi[:, 1]) / _PHYS["mu"]
    qin = 6.6e-5 * (1.0 + 0.2 * xi[:, 2])
    return [v[:, None, None] for v in (phi, kmu, phi * _PHYS["Dm"], qin)]


def _newton_step(F, J):
    """J d = -F by block elimination over the columns of the grid."""
    n, ny, nx, _ = F.shape
    m = 2 * ny
    D = torch.zeros((nx, n, ny, 2, ny, 2), dtype=torch.float64, device=F.device)
    i = torch.arange(ny, device=F.device)
    Jx = J.permute(2, 1, 0, 3, 4, 5)  # (nx, ny, n, 5, 2, 2)
    D[:, :, i, :, i, :] = Jx[:, :, :, 0].permute(1, 0, 2, 3, 4)
    D[:, :, i[1:], :, i[:-1], :] = Jx[:, 1:, :, 3].permute(1, 0, 2, 3, 4)
    D[:, :, i[:-1], :, i[1:], :] = Jx[:, :-1, :, 4].permute(1, 0, 2, 3, 4)
    D = D.reshape(nx, n, m, m)
    W = torch.zeros((nx, n, ny, 2, ny, 2), dtype=torch.float64, device=F.device)
    E = torch.zeros_like(W)
    W[:, :, i, :, i, :] = Jx[:, :, :, 1].permute(1, 0, 2, 3, 4)
    E[:, :, i, :, i, :] = Jx[:, :, :, 2].permute(1, 0, 2, 3, 4)
    W, E = W.reshape(nx, n, m, m), E.reshape(nx, n, m, m)
    b = -F.permute(2, 0, 1, 3).reshape(nx, n, m, 1)
    up, rhs = [], []
    for k in range(nx):
        A, r = D[k], b[k]
        if k:
            A = A - W[k] @ up[-1]
            r = r - W[k] @ rhs[-1]
        z = torch.linalg.solve(A, torch.cat([E[k], r], dim=2))
        up.append(z[:, :, :m])
        rhs.append(z[:, :, m:])
    d = [rhs[-1]]
    for k in range(nx - 2, -1, -1):
        d.append(rhs[k] - up[k] @ d[-1])
    return torch.stack(d[::-1]).reshape(nx, n, ny, 2).permute(1, 2, 0, 3)


def _exact_level0(xi, steps, tau):
    ny, nx, h = 16, 32, 1.0 / 16
    phi, kmu, PD, qin = _coefficients(xi)
    n = xi.shape[0]
    y = ((torch.arange(ny, dtype=torch.float64, device=xi.device) + 0.5) * h)[None, :, None]
    p = (_PHYS["rho0"] * _PHYS["g"] * (_PHYS["Ly"] - y)).expand(n, ny, nx).contiguous()
    c = torch.zeros_like(p)
    for _ in range(steps):
        co = c
        for _ in range(12):
            F, J = _system(p, c, co, phi, kmu, PD, qin, h, tau)
            if float(F.abs().max()) <= 1e-14:
                break
            d = _newton_step(F, J)
            p, c = p + d[..., 0], c + d[..., 1]
            if float(d[..., 1].abs().max()) <= 1e-14:
                break
    rho = _PHYS["rho0"] + _PHYS["drho"] * c
    mass = phi[:, 0, 0] * (rho * c).sum(dim=(1, 2)) * h * h
    point = 0.25 * (c[:, 3, 23] + c[:, 3, 24] + c[:, 4, 23] + c[:, 4, 24])  # the cells at (1.5, 0.25)
    return torch.stack([mass, point], dim=1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        if case["level"] or case["n"] > 300 or case["model"] != "uniform" or case["scheme"] != "cell" \
                or case["qoi"] != "standard":
            return None
        q = _exact_level0(prepare(case, seed)["xi"], case["steps0"], case["tau0"])
        return {"fine": q, "coarse": None, "status": None}
    if kind == "assemble":
        s = prepare(case, seed)
        new, old = s["new"], s["old"]
        h = 1.0 / new.shape[1]
        tau = 360.0 / (1 << case["level"])
        F, J = _system(new[..., 0], new[..., 1], old[..., 1], *_coefficients(s["xi"]), h, tau)
        return {"residual": F, "jacobian": J}
    if kind == "accumulate":
        s = prepare(case, seed)
        use = s["status"] == 0
        fine = s["fine"][use]
        out = []
        for v in (fine - s["near"][use] if case["coarse"] else fine, fine):
            mean = v.mean(dim=0)
            out.append(torch.stack([torch.full_like(mean, float(v.shape[0])), mean, (v - mean).square().sum(dim=0)], dim=1))
        return torch.stack(out)
    return None
