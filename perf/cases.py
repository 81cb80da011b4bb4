"""Performance cases: the calls that a user of the solver makes, over the sizes that the
repository's recipes, tests and benchmark use.

A case is a dict of plain values; "kind" says which call it is:

  step      assemble + build + solve of one linearised Newton system (Solver.assemble,
            Solver.build, Solver.solve), the call of every reservoir time step; with the FP64,
            FP32 or FP32 + BF16 hierarchies and with the plain or the learned Schur correction
  newton    one backward-Euler step by Newton's method (Solver.newton_step)
  assemble  Jacobian, residual and Schur approximation alone (Solver.assemble)
  spmv      products with the assembled Jacobian (Solver.spmv), as a user's own Krylov method
            or a residual check makes them
  amg       a standalone AMG hierarchy of a caller's CSR matrix and one V-cycle (thermo.AMG)
  probe     exact Schur columns, the training targets of the learned correction
            (Solver.probe_schur_columns)
  train     a validation gradient and some Adam steps of the per-cell network (thermo.MLP)

Inputs are those of the repository's recipes (permeability fields, five-spot wells, water),
generated here from the seed alone.
"""
import math

import numpy as np
import torch

from paper_1902_00095_gb300 import thermo

DAY = 86400.0
WATER = dict(rho0=999.0, c=5.5e-10, beta=2.5e-4, p0=101325.0, T0=288.7056, mu0=1.0e-3,
             T_mu0=288.7056, mu_coef=0.02, cv=4184.0, rho_r=2650.0, cr=920.0, kTf=0.6,
             kT_mix=0, mu_law=0, api=0.0)
GRAVITY = 9.81
CELL = 10.0  # metres, every direction
NF, NH, NO = 24, 64, 8  # the network: inputs, hidden units (two layers), outputs


def _step(name, field, nx, ny, nz, precision=0, learned=False):
    return dict(name=name, kind="step", field=field, nx=nx, ny=ny, nz=nz, precision=precision,
                learned=learned)


def listed():
    return [
        # the smallest grid of the repository's recipes: interactive use, latency throughout
        _step("step_iid_16x16x8", "iid", 16, 16, 8),
        # an ordinary sector model, FP64 throughout
        _step("step_grf_64x64x32", "grf", 64, 64, 32),
        # a ragged sector model with the smallest hierarchy storage (FP32 values, BF16 P and R)
        _step("step_grf_97x61x33_bf16", "grf", 97, 61, 33, precision=2),
        # the channelised mixed-precision workload with the learned Schur correction
        _step("step_channel_128x128x64_learned", "channel", 128, 128, 64, precision=1,
              learned=True),
        # the full-field layered workload, FP64 hierarchies: the benchmark's system
        _step("step_layered_256x256x64", "layered", 256, 256, 64),
        # the same system with FP32 hierarchies, the fastest configuration
        _step("step_layered_256x256x64_fp32", "layered", 256, 256, 64, precision=1),
        # one time step of a sector model: a handful of linearisations on one hierarchy structure
        dict(name="newton_grf_64x64x32", kind="newton", field="grf", nx=64, ny=64, nz=32, days=10.0),
        # linearisation alone at a full-field iterate (explicit coupling, residual checks)
        dict(name="assemble_layered_256x256x64", kind="assemble", field="layered", nx=256, ny=256,
             nz=64),
        # Jacobian products in a user's own Krylov method
        dict(name="spmv_grf_96x96x48", kind="spmv", field="grf", nx=96, ny=96, nz=48),
        # a standalone hierarchy and V-cycle of a caller's pressure matrix on an odd grid
        dict(name="amg_grf_65x51x31", kind="amg", field="grf", nx=65, ny=51, nz=31),
        # training targets of the learned correction on the training recipe's grid
        dict(name="probe_grf_32x32x16", kind="probe", field="grf", nx=32, ny=32, nz=16, cols=8),
        # part of a training epoch: 4096-sample batches, a validation pass as one gradient
        dict(name="train_batch4096", kind="train", batch=4096, steps=8, validation=10000),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step"] * 6 + ["newton", "assemble", "spmv", "amg", "probe", "train"])
    if kind == "train":
        return dict(kind="train", batch=log_int(500, 8192), steps=rng.randint(2, 8),
                    validation=log_int(500, 20000))
    # cells on a logarithmic scale up to what the kind is used for, then a shape of about as many
    most = {"newton": 150_000, "amg": 150_000, "probe": 20_000}.get(kind, 4_100_000)
    cells = math.exp(rng.uniform(math.log(2048), math.log(most)))
    nz = max(5, min(64, log_int(5, 64), int(cells / 256)))
    nx = max(12, min(256, int(math.sqrt(cells / nz) * rng.uniform(0.8, 1.25))))
    ny = max(12, min(256, int(cells / (nz * nx))))
    field = rng.choice(["grf", "grf", "channel", "layered"])
    case = dict(kind=kind, field=field, nx=nx, ny=ny, nz=nz)
    if kind == "step":
        case["precision"] = rng.choice([0, 0, 1, 2])
        case["learned"] = rng.random() < 0.25
    elif kind == "newton":
        case["field"], case["days"] = "grf", rng.choice([2.0, 5.0, 10.0])
    elif kind == "probe":
        case["field"], case["cols"] = "grf", rng.randint(2, 6)
    return case


# ------------------------------------------------------------------ inputs
def _gaussian_field(rng, shape, corr):
    """Unit-variance Gaussian field of the given correlation lengths (cells), by FFT."""
    spec = np.fft.rfftn(rng.standard_normal(shape))
    for axis, (n, ell) in enumerate(zip(shape, corr)):
        d = np.minimum(np.arange(n), n - np.arange(n))
        k = np.exp(-((d / ell) ** 2))
        k = np.fft.fft(k / k.sum()).real
        if axis == 2:
            k = k[: n // 2 + 1]
        spec *= k.reshape([-1 if a == axis else 1 for a in range(3)])
    f = np.fft.irfftn(spec, s=shape, axes=(0, 1, 2))
    return (f - f.mean()) / f.std()


def _problem(case, seed):
    """Fields, wells and states of one system, on the host."""
    rng = np.random.default_rng([seed, case["nx"], case["ny"], case["nz"]])
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    shape, n = (nz, ny, nx), nx * ny * nz
    kTr, kz, days = np.full(n, 2.0), 1.0, 10.0
    if case["field"] == "iid":
        logk = rng.normal(-13.0, 0.5, shape)
        days = 1.0
    elif case["field"] == "grf":
        logk = -13.0 + _gaussian_field(rng, shape, (2.0, 8.0, 8.0))
        kz = 0.1
    elif case["field"] == "channel":
        f = _gaussian_field(rng, shape, (2.0, 4.0, 16.0))
        sand = f >= np.quantile(f, 0.7)
        logk = np.where(sand, -12.0, -15.0)
        kTr = np.where(sand.ravel(), 3.0, 1.5)
    else:  # eight layers
        layer = np.minimum(np.arange(nz) // max(1, nz // 8), 7)
        logk = (-14.0 + 2.0 * layer / 7)[:, None, None] + rng.normal(0.0, 0.8, shape)
        days = 30.0
    K = (10.0 ** logk).ravel()
    well = lambda i, j, kind, value, T: dict(i=i, j=j, k0=0, k1=nz - 1, kind=kind, value=value,
                                             T_inj=T, U=0.0)
    if case["field"] == "iid":
        wells = [well(0, 0, 0, 1.0e-3, 450.0), well(nx - 1, ny - 1, 1, 10.0e6, 0.0)]
    else:
        wells = [well(i, j, 0, 1.0e-3, 450.0) for i in (0, nx - 1) for j in (0, ny - 1)]
        wells.append(well(nx // 2, ny // 2, 1, 10.0e6, 0.0))
    p_n, T_n = np.full(n, 15.0e6), np.full(n, 320.0)
    p_k, T_k = p_n.copy(), T_n.copy()
    if case["kind"] in ("assemble", "spmv", "probe"):  # an iterate of a Newton iteration
        p_k += 2.0e5 * rng.standard_normal(n)
        T_k += 5.0 * rng.standard_normal(n)
    return dict(nx=nx, ny=ny, nz=nz, Kx=K, Ky=K, Kz=kz * K, phi=np.full(n, 0.2), kTr=kTr,
                wells=wells, p_n=p_n, T_n=T_n, p_k=p_k, T_k=T_k,
                dt=case.get("days", days) * DAY, rng=rng)


def _params(rng, out_scale):
    """Parameters of the network: fan-in-scaled hidden layers and a small output layer."""
    w = lambda o, i, s: (rng.uniform(-1, 1, (o, i)) * s / math.sqrt(i)).ravel()
    return np.concatenate([w(NH, NF, 1.0), np.zeros(NH), w(NH, NH, 1.0), np.zeros(NH),
                           w(NO, NH, out_scale), np.zeros(NO)])


def _pressure_matrix(pr):
    """CSR matrix of the pressure equation: TPFA diffusion plus accumulation."""
    nx, ny, nz = pr["nx"], pr["ny"], pr["nz"]
    n = nx * ny * nz
    idx = np.arange(n).reshape(nz, ny, nx)
    rows, cols, vals = [], [], []
    diag = np.full(n, 1.0e3 * 0.2 * 5.5e-10 * 1.0e3 / pr["dt"])
    for axis, K in ((2, pr["Kx"]), (1, pr["Ky"]), (0, pr["Kz"])):
        lo = np.take(idx, np.arange(idx.shape[axis] - 1), axis).ravel()
        hi = np.take(idx, np.arange(1, idx.shape[axis]), axis).ravel()
        t = CELL * 2.0 * K[lo] * K[hi] / (K[lo] + K[hi]) * 1.0e6
        rows += [lo, hi]
        cols += [hi, lo]
        vals += [-t, -t]
        np.add.at(diag, lo, t)
        np.add.at(diag, hi, t)
    rows, cols, vals = (np.concatenate(a) for a in (rows + [idx.ravel()], cols + [idx.ravel()],
                                                    vals + [diag]))
    order = np.lexsort((cols, rows))
    rowptr = np.zeros(n + 1, np.int32)
    rowptr[1:] = np.cumsum(np.bincount(rows, minlength=n))
    return rowptr, cols[order].astype(np.int32), vals[order]


def _batch(rng, n):
    """Samples of the network: features, slots, S~ entries and diagonals, exact entries."""
    X = rng.standard_normal((n, NF)).astype(np.float32)
    slot = rng.integers(0, 7, n).astype(np.int32)
    Sd = 10.0 ** rng.uniform(4.0, 6.0, n)
    St = np.where(slot == 0, Sd, -Sd * rng.uniform(0.01, 0.3, n))
    return X, slot, St, Sd, St * (1.0 + 0.05 * np.tanh(X[:, :4].sum(axis=1)))


def prepare(case, seed):
    if case["kind"] == "train":
        rng = np.random.default_rng([seed, case["batch"]])
        params = _params(rng, 0.1)
        return dict(case=case, mlp=thermo.MLP(params), params=params,
                    validation=_batch(rng, case["validation"]),
                    batches=[_batch(rng, case["batch"]) for _ in range(case["steps"])])
    pr = _problem(case, seed)
    rng = pr.pop("rng")
    n = pr["nx"] * pr["ny"] * pr["nz"]
    if case["kind"] == "amg":
        rowptr, col, val = _pressure_matrix(pr)
        return dict(case=case, rowptr=rowptr, col=col, val=val, b=rng.standard_normal(n))
    solver = thermo.Solver(pr["nx"], pr["ny"], pr["nz"], WATER, CELL, CELL, CELL, GRAVITY)
    solver.set_fields(pr["Kx"], pr["Ky"], pr["Kz"], pr["phi"], pr["kTr"])
    solver.set_wells(pr["wells"])
    dev = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda")
    state = dict(case=case, solver=solver, dt=pr["dt"],
                 states=[dev(pr[k]) for k in ("p_k", "T_k", "p_n", "T_n")],
                 out=[torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2)])
    if case["kind"] == "step" and case["learned"]:
        state["mlp"] = thermo.MLP(_params(rng, 0.01))
        solver.set_schur_model(state["mlp"])
    if case["kind"] in ("spmv", "probe"):
        solver.assemble(*state["states"], pr["dt"])
    if case["kind"] == "spmv":
        state["x"] = [dev(1.0e5 * rng.standard_normal(n)), dev(rng.standard_normal(n))]
    if case["kind"] == "probe":
        solver.build()
        state["cols"] = np.sort(rng.choice(n, case["cols"], replace=False))
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "train":
        mlp = state["mlp"]
        mlp.set_params(state["params"])
        loss, grad = mlp.gradient(*state["validation"])
        losses = [mlp.train_step(*b, lr=2e-3) for b in state["batches"]]
        return {"validation_loss": loss, "gradient": grad, "losses": losses, "params": mlp.params()}
    if kind == "amg":
        amg = thermo.AMG(state["rowptr"], state["col"], state["val"])
        x = amg.vcycle(state["b"])
        levels = amg.info()
        amg.close()
        return {"x": x, "rows": levels[0], "entries": levels[1]}
    solver = state["solver"]
    if kind == "step":
        solver.assemble(*state["states"], state["dt"])
        solver.build(precision=case["precision"], schur=1 if case["learned"] else 0)
        x_p, x_T, info = solver.solve(rtol=1e-8, out=state["out"])
        return {"x_p": x_p, "x_T": x_T, "iterations": info["iters"]}
    if kind == "newton":
        p, T, info = solver.newton_step(state["states"][2], state["states"][3], state["dt"],
                                        max_newton=8, out=state["out"])
        return {"p": p, "T": T, "newton": info["newton_iters"], "linear": info["linear_iters"]}
    if kind == "assemble":
        solver.assemble(*state["states"], state["dt"], R_m=state["out"][0], R_e=state["out"][1])
        return {"R_m": state["out"][0], "R_e": state["out"][1]}
    if kind == "spmv":
        y_p, y_T = solver.spmv(*state["x"])
        return {"y_p": y_p, "y_T": y_T}
    entry, value, iters, status = solver.probe_schur_columns(state["cols"], rtol=1e-10)
    return {"entry": entry, "value": value, "iterations": iters, "status": status}


def work(case):
    """Inputs read once, outputs written once, and the arithmetic on them: 7-point rows of 2x2
    blocks, a nominal 15 Krylov iterations per solve with their two (A_pp) and one (Schur)
    V-cycles of about 8 operator passes each over 3 times the finest operator."""
    if case["kind"] == "train":
        macs = NF * NH + NH * NH + NH * NO
        samples = case["validation"] + case["batch"] * case["steps"]
        return {"bytes": samples * (4 * NF + 4 + 24) + 8 * 2 * (macs + 2 * NH + NO),
                "flops": 6 * macs * samples}
    n = case["nx"] * case["ny"] * case["nz"]
    vcycle = 8 * 3 * 2 * 7 * n
    solve = 15 * (3 * vcycle + 2 * 28 * n)
    if case["kind"] == "step":
        return {"bytes": 8 * n * (5 + 4 + 2), "flops": 400 * n + solve}
    if case["kind"] == "newton":
        return {"bytes": 8 * n * (5 + 2 + 2), "flops": 4 * (400 * n + solve)}
    if case["kind"] == "assemble":
        return {"bytes": 8 * n * (5 + 4 + 2), "flops": 400 * n}
    if case["kind"] == "spmv":
        return {"bytes": 8 * n * (28 + 2 + 2), "flops": 2 * 28 * n}
    if case["kind"] == "amg":
        return {"bytes": 12 * 7 * n + 16 * n, "flops": vcycle + 2 * 100 * n}
    return {"bytes": 8 * n * 7 * 4 + 96 * case["cols"], "flops": case["cols"] * 10 * vcycle}


# ------------------------------------------------- the same in plain torch
def _residual(pr, p, T):
    """(R_m, R_e) of the backward-Euler TPFA discretisation, upwinded, with wells."""
    f, n = WATER, p.numel()
    nx, ny, nz = pr["nx"], pr["ny"], pr["nz"]
    t = lambda a: torch.as_tensor(a, dtype=torch.float64, device=p.device)
    rho_of = lambda p, T: f["rho0"] * torch.exp(f["c"] * (p - f["p0"])) * torch.exp(
        f["beta"] * (T - f["T0"]))
    rho = rho_of(p, T)
    lam = rho / (f["mu0"] * torch.exp(-f["mu_coef"] * (T - f["T_mu0"])))
    p_n, T_n, phi = t(pr["p_n"]), t(pr["T_n"]), t(pr["phi"])
    rho_n = rho_of(p_n, T_n)
    kT = phi * t(pr["kTr"]) + (1.0 - phi) * f["kTf"]
    vol, cv = CELL ** 3, f["cv"]
    R_m = vol * phi * (rho - rho_n) / pr["dt"]
    R_e = vol * (phi * cv * (rho * T - rho_n * T_n)
                 + (1.0 - phi) * f["rho_r"] * f["cr"] * (T - T_n)) / pr["dt"]
    idx = torch.arange(n, device=p.device).reshape(nz, ny, nx)
    for axis, K in ((2, pr["Kx"]), (1, pr["Ky"]), (0, pr["Kz"])):
        m, K = idx.shape[axis], t(K)
        lo, hi = idx.narrow(axis, 0, m - 1).reshape(-1), idx.narrow(axis, 1, m - 1).reshape(-1)
        T_f = CELL * 2.0 * K[lo] * K[hi] / (K[lo] + K[hi])
        Tc_f = CELL * 2.0 * kT[lo] * kT[hi] / (kT[lo] + kT[hi])
        head = GRAVITY * CELL if axis == 0 else 0.0
        dphi = p[lo] - p[hi] - 0.5 * (rho[lo] + rho[hi]) * head
        low = dphi >= 0.0
        F = T_f * torch.where(low, lam[lo], lam[hi]) * dphi
        E = cv * torch.where(low, T[lo], T[hi]) * F + Tc_f * (T[lo] - T[hi])
        R_m = R_m.index_add(0, lo, F).index_add(0, hi, -F)
        R_e = R_e.index_add(0, lo, E).index_add(0, hi, -E)
    for w in pr["wells"]:
        k = torch.arange(w["k0"], w["k1"] + 1, device=p.device)
        c = w["i"] + nx * (w["j"] + ny * k)
        if w["kind"] == 0:
            q = -(w["value"] / k.numel()) * rho_of(p[c], torch.full_like(p[c], w["T_inj"]))
            R_m, R_e = R_m.index_add(0, c, q), R_e.index_add(0, c, q * cv * w["T_inj"])
        else:  # bottom-hole pressure, Peaceman index of a 5 m block, isotropic horizontally
            wi = 2.0 * math.pi * 5.0 * t(pr["Kx"])[c] / math.log(0.14 * math.sqrt(50.0) / 0.1)
            drop = p[c] - w["value"]
            q = wi * torch.where(drop > 0.0, drop, torch.zeros_like(drop)) * lam[c]
            R_m, R_e = R_m.index_add(0, c, q), R_e.index_add(0, c, q * cv * T[c])
    return R_m, R_e


def _stencil(pr, p, T):
    """The Jacobian's entries: {(variable, offset): (dR_m, dR_e)} by row. Cells of one colour
    (x + 2 y + 3 z mod 7) share no row of the 7-point pattern, so seven products per variable
    give every entry."""
    n, nx, ny = p.numel(), pr["nx"], pr["ny"]
    i = torch.arange(n, device=p.device)
    x, y, z = i % nx, (i // nx) % ny, i // (nx * ny)
    colour = (x + 2 * y + 3 * z) % 7
    zero = torch.zeros_like(p)
    out = {}
    moves = {(0, 0, 0): 0, (1, 0, 0): 1, (-1, 0, 0): -1, (0, 1, 0): nx, (0, -1, 0): -nx,
             (0, 0, 1): nx * ny, (0, 0, -1): -nx * ny}
    for var in range(2):
        cols = []
        for k in range(7):
            d = (colour == k).double()
            tangent = (d, zero) if var == 0 else (zero, d)
            cols.append(torch.func.jvp(lambda a, b: _residual(pr, a, b), (p, T), tangent)[1])
        for (ax, ay, az), off in moves.items():
            inside = ((x + ax >= 0) & (x + ax < nx) & (y + ay >= 0) & (y + ay < ny)
                      & (z + az >= 0) & (z + az < pr["nz"]))
            c = (colour + ax + 2 * ay + 3 * az) % 7
            out[var, off] = [torch.where(inside, torch.stack([v[e] for v in cols]).gather(
                0, c[None])[0], zero) for e in range(2)]
    return out


def _dense(stencil, var, eq, n, device):
    A = torch.zeros(n, n, dtype=torch.float64, device=device)
    i = torch.arange(n, device=device)
    for (v, off), rows in stencil.items():
        if v == var:
            ok = (i + off >= 0) & (i + off < n)
            A[i[ok], i[ok] + off] += rows[eq][ok]
    return A


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    t = lambda a: torch.as_tensor(a, dtype=torch.float64, device=device)
    if case["kind"] == "train":
        rng = np.random.default_rng([seed, case["batch"]])
        params = t(_params(rng, 0.1)).requires_grad_(True)
        X, slot, St, Sd, target = (torch.as_tensor(a, device=device)
                                   for a in _batch(rng, case["validation"]))
        sizes = [NH * NF, NH, NH * NH, NH, NO * NH, NO]
        W1, b1, W2, b2, W3, b3 = torch.split(params, sizes)
        gelu = lambda z: torch.nn.functional.gelu(z, approximate="tanh")
        h = gelu(X.double() @ W1.reshape(NH, NF).T + b1)
        h = gelu(h @ W2.reshape(NH, NH).T + b2)
        o = h @ W3.reshape(NO, NH).T + b3
        pred = St * torch.exp(o.gather(1, slot.long()[:, None])[:, 0])
        pred = pred + torch.where(slot == 0, o[:, 7] * Sd, torch.zeros_like(Sd))
        loss = (((pred - target) / Sd) ** 2).mean()
        loss.backward()
        return {"validation_loss": float(loss.detach()), "gradient": params.grad.cpu().numpy(),
                "losses": [None] * case["steps"], "params": None}
    if case["kind"] in ("newton", "amg"):
        return None
    n = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "step" and n > 2500 or case["kind"] == "probe" and n > 21_000:
        return None
    pr = _problem(case, seed)
    rng = pr.pop("rng")
    p, T = t(pr["p_k"]), t(pr["T_k"])
    if case["kind"] == "assemble":
        R_m, R_e = _residual(pr, p, T)
        return {"R_m": R_m, "R_e": R_e}
    if case["kind"] == "spmv":
        x = t(1.0e5 * rng.standard_normal(n)), t(rng.standard_normal(n))
        y = torch.func.jvp(lambda a, b: _residual(pr, a, b), (p, T), x)[1]
        return {"y_p": y[0], "y_T": y[1]}
    st = _stencil(pr, p, T)
    if case["kind"] == "step":
        A = torch.cat([torch.cat([_dense(st, v, e, n, device) for v in range(2)], 1)
                       for e in range(2)], 0)
        b = -torch.cat(_residual(pr, p, T))
        r = 1.0 / A.abs().amax(1)  # the two equations and unknowns differ by many orders
        A, b = A * r[:, None], b * r
        c = 1.0 / A.abs().amax(0)
        x = torch.linalg.solve(A * c, b) * c
        return {"x_p": x[:n], "x_T": x[n:], "iterations": None}
    cols = np.sort(rng.choice(n, case["cols"], replace=False))
    App, rhs = _dense(st, 0, 0, n, device), torch.zeros(n, len(cols), dtype=torch.float64,
                                                        device=device)
    nx, ny = case["nx"], case["ny"]
    A_TT = torch.zeros_like(rhs)
    offs = [-nx * ny, -nx, -1, 0, 1, nx, nx * ny]
    for q, j in enumerate(cols):
        for off in offs:
            if 0 <= j - off < n:
                rhs[j - off, q] += st[1, off][0][j - off]
                A_TT[j - off, q] += st[1, off][1][j - off]
    r = 1.0 / App.diagonal()
    zs = torch.linalg.solve(App * r[:, None], rhs * r[:, None])
    del App
    S = A_TT.clone()
    i = torch.arange(n, device=device)
    for off in offs:
        ok = (i + off >= 0) & (i + off < n)
        S[i[ok]] -= st[0, off][1][ok][:, None] * zs[i[ok] + off]
    S = S.cpu().numpy()
    value = np.zeros((len(cols), 7))
    for q, j in enumerate(cols):  # rows of column j, ascending, packed
        x, y, z = j % nx, (j // nx) % ny, j // (nx * ny)
        inside = [z > 0, y > 0, x > 0, True, x < nx - 1, y < ny - 1, z < case["nz"] - 1]
        rows = [j + off for off, ok in zip(offs, inside) if ok]
        value[q, :len(rows)] = S[rows, q]
    return {"entry": None, "value": value, "iterations": None, "status": None}
