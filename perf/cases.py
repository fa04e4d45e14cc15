"""Performance cases of the batched powered-descent solver.

Three kinds of call, each through the package's public binding:

  step    Solver.scp_step: one SCP iteration (discretization, prescaling, power
          iteration, PIPG, update) on a batch of references, as a program does
          that runs the SCP loop itself (its own line search, its own stop).
          The references are initial guesses with a small dispersion, the warm
          start is empty: the first iteration of a solve.
  solve   Solver.solve: whole SCP solves.
  grad    Solver.grad: whole solves and the gradients of fuel and touchdown
          error with respect to x0.

Whole solves and gradients are taken where every instance converges (few nodes,
or the 3-DoF model): a run that does not converge wanders, a change in the last
bit of its input then changes all of its output, and its values say nothing.
FP32 steps run the iteration counts they are given (`force`), as a program with
a fixed time budget does; with stop tests, the counts in FP32 depend on the
last bit.  Their results are returned as the FP32 numbers that they are.
"""
from __future__ import annotations

import numpy as np
import torch

from paper_2404_18034_gb300 import flops, inputs
from paper_2404_18034_gb300.pdg_mc import Solver


def listed():
    return [
        # guidance on board: one vehicle, one trajectory, the answer as soon as possible
        dict(_case("solve", B=1, n=10, mode=0), name="solve_one_n10"),
        # a Monte Carlo study of moderate size, whole solves by the persistent kernel
        dict(_case("solve", B=1024, n=10, mode=1), name="solve_n10_b1024"),
        # sensitivities of a dispersed batch (training, targeting): forward and adjoint
        dict(_case("grad", B=256, n=10), name="grad_n10_b256"),
        # a handful of vehicles (one formation): fewer instances than SMs
        dict(_case("step", B=24, n=15), name="step_n15_b24"),
        # the headline batch: 6-DoF, 15 nodes, FP64
        dict(_case("step", B=16384, n=15), name="step_n15_b16384"),
        # a fine grid: twice the nodes, few instances resident per SM
        dict(_case("step", B=2048, n=30), name="step_n30_b2048"),
        # the paper's full model: RCS torque (7 controls), its r(0) distribution
        dict(_case("step", B=2048, n=15, nu=7, kind="paper256"), name="step_nu7_n15_b2048"),
        # a mixed batch: node counts 10, 15, 20, 30 drawn per instance
        dict(_case("step", B=3000, n=30, uneven=True), name="step_uneven_b3000"),
        # the glide-slope row, an odd grid
        dict(_case("step", B=1500, n=17, glide=1), name="step_glide_n17_b1500"),
        # the translational 3-DoF model, a large batch
        dict(_case("step", B=12000, n=15, model="3dof"), name="step_3dof_n15_b12000"),
        # FP32 with a fixed iteration budget, 6-DoF
        dict(_case("step", B=16384, n=15, fp32=1), name="step_fp32_n15_b16384"),
        # FP32 with a fixed iteration budget, 3-DoF, a fine grid
        dict(_case("step", B=4096, n=30, model="3dof", fp32=1), name="step_fp32_3dof_n30_b4096"),
    ]


def _case(call, B, n, nu=4, model="6dof", kind="bj", fp32=0, uneven=False, soc=0, glide=0, mode=1):
    return dict(call=call, B=int(B), n=int(n), nu=int(nu), model=model, kind=kind, fp32=int(fp32),
                uneven=bool(uneven), soc=int(soc), glide=int(glide), mode=int(mode))


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    call = rng.choice(["step"] * 6 + ["solve", "grad"])
    model = rng.choice(["6dof", "6dof", "3dof"])
    kind = "bj"
    if call == "step":
        n = rng.randint(4, 32)
        # no dearer than 16384 instances of 15 nodes
        B = _log(rng, 1, 16384 * 15 // max(n, 15))
        nu = 7 if model == "6dof" and rng.random() < 0.25 else 4
        fp32 = int(rng.random() < 0.25 and n >= 16)
        kind = rng.choice(["bj", "bj", "paper256"])
        return _case(call, B, n, nu, model, kind, fp32, uneven=rng.random() < 0.25, glide=int(rng.random() < 0.2))
    n = rng.randint(8, 11) if model == "6dof" else rng.randint(8, 30)
    if call == "solve":
        mode = rng.choice([0, 1])
        # thrust cone by projection: the persistent form's option
        soc = int(mode == 1 and model == "3dof" and rng.random() < 0.3)
        return _case(call, _log(rng, 1, 2000), n, model=model, mode=mode, soc=soc)
    return _case(call, _log(rng, 1, 400), min(n, 16), model=model)


# ---------------------------------------------------------------------------
def _params(case):
    return inputs.load_params(nu=case["nu"], model=case["model"], soc_thrust=case["soc"], glide_slope=case["glide"])


def _nodes(case, seed):
    if not case["uneven"]:
        return None
    n = case["n"]
    return inputs.node_counts(case["B"], seed, sorted({max(2, n // 3), max(2, n // 2), max(2, (2 * n) // 3), n}))


def _guess(p, x0, n, counts):
    """Initial references of a batch (B, n, NX), (B, n, nu), padded with zeros
    past each instance's node count: straight lines from x0 to the target,
    normalized attitudes, hover thrust."""
    B, nx, nu = x0.shape[0], x0.shape[1] + 1, p["nu"]
    N = np.full(B, n) if counts is None else counts
    k = np.arange(n)
    live = k[None, :] < N[:, None]
    t = np.where(live, k[None, :] / (N[:, None] - 1.0), 0.0)[..., None]
    zf = p["z_f"]
    X = np.zeros((B, n, nx))
    X[..., :-1] = (1 - t) * x0[:, None, :] + t * zf[None, None, :-1]
    X[..., 0] = ((1 - t) * x0[:, None, :1] + t * 0.5 * (x0[:, None, :1] + p["m_dry"]))[..., 0]
    if nx == 15:
        q = X[..., 7:11]
        X[..., 7:11] = q / np.linalg.norm(q, axis=-1, keepdims=True)
    U = np.zeros((B, n, nu))
    U[..., 0] = X[..., 0] * np.linalg.norm(p["g_I"])
    U[..., -1] = p["tf_guess"]
    return X * live[..., None], U * live[..., None], live


def _inputs(case, seed):
    p = _params(case)
    x0 = inputs.dispersion(p, case["B"], seed, case["kind"])
    counts = _nodes(case, seed)
    return p, x0, counts


def _references(p, x0, n, counts, seed):
    """The guesses with a dispersion of 1 % of each component's scale (the
    first node stays at x0, attitudes stay unit)."""
    X, U, live = _guess(p, x0, n, counts)
    rng = np.random.default_rng(seed)
    dX = 0.01 * p["P_x"] * rng.standard_normal(X.shape)
    dX[:, 0] = 0
    dX[..., -1] = 0
    X += dX * live[..., None]
    U += 0.01 * p["P_u"][:p["nu"]] * rng.standard_normal(U.shape) * live[..., None]
    if X.shape[2] == 15:
        q = X[..., 7:11]
        X[..., 7:11] = np.where(live[..., None], q / np.maximum(np.linalg.norm(q, axis=-1, keepdims=True), 1e-9), 0)
    return X, U


# power and PIPG iterations of a step with a fixed budget
FORCE = (30, 500)


def prepare(case, seed):
    p, x0, counts = _inputs(case, seed)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    s = dict(case=case, solver=Solver(p, case["n"], case["fp32"]), x0=dev(x0), N=None if counts is None else dev(counts))
    B, n, nx, nu = case["B"], case["n"], x0.shape[1] + 1, p["nu"]
    if case["call"] == "step":
        X, U = _references(p, x0, n, counts, seed)
        s["X"], s["U"] = dev(X), dev(U)
        z = lambda *d: torch.zeros(*d, dtype=torch.float64, device="cuda")  # noqa: E731
        s["ws"] = dict(xh=z(B, n, nx), uh=z(B, n, nu), mup=z(B, n - 1, nx), mum=z(B, n - 1, nx), phi=z(B, n - 1, nx),
                       th=z(B, n - 1))
        s["force"] = torch.tensor([FORCE] * B, dtype=torch.int32, device="cuda") if case["fp32"] else None
    elif case["call"] == "grad":
        rng = np.random.default_rng(seed)
        s["gf"], s["gt"] = dev(1.0 + 0.1 * rng.standard_normal(B)), dev(1.0 + 0.1 * rng.standard_normal(B))
    return s


def run(s):
    S, case = s["solver"], s["case"]
    if case["call"] == "solve":
        return S.solve(s["x0"], s["N"], mode=case["mode"])
    if case["call"] == "grad":
        return S.grad(s["x0"], s["N"], s["gf"], s["gt"])
    # the reference is kept: the step works on the candidate
    X, U, ws = s["X"].clone(), s["U"].clone(), {k: v.clone() for k, v in s["ws"].items()}
    out = dict(S.scp_step(s["x0"], X, U, ws, s["N"], s["force"]), X=X, U=U, **ws)
    if case["fp32"]:
        out = {k: v.float() if v.dtype == torch.float64 else v for k, v in out.items()}
    return out


def work(case):
    """Bytes: the call's inputs read once and its outputs written once.  Flops:
    the method's own operations (flops.py) at the mean node count, for the
    iteration counts such a call runs: all of PIPG's (its tolerance is seldom
    met before the cap), about 40 of the power iteration, about 8 SCP
    iterations in a solve (7 for the 3-DoF model)."""
    p = _params(case)
    B, n, nu, m = case["B"], case["n"], case["nu"], case["model"]
    N = int(round(np.mean(_nodes(dict(case, B=4096), 1)))) if case["uneven"] else n
    nx = 15 if m == "6dof" else 8
    pw, pi = FORCE if case["fp32"] else (40, p["pipg_jmax"])
    one = flops.discretization(N, nu, p["rk4_substeps"], m) + pw * flops.power_iter(N, nu, m) + pi * flops.pipg_iter(N, nu, m)
    if case["call"] == "step":
        state = n * (nx + nu) * 2 + (n - 1) * (3 * nx + 1)
        return dict(bytes=B * (8 * (2 * state + nx + 2) + (4 if case["uneven"] else 0)), flops=B * one)
    its = 8 if m == "6dof" else 7
    if case["call"] == "solve":
        return dict(bytes=8 * B * (n * (nx + nu) + nx + 4), flops=B * its * one)
    # the adjoint: the last PIPG loop once more and once in reverse
    return dict(bytes=8 * B * (2 * nx + 4), flops=B * (its * one + 2 * pi * flops.pipg_iter(N, nu, m)))


# ---------------------------------------------------------------------------
# the same results in plain torch, 64 bits
# ---------------------------------------------------------------------------
def _dynamics(p, x, u):
    """f = s (F, sum |g|_+^2) of one state and control."""
    T, s, m, r, v = u[:3], u[-1], x[0], x[1:4], x[4:7]
    nT = torch.sqrt((T * T).sum())
    g = torch.tensor(p["g_I"], dtype=x.dtype, device=x.device)
    sec = 1.0 / np.cos(p["delta_max"])
    rows = [p["m_dry"] - m, -r[0], (v * v).sum() - p["v_max"] ** 2, p["T_min"] - nT]
    if not p["soc_thrust"]:
        rows += [nT - T[0] * sec, nT - p["T_max"]]
    if p["glide_slope"]:
        rows.append(np.tan(p["gamma_gs"]) ** 2 * (r[1] ** 2 + r[2] ** 2) - r[0] ** 2)
    if p["model"] == "3dof":
        F = [(-p["alpha_mdot"] * nT)[None], v, T / m + g]
    else:
        q, w = x[7:11], x[11:14]
        J, rT = (torch.tensor(p[k], dtype=x.dtype, device=x.device) for k in ("J_B", "r_T_B"))
        q0, q1, q2, q3 = q
        C = torch.stack([torch.stack([1 - 2 * (q2 * q2 + q3 * q3), 2 * (q1 * q2 - q0 * q3), 2 * (q1 * q3 + q0 * q2)]),
                         torch.stack([2 * (q1 * q2 + q0 * q3), 1 - 2 * (q1 * q1 + q3 * q3), 2 * (q2 * q3 - q0 * q1)]),
                         torch.stack([2 * (q1 * q3 - q0 * q2), 2 * (q2 * q3 + q0 * q1), 1 - 2 * (q1 * q1 + q2 * q2)])])
        qd = 0.5 * torch.stack([-w[0] * q1 - w[1] * q2 - w[2] * q3, w[0] * q0 + w[2] * q2 - w[1] * q3,
                                w[1] * q0 - w[2] * q1 + w[0] * q3, w[2] * q0 + w[1] * q1 - w[0] * q2])
        tq = torch.linalg.cross(rT, T) - torch.linalg.cross(w, J * w)
        rows += [2 * (q2 * q2 + q3 * q3) - (1 - np.cos(p["theta_max"])), (w * w).sum() - p["omega_max"] ** 2]
        if p["nu"] == 7:
            tq = tq + u[3:6]
            rows.append((u[3:6] ** 2).sum() - p["gamma_max"] ** 2)
        F = [(-p["alpha_mdot"] * nT)[None], v, C @ T / m + g, qd, tq / J]
    pen = torch.stack([torch.relu(row) ** 2 for row in rows]).sum()
    return s * torch.cat(F + [pen[None]])


def _discretize(p, X, U, jac=True):
    """RK4 over every interval of X, U (B, N, .): the end states, and A, B-, B+
    of the same steps."""
    nx, nu, N, ns = X.shape[2], U.shape[2], X.shape[1], p["rk4_substeps"]
    x, u0, u1 = X[:, :-1].reshape(-1, nx), U[:, :-1].reshape(-1, nu), U[:, 1:].reshape(-1, nu)
    f = lambda a, b: _dynamics(p, a, b)  # noqa: E731
    both = torch.func.vmap(lambda a, b: (f(a, b), torch.func.jacfwd(f, (0, 1))(a, b)))
    only = torch.func.vmap(f)
    h = 1.0 / ((N - 1) * ns)
    P = torch.cat([torch.eye(nx, dtype=X.dtype, device=X.device), X.new_zeros(nx, 2 * nu)], 1).expand(x.shape[0], -1, -1)

    def rhs(x, P, lp):
        u = (1 - lp) * u0 + lp * u1
        if not jac:
            return only(x, u), 0.0
        d, (Jx, Ju) = both(x, u)
        return d, Jx @ P + torch.cat([torch.zeros_like(Jx), (1 - lp) * Ju, lp * Ju], 2)

    for i in range(ns):
        a, A = rhs(x, P, i / ns)
        b, Bq = rhs(x + 0.5 * h * a, P + 0.5 * h * A, (i + 0.5) / ns)
        c, C = rhs(x + 0.5 * h * b, P + 0.5 * h * Bq, (i + 0.5) / ns)
        d, D = rhs(x + h * c, P + h * C, (i + 1) / ns)
        x, P = x + h / 6 * (a + 2 * b + 2 * c + d), P + h / 6 * (A + 2 * Bq + 2 * C + D)
    shape = X.shape[:1] + (N - 1,)
    return x.reshape(*shape, nx), P.reshape(*shape, nx, nx + 2 * nu) if jac else None


def _scaled(p, x0, X, U):
    """The scaled subproblem: K = [A- B- B+] per interval, w, eps, box, z_i, z_f."""
    nu, t = p["nu"], lambda a: torch.as_tensor(a, dtype=X.dtype, device=X.device)
    Px, Pu = t(p["P_x"]), t(p["P_u"][:nu])
    end, P = _discretize(p, X, U)
    K = P * torch.cat([Px, Pu, Pu]) / Px[:, None]
    N = X.shape[1]
    lo, hi = p["s_min"], min(p["s_max"], p["tf_max"]) if p["tf_max"] > 0 else p["s_max"]
    return dict(K=K, w=(end - X[:, 1:]) / Px, eps=(p["eps_ctcs"] - (X[:, 1:, -1] - X[:, :-1, -1])) / Px[-1],
                lo=(lo - U[..., -1]) / Pu[-1], hi=(hi - U[..., -1]) / Pu[-1],
                zi=(torch.nn.functional.pad(x0, (0, 1)) - X[:, 0]) / Px, zf=(t(p["z_f"]) - X[:, -1]) / Px,
                fix=t(p["fix_f"]).bool(), Px=Px, Pu=Pu, N=N)


def _fwd(q, x, u):
    return (q["K"] @ torch.cat([x[:, :-1], u[:, :-1], u[:, 1:]], 2)[..., None])[..., 0] - x[:, 1:]


def _adj(q, phi, th):
    """K^T (phi, theta) on x and u."""
    nx = phi.shape[2]
    g = (q["K"].transpose(2, 3) @ phi[..., None])[..., 0]
    nu = (g.shape[2] - nx) // 2
    pad = torch.nn.functional.pad
    gx = pad(g[..., :nx], (0, 0, 0, 1)) - pad(phi, (0, 0, 1, 0))
    gx = gx + pad((pad(th, (1, 0)) - pad(th, (0, 1)))[..., None], (nx - 1, 0))
    return gx, pad(g[..., nx:nx + nu], (0, 0, 0, 1)) + pad(g[..., nx + nu:], (0, 0, 1, 0))


def _power(p, q, ws, force):
    x, u, a, b = ws["xh"], ws["uh"], ws["mup"], ws["mum"]
    norm = lambda *v: torch.sqrt(sum((t * t).flatten(1).sum(1) for t in v))  # noqa: E731
    sig = norm(x, u, a, b)
    one = (sig == 0)[:, None, None]
    x, u, a, b = (torch.where(one, torch.ones_like(t), t) for t in (x, u, a, b))
    sig = norm(x, u, a, b)
    best, its, on = sig.clone(), torch.zeros_like(sig, dtype=torch.int32), torch.ones_like(sig, dtype=torch.bool)
    for j in range(1, (force or p["pow_jmax"]) + 1):
        phi = (_fwd(q, x, u) + a - b) / sig[:, None, None]
        th = (x[:, 1:, -1] - x[:, :-1, -1]) / sig[:, None]
        x, u = _adj(q, phi, th)
        a, b = phi, -phi
        s = norm(x, u, a, b)
        best, its = torch.where(on, s, best), torch.where(on, j, its)
        if not force:
            on = on & ((s - sig).abs() > p["pow_eps_abs"] + p["pow_eps_rel"] * torch.maximum(s, sig))
            if not on.any():
                break
        sig = s
    return (1 + p["pow_eps_buff"]) * best, its.int()


def _sector(p, q, T):
    """The node's thrust onto {|T| <= T_max, |(T_y, T_z)| <= tan(delta) T_x}."""
    a = np.tan(p["delta_max"])
    r = torch.sqrt(T[..., 1] ** 2 + T[..., 2] ** 2)
    t = (T[..., 0] + a * r) / (1 + a * a)
    side = (a * t / torch.where(r > 0, r, torch.ones_like(r)))[..., None]
    on = torch.cat([t[..., None], T[..., 1:] * side], -1)
    T = torch.where((r > a * T[..., 0])[..., None], torch.where((a * r <= -T[..., 0])[..., None], torch.zeros_like(T), on), T)
    n = torch.sqrt((T * T).sum(-1, keepdim=True))
    return torch.where(n > p["T_max"], T * (p["T_max"] / torch.where(n > 0, n, torch.ones_like(n))), T)


def _pipg(p, q, ws, sigma, U, force=None, counts=None):
    """PIPG from ws: `force` iterations, counts per instance (held), or with the
    stop test.  Returns the new state and each instance's iterations."""
    wp, rho = p["w_prox"], p["pipg_rho"]
    al = 2 / (wp + torch.sqrt(wp * wp + 4 * p["pipg_omega"] * sigma))
    a3, a2 = al[:, None, None], al[:, None]
    be3, be2 = p["pipg_omega"] * a3, p["pipg_omega"] * a2
    z = [ws[k] for k in ("xh", "uh", "mup", "mum", "phi", "th")]
    tl = list(z)
    B = sigma.shape[0]
    its, on = torch.zeros(B, dtype=torch.int32, device=sigma.device), torch.ones(B, dtype=torch.bool, device=sigma.device)
    cost = torch.zeros_like(z[0])
    cost[:, -1, 0] = p["w_cost"]
    top = lambda *v: torch.stack([t.abs().flatten(1).amax(1) for t in v]).amax(0)  # noqa: E731
    most = force or (int(counts.max()) if counts is not None else p["pipg_jmax"])
    last = torch.zeros_like(z[0], dtype=torch.bool)
    last[:, -1] = q["fix"]
    for j in range(1, most + 1):
        x, u, a, b, f, t = tl
        gx, gu = _adj(q, f, t)
        xn = (1 - a3 * wp) * x - a3 * (gx - cost)
        xn = torch.cat([q["zi"][:, None], torch.where(last, q["zf"][:, None], xn)[:, 1:]], 1)
        un = (1 - a3 * wp) * u - a3 * gu
        un = torch.cat([un[..., :-1], torch.minimum(torch.maximum(un[..., -1], q["lo"]), q["hi"])[..., None]], 2)
        if p["soc_thrust"]:
            T = _sector(p, q, U[..., :3] + q["Pu"][:3] * un[..., :3])
            un = torch.cat([(T - U[..., :3]) / q["Pu"][:3], un[..., 3:]], 2)
        an, bn = torch.relu(a - a3 * (p["w_ep"] + f)), torch.relu(b - a3 * (p["w_ep"] - f))
        dx = 2 * xn - x
        fn = f + be3 * (q["w"] + (2 * an - a) - (2 * bn - b) + _fwd(q, dx, 2 * un - u))
        tn = torch.relu(t + be2 * (dx[:, 1:, -1] - dx[:, :-1, -1] - q["eps"]))
        new = [xn, un, an, bn, fn, tn]
        run = on if counts is None else j <= counts
        keep = lambda m, v, w: torch.where(m.reshape(-1, *[1] * (v.dim() - 1)), v, w)  # noqa: E731
        old, every = z, force is None or counts is not None
        z = [keep(run, v, w) for v, w in zip(new, z)] if every else new
        tl = [keep(run, w + rho * (v - w), w) for v, w in zip(new, tl)] if every else [w + rho * (v - w) for v, w in zip(new, tl)]
        its = its + run.int()
        if every and counts is None and j % p["pipg_jcheck"] == 0:
            d, m = top(*(v - w for v, w in zip(z[:4], old))), torch.maximum(top(*z[:4]), top(*old[:4]))
            dd, dm = top(*(v - w for v, w in zip(z[4:], old[4:]))), torch.maximum(top(*z[4:]), top(*old[4:]))
            lim = lambda m: p["pipg_eps_abs"] + p["pipg_eps_rel"] * m  # noqa: E731
            on = on & ~((d <= lim(m)) & (dd <= lim(dm)))
            if not on.any():
                break
    return dict(zip(("xh", "uh", "mup", "mum", "phi", "th"), z)), its


def _step(p, x0, X, U, ws, force=None):
    """One SCP iteration; the new X, U, warm start and what a step reports."""
    q = _scaled(p, x0, X, U)
    sigma, pw = _power(p, q, ws, force and force[0])
    ws, pi = _pipg(p, q, ws, sigma, U, force and force[1])
    step = torch.maximum(ws["xh"].abs().flatten(1).amax(1), ws["uh"].abs().flatten(1).amax(1))
    return dict(ws, X=X + q["Px"] * ws["xh"], U=U + q["Pu"] * ws["uh"], sigma=sigma, step=step,
                defect=q["w"].abs().flatten(1).amax(1), iters=torch.stack([pw, pi], 1))


def _zeros(B, n, nx, nu, like):
    z = lambda *d: like.new_zeros(*d)  # noqa: E731
    return dict(xh=z(B, n, nx), uh=z(B, n, nu), mup=z(B, n - 1, nx), mum=z(B, n - 1, nx), phi=z(B, n - 1, nx), th=z(B, n - 1))


def _solve(p, x0, X, U):
    """Whole solves; also each instance's last iteration (its reference, warm
    start, sigma and PIPG count), which the gradient differentiates."""
    B, n, nx = X.shape
    ws = _zeros(B, n, nx, U.shape[2], X)
    on = torch.ones(B, dtype=torch.bool, device=X.device)
    status, scp, total = (torch.zeros(B, dtype=d, device=X.device) for d in (torch.int32, torch.int32, torch.int64))
    status += 1
    last = {}
    for _ in range(p["scp_jmax"]):
        r = _step(p, x0, X, U, ws)
        put = lambda new, old: torch.where(on.reshape(-1, *[1] * (new.dim() - 1)), new, old)  # noqa: E731
        now = dict(ws, X=X, U=U, sigma=r["sigma"], n=r["iters"][:, 1])
        last = {k: put(v, last.get(k, v)) for k, v in now.items()}
        X, U, ws = put(r["X"], X), put(r["U"], U), {k: put(r[k], ws[k]) for k in ws}
        scp, total = scp + on.int(), total + r["iters"][:, 1].long() * on
        done = (r["step"] <= p["scp_eps_step"]) & (r["defect"] <= p["scp_eps_defect"]) & \
            (X[:, -1, -1] - X[:, 0, -1] <= (n - 1) * p["eps_ctcs"])
        status = torch.where(on & done, 0, status).int()
        on = on & ~done
        if not on.any():
            break
    out = dict(X=X, U=U, tf=(0.5 * (U[:, :-1, -1] + U[:, 1:, -1])).sum(1) / (n - 1), fuel=X[:, 0, 0] - X[:, -1, 0],
               status=status, scp_iters=scp, pipg_iters=total)
    return out, last


def _grad(p, x0, X, U, gf, gt):
    """d (gf fuel + gt touch) / d x0 of each instance's last SCP iteration: its
    reference's first node moves with x0; the rest of the reference, the warm
    start, sigma and the PIPG count are held."""
    out, last = _solve(p, x0, X, U)
    x = x0.clone().requires_grad_(True)
    X = torch.cat([torch.nn.functional.pad(x, (0, 1))[:, None], last["X"][:, 1:]], 1)
    q = _scaled(p, x, X, last["U"])
    ws, _ = _pipg(p, q, last, last["sigma"], last["U"], counts=last["n"])
    X, U = X + q["Px"] * ws["xh"], last["U"] + q["Pu"] * ws["uh"]
    fuel = X[:, 0, 0] - X[:, -1, 0]
    end, _ = _discretize(dict(p, N=X.shape[1]), X, U, jac=False)
    zf = torch.as_tensor(p["z_f"], dtype=X.dtype, device=X.device)
    touch = 0.5 * (((end[:, -1] - zf) / q["Px"])[:, q["fix"]] ** 2).sum(1)
    (g,) = torch.autograd.grad((gf * fuel + gt * touch).sum(), x)
    return dict(grad=g, fuel=fuel.detach(), touch=touch.detach(), status=out["status"])


def exact(case, seed):
    n, B = case["n"], case["B"]
    if case["call"] == "grad" and B * n > 4096:
        return None  # the recorded loop would take too long
    p, x0, counts = _inputs(case, seed)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    if case["call"] != "step":
        X, U, _ = _guess(p, x0, n, counts)
        if case["call"] == "solve":
            with torch.no_grad():
                return _solve(p, dev(x0), dev(X), dev(U))[0]
        rng = np.random.default_rng(seed)
        gf, gt = dev(1.0 + 0.1 * rng.standard_normal(B)), dev(1.0 + 0.1 * rng.standard_normal(B))
        return _grad(p, dev(x0), dev(X), dev(U), gf, gt)
    X, U = _references(p, x0, n, counts, seed)
    nx, nu = X.shape[2], U.shape[2]
    x0, X, U = dev(x0), dev(X), dev(U)
    out = dict(_zeros(B, n, nx, nu, X), X=X.clone(), U=U.clone(), sigma=X.new_zeros(B), step=X.new_zeros(B),
               defect=X.new_zeros(B), iters=torch.zeros(B, 2, dtype=torch.int32, device=X.device))
    with torch.no_grad():
        for N in sorted(set(counts.tolist())) if counts is not None else [n]:
            at = torch.arange(B, device=X.device) if counts is None else torch.nonzero(dev(counts) == N)[:, 0]
            r = _step(p, x0[at], X[at, :N], U[at, :N], _zeros(len(at), N, nx, nu, X), FORCE if case["fp32"] else None)
            for k, v in r.items():
                if v.dim() == 1 or k == "iters":
                    out[k][at] = v
                else:
                    out[k][at, :v.shape[1]] = v
    return out
