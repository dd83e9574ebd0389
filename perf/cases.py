"""Performance cases of the micro-macro parareal framework.

Each case is one call (or one short sequence of calls) that a program using
this framework makes, at sizes of the repository's own workloads, tests and
benchmark.  ``listed()`` names them, ``draw()`` gives more of the same
ranges, ``prepare()`` makes what the program holds before the call, ``run()``
is the call, ``work()`` the bytes and operations it cannot do without and
``exact()`` the same results in 64-bit arithmetic from plain torch and numpy,
without this package.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1912_09240_gb300 import _lib as L
from paper_1912_09240_gb300.adjoint import fine_em, quantile_gradient, second_moment_gradient
from paper_1912_09240_gb300.batch import BatchSolver
from paper_1912_09240_gb300.fp_parareal import FPParareal
from paper_1912_09240_gb300.parareal import PararealSolver

DEV = "cuda"

# The systems of the repository's workloads: model parameters, fine step, grid.
FAMILIES = {
    "ou": dict(kind=L.PR_MODEL_OU, d=1, lam=1.0, beta=1.0, eps=0.1, tau_x=1.0, rates=(), dt=1e-3, lo=-4.0, hi=4.0),
    "double_well": dict(kind=L.PR_MODEL_DOUBLE_WELL, d=1, lam=0.5, beta=3.0, eps=1e-2, tau_x=1.0, rates=(), dt=1e-4,
                        lo=-3.0, hi=3.0),
    "multi": dict(kind=L.PR_MODEL_DW_MULTI, d=16, lam=0.5, beta=3.0, eps=1e-3, tau_x=1.0, rates=(), dt=1e-5, lo=-3.0,
                  hi=3.0),
    "chem": dict(kind=L.PR_MODEL_CHEM, d=1, lam=0.0, beta=1.0, eps=2.5e-2, tau_x=25.0,
                 rates=(60.0, 1.0, 4.8e-3, 0.666e-5, 0.833, 1.0), dt=1e-3, lo=0.0, hi=600.0),
    "advection": dict(kind=L.PR_MODEL_ADVECTION, d=1, lam=0.0, beta=1.0, eps=1.0, tau_x=1.0, rates=(), dt=1e-3,
                      lo=-12.0, hi=6.0),
}
ITERATORS = {"quantile": L.PR_ITER_QUANTILE, "add": L.PR_ITER_ADD, "mult": L.PR_ITER_MULT, "rot": L.PR_ITER_ROT}


def listed():
    return [
        # The headline workload from its initial ensemble on: the double well, 2^20 particles,
        # 50 slices x 1000 steps, pipelined, two iterations.  The largest case.
        dict(name="parareal_double_well", kind="parareal", family="double_well", precision="f32", n=1 << 20, K=50,
             steps=1000, bins=512, chunk=5, graph=False, matching="quantile", iters=2),
        # The plain binary64 workload in full (4096 particles, 8 x 125 steps), graph-replayed:
        # a small problem, where launches and the serial chain count.
        dict(name="parareal_ou_f64", kind="parareal", family="ou", precision="f64", n=4096, K=8, steps=125, bins=256,
             chunk=0, graph=True, matching="quantile", iters=4),
        # The chemical system's fine step of an iteration: 20 slices x 2000 steps of 10^5
        # particles, matching and both restrictions in the launch.
        dict(name="fine_chem", kind="fine", family="chem", precision="f32", d=1, n=100_000, slices=20, steps=2000,
             bins=600, match=True),
        # The 16-dimensional fast space, a pipelined chunk of four slices at a tenth of its particles.
        dict(name="fine_fast16", kind="fine", family="multi", precision="f32", d=16, n=400_000, slices=4, steps=1000,
             bins=1024, match=True),
        # The binary64 fine propagator that the binary32 one is measured against.
        dict(name="fine_f64", kind="fine", family="double_well", precision="f64", d=1, n=1 << 17, slices=2, steps=1000,
             bins=512, match=True),
        # Forward and backward through the autograd function: gradient of E[X_T^2] with respect
        # to the parameters and the initial state (the adjoint workload with 4 of its 20 slices).
        dict(name="adjoint_autograd", kind="adjoint", family="ou", n=1 << 18, K=4, steps=1000, dt=1e-4, ckpt=256,
             observable="autograd"),
        # Serving: 16 uneven OU problems (eps and particle counts over their ranges), two iterations.
        dict(name="batch_serving", kind="batch", problems=16, n_min=10_000, n_max=100_000, K=32, bins=256, iters=2,
             mix=1),
        # Restriction and matching as separate passes over all matched slices of the headline workload.
        dict(name="restrict_match", kind="transport", precision="f32", n=1 << 20, slices=49, bins=512, offset=0),
        # Matching that preserves the conditional: reweight, stratified resampling with the gather
        # of x and y, weighted restriction of the result, for a chunk of slices.
        dict(name="reweight_resample", kind="resample", precision="f32", d=1, n=1 << 20, slices=9, bins=512,
             mode="stratified"),
        # The Monte Carlo estimator: mean and second moment of every slice's end states.
        dict(name="moments", kind="moments", precision="f32", n=1 << 20, slices=49, order=2, weighted=False),
        # Parareal on densities (the linear advection case): the smallest calls, four iterations
        # of two coarse steps and a serial sweep each.
        dict(name="fp_parareal", kind="fp_parareal", bins=288, K=10, iterator="quantile", iters=4, eps_c=0.5,
             beta_c=1.0),
        # Setting up a solver's coarse propagator, as every solver and each run of a study does.
        dict(name="coarse_setup", kind="coarse", family="double_well", bins=512, dT=0.1),
    ]


# ---------------------------------------------------------------------------
# Drawn cases
# ---------------------------------------------------------------------------

def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _fit(n, cost_per_particle, budget):
    """The particle count, cut where the case would cost more than the budget (in particle-steps)."""
    return max(64, min(n, int(budget / cost_per_particle)))


def _draw_parareal(rng):
    family = rng.choice(["ou", "double_well", "chem"])
    f64 = rng.random() < 0.3
    K, steps = rng.randint(2, 50), _log_int(rng, 20, 1000)
    iters = rng.randint(1, 4)
    n = _fit(_log_int(rng, 1000, 1 << 20), K * steps * iters, 2e8 if f64 else 3e10)
    graph = rng.random() < 0.3
    return dict(kind="parareal", family=family, precision="f64" if f64 else "f32", n=n, K=K, steps=steps,
                bins=rng.randint(64, 640), chunk=rng.choice([0, 3, 5]), graph=graph,
                matching="quantile" if rng.random() < 0.75 else rng.choice(["resample", "resample_det", "reweight"]),
                iters=iters)


def _draw_fine(rng):
    family = rng.choice(["ou", "double_well", "multi", "chem"])
    f64 = rng.random() < 0.35
    d = rng.randint(2, 16) if family == "multi" else 1
    slices, steps = _log_int(rng, 1, 50), _log_int(rng, 7, 2000)
    n = _fit(_log_int(rng, 257, 1 << 20), slices * steps * (1 + d) / 2, 2e8 if f64 else 5e9)
    return dict(kind="fine", family=family, precision="f64" if f64 else "f32", d=d, n=n, slices=slices, steps=steps,
                bins=_log_int(rng, 64, 2000), match=rng.random() < 0.7)


def _draw_adjoint(rng):
    K, steps = rng.randint(1, 20), _log_int(rng, 25, 1000)
    n = _fit(_log_int(rng, 1000, 1 << 20), K * steps, 2e9)
    return dict(kind="adjoint", family=rng.choice(["ou", "double_well"]), n=n, K=K, steps=steps, dt=1e-4,
                ckpt=rng.choice([12, 64, 256, 301]),
                observable=rng.choice(["autograd", "second_moment", "quantile"]))


def _draw_batch(rng):
    n_min = _log_int(rng, 1000, 20_000)
    return dict(kind="batch", problems=rng.randint(3, 20), n_min=n_min, n_max=n_min * rng.randint(2, 10),
                K=rng.randint(4, 32), bins=rng.choice([128, 200, 256, 400]), iters=2, mix=rng.randint(0, 1 << 20))


def _draw_transport(rng):
    slices = rng.randint(1, 50)
    return dict(kind="transport", precision="f64" if rng.random() < 0.25 else "f32",
                n=_fit(_log_int(rng, 4096, 1 << 22), slices, 1 << 26), slices=slices, bins=_log_int(rng, 100, 2000),
                offset=rng.choice([0, 0, 1, 3]))


def _draw_resample(rng):
    slices = rng.randint(1, 12)
    return dict(kind="resample", precision="f64" if rng.random() < 0.25 else "f32", d=rng.choice([1, 1, 1, 3]),
                n=_fit(_log_int(rng, 4096, 1 << 21), slices, 1 << 24), slices=slices, bins=_log_int(rng, 64, 1024),
                mode=rng.choice(["stratified", "deterministic"]))


def _draw_moments(rng):
    slices = rng.randint(1, 50)
    return dict(kind="moments", precision="f64" if rng.random() < 0.25 else "f32",
                n=_fit(_log_int(rng, 4096, 1 << 22), slices, 1 << 26), slices=slices, order=rng.randint(1, 4),
                weighted=rng.random() < 0.4)


def _draw_fp_parareal(rng):
    return dict(kind="fp_parareal", bins=rng.randint(48, 640), K=rng.randint(4, 40),
                iterator=rng.choice(["quantile", "quantile", "add", "mult", "rot"]), iters=rng.randint(1, 5),
                eps_c=rng.choice([0.5, 1.0]), beta_c=rng.choice([0.5, 1.0, 2.0]))


def _draw_coarse(rng):
    family = rng.choice(["ou", "double_well", "chem", "advection"])
    return dict(kind="coarse", family=family, bins=rng.randint(100, 800),
                dT=2.0 if family == "chem" else rng.choice([0.0625, 0.1, 0.125, 0.2]))


def draw(rng):
    return rng.choice([_draw_parareal, _draw_fine, _draw_adjoint, _draw_batch, _draw_transport, _draw_resample,
                       _draw_moments, _draw_fp_parareal, _draw_coarse])(rng)


# ---------------------------------------------------------------------------
# What the program holds before the call
# ---------------------------------------------------------------------------

def _model(family, d=None):
    f = FAMILIES[family]
    return L.Model(f["kind"], f["d"] if d is None else d, f["lam"], f["beta"], f["eps"], f["tau_x"], f["rates"])


def _grid(family, bins):
    f = FAMILIES[family]
    return L.Grid(bins, f["lo"], f["hi"])


def _dtype(case):
    return torch.float64 if case["precision"] == "f64" else torch.float32


def _precision(case):
    return L.PR_F64 if case["precision"] == "f64" else L.PR_F32


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _initial(family, n, d, seed, dtype):
    """X_0 [n] and Y_0 [d][n] as the workloads draw them."""
    g = _gen(seed)
    z = torch.randn(1 + d, n, generator=g, device=DEV, dtype=torch.float64)
    if family == "chem":   # independent lognormals of mean 100 and standard deviation 20
        s2 = math.log1p(0.2 ** 2)
        v = torch.exp(math.log(100.0) - 0.5 * s2 + math.sqrt(s2) * z)
        x, y = v[0], v[1:]
    elif family == "ou":
        x, y = 1.0 + 0.1 * z[0], z[1:]
    else:
        x = -1.0 + 0.2 * z[0]
        y = x.expand(d, n)
    return x.to(dtype).contiguous(), y.to(dtype).contiguous()


def _later(family, n, slices, d, seed, dtype):
    """States of later slices, x [slices][n] and y [slices][d][n]: spread over the wells."""
    g = _gen(seed)
    x = torch.randn(slices, n, generator=g, device=DEV, dtype=torch.float32)
    u = torch.rand(slices, n, generator=g, device=DEV, dtype=torch.float32)
    f = torch.linspace(0.05, 0.5, slices, device=DEV).reshape(-1, 1)   # mass in the second well
    if family == "chem":
        x = torch.where(u < f, 340.0 + 18.0 * x, 100.0 + 11.0 * x)
    elif family == "ou":
        x = 1.0 - 1.5 * f + (0.1 + f) * x
    else:
        x = torch.where(u < f, 1.0, -1.0) + 0.28 * x
    e = torch.randn(slices, d, n, generator=g, device=DEV, dtype=torch.float32)
    y = (x * 1.2).unsqueeze(1) + 12.0 * e if family == "chem" else x.unsqueeze(1) + e
    return x.to(dtype).contiguous(), y.to(dtype).contiguous()


def _target(family, n, slices, bins, seed):
    """Target CDFs [slices][bins+1]: the restriction of another ensemble, a little further on."""
    x, _ = _later(family, min(n, 1 << 18), slices, 1, seed + 7919, torch.float64)
    scale = 100.0 if family == "chem" else 1.0
    return _restrict64(x * 1.01 + 0.02 * scale, _grid(family, bins))[1]


def _batch_problems(case, seed):
    rng = np.random.default_rng(case["mix"])
    m = case["problems"]
    eps = np.exp(rng.uniform(np.log(1e-3), np.log(1e-1), m))
    lam = rng.uniform(0.0, 1.0, m)
    n = np.rint(np.exp(rng.uniform(np.log(case["n_min"]), np.log(case["n_max"]), m))).astype(int)
    out = []
    for i in range(m):
        slice_dt = 2.0 / case["K"]
        steps = int(math.ceil(slice_dt / (eps[i] / 50.0)))
        out.append(L.Problem(L.Model(L.PR_MODEL_OU, 1, float(lam[i]), 1.0, float(eps[i])),
                             L.Grid(case["bins"], -4.0, 4.0), int(n[i]), case["K"], steps, slice_dt / steps, seed))
    return out


def _bytes_buffer(n):
    return torch.empty(max(int(n), 1), dtype=torch.uint8, device=DEV)


def _fp_models(case):
    adv = lambda eps, beta: L.Model(L.PR_MODEL_ADVECTION, 1, 0.0, beta, eps)
    return adv(1.0, 1.0), adv(case["eps_c"], case["beta_c"])


def _fp_start(case, seed):
    """R of N(m, 0.5^2) on [-12, 6], its mean around 1."""
    m = 1.0 + 0.2 * float(torch.rand(1, generator=_gen(seed), device=DEV).item())
    e = _edges64(L.Grid(case["bins"], -12.0, 6.0))
    c = 0.5 * (1.0 + torch.erf((e - m) / (0.5 * math.sqrt(2.0))))
    return ((c - c[0]) / (c[-1] - c[0])).to(DEV)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, seed=seed, rng=L.Rng(seed))
    if kind == "parareal":
        f = FAMILIES[case["family"]]
        s["solver"] = PararealSolver(_model(case["family"]), _grid(case["family"], case["bins"]), case["n"], case["K"],
                                     case["steps"], f["dt"], precision=_precision(case), rng=s["rng"], device=DEV,
                                     chunk=case["chunk"], graph=case["graph"], matching=case["matching"])
        s["x0"], s["y0"] = _initial(case["family"], case["n"], 1, seed, _dtype(case))
    elif kind == "fine":
        S, d, bins = case["slices"], case["d"], case["bins"]
        s["x"], s["y"] = _later(case["family"], case["n"], S, d, seed, _dtype(case))
        s["xo"], s["yo"] = torch.empty_like(s["x"]), torch.empty_like(s["y"])
        s["prior"] = s["target"] = None
        if case["match"]:
            s["prior"] = _restrict64(s["x"], _grid(case["family"], bins))[1]
            s["target"] = _target(case["family"], case["n"], S, bins, seed)
        s["counts"] = [torch.empty(S, bins, dtype=torch.int32, device=DEV) for _ in range(2)]
        s["cdf"] = [torch.empty(S, bins + 1, dtype=torch.float64, device=DEV) for _ in range(2)]
    elif kind == "adjoint":
        x, y = _initial(case["family"], case["n"], 1, seed, torch.float32)
        s["x0"], s["y0"] = x, y.reshape(-1)
        f = FAMILIES[case["family"]]
        s["theta"] = torch.tensor([f["lam"], f["beta"], f["eps"]], dtype=torch.float64)
    elif kind == "batch":
        probs = _batch_problems(case, seed)
        s["solver"] = BatchSolver(probs, device=DEV)
        n = sum(p.n for p in probs)
        s["x0"], y = _initial("ou", n, 1, seed, torch.float32)
        s["y0"] = y.reshape(-1)
    elif kind == "transport":
        x, _ = _later("double_well", case["n"], case["slices"], 1, seed, _dtype(case))
        # the ensemble `offset` elements into its buffer, as a slice of a larger array lies
        o, m = case["offset"], x.numel()
        s["x"] = torch.empty(m + o, dtype=x.dtype, device=DEV)[o:].reshape(x.shape)
        s["x"].copy_(x)
        s["xo"] = torch.empty(m + o, dtype=x.dtype, device=DEV)[o:].reshape(x.shape)
        s["target"] = _target("double_well", case["n"], case["slices"], case["bins"], seed)
        s["counts"] = torch.empty(case["slices"], case["bins"], dtype=torch.int32, device=DEV)
        s["cdf"] = torch.empty(case["slices"], case["bins"] + 1, dtype=torch.float64, device=DEV)
    elif kind == "resample":
        n, S, d = case["n"], case["slices"], case["d"]
        s["x"], s["y"] = _later("double_well", n, S, d, seed, _dtype(case))
        s["prior"] = _restrict64(s["x"], _grid("double_well", case["bins"]))[1]
        s["target"] = _target("double_well", n, S, case["bins"], seed)
        s["w"] = torch.empty(S, n, dtype=torch.float64, device=DEV)
        s["index"] = torch.empty(S, n, dtype=torch.int32, device=DEV)
        s["xo"], s["yo"] = torch.empty_like(s["x"]), torch.empty_like(s["y"])
        s["cdf"] = torch.empty(S, case["bins"] + 1, dtype=torch.float64, device=DEV)
        s["rs"] = _bytes_buffer(L.pr_resample_workspace(n, S))
        s["wr"] = _bytes_buffer(L.pr_restrict_weighted_workspace(S, case["bins"]))
    elif kind == "moments":
        n, S = case["n"], case["slices"]
        s["x"], _ = _later("double_well", n, S, 1, seed, _dtype(case))
        s["w"] = None
        if case["weighted"]:
            w = torch.rand(S, n, generator=_gen(seed + 1), device=DEV, dtype=torch.float64)
            s["w"] = w / w.sum(1, keepdim=True)
        s["out"] = torch.empty(S, case["order"], dtype=torch.float64, device=DEV)
        s["ws"] = _bytes_buffer(L.pr_moments_workspace(n, S, case["order"]))
    elif kind == "fp_parareal":
        fine, coarse = _fp_models(case)
        s["solver"] = FPParareal(L.Grid(case["bins"], -12.0, 6.0), fine, coarse, case["K"], 0.2,
                                 iterator=ITERATORS[case["iterator"]], device=DEV)
        s["cdf0"] = _fp_start(case, seed)
    elif kind == "coarse":
        # a horizon cut into slices of about dT, as the convergence studies vary it
        s["dT"] = _coarse_dT(case, seed)
        s["P"] = torch.empty(case["bins"], case["bins"], dtype=torch.float64, device=DEV)
    return s


def _coarse_dT(case, seed):
    return case["dT"] * (1.0 + 0.1 * float(np.random.default_rng(seed).random()))


# ---------------------------------------------------------------------------
# The calls
# ---------------------------------------------------------------------------

def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "parareal":
        sv = s["solver"]
        sv.set_initial(s["x0"], s["y0"])
        for _ in range(case["iters"]):
            sv.iterate()
        x, y, rho = sv.state()
        return {"rho": rho, "x": x, "y": y}
    if kind == "fine":
        (cs, ce), (ds, de) = s["counts"], s["cdf"]
        L.pr_fine_propagate(_model(case["family"], case["d"]), _precision(case), s["rng"], s["x"], s["y"], False,
                            s["xo"], s["yo"], case["n"], 0, case["slices"], case["steps"],
                            FAMILIES[case["family"]]["dt"], _grid(case["family"], case["bins"]), s["prior"],
                            s["target"], cs, ds, ce, de)
        return {"x": s["xo"], "y": s["yo"], "counts_start": cs, "cdf_start": ds, "counts_end": ce, "cdf_end": de}
    if kind == "adjoint":
        f = FAMILIES[case["family"]]
        if case["observable"] == "autograd":
            theta, x0, y0 = (s[k].detach().requires_grad_(True) for k in ("theta", "x0", "y0"))
            x, y = fine_em(theta, x0, y0, f["kind"], 1.0, s["rng"], 0, case["K"], case["steps"], case["dt"],
                           case["ckpt"])
            loss = (x * x).mean()
            loss.backward()
            return {"x": x.detach(), "y": y.detach(), "loss": loss.detach(), "theta_grad": theta.grad,
                    "x0_grad": x0.grad, "y0_grad": y0.grad}
        model = L.Model(f["kind"], 1, f["lam"], f["beta"], f["eps"])
        if case["observable"] == "second_moment":
            value, grad = second_moment_gradient(model, s["rng"], s["x0"], s["y0"], 0, case["K"], case["steps"],
                                                 case["dt"], case["ckpt"])
            return {"value": value, "grad": grad}
        q, dq, idx = quantile_gradient(model, s["rng"], s["x0"], s["y0"], 0, case["K"], case["steps"], case["dt"],
                                       512, case["ckpt"])
        return {"quantile": q, "grad": dq, "index": idx}
    if kind == "batch":
        sv = s["solver"]
        sv.set_initial(s["x0"], s["y0"])
        for _ in range(case["iters"]):
            sv.iterate()
        out = {}
        for i in range(case["problems"]):
            x, y = sv.fine_state(i)
            out["%02d" % i] = {"rho": sv.rho(i), "x": x, "y": y}
        return out
    if kind == "transport":
        grid = _grid("double_well", case["bins"])
        L.pr_restrict(_precision(case), s["x"], case["n"], case["slices"], grid, s["counts"], s["cdf"])
        L.pr_match(_precision(case), s["x"], s["xo"], case["n"], case["slices"], grid, s["cdf"], s["target"])
        return {"counts": s["counts"], "cdf": s["cdf"], "x": s["xo"]}
    if kind == "resample":
        grid, prec, n, S, d = _grid("double_well", case["bins"]), _precision(case), case["n"], case["slices"], case["d"]
        mode = L.PR_RESAMPLE_STRATIFIED if case["mode"] == "stratified" else L.PR_RESAMPLE_DETERMINISTIC
        L.pr_reweight(prec, s["x"], False, None, n, S, grid, s["prior"], s["target"], s["w"])
        L.pr_resample(prec, d, s["x"], s["y"], False, s["w"], n, S, 0, mode, s["rng"], s["index"], s["xo"], s["yo"],
                      s["rs"])
        L.pr_restrict_weighted(prec, s["x"], False, s["w"], n, S, grid, s["cdf"], s["wr"])
        return {"w": s["w"], "index": s["index"], "x": s["xo"], "y": s["yo"], "cdf": s["cdf"]}
    if kind == "moments":
        L.pr_moments(_precision(case), s["x"], case["n"], s["w"], case["n"], case["slices"], case["order"], s["out"],
                     s["ws"])
        return {"moments": s["out"]}
    if kind == "fp_parareal":
        sv = s["solver"]
        sv.set_initial(s["cdf0"])
        for _ in range(case["iters"]):
            sv.iterate()
        return {"rho": sv.rho}
    h = L.pr_coarse_create(_model(case["family"]), _grid(case["family"], case["bins"]), s["dT"])
    L.pr_coarse_matrix(h, s["P"])
    L.pr_coarse_destroy(h)
    return {"P": s["P"]}


# ---------------------------------------------------------------------------
# What one pass cannot do without
# ---------------------------------------------------------------------------

def _step_flops(d):
    """Floating-point operations of one Euler-Maruyama step of one particle: Box-Muller for
    1 + d normals (ten per pair) and the step itself (the generator's integer work not counted)."""
    return 5 * (1 + d) + 8 + 4 * d


def _sweep_flops(bins, slices):
    """A serial sweep: per slice a matrix-vector product and about 3 bins levels of quantiles."""
    return slices * (2 * bins * bins + 60 * bins)


def work(case):
    kind = case["kind"]
    sz = 8 if case.get("precision") == "f64" else 4
    if kind == "parareal":
        n, K, I = case["n"], case["K"], case["bins"]
        it = case["iters"]
        return {"bytes": sz * 2 * n + it * K * n * 4 * sz, "flops": it * (K * n * case["steps"] * _step_flops(1)
                                                                          + 2 * _sweep_flops(I, K))}
    if kind == "fine":
        n, S, d, I = case["n"], case["slices"], case["d"], case["bins"]
        return {"bytes": 2 * sz * S * n * (1 + d) + S * I * 40, "flops": S * n * case["steps"] * _step_flops(d)}
    if kind == "adjoint":
        n, t = case["n"], case["K"] * case["steps"]
        return {"bytes": 32 * n, "flops": n * t * (_step_flops(1) * (3 if case["observable"] == "autograd" else 2) + 20)}
    if kind == "batch":
        b = f = 0
        for p in _batch_problems(case, 0):
            b += case["iters"] * p.n * p.n_slices * 16
            f += case["iters"] * (p.n * p.n_slices * p.steps * _step_flops(1) + 2 * _sweep_flops(case["bins"], p.n_slices))
        return {"bytes": b, "flops": f}
    if kind == "transport":
        m = case["n"] * case["slices"]
        return {"bytes": m * sz * 3, "flops": 10 * m}
    if kind == "resample":
        m = case["n"] * case["slices"]
        # x and y read, w, the index and both states written; the weighted restriction reads x and w again
        return {"bytes": m * (2 * sz * (1 + case["d"]) + 8 + 4 + sz + 8), "flops": 10 * m}
    if kind == "moments":
        m = case["n"] * case["slices"]
        return {"bytes": m * (sz + (8 if case["weighted"] else 0)), "flops": 2 * case["order"] * m}
    if kind == "fp_parareal":
        I, K = case["bins"], case["K"]
        return {"bytes": 16 * I * I + (1 + case["iters"]) * (K + 1) * (I + 1) * 8,
                "flops": _sweep_flops(I, K) + case["iters"] * (4 * K * I * I + _sweep_flops(I, K))}
    I = case["bins"]
    # the matrix and its exponential: a squaring per factor 2 of the generator's norm, about 4 (I / 6)^2 dT
    return {"bytes": 8 * I * I, "flops": 2.0 * I ** 3 * max(1.0, math.log2(4.0 * I * I / 9.0 * case["dT"]))}


# ---------------------------------------------------------------------------
# The same results in 64 bits, from plain torch and numpy
# ---------------------------------------------------------------------------

def _edges64(grid):
    h = (grid.hi - grid.lo) / grid.bins
    return grid.lo + torch.arange(grid.bins + 1, dtype=torch.float64) * h


def _bins64(x, grid):
    """Bin of each particle: e_i <= x < e_{i+1}, the rest in the end bins."""
    e = _edges64(grid).to(x.device)
    return (torch.searchsorted(e, x, right=True) - 1).clamp_(0, grid.bins - 1)


def _restrict64(x, grid):
    """Counts [S][bins] and CDFs [S][bins+1] of x [S][n]."""
    counts = torch.stack([torch.bincount(_bins64(r.double(), grid), minlength=grid.bins) for r in x])
    cdf = torch.zeros(x.shape[0], grid.bins + 1, dtype=torch.float64, device=x.device)
    cdf[:, 1:] = counts.cumsum(1).double() / x.shape[1]
    return counts, cdf


def _match64(x, grid, prior, target):
    """X = c^{-1}(cbar(Xbar)), piecewise linear CDFs, lowest non-empty target bin; one slice."""
    e, h = _edges64(grid).to(x.device), (grid.hi - grid.lo) / grid.bins
    i = _bins64(x, grid)
    frac = ((x - e[i]) / h)
    below, above = frac < 0.0, frac > 1.0
    frac = frac.clamp(0.0, 1.0)
    u = prior[i] + frac * (prior[i + 1] - prior[i])
    full = (target[1:] > target[:-1]).nonzero().reshape(-1)
    j = full[torch.searchsorted(target[1:][full].contiguous(), u).clamp_(max=full.numel() - 1)]
    t = ((u - target[j]) / (target[j + 1] - target[j])).clamp(0.0, 1.0)
    xn = e[j] + t * h
    xn = torch.where(below, x + (xn - grid.lo), torch.where(above, x + (xn - grid.hi), xn))
    same = (prior[i] == target[i]) & (prior[i + 1] == target[i + 1])
    return torch.where(same, x, xn)


_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors holding 32-bit words (broadcast against each other)."""
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    c = [v if torch.is_tensor(v) else torch.tensor(v, dtype=torch.int64, device=DEV) for v in (c0, c1, c2, c3)]
    for _ in range(10):
        pa, pb = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = [((pb >> 32) & _M32) ^ c[1] ^ k0, pb & _M32, ((pa >> 32) & _M32) ^ c[3] ^ k1, pa & _M32]
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c


def _normals(w0, w1):
    u0, u1 = ((w >> 9).double().add_(0.5).mul_(1.0 / (1 << 23)) for w in (w0, w1))
    r, a = (-2.0 * u0.log()).sqrt_(), 2.0 * math.pi * u1
    return r * a.cos(), r * a.sin()


class _Noise:
    """The normals of step m for particles 0..n-1 of slices slice0..slice0+S-1: 1 + d tensors [S][n]."""

    def __init__(self, n, slices, d, seed, slice0=0, problem=0):
        self.p = torch.arange(n, dtype=torch.int64, device=DEV).reshape(1, -1)
        self.s = torch.arange(slice0, slice0 + slices, dtype=torch.int64, device=DEV).reshape(-1, 1)
        self.d, self.seed, self.hi = d, seed, problem << 8
        self.kept = {}

    def _block(self, c, g):
        """Block (c, p, slice, g): its four normals, kept until the counter moves on."""
        if self.kept.get(g, (None,))[0] != c:
            w = _philox(c, self.p, self.s, self.hi | g, self.seed)
            self.kept[g] = (c, _normals(w[0], w[1]) + _normals(w[2], w[3]))
        return self.kept[g][1]

    def __call__(self, m):
        q = 1 + self.d
        if q == 2:
            z = self._block(m >> 1, 0)
            return z[2:] if m & 1 else z[:2]
        f, t = q // 4, q % 4
        z = [v for g in range(f) for v in self._block(m, g)]
        for i in range((m & 3) * t, (m & 3) * t + t):
            z.append(self._block(m >> 2, f + i // 4)[i & 3])
        return z


def _chem_terms(k, y):
    y1, y2 = y * (y - 1.0), y * (y - 1.0) * (y - 2.0)
    return k[0] - k[1] * y + k[2] * y1 - k[3] * y2, k[0] + k[1] * y + k[2] * y1 + k[3] * y2


def _propagate64(family, x, y, steps, dt, seed, slice0=0):
    """Euler-Maruyama in 64 bits: x [S][n], y [S][d][n]."""
    f = FAMILIES[family]
    x, y = x.double().clone(), [v.double().clone() for v in y.unbind(1)]
    noise = _Noise(x.shape[1], x.shape[0], len(y), seed, slice0)
    ax, ay = dt / f["tau_x"], dt / f["eps"]
    sx, sy = math.sqrt(2.0 / f["beta"] * ax), math.sqrt(2.0 * ay)
    for m in range(steps):
        z = noise(m)
        if family == "chem":
            k = f["rates"]
            drift, twice_e = _chem_terms(k, y[0])
            xn = (x + (k[4] * y[0] - k[5] * x) * ax
                  + ((k[4] * y[0] + k[5] * x) * ax).clamp(min=0.0).sqrt() * z[0])
            y[0] = y[0] + drift * ay + (twice_e * ay).clamp(min=0.0).sqrt() * z[1]
        else:
            mean = sum(y) / len(y)
            grad = x - f["lam"] * mean if family == "ou" else x ** 3 - x + f["lam"] * mean
            xn = x - grad * ax + sx * z[0]
            for j in range(len(y)):
                y[j] = y[j] - (y[j] - x) * ay + sy * z[1 + j]
        x = xn
    return x, torch.stack(y, 1)


def _coarse64(model, grid, dT):
    """exp(A dT) of the finite volumes on the detailed-balance form, as a numpy array."""
    I = grid.bins
    e = _edges64(grid).numpy()
    mid, width = 0.5 * (e[1:] + e[:-1]), e[1:] - e[:-1]
    if model.kind == L.PR_MODEL_CHEM:
        k = model.rates
        y = 0.5 * np.arange(4001)
        net, twice_e = _chem_terms(k, y)
        r = -net / (0.5 * twice_e)
        inner = np.concatenate([[0.0], np.cumsum(0.25 * (r[1:] + r[:-1]))])
        lp = -inner - np.log(0.5 * twice_e)
        phi = np.exp(lp - lp.max())
        phi[[0, -1]] *= 0.5
        a = k[4] * (y * phi).sum() / phi.sum()
        diff = lambda x: 0.5 * (a + k[5] * x)
        log_rho = lambda x: -np.log(diff(x)) - (2.0 * x - 4.0 * a / k[5] * np.log1p(k[5] * x / a))
    else:
        lam, beta = model.lam, model.beta
        pot = {L.PR_MODEL_OU: lambda x: 0.5 * (1.0 - lam) * x * x,
               L.PR_MODEL_ADVECTION: lambda x: x / model.eps}.get(
                   model.kind, lambda x: 0.25 * x ** 4 - 0.5 * (1.0 - lam) * x * x)
        diff = lambda x: np.full_like(x, 1.0 / beta)
        log_rho = lambda x: np.log(beta) - pot(x) * beta
    xe = e[1:-1]
    coef = diff(xe) / (mid[1:] - mid[:-1]) / model.tau_x
    right = coef * np.exp(log_rho(xe) - log_rho(mid[1:])) / width[1:]     # flow out of cell e, rightmost of the edge
    left = coef * np.exp(log_rho(xe) - log_rho(mid[:-1])) / width[:-1]    # flow out of cell e - 1
    A = np.zeros((I, I))
    i = np.arange(I - 1)
    A[i + 1, i] += left
    A[i, i] -= left
    A[i, i + 1] += right
    A[i + 1, i + 1] -= right
    return torch.linalg.matrix_exp(torch.from_numpy(A * dT)).numpy()


def _coarse_step(P, cdf):
    m = P @ np.diff(cdf)
    m[m <= 1e-10] = 0.0
    c = np.concatenate([[0.0], np.cumsum(m)])
    return np.minimum(c / c[-1], 1.0)


def _quantiles(e, F, p):
    """Both one-sided quantiles of the piecewise linear CDF F at the levels p."""
    a = np.searchsorted(F, p, side="left")
    b = np.searchsorted(F, p, side="right") - 1
    hit = F[np.minimum(a, len(F) - 1)] == p
    k = np.clip(a, 1, len(F) - 1)
    span = F[k] - F[k - 1]
    t = (p - F[k - 1]) / np.where(span > 0.0, span, 1.0)
    inner = e[k - 1] + t * (e[k] - e[k - 1])
    inner = np.clip(inner, np.nextafter(e[k - 1], np.inf), np.nextafter(e[k], -np.inf))
    return np.where(hit, e[np.minimum(a, len(F) - 1)], inner), np.where(hit, e[b], inner)


def _pool(q):
    """Pool adjacent violators, equal weights."""
    sums, counts = [], []
    for v in q:
        s, c = float(v), 1
        while sums and sums[-1] * c > s * counts[-1]:
            s, c = sums.pop() + s, counts.pop() + c
        sums.append(s)
        counts.append(c)
    return np.repeat(np.array(sums) / np.array(counts), counts)


def _iterate64(name, e, a, b, c):
    """J(a, b, c) on CDFs at the edges e: the four iterators."""
    if name == "quantile":
        p = np.unique(np.concatenate([a, b, c]))
        (am, ap), (bm, bp), (cm, cp) = (_quantiles(e, F, p) for F in (a, b, c))
        q = np.stack([bm + (am - cm), bp + (ap - cp)], 1).reshape(-1)[1:-1]
        lev = np.repeat(p, 2)[1:-1]
        q = _pool(q)
        x = e[1:-1]
        j = np.searchsorted(q, x, side="right") - 1
        k, nxt = np.clip(j, 0, len(q) - 1), np.clip(j + 1, 0, len(q) - 1)
        span = q[nxt] - q[k]
        v = lev[k] + np.where(span > 0.0, (x - q[k]) / np.where(span > 0.0, span, 1.0), 0.0) * (lev[nxt] - lev[k])
        v = np.where(j < 0, 0.0, v)
        return np.concatenate([[0.0], np.clip(v, 0.0, 1.0), [1.0]])
    a, b, c = (np.diff(v) for v in (a, b, c))
    if name == "add":
        r = np.maximum(a + b - c, 0.0)
    elif name == "mult":
        r = np.where(c > 0.0, a * (b / np.where(c > 0.0, c, 1.0)), 0.0)
    else:
        u, v, w = np.sqrt(b * c).sum(), np.sqrt(b * a).sum(), np.sqrt(c * a).sum()
        r = ((u + 2.0 * u * w - v) / (1.0 + w) * np.sqrt(a) + np.sqrt(b) - (u + v) / (1.0 + w) * np.sqrt(c)) ** 2
    if not r.sum() > 0.0:
        r = b
    r = np.cumsum(r)
    return np.concatenate([[0.0], np.minimum(r[:-1] / r[-1], 1.0), [1.0]])


def _sweep64(P, e, name, rho0, fine, coarse):
    rho = [rho0]
    for n in range(len(fine) if name else coarse):
        a = _coarse_step(P, rho[-1])
        rho.append(_iterate64(name, e, a, fine[n], coarse[n]) if name else a)
    return rho


def _parareal64(case, seed):
    """The whole iteration in 64 bits (quantile matching and iterator, the OU and double-well systems)."""
    f, grid = FAMILIES[case["family"]], _grid(case["family"], case["bins"])
    K, steps, dt, n = case["K"], case["steps"], f["dt"], case["n"]
    e = _edges64(grid).numpy()
    P = _coarse64(_model(case["family"]), grid, steps * dt)
    x0, y0 = (v.double() for v in _initial(case["family"], n, 1, seed, _dtype(case)))
    cdf = lambda x: _restrict64(x.reshape(-1, n), grid)[1].cpu().numpy()
    rho0 = cdf(x0)[0]
    rho = _sweep64(P, e, None, rho0, None, K)
    prior_x, prior_y, prior = [x0] * K, [y0] * K, [rho0] * K
    for _ in range(case["iters"]):
        xs = [x0] + [_match64(prior_x[m], grid, torch.from_numpy(prior[m]).to(DEV), torch.from_numpy(rho[m + 1]).to(DEV))
                     for m in range(K - 1)]
        ys = [y0] + prior_y[:K - 1]
        start = cdf(torch.stack(xs))
        x, y = _propagate64(case["family"], torch.stack(xs), torch.stack(ys), steps, dt, seed)
        fine = cdf(x)
        rho = _sweep64(P, e, "quantile", rho0, fine, [_coarse_step(P, c) for c in start])
        prior_x, prior_y, prior = list(x), list(y), list(fine)
    return {"rho": torch.from_numpy(np.stack(rho)), "x": x, "y": y}


def _tangent64(case, seed):
    """X_T, Y_T [n] and their derivatives [5][n] with respect to (lambda, beta, eps, x0, y0)."""
    f = FAMILIES[case["family"]]
    lam, beta, eps, dt, S = f["lam"], f["beta"], f["eps"], case["dt"], case["steps"]
    x, y = _initial(case["family"], case["n"], 1, seed, torch.float32)
    x, y = x.double().reshape(-1), y.double().reshape(-1)
    dx, dy = (torch.zeros(5, x.numel(), dtype=torch.float64, device=DEV) for _ in range(2))
    dx[3], dy[4] = 1.0, 1.0
    rel, sx, sy = dt / eps, math.sqrt(2.0 * dt / beta), math.sqrt(2.0 * dt / eps)
    ou = case["family"] == "ou"
    for s in range(case["K"]):
        noise = _Noise(x.numel(), 1, 1, seed, s)
        for m in range(S):
            z = [v.reshape(-1) for v in noise(m)]
            nx, ny = sx * z[0], sy * z[1]
            sg = -1.0 if ou else 1.0
            grad = (x if ou else x ** 3 - x) + sg * lam * y
            slope = 1.0 if ou else (3.0 * x * x - 1.0)
            ndx = dx * (1.0 - dt * slope) - (sg * lam * dt) * dy
            ndx[0] -= sg * dt * y
            ndx[1] -= nx * (0.5 / beta)
            ndy = dy * (1.0 - rel) + rel * dx
            ndy[2] += (y - x) * (rel / eps) - ny * (0.5 / eps)
            x, y = x - grad * dt + nx, y - (y - x) * rel + ny
            dx, dy = ndx, ndy
    return x, y, dx, dy


def _reweight64(x, grid, prior, target):
    """Weights rho'_i / rhobar_i / n of one slice, the target mass the prior does not support moved
    half to the nearest supported bin on each side."""
    rb, rt = np.diff(prior.cpu().numpy()), np.diff(target.cpu().numpy())
    sup = np.flatnonzero(rb > 0.0)
    rn = np.where(rb > 0.0, rt, 0.0)
    for i in np.flatnonzero((rb <= 0.0) & (rt > 0.0)):
        k = np.searchsorted(sup, i)
        if 0 < k < len(sup):
            rn[sup[k - 1]] += 0.5 * rt[i]
            rn[sup[k]] += 0.5 * rt[i]
        else:
            rn[sup[min(k, len(sup) - 1)]] += rt[i]
    r = torch.from_numpy(np.where(rb > 0.0, rn / np.where(rb > 0.0, rb, 1.0), 0.0)).to(x.device)
    return r[_bins64(x, grid)] / x.numel()


def exact(case, seed):
    kind = case["kind"]
    if kind == "parareal":
        # a large ensemble takes too long in 64 bits; the resampled ones are chosen by integers,
        # and the chemical system's trajectories part at its saddle
        if case["n"] * case["K"] * case["steps"] * case["iters"] > 2e9 or case["matching"] != "quantile" \
                or case["family"] == "chem":
            return None
        return _parareal64(case, seed)
    if kind == "fine":
        grid = _grid(case["family"], case["bins"])
        if case["n"] * case["slices"] * case["steps"] * (1 + case["d"]) / 2 > 1.6e10:
            return None
        x, y = (v.double() for v in _later(case["family"], case["n"], case["slices"], case["d"], seed, _dtype(case)))
        if case["match"]:
            prior = _restrict64(x, grid)[1]
            target = _target(case["family"], case["n"], case["slices"], case["bins"], seed)
            x = torch.stack([_match64(x[i], grid, prior[i], target[i]) for i in range(len(x))])
        start = _restrict64(x, grid)[1]
        x, y = _propagate64(case["family"], x, y, case["steps"], FAMILIES[case["family"]]["dt"], seed)
        return {"x": x, "y": y, "counts_start": None, "cdf_start": start, "counts_end": None,
                "cdf_end": _restrict64(x, grid)[1]}
    if kind == "adjoint":
        if case["K"] * case["steps"] * max(case["n"], 1 << 17) > 1.6e9:
            return None
        x, y, dx, dy = _tangent64(case, seed)
        n = x.numel()
        if case["observable"] == "quantile":
            # the derivative is that of the particle holding a rank: no value of its own in 64 bits
            r = [max(1, math.ceil((j + 0.5) / 512 * n)) - 1 for j in range(512)]
            return {"quantile": x.sort()[0][torch.tensor(r, device=DEV)], "grad": None, "index": None}
        g = 2.0 / n * x * dx
        if case["observable"] == "second_moment":
            return {"value": (x * x).mean(), "grad": g[:3].sum(1)}
        return {"x": x, "y": y, "loss": (x * x).mean(), "theta_grad": g[:3].sum(1), "x0_grad": g[3], "y0_grad": g[4]}
    if kind == "batch":
        return None   # a whole run of many problems: their layers are cases of their own
    if kind == "transport":
        grid = _grid("double_well", case["bins"])
        x, _ = _later("double_well", case["n"], case["slices"], 1, seed, _dtype(case))
        prior = _restrict64(x, grid)[1]
        target = _target("double_well", case["n"], case["slices"], case["bins"], seed)
        return {"counts": None, "cdf": prior,
                "x": torch.stack([_match64(x[i].double(), grid, prior[i], target[i]) for i in range(len(x))])}
    if kind == "resample":
        grid = _grid("double_well", case["bins"])
        x, _ = _later("double_well", case["n"], case["slices"], case["d"], seed, _dtype(case))
        prior = _restrict64(x, grid)[1]
        target = _target("double_well", case["n"], case["slices"], case["bins"], seed)
        w = torch.stack([_reweight64(x[i].double(), grid, prior[i], target[i]) for i in range(len(x))])
        cdf = torch.zeros_like(prior)
        for i in range(len(x)):
            c = torch.bincount(_bins64(x[i].double(), grid), weights=w[i], minlength=grid.bins).cumsum(0)
            cdf[i, 1:] = c / c[-1]
        return {"w": w, "index": None, "x": None, "y": None, "cdf": cdf}
    if kind == "moments":
        x, _ = _later("double_well", case["n"], case["slices"], 1, seed, _dtype(case))
        w = None
        if case["weighted"]:
            w = torch.rand(*x.shape, generator=_gen(seed + 1), device=DEV, dtype=torch.float64)
            w = w / w.sum(1, keepdim=True)
        out = torch.empty(case["slices"], case["order"], dtype=torch.float64)
        for i in range(case["slices"]):
            v = x[i].double()
            for q in range(case["order"]):
                t = v ** (q + 1)
                out[i, q] = (t * w[i]).sum() if w is not None else t.mean()
        return {"moments": out}
    if kind == "fp_parareal":
        grid = L.Grid(case["bins"], -12.0, 6.0)
        e = _edges64(grid).numpy()
        F, C = (_coarse64(m, grid, 0.2) for m in _fp_models(case))
        rho0 = _fp_start(case, seed).cpu().numpy()
        rho = _sweep64(C, e, None, rho0, None, case["K"])
        for _ in range(case["iters"]):
            old = rho[:-1]
            rho = _sweep64(C, e, case["iterator"], rho0, [_coarse_step(F, v) for v in old],
                           [_coarse_step(C, v) for v in old])
        return {"rho": torch.from_numpy(np.stack(rho))}
    P = _coarse64(_model(case["family"]), _grid(case["family"], case["bins"]), _coarse_dT(case, seed))
    return {"P": torch.from_numpy(P)}
