"""The calls whose time matters to a user of the library, as measurable cases.

A case is a dict of plain values.  ``prepare`` builds what a program has in
hand before the call (initial densities, a handle, batch or server, output
buffers), ``run`` is one call sequence through the public Python binding, and
``exact`` gives the same outputs in 64 bits from plain torch.

Kinds of case:

* ``single``: one simulation.  A pass sets the initial densities, advances
  ``steps`` time steps and reads the densities and the FP64 mass, all in
  device memory (``distributions`` also exports every population).  ``tune``
  > 0: the handle was tuned once, as a program does before a long run.
* ``batch``: a (F, k) sweep of equal grids in one batch; a pass advances the
  whole batch and reads every instance's densities.  A batch cannot be set
  back to t = 0, so a repeated pass goes on from where the last one ended.
* ``serving``: a stream of uneven requests to a resident server, from host
  densities to host results.
* ``study``: the point-source convergence study (FP64 requests, host to host).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1007_3109_gb300 import binding as B
from paper_1007_3109_gb300 import inputs, studies

D_GS = (0.1, 0.05)  # diffusion constants of every Gray-Scott workload


def _single(name, **kw):
    case = dict(kind="single", lattice="D2Q9", model="gray_scott", precision="fp32", inplace=False, track_mass=False,
                tune=0, distributions=False)
    case.update(kw)
    return dict(name=name, **case)


def listed():
    return [
        # a probe or a parameter fit on a small grid: launches and latency count (one species, FP64, tau = 1)
        _single("decay_128_fp64", model="linear", precision="fp64", nx=128, ny=128, steps=100, distributions=True),
        # the 512^2 validation run in FP64 (bit-reproducible arithmetic), fields exported for analysis
        _single("gs_512_fp64", precision="fp64", nx=512, ny=512, steps=50, distributions=True),
        # the same run in FP32 on a tuned handle: the state stays in L2
        _single("gs_512_fp32", nx=512, ny=512, steps=200, tune=10, distributions=True),
        # a handle as it comes, on a ragged domain, with the mass tracked every step
        _single("gs_1531x1021_fp32", nx=1531, ny=1021, steps=50, track_mass=True),
        # the large pattern-formation run, tuned, called 20 steps at a time
        _single("gs_8192_fp32", nx=8192, ny=8192, steps=20, tune=3),
        # five-velocity lattice, large grid
        _single("gs_4096_d2q5_fp32", lattice="D2Q5", nx=4096, ny=4096, steps=40, tune=3),
        # 16-bit storage of the deviations, large grid
        _single("gs_4096_bf16", precision="fp32_bf16dev", nx=4096, ny=4096, steps=40, tune=3),
        # four species with a mass-action network of ten reaction steps
        _single("gs2x_2048_fp32", model="network", nx=2048, ny=2048, steps=20, tune=3),
        # phase-diagram sweep: 256 instances of 256^2, FP32 and 16-bit deviation storage
        dict(name="sweep_256_fp32", kind="batch", lattice="D2Q9", precision="fp32", n=16, nx=256, ny=256, steps=400),
        dict(name="sweep_256_bf16", kind="batch", lattice="D2Q9", precision="fp32_bf16dev", n=16, nx=256, ny=256,
             steps=400),
        # continuous batching of uneven requests (any side, three diffusion scales)
        dict(name="serving_fp32", kind="serving", precision="fp32", requests=12, side_min=64, side_max=1024,
             steps_min=500, steps_max=2000),
        # truncation-error study: point sources over a (D, kappa) grid at equal physical time
        dict(name="study_fp64", kind="study", n_d=8, n_kappa=8, side=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["single", "batch", "serving", "study"], [12, 4, 2, 1])[0]
    if kind == "batch":
        precision = rng.choice(["fp32", "fp32", "fp32_bf16dev", "fp32_fp16dev"])
        nx, ny = _log_int(rng, 64, 512), _log_int(rng, 64, 512)
        if precision != "fp32":
            nx = (nx + 3) // 4 * 4
        n = rng.randint(3, 16)
        return dict(kind="batch", lattice=rng.choice(["D2Q9", "D2Q9", "D2Q5"]), precision=precision, n=n, nx=nx, ny=ny,
                    steps=rng.randint(20, 100))
    if kind == "serving":
        lo = _log_int(rng, 64, 256)
        return dict(kind="serving", precision="fp32", requests=rng.randint(4, 12), side_min=lo,
                    side_max=rng.randint(lo + 32, 900), steps_min=rng.randint(200, 500),
                    steps_max=rng.randint(600, 1800))
    if kind == "study":
        return dict(kind="study", n_d=rng.randint(3, 8), n_kappa=rng.randint(2, 8), side=rng.randint(50, 100))
    model = rng.choices(["gray_scott", "linear", "network"], [6, 2, 1])[0]
    precision = rng.choices(["fp32", "fp64", "fp32_bf16dev", "fp32_fp16dev"], [6, 2, 2, 1])[0]
    if model == "network" and precision not in ("fp32", "fp64"):
        precision = "fp32"
    inplace = precision == "fp32" and rng.random() < 0.15
    top = 8192 if precision != "fp64" and model != "network" else 1024 if precision == "fp64" else 2048
    nx, ny = _log_int(rng, 64, top), _log_int(rng, 64, top)
    if precision in ("fp32_bf16dev", "fp32_fp16dev"):
        nx = (nx + 3) // 4 * 4
    most = 3e7 if precision == "fp64" else 1.2e9  # site-steps
    steps = max(10, min(_log_int(rng, 10, 400), int(most / (nx * ny))))
    return dict(kind="single", lattice=rng.choice(["D2Q9", "D2Q9", "D2Q5"]), model=model, precision=precision,
                inplace=inplace, track_mass=rng.random() < 0.25, tune=rng.choice([0, 3]), nx=nx, ny=ny, steps=steps,
                distributions=nx * ny <= 1 << 20 and rng.random() < 0.5)


# -- inputs --------------------------------------------------------------------

def _tau(D):
    return 3.0 * D + 0.5


def _spots(seed, nx, ny, gen_key, device):
    """u = 1, v = 0 with random 16 x 16 squares (u = 0.5, v = 0.25), one per 512 x 512 sites and at
    least one, plus 1 % uniform noise on every site; (2, ny, nx) float64."""
    g = torch.Generator(device=device)
    g.manual_seed((int(seed) * 7 + gen_key) & 0x7FFFFFFF)
    rho = (torch.rand((2, ny, nx), generator=g, device=device, dtype=torch.float64) - 0.5) * 0.02
    rho[0] += 1.0
    n = max(1, nx * ny // (512 * 512))
    rs = np.random.RandomState((int(seed) * 7 + gen_key) & 0x7FFFFFFF)
    side = min(16, nx, ny)
    for x, y in zip(rs.randint(0, nx - side + 1, n).tolist(), rs.randint(0, ny - side + 1, n).tolist()):
        rho[0, y:y + side, x:x + side] -= 0.5
        rho[1, y:y + side, x:x + side] += 0.25
    return rho


def _single_rho0(case, seed, device):
    nx, ny = case["nx"], case["ny"]
    if case["model"] == "linear":  # cosine mode plus noise (the decay workload's recipe)
        g = torch.Generator(device=device)
        g.manual_seed(int(seed) & 0x7FFFFFFF)
        x = torch.arange(nx, dtype=torch.float64, device=device)
        phase = 2 * math.pi * np.random.RandomState(int(seed) & 0x7FFFFFFF).rand()
        noise = (torch.rand((1, ny, nx), generator=g, device=device, dtype=torch.float64) - 0.5) * 2e-6
        return (1.0 + 0.1 * torch.cos(2 * math.pi * x / nx + phase))[None, None, :] + noise
    if case["model"] == "network":
        return torch.cat([_spots(seed, nx, ny, 0, device), _spots(seed, nx, ny, 3, device)])
    return _spots(seed, nx, ny, 0, device)


def _single_physics(case):
    """(taus, make_config keywords) of a single run."""
    if case["model"] == "linear":
        return [_tau(1.0 / 6.0)], dict(reaction="linear", kappa=1e-3)
    if case["model"] == "network":
        return [_tau(d) for d in D_GS * 2], dict(reaction="mass_action", network=inputs.coupled_gs_network())
    return [_tau(d) for d in D_GS], dict(reaction="gray_scott", F=0.037, k=0.06)


def _batch_fk(case):
    return inputs.sweep_params(case["n"])


def _batch_rho0(case, seed, i, device):
    """The noisy centred square of instance i."""
    nx, ny = case["nx"], case["ny"]
    g = torch.Generator(device=device)
    g.manual_seed((int(seed) * 65537 + i) & 0x7FFFFFFF)
    rho = (torch.rand((2, ny, nx), generator=g, device=device, dtype=torch.float64) - 0.5) * 0.02
    rho[0] += 1.0
    h = min(20, nx // 2, ny // 2)
    rho[0, ny // 2 - h:ny // 2 + h, nx // 2 - h:nx // 2 + h] -= 0.5
    rho[1, ny // 2 - h:ny // 2 + h, nx // 2 - h:nx // 2 + h] += 0.25
    return rho


def _requests(case, seed):
    """Serving requests [(side, scale, steps)]: sizes and step counts of the case (the same for every
    seed, spread evenly over the ranges), so that equal cases do equal work."""
    n = case["requests"]
    out = []
    for j in range(n):
        a = (j + 0.5) / n
        side = int(case["side_min"] + a * (case["side_max"] - case["side_min"]))
        steps = int(case["steps_min"] + ((5 * j + 2) % n + 0.5) / n * (case["steps_max"] - case["steps_min"]))
        out.append((side, (1, 2, 4)[j % 3], steps))
    order = np.random.RandomState(1238).permutation(n)
    return [out[j] for j in order]


def _request_rho0(side, seed, j):
    """Noisy square in host memory."""
    rs = np.random.RandomState((int(seed) * 131 + j) & 0x7FFFFFFF)
    rho = (rs.random_sample((2, side, side)) - 0.5) * 0.02
    rho[0] += 1.0
    c = side // 2
    rho[0, c - 20:c + 20, c - 20:c + 20] -= 0.5
    rho[1, c - 20:c + 20, c - 20:c + 20] += 0.25
    return rho


def _study_runs(case, seed):
    """[(config, rho0, steps)]: point sources of random place and mass, D log-spaced over the paper's
    range, kappa linear, D t = 8."""
    rs = np.random.RandomState(int(seed) & 0x7FFFFFFF)
    L, runs = case["side"], []
    for kappa in np.linspace(0.01, 0.033, case["n_kappa"]):
        for D in np.geomspace(0.02, 0.16, case["n_d"]):
            steps = max(1, int(round(8.0 / D)))
            cfg = dict(lattice="D2Q9", nspecies=2, nx=L, ny=L, tau=[_tau(float(D))] * 2, reaction="linear",
                       kappa=float(kappa), precision="fp64")
            rho0 = np.zeros((2, L, L))
            rho0[0, rs.randint(L), rs.randint(L)] = 0.5 + rs.rand()
            runs.append((cfg, rho0, steps))
    return runs


# -- the measured calls ----------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "single":
        taus, kw = _single_physics(case)
        S, nx, ny = len(taus), case["nx"], case["ny"]
        rho0 = _single_rho0(case, seed, "cuda")
        sim = B.Simulation(case["lattice"], S, nx, ny, taus, precision=case["precision"],
                           track_mass=case["track_mass"], inplace=case["inplace"], **kw)
        if case["tune"]:
            sim.init(rho0)
            sim.autotune(case["tune"])
        state = dict(kind=kind, sim=sim, rho0=rho0, steps=case["steps"], rho=torch.empty_like(rho0),
                     mass=torch.empty(S, dtype=torch.float64, device="cuda"), f=None)
        if case["distributions"]:
            state["f"] = torch.empty((S, sim.Q, ny, nx), dtype=torch.float64, device="cuda")
        return state
    if kind == "batch":
        F, k = _batch_fk(case)
        taus = [_tau(d) for d in D_GS]
        batch = B.Batch([dict(lattice=case["lattice"], nspecies=2, nx=case["nx"], ny=case["ny"], tau=taus,
                              reaction="gray_scott", F=float(F[i]), k=float(k[i]), precision=case["precision"])
                         for i in range(len(F))])
        for i in range(len(F)):
            batch.init(i, _batch_rho0(case, seed, i, "cuda"))
            torch.cuda.synchronize()
        return dict(kind=kind, batch=batch, n=len(F), steps=case["steps"],
                    rho=torch.empty((len(F), 2, case["ny"], case["nx"]), dtype=torch.float64, device="cuda"),
                    mass=torch.empty((len(F), 2), dtype=torch.float64, device="cuda"))
    if kind == "serving":
        server = B.Server(8 << 30, precision=case["precision"])
        reqs = []
        for j, (side, scale, steps) in enumerate(_requests(case, seed)):
            cfg = dict(lattice="D2Q9", nspecies=2, nx=side, ny=side, tau=[_tau(d * scale) for d in D_GS],
                       reaction="gray_scott", F=0.04, k=0.06, precision=case["precision"])
            reqs.append((_request_rho0(side, seed, j), steps, cfg))
        return dict(kind=kind, server=server, requests=reqs)
    return dict(kind=kind, runs=_study_runs(case, seed))


def run(state):
    kind = state["kind"]
    if kind == "single":
        sim = state["sim"]
        sim.init(state["rho0"])
        sim.step(state["steps"])
        B.lb_rd_moments(sim.h, state["rho"], state["mass"])
        out = {"rho": state["rho"], "mass": state["mass"]}
        if state["f"] is not None:
            B.lb_rd_get_distributions(sim.h, state["f"])
            out["f"] = state["f"]
        return out
    if kind == "batch":
        batch = state["batch"]
        batch.step(state["steps"])
        for i in range(state["n"]):
            B.lb_rd_batch_moments(batch.b, i, state["rho"][i], state["mass"][i])
        return {"rho": state["rho"], "mass": state["mass"]}
    if kind == "serving":
        server = state["server"]
        tickets = [server.submit(rho0, steps, **cfg) for rho0, steps, cfg in state["requests"]]
        results = [server.result(t) for t in tickets]
        return {"rho": [r[0] for r in results], "mass": np.stack([r[1] for r in results])}
    results, _, _ = studies.run_requests(state["runs"])
    return {"rho": np.stack([r[0] for r in results]), "mass": np.stack([r[1] for r in results])}


def _Q(lattice):
    return 9 if lattice == "D2Q9" else 5


def _flops(Q, S, network=False):
    """Floating-point operations of one site and step: the density sums, the relaxation with source
    (one fused multiply-add per population) and the reaction."""
    return S * ((Q - 1) + 2 * Q + 8) + (60 if network else 8)


def _state_bytes(Q, S, precision):
    return S * (8 * Q if precision == "fp64" else 4 * Q if precision == "fp32" else 4 + 2 * (Q - 1))


def work(case):
    kind = case["kind"]
    if kind == "single":
        S = len(_single_physics(case)[0])
        Q, sites = _Q(case["lattice"]), case["nx"] * case["ny"]
        # initial densities in, the state and the densities out (and the populations where exported)
        per = 16 * S + _state_bytes(Q, S, case["precision"]) + (8 * S * Q if case["distributions"] else 0)
        return {"bytes": sites * per, "flops": sites * case["steps"] * _flops(Q, S, case["model"] == "network")}
    if kind == "batch":
        Q, sites = _Q(case["lattice"]), case["n"] ** 2 * case["nx"] * case["ny"]
        return {"bytes": sites * (2 * _state_bytes(Q, 2, case["precision"]) + 16),
                "flops": sites * case["steps"] * _flops(Q, 2)}
    if kind == "serving":
        reqs = _requests(case, 0)
        return {"bytes": sum(32 * s * s for s, _, _ in reqs),
                "flops": sum(s * s * n * _flops(9, 2) for s, _, n in reqs)}
    runs = _study_runs(case, 0)
    sites = case["side"] ** 2
    return {"bytes": len(runs) * sites * 32, "flops": sum(n for _, _, n in runs) * sites * _flops(9, 2)}


# -- the same outputs in 64 bits, without the library ------------------------------

_E9 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]


def _evolve(rho0, taus, steps, lattice, source):
    """f after ``steps`` steps from equilibrium at rho0 (..., S, ny, nx): pre-collision populations
    (..., S, Q, ny, nx); ``source(rho)`` gives R of rho's shape."""
    e = _E9 if lattice == "D2Q9" else _E9[:5]
    w = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4 if lattice == "D2Q9" else [1 / 3] + [1 / 6] * 4
    dev = rho0.device
    wt = torch.tensor(w, dtype=torch.float64, device=dev)[:, None, None]
    om = 1.0 / torch.tensor(taus, dtype=torch.float64, device=dev)[..., None, None, None]
    f = wt * rho0.unsqueeze(-3)
    for _ in range(steps):
        f = _collide(f, wt, om, source)
        for i in range(1, len(e)):
            f[..., i, :, :] = torch.roll(f[..., i, :, :], (e[i][1], e[i][0]), (-2, -1))
    return f, wt, om


def _collide(f, wt, om, source):
    rho = f.sum(-3)
    R = source(rho)
    post = torch.addcmul(f, om, wt * rho.unsqueeze(-3) - f)
    return post.add_(wt * R.unsqueeze(-3))


def _gs_source(F, k):
    def source(rho):
        u, v = rho[..., 0, :, :], rho[..., 1, :, :]
        uvv = u * v * v
        return torch.stack([-uvv + F * (1 - u), uvv - (F + k) * v], -3)
    return source


def _network_source(rates, order, change):
    def source(rho):
        R = torch.zeros_like(rho)
        for r, a, nu in zip(rates, order, change):
            p = torch.full_like(rho[0], r)
            for j, n in enumerate(a):
                for _ in range(n):
                    p = p * rho[j]
            for s, c in enumerate(nu):
                if c:
                    R[s] += c * p
        return R
    return source


def _host(rho):
    return rho.cpu().numpy()


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if kind == "single":
        taus, kw = _single_physics(case)
        if case["model"] == "linear":
            def source(rho):
                return -kw["kappa"] * rho
        elif case["model"] == "network":
            source = _network_source(*kw["network"])
        else:
            source = _gs_source(kw["F"], kw["k"])
        f, wt, om = _evolve(_single_rho0(case, seed, dev), taus, case["steps"], case["lattice"], source)
        rho = f.sum(-3)
        out = {"rho": rho, "mass": rho.sum((-2, -1))}
        if case["distributions"]:
            out["f"] = _collide(f, wt, om, source)
        return out
    if kind == "batch":
        F, k = _batch_fk(case)
        rho, mass = [], []
        for i in range(0, len(F), 64):
            j = range(i, min(i + 64, len(F)))
            rho0 = torch.stack([_batch_rho0(case, seed, m, dev) for m in j])
            Fj, kj = (torch.tensor(np.asarray(a)[list(j)], device=dev)[:, None, None] for a in (F, k))
            f, _, _ = _evolve(rho0, [_tau(d) for d in D_GS], case["steps"], case["lattice"], _gs_source(Fj, kj))
            rho.append(f.sum(-3))
            mass.append(rho[-1].sum((-2, -1)))
        return {"rho": torch.cat(rho), "mass": torch.cat(mass)}
    if kind == "serving":
        rho = []
        for j, (side, scale, steps) in enumerate(_requests(case, seed)):
            rho0 = torch.from_numpy(_request_rho0(side, seed, j)).to(dev)
            f, _, _ = _evolve(rho0, [_tau(d * scale) for d in D_GS], steps, "D2Q9", _gs_source(0.04, 0.06))
            rho.append(_host(f.sum(-3)))
        return {"rho": rho, "mass": np.stack([r.sum((1, 2)) for r in rho])}
    rho = []
    runs = _study_runs(case, seed)
    for steps in sorted({n for _, _, n in runs}):  # one D per step count: its runs go together
        at = [j for j, r in enumerate(runs) if r[2] == steps]
        rho0 = torch.from_numpy(np.stack([runs[j][1] for j in at])).to(dev)
        kappa = torch.tensor([runs[j][0]["kappa"] for j in at], dtype=torch.float64, device=dev)[:, None, None]

        def source(r):
            return torch.stack([-kappa * r[:, 0], kappa * r[:, 0]], 1)
        f, _, _ = _evolve(rho0, runs[at[0]][0]["tau"], steps, "D2Q9", source)
        rho += list(zip(at, f.sum(-3)))
    rho = np.stack([_host(r) for _, r in sorted(rho, key=lambda a: a[0])])
    return {"rho": rho, "mass": rho.sum((2, 3))}
