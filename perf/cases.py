"""The work that users of this framework have it do, as cases to be timed.

A case is a dict of plain values.  ``kind`` says which public entry points a
pass goes through:

* ``run``: one sampling stride of a simulation, ``Lattice.step(steps)`` and
  ``Lattice.diag``, as the break-up driver and the calibration loop make it;
* ``batch``: ``Batch.step(steps)`` over many uneven ligaments, then the
  diagnostics and the density of every box;
* ``adjoint``: ``autograd.rollout`` of a ligament, its neck energy, and the
  gradient with respect to the initial density, G and tau;
* ``snapshot``: a new density from the caller's device tensor, a few steps,
  and the populations, density and velocity read back into device tensors.

Single- and half-precision runs return their series in the precision of the
run; the stored populations come as the run stores them.
"""

import math

import numpy as np
import torch

from paper_1905_09554_gb300 import autograd, lbm

# Coexistence densities of the flat interface per (operator, G): the end
# points of the initial tanh profile.
COEX = {("srt", -5.5): (2.306809, 0.104103), ("mrt", -5.5): (2.248703, 0.056949),
        ("srt", -5.3): (2.161682, 0.121367), ("mrt", -5.3): (2.10895, 0.078116)}
NP = {"f64": np.float64, "f32": np.float32, "f16": np.float16, "bf16": np.float16, "f16l": np.float16,
      "bf16l": np.float16}
TORCH = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16,
         "f16l": torch.float16, "bf16l": torch.bfloat16}
SIZE = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2, "f16l": 2, "bf16l": 2}


def _case(name, kind, nx, ny, nz, steps, storage="f32", coll="srt", rule="paper", tau=1.0, G=-5.5, G2=0.0, R0=0.0,
          eps=0.05, waves=1, boxes=1, every=0):
    return {"name": name, "kind": kind, "nx": nx, "ny": ny, "nz": nz, "steps": steps, "storage": storage,
            "coll": coll, "rule": rule, "tau": tau, "G": G, "G2": G2, "R0": R0 or min(nx, ny) / 4.0, "eps": eps,
            "waves": waves, "boxes": boxes, "every": every}


def listed():
    return [
        # the plain FP64 ligament that everything else is compared with, the smallest run: launches count
        _case("f64_srt_32x32x64", "run", 32, 32, 64, 50, "f64"),
        # a small FP32 ligament sampled every 5 steps on its way to break-up: latency and read-back count
        _case("f32_srt_64x64x144", "run", 64, 64, 144, 5),
        # the sharp-interface ligament R0 = 64 that the benchmark quotes, diagnostics every 50 steps
        _case("f32_srt_256x256x575", "run", 256, 256, 575, 50),
        # the sharp-interface sweep's FP64 MRT run at R0 = 32 (shear rates from tau = 1, the others 1)
        _case("f64_mrt_128x128x288", "run", 128, 128, 288, 10, "f64", "mrt", "shear"),
        # the precision form: R0 = 64, MRT, FP16 deviations from each cell's own density
        _case("f16l_mrt_256x256x575", "run", 256, 256, 575, 20, "f16l", "mrt", "shear"),
        # BF16 deviations from one reference density in a box with odd sides, off tau = 1
        _case("bf16_srt_97x85x131", "run", 97, 85, 131, 20, "bf16", "srt", "paper", 0.9),
        # the paper's own runs: Table 1's SRT ligament R0 = 42 and Table 2's MRT ligament R0 = 56 (the largest)
        _case("f32_srt_288x288x768_paper", "run", 288, 288, 768, 40, "f32", "srt", "paper", 0.83053, -5.3, R0=42,
              eps=0.1, waves=2),
        _case("f32_mrt_384x384x1024_paper", "run", 384, 384, 1024, 20, "f32", "mrt", "paper", 0.84575, -5.3, R0=56,
              eps=0.1, waves=2),
        # 64 uneven ligaments, R0 in {8, 12, 16}, kR0 uniform on [0.2, 1)
        _case("f32_batch64", "batch", 0, 0, 0, 50, R0=8.0, eps=0.03, boxes=64),
        # the differentiable form: 500 steps, checkpoints every 23, and the whole backward pass
        _case("f32_adjoint_64x64x180", "adjoint", 64, 64, 180, 500, R0=16.0, every=23),
        # the two-belt force at the same equation of state (surface tension set apart from it)
        _case("f32_twobelt_128x128x288", "run", 128, 128, 288, 10, "f32", "srt", "paper", 1.0, -7.0, 1.5),
        # a caller's own density stepped once and read back whole on the device
        _case("f64_snapshot_80x72x200", "snapshot", 80, 72, 200, 1, "f64", "srt", "paper", 0.9),
    ]


def draw(rng):
    """One more case of the listed ranges."""
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["run"] * 7 + ["batch", "adjoint", "snapshot"])
    coll = rng.choice(["srt", "mrt"])
    tau = rng.choice([1.0, 1.0, round(rng.uniform(0.65, 1.15), 4)])
    G = rng.choice([-5.5, -5.5, -5.3])
    c = dict(coll=coll, tau=tau, G=G, rule=rng.choice(["shear", "paper", "paper"]), eps=rng.choice([1 / 30, 0.05, 0.1]))
    if kind == "batch":
        c = dict(c, nx=0, ny=0, nz=0, steps=log(4, 60), storage=rng.choice(["f32", "f32", "f64"]),
                 boxes=log(2, 64), R0=8.0)
        if c["storage"] == "f64":
            c["steps"] = min(c["steps"], 12)
    elif kind == "adjoint":
        n = log(20, 64)
        c = dict(c, coll="srt", nx=n, ny=n + rng.randint(-3, 3), nz=log(24, 180), steps=log(20, 300),
                 storage="f32")
        c["every"] = max(1, round(math.sqrt(c["steps"])))
    else:
        small = kind == "snapshot"
        n = log(24, 120 if small else 300)
        nx = n if rng.random() < 0.5 else n + rng.randint(-7, 7)
        ny = n if rng.random() < 0.5 else n + rng.randint(-7, 7)
        nz = max(16, int(n * rng.uniform(1.0, 3.0)))
        storage = "f64" if small else rng.choice(["f32"] * 4 + ["f64"] * 2 + ["f16l", "bf16l", "f16", "bf16"])
        steps = rng.randint(1, 3) if small else log(2, 60)
        while nx * ny * nz * steps * (6 if storage == "f64" else 1) > 384 * 384 * 1024 * 15 and steps > 1:
            steps = max(1, steps // 2)
        c = dict(c, nx=nx, ny=ny, nz=nz, steps=steps, storage=storage)
        if not small and storage in ("f32", "f64") and rng.random() < 0.1:
            c.update(G=-7.0, G2=1.5, steps=min(steps, 8))
        if c["storage"] in ("f32", "f64") and coll == "mrt" and rng.random() < 0.15:
            c["rule"] = "general"
    got = _case("", kind, **c)
    del got["name"]
    return got


# ------------------------------------------------------------------- inputs
def _rates(c):
    """The 19 MRT rates in moment order; None for SRT."""
    if c["coll"] == "srt":
        return None
    s = [1.0] * 19
    if c["rule"] == "general":  # every moment at its own rate
        s = [0.8 + 0.04 * ((7 * k) % 19) for k in range(19)]
    for k in (9, 11, 13, 14, 15):
        s[k] = 1.0 / c["tau"]
    if c["rule"] == "paper":
        s[1] = 1.0 / c["tau"]
    return s


def _coex(c):
    return COEX[(c["coll"], -5.5 if c["G2"] else c["G"])]


def _density(nx, ny, nz, c, seed, R0):
    """Perturbed ligament along z with per-cell Gaussian noise, float64, on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    kw = dict(dtype=torch.float64, device="cuda")
    z = torch.arange(nz, **kw)[:, None, None]
    y = torch.arange(ny, **kw)[None, :, None] - 0.5 * (ny - 1)
    x = torch.arange(nx, **kw)[None, None, :] - 0.5 * (nx - 1)
    rl, rv = _coex(c)
    R = R0 * (1.0 + c["eps"] * torch.cos(2.0 * math.pi * c["waves"] * z / nz))
    rho = rv + 0.5 * (rl - rv) * (1.0 - torch.tanh((torch.sqrt(x * x + y * y) - R) / 2.0))
    return rho.add_(torch.randn((nz, ny, nx), generator=g, **kw), alpha=1e-3)


def _boxes(c):
    """(nx, ny, nz, R0) of the batch: R0 in {8, 12, 16}, kR0 uniform on [0.2, 1), box 4R0 x 4R0 x round(2 pi R0 / kR0)."""
    u = np.random.RandomState(c["boxes"]).random_sample((c["boxes"], 2))
    got = []
    for a, b in u:
        R0 = (8, 12, 16)[min(2, int(3 * a))]
        got.append((4 * R0, 4 * R0, int(round(2 * math.pi * R0 / (0.2 + 0.8 * b))), float(R0)))
    return got


def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        dims = _boxes(c)
        B = lbm.Batch([d[:3] for d in dims], G=c["G"], tau=c["tau"], collision=c["coll"], rates=_rates(c),
                      storage=c["storage"])
        for k, (v, d) in enumerate(zip(B.boxes, dims)):
            v.set_density(_density(*d[:3], c, seed + 1000 * k, d[3]))
        rho = [torch.empty(d[2], d[1], d[0], dtype=torch.float64, device="cuda") for d in dims]
        return {"case": c, "B": B, "rho": rho}
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    rho0 = _density(nx, ny, nz, c, seed, c["R0"])
    if c["kind"] == "adjoint":
        return {"case": c, "rho0": rho0.float().requires_grad_(True),
                "G": torch.tensor(c["G"], dtype=torch.float64, requires_grad=True),
                "tau": torch.tensor(c["tau"], dtype=torch.float64, requires_grad=True)}
    L = lbm.Lattice(nx, ny, nz, G=c["G"], G2=c["G2"], tau=c["tau"], collision=c["coll"], rates=_rates(c),
                    storage=c["storage"])
    if c["kind"] == "snapshot":
        kw = dict(dtype=torch.float64, device="cuda")
        return {"case": c, "L": L, "rho0": rho0, "f": torch.empty((19, nz, ny, nx), **kw),
                "rho": torch.empty((nz, ny, nx), **kw), "u": torch.empty((3, nz, ny, nx), **kw)}
    L.set_density(rho0)
    return {"case": c, "L": L}


# --------------------------------------------------------------------- runs
def run(state):
    c = state["case"]
    rl, rv = _coex(c)
    if c["kind"] == "batch":
        B, t = state["B"], NP[c["storage"]]
        B.step(c["steps"])
        d = [v.diag(rl, rv, raise_nonfinite=False) for v in B.boxes]
        for v, r in zip(B.boxes, state["rho"]):
            v.moments_device(r)
        return {"rho": torch.cat([r.reshape(-1).to(TORCH[c["storage"]]) for r in state["rho"]]),
                "area": np.concatenate([x["area_z"] for x in d]).astype(t),
                "maxrho": np.concatenate([x["maxrho_z"] for x in d]).astype(t)}
    if c["kind"] == "adjoint":
        rho0, G, tau = state["rho0"], state["G"], state["tau"]
        rho0.grad = G.grad = tau.grad = None
        rho = autograd.rollout(rho0, G, tau, c["steps"], every=c["every"], storage=c["storage"])
        autograd.neck_energy(rho, rl, rv).backward()
        return {"rho": rho.detach().float(), "d_rho0": rho0.grad, "d_G": G.grad.float(), "d_tau": tau.grad.float()}
    L = state["L"]
    if c["kind"] == "snapshot":
        L.set_density(state["rho0"])
        L.step(c["steps"])
        L.get_populations(state["f"])
        L.moments_device(state["rho"], *state["u"])
        return {"f": state["f"], "rho": state["rho"], "u": state["u"]}
    L.step(c["steps"])
    d = L.diag(rl, rv, raise_nonfinite=False)
    t = NP[c["storage"]]
    f = L.stored_populations().view(TORCH[c["storage"]]).view(19, c["nz"], c["ny"], c["nx"])
    return {"f": f, "mass": np.asarray(d["mass"], np.float64 if c["storage"] == "f64" else np.float32),
            "area": d["area_z"].astype(t), "maxrho": d["maxrho_z"].astype(t)}


def work(case):
    c = case
    cells = sum(d[0] * d[1] * d[2] for d in _boxes(c)) if c["kind"] == "batch" else c["nx"] * c["ny"] * c["nz"]
    per = 19 * SIZE[c["storage"]] + (4 if c["storage"].endswith("l") else 0)
    # the state in and the state out once; about 250 operations a cell and step (force 50, moments 40,
    # collision 150), 450 more for the 92 neighbours of the second belt, three times a step for its adjoint
    flops = cells * c["steps"] * (250.0 + (450.0 if c["G2"] else 0.0))
    if c["kind"] == "adjoint":
        return {"bytes": cells * 12.0, "flops": 4 * flops}
    if c["kind"] == "batch":
        return {"bytes": cells * (2.0 * per + SIZE[c["storage"]]), "flops": flops}
    if c["kind"] == "snapshot":
        return {"bytes": cells * (8.0 + 8.0 * 23), "flops": flops}
    return {"bytes": cells * 2.0 * per, "flops": flops}


# ------------------------------------------------- the same in 64 bits, plain torch
C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
     (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
     (0, -1, 1)]
W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
P8 = {1: 4 / 45, 2: 1 / 21, 3: 2 / 105, 4: 5 / 504, 5: 1 / 315, 6: 1 / 630, 8: 1 / 5040}  # second belt, by |e|^2


def _basis():
    """The 19 orthogonal moments (d'Humieres) as rows over the velocities."""
    rows = []
    for x, y, z in C:
        s = x * x + y * y + z * z
        rows.append([1, 19 * s - 30, (21 * s * s - 53 * s + 24) / 2, x, (5 * s - 9) * x, y, (5 * s - 9) * y, z,
                     (5 * s - 9) * z, 3 * x * x - s, (3 * s - 5) * (3 * x * x - s), y * y - z * z,
                     (3 * s - 5) * (y * y - z * z), x * y, y * z, x * z, (y * y - z * z) * x, (z * z - x * x) * y,
                     (x * x - y * y) * z])
    return torch.tensor(rows, dtype=torch.float64, device="cuda").T.contiguous()


def _at(a, c):
    """a at x + c."""
    return torch.roll(a, (-c[2], -c[1], -c[0]), (0, 1, 2))


def _force(rho, G, G2):
    psi = 1.0 - torch.exp(-rho)
    S = [torch.zeros_like(rho) for _ in range(3)]
    belts = [(c, G * w) for c, w in zip(C, W) if c != (0, 0, 0)]
    if G2:
        r = range(-2, 3)
        belts += [((x, y, z), G2 * P8[x * x + y * y + z * z] / 3) for x in r for y in r for z in r
                  if x * x + y * y + z * z in P8]
    for c, k in belts:
        p = _at(psi, c) * k
        S = [s + d * p if d else s for s, d in zip(S, c)]
    return [-psi * s for s in S]


def _collide(f, F, tau, rates, M):
    """Post-collision populations of a stack of planes."""
    rho = f.sum(0)
    j = [sum(c[k] * f[q] for q, c in enumerate(C) if c[k]) for k in range(3)]
    shift = tau if rates is None else 0.5
    u = [(j[k] + shift * F[k]) / rho for k in range(3)]
    uu = 1.0 - 1.5 * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2])
    feq, S = [], []
    for c, w in zip(C, W):
        cu = sum(c[k] * u[k] for k in range(3) if c[k]) if any(c) else torch.zeros_like(rho)
        feq.append(w * rho * (uu + 3.0 * cu + 4.5 * cu * cu))
        if rates is not None:
            S.append(w * sum((3.0 * (c[k] - u[k]) + 9.0 * cu * c[k]) * F[k] for k in range(3)))
    feq = torch.stack(feq)
    if rates is None:
        return f + (feq - f) / tau
    s = torch.tensor(rates, dtype=torch.float64, device=f.device)[:, None]
    d = s * (M @ (f - feq).reshape(19, -1)) - (1.0 - 0.5 * s) * (M @ torch.stack(S).reshape(19, -1))
    # the conserved rows do not depend on their rates: nothing for rho, the force for the momentum
    d[0] = 0.0
    for k, q in enumerate((3, 5, 7)):
        d[q] = -F[k].reshape(-1)
    return f - (M.T @ (d / (M * M).sum(1)[:, None])).reshape(f.shape)


def _run64(rho0, c, steps):
    """Populations and the density before the last step."""
    M, rates = _basis(), _rates(c)
    f = torch.stack([w * rho0 for w in W])
    nz = rho0.shape[0]
    slab = max(1, int(4e6 // rho0[0].numel()))
    rho = rho0
    for _ in range(steps):
        rho = f.sum(0)
        F = _force(rho, c["G"], c["G2"])
        for a in range(0, nz, slab):
            b = min(nz, a + slab)
            f[:, a:b] = _collide(f[:, a:b], [v[a:b] for v in F], c["tau"], rates, M)
        for q in range(1, 19):
            f[q] = torch.roll(f[q], C[q][::-1], (0, 1, 2))
    return f, rho


def _slices(rho, c):
    rl, rv = _coex(c)
    return ((rho - rv) / (rl - rv)).clamp_(0.0, 1.0).sum((1, 2)), rho.amax((1, 2))


def _adjoint64(rho0, c):
    n, (rl, rv) = c["steps"], _coex(c)
    G = torch.tensor(c["G"], dtype=torch.float64, device="cuda", requires_grad=True)
    tau = torch.tensor(c["tau"], dtype=torch.float64, device="cuda", requires_grad=True)
    w = torch.tensor(W, dtype=torch.float64, device="cuda")[:, None, None, None]

    def step(f):
        g = _collide(f, _force(f.sum(0), G, 0.0), tau, None, None)
        return torch.stack([torch.roll(g[q], C[q][::-1], (0, 1, 2)) for q in range(19)])

    states = [w * rho0]
    with torch.no_grad():
        for _ in range(n):
            states.append(step(states[-1]))
    rho = states.pop().sum(0).requires_grad_(True)
    R = torch.sqrt(((rho - rv) / (rl - rv)).sum((1, 2)) / math.pi)
    lam, = torch.autograd.grad(((R - R.mean()) ** 2).mean(), rho)
    lam, dG, dt = lam.expand(19, *lam.shape), 0.0, 0.0
    while states:
        f = states.pop().requires_grad_(True)
        lam, a, b = torch.autograd.grad(step(f), (f, G, tau), lam)
        dG, dt = dG + a, dt + b
    return {"rho": rho.detach(), "d_rho0": (w * lam).sum(0), "d_G": dG, "d_tau": dt}


def exact(case, seed):
    c = case
    if c["kind"] == "batch":
        rho, area, top = [], [], []
        for k, d in enumerate(_boxes(c)):
            r = _run64(_density(*d[:3], c, seed + 1000 * k, d[3]), c, c["steps"])[0].sum(0)
            a, m = _slices(r, c)
            rho.append(r.reshape(-1)), area.append(a), top.append(m)
        return {"rho": torch.cat(rho), "area": torch.cat(area), "maxrho": torch.cat(top)}
    rho0 = _density(c["nx"], c["ny"], c["nz"], c, seed, c["R0"])
    if c["kind"] == "adjoint":
        return _adjoint64(rho0.float().double(), c)
    f, before = _run64(rho0, c, c["steps"])
    rho = f.sum(0)
    if c["kind"] == "snapshot":
        F = _force(rho, c["G"], c["G2"])
        j = [sum(v[k] * f[q] for q, v in enumerate(C) if v[k]) for k in range(3)]
        return {"f": f, "rho": rho, "u": torch.stack([(j[k] + 0.5 * F[k]) / rho for k in range(3)])}
    area, top = _slices(rho, c)
    if SIZE[c["storage"]] == 2:  # stored: deviations from rest at density 1, or at the density before the step
        ref = before if c["storage"].endswith("l") else 1.0
        for q in range(19):
            f[q] -= W[q] * ref
    return {"f": f, "mass": rho.sum(), "area": area, "maxrho": top}
