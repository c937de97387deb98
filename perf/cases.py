"""What a user of the library runs, as cases that can be timed and checked.

A case is a dict of plain values.  `kind` says which entry point it calls:

  step       clot_species_step: `steps` species steps of a 2D channel or 3D duct
  ensemble   Ensemble.run: `steps` steps of `channels` uneven 2D channels
  split      clot_eta_solve, then clot_reaction_step: the reaction half of a
             split in which the caller transports the species itself
  eta        clot_eta_solve from a zero start, as when a run begins or resumes
  surrogate  clot_species_step_surrogate: steps whose reaction takes the network
  train      clot_surrogate_train: `steps` Adam steps of the network

A pass advances its state, as a user's time loop does: the next pass goes on
from where the last one stopped.  `exact` repeats a first pass in 64 bits with
plain torch, on the 32-bit inputs that `prepare` hands to the library.
"""
import functools
import math

import numpy as np
import torch

import paper_2304_09180_gb300 as clot

SPECIES = ("Pmu", "Pma", "Pba", "Pbse", "ADP", "S1", "S2", "E1", "E2", "S1b", "S2b", "E1b", "E2b", "C1", "C2")
PMU, PMA, PBA, PBSE, ADP, S1, S2, E1, E2, S1B, S2B, E1B, E2B, C1, C2 = range(15)
MOBILE = (PMU, PMA, ADP, S1, S2, E1, E2)
REACTING = tuple(s for s in range(15) if s != ADP)
UM = 1e-3  # one micrometre in mm

# The paper's parameters (mm, s, nmol, platelets); the numerics are the library's usual ones.
PARAMS = dict(
    Pmax=6.67e7, P0=2.5e5, kadh=3.3212e-8, kcohPmax=1.0e4, eta_t=0.1, eta_star=0.4, p_diam=3.0e-3, L_eta=6.0e-3,
    k_adp=0.34, adp_star=2.0e-3, k_e2=0.5, e2_star=1.0e-6, A_hat=2.0e-8, sigma_tf=6.0, sigma_dt=0.25,
    D_P=2.5e-5, D_adp=5.0e-4, D_chem=5.0e-5, N1=2700.0, N2=2000.0, N_A=6.02214076e14,
    kC0p=8.95e3, kC0m=1.0, kC0cat=1.15, kC1p=1.03e5, kC1m=1.0, kC1cat=30.0, kC2p=1.73e4, kC2m=1.0, kC2cat=0.23,
    kS1p=5.7e4, kS1m=0.17, kE1p=1.0e4, kE1m=2.5e-2, kS2p=1.0e4, kS2m=5.9, kE2p=1.0e4, kE2m=5.9,
    S1_plasma=1.7e-4, S2_plasma=1.4e-3, E0_wall=1.5e-7,
    M_rxn=2, limiter=1, flags=0, eta_tol=1e-6, eta_atol=1e-6, eta_maxit=100000, wait_s=0.0, kI=0.0, I_in=0.0,
    S1_ref=1.7e-4, S2_ref=1.4e-3)
FLAGS = {"euler": 0, "second": clot.HEUN | clot.STRANG, "lagged": clot.WALL_LAGGED}
TRAIN_BATCH = 16384


def listed():
    return [
        # the paper's thrombosis mesh, one step a call: a flow solver that hands over new fluxes each step
        dict(name="paper_mesh_one_step", kind="step", dim=2, nx=128, ny=32, nz=1, h=1.875, shear=1000, state="primed",
             order="euler", deviation=False, flow="deflected", M=2, steps=1),
        # a small channel from plasma on, the usual first run
        dict(name="channel_200x40_plasma", kind="step", dim=2, nx=200, ny=40, nz=1, h=1.5, shear=1000, state="plasma",
             order="euler", deviation=False, flow="parallel", M=2, steps=20),
        # a mesh of the convergence study: second order in time, deviation form
        dict(name="study_320x80_second", kind="step", dim=2, nx=320, ny=80, nz=1, h=0.375, shear=1000, state="plasma",
             order="second", deviation=True, flow="parallel", M=2, steps=20),
        # the fine 2D channel with a clot: the eta solve on fine cells
        dict(name="channel_1024x256_primed", kind="step", dim=2, nx=1024, ny=256, nz=1, h=0.25, shear=1500,
             state="primed", order="euler", deviation=False, flow="parallel", M=2, steps=10),
        # the 3D benchmark duct, from plasma on and with a clot
        dict(name="duct_512x128x128_plasma", kind="step", dim=3, nx=512, ny=128, nz=128, h=1.5, shear=1000,
             state="plasma", order="euler", deviation=False, flow="parallel", M=2, steps=8),
        dict(name="duct_512x128x128_primed", kind="step", dim=3, nx=512, ny=128, nz=128, h=1.5, shear=1000,
             state="primed", order="euler", deviation=False, flow="parallel", M=2, steps=8),
        # a duct of odd extents in a flow with all three components, the wall exchange placed as in the paper
        dict(name="duct_203x67x45_ragged", kind="step", dim=3, nx=203, ny=67, nz=45, h=1.5, shear=1000,
             state="primed", order="lagged", deviation=False, flow="deflected", M=2, steps=8),
        # many independent channels, the parameter-sweep workload
        dict(name="ensemble_256", kind="ensemble", channels=256, least=8, most=64, sizes=0, state="plasma", steps=60),
        # the library's reaction beside the caller's own transport
        dict(name="split_256x128x64", kind="split", dim=3, nx=256, ny=128, nz=64, h=1.5, shear=1000, state="primed",
             M=2),
        # a run that resumes without its eta
        dict(name="eta_512x128x128_cold", kind="eta", dim=3, nx=512, ny=128, nz=128, h=1.5, shear=1000,
             state="primed"),
        # stiff reaction substeps taken by the network
        dict(name="surrogate_256x128x64", kind="surrogate", dim=3, nx=256, ny=128, nz=64, h=1.5, shear=1000,
             state="primed", M=32, steps=4),
        # the network's training
        dict(name="train_65536", kind="train", rows=65536, steps=20),
    ]


def _spread(rng, lo, hi):
    """A whole number of [lo, hi], even over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("step2", "step2", "step2", "step3", "step3", "step3", "ensemble", "split", "eta", "surrogate",
                       "train"))
    if kind == "step2":
        ny = _spread(rng, 10, 256)
        nx = min(1024, int(ny * rng.uniform(2.5, 5.5)))
        return dict(kind="step", dim=2, nx=nx, ny=ny, nz=1, h=round(rng.uniform(0.25, 2.5), 3),
                    shear=rng.choice((500, 1000, 1500, 2000)), state=rng.choice(("plasma", "primed")),
                    order=rng.choice(("euler", "euler", "second", "lagged")), deviation=rng.random() < 0.25,
                    flow=rng.choice(("parallel", "deflected")), M=rng.choice((2, 2, 4)), steps=rng.choice((1, 5, 20)))
    if kind == "ensemble":
        return dict(kind="ensemble", channels=_spread(rng, 4, 256), least=8, most=rng.randint(12, 64),
                    sizes=rng.randrange(1000), state=rng.choice(("plasma", "primed")), steps=rng.choice((12, 30)))
    if kind == "train":
        return dict(kind="train", rows=TRAIN_BATCH * rng.randint(2, 8), steps=rng.randint(5, 30))
    ny, nz = _spread(rng, 16, 128), _spread(rng, 16, 128)
    nx = _spread(rng, 48, 512)
    if rng.random() < 0.6:
        nx -= nx % 4
    case = dict(kind=kind, dim=3, nx=nx, ny=ny, nz=nz, h=1.5, shear=rng.choice((500, 1000, 2000)), state="primed")
    if kind == "step3":
        case.update(kind="step", state=rng.choice(("plasma", "primed")),
                    order=rng.choice(("euler", "euler", "second", "lagged")), deviation=rng.random() < 0.25,
                    flow=rng.choice(("parallel", "deflected")), M=2, steps=rng.choice((1, 4, 8)))
    elif kind == "split":
        case.update(M=rng.choice((2, 4)))
    elif kind == "surrogate":
        case.update(nx=min(nx, 256), M=rng.choice((2, 8, 32)), steps=rng.choice((1, 4)))
    return case


# ------------------------------------------------------------------ inputs

def _desc(case):
    h, nx = case["h"] * UM, case["nx"]
    lo, hi = case.get("patch") or ((1 / 3, 2 / 3) if case["dim"] == 2 else (3 / 8, 5 / 8))
    hz = h if case["dim"] == 3 else 1.0
    return dict(dim=case["dim"], nx=nx, ny=case["ny"], nz=case["nz"], hx=h, hy=h, hz=hz, inj_x0=lo * nx * h,
                inj_x1=hi * nx * h, inj_z0=0.0, inj_z1=case["nz"] * hz if case["dim"] == 3 else 0.0,
                p_diam=PARAMS["p_diam"])


def _fluxes(desc, shear, flow):
    """Face fluxes (numpy, 64 bits) of a parabolic channel or duct flow of that
    floor shear; "deflected" adds a divergence-free roll between the walls."""
    nx, ny, nz, h, hz = desc["nx"], desc["ny"], desc["nz"], desc["hy"], desc["hz"]
    H = ny * h
    yf, xf = np.arange(ny + 1) * h, np.arange(nx + 1) / nx
    bump_y = (yf / H) * (1 - yf / H)
    if desc["dim"] == 2:
        psi = shear * (yf * yf / 2 - yf ** 3 / (3 * H))                    # stream function of the flow
        psi = np.broadcast_to(psi[:, None], (ny + 1, nx + 1)).copy()
        if flow == "deflected":
            psi += 0.2 * shear * H * H * bump_y[:, None] ** 2 * np.sin(3 * math.pi * xf)[None, :]
        return dict(fx=((psi[1:] - psi[:-1]) * hz).reshape(-1), fy=(-(psi[:, 1:] - psi[:, :-1]) * hz).reshape(-1),
                    fz=None)
    W = nz * h
    zf = np.arange(nz + 1) * h
    prim = lambda s, S: 4 * (S * s * s / 2 - s ** 3 / 3) / (S * S)         # of 4 s (S - s) / S^2
    iy, iz = np.diff(prim(yf, H)), np.diff(prim(zf, W))
    U = shear * H / 4
    fx = np.broadcast_to((U * iz[:, None] * iy[None, :])[:, :, None], (nz, ny, nx + 1)).copy()
    fy, fz = np.zeros((nz, ny + 1, nx)), np.zeros((nz + 1, ny, nx))
    if flow == "deflected":
        wave = np.sin(3 * math.pi * xf)
        a = 0.2 * U * H * bump_y ** 2                                      # roll in the x-y planes
        fx += iz[:, None, None] * np.diff(a)[None, :, None] * wave[None, None, :]
        fy -= iz[:, None, None] * a[None, :, None] * np.diff(wave)[None, None, :]
        b = 0.2 * U * W * ((zf / W) * (1 - zf / W)) ** 2                   # and in the x-z planes
        fx += np.diff(b)[:, None, None] * iy[None, :, None] * wave[None, None, :]
        fz -= b[:, None, None] * iy[None, :, None] * np.diff(wave)[None, None, :]
    return dict(fx=fx.reshape(-1), fy=fy.reshape(-1), fz=fz.reshape(-1))


def _dt(desc, fluxes):
    """Courant number 0.5, capped by explicit diffusion and by the reaction substep."""
    V = desc["hx"] * desc["hy"] * desc["hz"]
    worst = 0.0  # largest outflow of a cell over its volume is bounded by the sum over the axes
    for f in (fluxes["fx"], fluxes["fy"], fluxes["fz"]):
        if f is not None:
            worst += float(np.max(np.abs(f))) / V
    diff = 2 * PARAMS["D_adp"] * desc["dim"] / desc["hx"] ** 2
    return min(0.5 / worst, 0.2 * desc["hx"] ** 2 / PARAMS["D_adp"], 1e-4, 0.9 / (worst + diff))


def _shape_y(n, K):
    r = np.abs((np.arange(n) + 0.5) / n * 2 - 1)
    return K * r ** 18 * (1 - r)


def _inlet(desc):
    """Marginated platelets, plasma chemicals: [nz ny] Dirichlet values."""
    two = desc["dim"] == 2
    K, beta = (330.0 if two else 547.0), math.gamma(19) * math.gamma(2) / math.gamma(21)
    shape = 1 + _shape_y(desc["ny"], K)[None, :] + (0 if two else _shape_y(desc["nz"], K)[:, None])
    pmu = PARAMS["P0"] / (1 + (1 if two else 2) * K * beta) * shape.reshape(-1)
    return dict(pmu_in=pmu, s1_in=np.full(pmu.shape, PARAMS["S1_plasma"]), s2_in=np.full(pmu.shape, PARAMS["S2_plasma"]))


def _patch(desc):
    """Injury rectangle (i0, i1, k0, k1) and the number of adhesion rows."""
    x = (np.arange(desc["nx"]) + 0.5) * desc["hx"]
    i = np.nonzero((x >= desc["inj_x0"]) & (x <= desc["inj_x1"]))[0]
    rows = int(np.sum((np.arange(desc["ny"]) + 0.5) * desc["hy"] <= desc["p_diam"]))
    return int(i[0]), int(i[-1]), 0, desc["nz"] - 1, rows


def _state(desc, seed, state):
    """c [15, ncell], e0, c0 in 32 bits on the GPU: plasma with 1 % noise, or
    the same with a clot on the injury ("primed")."""
    gen = torch.Generator("cuda").manual_seed(seed)
    nx, ny, nz = desc["nx"], desc["ny"], desc["nz"]
    n, f32 = nx * ny * nz, dict(dtype=torch.float32, device="cuda")
    noise = lambda *s: 1 + 0.01 * torch.randn(*s, generator=gen, **f32)
    u = lambda lo, hi: lo + (hi - lo) * torch.rand(n, generator=gen, **f32)
    c = torch.zeros(15, n, **f32)
    pmu = torch.as_tensor(_inlet(desc)["pmu_in"], **f32)
    c[PMU] = pmu[:, None].expand(ny * nz, nx).reshape(-1) * noise(n)
    c[S1], c[S2] = PARAMS["S1_plasma"] * noise(n), PARAMS["S2_plasma"] * noise(n)
    i0, i1, k0, k1, _ = _patch(desc)
    ninj = (i1 - i0 + 1) * (k1 - k0 + 1)
    e0, c0 = PARAMS["E0_wall"] * noise(ninj), torch.zeros(ninj, **f32)
    if state == "plasma":
        return c, e0, c0
    x = (torch.arange(nx, **f32) + 0.5) * desc["hx"] - 0.5 * (desc["inj_x0"] + desc["inj_x1"])
    y = (torch.arange(ny, **f32) + 0.5) * desc["hy"]
    bump = torch.exp(-(x / (20 * UM)) ** 2)[None, None, :] * torch.exp(-(y / (8 * UM)) ** 2)[None, :, None]
    if desc["dim"] == 3:
        z = (torch.arange(nz, **f32) + 0.5 - nz / 2) * desc["hz"]
        bump = bump * torch.exp(-(z / (40 * UM)) ** 2)[:, None, None]
    floor = (torch.arange(ny, device="cuda") < 2)[None, :, None].expand(nz, ny, nx).reshape(-1)
    bump = bump.expand(nz, ny, nx).reshape(-1)
    bound = 0.9 * PARAMS["Pmax"] * bump * noise(n)
    c[PBSE] = torch.where(floor, 0.8 * bound, torch.zeros_like(bound))
    c[PBA] = torch.where(floor, 0.2 * bound, bound)
    c[PMA] = 0.05 * PARAMS["P0"] * bump * u(1.0, 1.1)
    c[PMU] *= 1 - 0.5 * bump
    cap1, cap2 = (PARAMS[k] / PARAMS["N_A"] * (c[PBA] + c[PBSE]) for k in ("N1", "N2"))
    c[C1], c[C2] = 0.02 * cap2 * u(0.5, 1.5), 0.02 * cap2 * u(0.5, 1.5)
    c[S1B], c[E1B] = cap1 * u(0.05, 0.3), cap1 * u(0.01, 0.1)
    c[S2B], c[E2B] = cap2 * u(0.05, 0.3), cap2 * u(0.01, 0.1)
    c[E1], c[E2], c[ADP] = 1e-7 * bump * u(0.5, 1.5), 5e-7 * bump * u(0.5, 1.5), 1e-3 * bump * u(0.5, 1.5)
    return c, 0.8 * e0, 0.2 * e0


def _fields(mesh, desc, seed, state):
    c, e0, c0 = _state(desc, seed, state)
    n, pitch, zeros = mesh.ncell, mesh.pitch, functools.partial(torch.zeros, dtype=torch.float32, device="cuda")
    full = zeros(15, pitch)
    full[:, :n] = c
    slots = int(PARAMS["sigma_tf"] / PARAMS["sigma_dt"] + 0.5) + 1
    return clot.Fields(full, e0, c0, zeros(n), zeros(n), zeros(slots, n), zeros(n))


def _padded(t):
    """t with its rows filled up to a multiple of 32 by zeros, the library's pitch."""
    return torch.nn.functional.pad(t, (0, -t.shape[-1] % 32))


def _mesh_inputs(case):
    desc = _desc(case)
    fluxes = _fluxes(desc, case["shear"], case.get("flow", "parallel"))
    return desc, fluxes, _inlet(desc), _dt(desc, fluxes)


def _step_flags(case):
    return FLAGS[case["order"]] | (clot.DEVIATION if case["deviation"] else 0)


@functools.lru_cache(maxsize=4)
def _channels(channels, least, most, sizes):
    """Cases of the ensemble's channels: uneven lengths, shears and patches."""
    rng = np.random.default_rng(sizes)
    out = []
    for _ in range(channels):
        nx, shear, frac = 8 * int(rng.integers(least, most + 1)), rng.uniform(500, 2000), rng.uniform(0.1, 0.5)
        out.append(dict(dim=2, nx=nx, ny=nx // 4, nz=1, h=1.5, shear=float(shear), patch=(0.5 - frac / 2, 0.5 + frac / 2)))
    return out


def _weights(seed):
    """A network as training leaves it: outputs of order 0.1."""
    rng = np.random.default_rng(seed + 77)
    W1 = rng.standard_normal((32, 64)) * math.sqrt(2 / 31) * (np.arange(32) < 31)[:, None]
    W2 = rng.standard_normal((64, 64)) * math.sqrt(2 / 64)
    W3 = rng.standard_normal((64, 16)) * 0.01 * (np.arange(16) < 14)[None, :]
    small = lambda n: 0.01 * rng.standard_normal(n)
    return np.concatenate([W1.ravel(), small(64), W2.ravel(), small(64), W3.ravel(), small(16) * (np.arange(16) < 14)])


def _scale():
    p = PARAMS
    cap1, cap2 = p["N1"] / p["N_A"] * p["Pmax"], p["N2"] / p["N_A"] * p["Pmax"]
    return [p["Pmax"]] * 4 + [p["adp_star"], p["S1_plasma"], p["S2_plasma"], 1e-8, 1e-8, cap1, cap2, cap1, cap2, cap2, cap2]


def _training_rows(n, seed):
    """Features and targets of random reaction states, 32 bits on the GPU."""
    gen = torch.Generator("cuda").manual_seed(seed)
    u = lambda lo, hi: lo + (hi - lo) * torch.rand(n, generator=gen, dtype=torch.float64, device="cuda")
    lu = lambda lo, hi: torch.exp(u(math.log(lo), math.log(hi)))
    p, c = PARAMS, torch.zeros(15, n, dtype=torch.float64, device="cuda")
    bound, split = p["Pmax"] * u(0, 0.9) * (u(0, 1) < 0.7), u(0, 1)
    c[PBSE], c[PBA], c[PMU], c[PMA] = bound * split, bound * (1 - split), lu(1e4, 2e6), lu(1e2, 1e6)
    c[ADP], c[S1], c[S2] = lu(1e-8, 5e-3), lu(1e-6, 3e-4), lu(1e-5, 2e-3)
    c[E1], c[E2] = lu(1e-12, 1e-6), lu(1e-12, 1e-5)
    cap1, cap2 = p["N1"] / p["N_A"] * bound, p["N2"] / p["N_A"] * bound
    for s, cap in ((S1B, cap1), (E1B, cap1), (S2B, cap2), (E2B, cap2), (C1, 0.5 * cap2), (C2, 0.5 * cap2)):
        c[s] = cap * u(0, 0.2)
    dt, g = 1.5625e-5, _affinity(u(0, 1))
    x, E, rho, floor = _features(c, g, dt)
    dc = _reaction(c, None, None, g, dt / 2, 2, None)[0] - c
    y = (dc - E) / (rho * (E.abs() + floor)).clamp_min(1e-300)
    y = torch.where(rho > 0, y, torch.zeros_like(y)).clamp(-4, 4)[list(REACTING)].T
    return x.float().contiguous(), torch.nn.functional.pad(y, (0, 2)).float().contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        x, y = _training_rows(case["rows"], seed)
        mlp = clot.Mlp(_weights(seed), _scale())
        z = functools.partial(torch.zeros, dtype=torch.float32, device="cuda")
        return dict(kind=kind, case=case, mlp=mlp, m=z(clot.MLP_NPARAM), v=z(clot.MLP_NPARAM), t=0, x=x, y=y,
                    work=z(clot.clot_surrogate_workspace(TRAIN_BATCH)))
    if kind == "ensemble":
        made = [_mesh_inputs(c) for c in _channels(case["channels"], case["least"], case["most"], case["sizes"])]
        ens = clot.Ensemble([m[0] for m in made])
        fields = [_fields(ens.meshes[q], m[0], seed * 1000 + q, case["state"]) for q, m in enumerate(made)]
        flat = {}  # one buffer for all channels, as their owner keeps them
        for name in ("c", "e0", "c0", "eta"):
            own = [getattr(f, name) for f in fields]
            rows = [_padded(t.reshape(-1)) for t in own]
            flat[name] = torch.cat(rows)
            for f, t, part in zip(fields, own, flat[name].split([r.numel() for r in rows])):
                setattr(f, name, part[:t.numel()].view_as(t))
        dev = lambda a: torch.as_tensor(a, dtype=torch.float32, device="cuda")
        args = (fields, [clot.Fluxes(ens.meshes[q], **m[1]) for q, m in enumerate(made)],
                [tuple(dev(m[2][k]) for k in ("pmu_in", "s1_in", "s2_in")) for m in made], [m[3] for m in made], PARAMS)
        ens.tune(*args, trials=3)
        return dict(kind=kind, case=case, ens=ens, args=args, flat=flat)
    desc, fluxes, inlet, dt = _mesh_inputs(case)
    mesh = clot.Mesh(desc)
    s = dict(kind=kind, case=case, mesh=mesh, dt=dt, fields=_fields(mesh, desc, seed, case["state"]),
             params=clot.Params(PARAMS, **inlet, M_rxn=case.get("M", 2), flags=_step_flags(case) if kind == "step" else 0))
    if kind in ("step", "surrogate"):
        s["fluxes"] = clot.Fluxes(mesh, **fluxes)
    if kind == "surrogate":
        s["mlp"] = clot.Mlp(_weights(seed), _scale())
    return s


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "train":
        loss = clot.clot_surrogate_train(s["mlp"], s["m"], s["v"], s["t"], 1e-3, s["x"], s["y"], TRAIN_BATCH,
                                         case["steps"], work=s["work"])
        s["t"] += case["steps"]
        return dict(w=s["mlp"].w, m=s["m"], v=s["v"], loss=loss)
    if kind == "ensemble":
        s["ens"].run(*s["args"], case["steps"])
        return s["flat"]
    mesh, f, prm = s["mesh"], s["fields"], s["params"]
    if kind == "eta":
        f.eta.zero_()
        clot.clot_eta_solve(mesh, f, prm)
        return dict(eta=f.eta)
    if kind == "split":
        clot.clot_eta_solve(mesh, f, prm)
        clot.clot_reaction_step(mesh, f, prm, s["dt"] / case["M"], case["M"])
    elif kind == "surrogate":
        clot.clot_species_step_surrogate(mesh, f, s["fluxes"], prm, s["mlp"], 1e-3, s["dt"], case["steps"])
    else:
        clot.clot_species_step(mesh, f, s["fluxes"], prm, s["dt"], case["steps"])
    return dict(c=f.c.unbind(0), e0=f.e0, c0=f.c0, eta=f.eta)


def work(case):
    """Bytes and operations of one pass.  A step reads and writes each cell's
    15 species once and reads its face fluxes, sigma and eta; a network row
    takes 7168 multiply-adds, three times that in training."""
    kind = case["kind"]
    if kind == "train":
        rows = TRAIN_BATCH * case["steps"]
        return dict(bytes=4.0 * rows * 48, flops=6.0 * rows * 7168)
    if kind == "ensemble":
        cells = sum(c["nx"] * c["ny"] for c in _channels(case["channels"], case["least"], case["most"], case["sizes"]))
        return dict(bytes=4.0 * 34 * cells * case["steps"], flops=600.0 * cells * case["steps"])
    n = case["nx"] * case["ny"] * case["nz"]
    if kind == "eta":
        return dict(bytes=4.0 * 3 * n, flops=30.0 * n)
    if kind == "split":
        return dict(bytes=4.0 * 32 * n, flops=400.0 * case["M"] * n)
    per = 400.0 * (2 if case.get("order") == "second" else 1) + (14336 if kind == "surrogate" else 0)
    return dict(bytes=4.0 * (32 + case["dim"]) * n * case["steps"], flops=per * n * case["steps"])


# ------------------------------------------------------------- in 64 bits

def _affinity(eta):
    p = PARAMS
    cube = lambda v: v ** 3
    g0 = (cube(p["eta_star"]) + cube(1 - p["eta_t"])) / cube(1 - p["eta_t"])
    u = (eta - p["eta_t"]).clamp_min(0)
    return g0 * u ** 3 / (p["eta_star"] ** 3 + u ** 3)


def _hindrance(theta):
    return torch.tanh(math.pi * (1 - theta.clamp(0, 1)))


def _rates(c, H, g):
    """Right-hand side of the cell reactions (no wall exchange)."""
    p, f = PARAMS, torch.zeros_like(c)
    adh = p["kadh"] * H * (p["Pmax"] - c[PBSE]) if H is not None else torch.zeros_like(c[0])
    act = p["k_adp"] * c[ADP] / (p["adp_star"] + c[ADP]) + p["k_e2"] * c[E2] / (p["e2_star"] + c[E2])
    coh = p["kcohPmax"] * g
    f[PMU] = -(adh + act) * c[PMU]
    f[PMA] = -(adh + coh) * c[PMA] + act * c[PMU]
    f[PBA] = coh * c[PMA] - adh * c[PBA]
    f[PBSE] = adh * (c[PMU] + c[PMA] + c[PBA])
    sites, held = c[PBA] + c[PBSE], c[C1] + c[C2]
    free1 = p["N1"] / p["N_A"] * sites - (c[S1B] + c[E1B] + held)
    free2 = p["N2"] / p["N_A"] * sites - (c[S2B] + c[E2B] + held)
    a1 = p["kC1p"] * c[S2B] * c[E1B] - p["kC1m"] * c[C1]
    a2 = p["kC2p"] * c[S1B] * c[E2B] - p["kC2m"] * c[C2]
    cat1, cat2 = p["kC1cat"] * c[C1], p["kC2cat"] * c[C2]
    for fluid, held_, free, name in ((S1, S1B, free1, "S1"), (S2, S2B, free2, "S2"), (E1, E1B, free1, "E1"),
                                     (E2, E2B, free2, "E2")):
        f[held_] = p["k%sp" % name] * free * c[fluid] - p["k%sm" % name] * c[held_]
        f[fluid] = -f[held_]
    f[S1B] -= a2
    f[S2B] -= a1
    f[E1B] += cat1 + cat2 - a1
    f[E2B] += cat1 + cat2 - a2
    f[C1], f[C2] = a1 - cat1, a2 - cat2
    return f


def _wall(desc, s1, w):
    """Flux J of S1 into the injury and the rates of w = (E0, C0)."""
    p, D = PARAMS, PARAMS["D_chem"] / (0.5 * desc["hy"])
    s1w = (D * s1 + p["kC0m"] * w[1]) / (D + p["kC0p"] * w[0])
    J, cat = p["kC0p"] * s1w * w[0] - p["kC0m"] * w[1], p["kC0cat"] * w[1]
    return J, cat, torch.stack((cat - J, J - cat))


def _reaction(c, w, H, g, h, M, where):
    """M RK4 steps of h; where = (desc, cells of the floor faces) couples the wall w = (E0, C0)."""
    def rhs(y, v):
        f = _rates(y, H, g)
        if where is None:
            return f, None
        desc, cells = where
        J, cat, fv = _wall(desc, y[S1, cells], v)
        f[S1, cells] -= J / desc["hy"]
        f[E1, cells] += cat / desc["hy"]
        return f, fv
    go = lambda v, a, k: None if v is None else v if k is None else v + a * k
    for _ in range(M):
        f, fv = rhs(c, w)
        acc, accv = f.clone(), fv
        for a, weight in ((h / 2, 2), (h / 2, 2), (h, 1)):
            f, fv = rhs(c + a * f, go(w, a, fv))
            acc += weight * f
            accv = None if fv is None else accv + weight * fv
        c = c + h / 6 * acc
        w = go(w, h / 6, accv)
    return c, w


def _transport(desc, c, flux, inlet, dt):
    """One explicit transport pass: van Leer faces, hindered platelets."""
    nx, ny, nz = desc["nx"], desc["ny"], desc["nz"]
    p, V, m = PARAMS, desc["hx"] * desc["hy"] * desc["hz"], list(MOBILE)
    c = c.view(15, nz, ny, nx)
    q = c[m]
    D = torch.tensor([p["D_P"], p["D_P"], p["D_adp"]] + [p["D_chem"]] * 4, dtype=c.dtype, device=c.device).view(7, 1, 1, 1)
    others = c[PMA] + c[PBA] + c[PBSE]
    theta = (c[PMU] + others) / p["Pmax"]
    W = _hindrance(theta)
    div = torch.zeros_like(q)
    for axis, (name, h) in enumerate((("fx", desc["hx"]), ("fy", desc["hy"]), ("fz", desc["hz"]))):
        n, d = (nx, ny, nz)[axis], 3 - axis
        if n < 2 and axis:
            continue
        shape = [nz, ny, nx]
        shape[d - 1] += 1
        F = flux[name].view(shape)
        cut = lambda t, lo, hi, dd: t.narrow(dd, lo, hi - lo)
        if n > 1:
            L, R, Fi = cut(q, 0, n - 1, d), cut(q, 1, n, d), cut(F, 1, n, d - 1)
            LL = torch.cat((cut(q, 0, 1, d), cut(q, 0, n - 2, d)), d)
            RR = torch.cat((cut(q, 2, n, d), cut(q, n - 1, n, d)), d)
            pos = Fi >= 0
            U, Dn, UU = torch.where(pos, L, R), torch.where(pos, R, L), torch.where(pos, LL, RR)
            a, b = U - UU, Dn - U
            same = a * b > 0
            face = torch.where(same, U + a * (b / torch.where(same, a + b, torch.ones_like(a))), U)
            del UU, Dn, U, a, b, same, LL, RR
            WL, WR = cut(W, 0, n - 1, d - 1), cut(W, 1, n, d - 1)
            adv, dif = Fi * face, -D * (V / h / h) * (R - L)
            adv[:2] *= torch.where(pos, WR, WL)
            dif[:2] *= torch.minimum(WL, WR)
            phi = adv + dif
            cut(div, 0, n - 1, d).add_(phi)
            cut(div, 1, n, d).sub_(phi)
            del phi, adv, dif, face
        if axis == 0:  # inlet (Dirichlet Pmu, S1, S2) and outlet
            last = q[..., -1] * F[..., -1]
            last[:2] *= W[..., -1]
            div[..., -1] += last
            pmu, s1, s2 = (inlet[k].view(nz, ny) for k in ("pmu_in", "s1_in", "s2_in"))
            Wb = _hindrance((pmu + others[..., 0]) / p["Pmax"])
            cP = q[..., 0]
            cb, out0 = cP.clone(), -F[..., 0]
            cb[0], cb[3], cb[4] = pmu, s1, s2
            out = out0 * cb
            out[:2] *= torch.where(out0 > 0, Wb, W[..., 0])
            dif = 2 * D[..., 0] * (V / h / h) * (cb - cP)
            dif[:2] *= torch.minimum(W[..., 0], Wb)
            div[..., 0] += out - dif
    out = c.clone()
    out[m] = q - dt / V * div
    return out.view(15, -1)


@functools.lru_cache(maxsize=64)
def _modes(n, c):
    """Orthonormal cosine modes of the zero-flux second difference, and c times its eigenvalues."""
    k = torch.arange(n, dtype=torch.float64, device="cuda")
    E = torch.cos(math.pi / n * k[:, None] * (k[None, :] + 0.5)) * math.sqrt(2 / n)
    E[0] /= math.sqrt(2)
    return E, c * (2 - 2 * torch.cos(math.pi * k / n))


def _eta(desc, c):
    """(I - L^2/4 lap) eta = theta_B by cosine transforms."""
    b = ((c[PBA] + c[PBSE]) / PARAMS["Pmax"]).view(desc["nz"], desc["ny"], desc["nx"])
    (Ez, lz), (Ey, ly), (Ex, lx) = (_modes(desc[n], PARAMS["L_eta"] ** 2 / 4 / desc[h] ** 2 if desc[n] > 1 else 0.0)
                                    for n, h in (("nz", "hz"), ("ny", "hy"), ("nx", "hx")))
    t = Ey @ (b @ Ex.T)
    t = (Ez @ t.reshape(desc["nz"], -1)).view_as(b)
    t = t / (1 + lz[:, None, None] + ly[None, :, None] + lx[None, None, :])
    t = (Ez.T @ t.reshape(desc["nz"], -1)).view_as(b)
    return (Ey.T @ (t @ Ex)).reshape(-1)


def _features(c, g, dt):
    """Network features, Euler increments, their relative size and the floors."""
    scale = torch.tensor(_scale(), dtype=c.dtype, device=c.device)[:, None]
    E = dt * _rates(c, None, g)
    rel = E / (c.abs() + 1e-6 * scale)
    r = rel[list(REACTING)]
    x = torch.zeros(c.shape[1], 32, dtype=c.dtype, device=c.device)
    x[:, :15] = torch.log1p(c.clamp_min(0) / scale).T
    x[:, 15], x[:, 16] = g, math.log(dt / 1e-5)
    x[:, 17:31] = (torch.sign(r) * torch.log1p(1e3 * r.abs())).T
    return x, E, r.abs().amax(0), 1e-6 * scale


def _network(w, x):
    at, parts = 0, []
    for shape in ((32, 64), (64,), (64, 64), (64,), (64, 16), (16,)):
        parts.append(w[at:at + math.prod(shape)].view(shape))
        at += math.prod(shape)
    W1, b1, W2, b2, W3, b3 = parts
    gelu = functools.partial(torch.nn.functional.gelu, approximate="tanh")
    return gelu(gelu(x @ W1 + b1) @ W2 + b2) @ W3 + b3


def _surrogate(c, w, H, g, dt, M, where, net):
    """The reaction over dt: the network's increment where it applies, RK4 elsewhere."""
    full, w2 = _reaction(c, w, H, g, dt / M, M, where)
    out = []
    for q in torch.arange(c.shape[1], device=c.device).split(1 << 18):
        y = c[:, q]
        x, E, rho, floor = _features(y, g[q], dt)
        v = torch.zeros_like(y)
        v[list(REACTING)] = _network(net, x)[:, :14].T
        dc = E + rho * v * (E.abs() + floor)
        big = (dc.abs() / (y.abs() + floor)).amax(0) > 1e-3
        out.append(torch.where(big | (H[q] > 0), full[:, q], y + dc))
    return torch.cat(out, 1), w2


def _train_exact(case, seed):
    x, y = (t.double() for t in _training_rows(case["rows"], seed))
    w = torch.as_tensor(_weights(seed), dtype=torch.float32, device="cuda").double()
    m, v, losses = torch.zeros_like(w), torch.zeros_like(w), []
    for t in range(case["steps"]):
        at = t * TRAIN_BATCH % (case["rows"] // TRAIN_BATCH * TRAIN_BATCH)
        w.requires_grad_(True)
        d = (_network(w, x[at:at + TRAIN_BATCH]) - y[at:at + TRAIN_BATCH])[:, :14]
        loss = d.square().mean()
        g, = torch.autograd.grad(loss, w)
        w = w.detach()
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        w = w - 1e-3 * (m / (1 - 0.9 ** (t + 1))) / ((v / (1 - 0.999 ** (t + 1))).sqrt() + 1e-8)
        losses.append(loss.detach())
    return dict(w=w, m=m, v=v, loss=torch.stack(losses))


def _run_exact(kind, case, seed, desc, fluxes, inlet, dt):
    """c, (E0, C0) and eta after one pass."""
    single = lambda a: torch.as_tensor(a, dtype=torch.float32, device="cuda").double()
    c, e0, c0 = (t.double() for t in _state(desc, seed, case["state"]))
    w, flux = torch.stack((e0, c0)), {k: None if v is None else single(v) for k, v in fluxes.items()}
    inlet = {k: single(v) for k, v in inlet.items()}
    i0, i1, k0, k1, rows = _patch(desc)
    nx, ny, nz = desc["nx"], desc["ny"], desc["nz"]
    H = torch.zeros(nz, ny, nx, dtype=torch.float64, device="cuda")
    H[k0:k1 + 1, :rows, i0:i1 + 1] = 1
    H = H.view(-1)
    cells = torch.arange(nx * ny * nz, device="cuda").view(nz, ny, nx)[k0:k1 + 1, 0, i0:i1 + 1].reshape(-1)
    where, order, M, eta = (desc, cells), case.get("order", "euler"), case.get("M", 2), None
    for _ in range(case.get("steps", 1)):
        eta = _eta(desc, c)
        g = _affinity(eta)
        if kind == "eta":
            break
        if kind == "split":
            c, w = _reaction(c, w, H, g, dt / M, M, where)
            continue
        if order == "second":
            c, w = _reaction(c, w, H, g, dt / 2 / M, M, where)
            c2 = _transport(desc, _transport(desc, c, flux, inlet, dt), flux, inlet, dt)
            c[list(MOBILE)] = 0.5 * (c + c2)[list(MOBILE)]
            c, w = _reaction(c, w, H, g, dt / 2 / M, M, where)
            continue
        start = c[S1, cells]
        c = _transport(desc, c, flux, inlet, dt)
        if order == "lagged":
            J, cat, _ = _wall(desc, start, w)
            c[S1, cells] -= dt / desc["hy"] * J
            c[E1, cells] += dt / desc["hy"] * cat
            s1, h = c[S1, cells], dt / M
            for _ in range(M):
                k1_ = _wall(desc, s1, w)[2]
                k2_ = _wall(desc, s1, w + h / 2 * k1_)[2]
                k3_ = _wall(desc, s1, w + h / 2 * k2_)[2]
                w = w + h / 6 * (k1_ + 2 * k2_ + 2 * k3_ + _wall(desc, s1, w + h * k3_)[2])
        where_ = None if order == "lagged" else where
        if kind == "surrogate":
            c, w = _surrogate(c, w, H, g, dt, M, where_, single(_weights(seed)))
        else:
            c, w2 = _reaction(c, w, H, g, dt / M, M, where_)
            w = w if order == "lagged" else w2
    return c, w, eta


def exact(case, seed):
    kind, plasma = case["kind"], case.get("state") == "plasma"
    if kind == "train":
        return _train_exact(case, seed)
    if kind == "ensemble":
        if case["channels"] * case["steps"] > 3000:  # about 6 ms a channel and step
            return None
        flat = dict(c=[], e0=[], c0=[], eta=[])
        for q, ch in enumerate(_channels(case["channels"], case["least"], case["most"], case["sizes"])):
            one = dict(ch, state=case["state"], steps=case["steps"])
            c, w, eta = _run_exact("step", one, seed * 1000 + q, *_mesh_inputs(one))
            for name, t in (("c", c), ("e0", w[0]), ("c0", w[1]), ("eta", eta)):
                flat[name].append(_padded(t).reshape(-1))
        return {name: None if name == "eta" and plasma else torch.cat(t) for name, t in flat.items()}
    c, w, eta = _run_exact(kind, case, seed, *_mesh_inputs(case))
    if kind == "eta":
        return dict(eta=eta)
    # From plasma on, hardly any platelet is bound at first: eta stays below what its solve resolves, and the
    # activated platelets, thrombin and what comes of it below the smallest 32-bit numbers.
    c = [None if plasma and s in (PMA, E2, E2B, C2) else row for s, row in enumerate(_padded(c).unbind(0))]
    return dict(c=c, e0=w[0], c0=w[1], eta=None if plasma else eta)
