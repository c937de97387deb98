"""What the eta solve promises however it is done: max |eta - eta_exact| within
the stopping rule's bound, max(eta_tol max theta_B, eta_atol), down to the
rounding of eta in 32 bits -- from a start far from the solution, at tight and
loose tolerances, for couplings from none to strong, and for the eta a step
corrects from its prediction.  Against the 64-bit solution by cosine transforms."""
import numpy as np
import pytest

import oracle as O
import synthetic as S
from test_gpu_eta_direct_tiles import exact_eta

pytestmark = pytest.mark.gpu

FLOOR = 1e-6  # of max theta_B: the rounding of theta_B, eta and the operator's coefficients in 32 bits


def _theta(c, p, d):
    th = (c[O.PBA].astype(np.float32).astype(np.float64) + c[O.PBSE].astype(np.float32)) / p["Pmax"]
    return th.reshape(d["nz"], d["ny"], d["nx"])


def _solve(d, p, start, eta_tol, eta_atol=1e-30, eta_maxit=100000, seed=2):
    import torch

    import paper_2304_09180_gb300 as clot
    c, e0, c0 = S.primed_state(d, p, seed=seed)
    ref = exact_eta(d, p, _theta(c, p, d)).reshape(-1)
    m = clot.Mesh(d)
    none = np.zeros(d["ny"] * d["nz"])
    prm = clot.Params(p, none, none, none, eta_tol=eta_tol, eta_atol=eta_atol, eta_maxit=eta_maxit)
    f = clot.Fields.from_host(m, p, c, e0, c0, eta=start(ref))
    clot.clot_eta_solve(m, f, prm)
    torch.cuda.synchronize()
    return np.max(np.abs(f.eta.double().cpu().numpy() - ref)) / np.max(_theta(c, p, d))


MESHES = {"channel": S.channel2d(200, 40, 200 * 1.5 * S.UM, 40 * 1.5 * S.UM),
          "fine": S.channel2d(400, 96, 100 * S.UM, 24 * S.UM), "duct": S.duct3d(70, 33, 40, 1.5 * S.UM)}
STARTS = {"zero": lambda ref: 0 * ref, "level": lambda ref: 0 * ref + 50.0,
          "rough": lambda ref: 10.0 * np.random.default_rng(1).standard_normal(ref.size)}


@pytest.mark.parametrize("start", STARTS)
@pytest.mark.parametrize("mesh", MESHES)
@pytest.mark.parametrize("eta_tol", [1e-5, 1e-6, 1e-9])
def test_error_within_the_rule_from_any_start(mesh, start, eta_tol):
    p = S.params_default()
    assert _solve(MESHES[mesh], p, STARTS[start], eta_tol) <= max(eta_tol, FLOOR)


@pytest.mark.parametrize("mesh", MESHES)
@pytest.mark.parametrize("L_eta", [1e-14, 1e-12, 1e-8, 1e-5, 6e-2])
def test_weak_and_strong_coupling(mesh, L_eta):
    p = S.params_default(L_eta=L_eta)
    assert _solve(MESHES[mesh], p, STARTS["zero"], 1e-6) <= max(1e-6, FLOOR)


@pytest.mark.parametrize("mesh", MESHES)
def test_no_iterations_allowed_leaves_eta(mesh):
    import paper_2304_09180_gb300 as clot
    p = S.params_default()
    d = MESHES[mesh]
    c, e0, c0 = S.primed_state(d, p, seed=2)
    m = clot.Mesh(d)
    none = np.zeros(d["ny"] * d["nz"])
    f = clot.Fields.from_host(m, p, c, e0, c0, eta=0.25 * np.ones(m.ncell))
    clot.clot_eta_solve(m, f, clot.Params(p, none, none, none, eta_maxit=0))
    assert np.all(f.eta.cpu().numpy() == 0.25)


@pytest.mark.parametrize("name", ["duct_300x24x20", "duct_203x67x45", "channel_301x40", "channel_900x72",
                                  "duct_60x256x256", "duct_61x320x330"])
@pytest.mark.parametrize("eta_tol", [1e-6, 1e-9])
def test_predicted_eta_of_a_step(name, eta_tol):
    """The eta a step used, solved from the prediction of the step before: the
    clot keeps the slab that is corrected inside the mesh.  The last two lie on
    either side of the rule that leaves wide cross sections to CG on a box."""
    import torch

    import paper_2304_09180_gb300 as clot
    p = S.params_default()
    cfg = S.config(name, p)
    d = cfg["desc"]
    mesh = clot.Mesh(d)
    f = clot.Fields.from_host(mesh, p, *S.primed_state(d, p, seed=2))
    fl = clot.Fluxes(mesh, **cfg["fluxes"])
    prm = clot.Params(p, **cfg["inlet"], eta_tol=eta_tol, eta_atol=1e-30)
    clot.clot_species_step(mesh, f, fl, prm, cfg["dt"], 3)
    c = f.to_host(mesh)["c"]  # the state the next step's eta is solved from
    clot.clot_species_step(mesh, f, fl, prm, cfg["dt"], 1)
    torch.cuda.synchronize()
    th = _theta(c, p, d)
    got = f.eta.double().cpu().numpy()
    assert np.max(np.abs(got - exact_eta(d, p, th).reshape(-1))) <= max(2 * eta_tol, FLOOR) * np.max(th)


@pytest.mark.parametrize("name", ["duct_45x24x20", "channel_131x40", "channel_1030x20"])
def test_nothing_bound_over_steps(name):
    """Transport alone of plain plasma: eta is zero in every step, from any start."""
    import paper_2304_09180_gb300 as clot
    p = S.params_default(eta_tol=1e-6)
    cfg = S.config(name, p)
    d = cfg["desc"]
    mesh = clot.Mesh(d)
    f = clot.Fields.from_host(mesh, p, *S.plasma_state(d, p, seed=2), eta=0.1 * np.ones(mesh.ncell))
    prm = clot.Params(p, **cfg["inlet"], flags=clot.NO_REACTION)
    for n in (1, 2, 3):
        clot.clot_species_step(mesh, f, clot.Fluxes(mesh, **cfg["fluxes"]), prm, cfg["dt"], n)
        assert np.all(f.eta.cpu().numpy() == 0.0)
