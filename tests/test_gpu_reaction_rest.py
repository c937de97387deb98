"""Cells at rest (nothing bound): the reaction over many substeps is the same
small factor every time.  Increments far below the rounding of P^{m,u} must
still add up, and P^{m,u} + P^{m,a} is conserved: against the 64-bit product of
the RK4 factors, to two roundings of each value."""
import numpy as np
import pytest

import oracle as O
import synthetic as S

pytestmark = pytest.mark.gpu


def _setup(adp, **over):
    import paper_2304_09180_gb300 as clot
    p = S.params_default(eta_tol=1e-6, **over)
    cfg = S.config("channel_60x16", p)
    c, e0, c0 = S.plasma_state(cfg["desc"], p, seed=3)
    c[O.ADP] = adp
    mesh = clot.Mesh(cfg["desc"])
    f = clot.Fields.from_host(mesh, p, c, e0, c0)
    return clot, p, cfg, mesh, f


def _off_the_floor(cfg):
    d = cfg["desc"]
    return np.arange(d["nx"] * d["ny"]) // d["nx"] > 6  # beyond the adhesion layer and the wall


@pytest.mark.parametrize("entry", ["reaction_step", "species_step"])
@pytest.mark.parametrize("M", [2, 32, 1000])
@pytest.mark.parametrize("Ah", [2e-8, 1e-5, 1e-3])
def test_small_increments_add_up(entry, M, Ah):
    import torch

    p0, A = S.params_default(), 0.1
    adp, h = float(np.float32(A * p0["adp_star"] / (p0["k_adp"] - A))), Ah / A
    clot, p, cfg, mesh, f = _setup(adp)
    start = f.to_host(mesh)["c"]
    prm = clot.Params(p, **cfg["inlet"], flags=clot.NO_ETA | clot.NO_TRANSPORT | clot.NO_SIGMA, M_rxn=M)
    if entry == "reaction_step":
        clot.clot_reaction_step(mesh, f, prm, h, M)
    else:
        clot.clot_species_step(mesh, f, clot.Fluxes(mesh, **cfg["fluxes"]), prm, M * h, 1)
    torch.cuda.synchronize()
    got = f.to_host(mesh)["c"]
    z = p["k_adp"] * adp / (p["adp_star"] + adp) * h
    lost = -np.expm1(M * np.log1p(-z + z * z / 2 - z ** 3 / 6 + z ** 4 / 24))  # fraction of P^{m,u} over M substeps
    rows = _off_the_floor(cfg)
    pmu, pma = start[O.PMU][rows].astype(np.float64), start[O.PMA][rows].astype(np.float64)
    moved, eps = lost * pmu, 2.0 ** -23
    # the values are rounded twice; the increment's factor a few times, its sum once a substep
    tol = (8 + M / 2) * eps * moved
    assert np.all(np.abs(got[O.PMU][rows] - (pmu - moved)) <= 2 * eps * pmu + tol)
    assert np.all(np.abs(got[O.PMA][rows] - (pma + moved)) <= 2 * eps * (pma + moved) + tol)


@pytest.mark.parametrize("entry", ["reaction_step", "species_step"])
@pytest.mark.parametrize("constant", ["adp_star", "e2_star"])
def test_no_activation_without_its_concentration(entry, constant):
    """A half-saturation constant of zero with none of the substance: no
    activation (0, not 0/0), the same bits as with the usual constant."""
    import torch

    out = []
    for over in ({}, {constant: 0.0}):
        clot, p, cfg, mesh, f = _setup(0.0, **over)
        prm = clot.Params(p, **cfg["inlet"], flags=clot.NO_ETA)
        if entry == "reaction_step":
            clot.clot_reaction_step(mesh, f, prm, 1e-5, 2)
        else:
            clot.clot_species_step(mesh, f, clot.Fluxes(mesh, **cfg["fluxes"]), prm, cfg["dt"], 1)
        torch.cuda.synchronize()
        out.append(f.to_host(mesh)["c"][:, _off_the_floor(cfg)])
    assert np.all(np.isfinite(out[1]))
    assert np.array_equal(*out)
