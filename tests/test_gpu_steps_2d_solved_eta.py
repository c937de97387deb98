"""Whole steps of a small 2D mesh in one launch when the eta passed in already
meets the stopping rule: the first solve of a call then only checks it.  The
solves of a launch share their barrier words, so this is where a step could
read what the step before left there.  Against the same steps launch by launch
(which per-kernel timing selects): the state within the parity bar, eta within
twice the stopping rule's bound (each side is within it of the solution)."""
import numpy as np
import pytest

import synthetic as S
from parity_util import species_errors

pytestmark = pytest.mark.gpu

TOL = 4e-6  # above the rounding of a solved eta's residual on these meshes


@pytest.mark.parametrize("maxit", [1000, 0])
@pytest.mark.parametrize("calls", [(1, 1, 1), (5, 2)], ids=str)
@pytest.mark.parametrize("name", ["channel_20x6", "channel_131x40", "channel_300x64"])
def test_solved_eta_on_entry(name, calls, maxit):
    import torch

    import paper_2304_09180_gb300 as clot
    p = S.params_default(eta_tol=1e-6)
    cfg = S.config(name, p)
    state = S.primed_state(cfg["desc"], p, seed=8)
    out = []
    for launches in (False, True):
        mesh = clot.Mesh(cfg["desc"])
        fl = clot.Fluxes(mesh, **cfg["fluxes"])
        f = clot.Fields.from_host(mesh, p, *state)
        clot.clot_eta_solve(mesh, f, clot.Params(p, **cfg["inlet"]))
        prm = clot.Params(p, **cfg["inlet"], flags=clot.binding.ETA_FRESH | clot.SYNC_STATUS, eta_tol=TOL, eta_maxit=maxit)
        for n in calls:
            if launches:
                clot.clot_profile_begin(mesh, max_launches=256)
            for _ in range(2):
                clot.clot_species_step(mesh, f, fl, prm, cfg["dt"], n)
            if launches:
                clot.clot_profile_end(mesh)
        torch.cuda.synchronize()
        out.append(f.to_host(mesh))
    a, b = out
    assert np.max(b["eta"]) > p["eta_t"]
    assert np.all(species_errors(a["c"], b["c"]) <= 1e-5)
    assert np.max(np.abs(a["eta"] - b["eta"])) <= 2 * TOL


@pytest.mark.parametrize("option", ["heun", "strang", "second", "lagged", "deviation"])
@pytest.mark.parametrize("name", ["channel_131x40", "channel_300x64"])
def test_options_with_eta_in_one_launch(name, option):
    """The stepping options with the eta solve, over several calls."""
    import torch

    import paper_2304_09180_gb300 as clot
    p = S.params_default(eta_tol=1e-6)
    cfg = S.config(name, p)
    state = S.primed_state(cfg["desc"], p, seed=9)
    flags = {"heun": clot.HEUN, "strang": clot.STRANG, "second": clot.HEUN | clot.STRANG, "lagged": clot.WALL_LAGGED,
             "deviation": clot.DEVIATION}[option]
    out = []
    for launches in (False, True):
        mesh = clot.Mesh(cfg["desc"])
        fl = clot.Fluxes(mesh, **cfg["fluxes"])
        f = clot.Fields.from_host(mesh, p, *state)
        prm = clot.Params(p, **cfg["inlet"], flags=flags)
        if launches:
            clot.clot_profile_begin(mesh, max_launches=1024)
        for n in (1, 4, 12):
            clot.clot_species_step(mesh, f, fl, prm, cfg["dt"], n)
        if launches:
            clot.clot_profile_end(mesh)
        torch.cuda.synchronize()
        out.append(f.to_host(mesh))
    a, b = out
    assert np.all(species_errors(a["c"], b["c"]) <= 1e-5)
    assert np.max(np.abs(a["eta"] - b["eta"])) <= 2e-6 * np.max(b["eta"])
