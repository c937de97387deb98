"""Whole steps of a small 2D mesh in one launch against the same steps launch by
launch (which per-kernel timing selects): the cell and face code is the same, so
without eta the state is equal bit for bit, for odd and even step counts split
over calls (the result lands in either buffer), the stepping options, and ADP
samples inside a call; with eta within the parity bar (its reductions run in
blocks of another size).  Meshes: one tile, tiles that end one cell in, odd and
even rows, the largest mesh taken and the first one not taken."""
import numpy as np
import pytest

import synthetic as S
from parity_util import species_errors

pytestmark = pytest.mark.gpu

TOL = 1e-5
OPTIONS = ("plain", "heun", "strang", "second", "lagged", "deviation", "partner")


def _run(cfg, params, state, calls, flags, option, launches, **over):
    import torch

    import paper_2304_09180_gb300 as clot
    flags |= {"heun": clot.HEUN, "strang": clot.STRANG, "second": clot.HEUN | clot.STRANG, "lagged": clot.WALL_LAGGED,
              "deviation": clot.DEVIATION}.get(option, 0)
    mesh = clot.Mesh(cfg["desc"])
    fl = clot.Fluxes(mesh, **cfg["fluxes"])
    prm = clot.Params(dict(params, **over), **cfg["inlet"], flags=flags)
    f = clot.Fields.from_host(mesh, dict(params, **over), *state, double_buffer=option == "partner")
    if launches:
        clot.clot_profile_begin(mesh, max_launches=8192)
    for n in calls:
        clot.clot_species_step(mesh, f, fl, prm, cfg["dt"], n)
    torch.cuda.synchronize()
    if launches:
        clot.clot_profile_end(mesh)
    return f.to_host(mesh), f


@pytest.mark.parametrize("option", OPTIONS)
@pytest.mark.parametrize("name", ["channel_20x6", "channel_33x9", "channel_64x16", "channel_131x40"])
def test_one_launch_equals_launch_by_launch_without_eta(name, option):
    import paper_2304_09180_gb300 as clot
    p = S.params_default()
    cfg = S.config(name, p)
    state = S.primed_state(cfg["desc"], p, seed=4)
    # two ADP samples within the run, the second inside a call
    over = dict(sigma_dt=6.5 * cfg["dt"], sigma_tf=6 * 6.5 * cfg["dt"])
    a, fa = _run(cfg, p, state, (1, 3, 2, 9), clot.NO_ETA, option, False, **over)
    b, fb = _run(cfg, p, state, (1, 3, 2, 9), clot.NO_ETA, option, True, **over)
    assert fa.n_samples == fb.n_samples == 2
    for k in ("c", "e0", "c0", "sigma"):
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("kind", ["plasma", "primed"])
@pytest.mark.parametrize("name", ["channel_20x6", "channel_131x40", "channel_300x64", "channel_608x128", "channel_640x128"])
def test_one_launch_with_eta_meets_the_parity_bar(name, kind):
    p = S.params_default(eta_tol=1e-6)
    cfg = S.config(name, p)
    state = (S.plasma_state if kind == "plasma" else S.primed_state)(cfg["desc"], p, seed=6)
    a, _ = _run(cfg, p, state, (1, 4, 12), 0, "plain", False)
    b, _ = _run(cfg, p, state, (1, 4, 12), 0, "plain", True)
    assert np.all(species_errors(a["c"], b["c"]) <= TOL)
    assert np.max(np.abs(a["eta"] - b["eta"])) <= 2e-6 * max(np.max(b["eta"]), 1.0)
