"""params.wait_s bounds the waits of the eta solve, not the steps of a small 2D
mesh in one launch: with a bound no wait could meet and no eta solve, the steps
run as with the usual bound and report no timeout."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", ["euler", "second"])
@pytest.mark.parametrize("name", ["channel_131x40", "channel_300x64"])
def test_steps_without_eta_are_not_bounded_by_the_eta_wait(name, order):
    import paper_2304_09180_gb300 as clot
    p = S.params_default()
    cfg = S.config(name, p)
    state = S.primed_state(cfg["desc"], p, seed=4)
    flags = clot.NO_ETA | clot.SYNC_STATUS | (clot.HEUN | clot.STRANG if order == "second" else 0)
    out = []
    for wait in (0.0, 1e-9):
        mesh = clot.Mesh(cfg["desc"])
        f = clot.Fields.from_host(mesh, p, *state)
        prm = clot.Params(p, **cfg["inlet"], flags=flags, M_rxn=50, wait_s=wait)
        clot.clot_species_step(mesh, f, clot.Fluxes(mesh, **cfg["fluxes"]), prm, cfg["dt"], 8)
        out.append(f.to_host(mesh)["c"])
    assert np.array_equal(*out)
