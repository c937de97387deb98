"""Runs of one ensemble that follow one another: the arguments and the graph a
run finds from the one before are used only where they are its own.  Without
eta the same steps on a new ensemble give the same bits."""
import numpy as np
import pytest

import synthetic as S
from test_gpu_ensemble import _channels, _specs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps", [(1, 1), (13, 8), (14, 15), (7, 2)])
def test_runs_in_turn_equal_runs_alone(steps):
    """A run with eta leaves its graph behind; the state is then set back, and
    runs without eta (the same arguments twice, then another dt) must give
    what a new ensemble gives: tolerance zero, the same kernels on the same
    values."""
    import torch

    import paper_2304_09180_gb300 as clot
    p = S.params_default(eta_tol=1e-6)
    off = dict(p, flags=clot.NO_ETA)
    specs = _specs(3, seed=5)
    sides = []
    for before in (True, False):
        ens, fields, fluxes, inlets, dts, states, _ = _channels(specs, p, seed=20)
        if before:
            ens.run(fields, fluxes, inlets, dts, p, 14)
            torch.cuda.synchronize()
            for c, f in enumerate(fields):  # everything back, in the same buffers: the same addresses
                fresh = clot.Fields.from_host(ens.meshes[c], p, *states[c])
                for k in ("c", "e0", "c0", "eta", "sigma", "hist", "bound_acc"):
                    getattr(f, k).copy_(getattr(fresh, k))
                f.t, f.t_last, f.n_samples, f.head = fresh.t, fresh.t_last, fresh.n_samples, fresh.head
        for n, scale in ((steps[0], 1.0), (steps[1], 1.0), (steps[0], 0.5)):
            ens.run(fields, fluxes, inlets, [scale * dt for dt in dts], off, n)
        torch.cuda.synchronize()
        sides.append([f.to_host(ens.meshes[c])["c"] for c, f in enumerate(fields)])
    for a, b in zip(*sides):
        assert np.array_equal(a, b)
