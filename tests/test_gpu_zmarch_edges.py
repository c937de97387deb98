"""The 3D fused step at the edges of its tiles, against the FP64 oracle, cell by
cell: rows of one, two and four-float multiples (its three ways of staging
planes), tiles that end one cell in or one short, a mesh end inside the halo,
one plane, runs of one plane and of several; in a flow with all three
components, so that every face advects, in the usual step and with the options
that take the general kernel.  Tolerance: that of the small-mesh parity test,
1e-5 of each species' maximum."""
import numpy as np
import pytest

import oracle as O
import synthetic as S
from parity_util import run_gpu, run_oracle

pytestmark = pytest.mark.gpu

MESHES = [(33, 9, 3), (34, 17, 13), (36, 9, 5), (65, 8, 2), (31, 7, 25), (66, 15, 4), (64, 16, 1), (32, 1, 6), (12, 10, 3)]


def _rolled(desc, shear):
    """The duct's fluxes plus divergence-free rolls in the x-y and x-z planes."""
    nx, ny, nz, h = desc["nx"], desc["ny"], desc["nz"], desc["hy"]
    fl = S.fluxes_duct3d(desc, shear)
    fx, fy, fz = (fl["fx"].reshape(nz, ny, nx + 1).copy(), fl["fy"].reshape(nz, ny + 1, nx).copy(),
                  fl["fz"].reshape(nz + 1, ny, nx).copy())
    U, wave = 0.05 * shear * ny * h * h * h, np.sin(3 * np.pi * np.arange(nx + 1) / nx)
    y, z = np.arange(ny + 1) / ny, np.arange(nz + 1) / nz
    a, b = U * (4 * y * (1 - y)) ** 2, U * (4 * z * (1 - z)) ** 2
    fx += np.diff(a)[None, :, None] * wave + np.diff(b)[:, None, None] * wave
    fy -= a[None, :, None] * np.diff(wave)
    fz -= b[:, None, None] * np.diff(wave)
    return dict(fx=fx.reshape(-1), fy=fy.reshape(-1), fz=fz.reshape(-1))


@pytest.mark.parametrize("flags", [0, "heun", "lagged"], ids=str)
@pytest.mark.parametrize("mesh", MESHES, ids=lambda m: "x".join(map(str, m)))
def test_tile_edges_match_the_oracle(mesh, flags):
    import paper_2304_09180_gb300 as clot
    p = S.params_default()
    cfg = S.config("duct_%dx%dx%d" % mesh, p)
    cfg["fluxes"] = _rolled(cfg["desc"], 1000.0)
    cfg["dt"] = 0.5 * S.stable_dt(cfg["desc"], cfg["fluxes"], p)
    state = S.primed_state(cfg["desc"], p, seed=sum(mesh))
    gf, of = {0: (0, 0), "heun": (clot.HEUN | clot.STRANG, O.TRANSPORT_RK2 | O.STRANG),
              "lagged": (clot.WALL_LAGGED, O.WALL_LAGGED)}[flags]
    ref = run_oracle(cfg, S.params_default(eta_tol=1e-10, flags=of), state, 4)
    gpu = run_gpu(cfg, p, state, 4, eta_tol=1e-6, flags=gf)
    for s in range(15):
        scale = np.max(np.abs(ref.c[s]))
        if scale > 0:
            assert np.max(np.abs(gpu["c"][s] - ref.c[s])) <= 1e-5 * scale, S.SPECIES[s]
