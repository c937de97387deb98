"""The direct eta solve where a block takes several tiles of a transform, one
after the other through the same shared memory: axes of one, two and three
stages of matrix rows (32 rows each), tiles of 32 and 64 modes, an axis of one
cell (no odd mode), on meshes of more tiles than the chip holds blocks.  Against
the 64-bit solution by cosine transforms along all axes; tolerance that of the
eta parity test, 2e-6 of max theta_B.  Solves from the same start give the same
bits."""
import numpy as np
import pytest
from scipy import fft

import oracle as O
import synthetic as S

pytestmark = pytest.mark.gpu

MESHES = [(256, 64, 64), (256, 128, 64), (128, 160, 96), (512, 1, 130), (203, 67, 131), (96, 190, 190)]


def exact_eta(desc, p, thB):
    """(I - L_eta^2 / 4 lap) eta = thB with zero-flux walls, 64 bits; thB [nz, ny, nx]."""
    lam = 1.0
    for ax, key in ((0, "hz"), (1, "hy"), (2, "hx")):
        n = thB.shape[ax]
        ev = 4 * np.sin(np.pi * np.arange(n) / (2 * n)) ** 2 * p["L_eta"] ** 2 / 4 / desc[key] ** 2
        lam = lam + (ev.reshape([-1 if a == ax else 1 for a in range(3)]) if n > 1 else 0.0)
    return fft.idctn(fft.dctn(thB, type=2, norm="ortho") / lam, type=2, norm="ortho")


@pytest.mark.parametrize("mesh", MESHES, ids=lambda m: "x".join(map(str, m)))
def test_several_tiles_a_block(mesh):
    import torch

    import paper_2304_09180_gb300 as clot
    nx, ny, nz = mesh
    p = S.params_default(eta_tol=1e-6)
    d = S.duct3d(nx, ny, nz, 1.5 * S.UM)
    rng = np.random.default_rng(nx + 7 * ny + 31 * nz)
    nc = nx * ny * nz
    c = np.zeros((15, nc))
    c[O.PBA] = p["Pmax"] * 0.5 * rng.random(nc) * (rng.random(nc) < 0.3)
    c[O.PBSE] = p["Pmax"] * 0.4 * rng.random(nc)
    thB = (c[O.PBA].astype(np.float32).astype(np.float64) + c[O.PBSE].astype(np.float32)) / p["Pmax"]
    ref = exact_eta(d, p, thB.reshape(nz, ny, nx)).reshape(-1)
    m = clot.Mesh(d)
    none = np.zeros(ny * nz)
    prm = clot.Params(p, none, none, none)
    wall = np.zeros(m.n_inj)
    f = clot.Fields.from_host(m, p, c, wall, wall)
    for start in (np.zeros(nc), 0.9 * ref + 0.02 * rng.random(nc)):
        first, eta0 = None, torch.as_tensor(start, dtype=torch.float32, device=f.eta.device)
        for _ in range(4):
            f.eta.copy_(eta0)
            clot.clot_eta_solve(m, f, prm)
            got = f.eta.clone()
            if first is None:
                first = got
                assert np.max(np.abs(got.double().cpu().numpy() - ref)) <= 2e-6 * np.max(thB)
            assert torch.equal(first, got)
