"""The direct eta solve (cosine transforms along y and z, a tridiagonal solve
per mode along x; App. A, Eq. eta) against the FP64 oracle at the sizes where
it can go wrong: the edges of its 32- and 64-row tiles and 64-column tiles, odd
and even extents (the folded middle row), single rows, columns and planes, each
number of cells a lane holds, the largest extents it takes and the first ones
it leaves to the iteration.  Tolerance: that of the eta parity test, 2e-6 of
max theta_B, from zero and from a perturbed solution."""
import numpy as np
import pytest

import oracle as O
import synthetic as S

pytestmark = pytest.mark.gpu

MESHES = [(1, 1, 1), (1, 7, 1), (5, 3, 1), (64, 32, 1), (63, 63, 1), (65, 65, 1), (130, 64, 1), (257, 129, 1),
          (516, 10, 1), (1024, 6, 1), (1025, 6, 1), (6, 512, 1), (6, 513, 1),
          (21, 9, 7), (34, 33, 5), (16, 64, 66), (33, 1, 65), (5, 130, 3), (40, 5, 129)]


@pytest.mark.parametrize("mesh", MESHES, ids=lambda m: "x".join(map(str, m)))
@pytest.mark.parametrize("h", [1.5, 0.3])
def test_direct_solve_matches_the_oracle(mesh, h):
    import torch

    import paper_2304_09180_gb300 as clot
    nx, ny, nz = mesh
    p = S.params_default(eta_tol=1e-6)
    dim = 3 if nz > 1 else 2
    h *= S.UM
    d = S.duct3d(nx, ny, nz, h) if dim == 3 else S.channel2d(nx, ny, nx * h, ny * h)
    rng = np.random.default_rng(nx + 7 * ny + 31 * nz)
    nc = nx * ny * nz
    c = np.zeros((15, nc))
    c[O.PBA] = p["Pmax"] * 0.5 * rng.random(nc) * (rng.random(nc) < 0.3)
    c[O.PBSE] = p["Pmax"] * 0.4 * rng.random(nc)
    thB = (c[O.PBA].astype(np.float32).astype(np.float64) + c[O.PBSE].astype(np.float32)) / p["Pmax"]
    ref, _ = O.eta_solve(d, p, thB)
    m = clot.Mesh(d)
    prm = clot.Params(p, np.zeros(ny * nz), np.zeros(ny * nz), np.zeros(ny * nz))
    start = 0.9 * ref + 0.02 * rng.random(nc)
    for eta in (None, start):
        f = clot.Fields.from_host(m, p, c, np.zeros(m.n_inj), np.zeros(m.n_inj), eta=eta)
        clot.clot_eta_solve(m, f, prm)
        torch.cuda.synchronize()
        got = f.eta.double().cpu().numpy()
        assert np.max(np.abs(got - ref)) <= 2e-6 * np.max(thB), (mesh, eta is None)


@pytest.mark.parametrize("L_eta,scale", [(0.0, 1.0), (6.0e-3, 0.0), (6.0e-3, 0.05)])
def test_uncoupled_empty_and_thin_states(L_eta, scale):
    """No coupling between cells (L_eta = 0): eta = theta_B.  Nothing bound:
    eta = 0 exactly.  max theta_B below the binding threshold eta_t, where the
    solve iterates: the stopping rule's bound."""
    import paper_2304_09180_gb300 as clot
    p = S.params_default(eta_tol=1e-6, L_eta=L_eta)
    cfg = S.config("duct_24x12x10", p)
    d = cfg["desc"]
    c, e0, c0 = S.primed_state(d, p, seed=6)
    c[O.PBA] *= scale
    c[O.PBSE] *= scale
    thB = (c[O.PBA].astype(np.float32).astype(np.float64) + c[O.PBSE].astype(np.float32)) / p["Pmax"]
    m = clot.Mesh(d)
    f = clot.Fields.from_host(m, p, c, e0, c0, eta=0.1 * np.ones(m.ncell))
    clot.clot_eta_solve(m, f, clot.Params(p, **cfg["inlet"]))
    got = f.eta.double().cpu().numpy()
    ref = thB if L_eta == 0.0 else O.eta_solve(d, p, thB)[0] if scale else np.zeros_like(thB)
    tol = 0.0 if scale == 0.0 else 2e-6 * max(np.max(thB), 1.0)
    assert np.max(np.abs(got - ref)) <= tol
