"""The TRI vertex flow with the dense lattice sum against the general TRI kernel.

The reference is the value part of a tangent flow (sr_flow_init_tangent), which runs the general
kernel on dual numbers in FP64 with the lattice-sum table summed entry by entry.  The state is
random, so every component, site and frequency counts; `odd` says whether the functions with an odd
number of in-plane spin indices are there (a graded lattice then takes the general form) or zero.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

MODELS = {
    "kagome_dm": (lambda: W.kagome_dm(1.0, 0.5), 6, 3),
    "kagome_dm_x": (lambda: W.rotated(W.kagome_dm(1.0, 0.4), np.array([[0, 0, 1.0], [1, 0, 0], [0, 1, 0]])), 6, 1),
    "honeycomb_hkg": (lambda: W.honeycomb_kitaev_gamma(0.1, -1.0, 0.5), 3, 0),
}


# sizes: one site in range, ragged tiles (5, 9, 13, 26 sites), the largest whose tangent flow fits
@pytest.mark.parametrize("name,L,N", [("kagome_dm", 1, 2), ("kagome_dm", 2, 9), ("kagome_dm", 4, 6), ("kagome_dm", 6, 4),
                                      ("kagome_dm_x", 3, 7), ("honeycomb_hkg", 1, 5), ("honeycomb_hkg", 4, 6),
                                      ("honeycomb_hkg", 6, 4)])
@pytest.mark.parametrize("odd", [False, True])
@pytest.mark.parametrize("mixed", [False, True])
def test_dense_matches_general(name, L, N, odd, mixed):
    import torch

    import paper_2109_13317_gb300 as sr
    make, ncoup, axis = MODELS[name]
    model = make()
    lat = sr.Lattice.from_model(model, L)
    mesh = sr.sr_frequency_mesh_exponential(N, 0.05, 20.0)
    lam = 0.7
    rng = np.random.default_rng(11 + N)
    G = rng.normal(size=(N * (N + 1) // 2, N, 16, lat.N_s))
    if not odd and axis:
        even = [((c // 4) in (0, axis)) == ((c % 4) in (0, axis)) for c in range(16)]
        G[:, :, ~np.array(even)] = 0.0
    gam = 0.2 * np.tanh(mesh)
    fl = sr.Flow(lat, mesh, lam, sr.SR_FP32_MIXED if mixed else sr.SR_FP64)
    fl.set_state(lam, torch.tensor(gam, device="cuda"), torch.tensor(G.reshape(-1), device="cuda"))
    ds, dG = fl.rhs(lam)
    # the same state as the value part of a tangent flow along one coupling direction
    dM = np.stack([c.M for c in model.couplings])[None]
    ft = sr.Flow(lat, mesh, lam, tangents=dM)
    tri = lambda x: torch.tensor(np.stack([x, 0 * x, 0 * x], -1).reshape(-1), device="cuda")  # noqa: E731
    ft.set_state(lam, tri(gam), tri(G.reshape(-1)))
    rs, rG = (x.view(-1, 3)[:, 0] for x in ft.rhs(lam))
    assert ncoup == len(model.couplings)
    assert (ds - rs).abs().max() <= 1e-13 * rs.abs().max()
    # sums of some thousands of products of order one: FP64 rounding 1e-16 and FP32 rounding 6e-8 of
    # the sum's scale per product, accumulating at most linearly over ~1e3 terms of one output
    tol = 1e-4 if mixed else 1e-12
    shape = fl.shape()
    for c in range(16):
        a, b = (x.view(shape)[:, :, c] for x in (dG, rG))
        assert (a - b).abs().max() <= tol * rG.abs().max(), c
