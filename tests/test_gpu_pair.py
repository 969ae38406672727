"""The SU2 / XYZ vertex flow on the packed state (eigenvalue rows, dense or listed lattice sum)
against the general kernel.

The reference is the value part of a tangent flow (sr_flow_init_tangent), which runs the general
kernel on dual numbers in FP64 (component products, the lattice-sum list summed entry by entry), or,
for a lattice too wide for it, the same SU(2) state on the XYZ core, whose products then exceed the
listed form.  The state is random, so every component, site and frequency counts, with the one
property that lookups rely on: the density vanishes at s = u, where the s <-> u relation flips its
sign (rows with |s| = |u| otherwise jump with the rounding of their arguments).
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

MODELS = {
    "square": lambda: W.square_j1j2(1.0, 0.5),
    "kagome": lambda: W.nn_heisenberg(W.kagome()),          # exchanged pairs differ
    "pyrochlore": lambda: W.nn_heisenberg(W.pyrochlore()),
    "honeycomb_hk": lambda: W.honeycomb_kitaev(0.2, -1.0),
}


# one and two sites, ragged rows and tiles, and the changes of kernel variant: FP32 tiles of 4 x 4
# (up to 20 sites), 8 x 4 one per thread (48) and two per thread (kagome range 9), FP64 lists of up
# to 128 and 1024 products and tiles beyond
@pytest.mark.parametrize("name,L,N", [("square", 1, 2), ("square", 2, 70), ("square", 3, 16), ("square", 7, 9), ("square", 9, 5),
                                      ("kagome", 1, 5), ("kagome", 5, 7), ("kagome", 7, 6), ("kagome", 8, 3), ("kagome", 9, 3), ("pyrochlore", 2, 11),
                                      ("pyrochlore", 6, 4), ("honeycomb_hk", 1, 3), ("honeycomb_hk", 3, 13),
                                      ("honeycomb_hk", 5, 8), ("honeycomb_hk", 7, 5)])
@pytest.mark.parametrize("mixed", [False, True])
def test_packed_matches_general(name, L, N, mixed):
    import torch

    import paper_2109_13317_gb300 as sr
    model = MODELS[name]()
    lat = sr.Lattice.from_model(model, L)
    mesh = sr.sr_frequency_mesh_exponential(N, 0.05, 20.0)
    lam = 0.7
    rng = np.random.default_rng(5 + N)
    fl = sr.Flow(lat, mesh, lam, sr.SR_FP32_MIXED if mixed else sr.SR_FP64)
    G = rng.normal(size=fl.shape())
    G[[i * (i + 3) // 2 for i in range(N)], :, 0] = 0.0
    gam = 0.2 * np.tanh(mesh)
    cuda = lambda x: torch.tensor(np.ascontiguousarray(x).reshape(-1), device="cuda")  # noqa: E731
    fl.set_state(lam, cuda(gam), cuda(G))
    ds, dG = fl.rhs(lam)
    if (name, L) == ("kagome", 9):
        ft = sr.Flow(sr.Lattice.from_model(model, L, backend=sr.SR_XYZ), mesh, lam)
        ft.set_state(lam, cuda(gam), cuda(G[:, :, [0, 1, 1, 1]]))
        rs, rG = ft.rhs(lam)
        rG = rG.view(ft.shape())[:, :, :2].reshape(-1)
    else:
        dM = np.stack([c.M for c in model.couplings])[None]
        ft = sr.Flow(lat, mesh, lam, tangents=dM)
        dual = lambda x: cuda(np.stack([x, 0 * x, 0 * x], -1))  # noqa: E731
        ft.set_state(lam, dual(gam), dual(G))
        rs, rG = (x.view(-1, 3)[:, 0] for x in ft.rhs(lam))
    assert (ds - rs).abs().max() <= 1e-13 * rs.abs().max()
    # sums of up to some thousands of products of order one: rounding of 1e-16 (FP64) and 6e-8 (FP32)
    # of the sum's scale per product, accumulating at most linearly over ~1e3 terms of one output
    tol = 1e-4 if mixed else 1e-12
    shape = fl.shape()
    for c in range(fl.n_comp):
        a, b = (x.view(shape)[:, :, c] for x in (dG, rG))
        assert (a - b).abs().max() <= tol * rG.abs().max(), c
