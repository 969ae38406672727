"""Right-hand side and adjoint of the SU2 / XYZ cores for states whose spin components differ in
size by orders of magnitude (XXZ- and Ising-like couplings, states with a dominant density), every
component on its own scale.

The reference is the tangent flow, which forms the products component by component in FP64: its
value part for the right-hand side, and its derivatives along single entries for the adjoint.  The
density vanishes at s = u, where the s <-> u relation flips its sign (see test_gpu_pair.py).
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _model(name, eps):
    if name == "square_su2":
        return W.square_j1j2(1.0, 0.5)
    cell = {"square_xxz": W.square, "kagome_xxz": W.kagome}[name]()
    m = W.nn_heisenberg(cell)
    for c in m.couplings:
        c.M = np.diag([eps, eps, 1.0])
    m.backend = "XYZ"
    return m


def _state(fl, scale, rng):
    G = rng.normal(size=fl.shape())
    G[[i * (i + 3) // 2 for i in range(fl.N)], :, 0] = 0.0
    return G * np.asarray(scale)[None, None, :, None]


def _scales(name, eps):
    return [1.0, eps] if name == "square_su2" else [1.0, eps, eps, 1.0]


def _cuda(x):
    import torch
    return torch.tensor(np.ascontiguousarray(x).reshape(-1), device="cuda")


CASES = [("square_su2", 3, 16), ("square_su2", 6, 9), ("square_xxz", 3, 16), ("square_xxz", 6, 7), ("kagome_xxz", 2, 9),
         ("kagome_xxz", 4, 5)]


@pytest.mark.parametrize("name,L,N", CASES)
@pytest.mark.parametrize("eps", [1e-3, 1e-6, 0.0])
@pytest.mark.parametrize("mixed", [False, True])
def test_weak_components_of_the_right_hand_side(name, L, N, eps, mixed):
    import paper_2109_13317_gb300 as sr
    model = _model(name, eps)
    lat = sr.Lattice.from_model(model, L)
    mesh = sr.sr_frequency_mesh_exponential(N, 0.05, 20.0)
    lam = 0.7
    fl = sr.Flow(lat, mesh, lam, sr.SR_FP32_MIXED if mixed else sr.SR_FP64)
    G = _state(fl, _scales(name, eps), np.random.default_rng(11 + N))
    gam = 0.2 * np.tanh(mesh)
    fl.set_state(lam, _cuda(gam), _cuda(G))
    _, dG = fl.rhs(lam)
    ft = sr.Flow(lat, mesh, lam, tangents=np.stack([c.M for c in model.couplings])[None])
    ft.set_state(lam, _cuda(np.stack([gam, 0 * gam, 0 * gam], -1)), _cuda(np.stack([G.reshape(-1), 0 * G.reshape(-1), 0 * G.reshape(-1)], -1)))
    rG = ft.rhs(lam)[1].view(-1, 3)[:, 0]
    # rounding of 1e-16 (FP64) and 6e-8 (FP32) of the sum's scale per product, accumulating at most
    # linearly over ~1e3 terms of one output; every product of a weak component has a weak factor
    tol = 1e-4 if mixed else 1e-12
    for c in range(fl.n_comp):
        a, b = (x.view(fl.shape())[:, :, c] for x in (dG, rG))
        assert (a - b).abs().max() <= tol * b.abs().max(), (c, float((a - b).abs().max()), float(b.abs().max()))
    fl.close()
    ft.close()


@pytest.mark.parametrize("name,L,N", [("square_su2", 3, 7), ("square_xxz", 3, 7), ("kagome_xxz", 2, 6)])
def test_weak_components_of_the_adjoint(name, L, N):
    """(J^T fbar)_i = <fbar, J e_i> at single entries i of a weak component."""
    import paper_2109_13317_gb300 as sr
    eps = 1e-8
    model = _model(name, eps)
    lat = sr.Lattice.from_model(model, L)
    mesh = sr.sr_frequency_mesh_exponential(N, 0.05, 20.0)
    lam = 0.7
    rng = np.random.default_rng(23 + L)
    fl = sr.Flow(lat, mesh, lam)
    G, fbar = _state(fl, _scales(name, eps), rng), _state(fl, _scales(name, eps), rng)
    gam = 0.2 * np.tanh(mesh)
    fl.set_state(lam, _cuda(gam), _cuda(G))
    bar = fl.rhs_adjoint(lam, _cuda(0 * gam), _cuda(fbar))[1].view(fl.shape())
    ft = sr.Flow(lat, mesh, lam, tangents=np.stack([c.M for c in model.couplings])[None])
    w = np.zeros(G.shape)
    zero = 0 * G.reshape(-1)
    fb = _cuda(fbar)
    for _ in range(8):
        at = (int(rng.integers(fl.npair)), int(rng.integers(N)), 1, int(rng.integers(lat.N_s)))
        w[at] = 1.0
        ft.set_state(lam, _cuda(np.stack([gam, 0 * gam, 0 * gam], -1)), _cuda(np.stack([G.reshape(-1), w.reshape(-1), zero], -1)))
        w[at] = 0.0
        terms = fb * ft.rhs(lam)[1].view(-1, 3)[:, 1]
        # rounding of 1e-16 per term, at most ~1e3 rounded terms per entry behind each of them
        assert abs(float(bar[at]) - float(terms.sum())) <= 1e-12 * float(terms.abs().sum()), at
    fl.close()
    ft.close()
