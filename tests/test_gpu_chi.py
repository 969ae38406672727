"""chi_ij of the SU2 / XYZ cores against the oracle, pair by pair, on lattices whose exchanged pairs
are read from other entries (pairs of frequencies with |w1| = |w2| have an argument that is exactly
zero, so (w1, w2) and (-w1, -w2) read one of the two each)."""
import numpy as np
import pytest

import workloads as W
from oracle import oracle as O
from tests.helpers import gpu_comp_map, oracle_to_gpu

pytestmark = pytest.mark.gpu

CASES = {
    "square": (lambda: W.square_j1j2(1.0, 0.5), 3, 9, 0.06),
    "kagome": (lambda: W.nn_heisenberg(W.kagome()), 3, 10, 0.06),
    "honeycomb_hk": (lambda: W.honeycomb_kitaev(0.2, -1.0), 3, 8, 0.35),
}


@pytest.mark.parametrize("name", CASES)
def test_pair_correlations_against_oracle(name):
    import torch

    import paper_2109_13317_gb300 as sr
    mk, L, N, lam = CASES[name]
    model = mk()
    mesh = O.mesh_exponential(N, 0.05, 10.0)
    lams = W.lambda_list(8.0, lam, 10)
    of = O.OracleFlow(model, L, mesh)
    for a, b in zip(lams[:-1], lams[1:]):
        of.euler(a, b)
    gam, G = of.get_state()
    lat = sr.Lattice.from_model(model, L)
    fl = sr.Flow(lat, mesh, lams[-1])
    fl.set_state(lams[-1], torch.tensor(gam, device="cuda"),
                 torch.tensor(oracle_to_gpu(of, lat, G, fl.n_comp).reshape(-1), device="cuda"))
    k = np.random.default_rng(3).uniform(-np.pi, np.pi, (17, 3))
    chi_o = of.chi(lams[-1])
    chik, chi = fl.measure(k)
    chi = chi.cpu().numpy()
    sites = fl.chi_sites()
    where = {(b,) + tuple(s): j for b in range(lat.N_basis) for j, s in enumerate(sites[b])}
    scale = max(np.abs(x).max() for x in chi_o)
    cm = gpu_comp_map(fl.n_comp)
    for b in range(lat.N_basis):
        for j, s in enumerate(sites[b]):
            exp = chi_o[b][of.find(b, s[:3], int(s[3])), cm]
            assert np.abs(chi[b, j] - exp).max() <= 1e-10 * scale, (b, tuple(s))
            rev = chi[int(s[3]), where[(int(s[3]), -s[0], -s[1], -s[2], b)]]
            assert np.abs(chi[b, j] - rev).max() <= 1e-10 * scale, (b, tuple(s))
    ck_o = of.chi_k(lams[-1], k, chi_o)
    assert np.abs(chik - ck_o).max() <= 1e-10 * np.abs(ck_o).max()
    kd = torch.tensor(k.reshape(-1), device="cuda")
    out = torch.empty(len(k), dtype=torch.float64, device="cuda")
    fl.measure_static(kd, out)
    assert np.abs(out.cpu().numpy() - ck_o).max() <= 1e-10 * np.abs(ck_o).max()
    fl.close()
