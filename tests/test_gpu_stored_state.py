"""The kernels on the stored state (flows without a packed copy: no plan for the lattice, no memory, or
switched off), against the oracle and against the packed form, alone, in the adjoint and in batches."""
import numpy as np
import pytest

import workloads as W
from oracle import oracle as O
from tests.helpers import oracle_to_gpu

pytestmark = pytest.mark.gpu

MODELS = {
    "square": lambda: W.square_j1j2(1.0, 0.5),
    "kagome": lambda: W.nn_heisenberg(W.kagome()),
    "honeycomb_hk": lambda: W.honeycomb_kitaev(0.2, -1.0),
    "kagome_dm": lambda: W.kagome_dm(1.0, 0.5),                    # graded TRI
    "honeycomb_hkg": lambda: W.honeycomb_kitaev_gamma(),           # ungraded TRI
}


def _flow(name, L, N, lams, mixed=True, packed=True):
    import paper_2109_13317_gb300 as sr
    lat = sr.Lattice.from_model(MODELS[name](), L)
    fl = sr.Flow(lat, O.mesh_exponential(N, 0.05, 10.0), lams[0], sr.SR_FP32_MIXED if mixed else sr.SR_FP64)
    assert fl.packed
    if not packed:
        fl.packed = False
        assert not fl.packed
    return lat, fl


def _rel(a, b):
    return float((a - b).abs().max() / b.abs().max())


@pytest.mark.parametrize("name,L,N", [("square", 3, 9), ("kagome", 3, 7), ("honeycomb_hk", 2, 8), ("kagome_dm", 2, 5), ("honeycomb_hkg", 1, 6)])
@pytest.mark.parametrize("mixed", [False, True])
def test_stored_state_matches_packed(name, L, N, mixed):
    lams = W.lambda_list(8.0, 1.0, 6)
    _, a = _flow(name, L, N, lams, mixed)
    _, b = _flow(name, L, N, lams, mixed, packed=False)
    for lam in lams[1:]:
        a.step(lam)
        b.step(lam)
    for x, y in zip(a.get_state(), b.get_state()):
        assert _rel(y, x) <= (1e-5 if mixed else 1e-12)
    x = a.rhs(lams[-1])[1]
    b.packed = True     # back again, on the same state
    b.set_state(lams[-1], *a.get_state())
    assert _rel(b.rhs(lams[-1])[1], x) == 0.0
    a.close()
    b.close()


@pytest.mark.parametrize("name,L,N", [("kagome", 3, 6), ("honeycomb_hk", 2, 6)])
@pytest.mark.parametrize("mixed", [False, True])
def test_stored_state_against_oracle(name, L, N, mixed):
    lams = W.lambda_list(8.0, 1.0, 6)
    of = O.OracleFlow(MODELS[name](), L, O.mesh_exponential(N, 0.05, 10.0))
    lat, fl = _flow(name, L, N, lams, mixed, packed=False)
    for p, q in zip(lams[:-1], lams[1:]):
        of.euler(p, q)
        fl.step(q)
    exp = oracle_to_gpu(of, lat, of.get_state()[1], fl.n_comp)
    got = fl.get_state()[1].cpu().numpy().reshape(exp.shape)
    for c in range(fl.n_comp):
        assert np.abs(got[:, :, c] - exp[:, :, c]).max() <= (1e-3 if mixed else 1e-10) * np.abs(exp[:, :, c]).max(), c
    fl.close()


@pytest.mark.parametrize("name,L,N", [("square", 3, 8), ("kagome", 2, 7), ("honeycomb_hk", 2, 6)])
def test_stored_state_adjoint(name, L, N):
    import torch
    lams = W.lambda_list(8.0, 1.0, 5)
    _, fl = _flow(name, L, N, lams, mixed=False)
    for lam in lams[1:]:
        fl.step(lam)
    rng = np.random.default_rng(2)
    fs, fG = (torch.tensor(rng.normal(size=n), device="cuda") for n in (fl.N, fl.n_gamma))
    packed = fl.rhs_adjoint(lams[-1], fs, fG)
    fl.packed = False
    for x, y in zip(fl.rhs_adjoint(lams[-1], fs, fG), packed):
        assert _rel(x, y) <= 1e-12
    fl.packed = True
    for x, y in zip(fl.rhs_adjoint(lams[-1], fs, fG), packed):
        assert _rel(x, y) <= 1e-12
    fl.close()


@pytest.mark.parametrize("mode,autotune", [(0, True), (1, True), (1, False), (2, False)])
def test_batch_takes_flows_on_the_stored_state(mode, autotune):
    import paper_2109_13317_gb300 as sr
    lams = W.lambda_list(8.0, 0.5, 8)
    cases = [("square", 2, 7, False), ("kagome", 3, 5, False), ("square", 3, 6, True), ("honeycomb_hk", 2, 5, False),
             ("honeycomb_hk", 1, 6, True), ("kagome_dm", 1, 4, False), ("honeycomb_hkg", 1, 4, True)]
    single = [_flow(n, L, N, lams, packed=p)[1] for n, L, N, p in cases]
    flows = [_flow(n, L, N, lams, packed=p)[1] for n, L, N, p in cases]
    for fl in single:
        for lam in lams[1:]:
            fl.step(lam)
    b = sr.Batch(flows)
    with pytest.raises(sr.SrError):     # the batch holds the buffers
        flows[2].packed = False
    b.force_launch(mode)
    b.run(lams, use_graph=True, autotune=autotune)
    for f1, f2 in zip(single, flows):
        for x, y in zip(f1.get_state(), f2.get_state()):
            assert _rel(y, x) <= 1e-5
    b.close()
    flows[2].packed = False
    for f in single + flows:
        f.close()


def test_mesh_beyond_31_bits_of_packed_values():
    """The largest meshes keep the packed form: its offsets count chunks of four values."""
    import torch

    import paper_2109_13317_gb300 as sr
    N, lam = 256, 0.7
    lat = sr.Lattice.from_model(MODELS["kagome"](), 7)
    mesh = sr.sr_frequency_mesh_exponential(N, 0.05, 20.0)
    fl = sr.Flow(lat, mesh, lam, sr.SR_FP32_MIXED)
    sr.Batch([fl]).close()
    assert 2 * 2 * (2 * lat.N_s) * N * fl.npair >= 2 ** 31
    assert fl.packed
    gen = torch.Generator(device="cuda").manual_seed(4)
    G = torch.randn(fl.n_gamma, dtype=torch.float64, device="cuda", generator=gen)
    G.view(fl.shape())[[i * (i + 3) // 2 for i in range(N)], :, 0] = 0.0    # no density at s = u
    fl.set_state(lam, torch.tensor(0.2 * np.tanh(mesh), device="cuda"), G)
    out = []
    for packed in (True, False):
        fl.packed = packed
        ds = torch.empty(N, dtype=torch.float64, device="cuda")
        fl.rhs_pairs(lam, fl.npair - 2, fl.npair, ds, G)    # (the flow has its own copy of the state)
        out.append(G.view(fl.shape())[-2:].clone())
    # as test_gpu_pair.py: rounding of 6e-8 per product, at most linearly over ~1e3 terms of an output
    for c in range(2):
        assert _rel(out[0][:, :, c], out[1][:, :, c]) <= 1e-4
    fl.close()


@pytest.mark.parametrize("mixed", [False, True])
def test_workspace_takes_the_room_of_the_packed_state(mixed):
    """A Dormand-Prince workspace that finds no memory beside the packed state takes its room; one that
    does not fit either way fails and leaves the flow as it was."""
    import gc

    import torch

    import paper_2109_13317_gb300 as sr
    mib = 1 << 20
    lat = sr.Lattice.from_model(MODELS["kagome"](), 7)
    mesh = sr.sr_frequency_mesh_exponential(64, 0.05, 20.0)
    prec = sr.SR_FP32_MIXED if mixed else sr.SR_FP64
    ref = sr.Flow(lat, mesh, 3.0, prec)
    ref.step(2.5, sr.SR_RK_FIXED)
    ref.packed = False           # (both forms' kernels are loaded before memory runs short)
    ref.step(2.4, sr.SR_RK_FIXED)
    ref.close()
    ref = sr.Flow(lat, mesh, 3.0, prec)
    ref.step(2.5, sr.SR_RK_FIXED)
    exp = [x.cpu() for x in ref.get_state()]
    ref.close()
    fl = sr.Flow(lat, mesh, 3.0, prec)
    part = (8 * fl.n_gamma + 2 * mib - 1) // (2 * mib) * 2 * mib
    spare = 40 * mib if mixed else 140 * mib       # less than the packed state gives back

    def hog(free):
        gc.collect()
        torch.cuda.empty_cache()
        return torch.empty(torch.cuda.mem_get_info()[0] - free, dtype=torch.uint8, device="cuda")

    h = hog(4 * part)
    try:
        with pytest.raises(sr.SrError):
            fl.step(2.5, sr.SR_RK_FIXED)
    finally:
        del h
    assert fl.packed
    h = hog(9 * part - spare)
    try:
        fl.step(2.5, sr.SR_RK_FIXED)
    finally:
        del h
        torch.cuda.empty_cache()
    assert not fl.packed
    for x, y in zip(fl.get_state(), exp):
        assert _rel(x.cpu(), y) <= (1e-5 if mixed else 1e-12)
    fl.close()
