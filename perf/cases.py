"""What the flow library is timed and checked on: right-hand sides, Euler steps with the structure
factor, the adjoint of a step and a batched sweep, over the three spin cores, both precisions and
the range of lattices, frequency meshes and cutoffs the flows run through.

The models are the ones the package is used for: the square J1-J2, kagome and pyrochlore Heisenberg
antiferromagnets (SU2 core), the honeycomb Heisenberg-Kitaev model (XYZ) and the kagome
Dzyaloshinskii-Moriya and honeycomb Kitaev-Gamma models (TRI).  A case starts from a vertex in the
middle of a flow, Gamma^{mu nu}_{ij}(s, t, u) = sum_f phi_f(s, t, u) M_f^{mu nu}_{ij}: the M_f are
built from powers of the model's own coupling matrix (so every lattice and spin symmetry holds) and
the phi_f are smooth functions on the scale of the cutoff with the frequency symmetries of the
parametrization; the seed sets their amplitudes.  Vertices and correlations of FP32-mixed flows
are handed on in single precision, the precision of their vertex integrals.  ``exact`` evaluates the same equations from that
form: interpolation and the frequency sums act on phi_f, the Pauli algebra and the lattice sums on
M_f, in 64 bits.
"""
import math
from functools import lru_cache

import numpy as np
import torch

import paper_2109_13317_gb300 as sr

S3 = math.sqrt(3.0)

# unit cells: primitive vectors, basis positions, bonds (from, to, cell offset)
CELLS = {
    "square": ([[1, 0, 0], [0, 1, 0], [0, 0, 1]], [[0, 0, 0]], [(0, 0, 1, 0, 0), (0, 0, 0, 1, 0)]),
    "honeycomb": ([[1.5, S3 / 2, 0], [1.5, -S3 / 2, 0], [0, 0, 1]], [[0, 0, 0], [1, 0, 0]],
                  [(0, 1, 0, 0, 0), (1, 0, 1, 0, 0), (1, 0, 0, 1, 0)]),
    "kagome": ([[2, 0, 0], [1, S3, 0], [0, 0, 1]], [[0, 0, 0], [1, 0, 0], [0.5, S3 / 2, 0]],
               [(0, 1, 0, 0, 0), (0, 2, 0, 0, 0), (1, 2, 0, 0, 0),
                (1, 0, 1, 0, 0), (2, 0, 0, 1, 0), (2, 1, -1, 1, 0)]),
    "pyrochlore": ([[0, 0.5, 0.5], [0.5, 0, 0.5], [0.5, 0.5, 0]],
                   [[0, 0, 0], [0, 0.25, 0.25], [0.25, 0, 0.25], [0.25, 0.25, 0]],
                   [(0, 1, 0, 0, 0), (0, 2, 0, 0, 0), (0, 3, 0, 0, 0),
                    (1, 2, 0, 0, 0), (1, 3, 0, 0, 0), (2, 3, 0, 0, 0),
                    (0, 1, -1, 0, 0), (0, 2, 0, -1, 0), (0, 3, 0, 0, -1),
                    (1, 2, 1, -1, 0), (1, 3, 1, 0, -1), (2, 3, 0, 1, -1)]),
}
MODELS = {"square_j1j2": ("square", "SU2"), "kagome_j1": ("kagome", "SU2"), "pyrochlore_j1": ("pyrochlore", "SU2"),
          "honeycomb_hk": ("honeycomb", "XYZ"), "honeycomb_hkg": ("honeycomb", "TRI"), "kagome_dm": ("kagome", "TRI")}
BACKEND = {"SU2": sr.SR_SU2, "XYZ": sr.SR_XYZ, "TRI": sr.SR_TRI}
N_COMP = {"SU2": 2, "XYZ": 4, "TRI": 16}


def couplings(model, g):
    """Interactions (from, to, 3 x 3 matrix) of a model; g: its second coupling (J2, K, D or Gamma)."""
    cell = MODELS[model][0]
    eye = np.eye(3)
    if model == "honeycomb_hk" or model == "honeycomb_hkg":
        out = []
        for c, to in enumerate([(0, 0, 0, 1), (0, -1, 0, 1), (-1, 0, 0, 1)]):
            M = 0.2 * eye
            M[c, c] += g if model == "honeycomb_hk" else -1.0
            if model == "honeycomb_hkg":
                a, b = [x for x in range(3) if x != c]
                M[a, b] += g
                M[b, a] += g
            out.append(((0, 0, 0, 0), to, M))
        return out
    if model == "kagome_dm":
        M = np.array([[1.0, g, 0.0], [-g, 1.0, 0.0], [0.0, 0.0, 1.0]])
        directed = [((0, 0, 0, 1), (0, 0, 0, 0)), ((0, 0, 0, 0), (0, 0, 0, 2)), ((-1, 0, 0, 1), (0, 0, 0, 0)),
                    ((0, 0, 0, 0), (0, -1, 0, 2)), ((0, 0, 0, 2), (0, 0, 0, 1)), ((0, -1, 0, 2), (-1, 0, 0, 1))]
        return [(f, t, M) for f, t in directed]
    out = [((0, 0, 0, f), (a, b, c, t), eye) for f, t, a, b, c in CELLS[cell][2]]
    if model == "square_j1j2" and g:
        out += [((0, 0, 0, 0), (1, 1, 0, 0), g * eye), ((0, 0, 0, 0), (1, -1, 0, 0), g * eye)]
    return out


# ---- the cases -----------------------------------------------------------------------------------

def case(name, what, model, g, L, n_freq, w_min, w_max, lam, ratio=0.98, mixed=False, kgrid=0):
    c = {"what": what, "model": model, "g": g, "L": L, "n_freq": n_freq, "w_min": w_min, "w_max": w_max,
         "lam": lam, "ratio": ratio, "mixed": mixed, "kgrid": kgrid}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest run of the README: every step of a short-range square flow, with its structure factor
        case("square_J1_L3_step", "step", "square_j1j2", 0.0, 3, 16, 0.005, 50.0, 1.1, 0.933, kgrid=16),
        # the headline workload's right-hand side in 64 bits (each stage of an adaptive flow is one)
        case("square_J1J2_L7_rhs", "rhs", "square_j1j2", 0.5, 7, 48, 0.001, 100.0, 0.87),
        # the same flow FP32-mixed, one Euler step and chi(k) on the 64 x 64 grid it is plotted on
        case("square_J1J2_L7_mixed", "step", "square_j1j2", 0.5, 7, 48, 0.001, 100.0, 0.87, mixed=True, kgrid=64),
        # a ragged kagome mesh in 64 bits: odd number of frequencies, exchange of inequivalent pairs
        case("kagome_L5_N37_step", "step", "kagome_j1", 0.0, 5, 37, 0.005, 50.0, 0.31, kgrid=33),
        # the three-dimensional lattice, the largest vertex of the configurations
        case("pyrochlore_L6_mixed_rhs", "rhs", "pyrochlore_j1", 0.0, 6, 64, 0.001, 100.0, 1.3, mixed=True),
        # the anisotropic core: right-hand side, FP32-mixed step, and the adjoint step of its gradient runs
        case("honeycomb_HK_L5_rhs", "rhs", "honeycomb_hk", -1.0, 5, 32, 0.005, 50.0, 0.5),
        case("honeycomb_HK_L5_mixed", "step", "honeycomb_hk", -1.0, 5, 32, 0.005, 50.0, 0.5, 0.966, mixed=True, kgrid=33),
        case("honeycomb_HK_L5_adjoint", "adjoint", "honeycomb_hk", -1.0, 5, 32, 0.005, 50.0, 0.5, 0.966),
        # all 16 basis functions: the Dzyaloshinskii-Moriya example at its range, a 64-bit right-hand
        # side at a smaller one, and symmetric off-diagonal couplings, which leave no component zero
        case("kagome_DM_L7_mixed", "step", "kagome_dm", 0.5, 7, 32, 0.005, 50.0, 0.6, mixed=True),
        case("kagome_DM_L4_rhs", "rhs", "kagome_dm", 0.5, 4, 24, 0.005, 50.0, 0.6),
        case("honeycomb_HKG_L4_mixed", "step", "honeycomb_hkg", 0.5, 4, 24, 0.005, 50.0, 0.6, mixed=True),
        # a coupling sweep: flows of uneven size stepped together
        dict(name="sweep_batch", what="batch", n=6, pick=0, lam=0.7, ratio=0.98),
    ]


def draw(rng):
    """One more case of the same ranges, no larger than the largest listed one."""
    logu = lambda a, b: math.exp(rng.uniform(math.log(a), math.log(b)))  # noqa: E731
    if rng.random() < 0.1:
        return dict(what="batch", n=rng.randint(2, 6), pick=rng.randint(1, 10 ** 6), lam=logu(0.1, 5.0), ratio=0.98)
    model = rng.choice(sorted(MODELS))
    core = MODELS[model][1]
    g = round({"square_j1j2": rng.uniform(0.0, 1.0), "honeycomb_hk": rng.uniform(-1.5, -0.5),
               "honeycomb_hkg": rng.uniform(0.2, 0.8), "kagome_dm": rng.uniform(0.1, 0.6)}.get(model, 0.0), 3)
    mixed = rng.random() < 0.5
    what = "adjoint" if core == "XYZ" and not mixed and rng.random() < 0.3 else rng.choice(["step", "rhs"])
    top_L = {"square": 9, "honeycomb": 6, "kagome": 7, "pyrochlore": 6}[MODELS[model][0]]
    top_n = {"SU2": 64, "XYZ": 40, "TRI": 32}[core]
    L = rng.randint(2, top_L)
    n = int(round(logu(10, top_n)))
    # the sizes whose single pass would cost more than the largest listed case
    if core == "TRI" and not mixed:
        L, n = min(L, 4), min(n, 24)
    elif model == "honeycomb_hkg":
        L = min(L, 5)
    elif model == "kagome_dm":
        n = min(n, 26 if L == 7 else 30)
    elif model == "pyrochlore_j1" and not mixed:
        L, n = min(L, 4), min(n, 40)
    elif model == "kagome_j1" and not mixed:
        L = min(L, 6)
    if what == "adjoint":
        L, n = min(L, 5), min(n, 32)
    w_min, w_max = rng.choice([(0.005, 50.0), (0.001, 100.0)])
    return case(None, what, model, g, L, n, w_min, w_max, round(logu(0.05, 20.0), 4), rng.choice([0.98, 0.966]), mixed,
                rng.choice([0, 16, 33, 64]) if what == "step" and core != "TRI" else 0)


def batch_instances(c):
    """The flows of a sweep: three in four square J1-J2, the rest kagome, uneven ranges and meshes."""
    rng = np.random.default_rng(c["pick"])
    out = []
    for i in range(c["n"]):
        square = i % 4 != 3
        out.append(case(None, "step", "square_j1j2" if square else "kagome_j1", round(float(rng.uniform(0, 1)), 3) if square else 0.0,
                        int(rng.integers(5, 8)) if square else int(rng.integers(4, 7)), int(rng.integers(32, 49)), 0.005, 50.0,
                        c["lam"], c["ratio"], True))
    return out


# ---- lattice geometry and the state --------------------------------------------------------------

@lru_cache(maxsize=64)
def geometry(model, g, L):
    """(sites, representatives, K): the sites within L bonds of the reference site in breadth-first
    order, the index of each irreducible site's representative (the first of its orbit under the
    symmetries of lattice and couplings), and per basis site b the powers K[b][n] (box of cells,
    basis, 3, 3) of the coupling matrix, scaled to a largest entry of one."""
    cell, core = MODELS[model]
    prim, basis, bonds = (np.asarray(x, dtype=float) for x in CELLS[cell])
    bonds = bonds.astype(int)
    nb = len(basis)
    links = [(f, t, (a, b, c)) for f, t, a, b, c in bonds] + [(t, f, (-a, -b, -c)) for f, t, a, b, c in bonds]

    def near(b0):
        depth, order = {(0, 0, 0, b0): 0}, [(0, 0, 0, b0)]
        for s in order:
            if depth[s] == L:
                continue
            for f, t, a, b, c in bonds:
                for x, y, sg in ((f, t, 1), (t, f, -1)):
                    if s[3] == x:
                        m = (s[0] + sg * a, s[1] + sg * b, s[2] + sg * c, y)
                        if m not in depth:
                            depth[m] = depth[s] + 1
                            order.append(m)
        return order

    sites = [near(b) for b in range(nb)]
    J = {}
    for f, t, M in couplings(model, g):
        d = tuple(t[k] - f[k] for k in range(3))
        for key, m in (((f[3], t[3], d), M), ((t[3], f[3], tuple(-x for x in d)), M.T)):
            J[key] = J.get(key, 0) + m
    # symmetries that fix the reference site: isometries of the lattice whose action on the
    # couplings is undone by one permutation (XYZ) or proper signed permutation (TRI) of x, y, z
    spins = [np.eye(3)]
    if core != "SU2":
        spins = [np.eye(3)[list(p)] for p in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))]
    if core == "TRI":
        spins = [np.diag(s) @ p for p in spins for s in np.array(np.meshgrid([1, -1], [1, -1], [1, -1])).T.reshape(-1, 3)]
        spins = [m for m in spins if np.linalg.det(m) > 0]
    inv = np.linalg.inv(prim)                       # cell coordinates of x: x @ inv
    cand = np.array(np.meshgrid(*[np.arange(-2, 3)] * 3)).T.reshape(-1, 3)
    gram, group = prim @ prim.T, []
    imgs = [cand[np.abs((cand @ prim) ** 2 @ np.ones(3) - gram[k, k]) < 1e-6] for k in range(3)]
    for a in imgs[0]:
        for b in imgs[1]:
            for c in imgs[2]:
                V = np.array([a, b, c]) @ prim
                if np.abs(V @ V.T - gram).max() > 1e-6:
                    continue
                O = (inv @ V)                       # row vectors: x -> x @ O, about basis site 0
                act = []
                for p in basis:
                    y = (p - basis[0]) @ O + basis[0]
                    hit = [(q, np.rint((y - basis[q]) @ inv).astype(int)) for q in range(nb)
                           if np.abs((y - basis[q]) @ inv - np.rint((y - basis[q]) @ inv)).max() < 1e-6]
                    act.append(hit[0] if hit else None)
                if any(x is None for x in act):
                    continue
                R = np.array([a, b, c])

                def image(s, R=R, act=act):
                    q, m = act[s[3]]
                    n = np.array(s[:3]) @ R + m
                    return (int(n[0]), int(n[1]), int(n[2]), q)

                def pair(f, t, d):
                    i, j = image((0, 0, 0, f)), image((d[0], d[1], d[2], t))
                    return i[3], j[3], tuple(j[k] - i[k] for k in range(3))

                if any(pair(*x) not in {(f, t, d) for f, t, d in links} for x in links):
                    continue
                moved = {k: J.get(pair(*k)) for k in J}
                if any(m is None for m in moved.values()):
                    continue
                if any(all(np.abs(moved[k] - s @ J[k] @ s.T).max() < 1e-5 for k in J) for s in spins):
                    group.append(image)
    at = {s: i for i, s in enumerate(sites[0])}
    seen, reps = set(), []
    for i, s in enumerate(sites[0]):
        if i in seen:
            continue
        reps.append(i)
        seen |= {at[h(s)] for h in group}
    # powers of the coupling matrix from each basis site
    flat = [0 if all(k[2][x] == 0 for k in J) and all(b[2 + x] == 0 for b in bonds) else L + 1 for x in range(3)]
    box = [2 * f + 1 for f in flat]
    K = []
    for b in range(nb):
        cur = np.zeros((*box, nb, 3, 3))
        cur[flat[0], flat[1], flat[2], b] = np.eye(3)
        powers = [cur]
        for _ in range(L):
            nxt = np.zeros_like(cur)
            for (f, t, d), M in J.items():
                src = cur[:, :, :, f] @ M
                # cells shifted by d; what leaves the box lies beyond the range
                to = tuple(slice(max(0, x), n + min(0, x)) for x, n in zip(d, box))
                fr = tuple(slice(max(0, -x), n + min(0, -x)) for x, n in zip(d, box))
                nxt[(*to, t)] += src[fr]
            cur = nxt
            powers.append(cur)
        K.append(powers)
    for n in range(L + 1):
        big = max(np.abs(K[b][n]).max() for b in range(nb))
        for b in range(nb):
            K[b][n] = K[b][n] / big
    return sites, reps, K, flat, J


IMAG = np.array([[(m == 0) != (n == 0) for n in range(4)] for m in range(4)])


def matrices(model, g, L, b, d, bj):
    """The real 4 x 4 matrices M_f of the pair ((0, b), (d, bj)): per power n of the coupling matrix
    the spin-spin part, the density part and, for TRI, the two density-spin parts."""
    core = MODELS[model][1]
    _, _, K, flat, _ = geometry(model, g, L)
    out = []
    for n in range(L + 1):
        k = K[b][n][d[0] + flat[0], d[1] + flat[1], d[2] + flat[2], bj]
        m = np.zeros((4 if core == "TRI" else 2, 4, 4))
        m[0, 1:, 1:] = k
        m[1, 0, 0] = np.trace(k) / 3
        if core == "TRI":
            v = np.array([k[1, 2] - k[2, 1], k[2, 0] - k[0, 2], k[0, 1] - k[1, 0]])
            m[2, 0, 1:] = v
            m[3, 1:, 0] = v
        out.append(m)
    return np.concatenate(out)


def parities(model, L):
    """Signs of the phi_f: under s <-> u, and under t -> -t (and u -> -u)."""
    n = 4 if MODELS[model][1] == "TRI" else 2
    return np.array(([1, -1, 1, -1][:n]) * (L + 1)), np.array(([1, 1, -1, -1][:n]) * (L + 1))


def mesh_of(c):
    n = c["n_freq"]
    return c["w_min"] * (c["w_max"] / c["w_min"]) ** (np.arange(n) / (n - 1))


def frequency_parts(c, w, seed, device):
    """phi_f on the whole mesh cube [s, t, u, f] (the half s < u by the s <-> u relation) and gamma."""
    rng = np.random.default_rng([seed, 77])
    model, L, lam = c["model"], c["L"], c["lam"]
    tri = MODELS[model][1] == "TRI"
    W = torch.as_tensor(w, dtype=torch.float64, device=device)
    S, T, U = W[:, None, None], W[None, :, None], W[None, None, :]
    tot = S + T + U + lam
    shape1 = lam / (lam + 0.5 * (S + U) + T)
    shape2 = torch.exp(-(S + U) / (lam + T))
    big = max(np.abs(m).max() for m in geometry(model, c["g"], L)[4].values())
    parts = []
    for n in range(L + 1):
        a = rng.normal(size=6) * 0.25 * math.exp(-0.45 * n)
        spin = a[0] * shape1 + 0.3 * a[1] * shape2
        if n == 1:
            spin = spin + big / 4          # the bare vertex J / 4
        parts += [spin, 0.5 * a[2] * (S - U) / tot]
        if tri:
            parts += [0.4 * a[3] * T * lam / tot ** 2, 0.4 * a[4] * T * (S - U) / tot ** 2]
    gam = lam * rng.uniform(0.1, 0.25) * torch.tanh(W / lam) + 0.05 * lam * W / (lam + W)
    return torch.stack([p.expand(len(w), len(w), len(w)) for p in parts], -1), gam


def stored(c, w, seed, device="cuda"):
    """The state in the library's layout: gamma(w), Gamma[pair(s, u)][t][component][site]."""
    core = MODELS[c["model"]][1]
    sites, reps, _, _, _ = geometry(c["model"], c["g"], c["L"])
    phi, gam = frequency_parts(c, w, seed, device)
    M = np.stack([matrices(c["model"], c["g"], c["L"], 0, sites[0][i][:3], sites[0][i][3]) for i in reps], -1)
    M = torch.as_tensor(components(M, core), device=device)                      # f, component, site
    i = torch.tril_indices(len(w), len(w), device=device)
    G = torch.tensordot(phi[i[0], :, i[1]], M, dims=1)                           # pair, t, component, site
    return gam.contiguous(), G.reshape(-1).contiguous()


def components(M, core):
    """Stored components of (f, 4, 4, site) arrays."""
    if core == "TRI":
        return M.reshape(M.shape[0], 16, -1)
    k = [0, 3] if core == "SU2" else [0, 1, 2, 3]
    return np.stack([M[:, a, a] for a in k], 1)


# ---- a user's program ----------------------------------------------------------------------------

def kpoints(n):
    x = np.linspace(-2 * np.pi, 2 * np.pi, n)
    return np.stack([*[k.ravel() for k in np.meshgrid(x, x, indexing="ij")], np.zeros(n * n)], 1)


def make_flow(c):
    cell, core = MODELS[c["model"]]
    prim, basis, bonds = CELLS[cell]
    lat = sr.Lattice(prim, basis, bonds, couplings(c["model"], c["g"]), c["L"], BACKEND[core])
    assert lat.N_s == len(geometry(c["model"], c["g"], c["L"])[1])
    mesh = sr.sr_frequency_mesh_exponential(c["n_freq"], c["w_min"], c["w_max"])
    return sr.Flow(lat, mesh, c["lam"], sr.SR_FP32_MIXED if c["mixed"] else sr.SR_FP64)


def prepare(c, seed):
    cs = batch_instances(c) if c["what"] == "batch" else [c]
    flows = [make_flow(x) for x in cs]
    st = {"what": c["what"], "mixed": c.get("mixed", c["what"] == "batch"), "lam": c["lam"], "next": c["lam"] * c["ratio"], "flows": flows,
          "states": [stored(x, f.mesh, seed + 1000 * i) for i, (x, f) in enumerate(zip(cs, flows))]}
    st["k"] = kpoints(c["kgrid"]) if c.get("kgrid") else None
    if c["what"] == "batch":
        st["batch"] = sr.Batch(flows)
    if c["what"] == "adjoint":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        f = flows[0]
        st["bar"] = [torch.randn(n, dtype=torch.float64, device="cuda", generator=gen) for n in (f.N, f.n_gamma)]
        st["out"] = [torch.empty_like(x) for x in st["bar"]]
        f.set_state(c["lam"], *st["states"][0])
    elif c["what"] == "rhs":
        flows[0].set_state(c["lam"], *st["states"][0])
    return st


def run(st):
    f = st["flows"][0]
    if st["what"] == "adjoint":
        return f.step_adjoint(st["lam"], st["next"], *st["bar"], *st["out"])
    if st["what"] == "rhs":
        return handed_on(st, f.rhs(st["lam"]))
    for g, (gam, G) in zip(st["flows"], st["states"]):
        g.set_state(st["lam"], gam, G)
    if st["what"] == "batch":
        st["batch"].run([st["lam"], st["next"]], use_graph=False, autotune=False)
        return [handed_on(st, g.get_state()) for g in st["flows"]]
    f.step(st["next"], sr.SR_EULER)
    out = handed_on(st, f.get_state())
    if st["k"] is not None:
        chi_k, chi_ij = f.measure(st["k"])
        out += [chi_k.astype(np.float32), chi_ij.float()] if st["mixed"] else [chi_k, chi_ij]
    return out


def handed_on(st, parts):
    return [parts[0], parts[1].float() if st["mixed"] else parts[1]]


# ---- what a pass cannot do without ---------------------------------------------------------------

def nodes_of(w, lam, gam=None, dgam=None):
    """Integration points and weights of every channel (s, t, u) and transfer frequency: the four
    points of the single-scale propagator where the cutoff function is resolved exactly, and the
    trapezoid rule on mesh and break points where both propagators lie above the cutoff.  Without
    gamma, points only."""
    odd = lambda f, x: np.sign(x) * np.interp(np.abs(x), w, f)  # noqa: E731
    out = []
    for ch in range(3):
        sg = 1.0 if ch == 2 else -1.0
        for v in w:
            other = (lambda x: v - x) if ch == 0 else (lambda x: x + sg * v)
            xs, ws = [], []
            for lm in (lam, -lam):
                # the point where the other propagator, or this one, carries the delta function
                first = v - lm if ch == 0 else lm - sg * v
                for x, partner in ((first, first), (lm, other(lm))):
                    xs.append(x)
                    keep = abs(partner) >= lam
                    if gam is None:
                        ws.append(float(keep))
                    else:
                        ws.append(-1.0 / ((partner + odd(gam, partner)) * (lm + odd(gam, lm))) / (2 * np.pi) if keep else 0.0)
            lim = {0: (v + lam, v - lam), 1: (v + lam, v - lam), 2: (lam - v, -v - lam)}[ch]
            p = np.sort(np.concatenate([-w, w, np.clip([lam, -lam, *lim], -w[-1], w[-1])]))
            mid, h = 0.5 * (p[1:] + p[:-1]), np.diff(p)
            seg = np.where((h > 0) & (np.abs(mid) >= lam) & (np.abs(other(mid)) >= lam), 0.5 * h, 0.0)
            q = np.concatenate([seg, [0.0]]) + np.concatenate([[0.0], seg])
            p, q = p[q != 0], q[q != 0]
            if gam is not None:
                y = other(p)
                gx, gy = p + odd(gam, p), y + odd(gam, y)
                q = q * -(odd(dgam, y) / (gx * gy * gy) + odd(dgam, p) / (gy * gx * gx)) / (2 * np.pi)
            out.append((np.concatenate([xs, p]), np.concatenate([ws, q])))
    return out


@lru_cache(maxsize=64)
def lattice_sum_terms(model, g, L):
    """Pairs (representative, j) with j within range of both sites."""
    sites, reps, _, _, _ = geometry(model, g, L)
    near = [{s: 1 for s in x} for x in sites]
    n = 0
    for i in reps:
        r = sites[0][i]
        n += sum((r[0] - s[0], r[1] - s[1], r[2] - s[2], r[3]) in near[s[3]] for s in sites[0])
    return n


def work(c):
    if c["what"] == "batch":
        all_ = [work(x) for x in batch_instances(c)]
        return {k: sum(x[k] for x in all_) for k in ("bytes", "flops")}
    w, core = mesh_of(c), MODELS[c["model"]][1]
    N, nc = len(w), N_COMP[core]
    Ns, P = len(geometry(c["model"], c["g"], c["L"])[1]), lattice_sum_terms(c["model"], c["g"], c["L"])
    cnt = np.array([len(x) for x, _ in nodes_of(w, c["lam"])]).reshape(3, N)
    i = np.arange(N)
    triples = np.stack([(i + 1) * N, np.full(N, N * (N + 1) // 2), (N - i) * N])   # triples at each transfer frequency
    nodes = (cnt * triples).sum(1)
    row = 2 * 4 * 2 * Ns * nc                               # two rows of four corners, one FMA each
    site = {"SU2": 11, "XYZ": 32, "TRI": 128}[core] * Ns    # products of two pair operators
    one = {"SU2": 4, "XYZ": 4, "TRI": 16}[core] * Ns * nc   # the two on-site terms
    # lattice sum: each distinct pair of sites once (two-component core), else the table's products
    lat = 2 * nc * min(P, Ns * Ns) if core == "SU2" else {"XYZ": 2 * 4, "TRI": 2 * 64}[core] * P
    flops = (nodes[0] + nodes[2]) * (row + site) + nodes[1] * (row + one + lat)
    entries = N * (N + 1) // 2 * N * nc * Ns
    if c["what"] == "adjoint":
        return {"bytes": 8.0 * 3 * entries, "flops": 3.0 * flops}   # the rows again, and both factors' adjoints
    return {"bytes": 8.0 * 2 * entries, "flops": float(flops)}


# ---- the same in 64 bits, from phi_f and M_f -----------------------------------------------------

PAULI = np.array([[[1, 0], [0, 1]], [[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]])
PP = np.einsum("aij,bjk,cki->abc", PAULI, PAULI, PAULI) / 2                       # sigma^a sigma^b -> sigma^c
PPPP = np.einsum("aij,bjk,ckl,dli->abcd", PAULI, PAULI, PAULI, PAULI) / 2


class Exact:
    """Right-hand side and correlations of a state given by phi_f and M_f."""

    def __init__(self, c, seed):
        self.c, self.dev = c, "cuda" if torch.cuda.is_available() else "cpu"
        self.w = mesh_of(c)
        self.N, self.L, self.core = len(self.w), c["L"], MODELS[c["model"]][1]
        self.cube, gam = frequency_parts(c, self.w, seed, self.dev)
        self.gam = gam.cpu().numpy()
        self.F = self.cube.shape[-1]
        ex, self.mixed = parities(c["model"], c["L"])
        # s < u reads sign * (u, t, s)
        lower = torch.tril(torch.ones(self.N, self.N, dtype=torch.bool, device=self.dev))[:, None, :, None]
        flipped = self.cube.transpose(0, 2) * torch.as_tensor(ex, dtype=torch.float64, device=self.dev)
        self.cube = torch.where(lower, self.cube, flipped).reshape(self.N ** 3, self.F)
        self.mixed = torch.as_tensor(self.mixed, dtype=torch.float64, device=self.dev)
        self.wt = torch.as_tensor(self.w, device=self.dev)

    def M(self, b, d, bj):
        return matrices(self.c["model"], self.c["g"], self.L, b, d, bj) * np.where(IMAG, 1j, 1.0)

    def axis(self, x):
        x = x.clamp(self.wt[0], self.wt[-1])
        k = (torch.searchsorted(self.wt, x.contiguous(), right=True) - 1).clamp(0, self.N - 2)
        f = (x - self.wt[k]) / (self.wt[k + 1] - self.wt[k])
        return k, f

    def lookup(self, s, t, u):
        """Coefficients of the M_f(ij) in Gamma_ij(s, t, u)."""
        swap, neg = (s < 0) ^ (u < 0), (t < 0) ^ (u < 0)
        s, t, u = torch.broadcast_tensors(s.abs(), t.abs(), u.abs())
        (ks, fs), (kt, ft), (ku, fu) = self.axis(s), self.axis(t), self.axis(u)
        out = 0
        for a in range(2):
            for b in range(2):
                for d in range(2):
                    wt = (fs if a else 1 - fs) * (ft if b else 1 - ft) * (fu if d else 1 - fu)
                    out = out + wt[..., None] * self.cube[((ks + a) * self.N + kt + b) * self.N + ku + d]
        if self.core == "TRI":
            # exchanged sites: the transpose of M_f(ji), which swaps the two density-spin parts
            # with a minus sign (they are odd under the exchange) and leaves the others
            v = out.unflatten(-1, (-1, 4))
            ex = torch.cat([v[..., :2], -v[..., 3:], -v[..., 2:3]], -1).flatten(-2)
            out = torch.where(swap[..., None], ex, out)
            out = torch.where(neg[..., None], out * self.mixed, out)
        return out

    def pairs(self):
        sites, reps, _, _, _ = geometry(self.c["model"], self.c["g"], self.L)
        return sites, [sites[0][i] for i in reps]

    def sigma(self):
        """d gamma / d Lambda."""
        lam, sites = self.c["lam"], self.pairs()[0]
        hartree = sum(self.M(0, s[:3], s[3])[:, 0, 0] for s in sites[0]).real
        fock = np.trace(self.M(0, (0, 0, 0), 0), axis1=1, axis2=2).real
        z = torch.zeros_like(self.wt)
        out = 0
        for w2 in (lam, -lam):
            a = self.lookup(self.wt + w2, z, self.wt - w2).cpu().numpy() @ hartree
            b = self.lookup(self.wt + w2, w2 - self.wt, z).cpu().numpy() @ fock
            out = out - (2 * a - b) / (w2 + math.copysign(np.interp(lam, self.w, self.gam), w2)) / (2 * np.pi)
        return out

    def structure(self):
        """Per irreducible site and component: the bilinear forms of the s, u and t channels."""
        sites, reps = self.pairs()
        near = [set(x) for x in sites]
        real = np.where(IMAG, -1j, 1.0)
        D = self.M(0, (0, 0, 0), 0)
        out = {k: [] for k in ("s", "u", "lat", "o2", "o3")}
        for r in reps:
            A = self.M(0, r[:3], r[3])
            E = self.M(r[3], (0, 0, 0), r[3])
            out["s"].append(np.einsum("fab,gcd,acm,bdn->fgmn", A, A, PP, PP, optimize=True) * real)
            out["u"].append(np.einsum("fab,gcd,cam,bdn->fgmn", A, A, PP, PP, optimize=True) * real)
            out["o2"].append(np.einsum("fml,gab,albn->fgmn", A, E, PPPP, optimize=True) * real)
            out["o3"].append(np.einsum("fkl,gan,lakm->fgmn", D, A, PPPP, optimize=True) * real)
            js = [s for s in sites[0] if (r[0] - s[0], r[1] - s[1], r[2] - s[2], r[3]) in near[s[3]]]
            X = np.stack([self.M(0, s[:3], s[3]) for s in js])
            Y = np.stack([self.M(s[3], (r[0] - s[0], r[1] - s[1], r[2] - s[2]), r[3]) for s in js])
            X = X.transpose(1, 2, 0, 3).reshape(self.F * 4, -1)
            Y = Y.transpose(0, 2, 1, 3).reshape(-1, self.F * 4)
            out["lat"].append((X @ Y).reshape(self.F, 4, self.F, 4).transpose(0, 2, 1, 3) * real)
        res = {}
        for k, v in out.items():
            v = np.stack(v, -1).real
            v = components(v.reshape(self.F ** 2, 4, 4, -1), self.core)
            res[k] = torch.as_tensor(v.reshape(self.F ** 2, -1), device=self.dev)
        return res

    def rhs(self):
        N, w = self.N, self.wt
        dgam = self.sigma()
        nodes = nodes_of(self.w, self.c["lam"], self.gam, dgam)
        st = self.structure()
        pi, pu = torch.tril_indices(N, N, device=self.dev)
        npair = len(pi)
        n_out = st["s"].shape[1]
        out = torch.zeros(npair * N, n_out, dtype=torch.float64, device=self.dev)
        idx = torch.arange(npair * N, device=self.dev)
        iS, iT, iU = pi[idx // N], idx % N, pu[idx // N]
        for ch in range(3):
            axis = (iS, iT, iU)[ch]
            for v in range(N):
                rows = (axis == v).nonzero()[:, 0]
                x, wx = (torch.as_tensor(a, device=self.dev) for a in nodes[ch * N + v])
                step = max(1, int(3e7 // (len(x) * self.F)))
                for a in range(0, len(rows), step):
                    k = rows[a:a + step]
                    s, t, u = (w[i[k]][:, None] for i in (iS, iT, iU))
                    w1p, w2p, w1, w2 = (s + t + u) / 2, (s - t - u) / 2, (s - t + u) / 2, (s + t - u) / 2
                    z = torch.zeros_like(x)[None]
                    if ch == 0:
                        A, B = self.lookup(s + z, w1p - x, x - w2p), self.lookup(s + z, x - w1, x - w2)
                    elif ch == 1:
                        A, B = self.lookup(w1 + x, t + z, w1p - x), self.lookup(x + w2p, t + z, x - w2)
                    else:
                        A, B = self.lookup(w1 + x, x - w2p, u + z), self.lookup(w1p + x, w2 - x, u + z)
                    A = A * wx[:, None]
                    bil = lambda p, q: (p.transpose(1, 2) @ q).flatten(1)  # noqa: E731
                    if ch != 1:
                        out[k] += bil(A, B) @ st["s" if ch == 0 else "u"]
                    else:
                        out[k] -= 2 * (bil(A, B) @ st["lat"])
                        C, D = self.lookup(w2p + x, w2 - x, -t + z), self.lookup(w1 + x, x - w1p, -t + z)
                        out[k] += bil(A, C) @ st["o2"] + bil(D * wx[:, None], B) @ st["o3"]
        return torch.as_tensor(dgam, device=self.dev), out.reshape(-1)

    def step(self):
        dg, dG = self.rhs()
        h = self.c["lam"] * (1 - self.c["ratio"])
        gam, G = stored(self.c, self.w, self.seed, self.dev)
        return gam - h * dg, G - h * dG


def exact(c, seed):
    """None where there is no such value: gradients with respect to the stored entries of the
    anisotropic cores depend on which of several symmetry-equivalent entries a lookup reads, and
    chi is that of the state after the step, which the phi_f no longer span."""
    if c["what"] == "adjoint":
        return None
    cs = batch_instances(c) if c["what"] == "batch" else [c]
    res = []
    for i, x in enumerate(cs):
        e = Exact(x, seed + 1000 * i)
        e.seed = seed + 1000 * i
        res.append(list(e.rhs() if c["what"] == "rhs" else e.step()))
    if c["what"] == "batch":
        return res
    return res[0] + ([None, None] if c.get("kgrid") else [])
