"""Performance cases of the enriched finite-element ChFSI library.

Each case is one call (or one short sequence of calls) that a user's program
makes on the public binding: the Chebyshev filter, Rayleigh-Ritz, the SCF step,
the density-to-Hamiltonian update between two filters, the learned initial
density, its training step, and the batched filter.  Geometries are the seeded
stand-ins of the paper's systems (a bare nucleus in a box, a C-O pair, diamond
silicon clusters, random clusters of H/C/O/Si atoms), written out here as the
plain descriptions that ``System`` takes.

A program keeps one ``System`` per geometry and brings new vectors, densities or
network weights to it: ``prepare`` makes those from the seed, the handles of the
last geometries used are kept between calls of ``prepare``.

``exact`` rebuilds the discrete problem in plain 64-bit torch: the operators from
their integrals over the handle's quadrature points (the points are part of the
problem's statement), every product as a dense or batched matrix product.
"""
import collections
import math

import numpy as np
import torch

import paper_1610_02121_gb300 as efe
from paper_1610_02121_gb300 import learned

DEV = "cuda"
F64 = torch.float64
KB = 3.166811563e-6          # Ha per kelvin
A_SI = 10.26                 # lattice constant of the silicon clusters (bohr)


# --------------------------------------------------------------------------- cases
def listed():
    return [
        # a bare nucleus in a 20-bohr box, 6^3 cells, plain FP64: the smallest real
        # eigenproblem, where launches and latency are what a user waits for
        {"name": "filter_nucleus_fp64", "do": "filter", "system": "nucleus", "size": 6, "n": 8, "m": 20,
         "precision": "fp64", "tail": 0, "engine": "dfma"},
        # a diatomic molecule in the mixed precision with the tensor-core FP64 tail: the
        # filter of every SCF iteration of a small molecule
        {"name": "filter_pair_mixed", "do": "filter", "system": "pair", "size": 1.0, "n": 12, "m": 24,
         "precision": "tf32x3", "tail": 2, "engine": "tensor"},
        # the first SCF iteration of the same molecule in plain FP64, as a whole call
        {"name": "scf_pair_fp64", "do": "scf", "system": "pair", "size": 1.0, "n": 12, "m": 12,
         "precision": "fp64", "tail": 0, "engine": "dfma"},
        # the 16-atom silicon cluster at its full mesh (1.5M nodes), 135 vectors, degree 20,
        # mixed: the ordinary production filter
        {"name": "filter_si16_mixed", "do": "filter", "system": "silicon", "size": 0.9, "n": 135, "m": 20,
         "precision": "tf32x3", "tail": 2, "engine": "tensor"},
        # the same cluster on the coarser mesh with every degree FP64-grade: what a user runs
        # to check a mixed result
        {"name": "filter_si16_fp64", "do": "filter", "system": "silicon", "size": 1.6, "n": 135, "m": 6,
         "precision": "fp64", "tail": 0, "engine": "tensor"},
        # Cholesky-QR and Rayleigh-Ritz of that block, with residuals
        {"name": "ritz_si16", "do": "ritz", "system": "silicon", "size": 1.6, "n": 135, "engine": "tensor"},
        # a block of many vectors: the coupling of many functions, column tiles, long rows
        {"name": "filter_wide_mixed", "do": "filter", "system": "silicon", "size": 1.6, "n": 640, "m": 8,
         "precision": "tf32x3", "tail": 2, "engine": "tensor"},
        # its Rayleigh-Ritz: the blocked dense eigensolver
        {"name": "ritz_wide", "do": "ritz", "system": "silicon", "size": 1.6, "n": 640, "engine": "tensor"},
        # density -> Hartree and xc potentials -> new Hamiltonian -> products with it: what
        # an SCF iteration does between two filters
        {"name": "fields_si16", "do": "fields", "system": "silicon", "size": 1.6, "n": 135, "precision": "fp64",
         "cols": 8, "engine": "tensor"},
        # the learned initial density of a cluster: superposed atoms, descriptors, network
        {"name": "start_si16", "do": "start", "system": "silicon", "size": 1.6, "engine": "tensor"},
        # one training step of its network on a minibatch
        {"name": "train_step", "do": "train", "rows": 8192},
        # eight small clusters of 1 to 6 atoms filtered together
        {"name": "batch_clusters", "do": "batch", "system": "clusters", "size": 1.2, "count": 8, "m": 20,
         "precision": "tf32x3", "tail": 2, "engine": "tensor"},
    ]


def draw(rng):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    do = rng.choice(["filter"] * 6 + ["ritz"] * 2 + ["scf", "fields", "start", "train", "batch"])
    if do == "train":
        return {"do": do, "rows": int(log(300, 60000))}
    if do == "batch":
        return {"do": do, "system": "clusters", "size": round(rng.uniform(1.2, 1.5), 2), "count": rng.randint(2, 8),
                "m": rng.randint(6, 20), "precision": rng.choice(["tf32x3", "fp32"]), "tail": rng.randint(0, 2),
                "engine": "tensor"}
    system = rng.choice(["nucleus", "pair", "cluster", "silicon"])
    if do in ("scf", "start") and system == "nucleus":
        system = "pair"
    c = {"do": do, "system": system,
         "size": {"nucleus": rng.randint(4, 9), "pair": round(rng.uniform(0.9, 1.4), 2),
                  "cluster": rng.randint(1, 6), "silicon": round(rng.uniform(1.4, 2.2), 2)}[system],
         "engine": rng.choice(["dfma", "tensor", "tensor"])}
    if do == "start":
        return c
    # vectors: a handful for a nucleus, up to some hundred for the clusters
    lo, hi = {"nucleus": (1, 20), "pair": (9, 300), "cluster": (12, 300), "silicon": (60, 480)}[system]
    c["n"] = int(log(lo, hi))
    if do in ("filter", "scf"):
        c["precision"] = rng.choice(["fp64", "tf32x3", "tf32x3", "fp32"]) if do == "filter" else "fp64"
        c["tail"] = rng.randint(0, 2)
        c["m"] = rng.randint(2, 4) if c["n"] > 64 else rng.randint(5, 24)
    if do == "scf":
        # room for the electrons: two a vector
        c["system"], c["size"] = "pair", round(rng.uniform(0.9, 1.4), 2)
        c["n"], c["m"] = rng.randint(11, 40), rng.randint(8, 14)
    if do == "filter" and rng.random() < 0.3:
        c["ld"] = c["n"] + rng.randint(1, 5)        # columns of a wider block
    if do == "fields":
        c["precision"], c["cols"] = rng.choice(["fp64", "fp32"]), rng.randint(1, 12)
        c["n"] = min(c["n"], 160)
    return c


# --------------------------------------------------------------------------- geometries
def _graded(lo, hi, must, h_min, h_max, growth=1.3, fine=2.0):
    """Break points of one axis: every coordinate in `must`, cells of at most h_min
    between them and `fine` bohr beyond, then growing to h_max at the box faces."""
    must = np.unique(np.round(np.asarray(must, dtype=np.float64), 12))
    inner = [must[0]]
    for a, b in zip(must[:-1], must[1:]):
        k = max(1, int(math.ceil((b - a) / h_min - 1e-9)))
        inner += list(a + (b - a) * np.arange(1, k + 1) / k)

    def outward(dist):
        k = max(1, int(math.ceil(fine / h_min - 1e-9)))
        lens = [fine / k] * k
        while sum(lens) < dist:
            lens.append(min(lens[-1] * growth, h_max))
        return np.cumsum(lens) * (dist / sum(lens))

    return np.concatenate([inner[0] - outward(inner[0] - lo)[::-1], inner, inner[-1] + outward(hi - inner[-1])])


def _exponents(Z):
    """Slater's-rules exponents of 1s and 2s/2p."""
    if Z <= 2:
        return (Z - 0.3 if Z > 1 else 1.0), max(0.5, (Z - 0.85 * (Z - 1)) / 2.0)
    n2 = min(Z - 2, 8)
    return Z - 0.3, (Z - 1.7 - (n2 - 1) * 0.35) / 2.0


def _atoms_system(atoms, Z, h_min, h_max, pad, gaussians, tau, depth, seed):
    rng = np.random.default_rng(seed)
    atoms = np.asarray(atoms, dtype=np.float64).reshape(-1, 3)
    lo, hi = atoms.min(axis=0), atoms.max(axis=0)
    funcs = []
    for ia, z in enumerate(Z):
        z1, z2 = (e * (1.0 + 0.05 * rng.uniform(-1, 1)) for e in _exponents(int(z)))
        for n, l, m, zeta in [(1, 0, 0, z1), (2, 0, 0, z2), (2, 1, -1, z2), (2, 1, 0, z2), (2, 1, 1, z2)]:
            funcs.append({"atom": ia, "n": n, "l": l, "m": m, "kind": "slater", "zeta": zeta, "r0": 2.0, "t": 1.0})
    return {"p": 4, "n_gauss": 6, "atoms": atoms, "Z": np.asarray(Z, dtype=np.float64), "funcs": funcs,
            "breaks": [_graded(lo[d] - pad, hi[d] + pad, atoms[:, d], h_min, h_max) for d in range(3)],
            "potential": {"nuclear": True, "omega": 0.0, "gauss_A": rng.uniform(-0.5, 0.5, gaussians),
                          "gauss_s": rng.uniform(1.0, 3.0, gaussians),
                          "gauss_c": lo + (hi - lo) * rng.uniform(0, 1, (gaussians, 3))},
            "quad": {"tau": tau, "max_depth": depth, "n": 6}}


def _random_cluster(count, h_min, seed):
    rng = np.random.default_rng(seed)
    side = (count / 0.012) ** (1.0 / 3.0)
    pos = []
    while len(pos) < count:
        c = np.round(rng.uniform(0.0, side, 3), 3)
        if all(np.linalg.norm(c - q) >= 3.0 for q in pos):
            pos.append(c)
    return _atoms_system(pos, rng.choice([1.0, 6.0, 8.0, 14.0], count), h_min, 4.0, 7.0, 0, 1e-8, 7, seed + 1)


def _systems(case):
    """The system descriptions of a case."""
    kind, size = case["system"], case["size"]
    if kind == "nucleus":
        b = np.linspace(-10.0, 10.0, int(size) + 1)
        f = [{"atom": 0, "n": n, "l": l, "m": m, "kind": "hydrogenic", "zeta": 0.0, "r0": 3.0, "t": 1.0}
             for n, l, m in [(1, 0, 0), (2, 0, 0), (2, 1, -1), (2, 1, 0), (2, 1, 1)]]
        # the nucleus sits on a mesh vertex (the one nearest the centre)
        at = b[(int(size) + 1) // 2]
        return [{"p": 4, "n_gauss": 6, "atoms": np.full((1, 3), at), "Z": np.ones(1), "funcs": f, "breaks": [b, b, b],
                 "potential": {"nuclear": True, "omega": 0.0, "gauss_A": np.zeros(0), "gauss_s": np.zeros(0),
                               "gauss_c": np.zeros((0, 3))},
                 "quad": {"tau": 1e-8, "max_depth": 8, "n": 6}}]
    if kind == "pair":
        return [_atoms_system([[0.0, 0.0, 0.0], [2.132, 0.0, 0.0]], [6.0, 8.0], size, 3.0, 6.0, 0, 1e-7, 6, 12)]
    if kind == "silicon":
        fcc = [[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]]
        base = np.array(fcc + [[x + .25 for x in p] for p in fcc])
        atoms = np.concatenate([base, base + [1.0, 0.0, 0.0]]) * A_SI
        return [_atoms_system(atoms, [14.0] * 16, size, 3.0 if size < 1.2 else 4.0, 10.0, 32, 1e-7, 7, 2)]
    if kind == "cluster":
        return [_random_cluster(int(size), 1.2, 500 + int(size))]
    return [_random_cluster(1 + (3 * i + 1) % 6, size, 700 + i) for i in range(case["count"])]


_KEPT = collections.OrderedDict()


def _handles(case):
    """The handles of a case's geometries with its potential set, and per handle the
    filter interval (a, b, a0).  The last two geometries are kept, as a program
    keeps its handle while vectors come and go."""
    key = tuple((k, case.get(k)) for k in ("do", "system", "size", "count", "engine"))
    if key in _KEPT:
        _KEPT.move_to_end(key)
        return _KEPT[key]
    while len(_KEPT) > 1:
        _KEPT.popitem(last=False)
    out = []
    for s in _systems(case):
        G = efe.System(s)
        G.set_potential_analytic()
        # the interval, in round numbers: a above the wanted levels, b above the
        # spectrum, a0 below it (the enrichment functions alone give the core levels)
        X = torch.zeros((G.rows, G.n_enrich), dtype=F64, device=DEV)
        X[G.n_nodes:] = torch.eye(G.n_enrich, dtype=F64, device=DEV)
        a0 = math.floor(1.05 * G.rayleigh_ritz(X, residuals=False)[0].min() - 1.0)
        b = G.upper_bound(_block(G, 1, 9, False)[:, 0].contiguous(), 10)
        p = 10.0 ** (math.floor(math.log10(b)) - 1)
        G.set_fp64_engine(case.get("engine", "dfma"))
        out.append((G, (1.0, math.ceil(1.02 * b / p) * p, float(a0))))
    _KEPT[key] = out
    return out


# --------------------------------------------------------------------------- inputs
def _interior(G):
    nx, ny, nz = (4 * (len(b) - 1) + 1 for b in G.system["breaks"])
    m = torch.zeros((nz, ny, nx), dtype=F64, device=DEV)
    m[1:-1, 1:-1, 1:-1] = 1.0
    return m.reshape(-1, 1)


def _block(G, n, seed, orbitals=True, ld=None):
    """A start block: (with `orbitals`) unit vectors on the first enrichment coefficients,
    normal values on the interior nodes and, without, on every coefficient."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    X = torch.zeros((G.rows, ld or n), dtype=F64, device=DEV)[:, :n]
    if orbitals:
        k = min(n, G.n_enrich)
        X[G.n_nodes:, :k] = torch.eye(G.n_enrich, k, dtype=F64, device=DEV)
        X[:G.n_nodes, k:] = torch.randn((G.n_nodes, n - k), generator=g, dtype=F64, device=DEV)
        # the seed moves the atomic orbitals too: a filter never meets bare unit vectors twice
        X[:G.n_nodes, :k] = 1e-3 * torch.randn((G.n_nodes, k), generator=g, dtype=F64, device=DEV)
    else:
        X[:] = torch.randn((G.rows, n), generator=g, dtype=F64, device=DEV)
    X[:G.n_nodes] *= _interior(G)
    return X


def _waves(G, X, seed):
    """Plane waves with a growing share of noise from the first column to the last: a
    start block whose Ritz values run from the smooth vectors' to the mesh's energies."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) + 77)
    x = np.array([-1.0, -math.sqrt(3 / 7), 0.0, math.sqrt(3 / 7)])
    n = X.shape[1]
    k = torch.randn((3, n), generator=g, dtype=F64, device=DEV)
    k /= k.norm(dim=0)
    wave = torch.polar(torch.ones(n, dtype=F64, device=DEV), 6.3 * torch.rand(n, generator=g, dtype=F64, device=DEV))
    for d, b in enumerate(np.asarray(b) for b in G.system["breaks"]):
        at = np.append((b[:-1, None] + 0.5 * np.diff(b)[:, None] * (x + 1.0)).reshape(-1), b[-1])
        ph = torch.tensor(at, dtype=F64, device=DEV)[:, None] * k[d]
        wave = wave * torch.polar(torch.ones_like(ph), ph).reshape([len(at) if j == 2 - d else 1 for j in range(3)] + [n])
    q = torch.linspace(0.05, 0.95, n, dtype=F64, device=DEV)      # the noise's part of each column's square
    X *= (0.5 * q / (1.0 - q)).sqrt()
    X[:G.n_nodes] += wave.real.reshape(-1, n) * _interior(G)
    return X


def _electron_cloud(G, q, seed):
    """A density of Gaussian clouds on the atoms holding their electrons."""
    rng = np.random.default_rng(int(seed))
    rho = torch.zeros(len(q), dtype=F64, device=DEV)
    for R, Z in zip(G.system["atoms"], G.system["Z"]):
        w = rng.uniform(0.8, 1.2)
        d2 = ((q[:, :3] - torch.tensor(R, dtype=F64, device=DEV)) ** 2).sum(dim=1)
        rho += float(Z) * torch.exp(-d2 / (2 * w * w)) / (2 * math.pi * w * w) ** 1.5
    return rho * (float(np.sum(G.system["Z"])) / float((q[:, 3] * rho).sum()))


def _shells(Z):
    """Occupied shells (n, exponent, electrons) of a neutral atom, Slater's rules."""
    Z = int(Z)
    out = [(1, Z - 0.30 if Z > 1 else 1.0, float(min(Z, 2)))]
    if Z > 2:
        n2 = min(Z - 2, 8)
        out.append((2, (Z - 1.7 - (n2 - 1) * 0.35) / 2.0, float(n2)))
    if Z > 10:
        n3 = min(Z - 10, 8)
        out.append((3, (Z - 8.8 - (n3 - 1) * 0.35) / 3.0, float(n3)))
    return out


def _net(rng):
    net = efe.Mlp(learned.DIMS, seed=int(rng.integers(1 << 30)))
    # small biases, as after some training
    net.params += torch.from_numpy(0.01 * rng.standard_normal(net.n_params)).to(net.params)
    return net


def prepare(case, seed):
    do = case["do"]
    rng = np.random.default_rng(int(seed))
    if do == "train":
        # mid-training: descriptors of unit scale, targets of a log density ratio, Adam moments
        net, n = _net(rng), case["rows"]
        g = torch.Generator(device=DEV)
        g.manual_seed(int(seed))
        X = torch.randn((n, learned.N_FEAT), generator=g, device=DEV)
        net.m.copy_(1e-3 * torch.randn(net.n_params, generator=g, device=DEV))
        net.v.copy_(1e-6 * (1.0 + torch.rand(net.n_params, generator=g, device=DEV)))
        net.t = 100
        y = torch.tanh(X[:, :8].sum(dim=1)) + 0.1 * torch.randn(n, generator=g, device=DEV)
        return {"do": do, "net": net, "X": X, "y": y, "c": torch.rand(n, generator=g, device=DEV)}
    hs = _handles(case)
    if do == "batch":
        X0 = [_block(G, _batch_n(G), seed + i) for i, (G, _) in enumerate(hs)]
        return {"do": do, "case": case, "B": efe.Batch([G for G, _ in hs]), "X0": X0, "X": [x.clone() for x in X0],
                "ab": [np.array(v) for v in zip(*[ab for _, ab in hs])]}
    G, ab = hs[0]
    s = {"do": do, "case": case, "G": G, "ab": ab}
    if do in ("filter", "ritz"):
        s["X0"] = _block(G, case["n"], seed, orbitals=do == "filter", ld=case.get("ld"))
        if do == "ritz":
            _waves(G, s["X0"], seed)
        s["X"] = torch.zeros((G.rows, case.get("ld") or case["n"]), dtype=F64, device=DEV)[:, :case["n"]]
    elif do == "scf":
        q = G.qpoints()
        s["X0"] = _block(G, case["n"], seed)
        s["X"] = s["X0"].clone()
        s["rho0"] = _electron_cloud(G, q, seed)
        s["rho_in"], s["rho_out"] = torch.empty_like(s["rho0"]), torch.empty_like(s["rho0"])
        s["ne"] = float(np.sum(G.system["Z"]))
    elif do == "fields":
        q = G.qpoints()
        d2 = torch.stack([((q[:, :3] - torch.tensor(R, dtype=F64, device=DEV)) ** 2).sum(dim=1)
                          for R in G.system["atoms"]])
        s["vext"] = -(torch.tensor(G.system["Z"], dtype=F64, device=DEV)[:, None] / d2.sqrt()).sum(dim=0)
        # orbitals of about unit norm: enrichment coefficients of order one, smaller classical values
        s["X"] = _block(G, case["n"], seed, orbitals=False)
        s["X"][:G.n_nodes] *= 0.02
        s["occ"] = torch.rand(case["n"], generator=torch.Generator(device=DEV).manual_seed(int(seed)), dtype=F64, device=DEV)
        s["Y"] = _block(G, case["cols"], seed + 1, orbitals=False)
    elif do == "start":
        s["shells"] = [_shells(z) for z in G.system["Z"]]
        s["ne"] = float(np.sum(G.system["Z"]))
        model = learned.DensityModel(seed=int(rng.integers(1 << 30)))
        model.net = _net(rng)
        model.offset = rng.uniform(0.0, 0.2, learned.N_FEAT)
        model.scale = rng.uniform(1.0, 4.0, learned.N_FEAT)
        s["model"] = model
    return s


def _phases(X0, X):
    """Ritz vectors carry an arbitrary sign: a program that follows them from step to
    step turns each to a positive overlap with its start block (here: the first column)."""
    X *= torch.sign(X0[:, 0] @ X)
    return X


def _batch_n(G):
    return int(math.ceil(0.6 * float(np.sum(G.system["Z"])))) + 8


def run(s):
    do = s["do"]
    if do == "train":
        net = s["net"]
        yh = net.forward(s["X"])
        loss, dy = net.wmse(yh, s["y"], s["c"])
        g = net.backward(s["X"], dy)
        net.adam(g)
        return {"y": yh, "loss": loss, "grad": g, "params": net.params, "m": net.m, "v": net.v}
    case = s["case"]
    if do == "batch":
        for x, x0 in zip(s["X"], s["X0"]):
            x.copy_(x0)
        s["B"].chfsi_step(s["X"], case["m"], *s["ab"], precision=case["precision"], fp64_tail=case["tail"])
        return s["X"]
    G = s["G"]
    if do == "filter":
        s["X"].copy_(s["X0"])
        return G.chfsi_step(s["X"], case["m"], *s["ab"], precision=case["precision"], fp64_tail=case["tail"])
    if do == "ritz":
        s["X"].copy_(s["X0"])
        eig, res = G.rayleigh_ritz(s["X"])
        return {"X": _phases(s["X0"], s["X"]), "eig": eig, "res": res}
    if do == "scf":
        s["X"].copy_(s["X0"])
        s["rho_in"].copy_(s["rho0"])
        G.scf_init(s["ne"], kT=500 * KB)
        r = G.scf_step(s["X"], s["rho_in"], s["rho_out"], case["m"], precision=case["precision"], fp64_tail=case["tail"])
        return {"rho_in": s["rho_in"], "rho_out": s["rho_out"], "eig": r["eig"], "occ": r["occ"],
                "terms": [r[k] for k in ("band", "xc", "hartree", "double_counting", "total", "drho")]}
    if do == "fields":
        rho = G.density(s["X"], s["occ"], precision=case["precision"])
        vh, phi, _ = G.hartree(rho)
        exc, vxc = G.xc_lda(rho)
        G.set_potential(s["vext"] + vh + vxc)
        return {"rho": rho, "vh": vh, "phi": phi, "exc": exc, "vxc": vxc, "HY": G.apply_H(s["Y"])}
    sad = G.sad_density(s["shells"], s["ne"])
    D = s["model"].descriptors(G)
    y = s["model"].net.forward(D)
    return {"sad": sad, "D": D, "y": y, "rho": G.learned_density(sad, y, learned.FLOOR, s["ne"])}


# --------------------------------------------------------------------------- work
def _filter_work(G, n, m, low):
    """Per degree: the operator and two vector blocks read, one written (8 bytes a value, 4
    in the mixed degrees); cell, coupling and enrichment products."""
    flops = m * n * (2.0 * 125 * 125 * G.n_cells + 8.0 * G.n_coupling + 4.0 * G.n_enrich ** 2)
    word = [4] * low + [8] * (m - low)
    per = 125.0 * 125 * G.n_cells + 2.0 * G.n_coupling + 2.0 * G.n_enrich ** 2 + 3.0 * G.rows * n
    return {"bytes": float(sum(word)) * per, "flops": flops}


def work(case):
    do = case["do"]
    if do == "train":
        d, n = learned.DIMS, case["rows"]
        w = sum(a * b for a, b in zip(d[:-1], d[1:]))
        return {"bytes": 4.0 * (n * (d[0] + 4) + 8 * w), "flops": 2.0 * n * (3 * w - d[0] * d[1])}
    hs = _handles(case)
    if do == "batch":
        ws = [_filter_work(G, _batch_n(G), case["m"], max(0, case["m"] - case["tail"])) for G, _ in hs]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    G = hs[0][0]
    if do == "filter":
        low = 0 if case["precision"] == "fp64" else max(0, case["m"] - case["tail"])
        return _filter_work(G, case["n"], case["m"], low)
    n = case.get("n", 0)
    apply = 2.0 * 125 * 125 * G.n_cells + 4.0 * G.n_coupling + 2.0 * G.n_enrich ** 2
    # Gram, two projections (symmetric), rotations by R^-1 and Psi, H and M applied; the dense
    # eigenproblem about 12 n^3; H X and M X once more for the residuals
    ritz = {"bytes": 8.0 * (3 * G.rows * n + 125.0 * 125 * G.n_cells + 2 * G.n_coupling),
            "flops": 3.0 * G.rows * n * n + 3.0 * G.rows * n * n + 2 * n * apply + 12.0 * n ** 3}
    if do == "ritz":
        return ritz
    # density per point and vector: a tensor-product interpolation (about 25 + 30 + 10 + 5 flops
    # a point on 6^3 boxes) and its square; descriptors and network per point; the cell
    # matrices written once
    point = 60.0 * G.n_qpoints
    cells = 8.0 * 125 * 125 * G.n_cells
    if do == "scf":
        f = _filter_work(G, n, case["m"], 0)
        return {"bytes": f["bytes"] + 2 * ritz["bytes"] + cells + 8.0 * 12 * G.n_qpoints,
                "flops": f["flops"] + 2 * ritz["flops"] + point * n}
    if do == "fields":
        return {"bytes": 8.0 * (G.rows * (n + 2 * case["cols"]) + 12 * G.n_qpoints) + 2 * cells,
                "flops": point * n + case["cols"] * apply + 2 * 3375.0 * 6 * G.n_cells * 6}
    d = learned.DIMS
    w = sum(a * b for a, b in zip(d[:-1], d[1:]))
    return {"bytes": G.n_qpoints * (8.0 * 6 + 4.0 * d[0]), "flops": 2.0 * w * G.n_qpoints}


# --------------------------------------------------------------------------- 64-bit values
class _Exact:
    """The discrete problem of one handle in dense 64-bit torch."""

    def __init__(self, G):
        self.G, s = G, G.system
        z = np.array([-1.0, -math.sqrt(3 / 7), 0.0, math.sqrt(3 / 7), 1.0])
        wz = np.array([0.1, 49 / 90, 32 / 45, 49 / 90, 0.1])
        coef = np.linalg.inv(np.vander(z, 5, increasing=True))        # columns: Lagrange polynomials
        self.coef = torch.tensor(coef, dtype=F64, device=DEV)
        self.dcoef = torch.tensor(coef[1:] * np.arange(1, 5)[:, None], dtype=F64, device=DEV)
        x, w = np.polynomial.legendre.leggauss(6)
        L = np.vander(x, 5, increasing=True) @ coef
        dL = np.vander(x, 4, increasing=True) @ (coef[1:] * np.arange(1, 5)[:, None])
        self.M1, self.K1 = L.T @ (w[:, None] * L), dL.T @ (w[:, None] * dL)
        self.brk = [torch.tensor(np.asarray(b), dtype=F64, device=DEV) for b in s["breaks"]]
        nc = self.nc = [len(b) - 1 for b in s["breaks"]]
        nn = self.nn = [4 * n + 1 for n in nc]
        k, j, i = torch.meshgrid(*[torch.arange(n, device=DEV) for n in nc[::-1]], indexing="ij")
        self.ijk = torch.stack([i.reshape(-1), j.reshape(-1), k.reshape(-1)])
        self.h = torch.stack([self.brk[d][self.ijk[d] + 1] - self.brk[d][self.ijk[d]] for d in range(3)])
        c, b, a = torch.meshgrid(*[torch.arange(5, device=DEV)] * 3, indexing="ij")
        loc = [a.reshape(-1), b.reshape(-1), c.reshape(-1)]
        g = [4 * self.ijk[d][:, None] + loc[d][None, :] for d in range(3)]
        self.nodes = g[0] + nn[0] * (g[1] + nn[1] * g[2])
        self.inside = _interior(G)[:, 0]
        w1 = torch.tensor(wz, dtype=F64, device=DEV)
        w3 = w1[loc[0]] * w1[loc[1]] * w1[loc[2]]
        self.D = torch.zeros(G.n_nodes, dtype=F64, device=DEV)
        self.D.index_add_(0, self.nodes.reshape(-1), (self.h.prod(dim=0)[:, None] / 8 * w3).reshape(-1))
        self.Dinv = self.inside / self.D
        q = G.qpoints()
        self.pts, self.w = q[:, :3], q[:, 3].contiguous()
        e = [torch.searchsorted(self.brk[d], self.pts[:, d].contiguous(), right=True) - 1 for d in range(3)]
        self.cell = e[0] + nc[0] * (e[1] + nc[1] * e[2])
        self.cnt = torch.bincount(self.cell, minlength=G.n_cells)
        self.off = torch.cumsum(self.cnt, 0) - self.cnt
        self.enr = []                                                  # per atom: functions, points, values, gradients
        for ia, (R, Z) in enumerate(zip(s["atoms"], s["Z"])):
            fs = [i for i, f in enumerate(s["funcs"]) if f["atom"] == ia]
            if fs:
                self.enr.append(self._functions(fs, R, Z))

    def basis(self, p, gradients=False):
        """Classical basis (and gradients) at the points p (indexes)."""
        e = self.cell[p]
        L, dL = [], []
        for d in range(3):
            h = self.h[d][e]
            xi = 2.0 * (self.pts[p, d] - self.brk[d][self.ijk[d][e]]) / h - 1.0
            pw = torch.stack([xi ** k for k in range(5)], dim=1)
            L.append(pw @ self.coef)
            dL.append((pw[:, :4] @ self.dcoef) * (2.0 / h)[:, None])

        def outer(x, y, z):
            return (z[:, :, None, None] * y[:, None, :, None] * x[:, None, None, :]).reshape(-1, 125)
        B = outer(*L)
        if not gradients:
            return B
        return B, [outer(*[dL[k] if k == d else L[k] for k in range(3)]) for d in range(3)]

    def _functions(self, fs, R, Z):
        s = self.G.system
        f0 = s["funcs"][fs[0]]
        rs = f0["r0"] * (1 + 1 / f0["t"])
        dx = self.pts - torch.tensor(R, dtype=F64, device=DEV)
        r = dx.square().sum(dim=1).sqrt()
        p = torch.nonzero(r < rs)[:, 0]
        dx, r = dx[p], r[p]
        rt = 1.0 - f0["t"] * (r - f0["r0"]) / f0["r0"]

        def u(x):
            y = torch.where(x > 0, x, torch.ones_like(x))
            v = torch.where(x > 0, torch.exp(-1.0 / y), torch.zeros_like(x))
            return v, v / (y * y)
        (ua, da), (ub, db) = u(rt), u(1.0 - rt)
        den = ua + ub
        hc, dh = ua / den, (da * ub + ua * db) / den ** 2 * (-f0["t"] / f0["r0"])
        E, Gr = [], []
        for i in fs:
            f = s["funcs"][i]
            n, l = f["n"], f["l"]
            if f["kind"] == "slater":
                zt = f["zeta"]
                c, k = (2 * zt) ** (n + 0.5) / math.sqrt(math.factorial(2 * n)), n - 1 - l
                ex = c * torch.exp(-zt * r)
                qv = ex * r ** k
                dq = ex * ((k * r ** (k - 1) if k > 0 else 0.0) - zt * r ** k)
            elif n == 1:
                qv = 2 * Z ** 1.5 * torch.exp(-Z * r)
                dq = -Z * qv
            elif l == 0:
                c, ex = Z ** 1.5 / (2 * math.sqrt(2)), torch.exp(-Z * r / 2)
                qv, dq = c * (2 - Z * r) * ex, c * ex * (Z * Z * r / 2 - 2 * Z)
            else:
                qv = Z ** 2.5 / (2 * math.sqrt(6)) * torch.exp(-Z * r / 2)
                dq = -0.5 * Z * qv
            v, dv = qv * hc, dq * hc + qv * dh
            if l == 0:
                P, ax = torch.full_like(r, 1 / math.sqrt(4 * math.pi)), None
            else:
                ax = {-1: 1, 0: 2, 1: 0}[f["m"]]
                P = math.sqrt(3 / (4 * math.pi)) * dx[:, ax]
            gr = (dv * P / r)[:, None] * dx
            if ax is not None:
                gr[:, ax] += v * math.sqrt(3 / (4 * math.pi))
            E.append(v * P)
            Gr.append(gr)
        return fs, p, torch.stack(E, dim=1), torch.stack(Gr, dim=1)

    def potential(self, extra=True):
        s, V = self.G.system, torch.zeros_like(self.w)
        for R, Z in zip(s["atoms"], s["Z"]):
            V -= float(Z) / (self.pts - torch.tensor(R, dtype=F64, device=DEV)).square().sum(dim=1).sqrt()
        if extra:
            pot = s["potential"]
            for A, sg, c in zip(pot["gauss_A"], pot["gauss_s"], pot["gauss_c"]):
                V += float(A) * torch.exp(-(self.pts - torch.tensor(c, dtype=F64, device=DEV)).square().sum(dim=1) / (2 * sg * sg))
        return V

    def build(self, V):
        G = self.G
        wV = self.w * V
        M1, K1 = self.M1, self.K1
        k3 = [np.kron(M1, np.kron(M1, K1)), np.kron(M1, np.kron(K1, M1)), np.kron(K1, np.kron(M1, M1))]
        k3 = torch.tensor(np.stack(k3), dtype=F64, device=DEV).reshape(3, -1)
        h = self.h
        cf = torch.stack([h[1] * h[2] / h[0], h[0] * h[2] / h[1], h[0] * h[1] / h[2]]) / 4.0
        self.Hcc = (cf.T @ k3).reshape(-1, 125, 125)
        for n in torch.unique(self.cnt).tolist():
            cells = torch.nonzero(self.cnt == n)[:, 0]
            for c in cells.split(max(1, 400000 // n)):
                p = (self.off[c][:, None] + torch.arange(n, device=DEV)).reshape(-1)
                B = self.basis(p).reshape(len(c), n, 125)
                self.Hcc[c] += torch.bmm(B.transpose(1, 2), wV[p].reshape(-1, n, 1) * B)
        nE = G.n_enrich
        self.Mec = torch.zeros((nE, G.n_nodes), dtype=F64, device=DEV)
        self.Hec = torch.zeros_like(self.Mec)
        self.Mee = torch.zeros((nE, nE), dtype=F64, device=DEV)
        self.Hee = torch.zeros_like(self.Mee)
        for fs, p, E, Gr in self.enr:
            for k in range(0, len(p), 200000):
                pk, sl = p[k:k + 200000], slice(k, k + 200000)
                B, dB = self.basis(pk, True)
                idx = self.nodes[self.cell[pk]].reshape(-1)
                for j, f in enumerate(fs):
                    e, gr = E[sl, j], Gr[sl, j]
                    self.Mec[f].index_add_(0, idx, ((self.w[pk] * e)[:, None] * B).reshape(-1))
                    hv = (wV[pk] * e)[:, None] * B
                    for d in range(3):
                        hv += (0.5 * self.w[pk] * gr[:, d])[:, None] * dB[d]
                    self.Hec[f].index_add_(0, idx, hv.reshape(-1))
        full = torch.full((len(self.w),), -1, dtype=torch.long, device=DEV)
        for fa, pa, Ea, Ga in self.enr:
            full.fill_(-1)
            full[pa] = torch.arange(len(pa), device=DEV)
            for fb, pb, Eb, Gb in self.enr:
                if fb[0] < fa[0]:
                    continue
                at = full[pb]
                kb = torch.nonzero(at >= 0)[:, 0]
                ka, pt = at[kb], pb[kb]
                ea, eb, w, wv = Ea[ka], Eb[kb], self.w[pt][:, None], wV[pt][:, None]
                m = ea.T @ (w * eb)
                hm = ea.T @ (wv * eb) + 0.5 * sum(Ga[ka, :, d].T @ (w * Gb[kb, :, d]) for d in range(3))
                ia, ib = torch.tensor(fa, device=DEV), torch.tensor(fb, device=DEV)
                for T, v in ((self.Mee, m), (self.Hee, hm)):
                    T[ia[:, None], ib[None, :]] = v
                    T[ib[:, None], ia[None, :]] = v.T
        self.Mec *= self.inside
        self.Hec *= self.inside
        S = self.Mee - (self.Mec * self.Dinv) @ self.Mec.T
        self.S = 0.5 * (S + S.T)
        return self

    def H(self, X):
        nn = self.G.n_nodes
        W = torch.zeros_like(X)
        for c in torch.arange(self.G.n_cells, device=DEV).split(2048):
            nd = self.nodes[c]
            W.index_add_(0, nd.reshape(-1), torch.bmm(self.Hcc[c], X[nd.reshape(-1)].reshape(len(c), 125, -1)).reshape(-1, X.shape[1]))
        W[:nn] += self.Hec.T @ X[nn:]
        W[:nn] *= self.inside[:, None]
        W[nn:] = self.Hec @ X[:nn] + self.Hee @ X[nn:]
        return W

    def M(self, X):
        nn = self.G.n_nodes
        return torch.cat([(self.D * self.inside)[:, None] * X[:nn] + self.Mec.T @ X[nn:], self.Mec @ X[:nn] + self.Mee @ X[nn:]])

    def Minv(self, X):
        nn = self.G.n_nodes
        dx = self.Dinv[:, None] * X[:nn]
        xe = torch.linalg.solve(self.S, X[nn:] - self.Mec @ dx)
        return torch.cat([dx - self.Dinv[:, None] * (self.Mec.T @ xe), xe])

    def filter(self, X, m, a, b, a0):
        e, c = 0.5 * (b - a), 0.5 * (b + a)
        s1 = s = e / (a0 - c)
        prev, Y = X, (s1 / e) * (self.Minv(self.H(X)) - c * X)
        for _ in range(2, m + 1):
            sn = 1.0 / (2.0 / s1 - s)
            prev, Y = Y, (2 * sn / e) * (self.Minv(self.H(Y)) - c * Y) - (s * sn) * prev
            s = sn
        return Y

    def ritz(self, X):
        Q = torch.linalg.qr(X)[0]
        HQ, MQ = self.H(Q), self.M(Q)
        Hp, Mp = Q.T @ HQ, Q.T @ MQ
        Li = torch.linalg.inv(torch.linalg.cholesky(0.5 * (Mp + Mp.T)))
        C = Li @ (0.5 * (Hp + Hp.T)) @ Li.T
        eps, Z = torch.linalg.eigh(0.5 * (C + C.T))
        Psi = Li.T @ Z
        return eps, Q @ Psi, ((HQ @ Psi) - (MQ @ Psi) * eps).norm(dim=0)

    def upper(self, v, k):
        v = v / (v @ self.M(v[:, None])[:, 0]).sqrt()
        vp, beta, al, be = torch.zeros_like(v), 0.0, [], []
        for _ in range(k):
            w = self.Minv(self.H(v[:, None]))[:, 0]
            alpha = w @ self.M(v[:, None])[:, 0]
            w = w - alpha * v - beta * vp
            beta = (w @ self.M(w[:, None])[:, 0]).sqrt()
            al.append(float(alpha))
            be.append(float(beta))
            vp, v = v, w / beta
        return float(np.linalg.eigvalsh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1)).max()) + be[-1]

    def at_points(self, X):
        """FE fields (columns of X) at every quadrature point, cell by cell in chunks."""
        for p in torch.arange(len(self.w), device=DEV).split(200000):
            B = self.basis(p)
            out = torch.empty((len(p), X.shape[1]), dtype=F64, device=DEV)
            cells, n = torch.unique_consecutive(self.cell[p], return_counts=True)
            at = 0
            for c, k in zip(cells.tolist(), n.tolist()):
                out[at:at + k] = B[at:at + k] @ X[self.nodes[c]]
                at += k
            yield p, out

    def density(self, X, occ):
        enr = torch.zeros((len(self.w), X.shape[1]), dtype=F64, device=DEV) if self.enr else None
        for fs, p, E, _ in self.enr:
            enr.index_add_(0, p, E @ X[self.G.n_nodes + torch.tensor(fs, device=DEV)])
        rho = torch.empty_like(self.w)
        for p, v in self.at_points(X):
            v = v + enr[p] if enr is not None else v
            rho[p] = 2.0 * v.square() @ occ
        return rho

    def hartree(self, rho):
        nn, wr = self.nn, self.w * rho
        Q = wr.sum()
        ctr = (wr[:, None] * self.pts).sum(dim=0) / Q
        b = torch.zeros(self.G.n_nodes, dtype=F64, device=DEV)
        for p in torch.arange(len(self.w), device=DEV).split(400000):
            b.index_add_(0, self.nodes[self.cell[p]].reshape(-1), (wr[p][:, None] * self.basis(p)).reshape(-1))
        K, M, ax = [], [], []
        for d in range(3):
            Kd, Md = np.zeros((nn[d], nn[d])), np.zeros((nn[d], nn[d]))
            br = np.asarray(self.G.system["breaks"][d])
            x = np.empty(nn[d])
            for i in range(self.nc[d]):
                hc, sl = br[i + 1] - br[i], slice(4 * i, 4 * i + 5)
                Kd[sl, sl] += 2 / hc * self.K1
                Md[sl, sl] += hc / 2 * self.M1
                x[sl] = br[i] + 0.5 * hc * (np.array([-1, -math.sqrt(3 / 7), 0, math.sqrt(3 / 7), 1]) + 1)
            K.append(torch.tensor(Kd, dtype=F64, device=DEV))
            M.append(torch.tensor(Md, dtype=F64, device=DEV))
            ax.append(torch.tensor(x, dtype=F64, device=DEV))

        def modes(A, u):         # A[2] (x) A[1] (x) A[0] on u[k][j][i]
            return torch.einsum("cC,CBA->cBA", A[2], torch.einsum("bB,CBA->CbA", A[1], torch.einsum("aA,CBA->CBa", A[0], u)))

        def stiff(u):
            return (modes([K[0], M[1], M[2]], u) + modes([M[0], K[1], M[2]], u) + modes([M[0], M[1], K[2]], u)) / (4 * math.pi)
        zz, yy, xx = torch.meshgrid(ax[2] - ctr[2], ax[1] - ctr[1], ax[0] - ctr[0], indexing="ij")
        inn = self.inside.reshape(nn[2], nn[1], nn[0])
        phi = (1 - inn) * Q / (xx * xx + yy * yy + zz * zz).sqrt()
        V, lam = [], []
        for d in range(3):
            Li = torch.linalg.inv(torch.linalg.cholesky(M[d][1:-1, 1:-1]))
            C = Li @ K[d][1:-1, 1:-1] @ Li.T
            l, W = torch.linalg.eigh(0.5 * (C + C.T))
            V.append(Li.T @ W)
            lam.append(l)
        den = lam[2][:, None, None] + lam[1][None, :, None] + lam[0][None, None, :]
        for _ in range(3):
            r = (b.reshape(inn.shape) - stiff(phi))[1:-1, 1:-1, 1:-1]
            phi[1:-1, 1:-1, 1:-1] += modes(V, modes([v.T for v in V], r) * (4 * math.pi) / den)
        phi = phi.reshape(-1)
        vh = torch.empty_like(self.w)
        for p, v in self.at_points(phi[:, None]):
            vh[p] = v[:, 0]
        return vh, phi


def _lda(rho):
    """Slater exchange and the Perdew-Zunger fit of the Ceperley-Alder correlation."""
    rho = rho.clamp(min=1e-30)
    ex = -0.75 * (3 * rho / math.pi) ** (1 / 3)
    rs = (3 / (4 * math.pi * rho)) ** (1 / 3)
    sq, lr = rs.sqrt(), rs.log()
    den = 1 + 1.0529 * sq + 0.3334 * rs
    lo = -0.1423 / den
    vlo = lo * (1 + 7 / 6 * 1.0529 * sq + 4 / 3 * 0.3334 * rs) / den
    hi = 0.0311 * lr - 0.048 + 0.0020 * rs * lr - 0.0116 * rs
    vhi = 0.0311 * lr + (-0.048 - 0.0311 / 3) + 2 / 3 * 0.0020 * rs * lr + (2 * -0.0116 - 0.0020) / 3 * rs
    return ex + torch.where(rs >= 1, lo, hi), 4 / 3 * ex + torch.where(rs >= 1, vlo, vhi)


def _fermi(eps, ne, kT):
    lo, hi = float(eps.min()) - 1.0 - 50 * kT, float(eps.max()) + 1.0 + 50 * kT
    for _ in range(200):
        mu = 0.5 * (lo + hi)
        f = torch.sigmoid(((mu - eps) / kT).clamp(-700, 700))
        lo, hi = (mu, hi) if 2 * float(f.sum()) < ne else (lo, mu)
    return f


def _layers(net):
    at, out = 0, []
    for a, b in zip(net.dims[:-1], net.dims[1:]):
        out.append((net.params[at:at + a * b].double().reshape(b, a), net.params[at + a * b:at + a * b + b].double()))
        at += a * b + b
    return out


def _forward(layers, X):
    for i, (W, b) in enumerate(layers):
        X = X @ W.T + b
        if i < len(layers) - 1:
            X = X * torch.sigmoid(X)
    return X[:, 0]


def exact(case, seed):
    do = case["do"]
    if do == "batch" and case["count"] * case["m"] > 400:
        return None
    s = prepare(case, seed)
    if do == "train":
        net, X, y, c = s["net"], s["X"].double(), s["y"].double(), s["c"].double()
        p = net.params.double().requires_grad_(True)
        at, layers = 0, []
        for a, b in zip(net.dims[:-1], net.dims[1:]):
            layers.append((p[at:at + a * b].reshape(b, a), p[at + a * b:at + a * b + b]))
            at += a * b + b
        yh = _forward(layers, X)
        loss = (c * (yh - y) ** 2).sum() / c.sum()
        g, = torch.autograd.grad(loss, p)
        t = net.t + 1
        m = 0.9 * net.m.double() + 0.1 * g
        v = 0.999 * net.v.double() + 0.001 * g * g
        q = p.detach() - 1e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
        return {"y": yh.detach(), "loss": float(loss.detach()), "grad": g, "params": q, "m": m, "v": v}
    if do == "batch":
        out = []
        for (G, ab), X in zip(_handles(case), s["X0"]):
            E = _Exact(G)
            out.append(E.build(E.potential()).filter(X, case["m"], *ab))
        return out
    G = s["G"]
    E = _Exact(G)
    if do == "start":
        sad = torch.zeros_like(E.w)
        A = torch.zeros((len(E.w), learned.N_FEAT), dtype=F64, device=DEV)
        nr, na = len(learned.RADIAL_MU), len(learned.ANG_MU)
        vec = torch.zeros((len(E.w), 4, na, 3), dtype=F64, device=DEV)
        mu, am = (torch.tensor(np.asarray(x), dtype=F64, device=DEV) for x in (learned.RADIAL_MU, learned.ANG_MU))
        for R, Z, sh in zip(G.system["atoms"], G.system["Z"], s["shells"]):
            dx = E.pts - torch.tensor(R, dtype=F64, device=DEV)
            r = dx.square().sum(dim=1).sqrt()
            for n, zt, ne in sh:
                c2 = (2 * zt) ** (2 * n + 1) / math.factorial(2 * n)
                sad += ne * c2 * r ** (2 * n - 2) * torch.exp(-2 * zt * r) / (4 * math.pi)
            sp = learned.SPECIES.index(float(Z))
            fc = torch.where(r < learned.R_CUT, 0.5 * (1 + torch.cos(math.pi * r / learned.R_CUT)), torch.zeros_like(r))
            A[:, sp * nr:(sp + 1) * nr] += torch.exp(-(r[:, None] - mu) ** 2 / (2 * learned.RADIAL_SIGMA ** 2)) * fc[:, None]
            g = torch.exp(-(r[:, None] - am) ** 2 / (2 * learned.ANG_SIGMA ** 2)) * fc[:, None]
            vec[:, sp] += g[:, :, None] * (dx / r[:, None])[:, None, :]
        A[:, 4 * nr:] = vec.square().sum(dim=3).reshape(len(E.w), -1)
        mdl = s["model"]
        D = (A - torch.tensor(mdl.offset, dtype=F64, device=DEV)) * torch.tensor(mdl.scale, dtype=F64, device=DEV)
        sad *= s["ne"] / (E.w * sad).sum()
        y = torch.cat([_forward(_layers(mdl.net), d) for d in D.split(500000)])
        rho = ((sad + learned.FLOOR) * torch.exp(y) - learned.FLOOR).clamp(min=0)
        return {"sad": sad, "D": D, "y": y, "rho": rho * (s["ne"] / (E.w * rho).sum())}
    if do == "fields":
        rho = E.density(s["X"], s["occ"])
        vh, phi = E.hartree(rho)
        exc, vxc = _lda(rho)
        return {"rho": rho, "vh": vh, "phi": phi, "exc": exc, "vxc": vxc, "HY": E.build(s["vext"] + vh + vxc).H(s["Y"])}
    if do == "filter":
        return E.build(E.potential()).filter(s["X0"], case["m"], *s["ab"])
    if do == "ritz":
        eps, X, res = E.build(E.potential()).ritz(s["X0"])
        return {"X": _phases(s["X0"], X), "eig": eps, "res": res}
    rho_in = s["rho0"]
    vh, _ = E.hartree(rho_in)
    exc, vxc = _lda(rho_in)
    E.build(E.potential(False) + vh + vxc)
    eps, X, _ = E.ritz(s["X0"])
    b = E.upper(X[:, -1], 10)
    eps, X, _ = E.ritz(E.filter(X, case["m"], float(eps.max()), b, float(eps.min())))
    f = _fermi(eps, s["ne"], 500 * KB)
    rho = E.density(X, f)
    vo, _ = E.hartree(rho)
    band, xc = 2 * float((f * eps).sum()), float((E.w * rho * _lda(rho)[0]).sum())
    har, dc = 0.5 * float((E.w * rho * vo).sum()), float((E.w * rho * (vh + vxc)).sum())
    at, Z = G.system["atoms"], G.system["Z"]
    zz = sum(Z[i] * Z[j] / np.linalg.norm(at[i] - at[j]) for i in range(len(Z)) for j in range(i))
    return {"rho_in": rho_in + 0.5 * (rho - rho_in), "rho_out": rho, "eig": eps, "occ": f,
            "terms": [band, xc, har, dc, band - dc + har + xc + float(zz), float((E.w * (rho - rho_in) ** 2).sum().sqrt())]}
