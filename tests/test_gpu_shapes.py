"""Sizes at the edges of the kernels' column tiles, thread splits and dispatch rules,
against the FP64 CPU oracle (products) or the general path (whole calls)."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_util import cuda_available, gpu_system, rel_err, to_dev, torch

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module")
def tiny_pair():
    from oracle.operators import Discretisation
    s = W.tiny(seed=11)
    return Discretisation(s), gpu_system(s)


# FP64 products: sums of up to a few thousand terms whose magnitudes exceed the result by
# at most ~1e3 here, at 2^-53 (DFMA) or a few 2^-48 (the tensor engine) a term: 1e-10 of
# the largest entry for H, 1e-11 for M (smaller terms), 1e-10 after the Schur solve
@pytest.mark.parametrize("engine", ["dfma", "tensor"])
@pytest.mark.parametrize("N", [5, 8, 9, 15, 16, 17, 31, 32, 65])
def test_products_at_tile_edges(tiny_pair, engine, N):
    d, G = tiny_pair
    X = W.random_block(d.system, N, seed=300 + N)
    wide = torch.zeros((X.shape[0], N + 3), dtype=torch.float64, device="cuda")
    wide[:, :N] = to_dev(X)
    G.set_fp64_engine(engine)
    try:
        for Xd in (to_dev(X), wide[:, :N]):
            assert rel_err(G.apply_H(Xd, torch.empty_like(wide)[:, :N]), d.apply_H_assembled(X)) < 1e-10
            assert rel_err(G.apply_M(Xd), d.apply_M_assembled(X)) < 1e-11
            assert rel_err(G.apply_Minv(Xd), d.apply_Minv_block(X)) < 1e-10
    finally:
        G.set_fp64_engine("dfma")


# FP64 engine's cell products: column tiles of 48 in groups of 16, few and many items per
# CTA (1 and 3 CTAs), column panels narrower than the block through the filter
@pytest.mark.parametrize("cap", [0, 1, 3])
@pytest.mark.parametrize("N", [9, 16, 17, 33, 47, 48, 49, 96, 97, 145])
def test_engine_cell_tiles(tiny_pair, cap, N):
    d, G = tiny_pair
    X = W.random_block(d.system, N, seed=700 + N)
    G.set_fp64_engine("tensor")
    G.set_grid_cap(cap)
    try:
        Y = G.apply_H(to_dev(X))
        assert rel_err(Y, d.apply_H_assembled(X)) < 1e-10
        assert torch.equal(Y, G.apply_H(to_dev(X)))          # reproducible, whatever the grid
        G.set_grid_cap(0)
        assert torch.equal(Y, G.apply_H(to_dev(X)))
    finally:
        G.set_grid_cap(0)
        G.set_fp64_engine("dfma")


# Cholesky-QR and Rayleigh-Ritz at the edges of the A^T B and A B tiles (16, 32, 48), against the
# oracle; the figures of the ordinary case (1e-9 on the Ritz values, 1e-8 on the residuals)
@pytest.mark.parametrize("N", [1, 2, 15, 16, 17, 32, 33, 48, 49])
def test_rayleigh_ritz_at_tile_edges(tiny_pair, N):
    from oracle.chfsi import cholqr, rayleigh_ritz
    d, G = tiny_pair
    X = W.random_block(d.system, N, seed=400 + N)
    eps_ref, _, res_ref = rayleigh_ritz(d.apply_H_assembled, d.apply_M_assembled, cholqr(X)[0])
    Xd = to_dev(X)
    eps, res = G.rayleigh_ritz(Xd)
    np.testing.assert_allclose(eps, eps_ref, atol=1e-9, rtol=1e-10)
    np.testing.assert_allclose(res, res_ref, atol=1e-8, rtol=1e-6)
    gram = (Xd.T @ G.apply_M(Xd)).cpu().numpy()
    np.testing.assert_allclose(gram, np.eye(N), atol=1e-10)


# the blocked eigensolver, Cholesky and triangular inverse at their block edges (16, 64) and
# at the size where they take over, on a problem whose Ritz values are the oracle's; the FP64
# engine's 2^-48 a term for the tall products gives the wider figure
@pytest.mark.parametrize("engine,tol", [("dfma", 1e-9), ("tensor", 1e-8)])
@pytest.mark.parametrize("N", [47, 50, 63, 64, 65, 97, 129, 150])
def test_blocked_dense_edges(tiny_pair, engine, tol, N):
    from oracle.chfsi import cholqr, rayleigh_ritz
    d, G = tiny_pair
    X = W.random_block(d.system, N, seed=500 + N)
    eps_ref, _, _ = rayleigh_ritz(d.apply_H_assembled, d.apply_M_assembled, cholqr(X)[0])
    G.set_fp64_engine(engine)
    try:
        Xd = to_dev(X)
        eps, _ = G.rayleigh_ritz(Xd)
    finally:
        G.set_fp64_engine("dfma")
    np.testing.assert_allclose(eps, eps_ref, atol=tol, rtol=tol)
    gram = (Xd.T @ G.apply_M(Xd)).cpu().numpy()
    np.testing.assert_allclose(gram, np.eye(N), atol=1e-8)


# FP32 network passes at the edges of the 128 x 128 x 16 tiles, with rows that do not allow
# 16-byte loads, against the oracle in FP64: the longest sums have max(dims, n) terms, so
# the largest entry is off by at most a few sqrt(max) roundings (2^-24 each); 1e-4 as in the
# ordinary FP32 case
@pytest.mark.parametrize("dims", [(64, 256, 256, 256, 1), (7, 33, 130, 1), (5, 1), (12, 128, 127, 1)])
@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 1000])
def test_network_at_tile_edges(dims, n):
    from oracle import learned as O
    from paper_1610_02121_gb300 import Mlp
    rng = np.random.default_rng(n + len(dims))
    flat = np.concatenate([x.reshape(-1) for x in O.init_params(dims, 3)]).astype(np.float32)
    flat += (0.05 * rng.standard_normal(len(flat))).astype(np.float32)
    params, at = [], 0
    for a, b in zip(dims[:-1], dims[1:]):
        params += [flat[at:at + a * b].reshape(b, a).astype(np.float64), flat[at + a * b:at + a * b + b].astype(np.float64)]
        at += a * b + b
    X = rng.standard_normal((n, dims[0])).astype(np.float32)
    dy = rng.standard_normal(n).astype(np.float32)
    y_ref, pre = O.forward(params, X.astype(np.float64))
    g_ref = np.concatenate([g.reshape(-1) for g in O.backward(params, X.astype(np.float64), pre, dy.astype(np.float64))])
    net = Mlp(dims, precision="fp32", params=flat)
    Xd = torch.from_numpy(X).cuda()
    assert rel_err(net.forward(Xd), y_ref) < 1e-4
    assert rel_err(net.backward(Xd, torch.from_numpy(dy).cuda()), g_ref) < 1e-4


# tensor-core cell products of the FP32 filter at the edges of the 16-column groups, the
# 160-column tile and the stage ring (one CTA walks every item; one item a CTA): one degree
# against the oracle at the operand's round-off times the cancellation factor (as in the
# ordinary case: 2^-11, 2^-24 and 2^-8 give 3e-3, 1e-5 and 3e-2)
@pytest.mark.parametrize("prec,tol", [("tf32", 3e-3), ("tf32x3", 1e-5), ("bf16", 3e-2)])
@pytest.mark.parametrize("N", [1, 5, 15, 16, 33, 64, 65, 96, 159, 160, 161])
def test_split_cell_tiles(tiny_pair, prec, tol, N):
    from oracle.chfsi import chebyshev_filter_scaled, lanczos_upper_bound
    d, G = tiny_pair
    X = W.random_block(d.system, N, seed=800 + N)
    b = 1.05 * lanczos_upper_bound(d.apply_Htilde, d.apply_M_assembled, W.lanczos_start(d.system), 10)
    ref = chebyshev_filter_scaled(d.apply_Htilde, X, 1, 0.2 * b, b, -1.0)
    out = []
    for cap in (0, 1):
        G.set_grid_cap(cap)
        try:
            Xd = to_dev(X)
            G.chfsi_step(Xd, 1, 0.2 * b, b, -1.0, precision=prec, fp64_tail=0)
        finally:
            G.set_grid_cap(0)
        out.append(Xd)
    assert rel_err(out[0], ref) < tol
    assert torch.equal(out[0], out[1])


# FP64 engine's tall products where the operand pieces of 128 rows and 96 columns and the
# 256-row groups of the segments end, against the oracle (figures of the blocked case)
@pytest.mark.parametrize("cap", [0, 3])
@pytest.mark.parametrize("N", [95, 96, 97, 127, 128, 129, 191, 193, 224])
def test_engine_tall_products(tiny_pair, cap, N):
    from oracle.chfsi import cholqr, rayleigh_ritz
    d, G = tiny_pair
    X = W.random_block(d.system, N, seed=900 + N)
    eps_ref, _, _ = rayleigh_ritz(d.apply_H_assembled, d.apply_M_assembled, cholqr(X)[0])
    G.set_fp64_engine("tensor")
    G.set_grid_cap(cap)
    try:
        Xd = to_dev(X)
        eps, _ = G.rayleigh_ritz(Xd)
    finally:
        G.set_grid_cap(0)
        G.set_fp64_engine("dfma")
    np.testing.assert_allclose(eps, eps_ref, atol=1e-8, rtol=1e-8)
    gram = (Xd.T @ G.apply_M(Xd)).cpu().numpy()
    np.testing.assert_allclose(gram, np.eye(N), atol=1e-8)


# descriptors: fewest and most Gaussians, widths at which most terms fall out of an FP32 sum
# and at which all stay, several atoms of a species; FP64 to rounding (arguments up to a few
# hundred: 1e-12 of the largest entry), FP32 to a few roundings of the largest entry (1e-6)
@pytest.mark.parametrize("width", [0.02, 0.45, 5.0, 1e-160])
@pytest.mark.parametrize("nr,nang", [(1, 0), (12, 4), (16, 8)])
def test_descriptor_sums(nr, nang, width):
    from paper_1610_02121_gb300 import learned as LR
    s = dict(W.tiny(seed=11))
    s["Z"] = np.ones(len(s["Z"]))
    G = gpu_system(s)
    p = LR.desc_params()
    p.n_radial, p.n_ang, p.radial_sigma, p.ang_sigma = nr, nang, width, max(width, 0.1)
    mu = np.linspace(0.3, 7.5, 16)
    for i in range(16):
        p.radial_mu[i] = mu[i]
    for i in range(8):
        p.ang_mu[i] = mu[2 * i]
    q = G.qpoints().cpu().numpy()[:, :3]
    ref = np.zeros((len(q), 4 * (nr + nang)))
    vec = np.zeros((len(q), nang, 3))
    with np.errstate(over="ignore", divide="ignore", invalid="ignore"):
        for a in np.asarray(s["atoms"]):
            d = q - a
            r = np.sqrt((d * d).sum(axis=1))
            fc = np.where(r < p.r_cut, 0.5 * (1 + np.cos(np.pi * r / p.r_cut)), 0.0)
            ref[:, :nr] += np.exp(-(r[:, None] - mu[None, :nr]) ** 2 / (2 * width * width)) * fc[:, None]
            g = np.exp(-(r[:, None] - mu[None, :2 * nang:2]) ** 2 / (2 * p.ang_sigma ** 2)) * fc[:, None]
            vec += g[:, :, None] * (d / np.maximum(r, 1e-12)[:, None])[:, None, :]
    ref[:, 4 * nr:4 * nr + nang] = (vec * vec).sum(axis=2)
    for prec, tol in (("fp64", 1e-12), ("fp32", 1e-6)):
        D = G.descriptors(p, precision=prec).double().cpu().numpy()
        assert D.shape == ref.shape
        assert np.abs(D - ref).max() <= tol * max(1.0, np.abs(ref).max())


# superposed atoms with one to three shells: every point to 1e-11 of its own value (the
# exponents reach a few hundred, at 2^-53 each; shells are left out below 2^-58 of the sum)
@pytest.mark.parametrize("Z", [(1, 1), (14, 1), (14, 14), (8, 14)])
def test_sad_points(tiny_pair, Z):
    from oracle import learned as OL
    d, G = tiny_pair
    q = G.qpoints().cpu().numpy()
    atoms = np.asarray(d.system["atoms"])
    shells = [W.sad_shells(Z[i % 2]) for i in range(len(atoms))]
    rho = G.sad_density(shells).cpu().numpy()
    ref = OL.sad_density(q[:, :3], atoms, shells)
    np.testing.assert_allclose(rho, ref, rtol=1e-11)


# superposed atoms far from their usual size: a density is linear in its occupations down to
# the smallest numbers, whatever part of it FP32 arithmetic can hold (2^-160 is exact in FP64
# and below FP32's range), so every point scales to rounding
@pytest.mark.parametrize("scale", [2.0 ** -160, 2.0 ** 160])
def test_sad_points_scale(tiny_pair, scale):
    d, G = tiny_pair
    shells = [W.sad_shells(z) for z in (14, 8)][:len(d.system["atoms"])]
    one = G.sad_density(shells)
    few = G.sad_density([[(n, z, o * scale) for n, z, o in s] for s in shells])
    torch.testing.assert_close(few / scale, one, rtol=1e-14, atol=0.0)


# dense eigenproblem of Rayleigh-Ritz on spectra from core levels (-90) to pairs 1e-4 apart: what
# is left off the diagonal of V^T C V turns a pair by itself over the gap.  The sweeps stop at
# 1e-15 of the norm; a product's sum of N terms adds a few sqrt(N) roundings of it.  (V^T C V
# and V^T V in extended precision; the mean value times V^T V - 1 belongs to the vectors' lengths.)
@pytest.mark.parametrize("N", [40, 49, 96, 135, 200])
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_eigenvectors_of_close_pairs(tiny_pair, N, seed):
    import ctypes as C
    from paper_1610_02121_gb300._lib import lib
    G = tiny_pair[1]
    rng = np.random.default_rng(seed + N)
    core = -90 + rng.uniform(-1, 1, N // 10)
    ev = rng.uniform(-1, 3, N - len(core))
    ev[1::8] = ev[0::8][:len(ev[1::8])] + 1e-4
    ev[2], ev[3] = 1e-7, -1e-7
    ev = np.concatenate([core, ev])
    Q, _ = np.linalg.qr(rng.standard_normal((N, N)))
    A = (Q * ev) @ Q.T
    A = (A + A.T) / 2
    G.reserve(N)
    Ad, V, w, E = to_dev(A), *(torch.empty(n, dtype=torch.float64, device="cuda") for n in (N * N, N, 9 * N * N))
    eig = lib().sym_eig
    eig.argtypes, eig.restype = [C.c_void_p, C.c_void_p, C.c_int] + [C.c_void_p] * 4, C.c_int
    assert eig(G.h, Ad.data_ptr(), N, V.data_ptr(), w.data_ptr(), E.data_ptr(),
               torch.cuda.current_stream().cuda_stream) == 0
    V = V.view(N, N).cpu().numpy().astype(np.longdouble)
    T, L = V.T @ (A.astype(np.longdouble) @ V), V.T @ V
    d = np.diag(T).copy()
    left = T - np.diag(d) - (d[:, None] + d[None, :]) / 2 * (L - np.diag(np.diag(L)))
    norm = np.linalg.norm(A)
    assert np.abs(left).max() <= (1e-15 + 4 * np.sqrt(N) * 2.0 ** -53) * norm


# Rayleigh-Ritz above 512 vectors (blocked Cholesky, block Jacobi with diagonalising visits, N x N
# products on the engine) and with the kernels of the largest blocks forced on smaller ones, against
# the oracle; the figures of the long tall products (1e-9 of the largest Ritz value; both engines)
@pytest.fixture(scope="module")
def wide_pair():
    from oracle.operators import Discretisation
    s = W.tiny(seed=11, cells=(3, 3, 3))
    return Discretisation(s), gpu_system(s)


@pytest.mark.parametrize("engine", ["dfma", "tensor"])
@pytest.mark.parametrize("N,forced", [(513, 0), (513, 1), (600, 0), (65, 1), (97, 1), (129, 1)])
def test_rayleigh_ritz_of_wide_blocks(wide_pair, engine, N, forced):
    from oracle.chfsi import cholqr, rayleigh_ritz
    d, G = wide_pair
    X = W.random_block(d.system, N, seed=1000 + N)
    eps_ref, _, res_ref = rayleigh_ritz(d.apply_H_assembled, d.apply_M_assembled, cholqr(X)[0])
    top = np.abs(eps_ref).max()
    G.set_fp64_engine(engine)
    G.set_option("dense_blocked", forced)
    try:
        Xd = to_dev(X)
        eps, res = G.rayleigh_ritz(Xd)
    finally:
        G.set_option("dense_blocked", 0)
        G.set_fp64_engine("dfma")
    np.testing.assert_allclose(eps, eps_ref, rtol=1e-9, atol=1e-9 * top)
    np.testing.assert_allclose(res, res_ref, rtol=1e-6, atol=1e-8 * top)
    gram = (Xd.T @ G.apply_M(Xd)).cpu().numpy()
    np.testing.assert_allclose(gram, np.eye(N), atol=1e-8)
