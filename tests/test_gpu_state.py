"""Handles and batches whose settings or workspaces change between calls: a recorded graph
must follow them, and no call may meet freed or stale memory."""
import pytest

import workloads as W
from tests.gpu_util import cuda_available, gpu_system, to_dev, torch

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]


@pytest.fixture()
def members():
    from paper_1610_02121_gb300 import Batch
    ss = [W.tiny(seed=11), W.tiny(seed=12, cells=(3, 2, 2))]
    Gs = [gpu_system(s) for s in ss]
    Xs = [to_dev(W.initial_block(s, N, seed=3 + i)) for i, (s, N) in enumerate(zip(ss, (12, 20)))]
    bounds = [[], [], []]
    for G, X in zip(Gs, Xs):
        e, _ = G.rayleigh_ritz(X)
        for v, x in zip(bounds, (e.max(), G.upper_bound(X[:, -1].contiguous(), 10), e.min())):
            v.append(x)
    B = Batch(Gs)
    yield Gs, Xs, bounds, B
    B.close()
    for G in Gs:
        G.close()


def _same_as_sequential(members, m, precision, tail):
    """One replayed or newly recorded step against the same step without a graph, bit for bit;
    the blocks' addresses stay those of the fixture."""
    Gs, Xs, (a, b, a0), B = members
    keep = [X.clone() for X in Xs]
    B.chfsi_step(Xs, m, a, b, a0, precision=precision, fp64_tail=tail, graph=True)
    got = [X.clone() for X in Xs]
    for X, k in zip(Xs, keep):
        X.copy_(k)
    B.chfsi_step(Xs, m, a, b, a0, precision=precision, fp64_tail=tail, graph=False)
    for g, X, k in zip(got, Xs, keep):
        assert torch.equal(g, X)
        X.copy_(k)


@pytest.mark.parametrize("precision,tail", [("fp64", 0), ("tf32x3", 2)])
def test_replayed_graph_follows_each_members_engine(members, precision, tail):
    """The recorded FP64 kernels are those of every member's engine, and the digit images of
    H are remade for the members that use them: a member that changes its engine and gets a
    new potential is recorded anew."""
    Gs = members[0]
    for G in Gs:
        G.set_fp64_engine("tensor")
    _same_as_sequential(members, 6, precision, tail)
    Gs[1].set_fp64_engine("dfma")
    q = Gs[1].qpoints()
    Gs[1].set_potential((-1.0 / (0.5 + (q[:, :3] ** 2).sum(dim=1).sqrt())).contiguous())
    _same_as_sequential(members, 6, precision, tail)
    Gs[1].set_fp64_engine("tensor")
    _same_as_sequential(members, 6, precision, tail)


@pytest.mark.parametrize("name,value", [("coupling_cols", 1), ("coupling_sparse", 1), ("grid_cap", 3),
                                        ("cell_scratch", 1)])
def test_replayed_graph_follows_options(members, name, value):
    Gs = members[0]
    Gs[0].set_fp64_engine("tensor")
    Gs[1].set_option("coupling_sparse", int(name == "coupling_cols"))
    _same_as_sequential(members, 6, "tf32x3", 1)
    Gs[1].set_option(name, value)
    _same_as_sequential(members, 6, "tf32x3", 1)
    Gs[1].set_option(name, 0)
    _same_as_sequential(members, 6, "tf32x3", 1)


def test_replayed_graph_follows_longer_recurrences(members):
    """A filter of a higher degree on one member remakes its coefficient buffers, which the
    recorded graph copies from: the batch records again."""
    Gs, Xs, (a, b, a0), B = members
    _same_as_sequential(members, 6, "tf32x3", 2)
    first = B.graph_nodes()
    Gs[1].chfsi_step(Xs[1].clone(), 40, a[1], b[1], a0[1])
    _same_as_sequential(members, 6, "tf32x3", 2)
    assert B.graph_nodes() == first


@pytest.mark.parametrize("stall", [1, 2, 3])
@pytest.mark.parametrize("what,precision,engine", [("filter", "tf32x3", "dfma"), ("filter", "fp64", "tensor"),
                                                   ("ritz", "fp64", "tensor")])
def test_waits_that_run_out_in_each_role(what, precision, engine, stall):
    """A barrier that never completes, for the MMA warp, the converters or copies, and the
    epilogue: every lane's wait runs out by its own clock, the warps leave as a whole, the call
    returns EFE_ERR_TIMEOUT, and the next one gives the bits of the one before."""
    from paper_1610_02121_gb300 import EfeError
    s = W.tiny(seed=11)
    G = gpu_system(s)
    X = to_dev(W.initial_block(s, 20, seed=2))
    e, _ = G.rayleigh_ritz(X)
    b = G.upper_bound(X[:, -1].contiguous(), 10)
    G.set_fp64_engine(engine)

    def call():
        Y = X.clone()
        if what == "ritz":
            G.rayleigh_ritz(Y)
        else:
            G.chfsi_step(Y, 3, e.max(), b, e.min(), precision=precision)
        return Y

    before = call()
    G.set_option("test_stall", stall)
    try:
        with pytest.raises(EfeError) as err:
            call()
        assert err.value.code == 5
    finally:
        G.set_option("test_stall", 0)
    assert torch.equal(before, call())
    G.close()


def test_handle_after_a_refused_reservation():
    """A reservation that the device has no memory for (50 million columns, 424 GB) is an error;
    the workspace that it gave up is not used again, and the next calls reserve their own."""
    from paper_1610_02121_gb300 import EfeError
    G = gpu_system(W.tiny(seed=11))
    X = to_dev(W.initial_block(G.system, 20, seed=2))
    e, _ = G.rayleigh_ritz(X)
    b = G.upper_bound(X[:, -1].contiguous(), 10)
    before = G.chfsi_step(X.clone(), 5, e.max(), b, e.min(), precision="tf32x3", fp64_tail=2)
    for _ in range(2):
        with pytest.raises(EfeError) as err:
            G.reserve(50_000_000)
        assert err.value.code == 7
    for N in (7, 20):
        Y = X[:, :N].clone()
        G.chfsi_step(Y, 5, e.max(), b, e.min(), precision="tf32x3", fp64_tail=2)
        assert N < 20 or torch.equal(before, Y)
    G.close()


# 48 columns of the 1,053 nodes and 12 cells of the tiny mesh: 14 B a value of the digit planes,
# 8 B a product
ONE_TILE = max(14 * 1053 * 48, 8 * 12 * 125 * 48)


@pytest.fixture(scope="module")
def oracle_H():
    from oracle.operators import Discretisation
    return Discretisation(W.tiny(seed=11)).apply_H_assembled


@pytest.mark.parametrize("N", [20, 48, 49, 100, 145])
def test_engine_cells_take_what_memory_there_is(oracle_H, N):
    """The FP64 engine's cell products where the device refuses their scratch: in 48-column
    panels the bits of one panel, and without any room the DFMA products, against the oracle
    (the engine's figure, 1e-10 of the largest entry).  A filter, which keeps its panels from
    degree to degree, and a call after the memory has come back."""
    from tests.gpu_util import rel_err
    G = gpu_system(W.tiny(seed=11))
    assert (G.n_nodes, G.n_cells) == (1053, 12)
    X = W.random_block(G.system, N, seed=700 + N)
    Xd = to_dev(X)
    ref = oracle_H(X)
    b = G.upper_bound(Xd[:, -1].contiguous(), 10)
    G.set_fp64_engine("tensor")

    def step():
        return G.chfsi_step(Xd.clone(), 3, 0.2 * b, b, -1.0)

    whole, filtered = G.apply_H(Xd), step()
    G.set_option("cell_scratch", ONE_TILE)
    assert torch.equal(G.apply_H(Xd), whole) and torch.equal(step(), filtered)
    G.set_option("cell_scratch", 1)
    assert rel_err(G.apply_H(Xd), ref) < 1e-10
    none = step()
    assert rel_err(none, filtered.cpu().numpy()) < 1e-9
    G.set_option("cell_scratch", 0)
    assert torch.equal(G.apply_H(Xd), whole) and torch.equal(step(), filtered)
    G.close()


@pytest.mark.parametrize("precision", ["fp64", "tf32", "tf32x3", "bf16"])
@pytest.mark.parametrize("N", [1, 5, 16, 33, 96, 159, 160, 161])
def test_cells_colour_by_colour(precision, N):
    """Without scratch the cell products go colour by colour and are added into the result in
    the kernel: the bits of the launch over all cells and its gather."""
    G = gpu_system(W.tiny(seed=11))
    X = to_dev(W.random_block(G.system, N, seed=800 + N))
    b = G.upper_bound(X[:, -1].contiguous(), 10)

    def step(cap):
        G.set_grid_cap(cap)
        return G.chfsi_step(X.clone(), 3, 0.2 * b, b, -1.0, precision=precision)

    at_once = step(0)
    G.set_option("cell_scratch", 1)
    assert torch.equal(step(0), at_once) and torch.equal(step(1), at_once)
    G.close()


def test_products_after_a_wait_that_ran_out():
    """The error flag of a call that timed out belongs to that call: the engine's products of
    the next one run."""
    from paper_1610_02121_gb300 import EfeError
    G = gpu_system(W.tiny(seed=11))
    X = to_dev(W.initial_block(G.system, 20, seed=2))
    b = G.upper_bound(X[:, -1].contiguous(), 10)
    G.set_fp64_engine("tensor")
    before = G.apply_H(X)
    G.set_option("test_stall", 1)
    with pytest.raises(EfeError):
        G.chfsi_step(X.clone(), 1, 0.2 * b, b, -1.0)
    G.set_option("test_stall", 0)
    after = G.apply_H(2.0 * X)
    assert torch.equal(after, 2.0 * before)
    G.close()


def test_narrow_filter_after_a_wide_one():
    """A block too wide for the dense-tile coupling kernels takes the many-function ones; a
    narrower block on the same handle takes the dense tiles again (mixed filter of degree 3,
    FP32-grade: 5e-5 of the largest entry, as in the mixed cases against the oracle)."""
    from tests.gpu_util import rel_err
    s = W.tiny(seed=11)
    wide, fresh = gpu_system(s), gpu_system(s)
    # (n_E + 32) rows of N floats and the pattern tile in 200 KB
    N = (200 * 1024 // 4 - 2048) // (wide.n_enrich + 32) // 4 * 4 + 8
    X = to_dev(W.random_block(s, N, seed=9))
    b = fresh.upper_bound(X[:, -1].contiguous(), 10)
    many = wide.chfsi_step(X.clone(), 3, 0.2 * b, b, -1.0, precision="tf32x3")
    for n in (20, N - 16, N):
        got = wide.chfsi_step(X[:, :n].clone(), 3, 0.2 * b, b, -1.0, precision="tf32x3")
        ref = fresh.chfsi_step(X[:, :n].clone(), 3, 0.2 * b, b, -1.0, precision="tf32x3")
        assert rel_err(got, ref.cpu().numpy()) < 5e-5
        assert rel_err(got, many[:, :n].cpu().numpy()) < 5e-5
    assert torch.equal(got, many)
    wide.close()
    fresh.close()
