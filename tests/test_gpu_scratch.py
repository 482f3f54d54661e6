"""Calls on a device with little room left (BTAS_WS_LIMIT refuses larger pieces of workspace): what faster paths ask for
beyond the ways they replaced is not needed, and the results are the same."""
import contextlib
import os

import numpy as np
import pytest

import gen
from tests.gpu_util import bits, dev, f32_matrix, host, int_matrix

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def btas():
    import paper_1701_04733_gb300 as m
    return m


@contextlib.contextmanager
def limit(nbytes):
    os.environ["BTAS_WS_LIMIT"] = str(nbytes)
    try:
        yield
    finally:
        del os.environ["BTAS_WS_LIMIT"]


@pytest.mark.parametrize("n", [40, 300, 1030])
def test_sssp_without_edge_lists(btas, oracle_mod, n):
    """Two vectors and 256 bytes, as one launch per product takes."""
    W = gen.random_graph(gen.BASE_SEED, 61 + n, n, 0.1, 1, 1000)
    want, info = btas.sssp(dev(W), 3, info=True)
    with limit(256 + 2 * ((4 * n + 255) // 256 * 256)):
        d, info1 = btas.sssp(dev(W), 3, info=True)
    np.testing.assert_array_equal(host(d), host(want))
    np.testing.assert_array_equal(host(d), oracle_mod.sssp(W, 3)[0])
    assert info1["iterations"] == info["iterations"]


@pytest.mark.parametrize("dt", ["i32", "f32"])
@pytest.mark.parametrize("trans_b", [False, True])
def test_product_without_aligned_copies(btas, oracle_mod, dt, trans_b):
    """Rows off 16 bytes, in a product large enough for aligned copies: room for B's transpose, or for nothing."""
    m, n, k = 700, 800, 801
    make = int_matrix if dt == "i32" else f32_matrix
    A, B = make(15, (m, k), 0), make(17, (k, n), 0)
    Bd = dev(np.ascontiguousarray(B.T)) if trans_b else dev(B)
    with limit(0 if trans_b else n * ((k + 3) // 4 * 4) * 4):
        C = btas.gemm(dev(A), Bd, 0, trans_b=trans_b)
    np.testing.assert_array_equal(bits(host(C)), bits(oracle_mod.tgemm(0, A, B)))


@pytest.mark.parametrize("n", [100, 1000, 2100])
def test_apsp_in_place_without_a_copy(btas, n):
    """Room for the squarings' workspace that the thread keeps (or Floyd-Warshall's panels), not for a copy of W."""
    W = gen.random_graph(gen.BASE_SEED, 63 + n, n, 0.02 if n > 100 else 0.2, 1, 100)
    want = host(btas.apsp(dev(W)))
    t = dev(W)
    with limit(n * n * 4 - 1):
        btas.apsp(t, out=t)
    np.testing.assert_array_equal(host(t), want)


def test_apsp_without_edge_lists(btas):
    """n = 8200: the lists take more than the 32 MiB a thread keeps, Floyd-Warshall's panels a third of that."""
    import torch
    W = dev(gen.random_graph(gen.BASE_SEED, 65, 8200, 0.002, 1, 1000))
    want = btas.apsp(W)
    with limit(12 << 20):
        D = btas.apsp(W)
        btas.apsp(W, out=W)
    assert torch.equal(D, want) and torch.equal(W, want)


@pytest.mark.parametrize("n", [130, 515])
def test_next_hops_without_edge_lists(btas, n):
    """Room for the matrices of the keyed squarings only; a sparse graph, whose first squaring would use the lists, and
    a W outside the domain, which they would have found."""
    W = gen.random_graph(gen.BASE_SEED, 67 + n, n, 0.05, 1, 100)
    D, N, info = btas.apsp_paths(dev(W), info=True)
    up = lambda x: (x + 255) // 256 * 256  # noqa: E731
    S = int(np.ceil(np.log2(n - 1)))
    pitch = (n + 3) // 4 * 4
    with limit(up((2 * S + 4) * 4) + 4 * up(n * n * 4) + 2 * up(n * pitch * 4)):
        D1, N1, info1 = btas.apsp_paths(dev(W), info=True)
        W[3, 5] = -1
        with pytest.raises(btas.BtasError) as ei:
            btas.apsp_paths(dev(W))
    assert ei.value.status == 1
    np.testing.assert_array_equal(host(D1), host(D))
    np.testing.assert_array_equal(host(N1), host(N))
    assert info1["squarings"] == info["squarings"]


def test_batch_needs_the_squarings_space_only(btas, oracle_mod):
    """A solve's lists lie in the space of its squarings; with no time for the relaxations the squarings take it over."""
    graphs = [gen.random_graph(gen.BASE_SEED, 69 + n, n, 0.1 if n > 10 else 0.5, 1, 100) for n in (3, 5, 9, 33, 300, 530)]

    def batch():
        b = btas.Batch()
        outs = [b.add_apsp(dev(W), dev(np.zeros_like(W))) for W in graphs]
        b.launch()
        b.wait()
        nbytes = b.workspace_bytes
        b.close()
        for W, D in zip(graphs, outs):
            np.testing.assert_array_equal(host(D), oracle_mod.floyd_warshall(W))
        return nbytes

    got = batch()
    os.environ["BTAS_RELAX_BUDGET"] = "-1"
    try:
        assert batch() == got
    finally:
        del os.environ["BTAS_RELAX_BUDGET"]
    os.environ["BTAS_BATCH_NO_RELAX"] = "1"
    try:
        squarings = batch()
    finally:
        del os.environ["BTAS_BATCH_NO_RELAX"]
    # lists of 32 rows are larger than the squarings' buffers of the smallest graphs only
    assert squarings <= got <= squarings + 3 * 4096
