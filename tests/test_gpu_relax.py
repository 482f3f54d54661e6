"""btas_apsp by relaxation over sorted edge lists: equal to the oracle's
Floyd-Warshall, and to the squarings, bit for bit on every form of graph and
size at which its lists, its 16-bit distances or its split over blocks change."""
import os

import numpy as np
import pytest

import gen
from tests.gpu_util import dev, host

pytestmark = pytest.mark.gpu

INF = 0x3FFFFFFF


@pytest.fixture(scope="module")
def btas():
    import paper_1701_04733_gb300 as m
    return m


def empty(n):
    W = np.full((n, n), INF, np.int32)
    np.fill_diagonal(W, 0)
    return W


def path(n):
    W = empty(n)
    W[np.arange(n - 1), np.arange(1, n)] = 3
    return W


def hidden_heavy_edge(n):
    """Vertex 0 has n - 60 light edges to dead ends (more than a list holds)
    and one heavy edge to the first of 50 vertices on a path, which only the
    row itself can show."""
    W = empty(n)
    W[0, 1:n - 60] = 1 + np.arange(n - 61) % 5
    W[0, n - 60] = 900
    W[np.arange(n - 60, n - 1), np.arange(n - 59, n)] = 2
    W[n - 1, 0] = 1
    return W


def two_blocks(n):
    """Two complete graphs without an edge between them: half of all distances stay INF."""
    W = gen.random_graph(gen.BASE_SEED, 31 + n, n, 1.0, 1, 50)
    h = n // 2
    W[:h, h:] = INF
    W[h:, :h] = INF
    return W


def zeros(n):
    W = gen.random_graph(gen.BASE_SEED, 37 + n, n, 0.1, 1, 3)
    W[W == 1] = 0
    return W


def equal_but_few(n):
    """Rows of equal weights, longer than a list, with light edges anywhere among them: the list keeps every
    light edge."""
    light = gen.random_graph(gen.BASE_SEED, 47 + n, n, 0.02, 1, 20)
    W = np.where(light < INF, light, 1000).astype(np.int32)
    np.fill_diagonal(W, 0)
    return W


def clamped(n):
    """Weights up to 2^28: three of them reach the clamp, and the distance is INF."""
    W = gen.random_graph(gen.BASE_SEED, 41 + n, n, 3.0 / n, 1 << 27, 1 << 28)
    W[0, 1] = 1 << 28
    return W


def random(p, w):
    return lambda n: gen.random_graph(gen.BASE_SEED, 43 + n, n, p, 1, w)


GRAPHS = {"empty": empty, "path": path, "two_blocks": two_blocks, "zeros": zeros, "clamped": clamped,
          "sparse": random(0.02, 100), "sparse_heavy": random(0.03, 10 ** 6), "dense_ties": random(1.0, 2),
          "equal_but_few": equal_but_few,
          "dense_heavy": random(0.6, 10 ** 6), "border": random(0.05, 12000)}


@pytest.mark.parametrize("n", [49, 64, 65, 256, 257, 513, 1100])
@pytest.mark.parametrize("graph", sorted(GRAPHS))
def test_equals_floyd_warshall(btas, oracle_mod, graph, n):
    W = GRAPHS[graph](n)
    ref = oracle_mod.floyd_warshall(W)
    ref[ref >= INF - (1 << 28)] = INF  # the encoding: sums from there on are INF
    np.testing.assert_array_equal(host(btas.apsp(dev(W))), ref)
    t = dev(W)  # in place
    btas.apsp(t, out=t)
    np.testing.assert_array_equal(host(t), ref)


@pytest.mark.parametrize("n,p,w", [(1217, 0.05, 100), (2047, 1.0, 7), (2048, 1.0, 10 ** 6), (3001, 0.01, 10 ** 6),
                                   (7001, 0.003, 1000)])
def test_larger_sizes_equal_the_squarings(btas, n, p, w):
    """Long rows (the sampled cutoff from n = 2048), one block of 1024 threads
    per SM from n = 7001, 32 bits without the split over blocks."""
    import torch
    W = dev(gen.random_graph(gen.BASE_SEED, 47 + n, n, p, 1, w))
    D, _ = btas.apsp(W, info=True)
    assert torch.equal(btas.apsp(W), D)


@pytest.mark.parametrize("n", [640, 2100])
def test_row_beyond_its_list(btas, oracle_mod, n):
    W = hidden_heavy_edge(n)
    np.testing.assert_array_equal(host(btas.apsp(dev(W))), oracle_mod.floyd_warshall(W))


def test_unaligned_matrices(btas, oracle_mod):
    import torch
    n = 128
    W = gen.random_graph(gen.BASE_SEED, 51, n, 0.1, 1, 100)
    a, b = (torch.empty(n * n + 1, dtype=torch.int32, device="cuda") for _ in range(2))
    w, d = a[1:].view(n, n), b[1:].view(n, n)
    w.copy_(dev(W))
    b[0] = 77
    btas.apsp(w, out=d)
    np.testing.assert_array_equal(host(d), oracle_mod.floyd_warshall(W))
    assert int(b[0]) == 77


@pytest.mark.parametrize("n", [100, 2100])
@pytest.mark.parametrize("in_place", [False, True])
def test_given_up_solves_still_finish(btas, n, in_place):
    """With no time allowed every block gives up after a few sweeps; the
    squarings (or Floyd-Warshall) then solve the graph, also in place."""
    W = path(n)
    ref = np.triu(3 * (np.arange(n)[None, :] - np.arange(n)[:, None]).astype(np.int32))
    ref[np.tril_indices(n, -1)] = INF
    os.environ["BTAS_RELAX_BUDGET"] = "0"
    try:
        t = dev(W)
        out = btas.apsp(t, out=t if in_place else None)
    finally:
        del os.environ["BTAS_RELAX_BUDGET"]
    np.testing.assert_array_equal(host(out), ref)


def test_given_up_solve_keeps_the_encoding(btas):
    """Floyd-Warshall instead: distances from INF - 2^28 on are INF, as the squarings give them."""
    import torch
    W = dev(clamped(2100))
    D, _ = btas.apsp(W, info=True)
    os.environ["BTAS_RELAX_BUDGET"] = "0"
    try:
        out = btas.apsp(W)
    finally:
        del os.environ["BTAS_RELAX_BUDGET"]
    assert torch.equal(out, D)


@pytest.mark.parametrize("value", [-1, (1 << 28) + 1])
def test_domain_violation_leaves_the_result_untouched(btas, value):
    n = 300
    W = gen.random_graph(gen.BASE_SEED, 53, n, 0.1, 1, 100)
    W[7, 250] = value
    out = dev(np.full((n, n), 19, np.int32))
    with pytest.raises(btas.BtasError) as ei:
        btas.apsp(dev(W), out=out)
    assert ei.value.status == 1
    assert (host(out) == 19).all()


def solve_batch(btas, graphs, graph=True):
    b = btas.Batch(graph=graph)
    outs = [b.add_apsp(dev(W), dev(np.full_like(W, 5))) for W in graphs]
    A = dev(gen.uniform_int(3, 9, (300, 200), 0, 1000))
    C = b.add_gemm(A, A, dev(np.zeros((300, 300), np.int32)), trans_b=True)
    results = []
    for _ in range(2):  # the second launch replays the plan
        b.launch()
        b.wait()
        results.append([host(o).copy() for o in outs + [C]])
    b.close()
    for x, y in zip(*results):
        np.testing.assert_array_equal(x, y)
    np.testing.assert_array_equal(results[0][-1], host(btas.gemm(A, A, trans_b=True)))
    return results[0][:-1]


@pytest.mark.parametrize("graph", [True, False])
def test_batched_relaxation(btas, oracle_mod, graph):
    """Every form of graph and the sizes around 2, a list task's rows and a list's capacity, beside a product."""
    graphs = [GRAPHS[g](n) for g in sorted(GRAPHS) for n in (33, 150)]
    graphs += [random(0.3, 100)(n) for n in (1, 2, 3, 7, 8, 9, 31, 32, 511, 512, 513, 700)]
    graphs.append(hidden_heavy_edge(640))
    for W, D in zip(graphs, solve_batch(btas, graphs, graph)):
        ref = oracle_mod.floyd_warshall(W)
        ref[ref >= INF - (1 << 28)] = INF
        np.testing.assert_array_equal(D, ref)


def test_batched_relaxation_given_up(btas, oracle_mod):
    """Long paths with no time allowed: their squarings run, the other solves' do not have to."""
    graphs = [path(100), random(0.2, 100)(60), path(300), random(0.05, 100)(300)]
    os.environ["BTAS_RELAX_BUDGET"] = "0"
    try:
        outs = solve_batch(btas, graphs)
    finally:
        del os.environ["BTAS_RELAX_BUDGET"]
    for W, D in zip(graphs, outs):
        np.testing.assert_array_equal(D, oracle_mod.floyd_warshall(W))
