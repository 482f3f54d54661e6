"""Batched APSP of matrices outside the domain, which a batch assumes and does not check: the graphs beside them are
unharmed, and in 32 bits the result is whatever the squarings make of them.  (Packed squarings rely on the domain to
know which operands the next one needs, so theirs is not a function of W outside it.)"""
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


def solve(btas, graphs):
    b = btas.Batch()
    outs = [b.add_apsp(dev(W), dev(np.full_like(W, 5))) for W in graphs]
    for _ in range(2):
        b.launch()
        b.wait()
    b.close()
    return [host(o) for o in outs]


@pytest.mark.parametrize("value", [-1, -(1 << 31), INF - 1, INF + 1, (1 << 31) - 1])
@pytest.mark.parametrize("where", ["an edge", "a diagonal entry", "no edge"])
def test_as_the_squarings_give_them(btas, oracle_mod, value, where):
    """Sparse rows (lists that end with pads), weights for 16 and for 32 bits, one wrong entry or every missing edge."""
    graphs = []
    for n, w in ((40, 9), (130, 100), (200, 10 ** 6)):
        W = gen.random_graph(gen.BASE_SEED, 91 + n, n, 0.05, 1, w)
        if where == "an edge":
            W[n // 2, n // 3] = value
        elif where == "a diagonal entry":
            W[n // 2, n // 2] = value
        else:
            W[W == INF] = value
        graphs += [W, gen.random_graph(gen.BASE_SEED, 95 + n, n, 0.1, 1, w)]
    got = solve(btas, graphs)
    os.environ["BTAS_BATCH_NO_RELAX"] = "1"
    try:
        want = solve(btas, graphs)
    finally:
        del os.environ["BTAS_BATCH_NO_RELAX"]
    for i, (x, y) in enumerate(zip(got, want)):
        if i % 2 or (i // 2 == 2 and value > 0):  # n = 200: distances too large for the packed squarings
            np.testing.assert_array_equal(x, y)
        if i % 2:
            np.testing.assert_array_equal(x, oracle_mod.floyd_warshall(graphs[i]))
