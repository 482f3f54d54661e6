"""btas_sssp in one cooperative launch, products over the frontier's edges: the
same distances and the same number of products as one launch per product, and
the oracle's distances, for rows within and beyond the edge lists."""
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


def graph(n, p, w, seed):
    return gen.random_graph(gen.BASE_SEED, seed + n, n, p, 1, w)


def mixed_rows(n):
    """A sparse graph with a few complete rows: lists and rows of W in one solve."""
    W = graph(n, 2.0 / n, 50, 71)
    W[n // 2, :] = 40 + np.arange(n) % 60
    W[3, :] = 200
    W[np.arange(n), np.arange(n)] = 0
    return W


def path(n):
    W = np.full((n, n), INF, np.int32)
    np.fill_diagonal(W, 0)
    W[np.arange(n - 1), np.arange(1, n)] = 1 << 20
    return W


CASES = {"sparse": lambda n: graph(n, min(1.0, 4.0 / n), 1000, 61), "dense": lambda n: graph(n, 1.0, 10 ** 6, 63),
         "heavy": lambda n: graph(n, min(1.0, 6.0 / n), 1 << 28, 65), "mixed": mixed_rows, "path": path}


@pytest.mark.parametrize("n", [4, 31, 64, 257, 1023, 1024, 1030])
@pytest.mark.parametrize("case", sorted(CASES))
def test_equals_one_launch_per_product(btas, oracle_mod, case, n):
    W = CASES[case](n)
    Wd, src = dev(W), n // 3
    d, info = btas.sssp(Wd, src, info=True)
    os.environ["BTAS_SSSP_NO_COOP"] = "1"
    try:
        d0, info0 = btas.sssp(Wd, src, info=True)
    finally:
        del os.environ["BTAS_SSSP_NO_COOP"]
    np.testing.assert_array_equal(host(d), host(d0))
    assert info["iterations"] == info0["iterations"]
    ref, _ = oracle_mod.sssp(W, src)
    ref[ref >= INF - (1 << 28)] = INF  # the encoding: sums from there on are INF
    np.testing.assert_array_equal(host(d), ref)
