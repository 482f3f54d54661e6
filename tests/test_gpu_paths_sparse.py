"""btas_apsp_paths with its first squaring over edge lists: the same distances,
next hops and number of squarings as the argmin kernel's, on ties, zero weights,
rows as long as the lists, and sizes where the matrices' rows are not aligned."""
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


def graph(n, p, lo, hi, seed):
    W = gen.random_graph(gen.BASE_SEED, seed + n, n, p, 1, hi - lo + 1)
    return np.where((W < INF) & ~np.eye(n, dtype=bool), W - 1 + lo, W).astype(np.int32)


def hub(n, more=0):
    """A row with n // 6 edges, the most that still takes the sparse squaring, and one with `more` above that."""
    W = graph(n, 2.0 / n, 1, 9, 83)
    for r, m in ((1, n // 6), (n - 2, n // 6 + more)):
        W[r] = INF
        W[r, :m + 1] = 3 + np.arange(m + 1) % 5
        W[r, r] = 0
    return W


CASES = {"ties": lambda n: graph(n, 0.05, 1, 3, 81), "zeros": lambda n: graph(n, 0.05, 0, 2, 82), "hub": hub,
         "one row too long": lambda n: hub(n, 1), "too heavy": lambda n: graph(n, 0.04, 49000, 49400, 88),
         "heavy": lambda n: graph(n, 0.04, 1, 49151, 84), "dense": lambda n: graph(n, 0.5, 1, 1000, 85),
         "empty": lambda n: graph(n, 0.0, 1, 1, 86)}


@pytest.mark.parametrize("n", [3, 33, 130, 515, 1030])
@pytest.mark.parametrize("case", sorted(CASES))
def test_equals_the_argmin_kernel(btas, case, n):
    W = dev(CASES[case](n))
    D, N, info = btas.apsp_paths(W, info=True)
    os.environ["BTAS_PATHS_NO_KEYED"] = "1"
    try:
        D0, N0, info0 = btas.apsp_paths(W, info=True)
    finally:
        del os.environ["BTAS_PATHS_NO_KEYED"]
    np.testing.assert_array_equal(host(D), host(D0))
    np.testing.assert_array_equal(host(N), host(N0))
    assert info["squarings"] == info0["squarings"]


@pytest.mark.parametrize("p", [0.08, 0.115, 0.13])
def test_rows_about_as_long_as_a_list(btas, p):
    """n = 4100: rows of about 330, 470 and 530 edges, where a list of 512 may be cut."""
    n = 4100
    W = dev(gen.random_graph(gen.BASE_SEED, 87, n, p, 1, 100))
    D, N = btas.apsp_paths(W)
    os.environ["BTAS_PATHS_NO_KEYED"] = "1"
    try:
        D0, N0 = btas.apsp_paths(W)
    finally:
        del os.environ["BTAS_PATHS_NO_KEYED"]
    import torch
    assert torch.equal(D, D0) and torch.equal(N, N0)
