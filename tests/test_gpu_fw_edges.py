"""Blocked Floyd-Warshall where its rows do not start on 16 bytes, called directly and
as what btas.apsp falls back to, and its encoding of long distances."""
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


def offset(W, by):
    """W on the device, `by` elements into its buffer; and the buffer."""
    import torch
    n = W.shape[0]
    buf = torch.full((n * n + 8,), 77, dtype=torch.int32, device="cuda")
    v = buf[by:by + n * n].view(n, n)
    v.copy_(dev(W))
    return v, buf


def untouched(buf, by, n):
    return bool((buf[:by] == 77).all()) and bool((buf[by + n * n:] == 77).all())


@pytest.mark.parametrize("packed", ["0", "1"])
@pytest.mark.parametrize("n", [4, 128, 132, 300, 516])
@pytest.mark.parametrize("by", [1, 2, 3])
def test_matrices_at_any_element(btas, oracle_mod, n, by, packed):
    """n a multiple of 4, so that the address alone decides against vectors: W, D and both (in place) off 16 bytes."""
    W = gen.random_graph(33, n, n, 0.05 if n > 10 else 0.5, 0, 100 if packed == "1" else 10 ** 6)
    ref = oracle_mod.floyd_warshall(W)
    w, wbuf = offset(W, by)
    d, dbuf = offset(np.zeros_like(W), by)
    os.environ["BTAS_FW_NO_U16"] = "0" if packed == "1" else "1"
    try:
        btas.apsp_fw(w, out=d)
        np.testing.assert_array_equal(host(d), ref)
        btas.apsp_fw(w, out=w)
    finally:
        del os.environ["BTAS_FW_NO_U16"]
    np.testing.assert_array_equal(host(w), ref)
    assert untouched(wbuf, by, n) and untouched(dbuf, by, n)


@pytest.mark.parametrize("in_place", [False, True])
def test_apsp_falls_back_to_it_at_any_element(btas, in_place):
    """n = 2100, given up by the relaxation."""
    n = 2100
    W = np.full((n, n), 0x3FFFFFFF, np.int32)
    np.fill_diagonal(W, 0)
    W[np.arange(n - 1), np.arange(1, n)] = 3
    ref = np.triu(3 * (np.arange(n)[None, :] - np.arange(n)[:, None]).astype(np.int32))
    ref[np.tril_indices(n, -1)] = 0x3FFFFFFF
    w, wbuf = offset(W, 1)
    d, dbuf = (w, wbuf) if in_place else offset(np.zeros_like(W), 1)
    os.environ["BTAS_RELAX_BUDGET"] = "0"
    try:
        btas.apsp(w, out=d)
    finally:
        del os.environ["BTAS_RELAX_BUDGET"]
    np.testing.assert_array_equal(host(d), ref)
    assert untouched(dbuf, 1, n)


@pytest.mark.parametrize("ahead", ["0", "1"])
@pytest.mark.parametrize("n", [3, 5, 128, 129, 300, 517])
def test_long_distances_keep_the_encoding(btas, oracle_mod, n, ahead):
    """Weights up to 2^28: three or more of them reach INF - 2^28, and the entry is INF, in every tile: the last
    pivot block's, which no product touches afterwards, included."""
    W = gen.random_graph(gen.BASE_SEED, 41 + n, n, min(0.5, 3.0 / n), 1 << 27, 1 << 28)
    W[np.arange(n - 1), np.arange(1, n)] = 1 << 28
    ref = oracle_mod.floyd_warshall(W)
    assert n < 128 or ((ref >= INF - (1 << 28)) & (ref < INF)).any()  # some entries need it
    ref[ref >= INF - (1 << 28)] = INF
    os.environ["BTAS_FW_NO_LOOKAHEAD"] = "0" if ahead == "1" else "1"
    try:
        np.testing.assert_array_equal(host(btas.apsp_fw(dev(W))), ref)
    finally:
        del os.environ["BTAS_FW_NO_LOOKAHEAD"]
    np.testing.assert_array_equal(host(btas.apsp(dev(W))), ref)
