"""Products whose tiles share their k range over several CTAs (merged into C with
atomics), on the 64 x 64 and 32 x 32 tiles, and products whose unaligned operands
are copied first: bit for bit the oracle's."""
import os

import numpy as np
import pytest

from tests.gpu_util import bits, dev, f32_matrix, host, int_matrix

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def btas():
    import paper_1701_04733_gb300 as m
    return m


def operands(dt, sr, m, n, k):
    make = int_matrix if dt == "i32" else f32_matrix  # signed values, a tenth of them the (+)-identity
    return make(11, (m, k), sr), make(13, (k, n), sr)


@pytest.mark.parametrize("cfg", ["6", "7"])
@pytest.mark.parametrize("dt", ["i32", "f32"])
@pytest.mark.parametrize("sr", [0, 1])
def test_split_tiles(btas, oracle_mod, cfg, dt, sr):
    """k steps that divide by the split and that do not, single rows and columns, tile edges, whole rows of C with no
    finite term."""
    for m, n, k in ((1, 1, 64), (31, 33, 95), (32, 64, 129), (65, 63, 200), (130, 70, 321)):
        A, B = operands(dt, sr, m, n, k)
        A[m // 2] = (0x3FFFFFFF if sr == 0 else -0x3FFFFFFF) if dt == "i32" else (np.inf if sr == 0 else -np.inf)
        ref = oracle_mod.tgemm(sr, A, B)
        for split in ("1", "2", "3", "7"):
            os.environ.update(BTAS_CFG=cfg, BTAS_SPLIT=split)
            try:
                C = btas.gemm(dev(A), dev(B), sr)
                Ct = btas.gemm(dev(A), dev(np.ascontiguousarray(B.T)), sr, trans_b=True)
            finally:
                del os.environ["BTAS_CFG"], os.environ["BTAS_SPLIT"]
            for X in (C, Ct):
                np.testing.assert_array_equal(bits(host(X)), bits(ref), err_msg=f"{m}x{n}x{k} split {split}")


@pytest.mark.parametrize("dt", ["i32", "f32"])
@pytest.mark.parametrize("sr", [0, 1])
def test_equal_shares(btas, oracle_mod, dt, sr):
    """All (tile, k step) units in equal shares for 304 CTAs: fewer units than CTAs (empty shares), parts of one tile,
    and shares that span tiles."""
    for m, n, k in ((100, 100, 70), (129, 257, 1000), (700, 650, 333)):
        A, B = operands(dt, sr, m, n, k)
        os.environ.update(BTAS_CFG="4", BTAS_SPLIT="0")
        try:
            C = btas.gemm(dev(A), dev(B), sr)
        finally:
            del os.environ["BTAS_CFG"], os.environ["BTAS_SPLIT"]
        np.testing.assert_array_equal(bits(host(C)), bits(oracle_mod.tgemm(sr, A, B)), err_msg=f"{m}x{n}x{k}")


@pytest.mark.parametrize("dt", ["i32", "f32"])
@pytest.mark.parametrize("m,n,k", [(1, 1, 5000), (33, 40, 3000), (700, 20, 130), (20, 900, 64), (513, 517, 1601)])
def test_default_choice(btas, oracle_mod, dt, m, n, k):
    """The sizes' own choice of tiles and split, with every form of call; (513, 517, 1601) also copies A, and B^T."""
    for sr in (0, 1):
        A, B = operands(dt, sr, m, n, k)
        ref = oracle_mod.tgemm(sr, A, B)
        Bt = np.ascontiguousarray(B.T)
        np.testing.assert_array_equal(bits(host(btas.gemm(dev(A), dev(B), sr))), bits(ref))
        np.testing.assert_array_equal(bits(host(btas.gemm(dev(A), dev(Bt), sr, trans_b=True))), bits(ref))
        np.testing.assert_array_equal(bits(host(btas.gemm(dev(A), dev(B), sr, checked=True))), bits(ref))
        C0 = operands(dt, sr, m, n, n)[1][:m] if m <= n else operands(dt, sr, n, n, m)[1]
        C0 = np.ascontiguousarray(C0)
        acc = btas.gemm(dev(A), dev(B), sr, out=dev(C0), accumulate=True)
        np.testing.assert_array_equal(bits(host(acc)), bits(oracle_mod.tgemm(sr, A, B, C0.copy())))
    assert btas.sync_status()[0] == 0


def test_pitched_output(btas, oracle_mod):
    """A split product into a column block of a wider matrix writes that block only."""
    import torch
    m, n, k = 50, 37, 2000
    A, B = operands("i32", 0, m, n, k)
    W = torch.full((m, 64), 9, dtype=torch.int32, device="cuda")
    btas.gemm(dev(A), dev(B), 0, out=W[:, 5:5 + n])
    got = host(W)
    np.testing.assert_array_equal(got[:, 5:5 + n], oracle_mod.tgemm(0, A, B))
    assert (got[:, :5] == 9).all() and (got[:, 5 + n:] == 9).all()
