"""Products whose k ranges stay whole (accumulate, checked, squarings): the choice of tiles against each of them, where
the last CTAs of an SM run alone."""
import os

import numpy as np
import pytest

from tests.gpu_util import bits, dev, f32_matrix, host, int_matrix

pytestmark = pytest.mark.gpu

SIZES = [(1000, 1000, 1000), (1024, 1024, 1024), (5000, 200, 300), (700, 700, 700)]


@pytest.fixture(scope="module")
def btas():
    import paper_1701_04733_gb300 as m
    return m


@pytest.mark.parametrize("dt", ["i32", "f32"])
@pytest.mark.parametrize("m,n,k", SIZES)
def test_choice_of_tiles(btas, dt, m, n, k):
    """Each side is the fastest of 6 rounds of 10 calls; the model's own error over 44 shapes is 5 %, and the choice was
    1.2 to 1.6 times the best at the first three sizes."""
    import torch
    if dt == "i32":
        A, B = (torch.randint(0, 1000, s, dtype=torch.int32, device="cuda") for s in ((m, k), (n, k)))
    else:
        A, B = torch.rand(m, k, device="cuda"), torch.rand(n, k, device="cuda")
    C = btas.gemm(A, B, 0, trans_b=True)

    def best():
        times = []
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                btas.gemm(A, B, 0, out=C, trans_b=True, accumulate=True)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    best()
    for attempt in range(4):  # a burst of other work on the host can spoil one
        chosen, fixed = best(), []
        for cfg in ("4", "6", "7"):
            os.environ["BTAS_CFG"] = cfg
            try:
                fixed.append(best())
            finally:
                del os.environ["BTAS_CFG"]
        if chosen < 1.12 * min(fixed):
            break
    assert chosen < 1.12 * min(fixed), (chosen, fixed)


@pytest.mark.parametrize("dt", ["i32", "f32"])
def test_accumulate_in_the_chosen_tiles(btas, oracle_mod, dt):
    make = int_matrix if dt == "i32" else f32_matrix
    m, n, k = 1000, 1000, 40
    A, B, C = make(3, (m, k), 0), make(5, (k, n), 0), make(7, (m, n), 0)
    got = btas.gemm(dev(A), dev(B), 0, out=dev(C), accumulate=True)
    np.testing.assert_array_equal(bits(host(got)), bits(oracle_mod.tgemm(0, A, B, C.copy())))
