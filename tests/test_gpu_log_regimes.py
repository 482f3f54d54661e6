"""BTAS_LOG=1 says what ran: the relaxation (or Floyd-Warshall after it) where that solved a plain call, and the squarings'
own lines, from the dispatch that chose them, where BTAS_APSP_NO_RELAX=1 keeps to them."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import sys
sys.path.insert(0, {root!r})
import torch
import gen
import paper_1701_04733_gb300 as btas
btas.apsp(torch.from_numpy(gen.random_graph(1, 1, {n}, {p}, 1, 100)).cuda())
"""


def lines(n, p, **env):
    r = subprocess.run([sys.executable, "-c", SCRIPT.format(root=ROOT, n=n, p=p)],
                       env=dict(os.environ, BTAS_LOG="1", **env), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return [x.split("] ", 1)[1] for x in r.stderr.splitlines() if x.startswith(f"[btas] apsp n={n}: ")]


@pytest.mark.parametrize("n,p,kernel", [(60, 0.1, "one-block kernel, int32"),
                                        (300, 0.1, "cooperative kernel, representations"),
                                        (2000, 0.1, "cooperative kernel, representations"),
                                        (2816, 0.5, "tiled kernels, representations"),
                                        (4608, 0.02, "tiled kernels, representations")])
def test_squarings(n, p, kernel):
    got = lines(n, p, BTAS_APSP_NO_RELAX="1")
    assert got[-1].startswith(f"apsp n={n}: {kernel}") and not any("relaxation" in x for x in got)
    assert len(got) == 1 + (n == 2816)  # which the cooperative kernel declines first
    if n == 2816:
        assert got[0] == f"apsp n={n}: too dense for the cooperative kernel's edge lists"


@pytest.mark.parametrize("n,p", [(60, 0.1), (300, 0.1), (2816, 0.5), (4608, 0.02)])
def test_relaxation(n, p):
    got = lines(n, p)
    assert got[-1].endswith("replaced by relaxation over sorted edge lists in 16 bits")
    assert not any("representations" in x or "int32" in x for x in got)


@pytest.mark.parametrize("n,last", [(600, "cooperative kernel, representations"),
                                    (2100, "tiled kernels replaced by blocked Floyd-Warshall")])
def test_given_up(n, last):
    got = lines(n, 0.01, BTAS_RELAX_BUDGET="-1")
    assert len(got) == 2 and got[0].endswith("in 16 bits, given up")
    assert got[1].startswith(f"apsp n={n}: {last}")
