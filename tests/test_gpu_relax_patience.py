"""When a relaxation is given up: graphs whose shortest paths have many edges are solved by it while that is cheaper
than the squarings, and the others left to them; the distances are the same."""
import os
import subprocess
import sys

import numpy as np
import pytest

from tests.gpu_util import dev, host

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
INF = 0x3FFFFFFF


@pytest.fixture(scope="module")
def btas():
    import paper_1701_04733_gb300 as m
    return m


def band(n, w, steps, wrap, both=True):
    """Edges from every vertex to those `steps` further on, around the end with `wrap`, and back with `both`."""
    rng = np.random.default_rng(n + w)
    W = np.full((n, n), INF, np.int32)
    for s in steps:
        i = np.arange(n if wrap else n - s)
        W[i, (i + s) % n] = rng.integers(1, w + 1, len(i))
        if both:
            W[(i + s) % n, i] = rng.integers(1, w + 1, len(i))
    np.fill_diagonal(W, 0)
    return W


def steep(n, w):
    """A complete graph whose shortest paths take every vertex on the way: all distances are known at once."""
    d = np.abs(np.arange(n)[:, None] - np.arange(n)[None, :])
    return np.minimum(d * d * w, 1 << 28).astype(np.int32)


GRAPHS = {"chain": lambda n, w: band(n, w, [1], False, both=False), "ring": lambda n, w: band(n, w, [1], True),
          "grid": lambda n, w: band(n, w, [1, int(n ** 0.5)], False), "lattice": lambda n, w: band(n, w, range(1, 9), True),
          "steep": steep}


@pytest.mark.parametrize("w", [7, 10 ** 6])
@pytest.mark.parametrize("shuffled", [False, True])
@pytest.mark.parametrize("graph", sorted(GRAPHS))
def test_long_paths(btas, oracle_mod, graph, shuffled, w):
    """One call at a time and as a batch; sizes on both sides of 2, 4 and 8 targets per block."""
    Ws = []
    for n in (65, 300, 500, 700):
        W = GRAPHS[graph](n, w)
        if shuffled:
            p = np.random.default_rng(n).permutation(n)
            W = np.ascontiguousarray(W[p][:, p])
        Ws.append(W)
    b = btas.Batch()
    outs = [b.add_apsp(dev(W), dev(np.zeros_like(W))) for W in Ws]
    b.launch()
    b.wait()
    b.close()
    for W, D in zip(Ws, outs):
        ref = oracle_mod.floyd_warshall(W)
        ref[ref >= INF - (1 << 28)] = INF
        np.testing.assert_array_equal(host(D), ref)
        np.testing.assert_array_equal(host(btas.apsp(dev(W))), ref)


SCRIPT = """
import sys
sys.path.insert(0, {root!r})
import paper_1701_04733_gb300 as btas
from tests.gpu_util import dev
from tests.test_gpu_relax_patience import GRAPHS
btas.apsp(dev(GRAPHS[{graph!r}]({n}, 7)))
"""


@pytest.mark.parametrize("graph,n,finishes", [("lattice", 1024, True), ("lattice", 2047, True), ("chain", 1024, False),
                                              ("chain", 2047, False)])
def test_goes_on_while_it_is_the_cheaper_way(graph, n, finishes):
    """Lattices of 16 neighbours: half of what the squarings take.  Chains: twice as much, which shows early."""
    r = subprocess.run([sys.executable, "-c", SCRIPT.format(root=ROOT, graph=graph, n=n)],
                       env=dict(os.environ, BTAS_LOG="1"), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [x for x in r.stderr.splitlines() if "relaxation" in x]
    assert len(lines) == 1 and ("given up" not in lines[0]) == finishes, lines
