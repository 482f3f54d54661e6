"""Which graphs btas_apsp_paths still squares over edge lists: no row of more than n / 6 edges, and from n = 800 on no
more than n / 8 per row on average."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import os
import sys
sys.path.insert(0, {root!r})
import numpy as np
import torch
import paper_1701_04733_gb300 as btas
n, rows, all_rows = {n}, {rows}, {all_rows}
W = np.full((n, n), 0x3FFFFFFF, np.int32)
W[np.arange(n), (np.arange(n) + 1) % n] = 2
W[5, :rows + 1] = 3
if all_rows:
    W[5] = 0x3FFFFFFF
    for d in range(1, rows + 1):
        W[np.arange(n), (np.arange(n) + d) % n] = 2 + d % 5
np.fill_diagonal(W, 0)
D, N = btas.apsp_paths(torch.from_numpy(W).cuda())
assert int((torch.from_numpy(W)[5] < 0x3FFFFFFF).sum()) - 1 == rows
os.environ["BTAS_PATHS_NO_KEYED"] = "1"
D0, N0 = btas.apsp_paths(torch.from_numpy(W).cuda())
assert torch.equal(D, D0) and torch.equal(N, N0)
"""


@pytest.mark.parametrize("n,rows,all_rows,lists", [
    (600, 100, False, True), (600, 101, False, False), (799, 133, True, True), (800, 133, False, True),
    (800, 134, False, False), (800, 100, True, True), (800, 101, True, False), (1030, 128, True, True),
    (1030, 129, True, False), (1030, 171, False, True), (1030, 172, False, False)])
def test_longest_row_and_average(n, rows, all_rows, lists):
    r = subprocess.run([sys.executable, "-c", SCRIPT.format(root=ROOT, n=n, rows=rows, all_rows=all_rows)],
                       env=dict(os.environ, BTAS_LOG="1"), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert any("first squaring over edge lists" in x for x in r.stderr.splitlines()) == lists
