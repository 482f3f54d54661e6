"""Tuned entries and products that only write C, whose untuned choice (k ranges shared over CTAs, smaller tiles) can be
faster than every kernel the tuner times: the entry then says so, also in a file, and tuning never costs time."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture()
def btas():
    import paper_1701_04733_gb300 as b
    b.build()
    b.lib()
    b.tune_clear()
    yield b
    b.tune_clear()


def line(**kv):
    e = {"arch": 103, "sms": 152, "semiring": 0, "dtype": 0, "m_bucket": 9, "n_bucket": 9, "k_bucket": 9, "variant": 1,
         "ns": 4, "cfg": 4, "group_m": 8, "candidates": 17, "tile_m": 128, "tile_n": 128, "seconds": 0.0302,
         "terms_per_second": 1.82e13}
    e.update(kv)
    return json.dumps(e)


def test_file_keeps_the_mark(btas, tmp_path):
    src, out = tmp_path / "in.jsonl", tmp_path / "out.jsonl"
    src.write_text(line() + "\n" + line(semiring=1, defaults=1) + "\n" + line(k_bucket=10, defaults=0) + "\n")
    assert btas.tune_load(str(src)) == 3
    btas.tune_save(str(out))
    got = {(e["semiring"], e["k_bucket"]): e for e in map(json.loads, out.read_text().splitlines())}
    assert got[(1, 9)]["defaults"] == 1
    assert "defaults" not in got[(0, 9)] and "defaults" not in got[(0, 10)]
    assert btas.tune_load(str(out)) == 3


SCRIPT = """
import sys
sys.path.insert(0, {root!r})
import torch
import paper_1701_04733_gb300 as btas
btas.tune_load({path!r})
A = torch.ones((333, 333), dtype=torch.int32, device="cuda")
C = btas.gemm(A, A, 0)
btas.gemm(A, A, 0, out=C, accumulate=True)
torch.cuda.synchronize()
"""


@pytest.mark.gpu
@pytest.mark.parametrize("marked", [False, True])
def test_marked_entry_leaves_plain_products_untuned(tmp_path, marked):
    import torch
    p = torch.cuda.get_device_properties(0)
    path = tmp_path / "t.jsonl"
    kv = {"defaults": 1} if marked else {}
    path.write_text(line(arch=p.major * 10 + p.minor, sms=p.multi_processor_count, cfg=0, ns=8, **kv) + "\n")
    r = subprocess.run([sys.executable, "-c", SCRIPT.format(root=ROOT, path=str(path))],
                       env=dict(os.environ, BTAS_LOG="1"), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    plain, accumulate = [x for x in r.stderr.splitlines() if "product 333x333x333" in x]
    assert ("(defaults)" if marked else "cfg 0 group 8 splits 1 shares 0 (autotuner)") in plain
    assert "cfg 0 group 8 splits 1 shares 0 (autotuner)" in accumulate


@pytest.mark.gpu
@pytest.mark.parametrize("m,n,k", [(1000, 1531, 777), (2000, 2000, 2000), (8192, 64, 8192)])
def test_tuning_costs_no_time(btas, m, n, k):
    """fp32 products between one and five waves of tiles, and a thin one.  Each side is the fastest of 5 rounds of 20
    calls; the bound is twice the 2 % and the noise that the tuner allows for, and was 10 to 20 % short of these."""
    import torch
    A, B = torch.rand(m, k, device="cuda"), torch.rand(k, n, device="cuda")

    def best():
        times = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                C = btas.gemm(A, B, btas.MINPLUS)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times), C

    best()
    for attempt in range(4):  # a burst of other work on the host can spoil one
        btas.tune_clear()
        untuned, C0 = best()
        btas.tune_gemm(btas.MINPLUS, btas.F32, m, n, k)
        tuned, C1 = best()
        assert torch.equal(C0, C1)
        if tuned < 1.05 * untuned:
            break
    assert tuned < 1.05 * untuned
