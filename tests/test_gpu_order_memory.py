"""Device memory of the four- to six-SNP scans (needs an sm_103 GPU): large tables of the smaller sets
are given back when the call returns, and are not made at all where they would take more than their
share of the memory that is free; the answer is the same."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
import oracle_pins as pins
from paper_2201_10956_gb300 import build as B
import paper_2201_10956_gb300 as epi

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# C(60, 5) tables of 32 four-byte counts: 700 MB
CHILD = """
import os, sys
sys.path[:0] = [{root!r}, {tests!r}]
import numpy as np, torch
import oracle_pins as pins
import paper_2201_10956_gb300 as epi
small, ph_s = pins.tiny_data(12, 60, 25, seed=71)
g, ph = pins.tiny_data(60, 60, 25, seed=72)
free = lambda: torch.cuda.mem_get_info()[0]
with epi.Handle(small, ph_s) as h, epi.Handle(g, ph) as big:
    h.scan_order(6, 5)
    before = free()
    sets, sc = big.scan_order(6, 5)
    print("kept", before - free())
    os.environ["EPI3_FAULT"] = "tables"
    sets_d, sc_d = big.scan_order(6, 5)
    assert np.array_equal(sets, sets_d) and np.array_equal(sc, sc_d)
"""


@pytest.fixture(scope="module", autouse=True)
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()
    return epi.load()


def test_large_tables_are_given_back():
    code = CHILD.format(root=ROOT, tests=os.path.join(ROOT, "tests"))
    r = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, EPI3_CACHE_MB="0"),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    assert int(r.stdout.split()[-1]) <= 300 << 20, r.stdout


@pytest.mark.parametrize("order,m", [(4, 30), (5, 15), (6, 12)])
def test_no_tables_where_memory_is_short(order, m, monkeypatch):
    monkeypatch.setenv("EPI3_FAULT", "lowmem")
    g, ph = pins.tiny_data(m, 150, 70, seed=2700 + order)
    osets, osc, _ = oracle.scan_order_topk(g, ph, order, 12)
    with epi.Handle(g, ph) as h:
        sets, sc = h.scan_order(order, 12)
        assert np.array_equal(sets, osets) and np.array_equal(sc, osc)
