"""The counted form of the four- to six-SNP scans (needs an sm_103 GPU): cells with genotype 2 from
the counts of smaller sets, FP32 scores and FP64 rescoring of the candidates -- against the oracle's
generic-order scan at the smallest set counts, ragged and one-sided classes, more samples than the
shared log-factorial table holds, sizes where the threshold comes from a sample, and data whose sets
tie by the thousand (the direct form answers then)."""
import numpy as np
import pytest

import oracle
import oracle_pins as pins
from paper_2201_10956_gb300 import build as B
import paper_2201_10956_gb300 as epi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()
    return epi.load()


def _check(g, ph, order, k):
    osets, osc, _ = oracle.scan_order_topk(g, ph, order, k)
    with epi.Handle(g, ph) as h:
        for _ in range(2):   # the second call takes the scratch as the first left it
            sets, sc = h.scan_order(order, k)
            assert np.array_equal(sets, osets), (sets[:3], osets[:3])
            assert np.array_equal(sc, osc)


@pytest.mark.parametrize("order,m,n,n1,k", [
    (4, 4, 1, 0, 1), (4, 5, 31, 16, 5), (4, 9, 128, 64, 126), (4, 33, 385, 1, 64), (4, 52, 260, 130, 20),
    (4, 12, 13000, 6000, 30), (5, 5, 129, 60, 1), (5, 6, 33, 33, 6), (5, 13, 500, 250, 200),
    (5, 23, 129, 40, 33), (5, 8, 20000, 9000, 12), (6, 6, 7, 3, 1), (6, 7, 256, 128, 7),
    (6, 12, 300, 100, 300), (6, 18, 130, 65, 9), (6, 8, 13500, 6500, 11)])
def test_counted_form_matches_oracle(order, m, n, n1, k):
    g, ph = pins.tiny_data(m, n, n1, seed=1700 + 10 * order + m)
    _check(g, ph, order, k)


@pytest.mark.parametrize("order,m", [(4, 26), (5, 14), (6, 13)])
def test_thousands_of_equal_sets(order, m):
    # copies of three SNPs: every set's score is one of a few values
    g, ph = pins.tiny_data(m, 200, 90, seed=1800 + order)
    g[:] = g[np.arange(m) % 3]
    _check(g, ph, order, 40)


@pytest.mark.parametrize("order,m", [(4, 15), (5, 11), (6, 9)])
def test_direct_form_without_memory_for_the_tables(order, m, monkeypatch):
    # the failed allocation is not reported by the launches that follow it
    monkeypatch.setenv("EPI3_FAULT", "tables")
    g, ph = pins.tiny_data(m, 150, 70, seed=1900 + order)
    _check(g, ph, order, 12)
