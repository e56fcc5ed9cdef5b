"""Pair and four- to six-SNP scans of data whose sets tie (needs an sm_103 GPU): the candidate list
overflowing once and fitting with the threshold it gave, thousands of candidates rescored and merged,
more ties at the k-th score than the list holds -- seen in the sample or only in the list --, with the
list as it is and cut to 1024 entries.  Answers identical to the oracle's, and the figures that tell
which way they came."""
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


def _scan(g, ph, order, k):
    """The stats of a scan whose answer is the oracle's."""
    if order == 2:
        osets, osc, _ = oracle.scan_pairs_topk(g, ph, k)
    else:
        osets, osc, _ = oracle.scan_order_topk(g, ph, order, k)
    with epi.Handle(g, ph) as h:
        for _ in range(2):   # the second call takes the scratch as the first left it
            sets, sc = h.scan_order(order, k)
            assert np.array_equal(sets, osets), (sets[:3], osets[:3])
            assert np.array_equal(sc, osc)
        return h.stats()


def _launches_before(order):   # sample and threshold; and tables, and counts of the smaller sets
    return 2 if order == 2 else order + 2


@pytest.mark.parametrize("order,m,k", [(2, 400, 500), (4, 40, 300), (5, 24, 500), (6, 20, 512)])
def test_second_pass_fits_the_list(monkeypatch, order, m, k):
    # the sample's threshold lets about 1200 to 1700 sets through, the list's own half of them
    monkeypatch.setenv("EPI3_FAULT", "cand")
    g, ph = pins.tiny_data(m, 120, 55, seed=2800 + order)
    st = _scan(g, ph, order, k)
    assert k <= st["n_rescored"] <= st["n_candidates"] <= 1024
    assert st["kernel_launches"] == _launches_before(order) + 2 * 5


@pytest.mark.parametrize("order,m,same,k", [(2, 700, 100, 40), (2, 400, 70, 512), (4, 60, 20, 40), (4, 45, 18, 512),
                                            (5, 16, 16, 40), (6, 15, 15, 512)])
def test_thousands_of_candidates_are_merged(order, m, same, k):
    # copies of an associated SNP: their sets tie below all others
    g, ph = pins.tiny_data(m, 300, 140, seed=2900 + order)
    rng = np.random.default_rng(order)
    g[rng.permutation(m)[:same]] = np.where(rng.random(300) < 0.9, 2 * ph, 1).astype(np.uint8)
    st = _scan(g, ph, order, k)
    assert 2048 < st["n_rescored"] <= st["n_candidates"] <= 1 << 18
    assert st["kernel_launches"] > _launches_before(order) + 5   # one pass, and merges


@pytest.mark.parametrize("order,m,same,n,n1,k", [(2, 200, 200, 300, 140, 20),
                                                 (4, 26, 26, 200, 90, 40), (4, 40, 20, 200, 90, 300),
                                                 (4, 16, 16, 131070, 65535, 30), (4, 18, 18, 33, 33, 7),
                                                 (5, 16, 16, 200, 90, 40), (6, 15, 15, 200, 90, 512)])
def test_more_ties_than_the_list_holds(monkeypatch, order, m, same, n, n1, k):
    # `same` SNPs without any variant: their sets have the least possible number of cells
    monkeypatch.setenv("EPI3_FAULT", "cand")
    g, ph = pins.tiny_data(m, n, n1, seed=3000 + order)
    g[np.random.default_rng(order).permutation(m)[:same]] = 0
    st = _scan(g, ph, order, k)
    assert st["n_candidates"] > 1024
    # one pass or two (its first threshold may lie above the ties), then every set and merges
    assert st["kernel_launches"] <= _launches_before(order) + 2 * 5 + 6
    assert st["n_rescored"] == st["n_triplets"]


def test_ties_that_only_the_list_shows(monkeypatch):
    # 46 copies of a strongly associated SNP: 1035 equal best pairs, of which the sample (every second
    # pair) holds so few that it does not expect the list to overflow; the list's threshold is no
    # lower than the sample's
    monkeypatch.setenv("EPI3_FAULT", "cand")
    m = 400
    g, ph = pins.tiny_data(m, 600, 290, seed=3100)
    rng = np.random.default_rng(1)
    for _ in range(2000):
        at = np.sort(rng.permutation(m)[:46])
        i, j = np.triu_indices(46, 1)
        even = int(np.sum((at[j] * (at[j] - 1) // 2 + at[i]) % 2 == 0))
        if 20 <= even <= 512:
            break
    assert even <= 512
    g[at] = np.where(rng.random(600) < 0.9, 2 * ph, 1).astype(np.uint8)
    st = _scan(g, ph, 2, 20)
    assert st["n_candidates"] == 1035 and st["n_rescored"] == m * (m - 1) // 2
    assert st["kernel_launches"] <= 2 + 5 + 6
