"""The four- to six-SNP scans of a few sets (needs an sm_103 GPU): the direct form's two launches up to
256 sets of four SNPs and eight of five or six, the counted form beyond; the oracle's answer on both
sides of the line."""
import math

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


@pytest.mark.parametrize("order,m,direct", [(4, 4, True), (4, 10, True), (4, 11, False), (5, 5, True), (5, 6, True),
                                            (5, 7, False), (6, 6, True), (6, 7, True), (6, 8, False)])
@pytest.mark.parametrize("n,n1", [(130, 60), (5000, 1)])
def test_form_by_the_number_of_sets(order, m, direct, n, n1):
    g, ph = pins.tiny_data(m, n, n1, seed=3200 + 10 * order + m)
    k = min(6, math.comb(m, order))
    osets, osc, _ = oracle.scan_order_topk(g, ph, order, k)
    with epi.Handle(g, ph) as h:
        sets, sc = h.scan_order(order, k)
        assert np.array_equal(sets, osets) and np.array_equal(sc, osc)
        assert (h.stats()["kernel_launches"] == 2) == direct
