"""The pairwise scan's thresholded form (needs an sm_103 GPU): the bound and the sampled threshold at
every class share, more pairs than the sample, long answers, and thousands of equal pairs (the
direct form answers then) -- identical to the oracle's exhaustive pair scan."""
import numpy as np
import pytest

import gen
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


def _check(g, ph, k):
    opr, osc, _ = oracle.scan_pairs_topk(g, ph, k)
    with epi.Handle(g, ph) as h:
        for _ in range(2):
            pr, sc = h.scan_pairs(k)
            assert np.array_equal(pr, opr) and np.array_equal(sc, osc)


@pytest.mark.parametrize("m,n,n1,k", [(3, 2, 1, 3), (256, 900, 450, 1), (257, 900, 30, 512), (513, 700, 690, 64),
                                      (300, 20000, 1, 20), (700, 1500, 0, 512), (150, 100000, 65000, 30)])
def test_filter_on_null_data(m, n, n1, k):
    d = gen.make_dataset(m, n, n1, (0.02, 0.5), 0, seed=1900 + m)
    _check(d.genotypes, d.phenotype, k)


@pytest.mark.parametrize("m,k", [(200, 512), (400, 3)])
def test_thousands_of_equal_pairs(m, k):
    g, ph = pins.tiny_data(m, 300, 140, seed=2000 + m)
    g[:] = g[np.arange(m) % 2]
    _check(g, ph, k)
