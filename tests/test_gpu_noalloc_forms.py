"""epi3_scan_noalloc on both sides of its switch (needs an sm_103 GPU): 8 cells counted where the pair
tables fit the static scratch beside the rest, all 27 beyond -- the oracle's answer either way, and on
calls of the two forms in turn, which share the scratch."""
import numpy as np
import pytest

import oracle
import oracle_pins as pins
from paper_2201_10956_gb300 import build as B
import paper_2201_10956_gb300 as epi
from paper_2201_10956_gb300 import epi3

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()
    return epi.load()


def _check(g, ph, k):
    import torch
    tr, sc = epi3.scan_noalloc(torch.from_numpy(g).cuda(), torch.from_numpy(ph).cuda(), k)
    otr, osc, _ = oracle.scan_topk(g, ph, k)
    assert np.array_equal(tr.cpu().numpy(), otr) and np.array_equal(sc.cpu().numpy(), osc)


# 32 bytes a pair in the 8 MiB: with 90 samples the pair tables fit up to 669 SNPs
@pytest.mark.parametrize("m,n,n1,k", [(640, 90, 41, 20), (669, 90, 41, 20), (670, 90, 41, 20), (720, 90, 60, 20),
                                      (1000, 70, 1, 5), (40, 40000, 17000, 512)])
def test_both_forms_match_the_oracle(m, n, n1, k):
    g, ph = pins.tiny_data(m, n, n1, seed=2400 + m)
    _check(g, ph, k)


def test_forms_in_turn():
    for m, n, n1, k in [(700, 80, 30, 12), (50, 900, 400, 300), (690, 64, 64, 7), (30, 128, 0, 9)]:
        g, ph = pins.tiny_data(m, n, n1, seed=2500 + m)
        _check(g, ph, k)


@pytest.mark.parametrize("m", [3, 4, 9, 10, 11, 12])
@pytest.mark.parametrize("n,n1", [(60, 25), (65536, 30001)])
def test_few_snps(m, n, n1):
    g, ph = pins.tiny_data(m, n, n1, seed=2450 + m)
    _check(g, ph, min(7, m * (m - 1) * (m - 2) // 6))
