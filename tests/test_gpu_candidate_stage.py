"""The candidate stage and its sampled threshold at their limits (needs an sm_103 GPU): thousands of
triplets tied at the k-th score, long answers of many samples, and answers around the length up to
which a shortened sample gives a threshold -- identical to the oracle's scan."""
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


def _check(g, ph, ks, path="auto"):
    otr, osc, _ = oracle.scan_topk(g, ph, max(ks))
    with epi.Handle(g, ph) as h:
        h.set_option("path", path)
        for k in ks:
            tr, sc = h.scan(k)
            assert np.array_equal(tr, otr[:k]) and np.array_equal(sc, osc[:k]), k


@pytest.mark.parametrize("m,n,n1", [(24, 1000, 400), (36, 1000, 999), (36, 40000, 20000), (36, 131072, 50000)])
def test_every_triplet_tied(m, n, n1):
    g = np.zeros((m, n), dtype=np.uint8)
    ph = np.zeros(n, dtype=np.uint8)
    ph[np.random.default_rng(n).permutation(n)[:n1]] = 1
    _check(g, ph, [1, 10, 512])


# 131 072 samples: the sample is cut to 512 triplets, which serve answers of up to 128 rows
@pytest.mark.parametrize("m,n,n1", [(40, 131072, 60000), (64, 131072, 60000), (50, 70000, 3000)])
@pytest.mark.parametrize("path", ["mma4c", "mma4", "popc8"])
def test_answers_around_the_shortened_sample(m, n, n1, path):
    g, ph = pins.tiny_data(m, n, n1, seed=2600 + m)
    _check(g, ph, [1, 127, 128, 129, 255, 256, 257, 512], path)
