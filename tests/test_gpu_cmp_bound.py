"""The compacted scan's runs, its table-free bound and its survivor queue (needs an sm_103 GPU):
sizes around the 64 x 32 tile edges and the 8-SNP blocks of its pair tables, class shares from
balanced to one-sided (the bound's parabola depends on them), null data whose k-th best lies in the
bulk of the scores (many survivors), several compaction ranges -- both epilogue forms, top-k
identical to the oracle's."""
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


def _check(g, ph, k, **options):
    otr, osc, _ = oracle.scan_topk(g, ph, k)
    with epi.Handle(g, ph) as h:
        h.set_option("path", "mma4c")
        for key, value in options.items():
            h.set_option(key, value)
        for form in ("plain", "split"):
            h.set_option("mma_form", form)
            tr, sc = h.scan(k)
            assert np.array_equal(tr, otr) and np.array_equal(sc, osc), form


@pytest.mark.parametrize("m", [8, 9, 31, 33, 63, 64, 65, 66, 95, 97, 127, 129, 193])
def test_tile_edges(m):
    g, ph = pins.tiny_data(m, 700, 300, seed=1300 + m)
    _check(g, ph, min(20, m * (m - 1) * (m - 2) // 6))


@pytest.mark.parametrize("n,n1", [(3000, 1500), (3000, 300), (3000, 2900), (3000, 1), (3000, 3000),
                                  (12000, 7000)])
def test_bound_on_null_data_at_every_class_share(n, n1):
    d = gen.make_dataset(90, n, n1, (0.05, 0.5), 0, seed=1400 + n1)
    _check(d.genotypes, d.phenotype, 300)


@pytest.mark.parametrize("mb", [1, 3])
def test_several_ranges(mb):
    g, ph = pins.tiny_data(300, 2100, 900, seed=1500 + mb)
    _check(g, ph, 40, cmp_buffer_mb=mb)
