"""What a batch says of itself (needs an sm_103 GPU): the form, the block and the launches of its scan,
for cohorts of one form and of several."""
import numpy as np
import pytest

import oracle_pins as pins
from paper_2201_10956_gb300 import build as B
import paper_2201_10956_gb300 as epi

pytestmark = pytest.mark.gpu

SHAPES = [(60, 400), (70, 900), (90, 300)]


@pytest.fixture(scope="module", autouse=True)
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()
    return epi.load()


def _stats(data):
    with epi.Batch(data) as b:
        b.scan(3)
        return b.stats(), b.paths()


@pytest.mark.parametrize("force,path,per_cohort,shared", [
    ("mma", epi.PATH_MMA4, 2, 1),         # seed and candidate stage; one launch for all tiles
    ("mma4c", epi.PATH_MMA4C, 5, 0),      # and sample lists, chunks and scan of the one range
    ("popc8", epi.PATH_POPC8, 3, 0)])     # and a scan
def test_cohorts_of_one_form(monkeypatch, force, path, per_cohort, shared):
    monkeypatch.setenv("EPI3_BATCH_PATH", force)
    data = [pins.tiny_data(m, n, n // 3, seed=2200 + m) for m, n in SHAPES]
    st, paths = _stats(data)
    assert np.all(paths == path) and st["path"] == path
    assert st["kernel_launches"] == per_cohort * len(data) + shared
    if force != "mma":
        with epi.Handle(*data[0]) as h:     # the block of the form's own kernel
            h.set_option("path", force)
            h.scan(3)
            assert st["block"] == h.stats()["block"]


def test_cohorts_of_several_forms():
    # the smallest share the one-hot launch, the larger ones are compacted
    data = [pins.tiny_data(m, 600, 250, seed=2300 + m) for m in (40, 260, 50, 300)]
    st, paths = _stats(data)
    assert paths.tolist() == [epi.PATH_MMA4, epi.PATH_MMA4C] * 2
    assert st["path"] == epi.PATH_AUTO
    assert st["kernel_launches"] == 2 * 2 + 1 + 2 * 5
