"""The tuner's file across versions of the kernels (needs an sm_103 GPU): lines written before the scan
forms changed say nothing about them, so their bucket is measured again; a line of this version
is taken."""
import os
import subprocess
import sys

import pytest

import paper_2201_10956_gb300 as epi

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = """
import sys
sys.path[:0] = [{root!r}, {tests!r}]
import oracle_pins as pins
import paper_2201_10956_gb300 as epi
g, ph = pins.tiny_data(130, 1100, 500, seed=61)
with epi.Handle(g, ph) as h:
    h.scan(4)
    print(h.stats()["path"])
"""


def _scan(cache):
    code = CHILD.format(root=ROOT, tests=os.path.join(ROOT, "tests"))
    r = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, EPI3_TUNE_CACHE=str(cache)),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    return int(r.stdout.split()[-1])


def test_lines_of_other_kernels_are_measured_again(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_10956_gb300 import build as B
    B.build()
    props = torch.cuda.get_device_properties(0)
    cache = tmp_path / "tune.tsv"
    sms = props.multi_processor_count
    old = f"{props.name}\t{sms}\t2\t1\t{epi.PATH_POPC8}\t0\t1\n" \
          f"{props.name}\t{sms}\t2\t1\t{epi.PATH_POPC8}\n"
    cache.write_text(old)
    path = _scan(cache)
    text = cache.read_text()
    assert text.startswith(old)
    new = text[len(old):].splitlines()
    assert len(new) == 1 and int(new[0].split("\t")[4]) == path
    # the new line is found again: nothing is appended
    assert _scan(cache) == path and cache.read_text() == text
