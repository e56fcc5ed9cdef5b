"""Outputs of a handle made with device pointers (needs an sm_103 GPU): wherever a copy can put
them -- arrays that are not aligned to their type, pinned host memory -- the scan does too, in every
scan form, and leaves the bytes around them alone."""
import ctypes

import numpy as np
import pytest

import oracle
import oracle_pins as pins
from paper_2201_10956_gb300 import build as B
import paper_2201_10956_gb300 as epi

pytestmark = pytest.mark.gpu

K = 9


@pytest.fixture(scope="module", autouse=True)
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()
    return epi.load()


@pytest.mark.parametrize("path", ["mma4c", "mma4", "popc8", "popc"])
@pytest.mark.parametrize("off_scores,off_trip", [(0, 0), (4, 0), (8, 2), (1, 3), (5, 4)])
def test_any_alignment(lib, path, off_scores, off_trip):
    import torch
    g, ph = pins.tiny_data(40, 500, 210, seed=2100)
    otr, osc, _ = oracle.scan_topk(g, ph, K)
    with epi.Handle(torch.from_numpy(g).cuda(), torch.from_numpy(ph).cuda()) as h:
        h.set_option("path", path)
        sc = torch.full((8 * K + 32,), 0xA5, dtype=torch.uint8, device="cuda")
        tr = torch.full((12 * K + 32,), 0xA5, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        rc = lib.epi3_scan(h._h, K, ctypes.c_void_p(tr.data_ptr() + off_trip),
                           ctypes.c_void_p(sc.data_ptr() + off_scores))
        assert rc == epi.OK, epi.last_error()
        s, t = sc.cpu().numpy(), tr.cpu().numpy()
    assert np.array_equal(s[off_scores:off_scores + 8 * K].copy().view(np.float64), osc)
    assert np.array_equal(t[off_trip:off_trip + 12 * K].copy().view(np.int32).reshape(K, 3), otr)
    assert np.all(s[:off_scores] == 0xA5) and np.all(s[off_scores + 8 * K:] == 0xA5)
    assert np.all(t[:off_trip] == 0xA5) and np.all(t[off_trip + 12 * K:] == 0xA5)


def test_pinned_host_outputs(lib):
    import torch
    g, ph = pins.tiny_data(40, 500, 210, seed=2100)
    otr, osc, _ = oracle.scan_topk(g, ph, K)
    with epi.Handle(torch.from_numpy(g).cuda(), torch.from_numpy(ph).cuda()) as h:
        sc = torch.zeros((K,), dtype=torch.float64, pin_memory=True)
        tr = torch.zeros((K, 3), dtype=torch.int32, pin_memory=True)
        rc = lib.epi3_scan(h._h, K, ctypes.c_void_p(tr.data_ptr()), ctypes.c_void_p(sc.data_ptr()))
        assert rc == epi.OK, epi.last_error()
    assert np.array_equal(sc.numpy(), osc) and np.array_equal(tr.numpy(), otr)
