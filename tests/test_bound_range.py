"""The table-free bounds over everything a data set can have (no GPU): the cell inequality on the two
curves it reduces to (one class's count + 1 equal to 1, the other's any real number) for every class
share down to 27 / 131126 and counts up to 131073, the reduction itself, and the library's own
constants (cmp_bound_terms, compiled for the host) against exact K2 values."""
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
P_LEAST = 27.0 / (131072 + 54)      # an all-control cohort of the most samples a handle takes
U_MOST = 131073.0                   # count + 1
HALF_LN_2PI = 0.9189385332046727


def _rest(us, p, p0):
    """The right side of the inequality (without the cell's own term)."""
    c = np.maximum(-np.log1p(-p0) / p0 ** 2, -np.log(p0) / (1 - p0) ** 2)
    h0, h1 = -p0 * np.log(p0) - (1 - p0) * np.log1p(-p0), np.log((1 - p0) / p0)
    eps = np.maximum(0.125, 0.2346 - p0 / 4)
    return us * (h0 + h1 * (p - p0) - c * (p - p0) ** 2) + 0.5 * np.log(us) \
        + 0.5 * np.log(p0 * (1 - p0)) - HALF_LN_2PI - eps


@pytest.mark.parametrize("small_is_minor", [True, False])
def test_cell_term_on_the_curves(small_is_minor):
    # grid steps of 3e-3 in ln p0 and ln us: D's second derivatives in these are of order 1 where it
    # is small, so that between grid points it is lower by 1e-5 at most; the margin asked is 5e-5
    shares = np.exp(np.linspace(math.log(P_LEAST), math.log(0.5), 2600))
    us = 2.0 + np.concatenate([[0.0], np.exp(np.linspace(math.log(1e-4), math.log(U_MOST), 7000))])
    p = 1.0 / us if small_is_minor else 1.0 - 1.0 / us
    for part in np.array_split(shares, 13):
        d = np.log(us - 1.0)[None, :] - _rest(us[None, :], p[None, :], part[:, None])
        assert d.min() > 5e-5, (d.min(), part[np.unravel_index(d.argmin(), d.shape)[0]])


def test_larger_counts_have_more_to_spare():
    rng = np.random.default_rng(5)
    for _ in range(3000):
        a = math.exp(rng.uniform(0.0, math.log(U_MOST)))
        counts = (1.0, a) if rng.random() < 0.5 else (a, 1.0)
        p0 = math.exp(rng.uniform(math.log(P_LEAST), math.log(0.5)))
        last = None
        for s in (1.0, 1.3, 2.0, 7.0, 100.0):
            u0, u1 = s * counts[0], s * counts[1]
            d = math.lgamma(u0 + u1) - math.lgamma(u0) - math.lgamma(u1) \
                - float(_rest(u0 + u1, u1 / (u0 + u1), p0))
            assert last is None or d >= last - 1e-12 * abs(last) - 3e-16 * (u0 + u1) * 30, (counts, p0, s)
            last = d


def test_library_constants_stay_below_k2(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / "bound_check"
    subprocess.check_call([nvcc, "-std=c++17", "-o", str(exe), os.path.join(HERE, "host", "bound_check.cu")])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and "bound ok" in out.stdout, out.stdout + out.stderr
