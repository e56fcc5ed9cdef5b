"""The cell inequality behind the compacted scan's table-free bound (no GPU): a cell's K2 term against
its parabola and half log, for class shares from 1/2 to 3e-4, every pair of cell counts up to 240 and
log-spaced ones up to 1e5."""
import math

import numpy as np
import pytest


def _lgamma(n):
    return np.array([math.lgamma(x) for x in n.ravel()]).reshape(n.shape)


@pytest.mark.parametrize("p0", [0.5, 0.497, 0.48, 0.46, 0.44, 0.42, 0.4, 0.37, 0.33, 0.3, 0.25, 0.2, 0.15, 0.1,
                                0.06, 0.03, 0.01, 0.003, 3e-4])
def test_cell_term_is_above_its_bound(p0):
    c = max(-math.log1p(-p0) / p0 ** 2, -math.log(p0) / (1 - p0) ** 2)
    h0, h1 = -p0 * math.log(p0) - (1 - p0) * math.log1p(-p0), math.log((1 - p0) / p0)
    eps = max(0.125, 0.2346 - p0 / 4)
    u = np.unique(np.concatenate([np.arange(1, 241), np.round(np.logspace(math.log10(240), 5, 80))])).astype(float)
    lg = _lgamma(u)
    u0, u1 = u[:, None], u[None, :]
    us = u0 + u1
    p = u1 / us
    k = _lgamma(us) - lg[:, None] - lg[None, :]
    bound = us * (h0 + h1 * (p - p0) - c * (p - p0) ** 2) + 0.5 * np.log(us) \
        + 0.5 * math.log(p0 * (1 - p0)) - 0.9189385332046727 - eps
    assert np.all(k >= bound - 1e-9 * us), float(np.max(bound - k))
