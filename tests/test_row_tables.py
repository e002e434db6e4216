"""The piecewise polynomials of the row tables (csrc/pt_device.cuh), restated
in 64 bits over the oracle's flux: for radius ratios over the tables' range
and three limb-darkening laws they stay within 2e-9 of the occulted flux
between the nodes, two orders below the FP32 path's 1e-6."""
import os
import re

import numpy as np
import pytest

import oracle

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = open(os.path.join(HERE, "..", "paper_1504_07433_gb300", "csrc", "pt_device.cuh")).read()
NA, NL = (int(x) for x in re.search(r"MT_NA = (\d+), MT_NL = (\d+)", SRC).groups())
Q = int(re.search(r"MT_Q = (\d+)", SRC).group(1))
PMIN, PMAX = (float(x) for x in re.search(r"MT_PMIN = ([0-9.e+-]+)f, MT_PMAX = ([0-9.e+-]+)f", SRC).groups())


def _depth(p, z, u1, u2):
    z = np.minimum(np.maximum(z, 0.0), (1.0 + p) * (1.0 - 1e-16))
    n = z.size
    return 1.0 - oracle.flux_quad_vec(np.full(n, p), z.ravel(), np.full(n, u1), np.full(n, u2)).reshape(z.shape)


@pytest.mark.parametrize("p", [PMIN, 1e-3, 0.01, 0.05, 0.1, 0.2, 0.35, PMAX])
def test_row_polynomials_within_2e9(p):
    x = np.cos((np.arange(Q) + 0.5) * np.pi / Q)
    V = np.linalg.inv(np.polynomial.chebyshev.chebvander(x, Q - 1))
    xt = np.linspace(-1.0, 1.0, 33)
    T = np.polynomial.chebyshev.chebvander(xt, Q - 1)
    for u1, u2 in ((0.0, 0.0), (0.9, 0.0), (0.4, 0.3)):
        for reg, n, length in (("A", NA, np.sqrt(1 - p)), ("B", NL, np.sqrt(p)), ("C", NL, np.sqrt(p))):
            s = (n - 0.5) * (1.0 - 2e-6) / length
            mid = np.where(np.arange(n) == 0, 0.25, np.arange(n))[:, None]
            half = np.where(np.arange(n) == 0, 0.25, 0.5)[:, None]
            w2 = ((mid + half * x) / s) ** 2
            wt2 = ((mid + half * xt) / s) ** 2
            wt2[-1, -1] = length ** 2   # the last interval ends 2e-6 beyond the region, where no look-up falls
            z = {"A": lambda q: (1 - p) - q, "B": lambda q: (1 - p) + q, "C": lambda q: (1 + p) - q}[reg]
            poly = _depth(p, z(w2), u1, u2) @ V.T @ T.T
            poly[-1, -1] = (_depth(p, z(w2), u1, u2)[-1] @ V.T
                            @ np.polynomial.chebyshev.chebvander((length * s - (n - 1)) / 0.5, Q - 1).ravel())
            err = np.abs(poly - _depth(p, z(wt2), u1, u2))
            assert err.max() <= 2e-9, (reg, u1, u2, err.max())
