"""The grid sums behind every dot product (integer fixed-point sums across a
warp, a block and the grid) on values a solver never meets together: wide
exponents, exact cancellation, zeros, subnormals, infinities and NaN.

x.y of rp_spmv on a diagonal system: y_i = d_i x_i, and the terms x_i y_i are
exact (powers of two times short integers), so the exact sum is known. Bound:
each term enters a sum of 32 lanes rounded to at most 2^-57 of the largest one
and every level rounds once, and a thread adds its own rows in FP64: with at
most r rows a thread, r + 8 roundings of 2^-53 of the sum of magnitudes.
"""
import dataclasses
import math

import numpy as np
import pytest
import torch

from paper_2510_08536_gb300 import build, repart

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@dataclasses.dataclass
class _Diagonal:
    n_cells: int
    lower_addr = upper_addr = iface_row = iface_nbr_rank = iface_nbr_col = np.zeros(0, np.int32)


def _terms(kind, n):
    rng = np.random.default_rng(n)
    x = np.ones(n)
    d = rng.integers(1, 1 << 20, n).astype(np.float64)
    if kind == "signed":
        d *= rng.choice([-1.0, 1.0], n)
    elif kind == "wide":
        d *= np.ldexp(1.0, rng.integers(-300, 300, n)) * rng.choice([-1.0, 1.0], n)
    elif kind == "cancel":
        h = n // 2
        d[h:2 * h] = -d[:h]
        d[2 * h:] = 0.0
    elif kind == "zero":
        d[:] = 0.0
    elif kind == "subnormal":
        d *= 5e-324
    return d, x


@pytest.mark.parametrize("kind", ["plain", "signed", "wide", "cancel", "zero", "subnormal"])
@pytest.mark.parametrize("n", [1, 31, 33, 257, 100003, 700001])
def test_dot_against_exact_sum(kind, n):
    build.build()
    d, x = _terms(kind, n)
    h = repart.build_repartition([_Diagonal(n)])
    repart.update_values_packed(h, torch.from_numpy(d).to(DEV))
    y = torch.zeros(n, dtype=torch.float64, device=DEV)
    xy = torch.full((1,), 7.0, dtype=torch.float64, device=DEV)
    xd = torch.from_numpy(x).to(DEV)
    repart.spmv(h, xd, y, xy)
    assert torch.equal(y.cpu(), torch.from_numpy(d * x))
    rows = -(-n // (152 * 8 * 256)) + 1
    bound = (rows + 8) * 2.0 ** -53 * math.fsum(np.abs(d * x))
    assert abs(float(xy[0]) - math.fsum(d * x)) <= bound
    again = torch.zeros_like(xy)
    repart.spmv(h, xd, y, again)
    assert torch.equal(xy, again)
    for bad, want in ((np.inf, math.inf), (-np.inf, -math.inf), (np.nan, math.nan)):
        d2 = d.copy()
        d2[n // 3] = bad
        repart.update_values_packed(h, torch.from_numpy(d2).to(DEV))
        repart.spmv(h, xd, y, xy)
        assert float(xy[0]) == want or (math.isnan(want) and math.isnan(float(xy[0])))
    h.close()
