"""Which way the value update of a sliced handle goes: one pass over the buffer, or
a permutation and a gather where too many of the slices hold more than 256 entries
(without S A S an eighth, of at most 384; with it a quarter). Bit for bit the same
values either way (the checks of test_gpu_passes): a few long slices among short
ones, at the lines and one more, and long ones only."""
import types

import numpy as np
import pytest

import test_gpu_passes as passes
from paper_2510_08536_gb300 import build, repart

pytestmark = pytest.mark.gpu


def _chain(slices, long_slices, reach=10):
    """A chain of cells; in the first `long_slices` slices every cell meets `reach` on either side."""
    n = 32 * slices - 5
    lo, up = [np.arange(n - 1)], [np.arange(1, n)]
    for d in range(2, reach + 1):
        i = np.arange(max(0, min(n, 32 * long_slices) - d))
        lo.append(i)
        up.append(i + d)
    lo, up = np.concatenate(lo), np.concatenate(up)
    o = np.lexsort((up, lo))
    z = np.zeros(0, np.int32)
    return [types.SimpleNamespace(n_cells=n, n_faces=len(lo), n_iface=0, lower_addr=lo[o].astype(np.int32),
                                  upper_addr=up[o].astype(np.int32), iface_row=z, iface_nbr_rank=z, iface_nbr_col=z)]


@pytest.mark.parametrize("kind", ["plain", "special"])
@pytest.mark.parametrize("slices,long_slices,reach", [
    (64, 1, 10), (64, 16, 10), (64, 17, 10), (64, 64, 10), (5000, 300, 10), (64, 8, 5), (64, 9, 5), (64, 17, 5)])
@pytest.mark.parametrize("fp32", [False, True])
def test_update_routes(slices, long_slices, reach, fp32, kind, monkeypatch):
    build.build()
    repart.load()
    monkeypatch.setitem(passes.SHAPES, "chain", (lambda: _chain(slices, long_slices, reach), {"want_fp32": fp32}))
    passes.test_update_bit_exact("chain", kind)
