"""grid_sum_unit, the grid sum of the resident iterations, by itself against exact
sums: no unit yet, units from totals near, above and below, both signs and
cancelling values, single values and totals out of the unit's range, infinities, NaN
and zeros, and blocks that give up.

Bounds. In a known unit: 155,648 threads round to half of 2^-79 of the last total at
most and 152 blocks to half of 2^-65, together below 2^-58 of it, then the total to
2^-53 of itself. The long way: three levels of sums rounded to 2^-53 each, and the
warps' own units 2^-57 of their largest value: below 2^-51 of the sum of magnitudes."""
import ctypes
import math

import numpy as np
import pytest
import torch

import device_probe

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _sums(v, last, blocks, threads, spin=1 << 24):
    lib = device_probe.load()
    vd, ld = torch.from_numpy(v).to(DEV), torch.from_numpy(np.asarray(last, np.float64)).to(DEV)
    out = torch.full((blocks, 2, 2), 7.0, dtype=torch.float64, device=DEV)
    bad = torch.full((blocks,), -1, dtype=torch.int32, device=DEV)
    torch.cuda.synchronize()
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    assert lib.probe_grid_sums(p(vd), p(ld), blocks, threads, ctypes.c_int64(spin), p(out), p(bad),
                               ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    return out.cpu().numpy(), bad.cpu().numpy()


def _shapes():
    return [(1, 32), (1, 1024), (7, 96), (None, 1024), (None, 768)]  # None: a block an SM


@pytest.mark.parametrize("kind", ["first", "near", "negative", "signs", "grown", "shrunk", "outlier", "wide", "zeros"])
@pytest.mark.parametrize("blocks,threads", _shapes())
def test_sums(blocks, threads, kind):
    blocks = blocks or torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(len(kind) + threads)
    n = blocks * threads
    v = rng.random((2, n))
    if kind == "negative":
        v = -v
    if kind == "signs":
        v = 2.0 * v - 1.0
    if kind == "wide":
        v = (2.0 * v - 1.0) * np.exp2(rng.integers(-300, 300, (2, n)))
    if kind == "zeros":
        v[:] = 0.0
    exact = np.array([math.fsum(r) for r in v])
    last, quick = exact * 1.3, kind in ("near", "negative", "signs", "grown")
    if kind == "first":
        last = np.zeros(2)
    if kind == "grown":  # 2^12 of the last total: in range still
        last = exact * 2.0 ** -12
    if kind == "shrunk":  # 2^-10 of it: taken again
        last = exact * 2.0 ** 10
    if kind == "outlier":  # one value of 2^10 of the last total
        last = np.full(2, 0.01)
        v[:, n // 2] = 10.24
        exact = np.array([math.fsum(r) for r in v])
    if kind == "wide":
        last = np.max(np.abs(v), axis=1) * 2.0 ** 40  # the total is far below
    out, bad = _sums(v, last, blocks, threads)
    assert (bad == 0).all()
    assert (out == out[:1]).all()  # all blocks hold the same totals
    first, second = out[0]
    long_way = 2.0 ** -51 * np.abs(v).sum(1)
    known = lambda unit_of: 2.0 ** -53 * np.abs(exact) + 2.0 ** -58 * np.abs(unit_of)  # noqa: E731
    assert (np.abs(first - exact) <= (known(last) if quick else long_way)).all()
    # the second sum of the same values in the unit of the first total: in range unless they cancel by 2^9
    in_range = np.abs(v).max() < 2.0 ** 9 * np.abs(exact).min()
    assert (np.abs(second - exact) <= (known(first) if in_range else long_way)).all()


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_special_values(value):
    v = np.random.default_rng(1).random((2, 4 * 128))
    v[1, 200] = value
    for last in ([0.0, 0.0], v[:, :200].sum(1) * 2.5):
        out, bad = _sums(v, last, 4, 128)
        assert (bad == 0).all() and (out == out[:1])[:, :, 0].all()
        assert np.allclose(out[0, :, 0], math.fsum(v[0]), rtol=2.0 ** -51, atol=0.0)
        same = np.isnan(out[..., 1]) if np.isnan(value) else out[..., 1] == value
        assert same.all()


@pytest.mark.parametrize("last", [0.0, 100.0])
def test_meeting_runs_out(last):
    _, bad = _sums(np.ones((2, 8 * 64)), [last, last], 8, 64, spin=0)
    assert (bad == 1).all()
