"""quot_rn, the quotient of positive doubles in integers that gives the resident
iterations their alpha, beta and omega: bit for bit the IEEE division, for
mantissas next to powers of two and all ones, at every exponent, at both ends of
the quotient's range (just above and below the smallest normal number and the
largest) and for operands that it leaves to the division itself."""
import ctypes

import numpy as np
import pytest
import torch

import device_probe

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _quotients(a, b):
    lib = device_probe.load()
    ad, bd = (torch.from_numpy(v).to(DEV) for v in (a, b))
    out = torch.empty_like(ad)
    p = [ctypes.c_void_p(t.data_ptr()) for t in (ad, bd, out)]
    assert lib.probe_quotients(*p, ctypes.c_int64(len(a)), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    return out.cpu().numpy()


def _mantissas(rng, n):
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    kind = rng.integers(0, 4, n)
    m[kind == 1] = rng.integers(0, 64, (kind == 1).sum(), dtype=np.uint64)
    m[kind == 2] = np.uint64((1 << 52) - 1) - rng.integers(0, 64, (kind == 2).sum(), dtype=np.uint64)
    m[kind == 3] &= np.uint64(0xFFFFF00000000)
    return m


@pytest.mark.parametrize("difference", [None, -1024, -1023, -1022, -1021, -1020, 0, 1020, 1021, 1022, 1023])
def test_quotient_is_the_division(difference):
    """difference: of the operands' exponents; None: any two."""
    rng = np.random.default_rng(3)
    n = 1 << 20
    ea, eb = rng.integers(0, 2048, n), rng.integers(0, 2048, n)
    if difference is not None:
        eb = rng.integers(max(1, 1 - difference), min(2046, 2046 - difference) + 1, n)
        ea = eb + difference
    a, b = ((_mantissas(rng, n) | e.astype(np.uint64) << np.uint64(52)).view(np.float64) for e in (ea, eb))
    a[0], b[0] = float.fromhex("0x1.000000000007bp-1022"), float.fromhex("0x1.8p+0")
    a[1], b[1] = 1.0, 0.0
    a[2], b[2] = 5e-324, 3.0
    with np.errstate(all="ignore"):
        want = a / b
    got = _quotients(a, b)
    same = (got.view(np.uint64) == want.view(np.uint64)) | (np.isnan(got) & np.isnan(want))
    k = np.flatnonzero(~same)
    assert len(k) == 0, (len(k), a[k[0]].hex(), b[k[0]].hex(), got[k[0]].hex(), want[k[0]].hex())
