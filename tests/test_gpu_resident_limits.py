"""Where the resident iterations stop short of the chip's shared memory: layouts
whose streamed products lose there. Sliced FP32 systems past L2 and CSR systems
whose rows find too little L1 take the streaming kernels; smaller ones, and the
uniform layout of the same size, stay resident. (Which form runs; the forms
themselves are tested for their results elsewhere.)"""
import numpy as np
import pytest
import torch

from paper_2510_08536_gb300 import build, repart, synth
from test_gpu_update_routes import _chain

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _staging(ranks):
    """diagonal = number of neighbours + 1, every coefficient -1"""
    out = []
    for r in ranks:
        d = np.ones(r.n_cells)
        for a in (r.lower_addr, r.upper_addr, r.iface_row):
            np.add.at(d, a, 1.0)
        out += [d, np.full(2 * len(r.lower_addr) + len(r.iface_row), -1.0)]
    return torch.from_numpy(np.concatenate(out)).to(DEV)


def _forms(ranks, **kw):
    h = repart.build_repartition(ranks, **kw)
    repart.update_values_packed(h, _staging(ranks))
    b = torch.ones(h.n, dtype=torch.float64, device=DEV)
    out = {}
    for name, f, precisions in (("pcg", repart.solve, ("fp64", "mixed_ru")), ("bicgstab", repart.solve_bicgstab, ("fp64", "mixed"))):
        for p in precisions:
            assert f(h, b, torch.zeros_like(b), tol=1e-3, precision=p)["status"] == 0
            out[name, p] = repart.solve_form(h) != "streaming"
    h.close()
    return out


CSR = {"layout": repart.RP_LAYOUT_CSR}


@pytest.mark.parametrize("name,ranks,kw,resident", [
    # rows of 21 entries, FP32 bytes with indices: 1.44M rows 151 MB, 320k rows 34 MB
    ("long_rows", lambda: _chain(45000, 45000), {}, {"pcg": (1, 0), "bicgstab": (0, 0)}),
    ("long_rows_small", lambda: _chain(10000, 10000), {}, {"pcg": (1, 1), "bicgstab": (1, 1)}),
    # rows of 7 entries, 2.1M rows: 30 KB of L1 are left to 64 and 50 KB of rows
    ("box_csr", lambda: synth.box_mesh(129, 129, 129, 2, 2, 2).ranks, CSR, {"pcg": (0, 0), "bicgstab": (0, 0)}),
    ("box_csr_small", lambda: synth.box_mesh(80, 80, 80, 2, 2, 2).ranks, CSR, {"pcg": (1, 1), "bicgstab": (1, 1)}),
    ("box_csr_parts", lambda: synth.box_mesh(126, 126, 126, 2, 2, 2).ranks, {"n_parts": 4, **CSR},
     {"pcg": (0, 0), "bicgstab": (0, 0)}),
    ("long_rows_csr", lambda: _chain(33000, 33000), CSR, {"pcg": (0, 1), "bicgstab": (0, 1)}),
    ("box", lambda: synth.box_mesh(126, 126, 126, 2, 2, 2).ranks, {}, {"pcg": (1, 1), "bicgstab": (0, 1)}),
])
def test_forms(name, ranks, kw, resident):
    build.build()
    repart.load()
    got = _forms(ranks(), **kw)
    want = {(s, p): bool(v) for s, ps in (("pcg", ("fp64", "mixed_ru")), ("bicgstab", ("fp64", "mixed")))
            for p, v in zip(ps, resident[s])}
    assert got == want
