"""The gradients where their walk through the buffer branches: one trip of the grid,
four trips a rank search, results that stream past L2, more than 128 ranks
(some without cells). One product, or for symmetric storage two and their sum: bit
for bit the oracle's."""
import types

import numpy as np
import pytest
import torch

from oracle import repart_oracle as O
from paper_2510_08536_gb300 import build, repart, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _empty():
    z = np.zeros(0, np.int32)
    return types.SimpleNamespace(n_cells=0, n_faces=0, n_iface=0, lower_addr=z, upper_addr=z, iface_row=z,
                                 iface_nbr_rank=z, iface_nbr_col=z)


@pytest.mark.parametrize("symmetric", [False, True])
@pytest.mark.parametrize("dims,ranks,empty", [
    ((1, 1, 1), (1, 1, 1), 1),       # a cell without faces
    ((21, 22, 23), (6, 6, 5), 3),    # 183 ranks, three of them empty
    ((58, 57, 59), (3, 2, 2), 0),    # four trips
    ((90, 86, 83), (5, 6, 7), 2),    # 212 ranks, streamed
    ((91, 87, 84), (2, 2, 2), 1),    # streamed
])
def test_gradient_routes(dims, ranks, empty, symmetric):
    build.build()
    repart.load()
    r = list(synth.box_mesh(*dims, *ranks).ranks) + [_empty() for _ in range(empty)]
    h = repart.build_repartition(r, symmetric=symmetric)
    (m,) = O.repartition_map(r, 1, symmetric)
    rng = np.random.default_rng(7)
    lam, x = rng.uniform(-1, 1, h.n), rng.uniform(-1, 1, h.n)
    ld, xd = torch.from_numpy(lam).to(DEV), torch.from_numpy(x).to(DEV)
    g = torch.full((h.n_slots,), 7.0, dtype=torch.float64, device=DEV)
    f = torch.full((sum(len(q.lower_addr) + len(q.iface_row) for q in r),), 7.0, dtype=torch.float64, device=DEV)
    repart.entry_grad(h, ld, xd, g)
    repart.face_grad(h, ld, xd, f)
    want = O.slot_grad(m.src_of, O.entry_grad(m.row_ptr, m.col_idx, lam, x), h.n_slots)
    assert np.array_equal(g.cpu().numpy(), want)
    assert np.array_equal(f.cpu().numpy(), O.face_grad_ldu(r, lam, x))
    h.close()
