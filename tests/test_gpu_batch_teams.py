"""The batch's own choice of team size: batches of one system, of fewer systems
than teams, of many small ones and of one large among small ones, whose choices
differ. Every system's residual is recomputed from its LDU coefficients (1e-9
asked for, the solver's own bound)."""
import numpy as np
import pytest
import torch

from oracle import repart_oracle as O
from paper_2510_08536_gb300 import build, repart, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("count,lo,hi", [(1, 20, 30), (1, 90000, 90001), (3, 500, 2000), (30, 200, 3000), (200, 30, 900)])
def test_default_team_size(count, lo, hi):
    build.build()
    repart.load()
    B = synth.Batch(count, lo, hi, seed=3)
    stg, b = B.staging(0.5, 100), B.rhs(0)
    h = repart.batch_build(B.systems)
    ro = np.cumsum([0] + [m.n_cells for m in B.meshes])
    so = np.cumsum([0] + [m.staging_size() for m in B.meshes])
    for precision in ("fp64", "mixed", "mixed_ru"):
        x = torch.zeros(B.n_rows, dtype=torch.float64, device=DEV)
        infos = repart.batch_update_solve(h, torch.from_numpy(stg).to(DEV), torch.from_numpy(b).to(DEV), x, 1e-9, precision)
        xs = x.cpu().numpy()
        for s, rank in enumerate(B.systems):
            xi, bi = xs[ro[s]:ro[s + 1]], b[ro[s]:ro[s + 1]]
            r = bi - O.ldu_matvec([rank], stg[so[s]:so[s + 1]], xi)
            assert infos[s]["status"] == 0 and np.linalg.norm(r) <= 1e-9 * np.linalg.norm(bi), (precision, s)
    h.close()
