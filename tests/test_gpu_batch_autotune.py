"""The autotuner does not leave a batch slower than it found it: 48 systems of 1k to
40k rows, whose own team size is none of those the autotuner goes through. Best of
five steps each; the next team size of its list is a seventh slower."""
import pytest
import torch

from paper_2510_08536_gb300 import build, repart, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_autotuned_shape_is_no_slower():
    build.build()
    repart.load()
    B = synth.Batch(48, 1000, 40000, seed=0)
    stg, b = (torch.from_numpy(v).to(DEV) for v in (B.staging(0.5, 100), B.rhs(0)))
    x = torch.zeros(B.n_rows, dtype=torch.float64, device=DEV)
    h = repart.batch_build(B.systems)

    def best():
        ms = []
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            repart.batch_update_solve(h, stg, b, x, 1e-9, "mixed_ru")
            e1.record()
            torch.cuda.synchronize()
            ms.append(e0.elapsed_time(e1))
        return min(ms[1:])

    own = best()
    shape = repart.batch_autotune(h, stg, b, x, tol=1e-9, precision="mixed_ru")
    tuned = best()
    assert tuned <= 1.05 * own, (own, tuned, shape)
    h.close()
