"""The two forms of the inner iterations in the bounds-checked build: cooperative
launches refused (as a driver under MPS refuses them) from the solve graph and
from the host loop, which then run the streaming kernels to the same residual;
and grid meetings that run out (their limit set to 0: every block gives up at its
first one), which end each solve with RP_DEVICE_TIMEOUT and leave the handle as good
as a fresh one; and solves of every resident form of the uniform layout, the forms
that the normal build runs on the same systems, with no access out of range.

A child process loads that library (the binding holds one library per process).
True residuals are recomputed with the oracle's matrix; 1e-9 is what the solves
are asked for."""
import multiprocessing as mp
import os
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


class _Systems:
    """A pressure and a momentum system on one ragged mesh, solved by a handle of the checked library."""

    def __init__(self, dims=(19, 17, 23), ranks=(2, 2, 2)):
        import torch

        from gpu_util import Case
        from oracle import repart_oracle as O
        from paper_2510_08536_gb300 import synth
        self.torch = torch
        c = Case(dims, ranks)
        self.ranks, self.n, self.b = c.mesh.ranks, c.mesh.n_cells, c.b
        mst = synth.momentum_staging(c.mesh, 0.5, 100)
        Am = O.csr_matrix(c.map.row_ptr, c.map.col_idx, O.update_values(c.map.src_of, mst))
        self.systems = {"pcg": (c.staging, c.A), "bicgstab": (mst, Am)}

    def dev(self, a):
        return self.torch.from_numpy(np.ascontiguousarray(a)).cuda()

    def solve(self, h, kind, precision):
        """(status, true relative residual, form)"""
        from paper_2510_08536_gb300 import repart
        stg, A = self.systems[kind]
        repart.update_values_packed(h, self.dev(stg))
        x = self.dev(np.zeros(self.n))
        f = repart.solve if kind == "pcg" else repart.solve_bicgstab
        info = f(h, self.dev(self.b), x, tol=1e-9, precision=precision)
        r = self.b - A @ x.cpu().numpy()
        return info["status"], float(np.linalg.norm(r) / np.linalg.norm(self.b)), repart.solve_form(h)


ALL = [("pcg", "fp64"), ("pcg", "mixed"), ("pcg", "mixed_ru"), ("bicgstab", "fp64"), ("bicgstab", "mixed")]


def _refused():
    from paper_2510_08536_gb300 import repart
    out = {}
    s = _Systems()
    for host_loop in (0, 1):
        h = repart.build_repartition(s.ranks, host_loop=host_loop)
        for refuse in (0, 1):
            repart.check_resident(h, refuse)
            for kind, precision in ALL:
                out[host_loop, refuse, kind, precision] = s.solve(h, kind, precision)
        h.close()
    return out


def _timeouts():
    from paper_2510_08536_gb300 import repart
    out = {}
    s = _Systems()
    for host_loop in (0, 1):
        h, fresh = (repart.build_repartition(s.ranks, host_loop=host_loop) for _ in range(2))
        for kind, precision in ALL:
            repart.check_resident(h, spin=0)
            try:
                out[host_loop, kind, precision, 0] = s.solve(h, kind, precision)
            except repart.RepartError as e:
                out[host_loop, kind, precision, 0] = e.status, repart.solve_form(h)
            repart.check_resident(h)
            out[host_loop, kind, precision, 1] = s.solve(h, kind, precision) == s.solve(fresh, kind, precision)
        h.close()
        fresh.close()
    return out


# rows where the forms change: one slice a warp, the matrix on chip, the matrix streamed (FP64)
FORMS = [
    ((19, 17, 23), {}, {"fp64": "resident_folded", "mixed": "resident_folded", "mixed_ru": "resident_folded"}),
    ((19, 17, 23), {"n_parts": 4}, {"fp64": "resident_folded", "mixed_ru": "resident_folded"}),
    ((61, 53, 67), {}, {"fp64": "resident_matrix", "mixed": "resident_matrix"}),
    ((61, 53, 67), {"n_parts": 2}, {"fp64": "resident_matrix", "mixed_ru": "resident_matrix"}),
    ((83, 79, 71), {}, {"fp64": "resident", "mixed_ru": "resident_matrix"}),
    ((83, 79, 71), {"n_parts": 2}, {"fp64": "resident", "mixed": "resident_matrix"}),
]


def _uniform():
    from paper_2510_08536_gb300 import repart
    out = {}
    for k, (dims, kw, forms) in enumerate(FORMS):
        s = _Systems(dims)
        h = repart.build_repartition(s.ranks, **kw)
        for precision in forms:
            out[k, "pcg", precision] = s.solve(h, "pcg", precision)
        for precision in ("fp64", "mixed"):
            out[k, "bicgstab", precision] = s.solve(h, "bicgstab", precision)
        h.close()
    return out


def _child(q, name):
    sys.path[:0] = [ROOT, HERE]
    try:
        from paper_2510_08536_gb300 import build, repart
        repart.load(build.build(check=True))
        repart.check_violations(reset=True)
        out = globals()[name]()
        out["violations"] = repart.check_violations(reset=True)
    except Exception:  # report to the parent
        import traceback
        out = {"error": traceback.format_exc()[-3000:]}
    q.put(out)


def _run(name):
    ctx = mp.get_context("spawn")
    q = ctx.Queue()
    p = ctx.Process(target=_child, args=(q, name))
    p.start()
    out = q.get(timeout=600)
    p.join(60)
    assert "error" not in out, out["error"]
    assert p.exitcode == 0
    assert out.pop("violations")[0] == 0
    return out


def test_grid_meetings_run_out():
    from paper_2510_08536_gb300 import repart
    for (host_loop, kind, precision, again), got in _run("_timeouts").items():
        case = (host_loop, kind, precision, got)
        if again:
            assert got is True, case
        else:
            assert got[0] == repart.RP_DEVICE_TIMEOUT and got[1] != "streaming", case


def test_uniform_forms():
    for (k, kind, precision), (status, residual, form) in _run("_uniform").items():
        want = FORMS[k][2][precision] if kind == "pcg" else "resident"
        assert status == 0 and residual <= 1e-9 and form == want, (FORMS[k][:2], kind, precision, status, residual, form)


def test_refused_cooperative_launches():
    for (host_loop, refuse, kind, precision), (status, residual, form) in _run("_refused").items():
        case = (host_loop, refuse, kind, precision, form)
        assert status == 0 and residual <= 1e-9, case
        assert (form == "streaming") == bool(refuse), case
