"""The resident forms of the PCG and BiCGStab iterations (one cooperative launch an inner run).

Against the oracle at the shapes where its split over the SMs changes: fewer
slices than SMs, ragged last slices, fewer warps than a full block, the
several-part and CSR layouts, and the FP64 form that keeps only r and q on chip.
Tolerances as in the parity tests: both sides run the same recurrence to 1e-9,
so the solutions agree to 1e-7 and the iteration counts to 2; true residuals
are recomputed with the oracle's matrix.

Solves of two handles on two streams from two threads, with launches of a
third stream between them: every result equals the one of a solve alone.
"""
import threading

import numpy as np
import pytest
import torch

from oracle import pcg_omp
from oracle import repart_oracle as O
from paper_2510_08536_gb300 import build, repart, synth
from gpu_util import Case

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    repart.load()
    torch.cuda.set_device(0)


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _solve(h, b, precision, stream=None):
    x = torch.zeros_like(b)
    info = repart.solve(h, b, x, tol=1e-9, precision=precision, stream=stream)
    return x, info


@pytest.mark.parametrize("dims,ranks,kw", [
    ((1, 1, 31), (1, 1, 1), {}),
    ((3, 11, 1), (1, 1, 1), {}),
    ((17, 17, 17), (2, 2, 2), {}),            # 154 slices: one SM more than one slice
    ((19, 23, 29), (2, 3, 2), {"n_parts": 3}),
    ((37, 29, 31), (2, 2, 2), {"layout": repart.RP_LAYOUT_CSR}),
    ((61, 53, 67), (3, 2, 4), {"symmetric": True}),
    ((83, 79, 71), (2, 1, 2), {"n_parts": 2}),  # FP32: matrix on chip, FP64: streamed
    ((97, 96, 95), (2, 2, 2), {}),            # matrix streamed
    ((109, 103, 101), (2, 2, 2), {}),         # FP64: r and q on chip only
])
def test_resident_solves(dims, ranks, kw):
    c = Case(dims, ranks, symmetric=kw.get("symmetric", False))
    ref = pcg_omp.pcg(c.map.row_ptr, c.map.col_idx, c.vals, c.dinv, c.b, tol=1e-9)
    h = repart.build_repartition(c.mesh.ranks, **kw)
    single = repart.build_repartition(c.mesh.ranks, host_loop=1, **kw)
    b = _t(c.b)
    for precision in ("fp64", "mixed", "mixed_ru"):
        repart.update_values_packed(h, _t(c.staging))
        x, info = _solve(h, b, precision)
        if c.mesh.n_cells < 100000:  # one iteration a launch: the same sums and states
            repart.update_values_packed(single, _t(c.staging))
            x1, info1 = _solve(single, b, precision)
            assert torch.equal(x, x1) and info == info1, precision
        xs = x.cpu().numpy()
        assert info["status"] == 0, (precision, info)
        assert c.true_rel_residual(xs) <= 1e-9, precision
        if precision == "fp64":
            assert np.linalg.norm(xs - ref.x) <= 1e-7 * np.linalg.norm(ref.x)
            assert abs(info["iterations"] - ref.iterations) <= 2
    h.close()
    single.close()


@pytest.mark.parametrize("dims,ranks,kw", [
    ((1, 1, 31), (1, 1, 1), {}),
    ((3, 11, 1), (1, 1, 1), {}),
    ((17, 17, 17), (2, 2, 2), {}),
    ((19, 23, 29), (2, 3, 2), {"n_parts": 3}),
    ((37, 29, 31), (2, 2, 2), {"layout": repart.RP_LAYOUT_CSR}),
    ((109, 103, 101), (2, 2, 2), {}),         # FP64: streaming
])
def test_resident_bicgstab(dims, ranks, kw):
    mesh = synth.box_mesh(*dims, *ranks)
    stg = synth.momentum_staging(mesh, 0.5, 100)
    (m,) = O.repartition_map(mesh.ranks, 1)
    vals = O.update_values(m.src_of, stg)
    A = O.csr_matrix(m.row_ptr, m.col_idx, vals)
    b = synth.uniform_vector(mesh, 0)
    ref = O.bicgstab(A, O.jacobi_inverse(m.row_ptr, m.col_idx, vals, m.diag_pos), b, tol=1e-9)
    hs = [repart.build_repartition(mesh.ranks, host_loop=k, **kw) for k in (0, 1)]
    for precision in ("fp64", "mixed"):
        out = []
        for h in hs:
            repart.update_values_packed(h, _t(stg))
            x = torch.zeros(h.n, dtype=torch.float64, device=DEV)
            info = repart.solve_bicgstab(h, _t(b), x, tol=1e-9, precision=precision)
            assert info["status"] == 0, (precision, info)
            out.append((x, info))
        assert torch.equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]  # one launch or one an iteration
        xs = out[0][0].cpu().numpy()
        assert np.linalg.norm(b - A @ xs) <= 1e-9 * np.linalg.norm(b), precision
        assert np.linalg.norm(xs - ref.x) <= 1e-7 * np.linalg.norm(ref.x)
        if precision == "fp64":
            assert abs(out[0][1]["iterations"] - ref.iterations) <= max(3, ref.iterations // 10)
    for h in hs:
        h.close()


def test_concurrent_solves():
    cases = [Case((24, 20, 18), (2, 1, 1), oracle_map=False), Case((48, 44, 40), (2, 2, 1), oracle_map=False)]
    hs = [repart.build_repartition(c.mesh.ranks) for c in cases]
    bs = [_t(c.b) for c in cases]
    for h, c in zip(hs, cases):
        repart.update_values_packed(h, _t(c.staging))
    alone = [[_solve(h, b, p)[0] for p in ("fp64", "mixed_ru")] for h, b in zip(hs, bs)]
    torch.cuda.synchronize()
    bad, stop = [], threading.Event()

    def work(k):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for _ in range(20):
                for p, want in zip(("fp64", "mixed_ru"), alone[k]):
                    x, info = _solve(hs[k], bs[k], p, s)
                    if info["status"] != 0 or not torch.equal(x, want):
                        bad.append((k, p, info))

    def noise():
        s, a = torch.cuda.Stream(), torch.ones(1 << 24, device=DEV)
        with torch.cuda.stream(s):
            while not stop.is_set():
                a.add_(1.0)
                s.synchronize()

    side = threading.Thread(target=noise)
    ts = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in [side] + ts:
        t.start()
    for t in ts:
        t.join()
    stop.set()
    side.join()
    assert not bad, bad
    for h in hs:
        h.close()
