"""The streaming kernels of the PCG and BiCGStab iterations, which systems take that
do not fit the chip's shared memory, or whose spin_limit is too small for grid
meetings.

Small ragged systems with such a limit, in every layout, the caller's x off a
16-byte boundary; one ragged mesh just above the resident forms' range; and waits:
spin_limit = 0 makes the mbarrier waits of the sliced products give up (from the
graph and from the host loop), while the CSR kernels, which wait for nothing, solve
as ever.

Tolerances as in the parity tests: both sides run the same recurrence to 1e-9, so
the FP64 solutions agree to 1e-7 and the iteration counts to 2 (BiCGStab: a tenth);
true residuals are recomputed with the oracle's matrix."""
import numpy as np
import pytest
import torch

from gpu_util import Case
from oracle import pcg_omp
from oracle import repart_oracle as O
from paper_2510_08536_gb300 import build, repart, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SMALL = (1 << 16) - 1  # too few polls for a grid meeting, plenty of mbarrier probes


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    repart.load()
    torch.cuda.set_device(0)


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _zeros(n):
    return torch.zeros(n + 1, dtype=torch.float64, device=DEV)[1:]  # 8 bytes off a 16-byte boundary


SHAPES = [
    ((1, 1, 31), (1, 1, 1), {}),
    ((17, 17, 17), (2, 2, 2), {}),
    ((61, 53, 67), (3, 2, 4), {"symmetric": True}),
    ((19, 23, 29), (2, 3, 2), {"n_parts": 3}),
    ((83, 79, 71), (2, 1, 2), {"n_parts": 2}),
    ((37, 29, 31), (2, 2, 2), {"layout": repart.RP_LAYOUT_CSR}),
    ((37, 29, 31), (2, 2, 2), {"layout": repart.RP_LAYOUT_CSR, "n_parts": 4}),
]


@pytest.mark.parametrize("dims,ranks,kw", SHAPES)
def test_streaming_pcg(dims, ranks, kw):
    c = Case(dims, ranks, symmetric=kw.get("symmetric", False))
    ref = pcg_omp.pcg(c.map.row_ptr, c.map.col_idx, c.vals, c.dinv, c.b, tol=1e-9)
    h = repart.build_repartition(c.mesh.ranks, spin_limit=SMALL, **kw)
    repart.update_values_packed(h, _t(c.staging))
    for precision in ("fp64", "mixed", "mixed_ru"):
        x = _zeros(c.mesh.n_cells)
        info = repart.solve(h, _t(c.b), x, tol=1e-9, precision=precision)
        xs = x.cpu().numpy()
        assert repart.solve_form(h) == "streaming"
        assert info["status"] == 0 and c.true_rel_residual(xs) <= 1e-9, (precision, info)
        if precision == "fp64":
            assert np.linalg.norm(xs - ref.x) <= 1e-7 * np.linalg.norm(ref.x)
            assert abs(info["iterations"] - ref.iterations) <= 2
    h.close()


@pytest.mark.parametrize("dims,ranks,kw", [s for s in SHAPES if not s[2].get("symmetric")])
def test_streaming_bicgstab(dims, ranks, kw):
    mesh = synth.box_mesh(*dims, *ranks)
    stg = synth.momentum_staging(mesh, 0.5, 100)
    (m,) = O.repartition_map(mesh.ranks, 1)
    vals = O.update_values(m.src_of, stg)
    A = O.csr_matrix(m.row_ptr, m.col_idx, vals)
    b = synth.uniform_vector(mesh, 0)
    ref = O.bicgstab(A, O.jacobi_inverse(m.row_ptr, m.col_idx, vals, m.diag_pos), b, tol=1e-9)
    h = repart.build_repartition(mesh.ranks, spin_limit=SMALL, **kw)
    repart.update_values_packed(h, _t(stg))
    for precision in ("fp64", "mixed"):
        x = _zeros(mesh.n_cells)
        info = repart.solve_bicgstab(h, _t(b), x, tol=1e-9, precision=precision)
        xs = x.cpu().numpy()
        assert repart.solve_form(h) == "streaming"
        assert info["status"] == 0 and np.linalg.norm(b - A @ xs) <= 1e-9 * np.linalg.norm(b), (precision, info)
        assert np.linalg.norm(xs - ref.x) <= 1e-7 * np.linalg.norm(ref.x)
        if precision == "fp64":
            assert abs(info["iterations"] - ref.iterations) <= max(3, ref.iterations // 10)
    h.close()


@pytest.mark.parametrize("kw", [{}, {"n_parts": 3}])
def test_just_above_the_resident_range(kw):
    c = Case((139, 131, 127), (3, 2, 2))
    mst = synth.momentum_staging(c.mesh, 0.5, 100)
    Am = O.csr_matrix(c.map.row_ptr, c.map.col_idx, O.update_values(c.map.src_of, mst))
    h = repart.build_repartition(c.mesh.ranks, **kw)
    for solve, stg, A, precisions in ((repart.solve, c.staging, c.A, ("fp64", "mixed", "mixed_ru")),
                                      (repart.solve_bicgstab, mst, Am, ("fp64", "mixed"))):
        repart.update_values_packed(h, _t(stg))
        for precision in precisions:
            x = _zeros(c.mesh.n_cells)
            info = solve(h, _t(c.b), x, tol=1e-9, precision=precision)
            assert repart.solve_form(h) == "streaming"
            r = c.b - A @ x.cpu().numpy()
            assert info["status"] == 0 and np.linalg.norm(r) <= 1e-9 * np.linalg.norm(c.b), (precision, info)
    h.close()


@pytest.mark.parametrize("host_loop", [0, 1])
@pytest.mark.parametrize("layout", ["sliced", "csr"])
def test_no_probe_at_all(layout, host_loop):
    mesh = synth.box_mesh(96, 96, 96, 2, 2, 2)  # several chunks a block: the producer's waits run out too
    csr = layout == "csr"
    h = repart.build_repartition(mesh.ranks, spin_limit=0, host_loop=host_loop,
                                 layout=repart.RP_LAYOUT_CSR if csr else repart.RP_LAYOUT_AUTO)
    b = _t(synth.uniform_vector(mesh, 0))
    for solve, stg, precisions in (
            (repart.solve, synth.Assembler(mesh).staging(synth.face_coeffs(mesh, 0.5, 100)), ("fp64", "mixed", "mixed_ru")),
            (repart.solve_bicgstab, synth.momentum_staging(mesh, 0.5, 100), ("fp64", "mixed"))):
        repart.update_values_packed(h, _t(stg))
        for precision in precisions:
            x = torch.zeros_like(b)
            if csr:
                assert solve(h, b, x, tol=1e-6, precision=precision)["status"] == 0
            else:
                with pytest.raises(repart.RepartError) as e:
                    solve(h, b, x, tol=1e-6, precision=precision)
                assert e.value.status == repart.RP_DEVICE_TIMEOUT, precision
            assert repart.solve_form(h) == "streaming"
    h.close()


def test_line_preconditioner_on_many_rows():
    """4.1M rows: the FP32 residual kernel held to the registers of eight blocks an SM.
    Iterations as in the line preconditioner's own tests: 1.25 of FP64's and 10."""
    c = Case((161, 163, 157), (2, 2, 2))
    h = repart.build_repartition(c.mesh.ranks, precond=repart.RP_PRECOND_LINE)
    repart.update_values_packed(h, _t(c.staging))
    its = {}
    for precision in ("fp64", "mixed_ru"):
        x = _zeros(c.mesh.n_cells)
        info = repart.solve(h, _t(c.b), x, tol=1e-9, precision=precision)
        assert info["status"] == 0 and c.true_rel_residual(x.cpu().numpy()) <= 1e-9, (precision, info)
        its[precision] = info["iterations"]
    assert its["mixed_ru"] <= 1.25 * its["fp64"] + 10, its
    h.close()
