"""The single passes over the matrix: the fused value update and the gradients in
buffer order, at the shapes where they branch: rows
longer than a warp's shared run, 8-bit and long offset tables, several parts,
ranks smaller than a warp's run, symmetric storage, and values outside the
range of the FP32 product of pairs.

The update is a permutation and conversions: every copy is compared bit for
bit with FP64 arithmetic on the same values. Gradients: one product (symmetric storage: two and their sum), bit for bit.
"""
import types

import numpy as np
import pytest
import torch

from oracle import repart_oracle as O
from paper_2510_08536_gb300 import build, repart, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    repart.load()
    torch.cuda.set_device(0)


def _graph(n, faces, reach, seed):
    """One rank whose cells meet at random faces (rows of any length up to 32)."""
    rng = np.random.default_rng(seed)
    lo = rng.integers(0, n - 1, faces)
    up = np.minimum(lo + 1 + rng.integers(0, reach, faces), n - 1)
    e = np.unique(np.stack([lo, up], 1)[lo < up], axis=0)
    deg = np.zeros(n, int)
    keep = []
    for i, (a, b) in enumerate(e):
        if deg[a] < 31 and deg[b] < 31:
            deg[a] += 1
            deg[b] += 1
            keep.append(i)
    e = e[keep].astype(np.int32)
    z = np.zeros(0, np.int32)
    return [types.SimpleNamespace(n_cells=n, n_faces=len(e), n_iface=0, lower_addr=e[:, 0], upper_addr=e[:, 1],
                                  iface_row=z, iface_nbr_rank=z, iface_nbr_col=z)]


SHAPES = {
    "box": (lambda: synth.box_mesh(23, 18, 21, 3, 2, 2).ranks, {}),
    "tiny_ranks": (lambda: synth.box_mesh(9, 8, 7, 4, 4, 3).ranks, {}),
    "parts": (lambda: synth.box_mesh(19, 16, 13, 2, 2, 2).ranks, {"n_parts": 4}),
    "symmetric": (lambda: synth.box_mesh(17, 11, 10, 2, 1, 3).ranks, {"symmetric": True}),
    "csr": (lambda: synth.box_mesh(13, 12, 11, 2, 2, 1).ranks, {"layout": repart.RP_LAYOUT_CSR}),
    "no_fp32": (lambda: synth.box_mesh(13, 12, 11, 2, 2, 1).ranks, {"want_fp32": False}),
    "long_rows": (lambda: _graph(701, 8000, 12, 1), {}),     # runs of more than 256 entries
    "long_tables": (lambda: _graph(997, 4000, 900, 2), {}),  # more than 16 and 32 offsets a slice
}


def _buffer(h, kind, seed):
    rng = np.random.default_rng(seed)
    v = -np.exp(rng.normal(0.0, 1.0, h.n_slots))
    if kind == "wide":
        v *= np.ldexp(1.0, rng.integers(-160, 160, h.n_slots))
        v[rng.integers(0, h.n_slots, 20)] = 0.0
        v[rng.integers(0, h.n_slots, 20)] = 1e-310
    return v


def _diagonal_positive(ranks, symmetric, v):
    at = 0
    for r in ranks:
        n, f, e = int(r.n_cells), len(r.lower_addr), len(r.iface_row)
        v[at:at + n] = np.abs(v[at:at + n]) + 1e-3
        at += n + f * (1 if symmetric else 2) + e
    return v


def _same(a, b):
    return np.array_equal(np.asarray(a).view(np.uint8), np.asarray(b).view(np.uint8))


@pytest.mark.parametrize("kind", ["plain", "wide", "special"])
@pytest.mark.parametrize("shape", SHAPES)
def test_update_bit_exact(shape, kind):
    ranks, kw = SHAPES[shape][0](), SHAPES[shape][1]
    h = repart.build_repartition(ranks, **kw)
    sym = kw.get("symmetric", False)
    v = _diagonal_positive(ranks, sym, _buffer(h, "plain", 0))
    fp32 = kw.get("want_fp32", True)
    repart.update_values_packed(h, torch.from_numpy(v).to(DEV))
    if fp32:  # the scaled values exist from here on, and every update refills them
        b = torch.ones(h.n, dtype=torch.float64, device=DEV)
        repart.solve(h, b, torch.zeros_like(b), tol=0.5, precision="mixed")
    v = _diagonal_positive(ranks, sym, _buffer(h, kind, 1))
    if kind == "special":
        rng = np.random.default_rng(3)
        off = np.flatnonzero(v < 0.0)
        v[rng.choice(off, 12, replace=False)] = np.repeat([np.inf, -np.inf, 3.5e38, 3.402823669e38], 3)
    repart.update_values_packed(h, torch.from_numpy(v).to(DEV))
    maps = O.repartition_map(ranks, kw.get("n_parts", 1), sym)
    got = repart.get_values(h)
    at = 0
    with np.errstate(over="ignore"):
        csr, base = [], 0
        for p, m in enumerate(maps):
            pm = repart.get_part_map(h, p)
            seg = v[pm["buf_off"]:pm["buf_off"] + pm["buf_len"]]
            csr.append(O.update_values(m.src_of, seg))
        csr = np.concatenate(csr)
        assert _same(got["vals"].cpu().numpy(), csr)
        if fp32:
            assert _same(got["vals32"].cpu().numpy(), csr.astype(np.float32))
        view = repart.get_sliced_view(h)
        assert (view is None) == (shape == "csr")
        if view is None:
            h.close()
            return
        pos = view["pos"].cpu().numpy()
        sliced = np.where(pos >= 0, csr[np.maximum(pos, 0)], 0.0)
        assert _same(view["vals"].cpu().numpy(), sliced)
        if fp32:
            assert _same(view["vals32"].cpu().numpy(), sliced.astype(np.float32))
        if len(maps) == 1 and fp32:
            (m,) = maps
            d = csr[m.diag_pos]
            s = 1.0 / np.sqrt(d)
            assert _same(got["dinv"].cpu().numpy(), 1.0 / d)
            assert _same(view["scale"].cpu().numpy(), s)
            rows = np.repeat(np.arange(h.n), np.diff(m.row_ptr))
            want = (csr * (s[rows] * s[m.col_idx])).astype(np.float32)
            assert _same(view["vals32s"].cpu().numpy(), np.where(pos >= 0, want[np.maximum(pos, 0)], np.float32(0)))
    h.close()


def test_scaled_values_of_a_large_mesh():
    """5M entries of wide draws: the rare entries near a rounding boundary are among them."""
    mesh = synth.box_mesh(96, 90, 84, 2, 2, 2)
    h = repart.build_repartition(mesh.ranks)
    b = torch.ones(h.n, dtype=torch.float64, device=DEV)
    for sigma, seed in ((0.5, 100), (4.0, 101)):
        stg = torch.from_numpy(synth.Assembler(mesh).staging(synth.face_coeffs(mesh, sigma, seed))).to(DEV)
        repart.update_values_packed(h, stg)
        repart.solve(h, b, torch.zeros_like(b), tol=0.5, precision="mixed")
        repart.update_values_packed(h, stg)
        m, view, vals = repart.get_part_map(h), repart.get_sliced_view(h), repart.get_values(h)["vals"]
        s = 1.0 / torch.sqrt(vals[m["diag_pos"].long()])
        rows = torch.repeat_interleave(torch.arange(h.n, device=DEV), m["row_ptr"].long().diff())
        want = (vals * (s[rows] * s[m["col_idx"].long()])).float()
        pos = view["pos"].long()
        assert torch.equal(view["vals32s"], torch.where(pos >= 0, want[pos.clamp(min=0)], torch.zeros((), device=DEV)))
    h.close()


def test_diagonal_reciprocal_and_root():
    """1/d and 1/sqrt(d) rounded as IEEE divisions and roots: mantissas next to
    powers of two and all ones, every exponent, and what has no such root."""
    rng = np.random.default_rng(11)
    n = 1 << 21
    mant = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    kind = rng.integers(0, 5, n)
    mant[kind == 1] = rng.integers(0, 64, (kind == 1).sum(), dtype=np.uint64)
    mant[kind == 2] = np.uint64((1 << 52) - 1) - rng.integers(0, 64, (kind == 2).sum(), dtype=np.uint64)
    mant[kind == 3] &= np.uint64(0xFFFFF00000000)
    expo = np.where(rng.random(n) < 0.5, rng.integers(1013, 1033, n), rng.integers(0, 2047, n)).astype(np.uint64)
    d = (mant | expo << np.uint64(52)).view(np.float64)
    d[:6] = [0.0, np.inf, 5e-324, 1.0, 2.0 ** -1022, np.finfo(np.float64).max]
    z = np.zeros(0, np.int32)
    rank = types.SimpleNamespace(n_cells=n, n_faces=0, n_iface=0, lower_addr=z, upper_addr=z, iface_row=z,
                                 iface_nbr_rank=z, iface_nbr_col=z)
    h = repart.build_repartition([rank])
    b = torch.ones(n, dtype=torch.float64, device=DEV)
    repart.update_values_packed(h, b)
    repart.solve(h, b, torch.zeros_like(b), tol=0.5, precision="mixed")  # the scaling exists from here on
    with np.errstate(all="ignore"):
        for sign in (1.0, -1.0):
            v = sign * d
            repart.update_values_packed(h, torch.from_numpy(v).to(DEV))
            s = 1.0 / np.sqrt(v)
            np.testing.assert_array_equal(repart.get_values(h)["dinv"].cpu().numpy(), 1.0 / v)
            view = repart.get_sliced_view(h)
            np.testing.assert_array_equal(view["scale"].cpu().numpy(), s)
            pos = view["pos"].cpu().numpy()
            np.testing.assert_array_equal(view["vals32s"].cpu().numpy()[pos >= 0], (v * (s * s)).astype(np.float32))
    h.close()


@pytest.mark.parametrize("shape", ["box", "tiny_ranks", "symmetric", "long_rows"])
def test_gradients(shape):
    ranks, kw = SHAPES[shape][0](), SHAPES[shape][1]
    if shape == "tiny_ranks":  # and a rank without cells between others
        z = np.zeros(0, np.int32)
        empty = types.SimpleNamespace(n_cells=0, n_faces=0, n_iface=0, lower_addr=z, upper_addr=z, iface_row=z,
                                      iface_nbr_rank=z, iface_nbr_col=z)
        ranks = list(ranks) + [empty]
    sym = kw.get("symmetric", False)
    h = repart.build_repartition(ranks, **kw)
    (m,) = O.repartition_map(ranks, 1, sym)
    rng = np.random.default_rng(5)
    lam, x = rng.uniform(-1, 1, h.n), rng.uniform(-1, 1, h.n)
    g = torch.full((h.n_slots,), 7.0, dtype=torch.float64, device=DEV)
    f = torch.full((sum(len(r.lower_addr) + len(r.iface_row) for r in ranks),), 7.0, dtype=torch.float64, device=DEV)
    ld, xd = torch.from_numpy(lam).to(DEV), torch.from_numpy(x).to(DEV)
    repart.entry_grad(h, ld, xd, g)
    repart.face_grad(h, ld, xd, f)
    want = O.slot_grad(m.src_of, O.entry_grad(m.row_ptr, m.col_idx, lam, x), h.n_slots)
    assert np.array_equal(g.cpu().numpy(), want)
    assert np.array_equal(f.cpu().numpy(), O.face_grad_ldu(ranks, lam, x))
    h.close()
