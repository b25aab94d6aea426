"""What is timed: the calls a CFD program makes of this library, through the Python binding.

A case is one call (or the few calls that always go together) on one mesh:

* ``update``  the value update of a time step (rp_update_values_packed);
* ``spmv``    y = A x with x.y (rp_spmv), what a program checks residuals with;
* ``step``    a time step: value update, then the pressure solve (rp_solve);
* ``momentum`` a time step of the non-symmetric momentum system (BiCGStab);
* ``grads``   the entry and face gradients of a solve with its adjoint at hand;
* ``autograd`` the differentiable solve, forward and backward;
* ``batch``   a time step of many uneven systems at once (rp_batch_update_solve).

Meshes, decompositions and coefficient draws are the synthetic workloads of
``synth`` at the sizes of the tests and the benchmark and between them. The
mesh is built once per shape; every draw of coefficients, right-hand sides and
gradients comes from the seed. Solves are asked for 1e-9 in FP64 (the
benchmark's tolerance, which the FP64 recurrence reproduces to rounding) and,
where the inner iteration is FP32 or BiCGStab, for 1e-12: the solution is then
settled far below the rounding of the inner iteration and can be compared.
"""
import functools
import math

import numpy as np
import torch

from paper_2510_08536_gb300 import autograd, repart, synth

DEV = "cuda"


def listed():
    def case(name, call, n, p, **kw):
        return dict(name=name, call=call, nx=n[0], ny=n[1], nz=n[2], px=p[0], py=p[1], pz=p[2], **kw)

    return [
        # the smallest call: the update of the 32^3 mesh of 8 ranks, all launches and latency
        case("update_32", "update", (32, 32, 32), (2, 2, 2), sigma=0.5),
        # the largest update: the headline mesh, 128 ranks; the program solves in mixed
        # precision, so the handle keeps the scaled FP32 system up to date as well
        case("update_256", "update", (256, 256, 256), (8, 4, 4), sigma=1.0, scaled=True),
        # a residual check on a mesh whose extents and ranks divide nothing evenly
        case("spmv_odd", "spmv", (171, 149, 163), (5, 3, 4), sigma=0.5),
        # the small time step, resident in L2: uniform coefficients, 8 ranks, FP64
        case("step_32_fp64", "step", (32, 32, 32), (2, 2, 2), sigma=0.0, precision="fp64"),
        # an odd mid-size time step in restarted refinement
        case("step_odd_mixed", "step", (97, 61, 83), (3, 2, 4), sigma=0.5, precision="mixed"),
        # the 128^3 time step of 64 ranks in FP64
        case("step_128_fp64", "step", (128, 128, 128), (4, 4, 4), sigma=0.5, precision="fp64"),
        # the headline: 256^3, 128 ranks, continued refinement
        case("step_256_mixed_ru", "step", (256, 256, 256), (8, 4, 4), sigma=1.0, precision="mixed_ru"),
        # 64 CPU ranks on 8 GPU parts: local and non-local matrices
        case("step_128_parts", "step", (128, 128, 128), (4, 4, 4), sigma=0.5, precision="mixed_ru", parts=8),
        # the momentum system, FP32 BiCGStab in FP64 refinement
        case("momentum_128_mixed", "momentum", (128, 128, 128), (4, 4, 4), sigma=0.5, precision="mixed"),
        # gradients of a solve whose adjoint is at hand
        case("grads_128", "grads", (128, 128, 128), (4, 4, 4), sigma=0.5),
        # a differentiable solve in a training loop, forward and backward
        case("autograd_64", "autograd", (64, 64, 64), (2, 2, 2), sigma=0.5, precision="fp64"),
        # many uneven systems at once
        dict(name="batch_48_mixed_ru", call="batch", count=48, lo=8000, hi=300000, shapes=0, sigma=0.5, precision="mixed_ru"),
    ]


def draw(rng):
    call = rng.choice(["update", "update", "spmv", "step", "step", "step", "momentum", "grads", "autograd", "batch"])
    if call == "batch":
        hi = int(math.exp(rng.uniform(math.log(4e4), math.log(3e5))))
        return dict(call=call, count=rng.randint(9, 48), lo=rng.randint(1000, 8000), hi=hi, shapes=rng.randrange(1 << 20),
                    sigma=rng.choice([0.25, 0.5, 1.0]), precision=rng.choice(["fp64", "mixed", "mixed_ru"]))
    # cells over the whole range (logarithmic) and uneven aspects; the iterative calls
    # stay below the headline's cost in FP64 too
    top = {"update": 256, "spmv": 256, "grads": 192, "step": 192, "momentum": 192, "autograd": 96}[call]
    c = math.exp(rng.uniform(math.log(11.0), math.log(float(top))))
    ext = [c, c * rng.uniform(0.6, 1.0), c * rng.uniform(0.6, 1.0)]
    rng.shuffle(ext)
    n = [max(6, int(round(e))) for e in ext]
    p = [rng.randint(1, 4 if e >= 16 else 2) for e in n]
    d = dict(call=call, nx=n[0], ny=n[1], nz=n[2], px=p[0], py=p[1], pz=p[2], sigma=rng.choice([0.0, 0.5, 0.5, 1.0]))
    if call == "update":
        d.update(scaled=rng.random() < 0.5, symmetric=rng.random() < 0.25, sigma=max(d["sigma"], 0.25))
    if call == "step":
        d.update(precision=rng.choice(["fp64", "mixed", "mixed_ru"]), symmetric=rng.random() < 0.2)
        kind = rng.random()
        if kind < 0.2:
            d["parts"] = p[2]  # ranks run x, y, z: p[2] divides their number
        elif kind < 0.3:
            d["line"] = True
    if call == "momentum":
        d.update(precision=rng.choice(["fp64", "mixed"]), sigma=max(d["sigma"], 0.25))
    if call == "autograd":
        d["precision"] = rng.choice(["fp64", "fp64", "mixed_ru"])
    return d


# ---------------------------------------------------------------- inputs


class _Mesh:
    """A decomposed mesh and where every slot of its coefficient buffer comes from."""

    def __init__(self, mesh, symmetric):
        self.mesh, self.symmetric, self.n = mesh, symmetric, mesh.n_cells
        self.slots = mesh.staging_size(symmetric)
        self._index = self._momentum = None

    def staging(self, sigma, gen):
        """Pressure system: lognormal face coefficients (sigma 0: all 1), assembled diagonal."""
        m = self.mesh
        if self._index is None:
            self._index = torch.from_numpy(synth.Assembler(m, self.symmetric).index).to(DEV)
        a = torch.ones(m.n_internal_faces + m.n_boundary_faces, dtype=torch.float64, device=DEV)
        if sigma > 0.0:
            a = torch.empty_like(a).log_normal_(0.0, sigma, generator=gen)
        d = torch.full((m.nz, m.ny, m.nx), synth.DIAG_SHIFT, dtype=torch.float64, device=DEV)
        self._add_faces(d, a, a)
        d[:, :, 0] += 2.0 * a[m.n_internal_faces:].reshape(m.nz, m.ny)
        return torch.cat([d.reshape(-1), -a])[self._index]

    def _add_faces(self, d, low, high):
        """Adds every internal face's coefficient to its low-side and its high-side cell."""
        m, at = self.mesh, 0
        for axis, ext in ((2, (m.nz, m.ny, m.nx - 1)), (1, (m.nz, m.ny - 1, m.nx)), (0, (m.nz - 1, m.ny, m.nx))):
            cnt = ext[0] * ext[1] * ext[2]
            d.narrow(axis, 0, ext[axis]).add_(low[at:at + cnt].reshape(ext))
            d.narrow(axis, 1, ext[axis]).add_(high[at:at + cnt].reshape(ext))
            at += cnt

    def momentum(self, sigma, gen):
        """Upwind convection-diffusion: lower and upper coefficients differ."""
        m = self.mesh
        nf = m.n_internal_faces
        if self._momentum is None:
            parts = []
            for r in m.ranks:
                row = r.cell_gid[r.iface_row]
                col = np.empty(r.n_iface, np.int64)
                for q in np.unique(r.iface_nbr_rank):
                    s = r.iface_nbr_rank == q
                    col[s] = m.ranks[q].cell_gid[r.iface_nbr_col[s]]
                parts += [r.cell_gid, m.n_cells + r.face_gid, m.n_cells + nf + r.face_gid,
                          m.n_cells + r.iface_face_gid + np.where(row < col, 0, nf)]
            flux = torch.from_numpy(synth._face_flux(m, synth.MOMENTUM_U0)).to(DEV)
            self._momentum = torch.from_numpy(np.concatenate(parts)).to(DEV), flux
        index, flux = self._momentum
        a = torch.empty(nf, dtype=torch.float64, device=DEV).log_normal_(0.0, sigma, generator=gen)
        up, lo = -(a + torch.clamp(-flux, min=0.0)), -(a + torch.clamp(flux, min=0.0))
        d = torch.full((m.nz, m.ny, m.nx), synth.MOMENTUM_CT, dtype=torch.float64, device=DEV)
        self._add_faces(d, -up, -lo)
        return torch.cat([d.reshape(-1), up, lo])[index]

    @functools.cached_property
    def entries(self):
        """(row, column, slot) of every stored coefficient of the merged matrix, rows and columns in merged order."""
        m = self.mesh
        off = np.concatenate([[0], np.cumsum([r.n_cells for r in m.ranks])])
        rows, cols, slots, at = [], [], [], 0
        for k, r in enumerate(m.ranks):
            cell, o = np.arange(r.n_cells), off[k]
            face = np.arange(r.n_faces) + at + r.n_cells
            low = face if self.symmetric else face + r.n_faces
            end = at + r.n_cells + r.n_faces * (1 if self.symmetric else 2)
            rows += [o + cell, o + r.lower_addr, o + r.upper_addr, o + r.iface_row]
            cols += [o + cell, o + r.upper_addr, o + r.lower_addr, off[r.iface_nbr_rank] + r.iface_nbr_col]
            slots += [at + cell, face, low, end + np.arange(r.n_iface)]
            at = end + r.n_iface
        return tuple(torch.from_numpy(np.concatenate(v).astype(np.int64)).to(DEV) for v in (rows, cols, slots))


@functools.lru_cache(maxsize=3)
def _mesh(n, p, symmetric):
    return _Mesh(synth.box_mesh(*n, *p), symmetric)


@functools.lru_cache(maxsize=2)
def _batch(count, lo, hi, shapes):
    return [_Mesh(synth.box_mesh(*d), False) for d in synth.batch_shapes(count, lo, hi, shapes)]


def _meshes(case):
    """The independent systems of a case: one merged mesh, or the batch's."""
    if case["call"] == "batch":
        return _batch(case["count"], case["lo"], case["hi"], case["shapes"])
    return [_mesh((case["nx"], case["ny"], case["nz"]), (case["px"], case["py"], case["pz"]), bool(case.get("symmetric")))]


def _inputs(case, seed):
    """The coefficient buffer and two vectors of merged rows, uniform in [-1, 1]."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    ms = _meshes(case)
    momentum = case["call"] == "momentum"
    buf = torch.cat([m.momentum(case["sigma"], gen) if momentum else m.staging(case["sigma"], gen) for m in ms])
    n = sum(m.n for m in ms)
    b, g = (torch.empty(n, dtype=torch.float64, device=DEV).uniform_(-1.0, 1.0, generator=gen) for _ in range(2))
    return buf, b, g


def _tol(case):
    return 1e-9 if case.get("precision", "fp64") == "fp64" and case["call"] in ("step", "batch") else 1e-12


def prepare(case, seed):
    call = case["call"]
    buf, b, g = _inputs(case, seed)
    if call == "batch":
        h = repart.batch_build([m.mesh.ranks[0] for m in _meshes(case)])
    else:
        (m,) = _meshes(case)
        h = repart.build_repartition(m.mesh.ranks, n_parts=case.get("parts", 1), symmetric=m.symmetric,
                                     want_transpose=call == "autograd",
                                     precond=repart.RP_PRECOND_LINE if case.get("line") else repart.RP_PRECOND_JACOBI)
    s = dict(call=call, h=h, buf=buf, b=b, g=g, x=torch.zeros_like(b), tol=_tol(case), precision=case.get("precision"))
    if call == "update" and case.get("scaled"):
        # a program that solves in mixed precision: its first time step lies behind it
        repart.update_values_packed(h, buf)
        repart.solve(h, b, s["x"], tol=0.1, precision="mixed_ru")
    if call == "spmv":
        repart.update_values_packed(h, buf)
        s.update(y=torch.empty_like(b), xy=torch.empty(1, dtype=torch.float64, device=DEV))
    if call == "grads":
        s.update(entry=torch.empty_like(buf), face=torch.empty(sum(r.n_faces + r.n_iface for r in m.mesh.ranks), dtype=torch.float64, device=DEV))
    if call == "autograd":
        buf.requires_grad_(True)
        b.requires_grad_(True)
    return s


def run(s):
    call, h = s["call"], s["h"]
    if call == "batch":
        repart.batch_update_solve(h, s["buf"], s["b"], s["x"], tol=s["tol"], precision=s["precision"])
        return s["x"]
    if call == "autograd":
        x = autograd.solve(h, s["buf"], s["b"], tol=s["tol"], precision=s["precision"])
        return (x.detach(), *torch.autograd.grad(x, (s["buf"], s["b"]), s["g"]))
    if call == "grads":
        repart.entry_grad(h, s["g"], s["b"], s["entry"])
        repart.face_grad(h, s["g"], s["b"], s["face"])
        return s["entry"], s["face"]
    if call == "spmv":
        repart.spmv(h, s["b"], s["y"], s["xy"])
        return s["y"], s["xy"]
    repart.update_values_packed(h, s["buf"])
    if call == "update":
        v = repart.get_values(h)  # views of the handle's memory: they have to keep it
        v["vals"].handle = v["vals32"].handle = v["dinv"].handle = h
        return v["vals"], v["vals32"], v["dinv"]
    if call == "momentum":
        repart.solve_bicgstab(h, s["b"], s["x"], tol=s["tol"], precision=s["precision"])
    else:
        repart.solve(h, s["b"], s["x"], tol=s["tol"], precision=s["precision"])
    return s["x"]


def work(case):
    ms = _meshes(case)
    n, nnz, slots = sum(m.n for m in ms), sum(m.mesh.nnz() for m in ms), sum(m.slots for m in ms)
    faces = (nnz - n) // 2
    # iterations of the solves, roughly: they grow with the longest mesh axis
    its = max(8.0 * max(m.mesh.nx, m.mesh.ny, m.mesh.nz) for m in ms)
    call = case["call"]
    if call == "update":  # buffer and permutation in; both copies of the values and the diagonals out
        return {"bytes": 8 * slots + 4 * nnz + 12 * nnz + 12 * n, "flops": 2 * n}
    if call == "spmv":  # values and columns, x in, y out
        return {"bytes": 12 * nnz + 4 * n + 16 * n, "flops": 2 * nnz + 2 * n}
    if call == "grads":  # two vectors and the addressing in, both gradients out
        return {"bytes": 32 * n + 2 * 8 * faces + 8 * slots + 8 * faces, "flops": 2 * nnz + 3 * faces}
    if call == "momentum":
        return {"bytes": 8 * slots + 16 * n, "flops": 150 * (4 * nnz + 20 * n)}
    if call == "autograd":
        return {"bytes": 16 * slots + 32 * n, "flops": 2.5 * its * (2 * nnz + 12 * n)}
    return {"bytes": 8 * slots + 16 * n, "flops": its * (2 * nnz + 12 * n)}


# ---------------------------------------------------------------- the same in 64 bits


def _csr(ms, buf, transpose=False):
    rows, cols, slots, ro, so = [], [], [], 0, 0
    for m in ms:
        r, c, s = m.entries
        rows.append(r + ro), cols.append(c + ro), slots.append(s + so)
        ro, so = ro + m.n, so + m.slots
    r, c, s = torch.cat(rows), torch.cat(cols), torch.cat(slots)
    if transpose:
        r, c = c, r
    order = torch.argsort(r * ro + c)
    ptr = torch.zeros(ro + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = torch.cumsum(torch.bincount(r, minlength=ro), 0)
    vals = buf[s[order]]
    return torch.sparse_csr_tensor(ptr, c[order], vals, (ro, ro)), vals, buf[s[r == c]][torch.argsort(r[r == c])]


def _cg(A, d, b):
    """A x = b by Jacobi-CG in 64 bits, restarted from the true residual until it stops falling."""
    x, last = torch.zeros_like(b), math.inf
    for _ in range(4):
        r = b - A @ x
        if not float(r.norm()) < 0.1 * last:
            break
        last = float(r.norm())
        y, z = torch.zeros_like(b), r / d
        p, rz, stop = z.clone(), torch.dot(r, z), 1e-6 * last
        for k in range(1, 20001):
            q = A @ p
            alpha = rz / torch.dot(p, q)
            y += alpha * p
            r -= alpha * q
            if k % 16 == 0 and float(r.norm()) <= stop:
                break
            z = r / d
            rz, old = torch.dot(r, z), rz
            p = z + (rz / old) * p
        x = x + y
    return x


def _bicgstab(A, d, b):
    x, last = torch.zeros_like(b), math.inf
    for _ in range(5):
        r = b - A @ x
        if not float(r.norm()) < 0.1 * last:
            break
        last = float(r.norm())
        h, y, rho = r.clone(), torch.zeros_like(b), torch.dot(r, r)
        p, stop = r.clone(), 1e-6 * last
        for k in range(2000):
            u = p / d
            v = A @ u
            alpha = rho / torch.dot(h, v)
            s = r - alpha * v
            w = s / d
            t = A @ w
            omega = torch.dot(t, s) / torch.dot(t, t)
            y += alpha * u + omega * w
            r = s - omega * t
            if float(r.norm()) <= stop:
                break
            rho, old = torch.dot(h, r), rho
            p = r + (rho / old) * (alpha / omega) * (p - omega * v)
        x = x + y
    return x


def exact(case, seed):
    call, ms = case["call"], _meshes(case)
    buf, b, g = _inputs(case, seed)
    if call == "grads":
        m = ms[0]
        r, c, s = m.entries
        entry = torch.zeros_like(buf).index_add_(0, s, -g[r] * b[c])
        face, off = [], 0
        offs = np.concatenate([[0], np.cumsum([q.n_cells for q in m.mesh.ranks])])
        for k, q in enumerate(m.mesh.ranks):
            lo = np.concatenate([offs[k] + q.lower_addr, offs[k] + q.iface_row]).astype(np.int64)
            hi = np.concatenate([offs[k] + q.upper_addr, offs[q.iface_nbr_rank] + q.iface_nbr_col]).astype(np.int64)
            lo, hi = torch.from_numpy(lo).to(DEV), torch.from_numpy(hi).to(DEV)
            face.append(-(g[lo] - g[hi]) * (b[lo] - b[hi]))
        return entry, torch.cat(face)
    A, vals, d = _csr(ms, buf)
    if call == "update":
        return vals, vals, 1.0 / d
    if call == "spmv":
        y = A @ b
        return y, torch.dot(b, y).reshape(1)
    if call == "momentum":
        return _bicgstab(A, d, b)
    x = _cg(A, d, b)
    if call == "autograd":
        lam = _cg(_csr(ms, buf, transpose=True)[0], d, g)
        r, c, s = ms[0].entries
        return x, torch.zeros_like(buf).index_add_(0, s, -lam[r] * x[c]), lam
    return x
