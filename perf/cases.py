"""The calls a user of libvie makes, as measurable cases.

A case names an array of meta-atoms (``array``, ``ns`` or ``atoms``, ``nv``), the
entry point (``kind``) and its options.  Kinds:

  apply    Operator.apply on a compressed operator (plain, fused with the
           preconditioner, or adjoint), in one of the four precisions;
  precond  Operator.precond (the block-diagonal preconditioner alone);
  rhs      Operator.rhs, the right-hand sides of a set of plane waves;
  fields   Operator.far_field, Operator.near_field and Operator.sigma of given
           currents (host arrays in, host arrays out);
  solve    Operator.solve on a compressed operator, the currents left on the device;
  request  geometry in, currents out: Operator(), compress(), solve().

Sizes, materials and incidence are those of workloads.py: square arrays of
dielectric cubes (side 0.2, pitch 0.4), lens-graded arrays of three cube sides,
and the gold Vogel spiral.
"""
import numpy as np
import torch

import workloads
from paper_2603_10586_gb300 import vie

PRECISION = {"c64": vie.C64, "c128": vie.C128, "bf16x3": vie.BF16X3, "c64_acc64": vie.C64_ACC64}
WIDE = ("c128", "c64_acc64")
MODE = {"plain": 0, "fused": vie.FUSE_PRECOND, "adjoint": vie.ADJOINT}


def listed():
    return [
        # a unit cell study or a test of a model: the smallest array of the parity
        # cases, one product; launches and latency are all there is
        dict(name="apply_small", kind="apply", array="square", ns=4, nv=3, nrhs=1, precision="c64", mode="plain"),
        # single-incidence solves of the 16 x 16 array of 6^3 cubes: the inner product of each step
        dict(name="apply_one", kind="apply", array="square", ns=16, nv=6, nrhs=1, precision="c64", mode="fused"),
        # the aperiodic, lossy array (gold atoms on a Vogel spiral): no two far blocks share factors
        dict(name="apply_spiral", kind="apply", array="spiral", atoms=500, nv=3, nrhs=1, precision="c64", mode="fused"),
        # a served request's inner product: 1 to 8 right-hand sides in complex float32
        dict(name="apply_serving", kind="apply", array="square", ns=28, nv=3, nrhs=5, precision="c64", mode="fused"),
        # the lens-graded array with 16 incidences: split-precision product on the tensor cores
        dict(name="apply_graded", kind="apply", array="graded", ns=24, nv=4, nrhs=16, precision="bf16x3", mode="fused"),
        # the 32-angle, two-polarisation sweep of the 32 x 32 array: one inner product for 64 right-hand sides
        dict(name="apply_sweep", kind="apply", array="square", ns=32, nv=4, nrhs=64, precision="bf16x3", mode="fused"),
        # the float64-accurate refinement residual of a multi-incidence solve
        dict(name="residual", kind="apply", array="square", ns=16, nv=4, nrhs=24, precision="c64_acc64", mode="plain"),
        # the all-float64 operator, the accuracy comparator
        dict(name="apply_double", kind="apply", array="square", ns=12, nv=3, nrhs=3, precision="c128", mode="plain"),
        # right-hand sides of the same sweep: every solve begins with them
        dict(name="rhs_sweep", kind="rhs", array="square", ns=32, nv=4, nrhs=64),
        # what a solve is read out as: far field, near field and cross sections
        dict(name="fields", kind="fields", array="square", ns=10, nv=3, nrhs=4, ndirs=181, npts=100),
        # a served request from geometry to currents
        dict(name="request", kind="request", array="square", ns=8, nv=3, nrhs=2, precision="c64"),
        # a multi-incidence solve on an operator at hand
        dict(name="solve", kind="solve", array="square", ns=16, nv=4, nrhs=32, precision="bf16x3"),
    ]


def _log(rng, lo, hi):
    """An integer in [lo, hi], uniform in its logarithm."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["apply"] * 5 + ["precond", "rhs", "fields", "request", "solve"])
    nv = rng.randint(2, 4)
    if kind in ("request", "solve"):
        c = dict(kind=kind, nv=nv, nrhs=_log(rng, 1, 32 if kind == "solve" else 8),
                 precision=rng.choice(["c64", "bf16x3"]))
        # (the lens-graded array is resonant: its solves take minutes)
        if rng.random() < 0.3:
            c.update(array="spiral", atoms=_log(rng, 5, 200), nv=min(nv, 3))
        else:
            c.update(array="square", ns=_log(rng, 3, 16 if kind == "solve" else 12))
        return c
    if kind == "fields":
        return dict(kind=kind, array="square", ns=_log(rng, 3, 10), nv=rng.randint(2, 3), nrhs=_log(rng, 1, 4),
                    ndirs=_log(rng, 1, 181), npts=_log(rng, 1, 100))
    if kind == "rhs":
        return dict(kind=kind, array=rng.choice(["square", "graded"]), ns=_log(rng, 3, 32), nv=nv,
                    nrhs=_log(rng, 1, 64))
    if kind == "precond":
        return dict(kind=kind, array=rng.choice(["square", "graded"]), ns=_log(rng, 3, 32), nv=nv,
                    nrhs=_log(rng, 1, 64), precision=rng.choice(["c64", "c128"]))
    precision = rng.choice(["c64", "c64", "bf16x3", "bf16x3", "c64_acc64", "c128"])
    nrhs = 1 if precision == "c64" and rng.random() < 0.4 else _log(rng, 1, 64 if precision == "bf16x3" else 12)
    c = dict(kind=kind, nv=nv, nrhs=nrhs, precision=precision, mode=rng.choice(["plain", "fused", "fused", "adjoint"]))
    if precision == "c128":
        c.update(array="square", ns=_log(rng, 3, 12), nv=min(nv, 3))
    elif rng.random() < 0.25:
        c.update(array="spiral", atoms=_log(rng, 5, 500), nv=rng.randint(2, 3))
    else:
        c.update(array=rng.choice(["square", "square", "graded"]), ns=_log(rng, 3, 28))
    return c


# ----------------------------------------------------------------------------
# geometry, operator, inputs
# ----------------------------------------------------------------------------
_CTX = []


def _context():
    """One context per process, as a program holds it."""
    if not _CTX:
        _CTX.append(vie.Context(0))
    return _CTX[0]


def _geometry(case, wavelength=1.0, eps=12.0):
    if case["array"] == "spiral":
        return workloads.vogel_gold(case["atoms"], nv=case["nv"])
    if case["array"] == "graded":
        return workloads.graded_array(case["ns"], case["nv"], seed=case["ns"], eps=eps, wavelength=wavelength)
    return workloads.square_array(case["ns"], case["nv"], eps=eps, wavelength=wavelength)


def _operator(case, geometry, compress=True):
    op = vie.Operator(_context(), geometry)
    if compress:
        op.compress(1e-4, vie.C128 if case.get("precision") == "c128" else vie.C64)
    return op


def _vectors(n, nrhs, wide, seed):
    """nrhs complex normal vectors of n entries (one per row), the Krylov vectors of a solve."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((nrhs, n), generator=g, device="cuda", dtype=torch.complex128 if wide else torch.complex64)


def _request(case, seed):
    """Geometry and plane waves of a request: wavelength and permittivity as in the serving stream."""
    rng = np.random.default_rng(seed)
    g = _geometry(case, wavelength=float(rng.uniform(0.97, 1.03)), eps=float(rng.uniform(11.0, 12.0)))
    kh, pol = workloads.random_directions(case["nrhs"], seed)
    return g, kh, pol


def _currents(n, nrhs, seed):
    """Host currents of n unknowns, complex normal, one column per right-hand side."""
    return workloads.random_complex(n, seed, nrhs)


def _directions(count, seed):
    rng = np.random.default_rng(seed + 1)
    d = rng.standard_normal((count, 3))
    return d / np.linalg.norm(d, axis=1, keepdims=True)


def _points(count, geometry, seed):
    """Points a third of a wavelength to three wavelengths above the array."""
    rng = np.random.default_rng(seed + 2)
    half = np.abs(geometry.centres[:, :2]).max() + 0.2
    return np.concatenate([rng.uniform(-half, half, (count, 2)), rng.uniform(0.35, 3.0, (count, 1))], 1)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, kind=kind)
    if kind == "request":
        st["geometry"], st["khat"], st["pol"] = _request(case, seed)
        n = st["geometry"].unknowns()
        st["I"] = torch.zeros((case["nrhs"], n), dtype=torch.complex128, device="cuda")
        return st
    g = _geometry(case)
    op = _operator(case, g, compress=kind in ("apply", "solve"))
    st["op"] = op
    if kind in ("apply", "precond"):
        x = _vectors(op.n, case["nrhs"], case["precision"] in WIDE, seed)
        st.update(x=x, y=torch.empty_like(x))
    elif kind in ("rhs", "solve"):
        st["khat"], st["pol"] = workloads.random_directions(case["nrhs"], seed, max_deg=60.0)
        st["I"] = torch.zeros((case["nrhs"], op.n), dtype=torch.complex128, device="cuda")
    else:
        st["khat"], st["pol"] = workloads.random_directions(case["nrhs"], seed)
        st["I"] = _currents(op.n, case["nrhs"], seed)
        st["dirs"] = _directions(case["ndirs"], seed)
        st["points"] = _points(case["npts"], g, seed)
    return st


def run(state):
    kind, case = state["kind"], state["case"]
    if kind == "apply":
        x, y = state["x"], state["y"]
        state["op"].apply(x.data_ptr(), y.data_ptr(), case["nrhs"], PRECISION[case["precision"]], MODE[case["mode"]])
        return y
    if kind == "precond":
        x, y = state["x"], state["y"]
        state["op"].precond(x.data_ptr(), y.data_ptr(), case["nrhs"], PRECISION[case["precision"]])
        return y
    if kind == "rhs":
        state["op"].rhs(state["khat"], state["pol"], state["I"].data_ptr())
        return state["I"]
    if kind == "fields":
        op, I = state["op"], state["I"]
        return {"far": op.far_field(I, state["dirs"]), "near": op.near_field(I, state["points"]),
                "sigma": op.sigma(I, state["khat"], state["pol"])}
    op = state.get("op")
    if kind == "request":
        op = vie.Operator(_context(), state["geometry"])
        op.compress(1e-4, vie.C64)
    op.solve(state["khat"], state["pol"], tol=1e-6, precision=PRECISION[case["precision"]],
             out_ptr=state["I"].data_ptr())
    if kind == "request":
        op.close()
    # the solve stops on a residual of 1e-6: its currents are handed on in single precision
    return state["I"].to(torch.complex64)


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------
_INFO = {}


def _info(case):
    """Sizes of the case's operator (ranks are found by the compression)."""
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _INFO:
        g = _request(case, 1)[0] if case["kind"] == "request" else _geometry(case)
        op = _operator(case, g, compress=case["kind"] in ("apply", "solve", "request"))
        _INFO[key] = dict(op.info(), n_voxels=g.n_atoms * case["nv"] ** 3)
        op.close()
    return _INFO[key]


def work(case):
    i, s, kind = _info(case), case["nrhs"], case["kind"]
    n, selfs, dense = i["n"], i["n_types"] * i["np"] ** 2, i["n_atoms"] * i["np"] ** 2
    cell = 16 if case.get("precision") in WIDE else 8
    if kind == "apply":
        fac = 16 if case["precision"] == "c128" else 8
        return {"bytes": fac * (i["stored_entries"] + selfs) + 2 * cell * n * s,
                "flops": 8 * (i["factor_entries"] + dense) * s}
    if kind == "precond":
        return {"bytes": cell * (selfs + 2 * n * s), "flops": 8 * dense * s}
    if kind == "rhs":
        # a plane wave factorises over the axes: one complex exponential product per unknown
        return {"bytes": 16 * n * s, "flops": 20 * n * s}
    if kind == "fields":
        # far field: directions x unknowns; near field: points x Gauss points (27 per voxel)
        ndirs = case["ndirs"] + 24 * 48
        return {"bytes": 3 * 16 * n * s + 48 * s * (case["npts"] + ndirs),
                "flops": s * (28 * ndirs * n + 100 * case["npts"] * 27 * i["n_voxels"])}
    # a solve: about fifty products (counted once, each with its share of the orthogonalisation)
    steps = 50
    flops = 8 * (i["factor_entries"] + dense) * s * steps + 16 * n * s * steps * steps // 2
    return {"bytes": steps * (8 * (i["stored_entries"] + selfs) + 16 * n * s) + 16 * n * s * steps * steps // 2,
            "flops": flops}


# ----------------------------------------------------------------------------
# the same results in 64 bits
# ----------------------------------------------------------------------------
def _gauss(q):
    """Gauss-Legendre nodes and weights on [0, 1]."""
    x, w = np.polynomial.legendre.leggauss(q)
    return 0.5 * (x + 1.0), 0.5 * w


class _Rooftops:
    """Rooftop basis of an nv^3-voxel cube with unit voxels, corner at the
    origin: the voxel below and above each face, and the charge sheet of a
    boundary face (include/vie.h has the ordering)."""

    def __init__(self, nv):
        self.nv = nv
        self.vox = np.array([(i, j, k) for i in range(nv) for j in range(nv) for k in range(nv)])
        num = lambda i: (i[0] * nv + i[1]) * nv + i[2]
        self.axis, self.lo, self.hi, self.sheet, corner = [], [], [], [], []
        for d in range(3):
            shape = [nv, nv, nv]
            shape[d] += 1
            for ijk in np.ndindex(*shape):
                below = list(ijk)
                below[d] -= 1
                self.axis.append(d)
                self.lo.append(num(below) if ijk[d] > 0 else -1)
                self.hi.append(num(ijk) if ijk[d] < nv else -1)
                edge = ijk[d] in (0, nv)
                self.sheet.append((len(corner), 1.0 if ijk[d] == 0 else -1.0) if edge else None)
                if edge:
                    corner.append((d, ijk))
        self.corner = corner
        self.np = len(self.axis)
        self.axis = np.array(self.axis)

    def voxel_points(self, q):
        """(nvox, q^3, 3) points, (q^3,) weights and (q^3, 3) local coordinates."""
        x, w = _gauss(q)
        xi = np.stack(np.meshgrid(x, x, x, indexing="ij"), -1).reshape(-1, 3)
        wt = np.einsum("i,j,k->ijk", w, w, w).ravel()
        return self.vox[:, None, :] + xi[None], wt, xi

    def sheet_points(self, q):
        """(nsheet, q^2, 3) points and (q^2,) weights of the boundary faces."""
        x, w = _gauss(q)
        ab = np.stack(np.meshgrid(x, x, indexing="ij"), -1).reshape(-1, 2)
        out = np.zeros((len(self.corner), q * q, 3))
        for s, (d, ijk) in enumerate(self.corner):
            out[s] = np.array(ijk, float)
            a, b = [e for e in range(3) if e != d]
            out[s, :, a] += ab[:, 0]
            out[s, :, b] += ab[:, 1]
        return out, np.outer(w, w).ravel()

    def currents(self, q):
        """Sparse map of the unknowns to point currents: for each axis d a matrix
        (np, nvox q^3) of w_f times the quadrature weight at the voxel points (h = 1)."""
        P, wt, xi = self.voxel_points(q)
        nq = len(wt)
        W = np.zeros((self.np, len(self.vox) * nq))
        for f in range(self.np):
            d = self.axis[f]
            if self.lo[f] >= 0:
                W[f, self.lo[f] * nq:(self.lo[f] + 1) * nq] = wt * xi[:, d]
            if self.hi[f] >= 0:
                W[f, self.hi[f] * nq:(self.hi[f] + 1) * nq] = wt * (1.0 - xi[:, d])
        return W

    def charges(self, q):
        """(np, nvox q^3) and (np, nsheet q'^2): charge times quadrature weight (h = 1)."""
        _, wt, _ = self.voxel_points(q)
        _, ws = self.sheet_points(q)
        nq, ns = len(wt), len(ws)
        V, S = np.zeros((self.np, len(self.vox) * nq)), np.zeros((self.np, len(self.corner) * ns))
        for f in range(self.np):
            if self.lo[f] >= 0:
                V[f, self.lo[f] * nq:(self.lo[f] + 1) * nq] = wt
            if self.hi[f] >= 0:
                V[f, self.hi[f] * nq:(self.hi[f] + 1) * nq] = -wt
            if self.sheet[f] is not None:
                s, sign = self.sheet[f]
                S[f, s * ns:(s + 1) * ns] = sign * ws
        return V, S


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _plane_waves(basis, g, vec, k):
    """T[w, a, f] = int w_f exp(j k vec_w . r) dV of atom a, for every vector w (64 bits)."""
    pts = basis.voxel_points(3)[0].reshape(-1, 3)
    W = _dev(basis.currents(3)).to(torch.complex128)
    out = torch.zeros((len(vec), g.n_atoms, basis.np), dtype=torch.complex128, device="cuda")
    v = _dev(vec)
    for t in range(len(g.sides)):
        h = g.sides[t] / basis.nv
        at = np.flatnonzero(g.types == t)
        if not len(at):
            continue
        # w_f = h^-2 profile, dV = h^3
        local = h * torch.exp(1j * k * h * (v @ _dev(pts).T)) @ W.T
        origin = torch.exp(1j * k * (v @ _dev(g.centres[at] - 0.5 * g.sides[t]).T))
        out[:, _dev(at)] = origin[:, :, None] * local[:, None, :]
    return out


def _exact_rhs(g, khat, pol):
    basis, k = _Rooftops(int(g.nvs[0])), 2.0 * np.pi / g.wavelength
    T = _plane_waves(basis, g, -np.asarray(khat), k)
    p = _dev(np.asarray(pol, complex))[:, _dev(basis.axis)]
    return (1j * k * T * p[:, None, :]).reshape(len(khat), -1)


def _exact_far(g, I, dirs):
    """F = -j k / (4 pi) (N - rhat (rhat . N)), (nrhs, ndirs, 3)."""
    basis, k = _Rooftops(int(g.nvs[0])), 2.0 * np.pi / g.wavelength
    cur = _dev(I.T).reshape(I.shape[1], g.n_atoms, basis.np)
    out = torch.zeros((I.shape[1], len(dirs), 3), dtype=torch.complex128, device="cuda")
    for i0 in range(0, len(dirs), 128):
        T = _plane_waves(basis, g, dirs[i0:i0 + 128], k)
        for d in range(3):
            sel = _dev(basis.axis == d)
            out[:, i0:i0 + 128, d] = torch.einsum("saf,waf->sw", cur[:, :, sel], T[:, :, sel])
    r = _dev(dirs).to(torch.complex128)
    return -1j * k / (4 * np.pi) * (out - r[None] * (out * r[None]).sum(-1, keepdim=True))


def _exact_near(g, I, points):
    """E = -j k int J g + (1 / (j k)) grad int q g, (nrhs, npts, 3)."""
    basis, k = _Rooftops(int(g.nvs[0])), 2.0 * np.pi / g.wavelength
    cur = _dev(I.T).reshape(I.shape[1], g.n_atoms, basis.np)
    W = _dev(basis.currents(3)).to(torch.complex128)
    V, S = (_dev(a).to(torch.complex128) for a in basis.charges(3))
    pv, ps = _dev(basis.voxel_points(3)[0].reshape(-1, 3)), _dev(basis.sheet_points(3)[0].reshape(-1, 3))
    r, E = _dev(points), torch.zeros((I.shape[1], len(points), 3), dtype=torch.complex128, device="cuda")
    for a in range(g.n_atoms):
        t = g.types[a]
        h = g.sides[t] / basis.nv
        o = _dev(g.centres[a] - 0.5 * g.sides[t])
        D = r[:, None, :] - (o + h * torch.cat([pv, ps]))[None]
        R = D.norm(dim=-1)
        G = torch.exp(-1j * k * R) / (4 * np.pi * R)
        # w_f = h^-2 profile; charges +-h^-3 in a voxel, +-h^-2 on a sheet
        c = cur[:, a]
        for d in range(3):
            sel = _dev(basis.axis == d)
            E[:, :, d] += -1j * k * h * (c[:, sel] @ W[sel]) @ G[:, :len(pv)].T
        q = c @ torch.cat([V, S], 1)
        K = -(1.0 + 1j * k * R) * G / R ** 2
        E += torch.einsum("sq,pq,pqd->spd", q, K, D.to(torch.complex128)) / (1j * k)
    return E


def _exact_fields(case, seed):
    g = _geometry(case)
    I = _currents(g.unknowns(), case["nrhs"], seed)
    khat, pol = workloads.random_directions(case["nrhs"], seed)
    x, w = np.polynomial.legendre.leggauss(24)
    ph = 2 * np.pi * np.arange(48) / 48
    st = np.sqrt(1 - x * x)
    sphere = np.stack([np.outer(st, np.cos(ph)), np.outer(st, np.sin(ph)), np.outer(x, np.ones(48))], -1).reshape(-1, 3)
    wt = np.repeat(w, 48) * (2 * np.pi / 48)
    F = _exact_far(g, I, sphere)
    sca = (F.abs() ** 2).sum(-1) @ _dev(wt)
    v0 = _exact_rhs(g, khat, pol) / (1j * 2 * np.pi / g.wavelength)
    ext = (_dev(I.T).conj() * v0).sum(-1).real
    return {"far": _exact_far(g, I, _directions(case["ndirs"], seed)),
            "near": _exact_near(g, I, _points(case["npts"], g, seed)), "sigma": torch.stack([ext, sca], 1)}


def _exact_product(case, seed):
    """The given factors and self blocks multiplied out in 64 bits (None where
    bringing the factors to the host takes too long)."""
    g = _geometry(case)
    op = _operator(case, g, compress=case["kind"] == "apply")
    info = op.info()
    if info["factor_entries"] > 150e6 or info["n_far_blocks"] > 8000:
        op.close()
        return None
    wide = case["precision"] in WIDE
    x = _vectors(op.n, case["nrhs"], wide, seed).to(torch.complex128).reshape(case["nrhs"], g.n_atoms, op.np)
    mode = case.get("mode", "precond")
    far = torch.zeros_like(x)
    if case["kind"] == "apply":
        for i in range(info["n_far_blocks"]):
            b = op.far_blocks(indices=[i])[0]
            t, s = _dev(b["tatoms"]).long(), _dev(b["satoms"]).long()
            Q, R = _dev(b["Q"]), _dev(b["R"])
            if mode == "adjoint":
                y = x[:, t].reshape(case["nrhs"], -1) @ Q.conj() @ R.conj()
                far[:, s] += y.reshape(case["nrhs"], len(s), op.np)
            else:
                y = x[:, s].reshape(case["nrhs"], -1) @ R.T @ Q.T
                far[:, t] += y.reshape(case["nrhs"], len(t), op.np)
    out = torch.zeros_like(x)
    for t in range(len(g.sides)):
        at = _dev(np.flatnonzero(g.types == t)).long()
        if not len(at):
            continue
        Z = _dev(op.export_block(0, t))
        if mode == "plain":
            out[:, at] = x[:, at] @ Z.T + far[:, at]
        elif mode == "adjoint":
            out[:, at] = x[:, at] @ Z.conj() + far[:, at]
        else:
            b = far[:, at] if mode == "fused" else x[:, at]
            y = torch.linalg.solve(Z, b.reshape(-1, op.np).T).T.reshape(b.shape)
            out[:, at] = x[:, at] + y if mode == "fused" else y
    op.close()
    return out.reshape(case["nrhs"], -1)


def _exact_currents(case, seed):
    """The dense system of the array (2-point rule between atoms, the given
    self blocks), solved in 64 bits; None above 8,000 unknowns."""
    if case["kind"] == "request":
        g, khat, pol = _request(case, seed)
    else:
        g = _geometry(case)
        khat, pol = workloads.random_directions(case["nrhs"], seed, max_deg=60.0)
    if g.unknowns() > 8000:
        return None
    basis, k = _Rooftops(int(g.nvs[0])), 2.0 * np.pi / g.wavelength
    W = _dev(basis.currents(2)).to(torch.complex128)
    C = torch.cat([_dev(a) for a in basis.charges(2)], 1).to(torch.complex128)
    pts = torch.cat([_dev(basis.voxel_points(2)[0].reshape(-1, 3)), _dev(basis.sheet_points(2)[0].reshape(-1, 3))])
    same = _dev(basis.axis[:, None] == basis.axis[None, :])
    nq, npf = W.shape[1], basis.np
    op = _operator(case, g, compress=False)
    Z = torch.zeros((g.n_atoms, npf, g.n_atoms, npf), dtype=torch.complex128, device="cuda")
    blocks = {}
    for a in range(g.n_atoms):
        for b in range(g.n_atoms):
            ta, tb = int(g.types[a]), int(g.types[b])
            if a == b:
                key = ("self", ta)
            else:
                key = (ta, tb) + tuple(np.round((g.centres[a] - g.centres[b]) * 1e9).astype(np.int64))
            if key not in blocks:
                ha, hb = g.sides[ta] / basis.nv, g.sides[tb] / basis.nv
                if a == b:
                    blocks[key] = _dev(op.export_block(0, ta))
                else:
                    oa, ob = (_dev(g.centres[c] - 0.5 * g.sides[g.types[c]]) for c in (a, b))
                    R = torch.cdist(oa + ha * pts, ob + hb * pts, compute_mode="donot_use_mm_for_euclid_dist")
                    G = torch.exp(-1j * k * R) / (4 * np.pi * R)
                    L = torch.where(same, ha * hb * (W @ G[:nq, :nq] @ W.T), 0)
                    blocks[key] = C @ G @ C.T - k * k * L
            Z[a, :, b, :] = blocks[key]
    op.close()
    n = g.n_atoms * npf
    return torch.linalg.solve(Z.reshape(n, n), _exact_rhs(g, khat, pol).T).T


def exact(case, seed):
    kind = case["kind"]
    if kind in ("apply", "precond"):
        return _exact_product(case, seed)
    if kind == "rhs":
        khat, pol = workloads.random_directions(case["nrhs"], seed, max_deg=60.0)
        return _exact_rhs(_geometry(case), khat, pol)
    if kind == "fields":
        return _exact_fields(case, seed)
    return _exact_currents(case, seed)
