"""The workloads this solver's speed is judged on, each run through the package's public entry points.

A case is a seismic wave-propagation set-up (mesh, material, order, relaxation mechanisms, time
clusters, simulations) and what one pass does with it:

* "advance": whole macro steps on the caller's stream, from DOFs that live in a device block the
  caller owns (the usual production loop; the pass returns that block's DOFs);
* "snapshot": set the DOFs from the host, advance, read all DOFs back (restart / snapshot output);
* "adjoint": misfit, material gradient, synthetic samples and initial-state gradient of an
  inversion step.

Meshes, materials and sources are those of this repository's generator (synth.py), configurations
and benchmark; initial wavefields are random modal fields from the seed with stresses, velocities
and memory variables in the ratios a wave of ~0.1 m/s has in rock. exact() is a plain FP64
evaluation of the same scheme in torch, by face quadrature instead of face matrices.
"""
import functools
import itertools
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2202_10313_gb300 import binding, synth

CFL = 0.5


def _advance(name, mesh, nx, ny, nz, order, mech, clusters, steps=1, fused=1, lam=0.8, receivers=0, sources=0):
    c = dict(kind="advance", mesh=mesh, nx=nx, ny=ny, nz=nz, order=order, mech=mech, clusters=clusters,
             steps=steps, fused=fused, lam=lam if clusters > 1 else 1.0, receivers=receivers, sources=sources)
    return dict(c, name=name) if name else c


def _other(kind, name, nx, ny, nz, order, clusters, steps, receivers, sources):
    return dict(_advance(name, "graded", nx, ny, nz, order, 0, clusters, steps, 1, 0.8, receivers, sources), kind=kind)


def listed():
    return [
        # the smallest call: one global step of the periodic verification cube (launch latency)
        _advance("cube_o3_gts_3k", "cube", 8, 8, 8, 3, 0, 1),
        # a tiny clustered problem with a source and receivers: many short phases per macro step
        _advance("box_o5_anelastic_360", "graded", 5, 4, 3, 5, 3, 3, receivers=4, sources=1),
        # order 3, anelastic: the cheap end of production runs, ragged size
        _advance("box_o3_anelastic_103k", "graded", 40, 33, 13, 3, 3, 4, receivers=16, sources=1),
        # order 4, elastic, odd sizes, several macro steps per call
        _advance("box_o4_elastic_39k", "graded", 31, 23, 9, 4, 0, 3, steps=4, receivers=16, sources=1),
        # order 4, anelastic, layer over a half-space (the verification benchmark's model)
        _advance("layer_o4_anelastic_111k", "layer", 34, 34, 16, 4, 3, 3, receivers=9, sources=1),
        # order 5, anelastic, global time stepping on a mid-size mesh
        _advance("box_o5_anelastic_gts_35k", "graded", 24, 24, 10, 5, 3, 1, steps=4, receivers=64, sources=1),
        # order 5, elastic, four clusters
        _advance("box_o5_elastic_192k", "graded", 40, 40, 20, 5, 0, 4, receivers=64, sources=1),
        # the headline workload at half the benchmark's mesh: order 5, anelastic, clustered
        _advance("box_o5_anelastic_1051k", "graded", 96, 96, 19, 5, 3, 5, receivers=64, sources=1),
        # fused simulations: 16 sources over one mesh, order 5, anelastic
        _advance("fused16_o5_anelastic_15k", "graded", 16, 16, 10, 5, 3, 4, fused=16, sources=16),
        # fused simulations: 4 sources, order 4, elastic, odd sizes
        _advance("fused4_o4_elastic_22k", "graded", 21, 19, 9, 4, 0, 3, steps=2, fused=4, receivers=8, sources=4),
        # restart / snapshot output: DOFs in from the host and out to it
        _other("snapshot", "snapshot_o4_elastic_20k", 21, 20, 8, 4, 2, 1, 8, 1),
        # one inversion step: misfit and gradients, order 4, elastic, clustered
        _other("adjoint", "adjoint_o4_elastic_47k", 28, 28, 10, 4, 2, 32, 16, 1),
    ]


def draw(rng):
    kind = rng.choice(["advance"] * 6 + ["snapshot", "adjoint"])
    order = rng.choice([3, 4, 5])
    # elements (times simulations), spread over the logarithm of the range
    if kind == "adjoint":
        nel, mech, fused = math.exp(rng.uniform(math.log(500), math.log(30000))), 0, 1
    elif kind == "snapshot":
        nel, mech, fused = math.exp(rng.uniform(math.log(200), math.log(40000))), 0, 1
    else:
        nel = math.exp(rng.uniform(math.log(150), math.log({3: 900e3, 4: 700e3, 5: 500e3}[order])))
        mech = rng.choice([0, 3, 3])
        fused = rng.choice([1, 1, 1, 4, 8, 16]) if nel > 5000 else 1
    nel /= fused
    clusters = rng.choice([1, 2, 3, 4, 5])
    if kind != "advance":
        clusters = min(clusters, 3)
    nz = max(3, min(24, int(round((nel / 6.0) ** (1.0 / 3.0) * rng.uniform(0.4, 0.9)))))
    nx = max(3, int(round(math.sqrt(nel / 6.0 / nz) * rng.uniform(0.8, 1.25))))
    ny = max(3, int(round(nel / 6.0 / nz / nx)))
    steps = 1 if nel * fused > 100e3 else rng.choice([1, 2, 3])
    receivers, sources = rng.choice([1, 8, 16, 64]), max(1, fused if fused > 1 else rng.choice([1, 2]))
    if kind == "adjoint":
        # finest steps of one sweep, as whole macro steps
        steps = max(2, rng.choice([12, 24, 40]) >> (clusters - 1))
    mesh = rng.choice(["graded", "graded", "layer"]) if kind == "advance" and nz >= 9 else "graded"
    return dict(_advance(None, mesh, nx, ny, nz, order, mech, clusters, steps, fused, rng.choice([0.7, 0.8, 0.9]),
                         receivers, sources), kind=kind)


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=3)
def _setting(kind, nx, ny, nz, mech):
    """Mesh and material (fixed by the case)."""
    if kind == "cube":
        mesh = synth.periodic_cube(nx)
        mat = synth.homogeneous(mesh["tet"].shape[0])
    elif kind == "layer":
        mesh = synth.permute_vertex_order(synth.layer_over_halfspace(nx, ny, 250.0, hz_layer=125.0, nz_below=nz - 8))
        mat = synth.loh3_materials(mesh)
    else:
        mesh = synth.permute_vertex_order(synth.graded_box(nx, ny, nz, 250.0, 125.0))
        mat = synth.random_layers(mesh)
    if not mech:
        mat = {k: mat[k] for k in ("rho", "vp", "vs")}
    return mesh, mat


def _case_setting(case):
    return _setting(case["mesh"], case["nx"], case["ny"], case["nz"], case["mech"])


def _points(case, seed):
    """Point sources and receivers of the case."""
    mesh, _ = _case_setting(case)
    rng = np.random.default_rng([seed, 17])
    lo, hi = mesh["xyz"].min(axis=0), mesh["xyz"].max(axis=0)
    fixed = np.random.default_rng(5)                     # positions belong to the case, the signals to the seed
    at = lo + (hi - lo) * (0.2 + 0.6 * fixed.random((case["sources"], 3)))
    m6 = rng.normal(size=(case["sources"], 6))
    m6 /= np.linalg.norm(m6, axis=1, keepdims=True)
    src = [dict(x=at[i], m6=m6[i], f0=float(rng.uniform(1.0, 4.0)), t0=0.0, m0=1e13,
                sim=i if case["fused"] > 1 else 0) for i in range(case["sources"])]
    n = int(math.ceil(math.sqrt(case["receivers"])))
    rec = synth.surface_receiver_grid(n, n, (lo[0], hi[0]), (lo[1], hi[1]))[:case["receivers"]] if n else []
    return src, rec


def _sizes(case):
    o = case["order"]
    return o * (o + 1) * (o + 2) // 6, o * (o + 1) // 2, 9 + 6 * case["mech"]


def _initial(case, seed, n_elem):
    """Random modal wavefield (F, K, NQ, B), FP32, the same on every call with this seed."""
    nb, _, nq = _sizes(case)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) * 7919 + 11)
    q = torch.empty(case["fused"], n_elem, nq, nb, device=dev)
    q.normal_(generator=gen)
    q *= (0.5 ** (4.0 * torch.arange(nb, device=dev) / nb))
    q *= torch.tensor([1e6] * 6 + [0.1] * 3 + [4e-4] * (nq - 9), device=dev)[:, None]
    return q


def _observed(case, seed):
    """Recorded velocities an inversion compares with (sample time, receiver, component)."""
    rng = np.random.default_rng([seed, 23])
    return 0.1 * rng.normal(size=(case["steps"] + 1, case["receivers"], 3))


def _split(q, rows):
    """Stresses, velocities and memory variables apart (they differ by orders of magnitude)."""
    out = dict(stress=q.narrow(rows, 0, 6), velocity=q.narrow(rows, 6, 3))
    if q.shape[rows] > 9:
        out["memory"] = q.narrow(rows, 9, q.shape[rows] - 9)
    return out


def prepare(case, seed):
    mesh, mat = _case_setting(case)
    nb, _, nq = _sizes(case)
    n, F = mesh["tet"].shape[0], case["fused"]
    s = binding.Solver(case["order"], case["mech"], device=0, n_fused=F)
    s.set_mesh(mesh["xyz"], mesh["tet"], mesh["face_bc"], mesh["period"])
    s.set_material(mat["rho"], mat["vp"], mat["vs"], mat.get("qp"), mat.get("qs"))
    src, rec = _points(case, seed)
    for p in src:
        s.add_point_source(p["x"], p["m6"], p["f0"], p["t0"], p["m0"], p["sim"])
    for x in rec:
        s.add_receiver(x, 0.01)
    s.use_torch_memory(case["clusters"])
    cl, _, _ = s.setup_clusters(case["clusters"], CFL, case["lam"])
    state = dict(case=case, solver=s, finest=case["steps"] * 2 ** (case["clusters"] - 1))
    q0 = _initial(case, seed, n)
    if case["kind"] == "snapshot":
        state["dofs"] = q0[0].cpu().numpy().astype(np.float64)
        return state
    # the DOFs are the first array of the caller's block: FP32, elements in cluster order, rows
    # padded to 16 bytes (fused: simulations innermost in groups of four)
    order = torch.from_numpy(np.argsort(cl, kind="stable")).to(q0.device)
    off = (-s._mem.data_ptr()) % 256
    if F == 1:
        qs = (nq * nb + 3) // 4 * 4
        flat = s._mem[off:off + 4 * n * qs].view(torch.float32).view(n, qs)
        q = flat[:, :nq * nb].unflatten(1, (nq, nb))
        q.copy_(q0[0][order])
    else:
        flat = s._mem[off:off + 4 * n * nq * nb * F].view(torch.float32)
        q = flat.view(n, F // 4, nq, nb, 4)
        q.copy_(q0[:, order].view(F // 4, 4, n, nq, nb).permute(2, 0, 3, 4, 1))
    state["rows"] = 1 if F == 1 else 2
    state["q"] = q
    if case["kind"] == "adjoint":
        state["data"] = _observed(case, seed)
    return state


def run(state):
    s = state["solver"]
    kind = state["case"]["kind"]
    if kind == "adjoint":
        J, grad, syn, dq0 = s.misfit_gradient(state["finest"], state["data"], want_dq0=True)
        # FP32 values in FP64 arrays: kept as FP32
        g = torch.from_numpy(grad.astype(np.float32))
        return dict(misfit=np.float32(J), rho=g[:, 0], lam=g[:, 1], mu=g[:, 2], samples=syn.astype(np.float32),
                    **_split(torch.from_numpy(dq0.astype(np.float32)), 1))
    if kind == "snapshot":
        s.set_dofs(state["dofs"])
        s.advance_steps(state["finest"])
        return _split(torch.from_numpy(s.get_dofs().astype(np.float32)), 1)
    s.advance_steps(state["finest"])
    return _split(state["q"], state["rows"])


# ------------------------------------------------------------------ work
@functools.lru_cache(maxsize=8)
def _nonzeros(order, mech):
    """Nonzeros of the three K_c summed over the derivatives (elastic: derivative d has degree
    order - 1 - d, anelastic: every mode) and the volume product, and of the four face matrices."""
    K, ft = _operators(order)[0], _face_matrices(order)
    on = np.abs(K) > 1e-7 * np.abs(K).max()
    size = [o * (o + 1) * (o + 2) // 6 for o in range(order + 1)]
    nk = on.sum()
    for d in range(order - 1):
        nk += on[:, :size[order - 1 - d], :size[order - d]].sum() if mech == 0 else on.sum()
    return int(nk), int((np.abs(ft) > 1e-7 * np.abs(ft).max()).sum())


@functools.lru_cache(maxsize=16)
def _updates(kind, nx, ny, nz, mech, order, clusters, lam):
    mesh, mat = _setting(kind, nx, ny, nz, mech)
    cl, _ = _clusters(_geometry(kind, nx, ny, nz, mech), mat["vp"], order, clusters, lam)
    return int(np.sum(2 ** (clusters - 1 - cl))), len(cl)


def work(case):
    nb, nf, nq = _sizes(case)
    o, m = case["order"], case["mech"]
    per_macro, n = _updates(case["mesh"], case["nx"], case["ny"], case["nz"], m, o, case["clusters"], case["lam"])
    nk, nft = _nonzeros(o, m)
    # an update: the derivatives and the volume product (three velocity gradients and three stress
    # divergences: 6 nonzeros' worth), traces and projections of 6 rows (velocity and traction), one star
    # application per derivative and per update, the relaxation of 6 m rows per derivative
    flops = 2 * (6 * nk + 2 * 6 * nft) + nb * o * (2 * 54 + 16 + 36 + 40 * m)
    # the DOFs in and out of every update, the time-integrated face states across every face
    upd_bytes = 4 * (2 * nq * nb + 4 * 6 * nf + 44)
    F, steps = case["fused"], case["steps"]
    fac = 1
    if case["kind"] == "adjoint":
        fac = 3                                          # the forward sweep, its states once more, the transpose
    w = dict(bytes=float(fac * F * steps * per_macro * upd_bytes), flops=float(fac * F * steps * per_macro * flops))
    if case["kind"] == "snapshot":
        w["bytes"] += 2.0 * 12 * n * nq * nb             # FP64 on the host, FP32 on the device, both ways
    return w


# ------------------------------------------------------------------ FP64 evaluation of the scheme
_FACES = ((0, 2, 1), (0, 1, 3), (0, 3, 2), (1, 2, 3))
_REF = np.array([[0.0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]])


def _jacobi(n, a, x):
    """P_n^(a,0)(x) by the three-term recurrence."""
    p0, p1 = np.ones_like(x), 0.5 * ((a + 2.0) * x + a)
    if n == 0:
        return p0
    for k in range(2, n + 1):
        c = 2.0 * k + a
        p0, p1 = p1, ((c - 1.0) * (c * (c - 2.0) * x + a * a) * p1 - 2.0 * (k + a - 1.0) * (k - 1.0) * c * p0) / (
            2.0 * k * (k + a) * (c - 2.0))
    return p1


def _modes(order):
    return [(d - k - j, j, k) for d in range(order) for k in range(d + 1) for j in range(d - k + 1)]


def _tet_rule(n):
    """Collapsed Gauss-Legendre rule of the reference tetrahedron."""
    g, w = np.polynomial.legendre.leggauss(n)
    g, w = 0.5 * (g + 1.0), 0.5 * w
    A, Bq, C = np.meshgrid(g, g, g, indexing="ij")
    W = np.einsum("i,j,k->ijk", w, w, w) * (1 - Bq) * (1 - C) ** 2
    return np.stack([A * (1 - Bq) * (1 - C), Bq * (1 - C), C], axis=-1).reshape(-1, 3), W.ravel()


def _tri_rule(n):
    g, w = np.polynomial.legendre.leggauss(n)
    g, w = 0.5 * (g + 1.0), 0.5 * w
    A, Bq = np.meshgrid(g, g, indexing="ij")
    return np.stack([A * (1 - Bq), Bq], axis=-1).reshape(-1, 2), (np.outer(w, w) * (1 - Bq)).ravel()


def _raw(order, x):
    s1, s2 = 1.0 - x[:, 1] - x[:, 2], 1.0 - x[:, 2]
    a, b, c = 2.0 * x[:, 0] / s1 - 1.0, 2.0 * x[:, 1] / s2 - 1.0, 2.0 * x[:, 2] - 1.0
    return np.stack([s1 ** i * _jacobi(i, 0.0, a) * s2 ** j * _jacobi(j, 2.0 * i + 1.0, b) * _jacobi(k, 2.0 * (i + j) + 2.0, c)
                     for i, j, k in _modes(order)], axis=1)


def _mono(order, x, diff=None):
    cols = []
    for i, j, k in _modes(order):
        e, f = [i, j, k], 1.0
        if diff is not None:
            f, e[diff] = float(e[diff]), max(e[diff] - 1, 0)
        cols.append(f * x[:, 0] ** e[0] * x[:, 1] ** e[1] * x[:, 2] ** e[2])
    return np.stack(cols, axis=1)


@functools.lru_cache(maxsize=8)
def _operators(order):
    """K_c, the basis as monomial coefficients, and the face rule."""
    x, w = _tet_rule(order + 2)
    v = _raw(order, x)
    v = v / np.sqrt((w[:, None] * v ** 2).sum(axis=0))
    coef = np.linalg.lstsq(_mono(order, x), v, rcond=None)[0]
    K = np.stack([(v * w[:, None]).T @ (_mono(order, x, c) @ coef) for c in range(3)])
    return K, coef, _tri_rule(order + 1)


def _phi(order, x):
    return _mono(order, x) @ _operators(order)[1]


@functools.lru_cache(maxsize=8)
def _face_matrices(order):
    """int_face phi_k psi_m, with the face basis from an orthonormalisation of the triangle's modes."""
    t, w = _operators(order)[2]
    s = 1.0 - t[:, 1]
    psi = np.stack([s ** i * _jacobi(i, 0.0, 2.0 * t[:, 0] / s - 1.0) * _jacobi(j, 2.0 * i + 1.0, 2.0 * t[:, 1] - 1.0)
                    for d in range(order) for j in range(d + 1) for i in [d - j]], axis=1)
    psi = psi / np.sqrt((w[:, None] * psi ** 2).sum(axis=0))
    bary = np.stack([1.0 - t.sum(axis=1), t[:, 0], t[:, 1]], axis=1)
    return np.stack([_phi(order, bary @ _REF[list(f)]).T @ (psi * w[:, None]) for f in _FACES])


@functools.lru_cache(maxsize=3)
def _geometry(kind, nx, ny, nz, mech):
    mesh, _ = _setting(kind, nx, ny, nz, mech)
    xyz, tet = mesh["xyz"], mesh["tet"]
    x = xyz[tet]
    J = np.stack([x[:, i] - x[:, 0] for i in (1, 2, 3)], axis=2)        # dx/dxi
    det, Jinv = np.linalg.det(J), np.linalg.inv(J)
    fv = np.array(_FACES)
    a, b, c = (x[:, fv[:, i]] for i in range(3))
    cr = np.cross(b - a, c - a)
    area = 0.5 * np.linalg.norm(cr, axis=2)
    normal = cr / (2.0 * area[..., None])
    ids = np.arange(len(xyz))
    if mesh["period"] is not None:
        key = np.round((xyz / mesh["period"] % 1.0) * 1e6).astype(np.int64) % 1000000
        ids = np.unique(key, axis=0, return_inverse=True)[1].ravel()
    vid = ids[tet]                                                      # (K, 4)
    trip = np.sort(vid[:, fv], axis=2).reshape(-1, 3)
    o = np.lexsort(trip.T[::-1])
    same = (trip[o][1:] == trip[o][:-1]).all(axis=1)
    i0, i1 = o[:-1][same], o[1:][same]
    nbr = np.full(4 * len(tet), -1, dtype=np.int64)
    nbr[i0], nbr[i1] = i1 // 4, i0 // 4
    nbr = nbr.reshape(-1, 4)
    # where the local face's vertices sit among the neighbour's
    vn = vid[np.maximum(nbr, 0)]                                        # (K, 4 faces, 4)
    pos = (vid[:, fv][..., None] == vn[:, :, None, :]).argmax(axis=3)  # (K, 4, 3)
    code = pos[..., 0] * 16 + pos[..., 1] * 4 + pos[..., 2]
    return dict(x0=x[:, 0], det=det, Jinv=Jinv, area=area, normal=normal, nbr=nbr, code=code, din=det / area.sum(axis=1),
                bc=np.asarray(mesh["face_bc"]))


def _clusters(geo, vp, order, clusters, lam):
    dt = CFL * geo["din"] / ((2.0 * order - 1.0) * vp)
    base = lam * dt.min()
    c = np.zeros(len(dt), dtype=np.int64)
    for l in range(1, clusters):
        c += dt >= base * 2.0 ** l
    nbr = geo["nbr"]
    while True:
        n = np.minimum(c, np.where(nbr >= 0, c[np.maximum(nbr, 0)] + 1, c[:, None]).min(axis=1))
        if (n == c).all():
            return c, base
        c = n


def _fit(q, omega):
    """Y_l of a constant quality factor by collocation at the relaxation frequencies."""
    wk, wl = omega[:, None], omega[None, :]
    qi = 1.0 / q
    M = (wl * wk + wl ** 2 * qi[:, None, None]) / (wl ** 2 + wk ** 2)
    return np.linalg.solve(M, np.repeat(qi[:, None, None], len(omega), axis=1))[..., 0]


_SIG = ((0, 3, 5), (3, 1, 4), (5, 4, 2))
_CHUNK = 1 << 16


class _Exact:
    """The clustered scheme in FP64, elements in the caller's order, one simulation."""

    def __init__(self, case, rho, lam, mu):
        self.case, self.o = case, case["order"]
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.geo = _geometry(case["mesh"], case["nx"], case["ny"], case["nz"], case["mech"])
        _, mat = _case_setting(case)
        t = self.t
        self.cl, self.delta = _clusters(self.geo, mat["vp"], self.o, case["clusters"], case["lam"])
        self.rho, self.lam, self.mu = rho, lam, mu
        K, _, (tri, w) = _operators(self.o)
        self.K = t(K)
        bary = np.stack([1.0 - tri.sum(axis=1), tri[:, 0], tri[:, 1]], axis=1)
        self.E = [t(_phi(self.o, bary @ _REF[list(f)])) for f in _FACES]
        self.w = t(w)
        self.Enb = {}
        for p in itertools.permutations(range(4), 3):
            self.Enb[p[0] * 16 + p[1] * 4 + p[2]] = t(_phi(self.o, bary @ _REF[list(p)]))
        for k in ("Jinv", "area", "normal", "det"):
            setattr(self, k, t(self.geo[k]))
        self.nbr = torch.from_numpy(self.geo["nbr"]).to(self.dev)
        self.m = case["mech"]
        if self.m:
            om = 2.0 * np.pi * 0.1 * 50.0 ** (np.arange(self.m) / (self.m - 1.0))
            ys, yp = _fit(mat["qs"], om), _fit(mat["qp"], om)
            l, u = lam.cpu().numpy()[:, None], mu.cpu().numpy()[:, None]
            self.om, self.yl, self.yu = om, t((l + 2 * u) * yp - 2 * u * ys), t(2 * u * ys)   # lam Y^lam, 2 mu Y^mu
        idx = [np.nonzero(self.cl == l)[0] for l in range(case["clusters"])]
        self.idx = [torch.from_numpy(i).to(self.dev) for i in idx]
        # per cluster, face and orientation: positions (in the cluster) of the elements with such a neighbour
        self.groups = []
        for i in idx:
            g = []
            for f in range(4):
                nb, code = self.geo["nbr"][i, f], self.geo["code"][i, f]
                for cd in np.unique(code[nb >= 0]):
                    g.append((f, int(cd), torch.from_numpy(np.nonzero((nb >= 0) & (code == cd))[0]).to(self.dev)))
            self.groups.append(g)

    def t(self, a):
        return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).to(self.dev)

    def star(self, Y, e):
        """sum_d A_d-like combination of (n, 3, 9, B): C : sym grad v, div sigma / rho, sym grad v."""
        W = torch.einsum("ncd,ncrb->ndrb", self.Jinv[e], Y)
        g = [[W[:, d, 6 + j] for j in range(3)] for d in range(3)]
        div = [sum(W[:, d, _SIG[i][d]] for d in range(3)) / self.rho[e][:, None] for i in range(3)]
        return self.hooke(g, e, div)

    def hooke(self, g, e, div):
        lam, mu = self.lam[e][:, None], self.mu[e][:, None]
        eps = [g[0][0], g[1][1], g[2][2], 0.5 * (g[0][1] + g[1][0]), 0.5 * (g[1][2] + g[2][1]), 0.5 * (g[0][2] + g[2][0])]
        tr = eps[0] + eps[1] + eps[2]
        out = [lam * tr + 2 * mu * eps[i] for i in range(3)] + [2 * mu * eps[i] for i in range(3, 6)] + list(div)
        return torch.stack(out, dim=1), torch.stack(eps, dim=1)

    def couple(self, th, e):
        """E^l theta^l summed over the mechanisms: stress rows (n, 6, B)."""
        s = 0.0
        for l in range(self.m):
            x = th[:, 6 * l:6 * l + 6]
            tr = x[:, :3].sum(dim=1, keepdim=True)
            y = -self.yu[e][:, l, None, None] * x
            s = s + torch.cat([y[:, :3] - self.yl[e][:, l, None, None] * tr, y[:, 3:]], dim=1)
        return s

    def predict(self, Q, e, dt):
        """T over dt and the elastic rows of T over dt/2; Q of elements e plus volume and local surface terms."""
        D, T, Th = Q, 0.0, 0.0
        for d in range(self.o):
            f = math.factorial(d + 1)
            T = T + dt ** (d + 1) / f * D
            Th = Th + (0.5 * dt) ** (d + 1) / f * D[:, :9]
            if d == self.o - 1:
                break
            out, eps = self.star(torch.einsum("cbk,nrk->ncrb", self.K, D[:, :9]), e)
            if self.m:
                out = torch.cat([out[:, :6] + self.couple(D[:, 9:], e), out[:, 6:]], dim=1)
                out = torch.cat([out] + [self.om[l] * (eps - D[:, 9 + 6 * l:15 + 6 * l]) for l in range(self.m)], dim=1)
            D = out
        Te = T[:, :9]
        out, eps = self.star(torch.einsum("ckb,nrk->ncrb", self.K, Te), e)
        V = -out
        if self.m:
            V = torch.cat([V[:, :6] + self.couple(T[:, 9:], e), V[:, 6:]], dim=1)
            V = torch.cat([V] + [self.om[l] * (-eps - T[:, 9 + 6 * l:15 + 6 * l]) for l in range(self.m)], dim=1)
        Q = Q + V
        for i in range(4):
            Q = Q + self.flux(Te @ self.E[i].T, e, i, True)
        return Q, Te, Th

    def flux(self, g, e, i, inner):
        """Contribution of one side's face states g (n, 9, points) to the DOFs of elements e, face i."""
        n = self.normal[e, i]
        nb, bc = self.nbr[e, i], torch.from_numpy(self.geo["bc"]).to(self.dev)[e, i]
        zi = [torch.sqrt((self.lam + 2 * self.mu) * self.rho), torch.sqrt(self.mu * self.rho)]
        has = (nb >= 0)[:, None, None]
        tr = torch.stack([sum(g[:, _SIG[a][d]] * n[:, d, None] for d in range(3)) for a in range(3)], dim=1)
        v = g[:, 6:9]
        N = n[:, :, None]
        tn, vn = (tr * N).sum(1, keepdim=True) * N, (v * N).sum(1, keepdim=True) * N
        vs, ts = 0.0, 0.0
        for z, tq, vq in ((zi[0], tn, vn), (zi[1], tr - tn, v - vn)):
            zm = z[e][:, None, None]
            zp = torch.where(has, z[nb.clamp(min=0)][:, None, None], zm)
            if inner:
                free = (bc == 2)[:, None, None]
                vs = vs + torch.where(free, vq - tq / zm, (zm * vq - tq) / (zm + zp))
                ts = ts + torch.where(free, torch.zeros_like(tq), (zp * tq - zm * zp * vq) / (zm + zp))
            else:
                vs = vs + (zp * vq + tq) / (zm + zp)
                ts = ts + (zm * tq + zm * zp * vq) / (zm + zp)
        grad = [[n[:, d, None] * vs[:, j] for j in range(3)] for d in range(3)]
        out, eps = self.hooke(grad, e, [ts[:, a] / self.rho[e][:, None] for a in range(3)])
        if self.m:
            out = torch.cat([out] + [self.om[l] * eps for l in range(self.m)], dim=1)
        s = (2.0 * self.area[e, i] / self.det[e])[:, None, None]
        return s * ((out * self.w) @ self.E[i])

    def macro(self, Q, s0, sources):
        """One macro step from finest step s0 (Q not modified in place)."""
        nc = self.case["clusters"]
        n, nb = Q.shape[0], Q.shape[2]
        B1, B2, B3 = (torch.zeros(n, 9, nb, dtype=Q.dtype, device=Q.device) for _ in range(3))
        cl = torch.from_numpy(self.cl).to(self.dev)
        for s in range(s0, s0 + 2 ** (nc - 1) + 1):
            for l in range(nc):
                if s == s0 or s % 2 ** l:
                    continue
                k = s // 2 ** l - 1
                e = self.idx[l]
                add = torch.zeros(len(e), Q.shape[1], nb, dtype=Q.dtype, device=Q.device)
                for f, code, pos in self.groups[l]:
                    for p in pos.split(_CHUNK):
                        ee = e[p]
                        nbr = self.nbr[ee, f]
                        rel = (cl[nbr] - l)[:, None, None]
                        x = torch.where(rel == 0, B1[nbr], torch.where(rel < 0, B3[nbr], B2[nbr] if k % 2 == 0 else B1[nbr] - B2[nbr]))
                        add = add.index_add(0, p, self.flux(x @ self.Enb[code].T, ee, f, False))
                Q = Q.index_add(0, e, add)
                for src in sources:
                    if self.cl[src["elem"]] == l:
                        amp = src["m6"] * (-src["m0"] * self.ricker(src, k * 2 ** l, (k + 1) * 2 ** l) / float(self.det[src["elem"]]))
                        inc = torch.zeros_like(Q[0])
                        inc[:6] = amp[:, None] * src["phi"][None, :]
                        Q = Q.index_add(0, torch.tensor([src["elem"]], device=self.dev), inc[None])
            if s == s0 + 2 ** (nc - 1):
                break
            for l in range(nc):
                if s % 2 ** l:
                    continue
                k = s // 2 ** l
                parts = []
                for e in self.idx[l].split(_CHUNK):
                    parts.append(self.predict(Q[e], e, self.delta * 2.0 ** l))
                if not parts:
                    continue
                e = self.idx[l]
                q, te, th = (torch.cat([p[j] for p in parts]) for j in range(3))
                Q, B1, B2 = Q.index_copy(0, e, q), B1.index_copy(0, e, te), B2.index_copy(0, e, th)
                B3 = B3.index_copy(0, e, te if k % 2 == 0 else B3[e] + te)
        return Q

    def ricker(self, src, a, b):
        gx, gw = np.polynomial.legendre.leggauss(self.o)
        t = self.delta * (0.5 * (a + b) + 0.5 * (b - a) * gx)
        u = (np.pi * src["f0"] * (t - src["t0"])) ** 2
        return 0.5 * (b - a) * self.delta * float(np.sum(gw * (1.0 - 2.0 * u) * np.exp(-u)))

    def place(self, x):
        """Lowest element that holds x, and the basis there."""
        xi = np.einsum("kcd,kd->kc", self.geo["Jinv"], np.asarray(x)[None] - self.geo["x0"])
        k = int(np.nonzero((xi.min(axis=1) >= -1e-12) & (xi.sum(axis=1) <= 1.0 + 1e-12))[0][0])
        return k, self.t(_phi(self.o, xi[k][None])[0])


def exact(case, seed):
    mesh, mat = _case_setting(case)
    n, F = mesh["tet"].shape[0], case["fused"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    rho, vp, vs = (torch.from_numpy(np.asarray(mat[k], dtype=np.float64)).to(dev) for k in ("rho", "vp", "vs"))
    mu = rho * vs * vs
    lam = rho * vp * vp - 2.0 * mu
    adj = case["kind"] == "adjoint"
    if adj:
        for p in (rho, lam, mu):
            p.requires_grad_(True)
    with torch.set_grad_enabled(adj):
        ex = _Exact(case, rho, lam, mu)
        src, rec = _points(case, seed)
        for p in src:
            p["elem"], p["phi"] = ex.place(p["x"])
            p["m6"] = ex.t(p["m6"])
        q0 = _initial(case, seed, n).double()
        period = 2 ** (case["clusters"] - 1)
        if not adj:
            order = torch.from_numpy(np.argsort(ex.cl, kind="stable")).to(dev)
            nb, _, nq = _sizes(case)
            sims = []
            for f in range(F):
                Q = q0[f]
                for m in range(case["steps"]):
                    Q = ex.macro(Q, m * period, [p for p in src if p["sim"] == f])
                sims.append(Q if case["kind"] == "snapshot" else Q[order])
            if F == 1:
                return _split(sims[0], 1)
            return _split(torch.stack(sims).view(F // 4, 4, n, nq, nb).permute(2, 0, 3, 4, 1), 2)
        Q = q0[0].requires_grad_(True)
        first = Q
        at = [ex.place(x) for x in rec]
        pe = torch.tensor([k for k, _ in at], device=dev)
        ph = torch.stack([p for _, p in at])
        sample = lambda q: torch.einsum("rcb,rb->rc", q[pe, 6:9], ph)  # noqa: E731
        syn = [sample(Q)]
        for m in range(case["steps"]):
            Q = checkpoint(ex.macro, Q, m * period, src, use_reentrant=False)
            syn.append(sample(Q))
        syn = torch.stack(syn)
        J = 0.5 * ((syn - ex.t(_observed(case, seed))) ** 2).sum()
        J.backward()
        return dict(misfit=float(J.detach()), rho=rho.grad, lam=lam.grad, mu=mu.grad, samples=syn.detach(), **_split(first.grad, 1))
