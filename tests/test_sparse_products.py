"""The generated sparse products of the predict kernel (contraction engine 'sparse') take
exactly the nonzero entries of the stiffness matrices K_c and of the face matrices F~_i
and of their transposes F^_i (Sec. III-A), and so do the products of the adjoint's reverse
predict pass, with values equal to the oracle's independently
built operators to FP32 rounding, and no term the oracle has is dropped. The generator lists every product term
(kind, part, output, k, value) it writes into the kernel."""
import os
import subprocess

import numpy as np
import pytest

from oracle.basis import Basis
from paper_2202_10313_gb300 import build


def _terms(order):
    build.build()
    exe = os.path.join(build.OUT_DIR, "gen_sparse")
    out = subprocess.run([exe, "--list", str(order)], capture_output=True, text=True, check=True).stdout
    rows = [l.split() for l in out.splitlines() if l.strip()]
    return [(r[0], int(r[1]), int(r[2]), int(r[3]), float(r[4])) for r in rows]


@pytest.mark.parametrize("order", [3, 4, 5])
def test_generated_terms_are_the_oracle_operators_nonzeros(order):
    ob = Basis(order)
    B = len(ob.K[0])
    F = ob.Ft[0].shape[1]
    terms = _terms(order)
    kmax = max(np.abs(k).max() for k in ob.K)
    fmax = max(np.abs(f).max() for f in ob.Ft)
    # the dense matrix each kind of product applies: time X K_c^T (out (c, b), sum over k of
    # K_c[b][k]); volume X K_c (K_c[k][b]); face traces X F~_i (F~_i[k][f])
    want = {"t": np.stack([ob.K[c] for c in range(3)]).reshape(3 * B, B),
            "v": np.stack([ob.K[c].T for c in range(3)]).reshape(3 * B, B),
            "g": np.stack([ob.Ft[i].T for i in range(4)]).reshape(4 * F, B)}
    # face projection: out (i, b) from the inputs (i, f), F^_i[f][b] = int psi_f phi_b = F~_i[b][f]
    proj = np.zeros((4 * B, 4 * F))
    for i in range(4):
        proj[i * B:(i + 1) * B, i * F:(i + 1) * F] = ob.Fh[i].T
    want["p"] = proj
    want["n"] = np.stack([ob.Ft[j].T for j in range(4)]).reshape(4 * F, B)
    # adjoint products: the four faces' transposed traces summed, out b from the inputs
    # (i, f), F~_i[b][f]; the reverse time kernel X K_c (as the volume kernel)
    want["s"] = np.concatenate([ob.Ft[i] for i in range(4)], axis=1)
    want["k"] = want["v"]
    scale = {"t": kmax, "v": kmax, "g": fmax, "p": fmax, "n": fmax, "s": fmax, "k": kmax}
    got = {k: np.zeros_like(v) for k, v in want.items()}
    part_of = {}
    for kind, part, o, k, val in terms:
        assert got[kind][o, k] == 0.0, "term listed twice"
        got[kind][o, k] = val
        assert part_of.setdefault((kind, o), part) == part, "output split over parts"
    for kind in want:
        w, g = want[kind], got[kind]
        if kind == "t":       # the kernel's full time variant writes outputs of degree <= O-2
            w = w.copy()
            nb1 = (order - 1) * order * (order + 1) // 6
            for c in range(3):
                assert np.abs(w[c * B + nb1:(c + 1) * B]).max() <= 1e-10 * scale[kind]
        # every nonzero of the oracle's operator is a term, within FP32 rounding of its value
        assert np.abs(g - w).max() <= 1e-6 * scale[kind], kind
        kept = g != 0.0
        assert np.all(np.abs(w[~kept]) <= 1e-10 * scale[kind]), kind
        assert np.all(np.abs(w[kept]) >= 1e-4 * scale[kind]), kind
    # multiply-adds per row, the paper's "all sparsity" count for these operators
    nk = sum(int(np.sum(np.abs(ob.K[c]) > 1e-9 * kmax)) for c in range(3))
    assert sum(1 for t in terms if t[0] == "t") == nk
    assert sum(1 for t in terms if t[0] == "v") == nk
    assert sum(1 for t in terms if t[0] == "k") == nk


@pytest.mark.parametrize("order", [3, 4, 5])
def test_row_form_terms_are_the_oracle_operators_nonzeros(order):
    """The row-form products of the forward kernels (gen_sparse --list-rows): per direction c the
    rows K_c (time) and K_c^T (volume), per face F~_i (traces) and F~_i^T (projection)."""
    build.build()
    exe = os.path.join(build.OUT_DIR, "gen_sparse")
    out = subprocess.run([exe, "--list-rows", str(order)], capture_output=True, text=True, check=True).stdout
    ob = Basis(order)
    B, F = len(ob.K[0]), ob.Ft[0].shape[1]
    kmax = max(np.abs(k).max() for k in ob.K)
    fmax = max(np.abs(f).max() for f in ob.Ft)
    block = lambda ms: np.concatenate([np.pad(m, ((0, 0), (i * m.shape[1], (len(ms) - 1 - i) * m.shape[1])))
                                       for i, m in enumerate(ms)])
    want = {"T": block([ob.K[c] for c in range(3)]), "V": block([ob.K[c].T for c in range(3)]),
            "P": block([ob.Ft[i] for i in range(4)])}
    # traces: the input mode is listed without its set
    g = np.zeros((4 * F, 4 * B))
    for i in range(4):
        g[i * F:(i + 1) * F, :B] = ob.Ft[i].T
    got = {k: np.zeros_like(v) for k, v in want.items()}
    got["G"], want["G"] = np.zeros_like(g), g
    for line in out.splitlines():
        kind, _, o, k, val = line.split()
        o, k = int(o), int(k)
        if kind == "P":
            assert k // F == o // B
        assert got[kind][o, k] == 0.0
        got[kind][o, k] = float(val)
    for kind in want:
        scale = kmax if kind in "TV" else fmax
        w = want[kind]
        if kind == "T":      # outputs of the top degree vanish and are not written
            nb1 = (order - 1) * order * (order + 1) // 6
            for c in range(3):
                assert np.abs(w[c * B + nb1:(c + 1) * B]).max() <= 1e-10 * kmax
        assert np.abs(got[kind] - w).max() <= 1e-6 * scale, kind
        assert np.all((np.abs(w) <= 1e-10 * scale) | (got[kind] != 0.0)), kind


@pytest.mark.parametrize("order", [3, 4, 5])
def test_row_form_parts_write_every_output_once(order):
    """Every variant of the row-form time products (modes k < nbasis(order - v) in, modes
    b < nbasis(order - 1 - v) out, the elastic kernel's truncation) and the neighbour kernel's parts of
    the projections (gen_sparse --list-parts): each output written by one part, with the oracle's
    entries."""
    build.build()
    exe = os.path.join(build.OUT_DIR, "gen_sparse")
    lines = subprocess.run([exe, "--list-parts", str(order)], capture_output=True, text=True, check=True).stdout.split("\n")
    ob = Basis(order)
    B, F = len(ob.K[0]), ob.Ft[0].shape[1]
    n = lambda o: o * (o + 1) * (o + 2) // 6
    want = {}
    for v in range(order - 1):
        w = np.zeros((3 * B, 3 * B))
        for c in range(3):
            w[c * B:c * B + n(order - 1 - v), c * B:c * B + n(order - v)] = ob.K[c][:n(order - 1 - v), :n(order - v)]
        want["T", v] = (w, {c * B + b for c in range(3) for b in range(n(order - 1 - v))})
    w = np.zeros((4 * B, 4 * F))
    for f in range(4):
        w[f * B:(f + 1) * B, f * F:(f + 1) * F] = ob.Ft[f]
    want["N", 0] = (w, set(range(4 * B)))
    got = {k: np.zeros_like(v[0]) for k, v in want.items()}
    written = {k: [] for k in want}
    for t in (x.split() for x in lines if x):
        if t[0] == "O":
            written[t[1], int(t[2])].append(int(t[4]))
        else:
            assert got[t[0], int(t[1])][int(t[3]), int(t[4])] == 0.0
            got[t[0], int(t[1])][int(t[3]), int(t[4])] = float(t[5])
    for k, (w, outs) in want.items():
        assert len(written[k]) == len(outs) and set(written[k]) == outs, k
        scale = max(np.abs(m).max() for m in (ob.K if k[0] == "T" else ob.Ft))
        assert np.abs(got[k] - w).max() <= 1e-6 * scale, k
        assert np.all((np.abs(w) <= 1e-10 * scale) | (got[k] != 0.0)), k
