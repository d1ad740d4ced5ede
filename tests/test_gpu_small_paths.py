"""Kernels and branches chosen by size, at the sizes where their index work can go
wrong, against the oracle:

* the adaptive column kernel with bitmaps (spai_adapt.cuh): orders around a bitmap
  word and a block's threads, rows longer than a warp, explicit zeros, and a
  restricted rho (which keeps the other kernel);
* the column kernel with its tile in registers (spai_mid.cuh) against the one with
  the tile in shared memory, bit for bit;
* the kernel of four small columns a warp against dense least squares;
* the refinement on one thread-block cluster (orders around its blocks' rows and
  their padding, scattered matrices with staged inputs) and on the grid just past
  the line, Gram-Schmidt rounds of several vectors on each and in a group of blocks.
"""
import numpy as np
import pytest

import oracle as O
from neartie import replay_gap
from paper_2202_10204_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

import paper_2202_10204_gb300 as S  # noqa: E402

# as in test_gpu_parity.py: a pattern that differs from the oracle's is a near-tie of rho;
# the solution's errors are within ten times the oracle's
NEAR_TIE = 512


@pytest.fixture(scope="module")
def ctx():
    c = S.Context(0, stream=torch.cuda.current_stream())
    yield c
    c.close()


def with_zeros(A, share, seed):
    rp, ci, va = A
    rows = np.repeat(np.arange(len(rp) - 1), np.diff(rp))
    va = va.copy()
    va[(np.random.default_rng(seed).random(len(va)) < share) & (ci != rows)] = 0.0
    return rp, ci, va


@pytest.mark.parametrize("n,per_col,uf,zeros,restricted", [
    (33, 4, "single", 0.0, False), (64, 5, "double", 0.0, False), (513, 12, "single", 0.0, False),
    (700, 36, "half", 0.0, False), (1025, 10, "single", 0.2, False), (400, 9, "single", 0.0, True)])
def test_adaptive_columns(ctx, n, per_col, uf, zeros, restricted):
    A = synth.random_sparse(n, per_col, seed=n, log10_scale=2.0)
    if zeros:
        A = with_zeros(A, zeros, 5)
    eps, beta, F = 0.2, 8, 30
    kw = dict(init=O.PAT_IDENTITY, adaptive=True, eps=eps, beta=beta, max_fill=F, uf=uf)
    P, st = S.spai_build(ctx, A, S.make_spai_opts(rho_restricted=restricted, **kw), per_column=True)
    rp, ci, va = P.export()
    ref = O.spai(A, rho_restricted=restricted, **kw)
    u = O.UNIT_ROUNDOFF[O.prec(uf)]
    same = np.zeros(n, bool)
    for k in range(n):
        J = ci[rp[k]:rp[k + 1]]
        same[k] = np.array_equal(J, ref["Jidx"][k][: ref["Jcnt"][k]])
        if not same[k] and not restricted:
            r = replay_gap(A, ref["d"], k, J, uf, eps, beta, F)
            assert r is not None and r[1] <= NEAR_TIE * u, (k, r)
    assert same.mean() >= 0.8
    # ||s_k|| as the kernel computed it, against the oracle's column in 64 bits
    tol = {"half": 2e-2, "single": 1e-4, "double": 1e-9}[uf]
    assert np.all(np.abs(st["colres"] - ref["colres64"])[same] <= tol)
    assert np.array_equal(st["nI"][same], ref["Icnt"][same])
    P.free()


def long_rows(n, seed):
    """Columns of four entries, three of them in rows of about 60 entries."""
    rng = np.random.default_rng(seed)
    M = np.zeros((n, n))
    for j in range(n):
        M[20 * rng.choice(n // 20, 3, replace=False), j] = rng.standard_normal(3)
        M[j, j] = 4.0
    rp = np.concatenate([[0], np.cumsum((M != 0).sum(1))])
    ci = np.nonzero(M)[1].astype(np.int32)
    return rp.astype(np.int64), ci, M[M != 0]


@pytest.mark.parametrize("uf", ["half", "single"])
@pytest.mark.parametrize("case", [7, 9, 11, 12, 13, 14, 15, 16, "long", "zeros"])
def test_register_tile_columns(ctx, uf, case):
    """Shadows of 3 to 10 slices of 32 rows, 1 to 16 pattern columns: both kernels do the
    same operations in the same order, so P, the norms and |I| are equal."""
    A = long_rows(600, 3) if case == "long" else synth.random_sparse(1200, 13 if case == "zeros" else case, seed=41)
    if case == "zeros":
        A = with_zeros(A, 0.3, 7)
    got = []
    for variant in (0, 3):  # the bin's own tile; the 32-column tile, always in shared memory
        for b in range(2, 9):
            S.tune_set(0, uf, b, variant)
        P, st = S.spai_build(ctx, A, S.make_spai_opts(init=O.PAT_A, max_fill=16, uf=uf), per_column=True)
        got.append((*P.export(), st["colres"], st["nI"]))
        P.free()
    for b in range(2, 9):
        S.tune_set(0, uf, b, -1)
    assert got[0][4].max() > 64
    for u, v in zip(*got):
        assert np.array_equal(u, v)


def stencil_1d(n, w):
    """Rows of the entries -w .. w around the diagonal: shadows of at most 4 w + 1 rows."""
    i, j = np.nonzero(np.abs(np.subtract.outer(np.arange(n), np.arange(n))) <= w)
    v = np.random.default_rng(n).standard_normal(len(i)) + 6.0 * (i == j)
    return np.searchsorted(i, np.arange(n + 1)).astype(np.int64), j.astype(np.int32), v


@pytest.mark.parametrize("uf", ["single", "double"])
@pytest.mark.parametrize("case", ["one", "three", "chain", "seven", "grid", "zeros", "mixed"])
def test_packed_columns(ctx, uf, case):
    """At most 16 shadow rows and 7 pattern columns; "mixed" has columns past either."""
    A = {"one": lambda: stencil_1d(1, 0), "three": lambda: stencil_1d(3, 2), "chain": lambda: stencil_1d(67, 1),
         "seven": lambda: stencil_1d(131, 3), "grid": lambda: synth.conv_diff_2d(13, 10.0, 1.0, 0.1, seed=3),
         "zeros": lambda: with_zeros(synth.conv_diff_2d(11, 10.0, 1.0, 0.1, seed=4), 0.2, 9),
         "mixed": lambda: synth.random_sparse(501, 4, seed=6)}[case]()
    n = len(A[0]) - 1
    P, st = S.spai_build(ctx, A, S.make_spai_opts(init=O.PAT_A, max_fill=16, uf=uf), per_column=True)
    rp, ci, va = P.export()
    P.free()
    ref = O.spai(A, init=O.PAT_A, max_fill=16, uf=uf)
    u = O.UNIT_ROUNDOFF[O.prec(uf)]
    M = np.zeros((n, n))
    M[np.repeat(np.arange(n), np.diff(A[0])), A[1]] = A[2]
    d = 1.0 / np.abs(M).max(1)
    assert np.array_equal(st["nI"], ref["Icnt"])
    small = (st["nI"] <= 16) & (np.diff(rp) <= 7)
    assert small.any() and (case == "mixed") != small.all()
    for k in range(n):
        J = ci[rp[k]:rp[k + 1]]
        assert np.array_equal(J, ref["Jidx"][k][: ref["Jcnt"][k]])
        B, e = (M[J] * d[J, None]).T, np.eye(n)[k]
        m = np.linalg.lstsq(B, e, rcond=None)[0]
        # Householder least squares in u_f (Higham, Accuracy and Stability, Theorem 20.3): gamma_{mn}
        # with a constant of a few, the values of B rounded to u_f themselves
        err = 8 * B.shape[1] * 16 * u * np.linalg.cond(B) ** 2 * np.abs(m).max()
        assert np.all(np.abs(va[rp[k]:rp[k + 1]] - m * d[J]) <= err * d[J] + u * np.abs(m * d[J]))
        assert abs(st["colres"][k] - np.linalg.norm(B @ m - e)) <= 8 * B.shape[1] * 16 * u * np.linalg.cond(B)


@pytest.mark.parametrize("kind,n,orth,prec", [
    ("grid", (1, 1, 7), 2, "single"), ("grid", (5, 13, 1), 0, "single"), ("grid", (9, 9, 7), 2, "double"),
    ("grid", (8, 9, 8), 2, "single"), ("grid", (23, 25, 21), 1, "single"), ("grid", (26, 21, 30), 0, "single"),
    ("grid", (16, 24, 16), 2, "double"), ("grid", (23, 23, 23), 2, "single"), ("grid", (24, 23, 23), 2, "single"),
    ("grid", (31, 31, 31), 0, "single"), ("grid", (29, 31, 33), 0, "double"), ("grid", (19, 20, 21), 0, "double"),
    ("random", 2100, 2, "single"), ("random", 8500, 2, "single"), ("random", 1500, 0, "double")])
def test_refinement_by_size(ctx, kind, n, orth, prec):
    A = synth.conv_diff_3d(n, 20.0, seed=5) if kind == "grid" else synth.random_sparse(n, 10, seed=5, log10_scale=1.0)
    b, x_true = synth.rhs(A, seed=6)
    tup = dict(uf="single", u="double", ug=prec, up=prec, ur="double")
    so = S.make_spai_opts(init=O.PAT_A, max_fill=30, uf="single")
    x = np.zeros_like(b)
    st = S.gmres_ir_solve(ctx, A, b, x, sopts=so, opts=S.make_ir_opts(tau=1e-4, orth=orth, **tup))
    P = O.assemble_P(O.spai(A, init=O.PAT_A, max_fill=30, uf="single"), prec, "single")
    ref = O.gmres_ir(A, b, P, tau=1e-4, orth=(O.ORTH_MGS, O.ORTH_CGS2, O.ORTH_MGS_ICWY)[orth], **tup)
    assert st["steps"] == ref["steps"]
    assert abs(st["total_its"] - ref["total_its"]) <= max(1, 0.1 * ref["total_its"])
    Ms = synth.to_scipy(A)
    den = abs(Ms).sum(axis=1).max() * np.max(np.abs(x_true)) + np.max(np.abs(b))
    for got, want in ((np.max(np.abs(b - Ms @ x)) / den, np.max(np.abs(b - Ms @ ref["x"])) / den),
                      (np.max(np.abs(x - x_true)), np.max(np.abs(ref["x"] - x_true)))):
        assert got <= 10 * max(want, 2.0 ** -53)
