"""Two routes to one result: the staged products of scattered systems whose input takes
several passes against the refinement on a grid, and the two adaptive column kernels
against one another."""
import numpy as np
import pytest

import oracle as O
from paper_2202_10204_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

import paper_2202_10204_gb300 as S  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    c = S.Context(0, stream=torch.cuda.current_stream())
    yield c
    c.close()


def errors(A, b, x, x_true):
    M = synth.to_scipy(A)
    den = abs(M).sum(axis=1).max() * np.max(np.abs(x_true)) + np.max(np.abs(b))
    return np.max(np.abs(b - M @ x)) / den, np.max(np.abs(x - x_true)) / np.max(np.abs(x_true))


@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("n,prec,orth", [
    (15001, "double", 2),   # a block of 3008 rows holds about 8000 staged entries: two passes
    (30011, "double", 2),   # four
    (13005, "double", 0),   # Gram-Schmidt rounds, quotients formed while staging: one or two
    (45003, "single", 2), (49999, "single", 2),   # about 36000: two
    (14999, "double", 1)])
def test_staged_products_in_passes(ctx, n, prec, orth, side):
    """A scattered system in a batch (a cluster, staged inputs) against itself alone on a grid: the same steps, its
    GMRES iterations within 10% and errors within ten times."""
    A = synth.random_sparse(n, 10, seed=n, log10_scale=1.0)
    b, x_true = synth.rhs(A, seed=6)
    so = S.make_spai_opts(init=O.PAT_A, max_fill=30, uf="single", side=side)
    io = S.make_ir_opts(uf="single", u="double", ug=prec, up=prec, ur="double", tau=1e-4, orth=orth, side=side)
    P, _ = S.spai_build(ctx, A, so)
    x1, x2 = np.zeros_like(b), np.zeros_like(b)
    alone = S.gmres_ir_solve(ctx, A, b, x1, P=P, opts=io)
    small = synth.conv_diff_2d(20, 10.0, 1.0, 0.1, seed=1)
    (st, _), rc = S.gmres_ir_solve_batch(ctx, [A, small], [b, np.ones(400)], [x2, np.zeros(400)], [P, None], io)
    P.free()
    assert rc[0] == 0 and st["grid"] < 17 <= alone["grid"]
    assert st["steps"] == alone["steps"]
    assert abs(st["total_its"] - alone["total_its"]) <= max(1, 0.1 * alone["total_its"])
    for got, want in zip(errors(A, b, x2, x_true), errors(A, b, x1, x_true)):
        assert got <= 10 * max(want, 2.0 ** -53)


@pytest.mark.parametrize("n,prec", [(2500, "double"), (6100, "double")])
def test_cgs2_on_a_cluster(ctx, n, prec):
    """Classical Gram-Schmidt in double on one cluster, against the oracle."""
    A = synth.random_sparse(n, 10, seed=n, log10_scale=1.0)
    b, x_true = synth.rhs(A, seed=6)
    tup = dict(uf="single", u="double", ug=prec, up=prec, ur="double")
    x = np.zeros_like(b)
    st = S.gmres_ir_solve(ctx, A, b, x, sopts=S.make_spai_opts(init=O.PAT_A, max_fill=30, uf="single"),
                          opts=S.make_ir_opts(tau=1e-4, orth=1, **tup))
    P = O.assemble_P(O.spai(A, init=O.PAT_A, max_fill=30, uf="single"), prec, "single")
    ref = O.gmres_ir(A, b, P, tau=1e-4, orth=O.ORTH_CGS2, **tup)
    assert st["grid"] <= 16 and st["steps"] == ref["steps"]
    assert abs(st["total_its"] - ref["total_its"]) <= max(1, 0.1 * ref["total_its"])
    for got, want in zip(errors(A, b, x, x_true), errors(A, b, ref["x"], x_true)):
        assert got <= 10 * max(want, 2.0 ** -53)


def beside_diagonal(A, total):
    """A and a diagonal block that fills the order up to `total`."""
    rp, ci, va = A
    n, more = len(rp) - 1, total - (len(rp) - 1)
    return (np.concatenate([rp, rp[-1] + 1 + np.arange(more)]),
            np.concatenate([ci, n + np.arange(more, dtype=np.int32)]).astype(np.int32), np.concatenate([va, np.ones(more)]))


@pytest.mark.parametrize("uf", ["half", "single", "double"])
@pytest.mark.parametrize("n,per_col,zeros", [(1200, 9, 0.0), (700, 36, 0.0), (1025, 14, 0.2)])
def test_adaptive_kernels_agree(ctx, uf, n, per_col, zeros):
    """Columns of a matrix whose bitmaps fit, and of the same matrix in one so large that they do not: equal bits."""
    A = synth.random_sparse(n, per_col, seed=n, log10_scale=2.0)
    if zeros:
        rows = np.repeat(np.arange(n), np.diff(A[0]))
        va = A[2].copy()
        va[(np.random.default_rng(5).random(len(va)) < zeros) & (A[1] != rows)] = 0.0
        A = (A[0], A[1], va)
    so = S.make_spai_opts(init=O.PAT_IDENTITY, adaptive=True, eps=0.2, alpha=12, beta=8, max_fill=30, uf=uf)
    got = []
    for M in (A, beside_diagonal(A, 120000 if uf == "double" else 460000)):
        P, st = S.spai_build(ctx, M, so, per_column=True)
        rp, ci, va = P.export()
        P.free()
        got.append((rp[:n + 1], ci[:rp[n]], va[:rp[n]], st["colres"][:n], st["nI"][:n], st["nJ"][:n], st["flags"][:n]))
    assert got[0][5].max() > 12
    for u, v in zip(*got):
        assert np.array_equal(u, v)


@pytest.mark.parametrize("shape,prec", [((32, 32, 27), "double"), ((32, 32, 28), "double"), ((33, 33, 34), "single"),
                                        ((34, 33, 34), "single")])
def test_gram_schmidt_groups_by_grid(ctx, shape, prec):
    """Grids just below and at the line from which the rounds run in a group (112 and 148 blocks)."""
    A = synth.conv_diff_3d(shape, 20.0, seed=5)
    b, x_true = synth.rhs(A, seed=6)
    tup = dict(uf="single", u="double", ug=prec, up=prec, ur="double")
    x = np.zeros_like(b)
    st = S.gmres_ir_solve(ctx, A, b, x, sopts=S.make_spai_opts(init=O.PAT_A, max_fill=30, uf="single"),
                          opts=S.make_ir_opts(tau=1e-4, orth=0, **tup))
    P = O.assemble_P(O.spai(A, init=O.PAT_A, max_fill=30, uf="single"), prec, "single")
    ref = O.gmres_ir(A, b, P, tau=1e-4, orth=O.ORTH_MGS, **tup)
    assert st["steps"] == ref["steps"]
    assert abs(st["total_its"] - ref["total_its"]) <= max(1, 0.1 * ref["total_its"])
    for got, want in zip(errors(A, b, x, x_true), errors(A, b, ref["x"], x_true)):
        assert got <= 10 * max(want, 2.0 ** -53)
