"""The largest orders that one system's refinement takes on a grid: a block keeps its rows
of w (one-reduction MGS: of u and w) in shared memory, and what it keeps beside them may
not grow."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

import paper_2202_10204_gb300 as S  # noqa: E402


def block_bytes(rows, kmax, orth, sg):
    """What a block of `rows` rows may take at most, its static variables among it."""
    sa = max(sg, 4)
    b = (1104 if sg == 8 else 976) + 40 * (kmax + 2) + 16 * (rows // 32 + 1) + rows * sg + 64
    if orth == 2:
        b += sg * rows + sa * (4 * (kmax + 1) + 2 * (kmax + 33)) + 4 * (kmax + 2) + 16 + 1024 * sa + 16
    return b


@pytest.mark.parametrize("orth,ug,kmax", [(0, "single", 500), (0, "single", 1024), (0, "double", 500),
                                          (1, "double", 1024), (2, "single", 500), (2, "single", 1024),
                                          (2, "double", 500), (2, "double", 1024), (2, "half", 500)])
def test_largest_order(orth, ug, kmax):
    props = torch.cuda.get_device_properties(0)
    blocks = props.multi_processor_count - (1 if orth == 2 else 0)
    room = props.shared_memory_per_block_optin
    sg = {"half": 2, "single": 4, "double": 8}[ug]
    rows = max(r for r in range(32, 1 << 17, 32) if block_bytes(r, kmax, orth, sg) <= room)
    n = rows * blocks
    A = (torch.arange(n + 1, device="cuda"), torch.arange(n, dtype=torch.int32, device="cuda"),
         torch.full((n,), 2.0, dtype=torch.float64, device="cuda"))
    b = torch.ones(n, dtype=torch.float64, device="cuda")
    x = torch.zeros_like(b)
    ctx = S.Context(0, stream=torch.cuda.current_stream())
    st = S.gmres_ir_solve(ctx, A, b, x, opts=S.make_ir_opts(
        uf="single", u="single", ug=ug, up="double" if ug == "double" else ug, ur="double", tau=1e-2, orth=orth,
        gmres_max_it=kmax, ir_max_steps=2))
    ctx.close()
    assert st["grid"] == props.multi_processor_count
    # A = 2 I: one column solves it but for the roundings of the basis
    assert float((x - 0.5).abs().max()) <= 1e-3 and np.isfinite(st["final_nbe"])


@pytest.mark.parametrize("orth", [0, 2])
def test_more_than_32_bits_of_entries(orth):
    """72 dense rows, one a slice and all in the first block: 2.3e9 entries of the slices' padded form."""
    n, dense = 1000000, 72
    cnt = torch.ones(n, dtype=torch.int64, device="cuda")
    rows = 32 * torch.arange(dense, device="cuda")
    cnt[rows] = n
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(cnt, 0, out=rowptr[1:])
    col = torch.empty(int(rowptr[-1]), dtype=torch.int32, device="cuda")
    val = torch.zeros(col.numel(), dtype=torch.float64, device="cuda")
    i = torch.arange(n, device="cuda")
    single = cnt == 1
    col[rowptr[:-1][single]] = i[single].to(torch.int32)
    val[rowptr[:-1][single]] = 2.0
    for r in rows.tolist():
        p = int(rowptr[r])
        col[p:p + n] = i.to(torch.int32)
        val[p + n - 1] = 1.0  # the last entry counts too
        val[p + r] = 2.0
    b = torch.full((n,), 2.0, dtype=torch.float64, device="cuda")
    b[rows] += 1.0
    x = torch.zeros_like(b)
    ctx = S.Context(0, stream=torch.cuda.current_stream())
    st = S.gmres_ir_solve(ctx, (rowptr, col, val), b, x, opts=S.make_ir_opts(
        uf="single", u="single", ug="single", up="single", ur="double", tau=1e-4, orth=orth, gmres_max_it=10, ir_max_steps=3))
    ctx.close()
    assert st["total_its"] <= 12 and float((x - 1.0).abs().max()) <= 1e-5
