"""Device functions of the refinement kernel by themselves, at the edges of their ranges:
probe_device.cu is compiled here and its kernels called with torch tensors."""
import ctypes as C
import math
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

from paper_2202_10204_gb300 import build as B  # noqa: E402

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("probe") / "libprobe.so")
    subprocess.run([B.nvcc(), "-shared", "-o", out, os.path.join(HERE, "probe_device.cu"), "-I", B.CSRC, "-O3",
                    "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", "-cudart", "shared"] + B.ARCH,
                   check=True)
    return C.CDLL(out)


def ptr(t):
    return C.c_void_p(t.data_ptr())


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def sell(probe, off, col, val, x, rows, scat, wide):
    out = torch.full((rows,), 7.0, dtype=val.dtype, device="cuda")
    assert probe.probe_sell(int(val.dtype == torch.float64), rows, ptr(off), ptr(col), ptr(val), ptr(x), ptr(out),
                            scat, wide) == 0
    return out.cpu().numpy()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("rows", [257, 288, 513])
def test_product_of_more_than_32_bits_of_entries(probe, dtype, rows):
    """The block's first eight slices hold 2^31 entries of value 0; the ones after them count."""
    rng = np.random.default_rng(rows)
    ns = (rows + 31) // 32
    w = np.array([1 << 23] * 8 + list(rng.integers(1, 9, ns - 8)))
    off = np.concatenate([[0], np.cumsum(32 * w)]).astype(np.int64)
    tail = int(off[-1] - off[8])
    col = torch.zeros(int(off[-1]), dtype=torch.int32, device="cuda")
    val = torch.zeros(int(off[-1]), dtype=dtype, device="cuda")
    c, v, x = rng.integers(0, rows, tail), rng.integers(-8, 9, tail), rng.integers(-8, 9, rows)  # (exact sums)
    col[off[8]:] = dev(c.astype(np.int32))
    val[off[8]:] = dev(v).to(dtype)
    got = [sell(probe, dev(off), col, val, dev(x).to(dtype), rows, scat, 1) for scat in (0, 1)]
    want = np.zeros(rows)
    for r in range(256, rows):
        q = off[r // 32] - off[8] + 32 * np.arange(w[r // 32]) + r % 32
        want[r] = np.dot(v[q], x[c[q]])
    assert np.array_equal(got[0], want) and np.array_equal(got[1], want)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("rows,width", [(1, 1), (31, 5), (33, 0), (257, 9), (513, 40), (1100, 13)])
def test_products_of_scattered_matrices(probe, dtype, rows, width):
    """Both orders of reading the entries, with places in entries and in columns, add a row's products in one order."""
    rng = np.random.default_rng(rows)
    ns = (rows + 31) // 32
    w = rng.integers(0, width + 1, ns)
    off = np.concatenate([[0], np.cumsum(32 * w)]).astype(np.int64)
    col = rng.integers(0, rows, off[-1] + 1).astype(np.int32)
    val = dev(rng.standard_normal(off[-1] + 1)).to(dtype)
    x = dev(rng.standard_normal(rows)).to(dtype)
    got = [sell(probe, dev(off), dev(col), val, x, rows, scat, wide) for scat in (0, 1) for wide in (0, 1)]
    assert all(np.array_equal(got[0], g) for g in got[1:])
    va, xa = val.double().cpu().numpy(), x.double().cpu().numpy()
    want = np.zeros(rows)
    for r in range(rows):
        q = off[r // 32] + 32 * np.arange(w[r // 32]) + r % 32
        want[r] = np.dot(va[q], xa[col[q]])
    assert np.abs(got[0] - want).max() <= 4 * (width + 1) * torch.finfo(dtype).eps * np.abs(va).max() * np.abs(xa).max()


def wsum_cases(n, rng):
    k = 32 * n
    x = rng.standard_normal(k)
    yield "alike", x
    yield "mixed", x * 10.0 ** rng.integers(-12, 12, k)
    yield "zeros", np.where(rng.random(k) < 0.8, 0.0, x)
    yield "all zero", np.zeros(k)
    yield "full words", np.full(k, 2.0 - 2.0 ** -52)
    yield "negative words", np.full(k, -(2.0 - 2.0 ** -52))
    y = np.concatenate([x[: k // 2], -x[: k // 2]])
    yield "cancels", y
    y = y.copy()
    y[3] += 2.0 ** -50
    yield "nearly cancels", y
    # one value dominates, the others lie just below half a unit of its last places
    for s in range(50, 60):
        y = np.full(k, 0.49 * 2.0 ** -s)
        y[rng.integers(k)] = 1.0
        yield "dominated", y
    # exponent fields around the ends of the integer sums' range
    for field in (99, 100, 101, 1999, 2000, 2001, 2046):
        y = x.clip(-1.9, 1.9) * 2.0 ** (field - 1023 - 8)
        y[0] = 1.5 * 2.0 ** (field - 1023)
        yield "field", y
    yield "subnormal", x * 2.0 ** -1070
    for bad in (np.inf, -np.inf, np.nan):
        y = x.copy()
        y[rng.integers(k)] = bad
        yield "non-finite", y
    y = x.copy()
    y[1], y[2] = np.inf, -np.inf
    yield "inf - inf", y


@pytest.mark.parametrize("n", [1, 2, 3, 5, 8])
def test_integer_sums(probe, n):
    """Within 32 n x 2^-58 of the largest value's power of two and one rounding of the exact sum; outside the
    exponents 100 .. 2000 the roundings of a chain of n and a tree of five levels; the same in every lane."""
    for name, x in wsum_cases(n, np.random.default_rng(n)):
        out = torch.zeros(32, dtype=torch.float64, device="cuda")
        assert probe.probe_wsum(n, ptr(dev(x)), ptr(out)) == 0
        got = out.cpu().numpy()
        assert np.array_equal(got, np.full(32, got[0]), equal_nan=True), name
        if not np.isfinite(x).all():
            with np.errstate(invalid="ignore"):
                assert np.array_equal(got[0], x.sum(), equal_nan=True), name
            continue
        try:
            want = math.fsum(x)
        except OverflowError:
            want = math.inf
        top = np.abs(x).max()
        field = int(np.float64(top).view(np.int64) >> 52)
        if 100 <= field <= 2000:
            tol = 32 * n * 2.0 ** -58 * 2.0 ** (field - 1023) + 0.5 * np.spacing(abs(want))
        else:
            tol = (n + 5) * 2.0 ** -53 * np.abs(x / 64).sum() * 64 if top < 2.0 ** 1000 else math.inf
        assert got[0] == want or abs(got[0] - want) <= tol, (name, got[0], want)


@pytest.mark.parametrize("cnt", [1, 2, 11, 12, 13, 38, 51])
def test_lane_sums(probe, cnt):
    """16 lanes' values in single: on any value's way ceil(log2 min(cnt, 12)) roundings of a tree, half as many as
    there are trees, one that joins the two chains, and four of the lanes' tree."""
    trees = -(-cnt // 12)
    steps = math.ceil(math.log2(min(cnt, 12))) + (trees + 1) // 2 + 4
    u = 2.0 ** -24
    for last in (0.49, 0.51, 0.99):
        # one lane's first value dominates; every further one lies below a unit of its last place
        x = np.full((16, cnt), last * 2.0 ** -23, dtype=np.float32)
        x[:, 0] = 1.0
        out = torch.zeros(1, dtype=torch.float32, device="cuda")
        assert probe.probe_lane_sum(cnt, ptr(dev(x)), ptr(out)) == 0
        want = math.fsum(x.astype(np.float64).ravel())
        assert abs(float(out) - want) <= 1.01 * steps * u * want


@pytest.mark.parametrize("cnt", [1, 2, 3, 14, 54])
def test_sums_in_turn(probe, cnt):
    """A thread's sum of squares in single: half as many roundings as squares, and one more."""
    u = 2.0 ** -24
    for last in (0.49, 0.51, 0.99):
        x = np.full(cnt, math.sqrt(last * 2.0 ** -23), dtype=np.float32)
        x[0] = 1.0
        out = torch.zeros(1, dtype=torch.float32, device="cuda")
        assert probe.probe_turns(cnt, ptr(dev(x)), ptr(out)) == 0
        want = math.fsum(x.astype(np.float64) ** 2)
        assert abs(float(out) - want) <= 1.01 * ((cnt + 1) // 2 + 1) * u * want


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_quotients(probe, dtype):
    """Owner and reader of a quotient form the same bits; they are a division's where the residual step is exact,
    within two units in the last place below, and a division's throughout where the reciprocal is out of range."""
    rng = np.random.default_rng(7)
    f = np.finfo(dtype)
    low = {np.float32: -100, np.float64: -960}[dtype]
    m = 1.0 + rng.integers(0, 1 << 23, 4000).astype(dtype) / (1 << 23)
    m[:200] = np.nextafter(dtype(2), dtype(0)) * np.ones(200, dtype)
    m[200:400] = 1
    divisors = [1.0, 3.0, float(np.nextafter(dtype(2), dtype(0))), 7e-3, 1e-20, 3e20, 1e-29, 9e29]
    slow = [2e30, 1e-31, float(f.tiny) / 8] if dtype is np.float32 else [2e250, 1e-251, 1e-310]
    if dtype is np.float64:
        divisors += [1e-200, 1e240, 3e-249]
    for d in divisors + slow:
        for lo, hi in ((-20, 20), (low, low + 8), (int(f.minexp) - int(f.nmant), low), (int(f.minexp), int(f.maxexp))):
            e = rng.integers(lo, hi, m.size)
            x = np.ldexp(m, e).astype(dtype) * rng.choice([-1, 1], m.size).astype(dtype)
            with np.errstate(all="ignore"):
                want = x / dtype(d)
            own, read = (torch.zeros(m.size, dtype=torch.float64 if f.bits == 64 else torch.float32, device="cuda")
                         for _ in range(2))
            fast = torch.zeros(1, dtype=torch.int32, device="cuda")
            assert probe.probe_quot(int(f.bits == 64), m.size, ptr(dev(x)), C.c_double(d), ptr(own), ptr(read), ptr(fast)) == 0
            own, read = own.cpu().numpy(), read.cpu().numpy()
            assert bool(fast) == (d in divisors), d
            keep = np.isfinite(want) & (np.abs(want) < f.max / 4)
            assert np.array_equal(own[keep], read[keep]), (d, lo)
            ok = keep & ((np.abs(x) >= 2.0 ** low) & (np.abs(want) >= 2 * f.tiny) if d in divisors else True)
            assert np.array_equal(own[ok], want[ok]), (d, lo)
            with np.errstate(all="ignore"):
                assert (np.abs(own - want)[keep] <= 2 * np.spacing(np.abs(want))[keep]).all(), (d, lo)
