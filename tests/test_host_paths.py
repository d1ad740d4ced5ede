"""The library's host side over a stand-in for the CUDA runtime (fake_cudart.cpp), so
without a GPU: which launches it makes, what it does when one is refused, and how long
the sources of its copies live."""
import bisect
import os
import subprocess
import sys
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def fake_lib(tmp_path_factory):
    from paper_2202_10204_gb300 import build as B
    B.build()
    objs = [os.path.join(B.OUT_DIR, s.replace(".cu", ".o")) for s in B.SOURCES]
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    out = str(tmp_path_factory.mktemp("fake") / "libspai_fake.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I" + inc, "-o", out,
                    os.path.join(ROOT, "tests", "fake_cudart.cpp")] + objs + ["-lpthread"], check=True)
    return out


def run(fake_lib, body):
    """Run `body` in a process of its own, where freed memory is overwritten; its last line is the result."""
    head = """
        import ctypes as C, sys
        import numpy as np
        sys.path.insert(0, %r)
        from paper_2202_10204_gb300 import _lib as S, synth
        S.LIB_PATH = %r
        L = S.lib()
        L.fake_get.restype = C.c_longlong
        L.fake_get.argtypes = [C.c_char_p]
        L.fake_set.argtypes = [C.c_char_p, C.c_longlong]
        get = lambda k: L.fake_get(k.encode())
        put = lambda k, v: L.fake_set(k.encode(), v)
        ctx = S.Context(0)
        def system(n):
            A = synth.conv_diff_2d(n, 10.0, 1.0, 0.1, seed=n)
            return A, np.ones(n * n)
    """ % (ROOT, fake_lib)
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(head) + textwrap.dedent(body)], capture_output=True,
                       text=True, cwd=ROOT, env=dict(os.environ, MALLOC_PERTURB_="165"), timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout.strip().splitlines()[-1]


@pytest.mark.parametrize("call", ["build", "solve", "build_right"])
def test_sources_of_copies_live_until_a_wait(fake_lib, call):
    """Host matrices, whose tables nothing waits for before the first kernel reads them."""
    out = run(fake_lib, """
        call = %r
        sys_ = [system(n) for n in (5, 9, 7, 12)]
        As = [s[0] for s in sys_]
        try:
            if call == "solve":
                S.gmres_ir_solve_batch(ctx, As, [s[1] for s in sys_], [np.zeros_like(s[1]) for s in sys_], None,
                                       S.make_ir_opts())
            else:
                S.spai_build_batch(ctx, As, S.make_spai_opts(side=int(call == "build_right")))
        except S.SpaiError as e:
            print(e)
        print(get("launches") > 0, get("stale_copies"))
    """ % call)
    assert out == "True 0"


def scratch_bytes(n, kmax, imax, sg=4, su=4, sp=4):
    """What gmres_ir_solve_noalloc may take of its fixed scratch for P = I, MGS and a matrix without entries."""
    nsl = (n + 31) // 32
    off = 0
    for b in (8 * 4 * 160 * 16, 24 + 4 * (imax + 1) + 8 * (imax + 1) + 24 + 64, su * n, su * n, sg * n, sp * n,
              sg * 32 * nsl * (kmax + 1), 8 * (kmax + 1) * kmax, 8 * (nsl + 1), 4 * nsl, 4, sp):
        off = (off + 255) // 256 * 256 + b
    return off


def test_noalloc_takes_what_fits_its_scratch(fake_lib):
    """Sizes that end within the last 256 bytes of the 32 MiB."""
    room = 32 << 20
    sizes = []
    for kmax in range(1, 500):
        n = bisect.bisect_right(range(1 << 20), room, key=lambda m: scratch_bytes(m, kmax, 10)) - 1
        if room - scratch_bytes(n, kmax, 10) < 256:
            sizes.append((n, kmax))
    assert len(sizes) >= 5
    out = run(fake_lib, """
        got = set()
        for n, kmax in %r:
            rp, ci, va, b, x = (np.zeros(n + 1, t) for t in (np.int64, np.int32, np.float64, np.float64, np.float64))
            p = lambda a: a.ctypes.data_as(C.c_void_p)
            A = S.spai_csr(n, 1, p(rp), p(ci), p(va), 1)
            o = S.make_ir_opts(uf="single", u="single", ug="single", up="single", ur="double", gmres_max_it=kmax)
            st = S.ir_stats()
            got.add(L.gmres_ir_solve_noalloc(C.byref(A), None, p(b), p(x), C.byref(o), None, C.byref(st)))
        print(sorted(got))
    """ % (sizes,))
    assert out == "[%d]" % 1  # (no kernel ran, so nothing converged)


@pytest.mark.parametrize("cluster_max", [16, 8, 2, 1])
@pytest.mark.parametrize("n", [8, 60, 150, 240])
def test_clusters_that_the_device_refuses(fake_lib, n, cluster_max):
    """A batch and a single system go on without a cluster of their usual size: on smaller ones, or on a grid."""
    out = run(fake_lib, """
        n, most = %d, %d
        put("cluster_max", most)
        o = S.make_ir_opts()
        A, b = system(n)
        a = S.gmres_ir_solve(ctx, A, b, np.zeros_like(b), opts=o)["rc"]
        one = get("cluster_launches"), get("grid_launches")
        sys_ = [system(n), system(7)]
        st, _ = S.gmres_ir_solve_batch(ctx, [s[0] for s in sys_], [s[1] for s in sys_],
                                    [np.zeros_like(s[1]) for s in sys_], None, o)
        print(a, [s["rc"] for s in st], one, all(s["grid"] <= most or get("grid_launches") > one[1] for s in st))
    """ % (n, cluster_max))
    # (nothing converges: no kernel ran); a single system up to 6144 rows takes a cluster of up to 16
    blocks = min((n * n + 63) // 64, 16)
    alone = n * n <= 6144 and blocks <= cluster_max
    assert out == "1 [1, 1] %s True" % ((1, 0) if alone else (0, 1),)


def test_launch_errors_are_reported(fake_lib):
    """An error of the launch itself is not taken for a cluster that is too large."""
    out = run(fake_lib, """
        put("cluster_error", 719)  # cudaErrorLaunchFailure
        A, b = system(30)
        try:
            print(S.gmres_ir_solve(ctx, A, b, np.zeros_like(b), opts=S.make_ir_opts())["rc"])
        except S.SpaiError as e:
            print(e.code, get("grid_launches"))
    """)
    assert out == "-7 0"
