"""Host code of the solvers on a stand-in for the CUDA runtime (fake_cudart.c, no GPU): the order of streams
when a call fails, and what happens inside a stream capture."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import glob
    from paper_2607_02335_gb300 import build as B
    B.build()
    d = str(tmp_path_factory.mktemp("fake"))
    fake, so = os.path.join(d, "fake.o"), os.path.join(d, "libfe_fake.so")
    subprocess.run(["gcc", "-O1", "-fPIC", "-c", os.path.join(HERE, "fake_cudart.c"), "-o", fake], check=True)
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", so, *sorted(glob.glob(os.path.join(B.BUILD, "*.o"))), fake],
                   check=True)
    return ctypes.CDLL(so)


def aligned(n):
    """n zeros on a 16-byte boundary, as the library's callers have to give."""
    a = np.zeros(n + 2)
    off = (-a.ctypes.data % 16) // 8
    return a[off:off + n]


def mesh(fe, lib, m, p):
    h = ctypes.c_void_p()
    desc = fe.fe_mesh_desc(*m, p, 0.1, fe.FE_GEOM_STORED, 1, 0)
    assert lib.fe_mesh_create(ctypes.byref(desc), None, ctypes.byref(h)) == 0
    return h


HOOK = ctypes.CFUNCTYPE(None, ctypes.c_char_p, ctypes.POINTER(ctypes.c_void_p))


def pointer_arg(args, k):
    return ctypes.cast(args[k], ctypes.POINTER(ctypes.c_void_p))[0]


@pytest.mark.parametrize("mixed", [False, True])
def test_a_solve_after_a_failed_allocation(lib, mixed):
    """Each allocation or launch of a mesh's first solve fails in turn; the next solve on the mesh reports no
    left-over error and runs on a whole workspace."""
    from paper_2607_02335_gb300 import fe
    p, m = 3, (2, 2, 2)
    b, x = aligned(8 * (p + 1) ** 3), aligned(8 * (p + 1) ** 3)
    opts = fe.fe_cg_opts(1e-10, 100, fe.FE_F32 if mixed else 0, 0, 0.1, None)
    seen = []

    def on_launch(name, args):
        if b"k_precond" in name:  # w, invmult, partials, count and sc
            seen.append(all(pointer_arg(args, k) for k in (0, 4, 6, 7, 8)))

    hook = HOOK(on_launch)
    failed = 0
    for n in range(1, 40):
        h, res = mesh(fe, lib, m, p), fe.fe_cg_result()
        lib.fake_fail_at(n)
        failed += lib.fe_cg_solve(h, ctypes.c_void_p(b.ctypes.data), ctypes.c_void_p(x.ctypes.data),
                                  ctypes.byref(opts), ctypes.byref(res), None) != 0
        lib.fake_fail_at(0)
        lib.fake_hook(hook)
        st = lib.fe_cg_solve(h, ctypes.c_void_p(b.ctypes.data), ctypes.c_void_p(x.ctypes.data),
                             ctypes.byref(opts), ctypes.byref(res), None)
        lib.fake_hook(None)
        assert st == 0, n  # a zero right-hand side
        assert seen and all(seen), n
        seen.clear()
        lib.fe_mesh_destroy(h)
    assert 15 < failed < 39  # every failable call of the solve, and a few solves beyond the last


def test_nothing_is_freed_under_a_forked_apply(lib):
    """A batched solve of three degrees, with each of its first calls that allocate, launch, fork or join
    failing in turn: the error is reported, and no buffer is freed while a forked stream still holds kernels
    that nothing orders before the free."""
    from paper_2607_02335_gb300 import fe
    shapes = [((2, 2, 2), 1), ((2, 2, 2), 2), ((2, 2, 2), 4)]
    meshes = [mesh(fe, lib, m, p) for m, p in shapes]
    vecs = [[aligned(8 * (p + 1) ** 3) for _, p in shapes] for _ in range(2)]
    arr = [(ctypes.c_void_p * 3)(*[v.ctypes.data for v in vs]) for vs in vecs]
    hs = (ctypes.c_void_p * 3)(*meshes)
    for mixed in (0, fe.FE_F32):
        opts = fe.fe_cg_opts(1e-10, 100, mixed, 0, 0.1, None)
        for n in range(1, 160):
            res = (fe.fe_cg_result * 3)()
            lib.fake_fail_at(n)
            st = lib.fe_cg_solve_batched(3, hs, arr[0], arr[1], ctypes.byref(opts), res, None)
            lib.fake_fail_at(0)
            assert st != 0, (mixed, n)
            assert lib.fake_unordered_frees() == 0, (mixed, n)


class Scal(ctypes.Structure):  # the start of CgScal (fe_cgcore.h)
    _fields_ = [(k, ctypes.c_double) for k in ("rz", "rz_new", "qp", "qz", "alpha", "beta", "rnorm2", "bnorm2",
                                               "relres", "best")] + [("done", ctypes.c_int)]


# single cells and pairs in FP64 (fused and separate iterations), FP32
@pytest.mark.parametrize("p,m,mixed", [(3, (2, 2, 2), False), (6, (2, 2, 2), False), (3, (24, 24, 24), False),
                                       (2, (3, 3, 3), True), (7, (2, 2, 2), True)])
def test_no_kernel_attribute_is_set_inside_a_capture(lib, p, m, mixed):
    """The iteration graph's capture holds launches only: each kernel was loaded and had its attributes set
    before."""
    from paper_2607_02335_gb300 import fe
    n = m[0] * m[1] * m[2] * (p + 1) ** 3
    b, x = aligned(n), aligned(n)
    opts = fe.fe_cg_opts(1e-10, 100, fe.FE_F32 if mixed else 0, 0, 0.1, None)

    def on_launch(name, args):
        if b"k_precond" in name:  # a right-hand side that is not zero, and a residual to iterate on
            sc = ctypes.cast(pointer_arg(args, 8), ctypes.POINTER(Scal))[0]
            sc.bnorm2 = sc.rnorm2 = sc.rz = sc.relres = 1.0

    hook = HOOK(on_launch)
    h, res, graphs = mesh(fe, lib, m, p), fe.fe_cg_result(), lib.fake_graphs()
    lib.fake_hook(hook)
    lib.fe_cg_solve(h, ctypes.c_void_p(b.ctypes.data), ctypes.c_void_p(x.ctypes.data), ctypes.byref(opts),
                    ctypes.byref(res), None)  # ends at the first replay, which the stand-in refuses
    lib.fake_hook(None)
    lib.fe_mesh_destroy(h)
    assert lib.fake_graphs() == graphs + 1
    assert lib.fake_attr_in_capture() == 0
