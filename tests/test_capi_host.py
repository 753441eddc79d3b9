"""C-ABI checks that need no GPU: the library loads, exports every function
that include/qbx.h declares, and its host-only functions behave."""
import ctypes
import os
import re

import numpy as np

import paper_1207_4461_gb300 as qbx

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_functions():
    names = []
    for fn in sorted(os.listdir(os.path.join(ROOT, "include"))):
        if not fn.endswith(".h"):
            continue
        src = open(os.path.join(ROOT, "include", fn)).read()
        src = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
        names += re.findall(r"^\s*(?:const\s+)?[A-Za-z_][\w\s\*]*?\b(qbx_\w+)\s*\(", src, flags=re.M)
    return sorted(set(names))


def test_library_exports_every_declared_symbol():
    L = qbx.lib()
    names = declared_functions()
    assert len(names) >= 15
    for n in names:
        assert hasattr(L, n), n
        assert isinstance(getattr(L, n), ctypes._CFuncPtr)


def test_version_and_error_string():
    L = qbx.lib()
    assert L.qbx_version() == 1
    assert isinstance(L.qbx_last_error(), bytes)


def test_host_gauss_legendre_matches_numpy():
    for q in (1, 3, 16, 64, 128):
        x, w = qbx.qbx_gauss_legendre(q)
        xn, wn = np.polynomial.legendre.leggauss(q)
        assert np.abs(x - xn).max() < 1e-15
        assert np.abs(w - wn).max() < 1e-14
        assert abs(w.sum() - 2.0) < 1e-14


def test_host_argument_errors_need_no_device():
    L = qbx.lib()
    x = np.zeros(4)
    assert L.qbx_gauss_legendre(0, x.ctypes.data_as(ctypes.c_void_p), x.ctypes.data_as(ctypes.c_void_p)) == 1
    assert L.qbx_gauss_legendre(qbx.MAX_P * 10, None, None) == 1
    h = ctypes.c_void_p()
    assert L.qbx_plan_create(ctypes.byref(h), 0, 0, 64, 0) == 1
    assert b"q_tgt" in L.qbx_last_error()
    assert L.qbx_apply(None, None, 0, 0, 0, qbx.c64(1.0, 0.0), 4, None, 1, 0, None, None, None, None) == 1
    assert b"plan" in L.qbx_last_error()
    assert L.qbx_apply_cfie(None, None, qbx.c64(1.0, 0.0), qbx.c64(1.0, 0.0), 4, None, 1, None, None) == 1
    assert b"plan" in L.qbx_last_error()


def test_workspace_bytes_formula():
    b = qbx.qbx_workspace_bytes(16384, 8192, 2, 1)
    assert b >= 16384 * 16 + 64 * 8192 * 2 * 16
    assert qbx.qbx_workspace_bytes(-1, 1, 1, 1) == 0


def test_shape_adjoint_workspace_bytes():
    """Holds the oversampled density, the centre gradients, coefficient
    columns and 64 splits of both sweeps; 0 for bad arguments."""
    M, p, nrhs = 128, 10, 1
    b = qbx.qbx_shape_adjoint_workspace_bytes(M, 16, 64, p, nrhs)
    n_t, n_s = M * 16, M * 64
    assert b >= n_s * 16 + 64 * (2 * n_t) * 4 * 16 + 64 * n_s * 3 * 16
    assert qbx.qbx_shape_adjoint_workspace_bytes(M, 16, 64, p, 2) > b
    assert qbx.qbx_shape_adjoint_workspace_bytes(0, 16, 64, p, 1) == 0
    assert qbx.qbx_shape_adjoint_workspace_bytes(M, 16, 64, -1, 1) == 0


def test_workspace_bytes_hold_the_cluster_arrays():
    """Beside 64 splits: node entries, coefficients (1 KB per node, column set
    and rhs), leaf contributions (1 KB per leaf, level, set and rhs) and lists
    (20 bytes per block and leaf), for one side and for two; the bound of these
    arrays ends at 8 GB."""
    for q_tgt, q_src in ((16, 64), (8, 32), (12, 40), (16, 16)):
        for M in (16, 100, 256, 1024, 4096):
            for sides in (1, 2):
                for ncoef, nset, ncset in ((1, 1, 1), (2, 2, 2), (2, 1, 3), (3, 2, 4), (4, 3, 5)):
                    for nrhs in (1, 3):
                        n_src, n_ctr = M * q_src, sides * M * q_tgt
                        leaves = M * (2 if q_src >= 32 and q_src % 2 == 0 else 1)
                        blocks = (M * q_tgt + 31) // 32
                        lev, nodes = 0, 0
                        while lev == 0 or leaves >> lev >= 8:
                            nodes += (leaves + (1 << lev) - 1) >> lev
                            lev += 1
                        supers = blocks + 7 if blocks >= 64 else 0
                        entries = nodes + blocks + supers
                        need = (entries * (32 + ncset * nrhs * 1024) + lev * leaves * nset * nrhs * 1024
                                + 20 * blocks * leaves + 20 * blocks + 5 * supers * leaves + 24 * supers + 10 * 256)
                        pairs = 3 * n_src * nrhs * 16 + 64 * n_ctr * ncoef * nrhs * 16
                        b = qbx.qbx_workspace_bytes(n_src, n_ctr, ncoef, nrhs)
                        assert pairs + need <= b < pairs + 4096 + 8 * 2**30, (q_tgt, q_src, M, sides, ncoef, nrhs)
    assert qbx.qbx_workspace_bytes(1 << 22, 1 << 20, 1, 1) <= 3 * 16 * 2**22 + 64 * 16 * 2**20 + 8 * 2**30 + 4096
    a, b, c = (ctypes.c_int() for _ in range(3))
    L = qbx.lib()
    assert L.qbx_debug_route(None, ctypes.byref(a), ctypes.byref(b), ctypes.byref(c)) == 1
