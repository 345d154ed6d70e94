"""The work plan of the tensor-core level solves on the CPU: every panel tile
taken exactly once (or zero), every row list right, and the solution of the
walked plan against a sparse direct solve (FP64 both: a few hundred roundings
of 1e-16 on these condition numbers, bounded at 1e-10 of the largest entry).
Grids from one node to several chunks per reduction; every split over a
cluster."""
import ctypes as C

import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spla

import gridgen


@pytest.fixture(scope="module")
def lib():
    from paper_1511_04519_gb300 import build
    build.build()
    from paper_1511_04519_gb300 import matex
    return matex.lib()


def _grid(layers, nx, ny):
    return gridgen.small_mesh(7, nx=nx, ny=ny, layers=layers, n_src=2, n_pads=2)


def _ptr(a, t):
    return a.ctypes.data_as(C.POINTER(t))


def _walk(lib, n, rp, ci, v, shift, alpha, width, version, cluster, b):
    x = np.zeros_like(b)
    info = np.zeros(4, np.int64)
    st = lib.matex_host_tensor_plan(
        C.c_int64(n), _ptr(rp, C.c_int64), _ptr(ci, C.c_int32), _ptr(v, C.c_double),
        _ptr(shift, C.c_double) if shift is not None else None, C.c_double(alpha), C.c_int32(width),
        C.c_int32(version), C.c_int32(cluster), C.c_int32(b.shape[0]), _ptr(b, C.c_double),
        _ptr(x, C.c_double), _ptr(info, C.c_int64))
    return st, x, info


@pytest.mark.parametrize("version", [0, 1])
@pytest.mark.parametrize("layers,nx,ny,width,cluster", [
    (1, 2, 2, 0, 1), (1, 7, 5, 0, 1), (1, 32, 32, 0, 2), (2, 23, 41, 0, 4), (3, 30, 29, 0, 8),
    (2, 40, 40, 24, 3), (1, 61, 3, 0, 1), (4, 20, 20, 130, 2)])
def test_plan_solves(lib, layers, nx, ny, width, cluster, version):
    p = _grid(layers, nx, ny) if nx * ny >= 4 else None
    G = p.G()
    rp, ci, v = (np.ascontiguousarray(a) for a in (p.g_rowptr, p.g_col, p.g_val))
    b = np.random.default_rng(3).standard_normal((3, p.n))
    st, x, info = _walk(lib, p.n, rp, ci, v, p.c, p.gamma, width, version, cluster, b)
    assert st == 0 and info[3] == 0, info
    A = (sp.diags(p.c) + p.gamma * G).tocsc()
    ref = spla.splu(A).solve(b.T).T
    assert np.abs(x - ref).max() <= 1e-10 * np.abs(ref).max()
    if layers >= 3:
        assert info[2] > 0  # reductions of several chunks


def test_single_node_and_disconnected(lib):
    # one node; and five that touch no other (five roots)
    for n in (1, 5):
        rp = np.arange(n + 1, dtype=np.int64)
        ci = np.arange(n, dtype=np.int32)
        v = np.linspace(1.0, 2.0, n)
        b = np.arange(1.0, n + 1.0)[None]
        st, x, info = _walk(lib, n, rp, ci, v, None, 1.0, 0, 1, 1, b)
        assert st == 0 and info[3] == 0
        assert np.allclose(x, b / v, rtol=1e-15)


def test_bad_arguments(lib):
    rp, ci, v, b = np.arange(2, dtype=np.int64), np.zeros(1, np.int32), np.ones(1), np.ones((1, 1))
    assert _walk(lib, 1, rp, ci, v, None, 1.0, 0, 2, 1, b)[0] == 1
    assert _walk(lib, 1, rp, ci, v, None, 1.0, 0, 0, 9, b)[0] == 1
