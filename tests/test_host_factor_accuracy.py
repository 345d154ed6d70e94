"""Accuracy of the factors that every solve uses, on the CPU: the solutions of the
fine structure's panels and of the tensor-core plan's larger ones against
iteratively refined ones (residuals in extended precision).

On a dominant matrix all pivots and row sums add values of one sign, so the
solution carries only the roundings along the elimination tree, about 15
supernodes of 4 roundings of 0.3 2^-53 each, 3e-16 root mean square: bounded at
8e-16.  (Pivots by subtraction from the diagonal gave 1.7e-15 to 4.2e-15, and the
larger panels up to 1.3 times more than the fine ones.)  Other SPD matrices are
eliminated by subtraction: 1e-12 on these condition numbers."""
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


def _ptr(a, t):
    return a.ctypes.data_as(C.POINTER(t))


def _solve(lib, A, shift, alpha, b, plan):
    """x of (diag(shift) + alpha A) x = b by the fine panels, or by the plan's."""
    A = sp.csr_matrix(A)
    A.sort_indices()
    rp, ci, v = A.indptr.astype(np.int64), A.indices.astype(np.int32), A.data.astype(np.float64)
    x, info = np.zeros_like(b), np.zeros(8, np.int64)
    head = [C.c_int64(A.shape[0]), _ptr(rp, C.c_int64), _ptr(ci, C.c_int32), _ptr(v, C.c_double),
            _ptr(shift, C.c_double) if shift is not None else None, C.c_double(alpha), C.c_int32(1024)]
    tail = [C.c_int32(b.shape[0]), _ptr(b, C.c_double), _ptr(x, C.c_double), _ptr(info, C.c_int64)]
    f = lib.matex_host_tensor_plan if plan else lib.matex_host_factor_solve
    st = f(*head, *([C.c_int32(1), C.c_int32(1)] if plan else []), *tail)
    return st, x


def _refined(A, shift, alpha, b):
    # alpha times the entries rounds as the factorisation has it; the diagonal's
    # two parts are kept apart
    M = sp.csr_matrix(A)
    M.sort_indices()
    M.data = alpha * M.data
    shift = np.zeros(M.shape[0]) if shift is None else shift
    lu = spla.splu((M + sp.diags(shift)).tocsc())
    val, sl = M.data.astype(np.longdouble), shift.astype(np.longdouble)
    x = np.zeros(b.shape, np.longdouble)
    for _ in range(4):
        r = np.stack([bq - np.add.reduceat(val * xq[M.indices], M.indptr[:-1]) - sl * xq for bq, xq in zip(b, x)])
        x = x + lu.solve(r.astype(np.float64).T).T
    return x


def _error(x, ref):
    return float(np.sqrt(((x - ref) ** 2).sum() / (ref ** 2).sum()))


@pytest.mark.parametrize("layers,nx,ny", [(1, 32, 32), (1, 100, 101), (2, 60, 57), (4, 40, 40)])
@pytest.mark.parametrize("which", ["M", "G"])
def test_grids(lib, layers, nx, ny, which):
    p = gridgen.small_mesh(9, nx=nx, ny=ny, layers=layers, n_src=3)
    rng = np.random.default_rng(nx)
    if which == "M":
        shift, alpha = p.c, p.gamma
        b = p.c * rng.standard_normal((4, p.n))
    else:
        shift, alpha = None, 1.0
        b = -rng.uniform(0.0, 1e-2, (4, p.n)) * (rng.random((4, p.n)) < 0.05)
    ref = _refined(p.G(), shift, alpha, b)
    for plan in (False, True):
        st, x = _solve(lib, p.G(), shift, alpha, b, plan)
        assert st == 0
        assert _error(x, ref) <= 8e-16, plan


@pytest.mark.parametrize("kind", ["positive entries", "not dominant"])
def test_other_spd_matrices(lib, kind):
    p = gridgen.small_mesh(9, nx=40, ny=37, layers=2, n_src=3)
    G = sp.csr_matrix(p.G())
    rng = np.random.default_rng(4)
    if kind == "positive entries":
        s = sp.diags(rng.choice([-1.0, 1.0], p.n))
        G = s @ G @ s
    else:  # a scaling of the unknowns: same signs, rows of either sum
        s = sp.diags(rng.uniform(0.2, 2.0, p.n))
        G = s @ G @ s
    b = rng.standard_normal((2, p.n))
    ref = _refined(G, None, 1.0, b)
    for plan in (False, True):
        st, x = _solve(lib, G, None, 1.0, b, plan)
        assert st == 0
        assert _error(x, ref) <= 1e-12


def test_indefinite_is_refused(lib):
    # dominant off-diagonals, a row that sums to less than zero
    G = sp.csr_matrix(np.array([[1.0, -2.0], [-2.0, 1.0]]))
    for plan in (False, True):
        assert _solve(lib, G, None, 1.0, np.ones((1, 2)), plan)[0] == 2
