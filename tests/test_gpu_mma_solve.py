"""Tensor-core level solves (FP16 digit products of an error-free split) against
the FP64 level solves and a sparse direct residual, at the edges of their tiles:
column counts around the 8- and 16-column halves of a block, grids whose
panels end inside a tile, both factors.

Tolerance: both paths round every product and sum at 2^-53 or below of the
largest term, so on condition numbers up to 1e4 they agree to about 1e-13 of a
column's largest entry; bounded at 1e-12, the residual at 1e-11."""
import numpy as np
import pytest
import scipy.sparse as sp

import gridgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_04519_gb300 import build
    build.build()
    from paper_1511_04519_gb300 import matex
    return matex


def _grid(layers, nx, ny):
    return gridgen.small_mesh(11, nx=nx, ny=ny, layers=layers, n_src=3, n_pads=4)


def _check(M, p, on, off, which, b):
    import torch
    x = on.solve(which, torch.from_numpy(b).cuda()).cpu().numpy()
    xf = off.solve(which, torch.from_numpy(b).cuda()).cpu().numpy()
    A = sp.csr_matrix(sp.diags(p.c) + p.gamma * p.G()) if which == 0 else p.G()
    for q in range(b.shape[0]):
        r = np.abs(A @ x[q] - b[q]).max()
        assert r <= 1e-11 * max(np.abs(b[q]).max(), np.abs(A).max() * np.abs(x[q]).max()), q
        assert np.abs(x[q] - xf[q]).max() <= 1e-12 * np.abs(xf[q]).max(), q


@pytest.mark.parametrize("layers,nx,ny", [(1, 2, 2), (1, 17, 9), (2, 31, 33), (3, 45, 40), (1, 120, 7)])
@pytest.mark.parametrize("ncols", [1, 2, 8, 9, 16, 17, 33])
def test_tile_edges(M, layers, nx, ny, ncols):
    p = _grid(layers, nx, ny) if nx * ny > 4 else gridgen.small_mesh(11, nx=2, ny=2, n_src=2, n_pads=2)
    on = M.Sim(p, tc_solve="on", resident="off")
    off = M.Sim(p, tc_solve="off", resident="off")
    assert on.setup_stats()["tc_solve_min_cols"] == 1
    rng = np.random.default_rng(ncols)
    for which in (0, 1):
        _check(M, p, on, off, which, rng.standard_normal((ncols, p.n)))


def test_refactored_capacitances(M):
    p = _grid(2, 30, 30)
    on, off = M.Sim(p, tc_solve="on", resident="off"), M.Sim(p, tc_solve="off", resident="off")
    c = p.c * np.random.default_rng(1).uniform(0.5, 2.0, p.n)
    on.set_caps(c)
    off.set_caps(c)
    p.c = c
    _check(M, p, on, off, 0, np.random.default_rng(2).standard_normal((5, p.n)))


def test_scales_zeros_and_non_finite_columns(M):
    """Columns far from 1 in size, zero columns and columns with an inf or a
    NaN: each column keeps to itself."""
    import torch
    p = _grid(2, 25, 27)
    on, off = M.Sim(p, tc_solve="on", resident="off"), M.Sim(p, tc_solve="off", resident="off")
    b = np.random.default_rng(5).standard_normal((9, p.n))
    b[0] *= 2.0 ** -900
    b[1] *= 2.0 ** 900
    b[2] = 0.0
    b[3, :] = 0.0
    b[3, 17] = 1e-3          # one entry: the response decays over many decades
    _check(M, p, on, off, 1, b)
    b[4, 3] = np.inf
    b[5, 8] = np.nan
    x = on.solve(1, torch.from_numpy(b).cuda()).cpu().numpy()
    assert not np.isfinite(x[4]).all() and not np.isfinite(x[5]).all()
    good = [0, 1, 2, 3, 6, 7, 8]
    assert np.isfinite(x[good]).all() and not x[2].any()


@pytest.mark.parametrize("ncols", [1, 8, 9, 40, 130])
def test_wide_separators(M, ncols):
    # a 512-column top and reductions of up to 32 K steps: clusters of 2 to 8 with
    # pieces of one chunk or several, the eight- and the four-warp kernel
    p = _grid(4, 50, 48)
    on = M.Sim(p, tc_solve="on", resident="off")
    off = M.Sim(p, tc_solve="off", resident="off")
    rng = np.random.default_rng(ncols)
    for which in (0, 1):
        _check(M, p, on, off, which, rng.standard_normal((ncols, p.n)))
