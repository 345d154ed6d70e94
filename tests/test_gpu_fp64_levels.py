"""The FP64 level kernels (tc_solve off, and where the tensor-core tiles do not fit
memory): every column block, the chunked reductions of wide supernodes, and the
persistent launch, at column counts that the default solves put on the tensor
cores.  Same products in another order: 1e-13 of a run's voltages, 1e-12 of a
solution's largest entry."""
import numpy as np
import pytest
import scipy.sparse as sp

import gridgen
from oracle import rmatex_ref as R
from tests.parity_util import oracle_m

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


@pytest.mark.parametrize("col_block", [2, 4, 8])
def test_column_blocks_agree(M, col_block):
    p = gridgen.small_mesh(8, nx=20, ny=20, layers=2, n_src=24, group_templates=[2] * 12, t_end=0.3e-9)
    base = M.Sim(p, col_block=1, resident="off", tc_solve="off").run().cpu().numpy()
    sim = M.Sim(p, col_block=col_block, resident="off", tc_solve="off")
    X = sim.run().cpu().numpy()
    assert sim.setup_stats()["tc_solve_min_cols"] == 0
    assert np.abs(X - base).max() <= 1e-13


@pytest.mark.parametrize("which", [0, 1])
def test_chunked_level_solves_on_the_bench_grid(M, which):
    import torch
    p = gridgen.config1()
    sim = M.Sim(p, solve_mode=1, tc_solve="off", include_dc=False, rows=np.arange(4, dtype=np.int32))
    A = sp.csr_matrix(sp.diags(p.c) + p.gamma * p.G()) if which == 0 else p.G()
    rng = np.random.default_rng(21)
    for ncols in (2, 5, 16, 64):
        b = torch.from_numpy(rng.standard_normal((ncols, p.n))).cuda()
        x = sim.solve(which, b)
        xu = torch.empty_like(b)
        M.matex_solve_noalloc(sim.ctx, which, ncols, b.data_ptr(), xu.data_ptr())  # unchunked
        torch.cuda.synchronize()
        xn, bn, xun = x.cpu().numpy(), b.cpu().numpy(), xu.cpu().numpy()
        for q in range(ncols):
            r = np.abs(A @ xn[q] - bn[q]).max()
            assert r <= 1e-11 * max(np.abs(bn[q]).max(), np.abs(A).max() * np.abs(xn[q]).max()), (ncols, q)
            assert np.abs(xn[q] - xun[q]).max() <= 1e-12 * np.abs(xun[q]).max(), (ncols, q)


@pytest.mark.parametrize("mode", [0, 1])
def test_persistent_and_level_solves_agree(M, mode):
    p = gridgen.small_mesh(13, nx=30, ny=30, layers=2, n_src=20, group_templates=[5] * 4, t_end=0.3e-9)
    ref = R.rmatex(p)
    sim = M.Sim(p, solve_mode=mode, tc_solve="off", replay_m=oracle_m(ref), resident="off")
    assert np.abs(sim.run().cpu().numpy() - ref.X).max() <= 1e-9 * p.vdd


@pytest.mark.parametrize("ncols", [2, 8, 13])
def test_column_blocks_of_single_solves(M, ncols):
    import torch
    p = gridgen.small_mesh(76, nx=37, ny=41, layers=2, n_src=16, group_templates=[1] * 16)
    b = torch.from_numpy(np.random.default_rng(ncols).standard_normal((ncols, p.n))).cuda()
    ref = M.Sim(p, col_block=1, solve_mode=1, tc_solve="off").solve(1, b)
    for kb in (2, 4, 8):
        x = M.Sim(p, col_block=kb, solve_mode=1, tc_solve="off").solve(1, b)
        assert (x - ref).abs().max() <= 1e-12 * ref.abs().max()
