"""Resident rounds on the largest grids that they take, where one work area for the
small dense steps fits beside the plan and the exponentials run one after another
on one warp: against the batched rounds with the same Krylov dimensions (the
same products in another order, 1e-12 V), for columns of one output interval
or less, of several, and of many outputs."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("dt_out", [5e-12, 40e-12, 150e-12])
def test_one_work_area(M, dt_out):
    # 3,042 nodes in two layers: 223 KB of shared memory with one work area, 268 with three
    p = gridgen.small_mesh(91, nx=39, ny=39, layers=2, n_src=12, group_templates=[2, 1, 3], t_end=1.2e-9,
                           dt_out=dt_out, start_hi=0.8e-9)
    a = M.Sim(p, resident="on")
    Xa = a.run().cpu().numpy()
    assert a.stats.resident == 1 and a.stats.max_m > 1
    Xb = M.Sim(p, resident="off", replay_m=a.m_sequence()).run().cpu().numpy()
    assert np.abs(Xa - Xb).max() <= 1e-12 * p.vdd
