"""Gram-Schmidt of the batched rounds (four launches over all columns) at the
edges of its node chunks (512 nodes and halves of 8192) and of its basis sizes
(1 to 10, two nodes per thread up to 8), against the resident rounds, which sum
the same products in another order: 1e-12 V for responses of at most 1 V."""
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


@pytest.mark.parametrize("nx,ny", [(7, 73), (16, 32), (27, 19), (31, 33), (32, 32), (9, 7)])
def test_against_resident_rounds(M, nx, ny):
    p = gridgen.small_mesh(71, nx=nx, ny=ny, n_src=12, group_templates=[2, 1, 3, 1])
    first = M.Sim(p, resident="on")
    first.run()
    n_seg = len(first.m_sequence())
    m = np.array([1 + k % 10 for k in range(n_seg)], dtype=np.int32)
    a = M.Sim(p, resident="on", replay_m=m)
    Xa = a.run().cpu().numpy()
    b = M.Sim(p, resident="off", replay_m=m)
    Xb = b.run().cpu().numpy()
    assert a.stats.resident == 1 and b.stats.resident == 0
    assert b.stats.max_m == a.stats.max_m
    assert np.abs(Xa - Xb).max() <= 1e-12 * p.vdd


def test_wide_round_with_full_chunks(M):
    # 64 columns of 78,961 nodes: blocks of 4096 nodes, the last one partly filled
    p = gridgen.small_mesh(72, nx=281, ny=281, n_src=64, group_templates=[1] * 64)
    a = M.Sim(p, resident="off")
    Xa = a.run().cpu().numpy()
    # one group at a time: the same columns in blocks of 512 nodes
    b = M.Sim(p, resident="off", replay_m=a.m_sequence())
    b.one_group_at_a_time(True)
    Xb = b.run().cpu().numpy()
    assert np.abs(Xa - Xb).max() <= 1e-12 * p.vdd
