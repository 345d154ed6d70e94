"""Gram-Schmidt of the batched rounds at its larger basis sizes (11 to 20, one node
per thread), and columns whose norm overflows, against the resident rounds: the
same products in another order, 1e-12 V for responses of at most 1 V (columns
of more dimensions than they need are orthogonalised against rounding noise,
which the Hessenberg matrix leaves out at breakdown)."""
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


@pytest.mark.parametrize("nx,ny", [(31, 33), (40, 41)])
def test_bases_of_up_to_twenty(M, nx, ny):
    # time constants over four decades, so that twenty vectors are independent
    p = gridgen.small_mesh(73, nx=nx, ny=ny, n_src=12, group_templates=[2, 1, 3, 1], c_range=(1e-15, 1e-11))
    first = M.Sim(p, resident="on")
    first.run()
    m = np.array([11 + k % 10 for k in range(len(first.m_sequence()))], dtype=np.int32)
    a = M.Sim(p, resident="on", replay_m=m)
    Xa = a.run().cpu().numpy()
    b = M.Sim(p, resident="off", replay_m=m)
    Xb = b.run().cpu().numpy()
    assert a.stats.resident == 1 and b.stats.resident == 0
    assert a.stats.max_m == b.stats.max_m == 20
    assert np.abs(Xa - Xb).max() <= 1e-12 * p.vdd


@pytest.mark.parametrize("bad", [-1e290, -1e300])
def test_overflowing_column(M, bad):
    """One group's response overflows: the same outputs are finite on both paths."""
    p = gridgen.small_mesh(74, nx=20, ny=19, n_src=8, group_templates=[1] * 8, t_end=2e-9)
    m = np.full(M.Sim(p).n_segments, 3, np.int32)
    v = np.array(p.pwl_v, dtype=np.float64)
    v[1] = bad
    X = [M.Sim(p, resident=r, replay_m=m).run_host(v) for r in ("on", "off")]
    ok = [np.isfinite(x) for x in X]
    assert np.array_equal(ok[0], ok[1])
    assert ok[0][0].all() and not ok[0][-1].any()
    assert np.abs(X[0][ok[0]] - X[1][ok[0]]).max() <= 1e-12 * p.vdd
