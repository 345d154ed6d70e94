"""Tensor-core recombination of columns that differ by more than the digits of one
exponent hold, against the FP64 kernel on the same run: a column with an
inf or NaN among finite ones, a column of small currents beside one of large
ones."""
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


@pytest.mark.parametrize("tail_eps", [0.0, 1e-12])
@pytest.mark.parametrize("bad", [-1e290, -1e300])
def test_non_finite_column_keeps_to_its_outputs(M, bad, tail_eps):
    """The group that starts last gets a current whose response overflows (at
    -1e290 its norm, at -1e300 its slope already): the outputs before
    its start, which share rounds and tiles with it, stay finite (both kernels
    sum the same products: 1e-13 V there), those from its start on are not."""
    p = gridgen.small_mesh(65, nx=60, ny=55, layers=2, n_src=40, group_templates=[1] * 20, t_end=3e-9,
                           dt_out=5e-12)
    clean = M.Sim(p, resident="off", tail_eps=tail_eps)
    clean.run()
    m = clean.m_sequence()
    if tail_eps == 0.0:
        assert clean.stats.tc_rounds > 0
    first = np.asarray(p.pwl_t)[np.asarray(p.pwl_off)[:-1]]
    start = np.array([first[np.asarray(p.src_group) == g].min() for g in range(p.n_groups)])
    late = int(np.argmax(start))
    v = np.array(p.pwl_v, dtype=np.float64)
    s = int(np.flatnonzero(np.asarray(p.src_group) == late)[0])
    v[p.pwl_off[s] + 1] = bad
    X = [M.Sim(p, resident="off", recombine=r, replay_m=m, tail_eps=tail_eps).run_host(v)
         for r in ("auto", "fp64")]
    ok = [np.isfinite(x) for x in X]
    assert np.array_equal(ok[0], ok[1])
    before = np.arange(X[0].shape[0]) * p.dt_out < start[late]
    assert before.sum() > 20 and ok[0][before].all() and not ok[0][~before][1:].any()
    assert np.abs(X[0][before] - X[1][before]).max() <= 1e-13 * p.vdd


@pytest.mark.parametrize("ratio", [1.0, 1e-6, 1e-12])
def test_small_currents_beside_large_ones(M, ratio):
    """Two groups with the same pulse at the ends of a long strip with pads along
    it, one of them scaled by ratio, no DC part: each end has its own group's
    response, the other one's is 1e-20 there and less.  At every node the two
    kernels (on FP64 solves) agree to 1e-13 of what their terms there are: about
    40 terms of either, each off by 2^-53 of the largest, which is |z| + L |z'| +
    |w| of Eq. 5/6 or a few times that for a basis vector."""
    import scipy.sparse.linalg as spla
    q = gridgen.small_mesh(66, nx=400, ny=12, layers=1, n_src=2, group_templates=[1], n_pads=60, t_end=2e-9)
    nodes, peak = [5, q.n - 6], [1e-2, 1e-2 * ratio]
    t = np.array([50e-12, 90e-12, 160e-12])
    p = gridgen.with_sources(q, nodes, [0, 3, 6], np.tile(t, 2),
                             [0, -peak[0], 0, 0, -peak[1], 0], [0, 1], 2)
    lu = spla.splu(p.G().tocsc())
    terms = np.zeros(p.n)
    for node, i in zip(nodes, peak):
        e = np.zeros(p.n)
        e[node] = i
        z = np.abs(lu.solve(e))
        terms += 2.0 * z + np.abs(lu.solve(p.c * z)) / np.diff(t).min()
    kw = dict(resident="off", tc_solve="off", include_dc=False)
    a = M.Sim(p, **kw)
    Xa = a.run().cpu().numpy()
    Xb = M.Sim(p, recombine="fp64", replay_m=a.m_sequence(), **kw).run().cpu().numpy()
    worst = (np.abs(Xa - Xb).max(axis=0) / terms).max()
    assert worst <= 1e-13, worst
