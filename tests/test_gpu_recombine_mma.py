"""Tensor-core recombination (V y and -P as one contraction of FP16 digits)
against the FP64 kernel on the same run, at the edges of its tiles: node counts
around 8 and 32, output counts around 16, more K steps than one launch takes,
segments of a few outputs beside long ones, one group at a time, no DC part (so
that the small load response stands alone), tail skipping.

Both sum the same products, rounded at 2^-53 of the largest term or below, at
most a few hundred terms of at most 1 V: 1e-13 V; with tail skipping both stay
within eps per group of the exact run."""
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


def _both(M, p, serial=False, **kw):
    a = M.Sim(p, resident="off", **kw)
    a.one_group_at_a_time(serial)
    Xa = a.run().cpu().numpy()
    Xr = a.run().cpu().numpy()  # graph replay
    b = M.Sim(p, resident="off", recombine="fp64", replay_m=a.m_sequence(), **kw)
    Xb = b.run().cpu().numpy()
    assert np.abs(Xa - Xr).max() <= 1e-13
    return Xa, Xb, a


@pytest.mark.parametrize("nx,ny,layers,outputs", [(41, 43, 2, 15), (64, 61, 1, 16), (73, 57, 2, 17),
                                                  (91, 89, 1, 401)])
def test_node_and_output_edges(M, nx, ny, layers, outputs):
    p = gridgen.small_mesh(61, nx=nx, ny=ny, layers=layers, n_src=60, group_templates=[2, 1, 3] * 10,
                           t_end=outputs * 10e-12, dt_out=10e-12)
    Xa, Xb, _ = _both(M, p, include_dc=False)
    assert np.abs(Xa - Xb).max() <= 1e-13
    # the response alone: relative to its own size as well
    assert np.abs(Xa - Xb).max() <= 1e-11 * np.abs(Xb).max()


def test_more_steps_than_one_launch(M):
    p = gridgen.small_mesh(62, nx=45, ny=47, layers=1, n_src=260, group_templates=[1] * 260,
                           t_end=0.4e-9, dt_out=5e-12, start_hi=0.02e-9)
    p.tol = 1e-11
    Xa, Xb, a = _both(M, p)
    assert (a.stats.sum_m + 2 * 260 * a.stats.rounds) > 56 * 16 * a.stats.rounds
    assert np.abs(Xa - Xb).max() <= 1e-13


def test_one_group_at_a_time(M):
    p = gridgen.small_mesh(63, nx=95, ny=93, layers=1, n_src=9, group_templates=[1, 2, 3], t_end=3e-9)
    Xa, Xb, _ = _both(M, p, serial=True)
    assert np.abs(Xa - Xb).max() <= 1e-13


def test_tail_cut(M):
    p = gridgen.small_mesh(64, nx=60, ny=50, layers=2, n_src=40, group_templates=[1] * 40, t_end=4e-9)
    eps = 1e-10
    Xa, Xb, _ = _both(M, p, tail_eps=eps)
    exact = M.Sim(p, resident="off").run().cpu().numpy()
    assert np.abs(Xa - exact).max() <= eps * p.n_groups
    assert np.abs(Xb - exact).max() <= eps * p.n_groups
