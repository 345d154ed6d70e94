"""Which rounds a default transient takes on the grids that fit both, and what new
inputs do there: the choice by the rounds' own time, the one run on resident
rounds in place of a plain run and a new recording, and the recording that stays
for the currents it was made with.

Both paths sum the same products in another order (1e-12 V with equal Krylov
dimensions); where new currents leave the dimensions to the run itself, a
residual within rounding of tol may move one segment: 10 tol."""
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


# single-layer and two-layer grids of the workloads measured in perf/cases.py: few
# columns in many rounds of one or two Arnoldi steps (resident rounds 0.80 to 0.84 of
# the batched ones' time at 3,000 nodes), many columns (1.2 to 1.4 times)
WORKLOADS = [
    dict(layers=1, nx=49, ny=67, n_src=415, groups=4, templates=8, steps=497),
    dict(layers=1, nx=55, ny=55, n_src=60, groups=1, templates=8, steps=600),
    dict(layers=2, nx=32, ny=32, n_src=60, groups=1, templates=8, steps=600),
    dict(layers=2, nx=39, ny=39, n_src=60, groups=24, templates=36, steps=600),
    dict(layers=1, nx=55, ny=55, n_src=72, groups=48, templates=72, steps=600),
]


@pytest.mark.parametrize("case", WORKLOADS, ids=lambda c: "%dx%dx%d-%dgroups" % (
    c["layers"], c["nx"], c["ny"], c["groups"]))
def test_default_run_is_the_faster_of_both(M, case):
    """Repeated runs and runs with new currents (after the first few): within 15 % of
    the faster of both paths (the runs of one path differ by 1 to 3 %; a wrong
    choice costs 20 % and more)."""
    import time
    import torch
    from perf import cases
    p = cases._run_grid(case, 3)
    ms = {}
    for mode in ("on", "off", "auto"):
        sim = M.Sim(p, resident=mode)
        out = torch.empty((sim.n_times, sim.n_rows), dtype=torch.float64, device="cuda")

        def timed(v=None):
            torch.cuda.synchronize()
            t = time.perf_counter()
            if v is not None:
                sim.set_sources(v)
            sim.run(out)
            return time.perf_counter() - t

        timed(), timed(), timed()
        repeated = min(timed() for _ in range(5))
        rng = np.random.default_rng(1)
        new = [timed(p.pwl_v * np.repeat(rng.uniform(0.5, 1.5, p.n_src), 3)) for _ in range(7)]
        ms[mode] = repeated, float(np.median(new[2:]))
    for k in range(2):
        assert ms["auto"][k] <= 1.15 * min(ms["on"][k], ms["off"][k]), ms


@pytest.fixture()
def batched_choice(M):
    """A context that fits the resident rounds and has chosen the batched ones (3,042
    nodes, many columns: 4.0 ms against 5.5 ms)."""
    p = gridgen.small_mesh(93, nx=39, ny=39, layers=2, n_src=60, group_templates=[1] * 24, t_end=3e-9)
    sim = M.Sim(p)
    assert sim.setup_stats()["resident"] == 0
    return p, sim


def _scaled(p, a):
    return np.asarray(p.pwl_v) * a[np.repeat(np.arange(p.n_src), np.diff(p.pwl_off))]


def test_new_currents_take_the_resident_rounds(M, batched_choice):
    p, sim = batched_choice
    first = sim.run().cpu().numpy()
    assert sim.stats.resident == 1  # nothing recorded yet
    for replay in (0, 1, 1):
        assert np.abs(sim.run().cpu().numpy() - first).max() <= 10 * p.tol
        assert (sim.stats.resident, sim.stats.graph_replay) == (0, replay)
    ref = M.Sim(p, resident="on")
    took = []
    for k in range(4):
        # from a hundredth to a hundred times: other Krylov dimensions
        v = _scaled(p, 10.0 ** np.random.default_rng(k).uniform(-2, 2, p.n_src))
        X, Y = sim.run_host(v), ref.run_host(v)
        took.append(sim.stats.resident)
        assert sim.stats.graph_replay == 1 - took[-1]
        if took[-1]:
            assert np.array_equal(X, Y)  # the same code on the same data
            assert np.array_equal(sim.m_sequence(), ref.m_sequence())
            assert sim.stats.sum_m == ref.stats.sum_m
        assert np.abs(X - Y).max() <= 10 * p.tol
    assert 1 in took and took == sorted(took)  # once they changed the counts, at once
    # the setup's currents again: new ones to this run, then the recording's own
    back = sim.run_host(p.pwl_v)
    assert sim.stats.resident == 1
    again = sim.run().cpu().numpy()
    assert sim.stats.resident == 0
    for X in (back, again):
        assert np.abs(X - first).max() <= 10 * p.tol


def test_new_capacitances(M, batched_choice):
    p, sim = batched_choice
    sim.run()
    c = p.c * np.random.default_rng(3).uniform(0.1, 10.0, p.n)
    sim.set_caps(c)
    X = sim.run().cpu().numpy()
    q = gridgen.with_sources(p, p.src_node, p.pwl_off, p.pwl_t, p.pwl_v, p.src_group, p.n_groups)
    q.c = c
    Y = M.Sim(q, resident="off").run().cpu().numpy()
    assert np.abs(X - Y).max() <= 10 * p.tol


def test_batch_and_serial_after_new_currents(M, batched_choice):
    """A batch records the context whatever was set before; one group at a time
    works on either path."""
    p, sim = batched_choice
    v = _scaled(p, 10.0 ** np.random.default_rng(9).uniform(-2, 2, p.n_src))
    Y = M.Sim(p, resident="on").run_host(v)
    sim.run()
    sim.set_sources(v)
    batch = M.Batch([sim])
    for _ in range(2):
        outs, _ms = batch.run()
        assert sim.stats.resident == 0
        assert np.abs(outs[0].cpu().numpy() - Y).max() <= 10 * p.tol
    batch.close()
    sim.set_sources(v)
    sim.one_group_at_a_time(True)
    assert np.abs(sim.run().cpu().numpy() - Y).max() <= 10 * p.tol
