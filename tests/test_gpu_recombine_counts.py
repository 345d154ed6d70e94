"""matex_stats counts what ran: every round whose recombination ran on the tensor
cores, exact, with tail skipping and one group at a time, on the grids whose
results the other tests compare with the FP64 kernel; and the supernodes of the
tensor-core solves."""
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


def _edge(nx, ny, layers, outputs):
    return dict(seed=61, nx=nx, ny=ny, layers=layers, n_src=60, group_templates=[2, 1, 3] * 10,
                t_end=outputs * 10e-12, dt_out=10e-12)


GRIDS = {
    "15 outputs": (_edge(41, 43, 2, 15), {}),
    "16 outputs": (_edge(64, 61, 1, 16), {}),
    "17 outputs": (_edge(73, 57, 2, 17), {}),
    "401 outputs": (_edge(91, 89, 1, 401), {}),
    "260 groups": (dict(seed=62, nx=45, ny=47, layers=1, n_src=260, group_templates=[1] * 260, t_end=0.4e-9,
                        dt_out=5e-12, start_hi=0.02e-9), {}),
    "tail": (dict(seed=64, nx=60, ny=50, layers=2, n_src=40, group_templates=[1] * 40, t_end=4e-9),
             dict(tail_eps=1e-10)),
    "serial": (dict(seed=63, nx=95, ny=93, layers=1, n_src=9, group_templates=[1, 2, 3], t_end=3e-9), {}),
}


@pytest.mark.parametrize("name", GRIDS)
def test_rounds_on_the_tensor_cores(M, name):
    kw, opts = GRIDS[name]
    p = gridgen.small_mesh(kw["seed"], **{k: v for k, v in kw.items() if k != "seed"})
    counts = {}
    for path in ("auto", "fp64"):
        sim = M.Sim(p, resident="off", recombine=path, **opts)
        sim.one_group_at_a_time(name == "serial")
        sim.run()
        counts[path] = sim.stats.tc_rounds
        sim.run()
        assert sim.stats.graph_replay == 0 or sim.stats.tc_rounds == counts[path]
    assert counts["auto"] > 0 and counts["fp64"] == 0, counts


def test_supernodes_of_the_plan(M):
    p = gridgen.small_mesh(75, nx=20, ny=18, layers=1, n_src=4)  # none 64 columns wide
    assert M.Sim(p, tc_solve="on").setup_stats()["tc_solve_supernodes"] > 1
    assert M.Sim(p, tc_solve="off").setup_stats()["tc_solve_supernodes"] == 0
