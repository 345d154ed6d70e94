"""A context set up on a non-blocking side stream, with work of another stream in
between: the solves before and after new capacitances, 1 and 5 columns, equal
those of a context on the default stream.  Same kernels, the order of FP64
atomics apart, which condition numbers up to 1e4 carry to 1e-12 of the largest
entry."""
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


@pytest.mark.parametrize("tc_solve", ["on", "off"])
def test_side_stream_setup_and_new_capacitances(M, tc_solve):
    import torch
    p = gridgen.small_mesh(81, nx=70, ny=65, layers=2, n_src=8, group_templates=[1] * 8)
    c = p.c * np.random.default_rng(1).uniform(0.2, 5.0, p.n)
    b = torch.from_numpy(np.random.default_rng(2).standard_normal((5, p.n))).cuda()
    torch.cuda.synchronize()

    def solves(sim):
        out = [sim.solve(w, b[:k].contiguous()) for w in (0, 1) for k in (1, 5)]
        sim.set_caps(c)
        return out + [sim.solve(w, b[:k].contiguous()) for w in (0, 1) for k in (1, 5)]

    ref = solves(M.Sim(p, tc_solve=tc_solve, resident="off"))
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        got = solves(M.Sim(p, tc_solve=tc_solve, resident="off"))
    side.synchronize()
    for x, y in zip(got, ref):
        assert (x - y).abs().max() <= 1e-12 * y.abs().max()
    assert (ref[0] - ref[4]).abs().max() > 1e-3 * ref[0].abs().max()  # the capacitances matter
