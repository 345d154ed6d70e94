"""What the digits of the tensor-core solves keep: 55 bits below the largest entry of
a panel row and of a right-hand side over 128 terms.  A solution is then accurate
relative to its largest entry, on responses that fall over 8 to 50 decades as on
flat ones: each of about 15 levels is off by at most 128 terms of 2^-54 of the
largest product, in the mean square by some units of 1e-16 in all, bounded at
1e-14 of the largest entry.  Entries far below it keep the digits that this
leaves; with tc_solve off they keep all (every product of a dominant matrix and
a right-hand side of one sign has that sign)."""
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


@pytest.mark.parametrize("layers,nx,ny,gamma", [(1, 400, 12, 1e-13), (1, 400, 12, 1e-11), (1, 110, 100, 1e-13),
                                                (2, 100, 100, 1e-11)])
@pytest.mark.parametrize("which", [0, 1])
def test_graded_solutions(M, layers, nx, ny, gamma, which):
    import torch
    p = gridgen.small_mesh(66, nx=nx, ny=ny, layers=layers, n_src=2, group_templates=[1, 1], n_pads=2)
    p.gamma = gamma
    b = np.zeros((5, p.n))
    b[0, 5] = b[1, p.n // 2] = b[2, p.n - 3] = 1.0
    b[3, 5], b[3, p.n - 6] = 1.0, 1e-12          # a small one far from a large one
    b[4] = 10.0 ** -np.linspace(0.0, 30.0, p.n)  # graded within every supernode
    b = torch.from_numpy(b).cuda()
    on = M.Sim(p, tc_solve="on", resident="off").solve(which, b)
    off = M.Sim(p, tc_solve="off", resident="off").solve(which, b)
    size = off.abs().max(dim=1, keepdim=True).values
    assert float(((on - off).abs() / size).max()) <= 1e-14
    # the FP64 kernels entry by entry, against the persistent ones' other order
    alt = M.Sim(p, tc_solve="off", solve_mode=0, resident="off").solve(which, b)
    assert float(((alt - off).abs() / off.abs()).max()) <= 1e-12
