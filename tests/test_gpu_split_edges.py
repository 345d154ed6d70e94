"""Edges of the digit split of the tensor-core solves: mantissas just below a power of
two, where rounding or the leading digit would run over (all of them in one
chunk, with both signs), the ends of the exponent range, and values next to
them.  On a diagonal matrix of powers of two either substitution rounds a lone
product to a whole number of at least 2^51.98: 2^-51.98 in all; on a grid the
path agrees with the FP64 kernels to 1e-14 of the largest entry (15 levels of a
few units of 2^-53)."""
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


def _mantissas(rng, n):
    near = [2.0 - 2.0 ** -k for k in range(1, 53)] + [1.0 + 2.0 ** -k for k in range(1, 53)]
    near += [1.984375, np.nextafter(1.984375, 0), 127.5 / 64, 127 / 64, 1.0]
    return rng.choice(near, n) * rng.choice([-1.0, 1.0], n)


@pytest.mark.parametrize("scale", [0, -1020, 1022, -500, 700])
def test_diagonal_matrix(M, scale):
    import torch
    n = 500
    rng = np.random.default_rng(scale + 2000)
    d = 2.0 ** rng.integers(0, 2, n)
    p = gridgen.small_mesh(3, nx=20, ny=25, n_src=2)
    p.g_rowptr, p.g_col, p.g_val = np.arange(n + 1, dtype=np.int64), np.arange(n, dtype=np.int32), d
    sim = M.Sim(p, tc_solve="on", resident="off")
    b = np.stack([_mantissas(rng, n) for _ in range(9)]) * 2.0 ** scale
    x = sim.solve(1, torch.from_numpy(b).cuda()).cpu().numpy()
    assert (np.abs(x - b / d) <= 2.0 ** -51.98 * np.abs(b / d)).all()


@pytest.mark.parametrize("layers,nx,ny", [(1, 40, 41), (2, 45, 44)])
@pytest.mark.parametrize("kind", ["near two", "just below two", "powers of two"])
def test_grid(M, layers, nx, ny, kind):
    import torch
    p = gridgen.small_mesh(97, nx=nx, ny=ny, layers=layers, n_src=3)
    rng = np.random.default_rng(nx)
    b = {"near two": lambda: np.stack([_mantissas(rng, p.n) for _ in range(10)]),
         "just below two": lambda: np.full((10, p.n), np.nextafter(2.0, 0.0)),
         "powers of two": lambda: np.full((10, p.n), 2.0 ** 52)}[kind]()
    b = torch.from_numpy(b).cuda()
    on, off = (M.Sim(p, tc_solve=t, resident="off") for t in ("on", "off"))
    for which in (0, 1):
        x, y = on.solve(which, b), off.solve(which, b)
        assert float(((x - y).abs().max(dim=1).values / y.abs().max(dim=1).values).max()) <= 1e-14
