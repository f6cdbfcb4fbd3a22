"""ugks_residual and ugks_residual_sums of one step against the states before and
after it, at cell counts around the units their sums are formed in."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2412_06546_gb300 import _lib, cases as cs  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2412_06546_gb300 import build
    build.build()


@pytest.mark.parametrize("nx,ny", [(1, 1), (31, 1), (8, 4), (33, 1), (128, 64), (256, 256), (65537, 1), (400, 300)])
def test_residual_of_one_step(nx, ny):
    """Partials of 32 cells, folded by eight above 2,048 of them, 512 threads over
    them in ugks_residual: 1 cell to 120,000."""
    mesh = cs.quad_mesh(nx, ny, left=("wall", 0), right=("wall", 0), bottom=("wall", 0), top=("wall", 0))
    g = _lib.Case(mesh, cs.cartesian_vgrid((6, 5), (-5, -5), (5, 5)),
                  cs.params(0.5, walls=[{"T": 1.4, "U": [0.5, 0, 0]}]), cs.smooth_state(mesh, 3, 0.2), patch_cells=16)
    assert np.all(g.residual() == 0.0) and np.all(g.residual_sums() == 0.0)
    f, W0 = g.state()
    g.set_state(f * cs.perturbation(f.shape, 7, 0.2), W0)
    g.step(1)
    _, W1 = g.state(with_f=False)
    s, r = g.residual_sums(), g.residual()
    g.close()
    # W1 - W0 carries the rounding of W1 where the step's own sum does not: 1e-16 |W| of
    # changes that the perturbation makes no smaller than 1e-5 |W| in the root mean square
    assert np.allclose(s, np.concatenate([((W1 - W0) ** 2).sum(0), (W0 ** 2).sum(0)]), rtol=1e-9, atol=1e-25)
    assert np.allclose(r, np.sqrt(s[:4]) / np.sqrt(s[4:]), rtol=1e-13, atol=0)
