"""Velocity sets that cannot carry a slope system are reported, not answered."""
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


@pytest.mark.parametrize("precision", [_lib.FP64, _lib.FP32])
@pytest.mark.parametrize("n", [2, 3, 5, 8])
@pytest.mark.parametrize("dim", [2, 3])
def test_velocities_in_one_plane_fail(dim, n, precision):
    """Velocities on a line (2D) or in a plane (3D): the moment matrix of every face
    is singular, so that rounding makes a pivot of some face negative; ugks_check
    reports a numeric failure after one step."""
    rng = np.random.default_rng(10 * n + dim)
    mesh = cs.periodic_tri_mesh(6, 5) if dim == 2 else cs.hex_mesh(4, 4, 3)
    n = n ** (dim - 1)
    axes = np.linalg.qr(rng.normal(size=(dim, dim)))[0][:dim - 1]
    u = rng.uniform(-3.0, 3.0, size=(n, dim - 1)) @ axes + 0.5 * rng.normal(size=dim)
    vg = {"dim": dim, "u": u, "w": np.full(n, 6.0 ** dim / n), "cart_n": [0, 0, 0]}
    walls = [{"T": 1.0, "U": [0.0, 0.0, 0.0]}]
    g = _lib.Case(mesh, vg, cs.params(0.1, walls=walls), cs.smooth_state(mesh, 3, 0.1), precision=precision,
                  patch_cells=16)
    g.step(1)
    with pytest.raises(Exception, match="non-finite or non-positive"):
        g.check()
    g.close()
