"""The flux pass where the last velocity tile of a row or of a chunk is short (a
tile of 128 on rows padded to 64), and over several chunks of the flux buffer,
against the oracle."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2412_06546_gb300 import _lib, cases as cs  # noqa: E402
import test_gpu_flux_pass as flux  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2412_06546_gb300 import build
    build.build()


def _meshes():
    tri = cs.cylinder_case(n_cells=700, nvx=4, nvy=4, mach=2.0)
    quads = cs.quad_mesh(9, 7)
    return {"walls and far field": (tri["mesh"], tri["params"]), "periodic": (cs.periodic_tri_mesh(8, 7), cs.params(0.1)),
            "quadrilaterals": (quads, cs.params(0.1)), "any face count": (flux.merged(quads, 2, 7, 6), cs.params(0.1))}


@pytest.mark.parametrize("precision", [_lib.FP64, _lib.FP32])
@pytest.mark.parametrize("nv", [(24, 24), (8, 8), (20, 15)])
@pytest.mark.parametrize("kind", ["walls and far field", "periodic", "quadrilaterals", "any face count"])
def test_short_last_tile(kind, nv, precision):
    """576, 64 and 320 padded velocities in tiles of 128: half a tile at the end,
    or half a tile in all."""
    mesh, params = _meshes()[kind]
    vg = cs.cartesian_vgrid(nv, (-6.0, -6.0), (6.0, 6.0))
    info = flux._compare(mesh, vg, dict(params, walls=flux.WALL), precision, patch_cells=16, vtile=128)
    assert info["vtile"] == 128 and info["nv_pad"] % 128 == 64


@pytest.mark.parametrize("precision,vtile,group", [(_lib.FP32, 128, 0), (_lib.FP64, 128, 0), (_lib.FP32, 64, 3),
                                                   (_lib.FP64, 32, 9), (_lib.FP32, 32, 1024)])
def test_several_chunks(precision, vtile, group):
    """1,472 padded velocities in two chunks or more (the last one shorter, and for
    tiles of 128 ending in half a tile): ten launches of the step and two per chunk."""
    c = cs.cylinder_case(n_cells=900, nvx=46, nvy=32, mach=2.0)
    info = flux._compare(c["mesh"], c["vgrid"], dict(c["params"], walls=flux.WALL), precision, patch_cells=16,
                         vtile=vtile, tile_group=group)
    assert info["n_wall_faces"] > 0 and info["nv_pad"] == 1472
    assert info["kernel_launches_per_step"] >= 10 + 2 * 2
