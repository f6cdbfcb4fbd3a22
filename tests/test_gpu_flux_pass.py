"""The flux and stage-1 passes over the entry layouts, tiles and chunks they
distinguish, against the oracle: cells of 3 to 10 faces (kernels for 3, 4 and 6
entries per cell with padding entries, and the loop over any count), velocity
counts that end in a short tile, a short group and a short chunk."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2412_06546_gb300 import _lib, cases as cs  # noqa: E402

FP64_TOL, FP32_TOL = 1e-12, 1e-5     # of max |x|, the parity bars of the step


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2412_06546_gb300 import build
    build.build()
    oracle.build()


def merged(mesh, group, seed, pairs):
    """The mesh with `pairs` seeded clusters of `group` face-connected cells
    each merged into one cell that keeps all outer faces."""
    rng = np.random.default_rng(seed)
    fc, C = np.asarray(mesh["face_cells"]), len(mesh["cell_vol"])
    inner = np.asarray(mesh["face_type"]) == cs.INTERIOR
    nbrs = [[] for _ in range(C)]
    for a, b in fc[inner]:
        nbrs[a].append(b)
        nbrs[b].append(a)
    lab = np.arange(C)
    used = np.zeros(C, bool)
    done = 0
    for c in rng.permutation(C):
        cluster = [c]
        while len(cluster) < group:
            more = [n for x in cluster for n in nbrs[x] if not used[n] and n not in cluster]
            if not more:
                break
            cluster.append(more[0])
        if len(cluster) < group or used[c]:
            continue
        used[cluster] = True
        lab[cluster] = cluster[0]
        done += 1
        if done == pairs:
            break
    ids, new = np.unique(lab, return_inverse=True)
    vol = np.bincount(new, mesh["cell_vol"])
    xc = np.stack([np.bincount(new, mesh["cell_vol"] * mesh["cell_xc"][:, d]) / vol
                   for d in range(mesh["dim"])], 1)
    nfc = np.where(fc >= 0, new[np.maximum(fc, 0)], -1)
    keep = nfc[:, 0] != nfc[:, 1]
    out = {"dim": mesh["dim"], "cell_xc": xc, "cell_vol": vol, "face_cells": nfc[keep]}
    for k in ("face_n", "face_S", "face_xc", "face_type", "face_tag", "face_shift"):
        out[k] = np.asarray(mesh[k])[keep]
    return out


def _faces_per_cell(mesh):
    fc = np.asarray(mesh["face_cells"])
    return np.bincount(fc[fc >= 0])


def _compare(mesh, vg, pr, precision, **tiling):
    init = cs.smooth_state(mesh, 3, 0.1)
    o = oracle.OracleCase(mesh, vg, pr, init, n_threads=0)
    g = _lib.Case(mesh, vg, pr, init, precision=precision, **tiling)
    f, W, _ = o.state()
    f = (f * cs.perturbation(f.shape, 4, 0.05)).astype(np.float32).astype(np.float64)
    o.set_state(f, W)
    g.set_state(f, W)
    o.step(2)
    g.step(2)
    fo, Wo, _ = o.state()
    fg, Wg = g.state()
    tol = FP64_TOL if precision == _lib.FP64 else FP32_TOL
    for a, b in ((fg, fo), (Wg, Wo)):
        assert np.abs(a - b).max() <= tol * np.abs(b).max()
    info = g.info()
    g.close()
    return info


WALL = [{"T": 1.0, "U": [0.0, 0.0, 0.0]}, {"T": 1.1, "U": [0.2, 0.0, 0.0]}]


@pytest.mark.parametrize("precision", [_lib.FP64, _lib.FP32])
@pytest.mark.parametrize("dim,group,most", [(2, 1, 4), (2, 2, 6), (2, 4, 10), (3, 1, 6), (3, 2, 10)])
def test_cells_of_any_face_count(precision, dim, group, most):
    """Boxes with some of the cells merged: quadrilaterals (4 entries) and
    hexahedra (6), and mixed cells of up to 10 faces (the loop)."""
    mesh = cs.quad_mesh(9, 7) if dim == 2 else cs.hex_mesh(4, 3, 4, sides={"z+": ("wall", 1)})
    if group > 1:
        mesh = merged(mesh, group, 7, 6)
    assert _faces_per_cell(mesh).max() == most
    vg = cs.cartesian_vgrid((11, 9, 8)[:dim], (-4.0,) * dim, (4.0,) * dim)
    _compare(mesh, vg, cs.params(0.1, walls=WALL), precision)


@pytest.mark.parametrize("precision", [_lib.FP64, _lib.FP32])
def test_triangles_padded_to_four_entries(precision):
    """Periodic triangles (3 entries), and with pairs merged into
    quadrilaterals, whose mesh pads the triangles with a fourth entry."""
    vg = cs.cartesian_vgrid((10, 9), (-4.0, -4.0), (4.0, 4.0))
    mesh = cs.periodic_tri_mesh(8, 7)
    for m, most in ((mesh, 3), (merged(mesh, 2, 5, 9), 4)):
        assert _faces_per_cell(m).max() == most and _faces_per_cell(m).min() == 3
        _compare(m, vg, cs.params(0.1), precision)


@pytest.mark.parametrize("precision,vtile,group", [(_lib.FP64, 32, 1), (_lib.FP64, 64, 3), (_lib.FP64, 0, 0),
                                                   (_lib.FP32, 32, 5), (_lib.FP32, 64, 2), (_lib.FP32, 128, 0),
                                                   (_lib.FP32, 0, 0)])
def test_chunks_and_short_ends(precision, vtile, group):
    """A velocity set larger than one chunk of the flux buffer (more launches
    than the 11 of a step in one chunk), whose last tile, group and chunk are
    short for some of the tilings."""
    c = cs.cylinder_case(n_cells=900, nvx=43, nvy=41, mach=2.0)
    tiling = {"patch_cells": 16, "vtile": vtile, "tile_group": group} if vtile else {}
    info = _compare(c["mesh"], c["vgrid"], dict(c["params"], walls=WALL), precision, **tiling)
    assert info["kernel_launches_per_step"] > 11
