"""The moment groups of stage 1 (ugks_params.gather_tile_group): with a fixed tiling
a group depends on the velocity set alone, whatever the flux buffer of the mesh can hold,
so that subdomains sum the moments of a cell as the whole mesh does, and
ugks_info reports the group that is used."""
import functools

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2412_06546_gb300 import _lib, cases as cs, decompose as dc  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2412_06546_gb300 import build
    build.build()


@functools.lru_cache(maxsize=None)
def _case(name):
    if name == "cylinder":
        return cs.cylinder_case(n_cells=5000, nvx=32, nvy=30, mach=3.0)
    n, nv = {"box": ((14, 13, 14), 12), "box 3": ((20, 20, 20), 3), "box 8": ((20, 20, 20), 8)}[name]
    mesh = cs.hex_mesh(*n)
    return {"mesh": mesh, "vgrid": cs.cartesian_vgrid((nv,) * 3, (-4.0,) * 3, (4.0,) * 3),
            "params": cs.params(0.1, walls=[{"T": 1.1, "U": [0.2, 0.0, 0.0]}]), "init": cs.smooth_state(mesh, 3, 0.1)}


def _perturbed(case, precision):
    g = _lib.Case(case["mesh"], case["vgrid"], case["params"], case["init"], precision=precision, patch_cells=16)
    f, W = g.state()
    g.close()
    f = f * cs.perturbation(f.shape, 7, 0.1)
    return (f.astype(np.float32).astype(np.float64) if precision == _lib.FP32 else f), W


@pytest.mark.parametrize("name,precision,vtile,group,chunks", [
    ("cylinder", _lib.FP32, 64, 15, 2), ("cylinder", _lib.FP32, 32, 28, 3), ("cylinder", _lib.FP64, 32, 1024, 2),
    ("cylinder", _lib.FP64, 64, 14, 3), ("cylinder", _lib.FP32, 64, 0, 2), ("box", _lib.FP64, 32, 0, 4),
    ("box", _lib.FP32, 64, 1024, 4), ("box", _lib.FP32, 128, 12, 4), ("box", _lib.FP64, 32, 50, 5),
    ("box", _lib.FP64, 64, 1024, 4)])
def test_group_is_used_on_every_mesh(name, precision, vtile, group, chunks):
    """Groups of which the whole mesh's flux buffer holds a part (``chunks`` per
    step in all, the last group shorter in some) and a subdomain's a part or
    all: three decomposed steps bitwise equal the undivided ones, also in W,
    and the reported group is the caller's, at most all tiles (0: up to 1,024
    velocities, equal groups in multiples of 128)."""
    case = _case(name)
    mesh, vg, pr = case["mesh"], case["vgrid"], case["params"]
    case = dict(case, params=dict(pr, dt=_lib.cfl_dt(mesh, vg, pr["cfl"])))
    tiling = {"patch_cells": 32, "vtile": vtile, "threads": 256, "tile_group": group}
    full = _lib.Case(mesh, vg, case["params"], case["init"], precision=precision, **tiling)
    dec = dc.DecomposedCase(case, 16 if name == "cylinder" else 12, precision, **tiling)
    info = full.info()
    assert info["kernel_launches_per_step"] == 10 + 2 * chunks
    tiles = -(-info["nv_pad"] // vtile)
    used = min(group, tiles) if group else {"cylinder": 960, "box": 896}[name] // vtile
    for c in [full] + dec.cases:
        assert c.info()["gather_tile_group"] == used
    f, W = _perturbed(case, precision)
    full.set_state(f, W)
    dec.set_state(f, W)
    full.step(3)
    dec.step(3)
    (ff, Wf), (fd, Wd) = full.state(), dec.state()
    full.close()
    dec.close()
    assert np.array_equal(Wd, Wf), np.abs(Wd - Wf).max()
    assert np.array_equal(fd, ff)


@pytest.mark.parametrize("precision", [_lib.FP32, _lib.FP64])
@pytest.mark.parametrize("nv,group", [((24, 24), 0), ((24, 24), 3), ((41, 37), 0), ((41, 37), 1), ((41, 37), 5)])
def test_reported_tiling_gives_the_same_groups(precision, nv, group):
    """The autotuned tiling that ugks_info reports, fed back, gives the same moment
    groups: W after three steps is bitwise the same.  A caller's group is of
    default tiles whatever tile the autotuner takes."""
    case = cs.cylinder_case(n_cells=3000, nvx=nv[0], nvy=nv[1], mach=3.0)
    f, W = _perturbed(case, precision)
    out = []
    tiling = {"tile_group": group}
    for _ in range(2):
        g = _lib.Case(case["mesh"], case["vgrid"], case["params"], case["init"], precision=precision, **tiling)
        i = g.info()
        if group:
            assert i["gather_tile_group"] * i["vtile"] == group * (64 if precision == _lib.FP32 else 32)
        tiling = {"patch_cells": i["patch_cells"], "vtile": i["vtile"], "threads": i["gather_threads"],
                  "tile_group": i["gather_tile_group"]}
        g.set_state(f, W)
        g.step(3)
        out.append(g.state())
        g.close()
    assert np.array_equal(out[0][1], out[1][1]), np.abs(out[0][1] - out[1][1]).max()
    assert np.array_equal(out[0][0], out[1][0])


@pytest.mark.parametrize("precision", [_lib.FP32, _lib.FP64])
@pytest.mark.parametrize("tiling", [{}, {"patch_cells": 16, "vtile": 32, "tile_group": 1024},
                                    {"patch_cells": 16, "vtile": 32, "tile_group": 1}])
def test_footprint_estimate_bounds_the_device_bytes(precision, tiling):
    """The server admits by an estimate that is no less than what a case holds:
    two- and three-dimensional requests of few and of many velocities."""
    import ctypes as ct
    for case in (_case("box 3"), _case("box 8"), cs.cavity_case(n=60, nv=2), cs.cavity_case(n=60, nv=24),
                 _case("cylinder")):
        srv = _lib.Server(1 << 40, 8, 10)
        (m, v, p), keep = _lib.make_structs(case["mesh"], case["vgrid"], case["params"], case["init"], precision,
                                            **tiling)
        t = ct.c_uint64()
        _lib.check(_lib.load().ugks_server_submit(srv._h, ct.byref(m), ct.byref(v), ct.byref(p), 1e-12, 1, -1.0,
                                                  ct.byref(t)))
        estimate = srv.poll(t.value)["footprint_bytes"]
        srv.close()
        g = _lib.Case(case["mesh"], case["vgrid"], case["params"], case["init"], precision=precision, **tiling)
        assert g.info()["device_bytes"] <= estimate
        g.close()


@pytest.mark.parametrize("case,fp32,fp64", [
    (lambda: cs.cavity_case(n=60, nv=2), 26138376, 43120296), (lambda: cs.cavity_case(n=60, nv=24), 56104200, 103015080),
    (lambda: cs.cylinder_case(n_cells=8000, nvx=30, nvy=25, mach=3.0), 137878443, 260162397)])
def test_footprint_estimate_admits_what_it_admitted(case, fp32, fp64):
    """Automatic tilings: no more than when the flux buffer was bounded by a copy of
    f, so that no budget that held a request refuses it."""
    c = case()
    for precision, was in ((_lib.FP32, fp32), (_lib.FP64, fp64)):
        srv = _lib.Server(1 << 40, 8, 10)
        estimate = srv.poll(srv.submit(c, 1e-12, 1, precision=precision))["footprint_bytes"]
        srv.close()
        assert estimate <= was
