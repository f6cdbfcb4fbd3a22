"""The plain 64-bit step of the performance cases against the CPU oracle, for each
kind of set-up: the reference that rounding errors are quoted against."""
import importlib.util
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def perf():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    spec = importlib.util.spec_from_file_location("perf_cases", os.path.join(ROOT, "perf", "cases.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    return m


@pytest.mark.parametrize("case", [
    {"kind": "cavity", "n": 9, "nvx": 14, "nvy": 13}, {"kind": "cylinder", "cells": 1000, "nvx": 20, "nvy": 17},
    {"kind": "cylinder_dvs", "cells": 1000, "nv": 600}, {"kind": "hex", "nx": 5, "ny": 4, "nz": 6, "nvx": 9, "nvy": 8, "nvz": 7},
    {"kind": "body", "h0": 1.4, "surface": 3000, "nvx": 9, "nvy": 8, "nvz": 8},
    {"kind": "body_dvs", "h0": 1.4, "surface": 3000, "nv": 700}], ids=lambda c: c["kind"])
def test_plain_step_is_the_oracles(perf, case):
    """One step in 64 bits each, 1e-13 of the largest value (sums over up to 700
    velocities in another order, 1e-16 a term)."""
    case = dict(case, precision="fp64", steps=1)
    (got,) = perf.exact(case, 11)
    (setup,), (seed,) = perf._setups(case), perf._seeds(case, 11)
    f, W = perf._state(setup, torch.float64, seed)
    o = oracle.OracleCase(setup["mesh"], setup["vgrid"], setup["params"], setup["init"], n_threads=0)
    o.set_state(f.cpu().numpy().reshape(o.state()[0].shape), W.cpu().numpy())
    o.step(1)
    fo, Wo, qo = o.state()
    for name, a, b in (("f", got["f"], fo), ("W", got["W"], Wo), ("q", got["q"], qo)):
        err = np.abs(a.cpu().numpy().reshape(b.shape) - b).max() / np.abs(b).max()
        print(case["kind"], name, f"{err:.1e}")
        assert err <= 1e-13, (name, err)
