"""The FP64 arithmetic of one cell or face against extended precision: no less
accurate than the formula written out in ordinary double precision."""
import ctypes as ct
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
EXP_NEG, TIME_INTEGRALS, PRIM2, PRIM3 = range(4)
LD = np.longdouble
# a root mean square over 2e4 samples scatters by well under 1 %, and the CUDA and the
# host library round exp and expm1 differently (0.25 units in the last place in the mean)
SAMPLES, SCATTER = 20000, 1.15


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2412_06546_gb300 import build
    so = str(tmp_path_factory.mktemp("probe") / "scalar_probe.so")
    subprocess.run([build.NVCC] + build.ARCH + build.FLAGS + ["-I", build.CSRC, "-shared", "-o", so,
                                                              os.path.join(HERE, "scalar_probe.cu"), "-lcudart"],
                   check=True, capture_output=True)
    fn = ct.CDLL(so).scalar_probe
    dp = ct.POINTER(ct.c_double)
    fn.argtypes = [ct.c_int, dp, ct.c_int, dp, ct.c_int, ct.c_int]

    def run(what, x, nout):
        x = np.ascontiguousarray(x, dtype=np.float64).reshape(len(x), -1)
        out = np.empty((len(x), nout))
        assert fn(what, x.ctypes.data_as(dp), x.shape[1], out.ctypes.data_as(dp), nout, len(x)) == 0
        return out
    return run


def _rms(x, exact):
    return np.sqrt(np.mean((((x - exact) / exact).astype(np.float64)) ** 2, axis=0))


def _integrals(dt, x, series):
    """q1..q5 in the type of dt and x, by series or by the bracketed forms."""
    one = x.dtype.type(1)
    if series:
        s = [np.zeros_like(x) for _ in range(5)]
        fact, p1, p2 = one, np.ones_like(x), np.ones_like(x)      # 1/j!, x^(j-1), x^(j-2)
        for j in range(1, 31):
            fact = fact / j
            sg = one if j & 1 else -one
            s[0] = s[0] + sg * p1 * fact
            if j >= 2:
                s[1] = s[1] + sg * (j - one) * p2 * fact
                s[2] = s[2] - sg * p1 * fact
            if j >= 3:
                s[3] = s[3] + sg * (2 - one * j) * p2 * fact
                s[4] = s[4] + sg * p2 * fact
            p1, p2 = p1 * x, p1
        return np.stack([dt * s[0], dt * dt * s[1], dt * s[2], dt * dt * s[3], dt * dt * s[4]], 1)
    e, E = np.exp(-x), -np.expm1(-x)
    ix = one / x
    ix2 = ix * ix
    return np.stack([dt * E * ix, dt * dt * (x * e - E) * ix2, dt * (x - E) * ix,
                     dt * dt * (2 * E - x * (1 + e)) * ix2, dt * dt * (x * x / 2 - x + E) * ix2], 1)


@pytest.mark.parametrize("lo,hi", [(1e-8, 1e-3), (1e-3, 0.05), (0.05, 0.5), (0.5, 0.7), (0.7, 1.0), (1.0, 2.0),
                                   (2.0, 10.0), (10.0, 300.0)])
def test_time_integrals(probe, lo, hi):
    """q1..q5 over x = dt / tau: below 1/2 against their alternating series, above
    against the bracketed forms with exp and expm1, both in double precision."""
    rng = np.random.default_rng(3)
    x = np.minimum(np.exp(rng.uniform(np.log(lo), np.log(hi), SAMPLES)), np.nextafter(hi, 0.0))
    dt = rng.uniform(0.5, 1.5, SAMPLES)
    exact = _integrals(dt.astype(LD), x.astype(LD), hi <= 2.0)
    here = _rms(probe(TIME_INTEGRALS, np.stack([dt, x], 1), 5), exact)
    plain = _rms(_integrals(dt, x, hi <= 0.5), exact)
    assert np.all(here <= SCATTER * plain), (here, plain)


def test_exp_neg(probe):
    """The Maxwellians' exponential on [-700, 700): within one unit in the last
    place (reduction and polynomial 2^-60, the table's remainder 2^-106, three
    roundings of which the last is half a unit), no less accurate in the root
    mean square than numpy's, exact at 0 and -0."""
    rng = np.random.default_rng(5)
    x = np.concatenate([-np.exp(rng.uniform(np.log(1e-12), np.log(700.0), 8 * SAMPLES)), rng.uniform(-700, 0, 8 * SAMPLES),
                        rng.uniform(0, 700, SAMPLES), [-699.9999999, np.nextafter(-700.0, 0), -1e-300, 5e-324]])
    y = probe(EXP_NEG, x, 1)[:, 0]
    exact = np.exp(x.astype(LD))
    ulp = np.abs((y - exact) / np.spacing(exact.astype(np.float64)))
    assert ulp.max() <= 1.0, ulp.max()
    plain = (np.exp(x) - exact) / np.spacing(exact.astype(np.float64))
    assert np.sqrt(np.mean(ulp ** 2)) <= SCATTER * np.sqrt(np.mean(plain.astype(np.float64) ** 2))
    assert np.all(probe(EXP_NEG, np.array([0.0, -0.0]), 1) == 1.0)


def test_exp_neg_beyond_its_range(probe):
    """Nothing at or below -700 (the true values are under 1e-304), the library's
    exp from 700 on, NaN and infinities as exp has them."""
    x = np.array([-700.0, -700.5, -745.0, -1e4, -1e308, -np.inf])
    assert np.all(probe(EXP_NEG, x, 1) == 0.0) and np.exp(-700.0) < 1e-304
    x = np.array([700.0, 705.25, 709.7])
    assert np.allclose(probe(EXP_NEG, x, 1)[:, 0], np.exp(x.astype(LD)).astype(np.float64), rtol=3e-16, atol=0)
    x = np.array([710.0, 1e300, np.inf])
    assert np.all(probe(EXP_NEG, x, 1) == np.inf)
    assert np.all(np.isnan(probe(EXP_NEG, np.array([np.nan, -np.nan]), 1)))


def _primitive(W):
    """U, T, lam and the prefactor of a Maxwellian, in the type of W."""
    D = W.shape[1] - 2
    pi = W.dtype.type("3.14159265358979323846264338327950288")
    U = W[:, 1:-1] / W[:, :1]
    ke = np.zeros_like(W[:, 0])
    for d in range(D):
        ke = ke + U[:, d] * U[:, d]
    T = W.dtype.type(2) / 3 * (W[:, -1] / W[:, 0] - ke / 2)
    lam = 1 / (2 * T)
    a = lam / pi
    return np.column_stack([U, T, lam, W[:, 0] * a if D == 2 else W[:, 0] * a * np.sqrt(a)])


@pytest.mark.parametrize("D,what", [(2, PRIM2), (3, PRIM3)])
def test_primitive_variables(probe, D, what):
    """(rho, rho U, rho E) over six decades of density and three of temperature to
    U, T, lambda and the prefactor: the root mean square errors of the formulas
    with IEEE divisions, on the same states (3 % for what the contraction of a
    product and a sum changes at either side)."""
    rng = np.random.default_rng(7)
    rho, T = np.exp(rng.uniform(-7, 7, 10 * SAMPLES)), np.exp(rng.uniform(np.log(0.1), np.log(100.0), 10 * SAMPLES))
    U = rng.normal(size=(10 * SAMPLES, D)) * np.sqrt(T)[:, None]
    W = np.column_stack([rho, rho[:, None] * U, rho * (0.5 * (U * U).sum(1) + 1.5 * T)])
    exact = _primitive(W.astype(LD))
    here, plain = _rms(probe(what, W, D + 3), exact), _rms(_primitive(W), exact)
    assert np.all(here <= 1.03 * plain), (here, plain)
