"""The eigensolver's device code by itself (eig_probe.cu): what an unreduced subspace matrix hardly
ever holds, but the code has to take."""

import ctypes as C
import math
import os
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1307_3218_gb300 import build as b
    out = str(tmp_path_factory.mktemp("probe") / "eig_probe.so")
    r = subprocess.run([b.nvcc(), *b.ARCH, *b.FLAGS, "-shared", os.path.join(HERE, "eig_probe.cu"), "-o", out],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return C.CDLL(out)


def _ptr(a):
    return a.ctypes.data_as(C.c_void_p)


def _ql(probe, d, e, nl=4, bits=0):
    """Levels, column scales and sweep counts of the tridiagonal matrices (d, e), e of d's length; a
    scale below 2^-bits counts as lost (0: the library's bound)."""
    d, e = np.array(d, float), np.array(e, float)
    ns = np.zeros(d.shape[0], np.int32)
    assert probe.eig_probe_ql(d.shape[0], d.shape[1], nl, bits, _ptr(d), _ptr(e), _ptr(ns)) == 0
    return d, e, ns


@pytest.mark.parametrize("d,e", [
    ([0.0, 0.0], [0.0, 0.0]),
    ([0.0, 0.0, 0.0, 2.0], [0.0, 0.0, 1.0, 0.0]),
    ([1.0, 0.0, 0.0, 3.0], [1.0, 0.0, 0.5, 0.0]),          # two blocks joined by an exact zero
    ([1e-300, -2e-300, 1e-300], [0.0, 1e-320, 0.0]),       # a coupling below the levels' precision
], ids=["zero", "zeros-first", "joined", "tiny"])
def test_negligible_couplings_of_zero_levels(probe, d, e):
    """A coupling |e| <= eps (|d| + |d'|) splits the matrix, also where all three are zero."""
    lv, _, ns = _ql(probe, [d] * 5, [e] * 5)
    want = np.linalg.eigvalsh(np.diag(d) + np.diag(e[:-1], 1) + np.diag(e[:-1], -1))
    assert np.all(ns >= 0)
    for row in lv:
        np.testing.assert_allclose(np.sort(row), want, rtol=0, atol=8 * np.finfo(float).eps * np.abs(want).max())


@pytest.mark.parametrize("bits", [2, 4, 8])
@pytest.mark.parametrize("n", [2, 5, 20, 60])
def test_every_lost_scale_is_reported(probe, n, bits):
    """The scales only shrink, so a subspace has lost one exactly when one of those it ends with lies
    below the bound, in whichever column: with a bound that ordinary matrices reach."""
    rng = np.random.default_rng(n)
    d, e = rng.standard_normal((256, n)), rng.standard_normal((256, n))
    _, w, ns = _ql(probe, d, e, nl=32, bits=bits)
    w0, ns0 = _ql(probe, d, e, nl=32)[1:]
    np.testing.assert_array_equal(w, w0)
    assert np.all(ns0 >= 0)
    np.testing.assert_array_equal(ns < 0, np.abs(w).min(axis=1) < 2.0 ** -bits)


def _ulps(got, exact):
    """|got - exact| in units of got's last place; exact in 50 digits."""
    return np.array([float(abs(Decimal(float(g)) - e) / Decimal(math.ulp(float(g)))) for g, e in zip(got, exact)])


def test_series_reciprocals(probe):
    """series_rsqrt and series_rcp over mantissas, signs and the exponents whose results are normal.
    With a 20-bit estimate, e = 1 - a y^2 is about 2^-19 and known to 2^-53: half of that on the result
    is at most half a unit of its last place, the last rounding another half, what the series leaves out
    (5/16 e^3) 0.02.  e = 1 - a y is exact to 2^-73: half a unit, and e^3 = 0.008.  CUDA's rsqrt is within
    one unit, its quotient correctly rounded."""
    rng = np.random.default_rng(0)
    edge = np.array([1.0, 1.0 + 2.0 ** -52, 1.5, np.sqrt(2.0), 2.0 - 2.0 ** -52])
    near = np.concatenate([rng.uniform(1.0, 2.0, 4000), np.linspace(1.0, 2.0, 2000, endpoint=False)])
    x = np.concatenate([
        np.ldexp(np.tile(edge, 2044), np.repeat(np.arange(-1021, 1023), edge.size) - 1),   # every exponent
        near, 2.0 * near,
        np.ldexp(rng.uniform(1.0, 2.0, 6000), rng.integers(-1021, 1020, 6000))])
    x = np.concatenate([x, -x[::7]])
    out = np.zeros((4, x.size))
    assert probe.eig_probe_series(x.size, _ptr(x), _ptr(out)) == 0
    getcontext().prec = 50
    pos = x > 0
    d = [Decimal(float(v)) for v in x]
    root = [1 / v.sqrt() for v, p in zip(d, pos) if p]
    assert _ulps(out[0][pos], root).max() <= 1.05
    assert (np.abs(out[0] - out[1])[pos] / np.spacing(out[1][pos])).max() <= 2.05
    assert _ulps(out[2], [1 / v for v in d]).max() <= 0.55
    assert (np.abs(out[2] - out[3]) / np.spacing(np.abs(out[3]))).max() <= 1.05
