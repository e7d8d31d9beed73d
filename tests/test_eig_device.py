"""The eigensolver's device code by itself (eig_probe.cu): what an unreduced subspace matrix hardly
ever holds, but the code has to take."""

import ctypes as C
import os
import subprocess

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
