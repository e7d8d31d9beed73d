"""The estimate that the default batch size is taken from covers what a batch takes, for single
structures, regions and unions of members (whose tiles are the whole union's).  No GPU."""

import ctypes as C
import os
import subprocess

import pytest

from paper_1307_3218_gb300 import build as b

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    lib = b.build()
    tag = os.path.basename(lib)[len("libmarnoldi_"):-len(".so")]
    objs = [os.path.join(b.BUILD, f"{os.path.splitext(s)[0]}_{tag}.o") for s in b.SOURCES if s != "api.cu"]
    out = str(tmp_path_factory.mktemp("probe") / "plan_probe.so")
    r = subprocess.run([b.nvcc(), *b.ARCH, *b.FLAGS, "-shared", os.path.join(HERE, "plan_probe.cu"), *objs, "-o", out],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return C.CDLL(out)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("m_vec,atoms,region", [
    (256, 64, 0), (4000, 1000, 0), (4004, 1001, 0), (16384, 4096, 0),        # one structure
    (1024, 6000, 256), (128, 6000, 32),                                      # regions
    (256, 4096, 0), (32, 4096, 0), (4096, 4096, 0), (2000, 3 * 504, 0),      # unions of members
])
@pytest.mark.parametrize("nu", [1, 4, 30, 100])
def test_estimate_covers_the_plan(probe, m_vec, atoms, region, prec, nu):
    maxrow, B = 12, 4096
    per, taken = C.c_uint64(), C.c_uint64()
    assert probe.plan_probe(C.c_int64(m_vec), prec, nu, region, maxrow, C.c_int64(atoms), C.c_int64(B),
                            C.byref(per), C.byref(taken)) == 0
    assert taken.value <= B * per.value + 32 * 256   # the pieces' alignment
