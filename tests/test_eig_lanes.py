"""The QL kernel's shared memory fits a CTA for every subspace size and chunk, its static arrays
(below 2 KB) included.  No GPU."""

import ctypes as C
import os
import subprocess

from paper_1307_3218_gb300 import build as b

HERE = os.path.dirname(os.path.abspath(__file__))


def test_ql_shared_memory_fits(tmp_path):
    out = str(tmp_path / "eig_probe.so")
    r = subprocess.run([b.nvcc(), *b.ARCH, *b.FLAGS, "-Xptxas", "-v", "-shared", os.path.join(HERE, "eig_probe.cu"),
                        "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lines = (r.stdout + r.stderr).splitlines()
    at = [i for i, ln in enumerate(lines) if "Compiling" in ln and "eig_ql_kernel" in ln]
    static = [int(ln.split(" bytes smem")[0].split()[-1]) for i in at for ln in lines[i:i + 4] if " bytes smem" in ln]
    assert static and max(static) <= 2048
    probe = C.CDLL(out)
    probe.eig_probe_ql_smem.restype = C.c_int64
    for nu in range(1, 321):
        for nb in (1, 152, 153, 2432, 2433, 100000):
            assert 0 < probe.eig_probe_ql_smem(nu, nb) + max(static) <= 227 * 1024, (nu, nb)
