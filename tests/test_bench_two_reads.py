"""bench.gs_two_reads, the bytes behind the Gram-Schmidt roofline: per column and step, every stored
vector's S w_i and w_i once, written out over a small structure's supports and over dense vectors."""

import numpy as np
import pytest

import bench
from tbsynth import amorphous_system


@pytest.mark.parametrize("vbytes", [4, 8])
@pytest.mark.parametrize("nu", [1, 2, 7, 12])
def test_two_reads_step_by_step(nu, vbytes):
    t = amorphous_system(90, seed=3, check_spd=False)
    m_pad = 512
    cols = np.array([0, 5, 17, 200, 359])
    tc = bench.support_counts(t, cols, nu, m_pad)

    def bytes_of(E):
        total = 0
        for n in range(nu):
            total += (2 if vbytes == 4 else 1) * E[n + 1] + E[n]             # u (and its lo word), w_n
            total += sum(E[i + 1] for i in range(n + 1))                     # S w_i
            total += sum(E[i + 1] for i in range(n + 1))                     # w_i: a_i and the subtraction
            total += E[n + 1] if n + 1 < nu else 0                           # the new w
        return vbytes * total

    by, _ = bench.gs_algorithmic_support(nu, tc, vbytes)
    assert bench.gs_two_reads(nu, by, tc, t.M, vbytes, len(cols)) == sum(bytes_of(32 * c) for c in tc)
    by, _ = bench.gs_algorithmic(nu, t.M, vbytes, len(cols))
    want = len(cols) * bytes_of(np.full(nu + 2, t.M))
    assert bench.gs_two_reads(nu, by, None, t.M, vbytes, len(cols)) == want
