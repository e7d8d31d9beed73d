"""Gram-Schmidt of few columns (several groups of threads per column) against that of many (one
group): every sum in the same order, so the same bits.  One to four passes of the second sweep,
one block of stored vectors and several rounds of totals, partial tiles, regions, breakdown, nu past
the 254 hops of the support search."""

import numpy as np
import pytest

from tbsynth import amorphous_system, tiny_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("atoms,nu,region,prec", [
    (45, 3, 0, 0), (45, 3, 0, 1), (60, 34, 0, 0), (64, 33, 0, 1),       # vectors of 256 entries
    (250, 70, 0, 0), (250, 70, 0, 1), (500, 37, 0, 0), (505, 40, 0, 1), (1001, 30, 0, 0), (1001, 66, 0, 1),
    (1500, 30, 0, 1), (2048, 20, 0, 1),                                 # 8,192 FP32 entries
    (2100, 34, 0, 1), (4001, 24, 0, 1),                                 # 16,384, chains in pairs
    (1000, 320, 0, 0), (1500, 320, 0, 1), (2049, 320, 0, 1),            # the most shared memory
    (600, 20, 300, 0), (600, 20, 300, 1), (90, 257, 0, 0), (90, 260, 0, 1), (48, 12, 0, 0),
])
def test_bits_do_not_depend_on_the_column_count(atoms, nu, region, prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1307_3218_gb300 as m
    # 48 atoms: isolated ones, whose columns break down
    t = tiny_system(48, seed=1) if atoms == 48 else amorphous_system(atoms, seed=6, check_spd=False)
    cols = np.arange(t.M)[t.orbital_mask.astype(bool)][-180:]
    ctx = m.setup_system(t, prec)

    def solve(batch):
        m.marnoldi_set_batch(ctx, batch)
        m.marnoldi_solve(ctx, cols, nu, region, 0.0, 0.1, mu_fixed=4.0)
        return (*m.marnoldi_density(ctx), *m.marnoldi_column_stats(ctx))

    many, few = solve(cols.size), solve(44)
    m.marnoldi_destroy(ctx)
    assert cols.size > 152
    for a, b in zip(many, few):
        np.testing.assert_array_equal(a, b)
