"""The regional product of an atom's four columns together (staged blocks, packed columns) against
the same columns one by one, bit for bit: region sizes around the 32 rows of a
warp and the 128 of a CTA, and with columns left out of some atoms."""

import numpy as np
import pytest

from tbsynth import amorphous_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_reg,nu", [(3, 7), (31, 9), (32, 9), (33, 10), (127, 8), (129, 12), (260, 12)])
def test_groups_equal_single_columns(n_reg, nu):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1307_3218_gb300 as m
    t = amorphous_system(300, seed=4, check_spd=False)
    ctx = m.setup_system(t, m.MARNOLDI_MIXED)
    cols = np.concatenate([np.arange(40, 48), [60, 61, 63], np.arange(1196, 1200)])

    def levels(c):
        m.marnoldi_solve(ctx, c, nu, n_reg, 0.0, 0.1, mu_fixed=4.0)
        return m.marnoldi_column_stats(ctx)

    nue, eps, w = levels(cols)
    for q, c in enumerate(cols):
        n1, e1, w1 = levels([c])
        assert n1[0] == nue[q]
        np.testing.assert_array_equal(e1[0], eps[q])
        np.testing.assert_array_equal(w1[0], w[q])
    m.marnoldi_destroy(ctx)
