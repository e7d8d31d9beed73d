"""The mixed-precision regional product of groups of one to four columns of an atom, in every
selection of its orbitals, against the columns alone, bit for bit; rows in one warp and in several."""

import itertools

import numpy as np
import pytest

from tbsynth import amorphous_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_reg", [20, 64, 150])
def test_every_selection_of_an_atoms_columns(n_reg):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1307_3218_gb300 as m
    t = amorphous_system(200, seed=8, check_spd=False)
    ctx = m.setup_system(t, m.MARNOLDI_MIXED)
    sets = [s for n in range(1, 5) for s in itertools.combinations(range(4), n)]
    atoms = [3 + 11 * q for q in range(len(sets))]
    cols = np.concatenate([4 * a + np.array(s) for a, s in zip(atoms, sets)])

    def levels(c):
        m.marnoldi_solve(ctx, c, 10, n_reg, 0.0, 0.1, mu_fixed=4.0)
        return m.marnoldi_column_stats(ctx)

    together = levels(cols)
    for q, c in enumerate(cols):
        for a, b in zip(levels([c]), together):
            np.testing.assert_array_equal(a[0], b[q])
    m.marnoldi_destroy(ctx)
