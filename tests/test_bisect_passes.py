"""The Fermi bisection with three counts per pass (few levels) against one count per
pass (many): the same halvings, so the same mu, N and E to the last bit."""

import pytest

from tbsynth import amorphous_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kT", [0.02, 0.2])
def test_three_counts_equal_one_by_one(kT):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1307_3218_gb300 as m
    sizes, nu = (160, 200, 216, 240), 30
    assert 4 * max(sizes) * nu < 152 * 512 < 4 * sum(sizes) * nu   # alone below the line, together above
    systems = [amorphous_system(n, seed=20 + q, check_spd=False) for q, n in enumerate(sizes)]
    n, rp, ci, H, S, mask, offs, _ = m.union_of(systems)
    ctx = m.marnoldi_setup(n, rp, ci, H, S, mask, precision=m.MARNOLDI_FP64)
    m.marnoldi_set_members(ctx, offs, [t.n_electrons for t in systems])
    m.marnoldi_solve(ctx, None, nu, 0, 0.0, kT)
    together = [m.marnoldi_member_energy(ctx, q) for q in range(len(sizes))]
    m.marnoldi_destroy(ctx)
    for t, got in zip(systems, together):
        ctx = m.setup_system(t, m.MARNOLDI_FP64)
        m.marnoldi_solve(ctx, None, nu, 0, t.n_electrons, kT)
        assert tuple(m.marnoldi_energy(ctx)) == tuple(got)
        m.marnoldi_destroy(ctx)


def test_no_bracket_is_refused_alike():
    """A level range that cannot hold the electrons ends in the same error on both routes."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1307_3218_gb300 as m
    for atoms in (64, 700):   # below and above the line
        t = amorphous_system(atoms, seed=5, check_spd=False)
        ctx = m.setup_system(t, m.MARNOLDI_FP64)
        with pytest.raises(m.MarnoldiError, match="outside"):
            m.marnoldi_solve(ctx, None, 30, 0, 1e6, 0.1)
        m.marnoldi_destroy(ctx)
