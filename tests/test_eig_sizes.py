"""The subspace eigensolve at the edges of its kernels, against the oracle: one warp per
tridiagonalisation and several, one subspace per QL warp and many, a breakdown that leaves a few
levels, H_sub in shared and in global memory, more pattern rows than a warp or a CTA holds."""

import numpy as np
import pytest

import oracle
from tbsynth import amorphous_system, build_tb, diamond, tiny_system

pytestmark = pytest.mark.gpu

KT, MU = 0.1, 3.0


def _dense():
    """A compressed cell: up to 47 blocks per row, overlaps scaled to stay positive definite."""
    t = build_tb(diamond(3, a=2.2, jitter=0.02, seed=0), check_spd=False)
    row = np.repeat(np.arange(t.n_block_rows), np.diff(t.row_ptr))
    t.S[row != t.col_idx] *= 0.2
    return t


@pytest.mark.parametrize("make,nu,ncols", [
    (lambda: amorphous_system(100, seed=1, check_spd=False), 2, 1),
    (lambda: amorphous_system(100, seed=1, check_spd=False), 3, 153),
    (lambda: amorphous_system(100, seed=1, check_spd=False), 32, 305),
    (lambda: amorphous_system(100, seed=1, check_spd=False), 33, 33),
    (lambda: amorphous_system(200, seed=2, check_spd=False), 129, 9),
    (lambda: tiny_system(8, seed=1), 12, 32),              # isolated atoms: breakdown
], ids=["nu2", "nu3", "nu32", "nu33", "nu129", "breakdown"])
def test_against_oracle(make, nu, ncols):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1307_3218_gb300 as m
    t = make()
    cols = np.sort(np.random.default_rng(nu).choice(t.M, size=min(ncols, t.M), replace=False))
    ctx = m.setup_system(t, m.MARNOLDI_FP64)
    m.marnoldi_solve(ctx, cols, nu, 0, 0.0, KT, mu_fixed=MU)
    rho, rhoE = m.marnoldi_density(ctx)
    nue, eps, w = m.marnoldi_column_stats(ctx)
    m.marnoldi_destroy(ctx)
    ref = oracle.solve(t, nu=nu, kT=KT, mu_fixed=MU, cols=cols)
    np.testing.assert_array_equal(nue, ref.cols.nu_eff)
    assert np.all(np.diff(np.where(np.arange(nu) < nue[:, None], eps, np.inf)[:, :2], axis=1)[nue > 1] >= 0)
    mask = ~np.isnan(ref.rho)
    assert np.abs(rho[mask] - ref.rho[mask]).max() <= 1e-10 * np.abs(ref.rho[mask]).max()
    assert np.abs(rhoE[mask] - ref.rhoE[mask]).max() <= 1e-10 * np.abs(ref.rhoE[mask]).max()


def test_many_pattern_rows():
    """More than 128 rows of R: a CTA's threads take several."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1307_3218_gb300 as m
    t = _dense()
    assert 4 * int(np.diff(t.row_ptr).max()) + 2 > 128
    cols = np.arange(0, t.M, 17)
    ctx = m.setup_system(t, m.MARNOLDI_FP64)
    m.marnoldi_solve(ctx, cols, 24, 0, 0.0, KT, mu_fixed=MU)
    rho, rhoE = m.marnoldi_density(ctx)
    m.marnoldi_destroy(ctx)
    ref = oracle.solve(t, nu=24, kT=KT, mu_fixed=MU, cols=cols)
    mask = ~np.isnan(ref.rho)
    assert np.abs(rho[mask] - ref.rho[mask]).max() <= 1e-10 * np.abs(ref.rho[mask]).max()
    assert np.abs(rhoE[mask] - ref.rhoE[mask]).max() <= 1e-10 * np.abs(ref.rhoE[mask]).max()
