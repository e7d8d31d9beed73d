"""The Gram-Schmidt kernel at the edges of its shapes, against the oracle: one chunk and several,
a last block of one to four stored vectors, totals in one round of 32 vectors and in several, a
partial last tile, each number of chains of partial sums (256, 512, 1,024), both precisions."""

import numpy as np
import pytest

import oracle
from tbsynth import amorphous_system

pytestmark = pytest.mark.gpu

KT, MU = 0.1, 4.0


@pytest.mark.parametrize("atoms,nu,prec,shape", [
    (40, 33, 0, (1, 256)), (64, 34, 1, (1, 256)),       # one chunk, 32 + 1 and 32 + 2 vectors
    (250, 65, 1, (4, 256)), (300, 35, 1, (8, 256)),     # two- and three-stage rings, partial tiles
    (1000, 36, 0, (16, 256)),                           # passes of four chunks in sweep 2
    (1100, 37, 1, (16, 512)), (1100, 37, 0, (8, 1024)),
    (2060, 9, 0, (16, 1024)),
])
def test_against_oracle(atoms, nu, prec, shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1307_3218_gb300 as m
    t = amorphous_system(atoms, seed=5, check_spd=False)
    cols = np.sort(np.random.default_rng(atoms).choice(t.M, size=12, replace=False))
    ctx = m.setup_system(t, prec)
    m.marnoldi_solve(ctx, cols, nu, 0, 0.0, KT, mu_fixed=MU)
    assert m.marnoldi_gs_shape(ctx) == shape
    rho, rhoE = m.marnoldi_density(ctx)
    m.marnoldi_destroy(ctx)
    ref = oracle.solve(t, nu=nu, kT=KT, mu_fixed=MU, cols=cols)
    mask = ~np.isnan(ref.rho)
    err, errE = np.abs(rho[mask] - ref.rho[mask]).max(), np.abs(rhoE[mask] - ref.rhoE[mask]).max()
    if prec == 0:
        assert err <= 1e-10 * np.abs(ref.rho[mask]).max() and errE <= 1e-10 * np.abs(ref.rhoE[mask]).max()
    else:
        assert err <= 1e-5 and errE <= 1e-4
