"""The batch workspace is not cleared between solves: a solve reads only what it wrote.  Device
memory that the allocator hands out full of 0xff bytes (NaN in every float) changes no bit of any
result: FP64 and mixed, global and regional mode, partial tiles, padded vectors, several batches,
breakdown, and nu past the 254 hops of the support search."""

import numpy as np
import pytest

from tbsynth import amorphous_system, tiny_system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def m():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1307_3218_gb300 as mm
    from paper_1307_3218_gb300 import build as b
    b.build()
    mm.load()
    mm.setup_system(tiny_system(8, seed=1))   # the default allocator is chosen on the first setup
    yield mm
    mm.use_torch_allocator()


def _solve(m, t, prec, nu, region, batch):
    ctx = m.setup_system(t, prec)
    if batch:
        m.marnoldi_set_batch(ctx, batch)
    m.marnoldi_solve(ctx, None, nu, region, t.n_electrons, 0.1)
    out = (*m.marnoldi_density(ctx), *m.marnoldi_column_stats(ctx), np.array(m.marnoldi_energy(ctx)))
    m.marnoldi_destroy(ctx)
    return out


@pytest.mark.parametrize("atoms,prec,nu,region,batch", [
    (90, 0, 30, 0, 0), (90, 1, 30, 0, 100), (300, 1, 30, 0, 0), (130, 0, 20, 50, 100), (130, 1, 20, 50, 0),
    (90, 0, 260, 0, 0), (90, 1, 255, 0, 0), (8, 0, 12, 0, 0),
])
def test_poisoned_memory_changes_nothing(m, atoms, prec, nu, region, batch):
    import torch
    t = tiny_system(8, seed=1) if atoms == 8 else amorphous_system(atoms, seed=9, check_spd=False)
    m.use_torch_allocator()
    want = _solve(m, t, prec, nu, region, batch)
    held = {}

    def alloc(nbytes, stream, user):
        a = torch.full((int(nbytes),), 255, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        held[a.data_ptr()] = a
        return a.data_ptr()

    def free(ptr, nbytes, stream, user):
        torch.cuda.synchronize()
        held.pop(ptr, None)

    m.marnoldi_set_allocator(alloc, free)
    try:
        got = _solve(m, t, prec, nu, region, batch)
    finally:
        m.use_torch_allocator()
    assert not held
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)
