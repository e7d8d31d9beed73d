"""The uncleared batch workspace under a union of members, whose tiles outnumber the vectors'
positions: device memory full of 0xff bytes (NaN in every float), and a workspace that a larger solve
of the same context has used, change no bit of any member's result."""

import numpy as np
import pytest

from tbsynth import amorphous_system, tiny_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,nu,batch", [(0, 30, 0), (1, 30, 100), (1, 12, 0), (0, 31, 77), (1, 200, 0)])
def test_poisoned_memory_changes_no_member(prec, nu, batch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1307_3218_gb300 as m
    # partial last tiles, a member far shorter than the others, one of isolated atoms
    systems = [amorphous_system(n, seed=n, check_spd=False) for n in (90, 61, 200, 47)] + [tiny_system(9, seed=1)]
    n, rp, ci, H, S, mask, offs, _ = m.union_of(systems)
    m.marnoldi_destroy(m.setup_system(systems[0]))   # the default allocator is chosen on the first setup

    def solve(before=None):
        ctx = m.marnoldi_setup(n, rp, ci, H, S, mask, precision=prec)
        m.marnoldi_set_batch(ctx, batch)
        if before:
            m.marnoldi_solve(ctx, None, before, 0, sum(t.n_electrons for t in systems), 0.1)
        m.marnoldi_set_members(ctx, offs, [t.n_electrons for t in systems])
        m.marnoldi_solve(ctx, None, nu, 0, 0.0, 0.1)
        out = (*m.marnoldi_density(ctx), *m.marnoldi_column_stats(ctx),
               np.array([m.marnoldi_member_energy(ctx, q) for q in range(len(systems))]))
        m.marnoldi_destroy(ctx)
        return out

    m.use_torch_allocator()
    want = solve()
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
        poisoned, reused = solve(), solve(before=nu + 20)
    finally:
        m.use_torch_allocator()
    assert not held
    for got in (poisoned, reused):
        for a, b in zip(got, want):
            np.testing.assert_array_equal(a, b)
