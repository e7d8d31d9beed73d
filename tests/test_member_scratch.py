"""A solve of members keeps to its two allocations (the column state and the batch workspace), also
when the workspace of a small batch does not hold every member's bisection at once."""

import pytest

from tbsynth import tiny_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("members", [2, 64, 200])
def test_no_allocation_for_the_bisections(members, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1307_3218_gb300 as m
    systems = [tiny_system(8, seed=q % 5) for q in range(members)]
    n, rp, ci, H, S, mask, offs, _ = m.union_of(systems)
    m.marnoldi_destroy(m.setup_system(systems[0]))   # the default allocator is chosen on the first setup

    def solve(batch):
        ctx = m.marnoldi_setup(n, rp, ci, H, S, mask, precision=precision)
        m.marnoldi_set_members(ctx, offs, [t.n_electrons for t in systems])
        m.marnoldi_set_batch(ctx, batch)
        before = len(sizes)
        m.marnoldi_solve(ctx, None, 4, 0, 0.0, 0.1)
        made = len(sizes) - before
        out = [m.marnoldi_member_energy(ctx, q) for q in range(members)]
        m.marnoldi_destroy(ctx)
        return made, out

    sizes, held = [], {}

    def alloc(nbytes, stream, user):
        a = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
        sizes.append(int(nbytes))
        held[a.data_ptr()] = a
        return a.data_ptr()

    def free(ptr, nbytes, stream, user):
        torch.cuda.synchronize()
        held.pop(ptr, None)

    m.marnoldi_set_allocator(alloc, free)
    try:
        whole, one = solve(0), solve(1)
    finally:
        m.use_torch_allocator()
    assert not held
    assert whole[0] == one[0] == 2
    assert whole[1] == one[1]
