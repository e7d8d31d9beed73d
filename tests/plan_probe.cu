// Host entry for the test of the solve's memory plan (no GPU), one translation unit with the library's
// host code and linked with its other objects.
#include "api.cu"

// Bytes per batch column of the estimate behind the default batch size, and what a batch of B
// columns takes of the plan (everything but the eigensolver's scratch, which is bounded by itself).
extern "C" int plan_probe(int64_t m_vec, int prec, int nu, int region_atoms, int maxrow, int64_t atoms, int64_t B,
                          uint64_t *per_column, uint64_t *taken)
{
    const int64_t ntile = region_atoms > 0 ? 0 : (atoms + 7) / 8;
    SolvePlan p;
    if (!plan_solve(m_vec, prec, nu, region_atoms, maxrow, B, 4 * maxrow * B, B, ntile, p)) return 1;
    *per_column = per_column_bytes(column_shape(m_vec, prec), prec == 0 ? 8 : 4, nu, region_atoms, maxrow, ntile);
    *taken = p.oED;
    return 0;
}
