// Regional (projection) mode of the multiple Arnoldi method on sm_103a.
//
// The method's cost is order-N (arXiv:1307.3218, Section 1): each column's
// Krylov process touches only a neighbourhood of its atom.  In regional mode
// the process for column j = 4 J + b runs on the principal sub-pair of (H, S)
// over J's projection region R_J: the n_reg atoms nearest J by squared
// minimum-image distance (ties to the lower atom index), kept in ascending
// atom index.  Local orbital 4 p + a is orbital a of atom R_J[p].
//
// Per batch column c (a region depends only on the column's atom, so of a
// run of batch columns of one atom only the first, its leader, searches):
//   region_kernel:     candidates from the cell list within radius r_s,
//                      bitonic sort by (d^2, index), the first n_reg sorted
//                      again by index -> reg[c][p]
//   local_bsr_kernel:  copies the leader's region to the other columns of
//                      its run; for every local block row p, the blocks of global row
//                      R_J[p] whose column atom lies in R_J (binary search):
//                      local column lci and global block index lgk, stored
//                      slot-major ([c][slot][p]) so that lanes over p coalesce
//   init_regional:     k_1 = e_{jl} / sqrt(S_jj), S k_1 from row j's local blocks
//   spmm_regional_hs:  H_local x and S_local x in one pass per group of one
//                      atom's columns (each block read once for the group),
//                      x and y of length m_pad >= 4 n_reg, matrix values
//                      gathered from the global BSR through lgk
#include "gs_common.cuh"

#include <climits>
#include <type_traits>

namespace marnoldi {
namespace {

constexpr int kRegionThreads = 256;

// Squared minimum-image distance, summed as (dx^2 + dy^2) + dz^2 with every
// operation rounded separately (no contraction), so the host-side checker can
// reproduce the same values.  The image rint(d / box) comes from d * (1 / box)
// unless that lies within 2^-20 of a half or is large: a division costs about
// ten instructions on the FP64 pipe, the rest of a coordinate eight.
__device__ __forceinline__ double min_image_d2(const double *pi, const double *pj,
                                               const double *box, const double *inv)
{
    double d2 = 0.0;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        double d = __dsub_rn(pi[q], pj[q]);
        const double t = d * inv[q];
        double r = rint(t);
        // high words: |t| < 2^20 (t is then within 2^-31 of d / box), |t - r| < 1/2 - 2^-20
        if ((__double2hiint(t) & 0x7fffffff) >= 0x41300000 ||
            (__double2hiint(t - r) & 0x7fffffff) >= 0x3fdffffc)
            r = rint(__ddiv_rn(d, box[q]));
        d = __dsub_rn(d, __dmul_rn(box[q], r));
        d2 = q == 0 ? __dmul_rn(d, d) : __dadd_rn(d2, __dmul_rn(d, d));
    }
    return d2;
}

__device__ __forceinline__ bool key_less(uint64_t da, int ia, uint64_t db, int ib)
{
    return da < db || (da == db && ia < ib);
}

// In-place bitonic sort of n (a power of two) (key, index) pairs in shared
// memory.  A distance's key is its bit pattern, which orders non-negative
// doubles as their values: a comparison on the FP64 pipe holds the warp's
// scheduler for 64 cycles (6,000 regions of 256 atoms: 6.0 -> 5.4 ms).
__device__ void bitonic_sort(uint64_t *key, int *idx, int n)
{
    for (int size = 2; size <= n; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int t = threadIdx.x; t < n / 2; t += blockDim.x) {
                const int lo = 2 * stride * (t / stride) + (t % stride);
                const int hi = lo + stride;
                const bool up = ((lo & size) == 0);
                const bool sw = up ? key_less(key[hi], idx[hi], key[lo], idx[lo])
                                   : key_less(key[lo], idx[lo], key[hi], idx[hi]);
                if (sw) {
                    const uint64_t tk = key[lo]; key[lo] = key[hi]; key[hi] = tk;
                    const int ti = idx[lo]; idx[lo] = idx[hi]; idx[hi] = ti;
                }
            }
            __syncthreads();
        }
    }
}

// One CTA per leader; a warp takes a row of cells along x, whose atoms are one
// run of cell_atoms (two where the row wraps), so that the lanes are full: an
// FP64 instruction holds its scheduler as long for one lane as for 32.  256
// threads: eight CTAs per SM hide one another's barriers.  With the lists'
// kernel below searching once per run, 6,000 regions of 256 atoms: 5.4 -> 2.7 ms.
__global__ void __launch_bounds__(kRegionThreads) region_kernel(
    const double *__restrict__ pos, const double *__restrict__ box,
    const int *__restrict__ cell_start, const int *__restrict__ cell_atoms, int3 ncell,
    double cell_edge_x, double cell_edge_y, double cell_edge_z, const int64_t *__restrict__ cols,
    int n_reg, double rs2, int hx, int hy, int hz, int cap, int *__restrict__ reg,
    int *__restrict__ rstat)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint64_t *key = reinterpret_cast<uint64_t *>(smem_raw);
    int *idx = reinterpret_cast<int *>(key + cap);
    __shared__ int count;
    __shared__ double bx[3], ib[3], pj[3];
    const int c = blockIdx.x;
    const int J = (int)(cols[c] >> 2);
    if (c > 0 && (cols[c - 1] >> 2) == J) {   // not a leader: local_bsr_kernel copies the region
        if (threadIdx.x == 0) rstat[c] = 0;
        return;
    }
    if (threadIdx.x < 3) {
        bx[threadIdx.x] = box[threadIdx.x];
        ib[threadIdx.x] = 1.0 / box[threadIdx.x];
        pj[threadIdx.x] = pos[3 * (int64_t)J + threadIdx.x];
    }
    if (threadIdx.x == 0) count = 0;
    __syncthreads();
    const int cx = min(ncell.x - 1, max(0, (int)(pj[0] / cell_edge_x)));
    const int cy = min(ncell.y - 1, max(0, (int)(pj[1] / cell_edge_y)));
    const int cz = min(ncell.z - 1, max(0, (int)(pj[2] / cell_edge_z)));
    // distinct cells of the cube [c - h, c + h] (the whole axis when it wraps onto itself)
    const int nx = min(2 * hx + 1, ncell.x), ny = min(2 * hy + 1, ncell.y), nz = min(2 * hz + 1, ncell.z);
    const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    const int gx0 = nx == ncell.x ? 0 : ((cx - hx) % ncell.x + ncell.x) % ncell.x;
    const int wrap = max(0, gx0 + nx - ncell.x);   // cells of the row at the start of the axis
    for (int q = threadIdx.x >> 5; q < ny * nz; q += warps) {
        const int oy = q % ny, oz = q / ny;
        const int gy = ((ny == ncell.y ? oy : cy - hy + oy) % ncell.y + ncell.y) % ncell.y;
        const int gz = ((nz == ncell.z ? oz : cz - hz + oz) % ncell.z + ncell.z) % ncell.z;
        const int row = (gz * ncell.y + gy) * ncell.x;
        const int s0 = cell_start[row + gx0], n0 = cell_start[row + gx0 + nx - wrap] - s0;
        const int s1 = cell_start[row], n1 = cell_start[row + wrap] - s1;
        for (int s = lane; s < n0 + n1; s += 32) {
            const int a = cell_atoms[s < n0 ? s0 + s : s1 + s - n0];
            const double d2 = min_image_d2(pos + 3 * (int64_t)a, pj, bx, ib);
            if (d2 <= rs2) {
                const int slot = atomicAdd(&count, 1);
                if (slot < cap) {
                    key[slot] = (uint64_t)__double_as_longlong(d2);
                    idx[slot] = a;
                }
            }
        }
    }
    __syncthreads();
    const int cnt = count;
    if (cnt < n_reg || cnt > cap) {   // uniform: the host widens or narrows r_s and retries
        if (threadIdx.x == 0) rstat[c] = cnt < n_reg ? 1 : 2;
        return;
    }
    int n2 = 1;
    while (n2 < cnt) n2 <<= 1;
    for (int s = cnt + threadIdx.x; s < n2; s += blockDim.x) {
        key[s] = UINT64_MAX;
        idx[s] = INT_MAX;
    }
    __syncthreads();
    bitonic_sort(key, idx, n2);
    // the n_reg nearest, again in ascending atom index: second sort with the
    // atom index as key (m2 <= n2 <= cap, cap a power of two)
    int m2 = 1;
    while (m2 < n_reg) m2 <<= 1;
    for (int s = threadIdx.x; s < m2; s += blockDim.x) {
        const bool in = s < n_reg;
        const int a = in ? idx[s] : INT_MAX;
        key[s] = in ? (uint64_t)a : UINT64_MAX;
        idx[s] = a;
    }
    __syncthreads();
    bitonic_sort(key, idx, m2);
    for (int s = threadIdx.x; s < n_reg; s += blockDim.x) reg[(int64_t)c * n_reg + s] = idx[s];
    if (threadIdx.x == 0) rstat[c] = 0;
}

// The leader's CTAs search, in the region's copy in shared memory, and write
// the lists of every column of the run.
__global__ void __launch_bounds__(256) local_bsr_kernel(
    const int64_t *__restrict__ rp, const int32_t *__restrict__ ci, const int64_t *__restrict__ cols,
    int nb, int *__restrict__ reg, int n_reg, int maxrow, int *__restrict__ lcnt, int *__restrict__ lci,
    int *__restrict__ lgk)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int *R = reinterpret_cast<int *>(smem_raw);
    const int c = blockIdx.y;
    const int64_t J = cols[c] >> 2;
    if (c > 0 && (cols[c - 1] >> 2) == J) return;
    for (int q = threadIdx.x; q < n_reg; q += blockDim.x) R[q] = reg[(int64_t)c * n_reg + q];
    __syncthreads();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n_reg) return;
    int end = c + 1;
    while (end < nb && (cols[end] >> 2) == J) ++end;
    const int I = R[p];
    const int64_t step = (int64_t)maxrow * n_reg;
    int cnt = 0;
    for (int64_t k = rp[I]; k < rp[I + 1]; ++k) {
        const int q = find_sorted(R, n_reg, ci[k]);
        if (q >= 0) {
            int64_t at = c * step + (int64_t)cnt * n_reg + p;
            for (int m = c; m < end; ++m, at += step) {
                lci[at] = q;
                lgk[at] = (int)k;
            }
            ++cnt;
        }
    }
    for (int m = c; m < end; ++m) {
        lcnt[(int64_t)m * n_reg + p] = cnt;
        if (m > c) reg[(int64_t)m * n_reg + p] = I;
    }
}

// k_1 = e_{jl} / sqrt(S_jj) and S k_1 from row j's local blocks (S symmetric).
template <typename VT>
__global__ void init_regional_kernel(const double *__restrict__ Sv, const double *__restrict__ sdiag,
                                     const int64_t *__restrict__ cols, const int *__restrict__ reg,
                                     int n_reg, int maxrow, const int *__restrict__ lcnt,
                                     const int *__restrict__ lci, const int *__restrict__ lgk,
                                     VT *__restrict__ K, VT *__restrict__ SK,
                                     double *__restrict__ scale, int *__restrict__ status,
                                     int *__restrict__ nu_eff, int nu, int64_t m_pad,
                                     const uint16_t *__restrict__ tinv, int nb)
{
    const int c = blockIdx.x;
    const int64_t j = cols[c];
    const int J = (int)(j >> 2), b = (int)(j & 3);
    VT *k0 = K + (int64_t)c * nu * m_pad;
    VT *sk0 = SK + (int64_t)c * nu * m_pad;
    for (int64_t r = threadIdx.x; r < m_pad; r += blockDim.x) {
        k0[r] = VT(0);
        sk0[r] = VT(0);
    }
    __syncthreads();
    // J is always inside its own region (distance 0); the guard only keeps the
    // writes in bounds should a region ever lack it (the column is then failed)
    const int pJ = find_sorted(reg + (int64_t)c * n_reg, n_reg, J);
    if (pJ < 0) {
        if (threadIdx.x == 0) {
            status[c] = 2;
            nu_eff[c] = 1;
        }
        return;
    }
    const double inv = 1.0 / sqrt(sdiag[j]);
    if (threadIdx.x == 0) {
        k0[vpos(tinv, nb, c, 4 * pJ + b)] = (VT)inv;
        scale[(int64_t)c * nu] = 1.0;
        status[c] = 0;
        nu_eff[c] = nu;
    }
    const int64_t base = (int64_t)c * maxrow * n_reg;
    const int cnt = lcnt[(int64_t)c * n_reg + pJ];
    for (int s = threadIdx.x; s < cnt; s += blockDim.x) {
        const int q = lci[base + (int64_t)s * n_reg + pJ];
        const int64_t k = lgk[base + (int64_t)s * n_reg + pJ];
#pragma unroll
        for (int a = 0; a < 4; ++a) sk0[vpos(tinv, nb, c, 4 * q + a)] = (VT)(Sv[16 * k + 4 * b + a] * inv);
    }
}

// y = H_local x and, with kS, S_local x in one pass (both feed the same
// Gram-Schmidt step and share the local block list, so the x gathers and the
// index reads serve both).  Lanes run over local block rows, so the
// local-structure reads coalesce and the x gathers stay inside the columns'
// short local vectors.  FP64: FMAs; mixed precision: see group_rows.  Rows whose
// support tile lies more than `lim` hops from the column's atom are exact zeros
// and are written without being computed.
//
// The NC batch columns c0 .. c0 + NC - 1 belong to one atom here: a column's
// region, local block lists and tile order depend only on its atom, so one
// pass over the blocks, each block read once, serves all NC columns (the
// lanes read different blocks, so the block reads are what the L1 spends its
// time on).  Every column's sums run in the same order as alone.
template <bool kS, int NC>
__device__ __forceinline__ void regional_rows(
    int p, int c0, int n_reg, int maxrow, const int *__restrict__ lcnt, const int *__restrict__ lci,
    const int *__restrict__ lgk, const double *__restrict__ Hv, const double *__restrict__ Sv,
    const double *__restrict__ X, int64_t ldx, double *__restrict__ U, int64_t ldu, double *__restrict__ SY,
    int64_t ldsy, int ncols, const uint8_t *__restrict__ thop, const uint16_t *__restrict__ tinv, int lim)
{
    const int64_t base = (int64_t)c0 * maxrow * n_reg;
    const bool act = (int)thop[(int64_t)(p >> 3) * ncols + c0] <= lim;
    const int cnt = act ? lcnt[(int64_t)c0 * n_reg + p] : 0;
    double acc[NC][4], sacc[NC][4];
#pragma unroll
    for (int m = 0; m < NC; ++m)
#pragma unroll
        for (int a = 0; a < 4; ++a) acc[m][a] = sacc[m][a] = 0.0;
    for (int s = 0; s < cnt; ++s) {
        const int q = lci[base + (int64_t)s * n_reg + p];
        const int64_t k = lgk[base + (int64_t)s * n_reg + p];
        if (!in_range(q, n_reg, kChkRegionCol)) continue;
        const int64_t xp = 32 * (int64_t)tinv[(int64_t)(q >> 3) * ncols + c0] + 4 * (q & 7);
        if (!in_range(xp, ldu - 3, kChkRegionGather)) continue;
        double xv[NC][4];
#pragma unroll
        for (int m = 0; m < NC; ++m) load4(X + (int64_t)(c0 + m) * ldx + xp, xv[m]);
        const double *Hb = Hv + 16 * k;
        const double *Sb = Sv + 16 * k;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            double hr[4], sr[4];
            load4(Hb + 4 * a, hr);
            if constexpr (kS) load4(Sb + 4 * a, sr);
#pragma unroll
            for (int m = 0; m < NC; ++m) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    acc[m][a] = fma(hr[e], xv[m][e], acc[m][a]);
                    if constexpr (kS) sacc[m][a] = fma(sr[e], xv[m][e], sacc[m][a]);
                }
            }
        }
    }
    const int64_t yp = 32 * (int64_t)tinv[(int64_t)(p >> 3) * ncols + c0] + 4 * (p & 7);
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        const int64_t c = c0 + m;
        store4(U + c * ldu + yp, acc[m]);
        if constexpr (kS) store4(SY + c * ldsy + yp, sacc[m]);
    }
}

// Columns of one atom that share a pass over the blocks: what the registers
// allow (FP64 accumulators for four columns would leave one CTA per SM).
template <typename VT>
constexpr int reg_group()
{
    return sizeof(VT) == 4 ? 4 : 2;
}

// FP64: thread (x, y) of a 32x8 CTA takes local row p = 32 blockIdx.x + x of
// group g = 8 blockIdx.y + y, the batch columns gstart[g] .. gstart[g + 1] - 1 of
// one atom (the host splits the batch into runs of one atom's columns of at
// most G = reg_group<VT>()).  A full group takes one shared pass; a shorter one
// (an atom with fewer real orbitals, or a run cut by the batch) runs its
// columns one by one.  Bound by the FP64 pipe.
template <bool kS>
__global__ void __launch_bounds__(256) spmm_regional_hs_kernel(
    int n_reg, int maxrow, const int *__restrict__ lcnt, const int *__restrict__ lci,
    const int *__restrict__ lgk, const double *__restrict__ Hv, const double *__restrict__ Sv,
    const double *__restrict__ X, int64_t ldx, double *__restrict__ U, int64_t ldu,
    double *__restrict__ SY, int64_t ldsy, int ncols, const int *__restrict__ gstart, int ngroups,
    const uint8_t *__restrict__ thop, const uint16_t *__restrict__ tinv, int lim)
{
    constexpr int G = reg_group<double>();
    const int p = blockIdx.x * 32 + threadIdx.x;
    const int g = blockIdx.y * 8 + threadIdx.y;
    if (p >= n_reg || g >= ngroups) return;
    // clipped to ncols: a run of the autotuner covers the batch's first columns only
    const int c0 = gstart[g], c1 = min(gstart[g + 1], ncols);
    if (c0 >= c1) return;
    if (c1 - c0 == G) {
        regional_rows<kS, G>(p, c0, n_reg, maxrow, lcnt, lci, lgk, Hv, Sv, X, ldx, U, ldu, SY, ldsy, ncols, thop, tinv,
                             lim);
    } else {
#pragma unroll 1
        for (int c = c0; c < c1; ++c)
            regional_rows<kS, 1>(p, c, n_reg, maxrow, lcnt, lci, lgk, Hv, Sv, X, ldx, U, ldu, SY, ldsy, ncols, thop,
                                 tinv, lim);
    }
}

// Mixed precision, NC columns of one atom: one warp per 32 rows of the group, a
// lane per local row.  H by exact products and two-sums over its hi + lo values,
// output as a (hi, lo) pair (the subspace matrix entries use it), S by FMAs over
// its hi values.  A lane's block is its own (the lanes' blocks are 32
// different ones), and reading it 16 bytes at a time looked up 32 lines per
// load, which kept the L1 at 87 %; here twelve lanes copy one block together
// (its lines are looked up once) into the warp's shared memory, from where each
// lane reads its own.  The columns go through packed instructions in pairs;
// every column's sums run in the same order as alone.  24,000 columns, 256-atom
// regions, nu = 30: 20.4 ms, 27.2 with a lane reading its own block; 4,000
// columns, nu = 100: 13.2 (19.0).  An odd NC (an atom with fewer real orbitals, or
// a run cut by the batch) takes its last column for both halves of a pair.  Groups
// of one, two and three columns of 2,000 atoms: 4.6, 4.8 and 7.2 ms; one column
// after another, a lane reading its own block, 7.5, 14.5 and 21.4.  (NC at run time
// instead: 21.8 ms for the 24,000 columns.)  The warps need nothing of each other, so a CTA
// is one: no CTA waits for its longest warp, and a few groups, or regions of few
// rows, still spread over the SMs.  With a CTA of four warps per group that went
// over all its rows: one atom of a 1,024-atom region, nu = 30, 3.4 ms, now 0.61;
// 100 columns, one per atom, of 1,000-atom regions 3.6 -> 1.75; 8,000 columns of
// 32-atom regions, nu = 20, 1.6 -> 0.86.  The rows of a group run fastest in the
// grid, so that they share the group's x in L2.
constexpr int kRegPitch = 52;   // floats per staged block: H hi and lo, S hi, and 4 that spread the banks

template <bool kS, int NC>
__device__ __forceinline__ void group_rows(
    float *blk, int p, int c0, int n_reg, int maxrow, const int *__restrict__ lcnt,
    const int *__restrict__ lci, const int *__restrict__ lgk, const float *__restrict__ Hv,
    const float *__restrict__ Sv, const float *__restrict__ X, int64_t ldx, float *__restrict__ U,
    float *__restrict__ Ulo, int64_t ldu, float *__restrict__ SY, int64_t ldsy, int ncols,
    const uint8_t *__restrict__ thop, const uint16_t *__restrict__ tinv, int lim)
{
    constexpr int kPieces = kS ? 12 : 8, NP = (NC + 1) / 2, G = 2 * NP;
    const int lane = threadIdx.x;
    const float *xc = X + (int64_t)c0 * ldx;
    const int64_t base = (int64_t)c0 * maxrow * n_reg;
    const uint32_t sb = (uint32_t)__cvta_generic_to_shared(blk);
    const bool row = p < n_reg;
    const bool act = row && (int)thop[(int64_t)(p >> 3) * ncols + c0] <= lim;
    const int cnt = act ? lcnt[(int64_t)c0 * n_reg + p] : 0;
    const int most = __reduce_max_sync(kFull, cnt);
    uint64_t hi[NP][4], lo[NP][4], sy[NP][4];   // column pairs (0, 1) and (2, 3)
#pragma unroll
    for (int h = 0; h < NP; ++h)
#pragma unroll
        for (int a = 0; a < 4; ++a) hi[h][a] = lo[h][a] = sy[h][a] = 0;
    auto block_of = [&](int s) { return s < cnt ? lgk[base + (int64_t)s * n_reg + p] : -1; };
    auto column_of = [&](int s) { return s < cnt ? lci[base + (int64_t)s * n_reg + p] : -1; };
    // position of local column q's entries, -1 for none
    auto position = [&](int q) {
        if (q < 0 || !in_range(q, n_reg, kChkRegionCol)) return -1;
        const int xp = 32 * (int)tinv[(int64_t)(q >> 3) * ncols + c0] + 4 * (q & 7);
        return in_range(xp, ldu - 3, kChkRegionGather) ? xp : -1;
    };
    auto copy = [&](int s, int k) {   // the lanes' blocks of slot s, k this lane's
        const uint32_t st = sb + (s & 1) * (32 * kRegPitch * 4);
#pragma unroll
        for (int r = 0; r < kPieces; ++r) {
            const int item = 32 * r + lane, b = item / kPieces, piece = item - b * kPieces;
            const int kb = __shfl_sync(kFull, k, b);
            const float *src = (piece < 8 ? Hv : Sv) + 32 * (int64_t)kb + 4 * (piece < 8 ? piece : piece - 8);
            if (kb >= 0)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(st + 4 * (b * kRegPitch + 4 * piece)),
                             "l"(src)
                             : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto gather = [&](int xp, float4 (&x)[G]) {
#pragma unroll
        for (int m = 0; m < G; ++m)
            if (xp >= 0) x[m] = __ldg(reinterpret_cast<const float4 *>(xc + (m < NC ? m : NC - 1) * ldx + xp));
    };
    // blocks are copied one slot ahead, x one, the positions two, the indices three
    copy(0, block_of(0));
    int kn = block_of(1), x0p = position(column_of(0)), x1p = position(column_of(1)), q2 = column_of(2);
    float4 xv[G], xw[G];
    gather(x0p, xv);
    for (int s = 0; s < most; ++s) {
        __syncwarp();   // slot s - 1 has been read
        if (s + 1 < most) copy(s + 1, kn);
        else asm volatile("cp.async.commit_group;" ::: "memory");
        gather(x1p, xw);
        const int x2p = position(q2);
        q2 = column_of(s + 3);
        kn = block_of(s + 2);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
        if (x0p >= 0) {
            uint64_t x[NP][4], nx[NP][4];
#pragma unroll
            for (int h = 0; h < NP; ++h) {
                const float4 u = xv[2 * h], v = xv[2 * h + 1];
                x[h][0] = pack_x2(u.x, v.x);
                x[h][1] = pack_x2(u.y, v.y);
                x[h][2] = pack_x2(u.z, v.z);
                x[h][3] = pack_x2(u.w, v.w);
#pragma unroll
                for (int e = 0; e < 4; ++e) nx[h][e] = neg_x2(x[h][e]);
            }
            const float *B = blk + (s & 1) * (32 * kRegPitch) + lane * kRegPitch;
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const float4 h4 = *reinterpret_cast<const float4 *>(B + 4 * a);
                const float4 l4 = *reinterpret_cast<const float4 *>(B + 16 + 4 * a);
                const float hv[4] = {h4.x, h4.y, h4.z, h4.w}, lv[4] = {l4.x, l4.y, l4.z, l4.w};
                float sv[4] = {0.f, 0.f, 0.f, 0.f};
                if constexpr (kS) {
                    const float4 s4 = *reinterpret_cast<const float4 *>(B + 32 + 4 * a);
                    sv[0] = s4.x; sv[1] = s4.y; sv[2] = s4.z; sv[3] = s4.w;
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint64_t hp = pack_x2(hv[e], hv[e]), lp = pack_x2(lv[e], lv[e]);
#pragma unroll
                    for (int h = 0; h < NP; ++h) spmm_add(hi[h][a], lo[h][a], hp, lp, x[h][e], nx[h][e]);
                    if constexpr (kS) {
                        const uint64_t sp = pack_x2(sv[e], sv[e]);
#pragma unroll
                        for (int h = 0; h < NP; ++h) sy[h][a] = fma_x2(sp, x[h][e], sy[h][a]);
                    }
                }
            }
        }
        x0p = x1p;
        x1p = x2p;
#pragma unroll
        for (int m = 0; m < G; ++m) xv[m] = xw[m];
    }
    if (!row) return;
    const int64_t yp = 32 * (int64_t)tinv[(int64_t)(p >> 3) * ncols + c0] + 4 * (p & 7);
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        const int64_t c = c0 + m;
        float yh[4], yl[4], ys[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int sh = 32 * (m & 1);
            const float fh = __uint_as_float((unsigned)(hi[m >> 1][a] >> sh));
            const float fl = __uint_as_float((unsigned)(lo[m >> 1][a] >> sh));
            yh[a] = __fadd_rn(fh, fl);
            yl[a] = __fsub_rn(fl, __fsub_rn(yh[a], fh));
            ys[a] = __uint_as_float((unsigned)(sy[m >> 1][a] >> sh));
        }
        store4(U + c * ldu + yp, yh);
        store4(Ulo + c * ldu + yp, yl);
        if constexpr (kS) store4(SY + c * ldsy + yp, ys);
    }
}

template <bool kS>
__global__ void __launch_bounds__(32, 12) spmm_regional_group_kernel(
    int n_reg, int maxrow, const int *__restrict__ lcnt, const int *__restrict__ lci,
    const int *__restrict__ lgk, const float *__restrict__ Hv, const float *__restrict__ Sv,
    const float *__restrict__ X, int64_t ldx, float *__restrict__ U, float *__restrict__ Ulo, int64_t ldu,
    float *__restrict__ SY, int64_t ldsy, int ncols, const int *__restrict__ gstart,
    const uint8_t *__restrict__ thop, const uint16_t *__restrict__ tinv, int lim)
{
    static_assert(reg_group<float>() == 4, "two pairs of columns");
    __shared__ __align__(16) float blk[2 * 32 * kRegPitch];   // two stages of 32 blocks
    const int g = blockIdx.y, p = 32 * (int)blockIdx.x + (int)threadIdx.x;
    // clipped to ncols: a run of the autotuner covers the batch's first columns only
    const int c0 = gstart[g], nc = min(gstart[g + 1], ncols) - c0;
    auto rows = [&](auto n) {
        group_rows<kS, decltype(n)::value>(blk, p, c0, n_reg, maxrow, lcnt, lci, lgk, Hv, Sv, X, ldx, U, Ulo, ldu, SY,
                                           ldsy, ncols, thop, tinv, lim);
    };
    switch (nc) {
    case 4: rows(std::integral_constant<int, 4>()); break;
    case 3: rows(std::integral_constant<int, 3>()); break;
    case 2: rows(std::integral_constant<int, 2>()); break;
    case 1: rows(std::integral_constant<int, 1>()); break;
    default: break;   // past ncols
    }
}

}  // namespace

int regional_group(int prec) { return prec == 0 ? reg_group<double>() : reg_group<float>(); }

cudaError_t launch_spmm_regional_hs(const DeviceMatrix &A, const RegionMaps &rm, const KrylovBatch &b,
                                    const void *X, int64_t ldx, void *SY, int64_t ldsy, int lim,
                                    cudaStream_t s)
{
    if (!b.thop || !b.tinv || b.ntile * 8 < rm.n_reg) return cudaErrorInvalidValue;
    const dim3 block(32, 8);
    if (!rm.gstart || rm.ngroups < 1) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)((rm.n_reg + 31) / 32), (unsigned)((rm.ngroups + 7) / 8));
    const int64_t ldu = b.shape.m_pad;
    if (b.prec == 0) {
        if (SY)
            spmm_regional_hs_kernel<true><<<grid, block, 0, s>>>(
                rm.n_reg, rm.maxrow, rm.lcnt, rm.lci, rm.lgk, A.Hd, A.Sd, (const double *)X, ldx, (double *)b.U, ldu, (double *)SY, ldsy, b.nb, rm.gstart, rm.ngroups, b.thop, b.tinv, lim);
        else
            spmm_regional_hs_kernel<false><<<grid, block, 0, s>>>(
                rm.n_reg, rm.maxrow, rm.lcnt, rm.lci, rm.lgk, A.Hd, A.Sd, (const double *)X, ldx, (double *)b.U, ldu, nullptr, 0, b.nb, rm.gstart, rm.ngroups, b.thop, b.tinv, lim);
    } else {
        const dim3 ggrid(grid.x, (unsigned)rm.ngroups);
        auto go = [&](auto kernel) {
            kernel<<<ggrid, 32, 0, s>>>(
                rm.n_reg, rm.maxrow, rm.lcnt, rm.lci, rm.lgk, A.Hf, A.Sf, (const float *)X, ldx, (float *)b.U,
                (float *)b.Ulo, ldu, (float *)SY, ldsy, b.nb, rm.gstart, b.thop, b.tinv, lim);
        };
        SY ? go(spmm_regional_group_kernel<true>) : go(spmm_regional_group_kernel<false>);
    }
    return cudaGetLastError();
}

cudaError_t launch_region(const RegionMaps &rm, const KrylovBatch &b, double rs, int cap,
                          cudaStream_t s)
{
    const int hx = (int)ceil(rs / rm.cell_edge[0]), hy = (int)ceil(rs / rm.cell_edge[1]),
              hz = (int)ceil(rs / rm.cell_edge[2]);
    const size_t smem = (size_t)cap * (sizeof(double) + sizeof(int));
    cudaError_t e = allow_dynamic_smem((const void *)region_kernel, smem);
    if (e != cudaSuccess) return e;
    region_kernel<<<b.nb, kRegionThreads, smem, s>>>(rm.pos, rm.box, rm.cell_start, rm.cell_atoms,
                                           make_int3(rm.ncell[0], rm.ncell[1], rm.ncell[2]),
                                           rm.cell_edge[0], rm.cell_edge[1], rm.cell_edge[2],
                                           b.cols, rm.n_reg, rs * rs, hx, hy, hz, cap, rm.reg,
                                           rm.rstat);
    return cudaGetLastError();
}

cudaError_t launch_local_bsr(const DeviceMatrix &A, const RegionMaps &rm, const KrylovBatch &b,
                             cudaStream_t s)
{
    const dim3 grid((unsigned)((rm.n_reg + 255) / 256), (unsigned)b.nb);
    local_bsr_kernel<<<grid, 256, rm.n_reg * sizeof(int), s>>>(A.rp, A.ci, b.cols, b.nb, rm.reg, rm.n_reg, rm.maxrow, rm.lcnt,
                                          rm.lci, rm.lgk);
    return cudaGetLastError();
}

cudaError_t launch_init_regional(const DeviceMatrix &A, const RegionMaps &rm, const KrylovBatch &b,
                                 cudaStream_t s)
{
    if (b.prec == 0)
        init_regional_kernel<double><<<b.nb, 256, 0, s>>>(
            A.Sd, A.sdiag, b.cols, rm.reg, rm.n_reg, rm.maxrow, rm.lcnt, rm.lci, rm.lgk,
            (double *)b.K, (double *)b.SK, b.scale, b.status, b.nu_eff, b.nu, b.shape.m_pad,
            b.tinv, b.nb);
    else
        init_regional_kernel<float><<<b.nb, 256, 0, s>>>(
            A.Sd, A.sdiag, b.cols, rm.reg, rm.n_reg, rm.maxrow, rm.lcnt, rm.lci, rm.lgk,
            (float *)b.K, (float *)b.SK, b.scale, b.status, b.nu_eff, b.nu, b.shape.m_pad,
            b.tinv, b.nb);
    return cudaGetLastError();
}


MARNOLDI_CHECK_TAKE(region)

}  // namespace marnoldi
