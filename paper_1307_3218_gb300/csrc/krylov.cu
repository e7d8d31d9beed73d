// Krylov-subspace build of the multiple Arnoldi method on sm_103a.
//
// For a batch of columns j, builds a basis of
// span{e_j, H e_j, ..., H^(nu-1) e_j} (arXiv:1307.3218, Section 2: the subspace
// L_nu^(j) containing e_j whose nu x nu *standard* eigenproblem replaces
// H phi = eps S phi, Eq. 2), its S-Gram matrix and the explicit subspace
// matrix of the stored vectors; the eigensolve turns them into the
// S-orthonormal basis K and H_sub = K^T H K.
//
// The basis is stored unnormalised: slot i holds w_i and S w_i, and
// k_i = s_i w_i with s_i = 1 / ||w_i||_S.  One Krylov step n, for every column:
//   spmm_hs:  H w_n into U (accurate (hi, lo) in mixed precision) and, for
//             n >= 1, S w_n into slot n (one gather of w_n for both)
//   gs:       beta_n^2 = w_n . S w_n; stop the column when
//             beta_n^2 <= tau^2 (beta_n^2 + |projection of u_{n-1}|_S^2), i.e.
//             ||w_n||_S <= tau ||u_{n-1}||_S; else s_n = 1 / beta_n, the
//             entries k_i . H k_n, the Gram column k_i . S k_n, and
//             w_{n+1} = s_n H w_n - (its S-projection on span(K)) into slot n+1
//
// Inner products are accumulated to FP64 accuracy where the result needs it;
// in mixed precision the vectors, the SpMM and the Gram-Schmidt updates are
// FP32.  Reductions use a fixed order (trees over the lanes, then over the
// warps), so results do not depend on scheduling.
#include "gs_common.cuh"

#include <cstdio>
#include <type_traits>

namespace marnoldi {

const char *kernel_name(int kind)
{
    static const char *names[KK_NKINDS] = {"init",   "spmm_H", "gs",      "spmm_S", "eigsub",
                                           "minmax", "count",  "density", "green", "region", "support", "spmm_HS",
                                           "bisect_step", "force", "eigenstate"};
    return (kind >= 0 && kind < KK_NKINDS) ? names[kind] : "?";
}

// A shape {vpt, threads} of gs_kernel names its partial sums: `threads` chains
// of vpt values each (m_pad = vpt threads), on a CTA of threads / 4 threads.
// Vectors up to 4096 entries take 256 chains, FP32 vectors up to 8192 entries
// 512, longer FP32 vectors 256 pairs of chains (shape {64, 288}; {32, 544}, 512
// pairs, is the other pair shape), the rest 1024 chains.  vpt is the power of
// two that covers m.
ColumnShape column_shape(int64_t m, int prec)
{
    if (prec == 1 && m > 4096 && m <= 8192) return ColumnShape{16, 512, 8192};
    if (prec == 1 && m > 8192 && m <= 16384) return ColumnShape{64, 288, 16384};
    const int T = m <= 4096 ? 256 : 1024;
    int v = 1;
    while (v < 16 && (int64_t)v * T < m) v *= 2;
    return ColumnShape{v, T, (int64_t)v * T};
}

int column_shape_candidates(int64_t m_pad, int prec, ColumnShape *out)
{
    int n = 0;
    for (int T : {256, 512, 1024})
        for (int v = 1; v <= 16; v *= 2)
            if ((int64_t)v * T == m_pad) out[n++] = ColumnShape{v, T, m_pad};
    for (const ColumnShape st : {ColumnShape{32, 544, 16384}, ColumnShape{64, 288, 16384}})
        if (m_pad == st.m_pad && gs_pair_shape(st, prec)) out[n++] = st;
    return n;
}

bool gs_pair_shape(const ColumnShape &s, int prec)
{
    return prec == 1 && s.m_pad == 16384 &&
           ((s.vpt == 32 && s.threads == 544) || (s.vpt == 64 && s.threads == 288));
}

namespace {

// ------------------------------------------------------------------ init
// k_1 = e_j / sqrt(S_jj); S k_1 = (column j of S) / sqrt(S_jj), read from block
// row j/4 (S is symmetric: S[4I+a][j] = S[j][4I+a]).
// Entries are stored at their positions in the column's tile order.
template <typename VT>
__global__ void init_kernel(const int64_t *__restrict__ rp, const int32_t *__restrict__ ci,
                            const double *__restrict__ Sv, const double *__restrict__ sdiag,
                            const int64_t *__restrict__ cols, VT *__restrict__ K,
                            VT *__restrict__ SK, double *__restrict__ scale,
                            int *__restrict__ status, int *__restrict__ nu_eff, int nu,
                            int64_t m_pad, const uint16_t *__restrict__ tinv, int nb, VT *__restrict__ panel,
                            int ntile)
{
    const int c = blockIdx.x;
    const int64_t j = cols[c];
    const int64_t J = j >> 2;
    const int b = (int)(j & 3);
    VT *k0 = K + (int64_t)c * nu * m_pad;
    VT *sk0 = SK + (int64_t)c * nu * m_pad;
    for (int64_t r = threadIdx.x; r < m_pad; r += blockDim.x) {
        k0[r] = VT(0);
        sk0[r] = VT(0);
    }
    __syncthreads();
    const double inv = 1.0 / sqrt(sdiag[j]);
    if (threadIdx.x == 0) {
        k0[vpos(tinv, nb, c, j)] = (VT)inv;
        panel[panel_pos(ntile, c, J) + b] = (VT)inv;
        scale[(int64_t)c * nu] = 1.0;
        status[c] = 0;
        nu_eff[c] = nu;
    }
    for (int64_t k = rp[J] + threadIdx.x; k < rp[J + 1]; k += blockDim.x) {
        const int64_t I = ci[k];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int64_t q = vpos(tinv, nb, c, 4 * I + a);
            if (in_range(q, m_pad, kChkInitPos)) sk0[q] = (VT)(Sv[16 * k + 4 * b + a] * inv);
        }
    }
}

// ------------------------------------------------------------------ SpMM
__device__ __forceinline__ void lds_x4(uint32_t a, uint64_t (&v)[4])
{
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(v[0]), "=l"(v[1]) : "r"(a));
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(v[2]), "=l"(v[3]) : "r"(a + 16));
}
__device__ __forceinline__ void lds_d4(uint32_t a, double (&v)[4])
{
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "r"(a));
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v[2]), "=d"(v[3]) : "r"(a + 16));
}
// H x and S x for the same panel in one pass (both feed the Gram-Schmidt step
// of the same Krylov vector, and H and S share their block pattern): each x
// entry is gathered once for both products.  A warp takes one block row for 32 NC
// columns, a lane the columns 32 NC g + lane (+ 32); a CTA's W
// warps take W consecutive rows, which share most of their neighbours.  Rows
// run fastest in the grid, so the CTAs in flight work on a few column groups
// whose input panels stay in L2.
//
// The input is the panel that the Gram-Schmidt step wrote beside the vector's
// slot: atom-major, kPanel columns side by side, zero outside the supports.
// Gathering a block's x from the columns' own slots, each in its own tile
// order, touched 32 lines per load and held the L1 at 75 %: 16,384 columns of
// 4,096 atoms, nu = 30, 190.1 ms, now 145.7 (the Gram-Schmidt step pays 9 ms for
// the panel; 13 with 16 columns side by side, whose product is 0.8 ms faster).
// Column c's y are stored in its tile order: block row I at position
// 8 tinv[I / 8] + I % 8 (4 entries each).  Support: row I of column c vanishes
// when its tile lies more than `lim` hops from the column's atom (thop > lim;
// the input vanishes beyond lim - 1); a warp with no live lane only writes
// zeros.
//
// FP64: plain FMAs.  Mixed precision (matrix blocks stored as 16 "hi" then 16
// "lo" FP32 values, hi + lo = the FP64 value to about 2^-48): the subspace
// matrix entries h_{i,n} = k_i . u take u = H k_n at face value, so u is
// formed to about 2^-48: each product with hi is split exactly (p + e,
// e = fma(h, x, -p)) and summed with exact two-sums, the lo products and the
// errors collect in a second FP32 word, and u is written as a normalised
// (hi, lo) FP32 pair; the Krylov vector itself continues from the hi word.
// S x is plain FP32 with the hi values: its rounding only perturbs the
// Gram-Schmidt coefficients and the norms, which G and the subspace Galerkin
// step absorb.  A lane's two columns share one packed instruction (f32x2).
//
// What bounds it: the FP32 pipe, 68 % busy (12 operations per matrix entry and
// column); FP64: the FP64 pipe.  The warp's blocks go through its own two slots
// of shared memory, each value twice (FP32), so that one 16-byte broadcast read
// gives two packed operands; block q + 2 is on its way from L2 and block q + 1's
// x entries are loaded while block q computes.
template <typename VT> struct SpmmCfg {
    static constexpr bool kF = sizeof(VT) == 4;
    // shared memory per block: H hi, H lo and S, each value twice (FP32); H and S (FP64)
    static constexpr int kSmem = kF ? 48 * 8 : 32 * 8;
};

template <typename VT, bool kS, int W, int NC>
__global__ void __launch_bounds__(32 * W, (sizeof(VT) == 4 ? 20 : 16) / W) spmm_hs_kernel(
    int nbr, const int64_t *__restrict__ rp, const int32_t *__restrict__ ci,
    const VT *__restrict__ Hv, const VT *__restrict__ Sv, const VT *__restrict__ panel, int ntile,
    VT *__restrict__ U, VT *__restrict__ Ulo, int64_t ldu, VT *__restrict__ SY, int64_t ldsy,
    int ncols, const uint8_t *__restrict__ thop, const uint16_t *__restrict__ tinv, int lim)
{
    using Cfg = SpmmCfg<VT>;
    constexpr bool kF = Cfg::kF;
    static_assert(!kF || NC == 2, "FP32 columns go in pairs");
    __shared__ __align__(16) unsigned char blk[W][2][Cfg::kSmem];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int I = (int)blockIdx.x * W + warp, tile = I >> 3;
    if (I >= nbr) return;   // uniform over the warp
    int cc[NC];
    bool act = false;
    int64_t yo[NC];
#pragma unroll
    for (int h = 0; h < NC; ++h) {
        cc[h] = (int)blockIdx.y * (32 * NC) + 32 * h + lane;
        act |= cc[h] < ncols && (int)thop[(int64_t)tile * ncols + cc[h]] <= lim;
        // no position: past the columns, or a row of another structure of a
        // union, whose tiles may sit past this column's positions
        yo[h] = cc[h] < ncols ? 32 * (int64_t)tinv[(int64_t)tile * ncols + cc[h]] + 4 * (I & 7) : ldu;
    }
    uint64_t hi[4], lo[4], sy[4];   // FP32: per row entry, the two columns
    double hd[NC][4], sd[NC][4];    // FP64
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        hi[a] = lo[a] = sy[a] = 0;
#pragma unroll
        for (int h = 0; h < NC; ++h) hd[h][a] = sd[h][a] = 0.0;
    }
    if (__any_sync(kFull, act)) {
        const int64_t k0 = rp[I];
        const int nk = (int)(rp[I + 1] - k0);
        const VT *xp0 = panel + panel_pos(ntile, cc[0], 0);
        const int dx = 32 / kPanel * ntile * (32 * kPanel);   // to the column 32 further
        int jv = 0;   // column atoms of blocks 32 (q / 32) + lane
        auto column = [&](int q) {
            if ((q & 31) == 0) jv = k0 + q + lane < k0 + nk ? ci[k0 + q + lane] : 0;
            return __shfl_sync(kFull, jv, q & 31);
        };
        // this lane's 16 bytes of a block: H (lanes 0-7), then S (FP32: its hi
        // values only, lanes 8-11; FP64: lanes 8-15)
        const bool loads = lane < 8 || (kS && lane < (kF ? 12 : 16));
        const float4 *src = reinterpret_cast<const float4 *>(lane < 8 ? Hv : Sv) + 8 * k0 + (lane & 7);
        auto fetch = [&](int q) { return loads && q < nk ? __ldg(src + 8 * q) : make_float4(0.f, 0.f, 0.f, 0.f); };
        auto stage = [&](int q, const float4 &v) {
            if (!loads) return;
            float4 *d = reinterpret_cast<float4 *>(blk[warp][q & 1]);
            if constexpr (kF) {
                d[2 * lane] = make_float4(v.x, v.x, v.y, v.y);
                d[2 * lane + 1] = make_float4(v.z, v.z, v.w, v.w);
            } else {
                d[lane] = v;
            }
        };
        auto gather = [&](int J, VT (&x)[NC][4]) {
            if (!in_range(J, 8 * ntile, kChkSpmmGather)) J = 0;
            const VT *p = xp0 + J * (4 * kPanel);
#pragma unroll
            for (int h = 0; h < NC; ++h) load4(p + h * dx, x[h]);
        };
        VT xn[NC][4];
        float4 v = fetch(0);
        gather(column(0), xn);
        stage(0, v);
        v = fetch(1);
#pragma unroll 1
        for (int q = 0; q < nk; ++q) {
            __syncwarp();   // block q is staged, block q - 1 read
            VT x[NC][4];
#pragma unroll
            for (int h = 0; h < NC; ++h)
#pragma unroll
                for (int e = 0; e < 4; ++e) x[h][e] = xn[h][e];
            if (q + 1 < nk) {
                stage(q + 1, v);
                gather(column(q + 1), xn);
                v = fetch(q + 2);
            }
            const uint32_t sb = (uint32_t)__cvta_generic_to_shared(blk[warp][q & 1]);
            if constexpr (kF) {
                uint64_t xp[4], nx[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    xp[e] = pack_x2(x[0][e], x[1][e]);
                    nx[e] = neg_x2(xp[e]);
                }
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    uint64_t h4[4], l4[4], s4[4];
                    lds_x4(sb + 32 * a, h4);
                    lds_x4(sb + 128 + 32 * a, l4);
                    if constexpr (kS) lds_x4(sb + 256 + 32 * a, s4);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        spmm_add(hi[a], lo[a], h4[e], l4[e], xp[e], nx[e]);
                        if constexpr (kS) sy[a] = fma_x2(s4[e], xp[e], sy[a]);
                    }
                }
            } else {
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    double h4[4], s4[4];
                    lds_d4(sb + 32 * a, h4);
                    if constexpr (kS) lds_d4(sb + 128 + 32 * a, s4);
#pragma unroll
                    for (int e = 0; e < 4; ++e)
#pragma unroll
                        for (int h = 0; h < NC; ++h) {
                            hd[h][a] = fma(h4[e], x[h][e], hd[h][a]);
                            if constexpr (kS) sd[h][a] = fma(s4[e], x[h][e], sd[h][a]);
                        }
                }
            }
        }
    }
#pragma unroll
    for (int h = 0; h < NC; ++h) {
        if (yo[h] >= ldu) continue;
        if constexpr (kF) {
            float yh[4], yl[4], ys[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) {   // renormalise: yh = fl(hi + lo), yl = the rest
                const float fh = h ? lane_y(hi[a]) : lane_x(hi[a]), fl = h ? lane_y(lo[a]) : lane_x(lo[a]);
                yh[a] = __fadd_rn(fh, fl);
                yl[a] = __fsub_rn(fl, __fsub_rn(yh[a], fh));
                ys[a] = h ? lane_y(sy[a]) : lane_x(sy[a]);
            }
            store4(U + (int64_t)cc[h] * ldu + yo[h], yh);
            store4(Ulo + (int64_t)cc[h] * ldu + yo[h], yl);
            if constexpr (kS) store4(SY + (int64_t)cc[h] * ldsy + yo[h], ys);
        } else {
            store4(U + (int64_t)cc[h] * ldu + yo[h], hd[h]);
            if constexpr (kS) store4(SY + (int64_t)cc[h] * ldsy + yo[h], sd[h]);
        }
    }
}

// ------------------------------------------------------------------ Gram-Schmidt
// One CTA per column, of G groups of T = C / 4 threads, for vectors of m_pad =
// nchunk C entries; G = 1, or 2 or 4 where columns are few (gs_shape).  The groups
// share a step's work without touching a sum: in sweep 1 they take the blocks of
// stored vectors in turn, in sweep 2 the passes of four chunks (whose sums a_i
// are then added in the order of the passes at the end), and the scalar step
// runs on all warps.  Vectors are stored in the column's tile order (tiles of 32 entries
// by hop count from the column's atom), and vector i vanishes past its first
// tcnt[i + 1] tiles (S w_i reaches one hop further than w_i), so each sweep
// reads a prefix; the entries past a support are exact zeros, so no sum
// changes.  Thread t owns four entries of every chunk of C (FP32: positions
// 4 t .. 4 t + 3, one 16-byte load; FP64: 2 t, 2 t + 1 and C / 2 further, two).
//
// Orthogonalisation (one pass, with the exact S-Gram matrix).  The stored
// vectors w_i, scaled to unit S-norm (k_i = s_i w_i), are S-orthonormal only
// up to rounding; their Gram matrix G = K^T S K = L L^T is kept exactly
// through L^-1 (its new row every step from G's new column), so that every
// solve with G is a pair of matrix-vector products.  Step n makes two sweeps
// over the stored vectors i <= n, in blocks of kGsBlock:
//   1. over S w_i:  b_i = (S w_i) . u    right-hand side of the S-projection of u
//                   g_i = (S w_i) . w_n  G's column n (g_n = beta_n^2)
//      then, in FP64 over the CTA, the norm, the breakdown test and the
//      S-projection coefficients c = G^-1 p of s_n u onto span(K);
//   2. over w_i:    w_{n+1} = s_n u - sum_i c_i k_i, and
//                   a_i = w_i . u        H_sub entries of the stored basis (u = H w_n)
// a_i feeds nothing before the eigensolve, so it needs no sweep of its own:
// two vector reads per stored vector and step, where a first sweep with a, b
// and g and a second for the subtraction read three.  Whatever rounding leaves
// along span(K) is carried by G, so the subspace problem, solved on
// L^-1 H_sub L^-T, is the exact Rayleigh-Ritz projection on the stored
// vectors.  The subspace is span{e_j, H e_j, ...} whatever the coefficients,
// so in exact arithmetic this is the method's Arnoldi basis.
//
// In mixed precision a_i and g_i are accumulated error-free (exact FP32
// products, two-sums, (hi, lo) pairs; the lo word of u, which only corrects
// a_i by about 2^-24, through plain FMAs).  b_i is summed with plain FMAs in C
// chains per CTA (one per position modulo C; the sums of the chains stay
// accurate): its rounding only leaves a component of w_{n+1} along span(K) at
// the level the FP32 subtraction leaves anyway, which G records.  The chains
// of b and g, and the tree that adds them up, are those of a CTA of C threads
// of one entry per chunk each, so a shape's results do not depend on how many
// of its chains a thread carries.  (Vectors of 16,384 FP32 entries join
// neighbouring chains in pairs first.)  The coefficients and G are FP64.
//
// What bounds it: FP32 vectors, the issue slots (54 % at 0.51 of the HBM
// bandwidth; about 32 FP32 operations per entry and stored vector, in packed
// pairs) and the reductions, a fixed cost per warp and block of four vectors:
// four entries per thread and chunk divide them by four against one thread per
// chain.  FP64 vectors: the two-lane FP64 pipe, 93 % busy (four FMAs per entry
// and stored vector).  Every copy goes through a ring in shared memory that
// each thread fills for itself (cp.async), so that no registers wait for HBM
// and a warp needs no barrier before its block's sums.
// Per solve, against one thread per chain and a, b and g in one sweep (three
// vector reads): 8,192 columns of 8,192 FP32 entries, nu = 30: 46.5 ms (was
// 121.1); 24,000 of 1,024, nu = 30: 27.7 (47.8); 4,000 of 1,024, nu = 100: 50.8
// (86.3); 2,048 of 2,048, nu = 100: 45.2 (72.0).  FP64: 4,004 of 4,096, nu = 30:
// 50.8 (65.0); 2,048 of 16,384, nu = 30: 82.6 (100.1); 348 of 4,096, nu = 300:
// 531 (681).  16,384 columns of 16,384 FP32 entries, nu = 30: 160.8 ms, where a
// kernel with the stored vectors streamed by a producer warp's bulk copies, two
// CTAs per SM, took 227.7: it read each vector three times and its 16 consumer
// warps per SM waited for their own arithmetic's latency.  More ring stages hold
// back CTAs: 161.4 ms with four, 165.4 with five.  The input panel of the next
// product, written too since (see the SpMM), added 2.3 ms to the first figure, 0.7 to
// the 2,048 columns and 10 to the last.

// Four entries of a vector: FP32 as two packed pairs, FP64 as four doubles.
template <typename VT> struct Quad;
template <> struct Quad<float> {
    uint64_t p[2];
    __device__ __forceinline__ void lds(uint32_t a, int)
    {
        asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(p[0]), "=l"(p[1]) : "r"(a));
    }
};
template <> struct Quad<double> {
    double d[4];
    __device__ __forceinline__ void lds(uint32_t a, int h)
    {
        asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(d[2 * h]), "=d"(d[2 * h + 1]) : "r"(a));
    }
};

// 16 bytes global -> shared without a register; groups of such copies per thread.
__device__ __forceinline__ void copy16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Dynamic shared memory: the ring (R stages of six quads per thread: four
// stored vectors, u, and w_n or u's lo word), six FP64 arrays of nu entries, the
// partial sums (sweep 1: b and g for kSpan vectors and C / 32 groups of 32
// chains, FP64 per warp; sweep 2: a per vector and warp, with several groups
// also per pass), the coefficients and the support counts.
template <typename VT, int C, int R, int G, bool kPairs>
struct GsCfg {
    static constexpr int T = C / 4;                               // threads of a group
    static constexpr int NW = T / 32;
    static constexpr int TA = G * T;                              // threads of the CTA
    static constexpr int NP = kPairs ? C / 64 : sizeof(VT) == 4 ? C / 32 : NW;   // partial sums per total
    static constexpr int kSpan = 32;                              // stored vectors per round of totals
    static constexpr int kHalves = sizeof(VT) == 4 ? 1 : 2;       // 16-byte pieces per quad
    static constexpr int kStage = 6 * kHalves * TA * 16;          // bytes
    static constexpr int kPass = 4;                               // chunks per pass of sweep 2 (16 entries per thread)
    // registers: FP32 96 (FP32 at 80: 54.8 against 46.6 ms on 8,192-entry
    // vectors), FP64 (bound by its pipe, which few warps fill) about 150, but two
    // CTAs for C = 1024 (91 against 96 ms on 16,384-entry vectors)
    static constexpr int kMinCtas = G > 1 ? 2 : sizeof(VT) == 4 ? 640 / T : C == 1024 ? 2 : 416 / T;
    static constexpr __host__ __device__ int parts(int nu, int nchunk)   // doubles
    {
        const int a = nu * NW * (G > 1 ? (nchunk + kPass - 1) / kPass : 1);
        return 2 * kSpan * NP > a ? 2 * kSpan * NP : a;
    }
    static size_t smem(int nu, int nchunk)
    {
        return (size_t)R * kStage + ((size_t)nu * 6 + parts(nu, nchunk)) * sizeof(double) + (size_t)nu * sizeof(VT) +
               (size_t)(nu + 2) * sizeof(int);
    }
};

// f(integral constant count) for a run-time count in 1 .. N: a block's loops
// over its vectors unroll for each count, so a short last block costs no FP64
// work on vectors that do not exist (and no branch between independent FMAs).
template <int N, typename F>
__device__ __forceinline__ void for_count(int count, F &&f)
{
    if constexpr (N > 1) {
        if (count < N) {
            for_count<N - 1>(count, f);
            return;
        }
    }
    f(std::integral_constant<int, N>());
}

// The sums over groups of 32 chains of b and g for a block's four vectors
// (FP32): bq[l], gq[l] hold the thread's four chains e.  A group is the chains
// of eight lanes; its 32 chains x_0 .. x_31 are added in the tree of a
// 32-lane reduce-scatter over twelve slots (slot 4 + l for b_l, 8 + l for
// g_l): halves 16, 8, 4, 2, 1 apart, the first operand of each two-sum being
// the half that the slot's number selects.  Lane j of the group ends with
// q = j / 4 (b, g), l = j % 4.
__device__ __forceinline__ uint64_t sel_x2(bool c, uint64_t a, uint64_t b) { return c ? a : b; }
__device__ __forceinline__ PairAcc sel_x2(bool c, const PairAcc &a, const PairAcc &b)
{
    PairAcc r;
    r.hi = sel_x2(c, a.hi, b.hi);
    r.lo = sel_x2(c, a.lo, b.lo);
    return r;
}
__device__ __forceinline__ PairAcc shfl_x2(const PairAcc &a, int o)
{
    PairAcc r;
    r.hi = __shfl_xor_sync(kFull, a.hi, o);
    r.lo = __shfl_xor_sync(kFull, a.lo, o);
    return r;
}
// Per lane of the pair, first.merge(second), own being the first when
// own_first: hi and the two-sum's error are symmetric in the operands, only
// lo = lo_first + (lo_second + error) is not.
__device__ __forceinline__ PairAcc merge_x2(bool own_first, const PairAcc &own, const PairAcc &other)
{
    PairAcc r;
    uint64_t err;
    asm("{\n\t.reg .b64 bb, t, u;\n\t"
        "add.rn.f32x2 %0, %2, %3;\n\t"
        "sub.rn.f32x2 bb, %0, %2;\n\t"
        "sub.rn.f32x2 t, %0, bb;\n\t"
        "sub.rn.f32x2 t, %2, t;\n\t"
        "sub.rn.f32x2 u, %3, bb;\n\t"
        "add.rn.f32x2 %1, t, u;\n\t}"
        : "=&l"(r.hi), "=l"(err)
        : "l"(own.hi), "l"(other.hi));
    asm("{\n\t.reg .b64 t;\n\t"
        "add.rn.f32x2 t, %2, %3;\n\t"
        "add.rn.f32x2 %0, %1, t;\n\t}"
        : "=l"(r.lo)
        : "l"(sel_x2(own_first, own.lo, other.lo)), "l"(sel_x2(own_first, other.lo, own.lo)), "l"(err));
    return r;
}
__device__ __forceinline__ DotAcc<float> chain_tree(const uint64_t (&bq)[kGsBlock][2], const PairAcc (&gq)[kGsBlock][2])
{
    const int lane = threadIdx.x & 31;
    const bool j2 = (lane & 4) != 0, j1 = (lane & 2) != 0, j0 = (lane & 1) != 0;
    // 16 chains apart = 4 lanes apart: lanes 0-3 take b, lanes 4-7 g; both
    // keep their own half first
    PairAcc a[4][2];
#pragma unroll
    for (int l = 0; l < 4; ++l)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            PairAcc b;
            b.hi = bq[l][h];
            a[l][h] = merge_x2(true, sel_x2(j2, gq[l][h], b), shfl_x2(sel_x2(j2, b, gq[l][h]), 4));
        }
    // 8 chains = 2 lanes apart: lane bit 1 takes vectors l / 2; b's first
    // operand is the upper half, g's the lower
    PairAcc c2[2][2];
#pragma unroll
    for (int l = 0; l < 2; ++l)
#pragma unroll
        for (int h = 0; h < 2; ++h)
            c2[l][h] = merge_x2(j1 != j2, sel_x2(j1, a[l + 2][h], a[l][h]), shfl_x2(sel_x2(j1, a[l][h], a[l + 2][h]), 2));
    // 4 chains = 1 lane apart: lane bit 0 takes l % 2; the first operand is the
    // half numbered l / 2
    PairAcc c1[2];
#pragma unroll
    for (int h = 0; h < 2; ++h)
        c1[h] = merge_x2(j0 == j1, sel_x2(j0, c2[1][h], c2[0][h]), shfl_x2(sel_x2(j0, c2[0][h], c2[1][h]), 1));
    // 2 chains apart (first: the half numbered l % 2), then neighbours
    return merge_x2(!j0, c1[0], c1[1]).joined();
}

// The same for chains in pairs: two neighbouring chains are joined first (b by
// a plain addition, g by a two-sum, lower lane first) and the 32 pairs of 16
// lanes added in that tree.  Lanes j and j + 1 (j even) end with q = j / 8 % 2,
// l = j / 2 % 4 of their 16 lanes.
__device__ __forceinline__ DotAcc<float> pair_tree(const uint64_t (&bq)[kGsBlock][2], const PairAcc (&gq)[kGsBlock][2])
{
    const int lane = threadIdx.x & 31;
    const bool j3 = (lane & 8) != 0, j2 = (lane & 4) != 0, j1 = (lane & 2) != 0, j0 = (lane & 1) != 0;
    PairAcc a[4];
#pragma unroll
    for (int l = 0; l < 4; ++l) {
        PairAcc b, g;
        b.hi = pack_x2(__fadd_rn(lane_x(bq[l][0]), lane_y(bq[l][0])), __fadd_rn(lane_x(bq[l][1]), lane_y(bq[l][1])));
        const DotAcc<float> g0 = gq[l][0].joined(), g1 = gq[l][1].joined();
        g.hi = pack_x2(g0.hi, g1.hi);
        g.lo = pack_x2(g0.lo, g1.lo);
        a[l] = merge_x2(true, sel_x2(j3, g, b), shfl_x2(sel_x2(j3, b, g), 8));
    }
    PairAcc c2[2];
#pragma unroll
    for (int l = 0; l < 2; ++l)
        c2[l] = merge_x2(j2 != j3, sel_x2(j2, a[l + 2], a[l]), shfl_x2(sel_x2(j2, a[l], a[l + 2]), 4));
    const PairAcc c1 = merge_x2(j1 == j2, sel_x2(j1, c2[1], c2[0]), shfl_x2(sel_x2(j1, c2[0], c2[1]), 2));
    return merge_x2(j0 == j1, c1, shfl_x2(c1, 1)).joined();
}

template <typename VT, int C, int R, int G = 1, bool kPairs = false>
__global__ void __launch_bounds__(G * C / 4, GsCfg<VT, C, R, G, kPairs>::kMinCtas) gs_kernel(
    VT *__restrict__ K, const VT *__restrict__ SK, const VT *__restrict__ U, const VT *__restrict__ Ulo,
    double *__restrict__ Hsub, double *__restrict__ Lsub, double *__restrict__ scale,
    double *__restrict__ cn2, int *__restrict__ status, int *__restrict__ nu_eff,
    const int *__restrict__ tcnt, const uint16_t *__restrict__ tord, VT *__restrict__ panel, int ntile, int64_t MP,
    int n, int nu, int need_w, double tau2)
{
    using Cfg = GsCfg<VT, C, R, G, kPairs>;
    constexpr bool kF = sizeof(VT) == 4;
    constexpr int T = Cfg::T, TA = Cfg::TA, NW = Cfg::NW, NP = Cfg::NP, kB = kGsBlock, kH = Cfg::kHalves;
    constexpr int TPC = C / 32;           // tiles per chunk
    constexpr int SC = Cfg::kPass;
    const int c = blockIdx.x;
    if (status[c] != 0) return;
    const int ta = threadIdx.x;                              // thread of the CTA
    const int group = G > 1 ? ta / T : 0, tid = G > 1 ? ta % T : ta;   // its group, thread and warp of the group
    const int warp = tid >> 5, lane = tid & 31;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *ssc = reinterpret_cast<double *>(smem_raw + R * Cfg::kStage);   // s_i, then s_n
    double *tb = ssc + nu, *tg = tb + nu;                   // the sweep's totals
    double *lrow = tg + nu;                                 // L^-1 G_{<n, n}
    double *nrow = lrow + nu;                               // the new row n of L^-1
    double *zc = nrow + nu;                                 // L^-1 p
    double *part = zc + nu;                                 // partial sums
    VT *coef = reinterpret_cast<VT *>(part + Cfg::parts(nu, (int)(MP / C)));   // subtraction coefficients c_i s_i
    int *cnt_s = reinterpret_cast<int *>(coef + nu);
    __shared__ int bc_stop;
    __shared__ double bc_dinv;
    const int64_t base = (int64_t)c * nu * MP;
    for (int i = ta; i < n; i += TA) ssc[i] = scale[(int64_t)c * nu + i];
    for (int L = ta; L <= n + 1; L += TA) {
        const int t = tcnt[(int64_t)c * (nu + 2) + L];
        cnt_s[L] = in_range(t, MP / 32 + 1, kChkSupportCount) ? t : (int)(MP / 32);
    }
    __syncthreads();
    const int cnt_u = cnt_s[n + 1];                     // tiles of u's support (and of w_{n+1})
    const int nb1 = (n + kB) / kB;                      // blocks of stored vectors
    const int nch_u = (cnt_u + TPC - 1) / TPC, nch_all = (int)(MP / C);
    // chunks of block b (its last vector has the largest support; u's is the last block's)
    auto chunks = [&](int b) { return (cnt_s[min(b * kB + kB, n + 1)] + TPC - 1) / TPC; };
    // this thread's entries of a chunk: 16-byte piece h at position off + h C / 2
    const int off = kF ? 4 * tid : 2 * tid;
    constexpr int kHT = TPC / 2;                        // tiles from a piece to the next
    const char *Ut = reinterpret_cast<const char *>(U + (int64_t)c * MP + off);
    const int64_t dW = reinterpret_cast<const char *>(K + base + (int64_t)n * MP) -
                       reinterpret_cast<const char *>(U + (int64_t)c * MP);      // w_n, from u
    const int64_t dL = kF ? reinterpret_cast<const char *>(Ulo) - reinterpret_cast<const char *>(U) : 0;   // u's lo word
    const uint32_t vb = (uint32_t)(MP * sizeof(VT));    // bytes of a vector
    constexpr uint32_t kCB = C * sizeof(VT);            // bytes of a chunk
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(smem_raw) + 16 * ta;
    auto piece = [&](uint32_t slot, int j, int h) { return slot + (j * kH + h) * (TA * 16); };

    // One stage: a chunk of a block's vectors (nbk of them, at src and vb
    // apart), of u and of a sixth vector (d6 bytes from u).  Every thread
    // copies what it alone reads, so a stage needs no barrier, only the
    // thread's own wait.  Tiles from cnt on, past the support of the block's
    // last vector, are neither copied nor read; a shorter vector of the block
    // holds exact zeros up to there, and so does w_n.
    auto copy_stage = [&](uint32_t slot, const char *src, const char *u, int64_t d6, bool six, int nbk, int k, int cnt) {
#pragma unroll
        for (int h = 0; h < kH; ++h)
            if (k + h * kHT < cnt) {
#pragma unroll
                for (int l = 0; l < kB; ++l)
                    if (l < nbk) copy16(piece(slot, l, h), src + l * vb + h * (kCB / 2));
                copy16(piece(slot, 4, h), u + h * (kCB / 2));
                if (six) copy16(piece(slot, 5, h), u + d6 + h * (kCB / 2));
            }
    };
    // the next stage to copy: block pb, chunk pv (of the pass at chunk p0 in sweep 2)
    uint32_t pslot = ring;
    int pb = group, pv = 0, p0 = 0, pch = chunks(pb), pcnt = cnt_s[min(pb * kB + kB, n + 1)];
    const char *ps = reinterpret_cast<const char *>(SK + base + off) + (int64_t)pb * kB * vb, *pu = Ut;
    int pk = off >> 5;   // tile of the thread's first piece
    auto issue1 = [&] {   // sweep 1: the group's blocks in order, then nothing
        if (pb < nb1) {
            copy_stage(pslot, ps, pu, dW, true, n + 1 - pb * kB, pk, pcnt);
            ps += kCB;
            pu += kCB;
            pk += TPC;
            if (++pv == pch) {
                ps += (int64_t)(G * kB) * vb - (int64_t)pch * kCB;
                pu = Ut;
                pk = off >> 5;
                pv = 0;
                if ((pb += G) < nb1) {
                    pch = chunks(pb);
                    pcnt = cnt_s[min(pb * kB + kB, n + 1)];
                }
            }
        }
        copy_commit();
        pslot = pslot == ring + (R - 1) * Cfg::kStage ? ring : pslot + Cfg::kStage;
    };
    auto seek2 = [&] {   // sweep 2: to block pb of the pass at chunk p0
        pch = min(SC, chunks(pb) - p0);
        pcnt = cnt_s[min(pb * kB + kB, n + 1)];
        ps = reinterpret_cast<const char *>(K + base + off) + (int64_t)pb * kB * vb + p0 * kCB;
        pu = Ut + p0 * kCB;
        pk = (off >> 5) + p0 * TPC;
        pv = 0;
    };
    auto issue2 = [&] {   // the group's passes of SC chunks, in each the blocks that reach it, last first
        if (p0 < nch_u) {
            copy_stage(pslot, ps, pu, dL, kF, n + 1 - pb * kB, pk, pcnt);
            ps += kCB;
            pu += kCB;
            pk += TPC;
            if (++pv == pch) {
                if (--pb < 0 || chunks(pb) <= p0) {
                    pb = nb1 - 1;
                    p0 += G * SC;
                }
                if (p0 < nch_u) seek2();
            }
        }
        copy_commit();
        pslot = pslot == ring + (R - 1) * Cfg::kStage ? ring : pslot + Cfg::kStage;
    };

    // ---- sweep 1: b_i and g_i, in rounds of kSpan vectors, the groups taking blocks in turn
    constexpr int kRound = Cfg::kSpan / kB;
    static_assert(kRound % G == 0, "every group keeps its place from round to round");
    uint32_t slot = ring;
    auto next = [&] { slot = slot == ring + (R - 1) * Cfg::kStage ? ring : slot + Cfg::kStage; };
#pragma unroll 1
    for (int s = 0; s + 1 < R; ++s) issue1();
#pragma unroll 1
    for (int b0 = 0; b0 < nb1; b0 += kRound) {
        const int b1 = min(b0 + kRound, nb1);
#pragma unroll 1
        for (int b = b0 + group; b < b1; b += G) {
            const int i0 = b * kB, nch = chunks(b), cnt = cnt_s[min(i0 + kB, n + 1)];
            int k = off >> 5;
            if constexpr (kF) {
                uint64_t bq[kB][2];
                PairAcc gq[kB][2];
#pragma unroll
                for (int l = 0; l < kB; ++l) bq[l][0] = bq[l][1] = 0;
#pragma unroll 1
                for (int v = 0; v < nch; ++v, k += TPC) {
                    issue1();
                    copy_wait<R - 1>();
                    if (k < cnt) {
                        Quad<float> u, w;
                        u.lds(piece(slot, 4, 0), 0);
                        w.lds(piece(slot, 5, 0), 0);
                        const uint64_t nw[2] = {neg_x2(w.p[0]), neg_x2(w.p[1])};
#pragma unroll
                        for (int l = 0; l < kB; ++l) {
                            if (i0 + l > n) break;
                            Quad<float> sr;
                            sr.lds(piece(slot, l, 0), 0);
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                bq[l][h] = fma_x2(sr.p[h], u.p[h], bq[l][h]);
                                gq[l][h].add(sr.p[h], w.p[h], nw[h]);
                            }
                        }
                    }
                    next();
                }
                const DotAcc<float> r = kPairs ? pair_tree(bq, gq) : chain_tree(bq, gq);
                const int j = kPairs ? (lane & 15) >> 1 : lane & 7, i = i0 + (j & 3);
                const int grp = kPairs ? 2 * warp + (lane >> 4) : 4 * warp + (lane >> 3);
                if (i <= n) part[((i % Cfg::kSpan) * 2 + (j >> 2)) * NP + grp] = r.pack();
            } else {
                DotAcc<VT> acc[2 * kB];   // [l] b, [kB + l] g
                for_count<kB>(min(kB, n + 1 - i0), [&](auto nbk) {
#pragma unroll 1
                    for (int v = 0; v < nch; ++v, k += TPC) {
                        issue1();
                        copy_wait<R - 1>();
#pragma unroll
                        for (int h = 0; h < kH; ++h)
                            if (k + h * kHT < cnt) {
                                Quad<VT> sr[nbk], u, w;
                                u.lds(piece(slot, 4, h), h);
                                w.lds(piece(slot, 5, h), h);
#pragma unroll
                                for (int l = 0; l < nbk; ++l) sr[l].lds(piece(slot, l, h), h);
#pragma unroll
                                for (int e = 2 * h; e < 2 * h + 2; ++e)
#pragma unroll
                                    for (int l = 0; l < nbk; ++l) {
                                        if (need_w) acc[l].add(sr[l].d[e], u.d[e]);
                                        acc[kB + l].add(sr[l].d[e], w.d[e]);
                                    }
                            }
                        next();
                    }
                });
                const DotAcc<VT> r = warp_scatter(acc);   // slot lane / 4
                const int q = lane >> 4, i = i0 + ((lane >> 2) & 3);
                if ((lane & 3) == 0 && i <= n) part[((i % Cfg::kSpan) * 2 + q) * NP + warp] = r.pack();
            }
        }
        // totals of the round: the groups of chains (warps) in the tree of a butterfly reduction
        const int j0 = b0 * kB;
        __syncthreads();
        for (int x = ta; x < 2 * (min(b1 * kB, n + 1) - j0); x += TA) {
            DotAcc<VT> v[NP];
#pragma unroll
            for (int j = 0; j < NP; ++j) v[j].unpack(part[x * NP + j]);
            if constexpr (kPairs) {   // in order
#pragma unroll
                for (int j = 1; j < NP; ++j) v[0].merge(v[j]);
            } else {
#pragma unroll
                for (int o = NP / 2; o > 0; o >>= 1)
#pragma unroll
                    for (int j = 0; j < o; ++j) v[j].merge(v[j + o]);
            }
            ((x & 1) ? tg : tb)[j0 + (x >> 1)] = v[0].value();
        }
        __syncthreads();
    }

    // the first stages of sweep 2 are copied during the scalar step
    pslot = slot = ring;
    pb = nb1 - 1;
    p0 = group * SC;
    seek2();
#pragma unroll 1
    for (int s = 0; s + 1 < R; ++s) issue2();

    // ---- scalars: the norm, G's column, the new row of L^-1, the coefficients
    {
        const GsScalarSmem<VT> sm{ssc, tb, tg, lrow, nrow, zc, coef, bc_stop, bc_dinv};
        if (!gs_scalars<VT, TA>(c, n, nu, need_w, tau2, ta, Lsub, scale, cn2, status, nu_eff, sm,
                               [] { __syncthreads(); })) {
            copy_wait<0>();
            return;
        }
    }

    // ---- sweep 2: w_{n+1} = s_n u - sum_i coef_i w_i and a_i = w_i . u, last
    // block first (its support is u's), SC chunks at a time with w_{n+1} in
    // registers.  FP32 vectors: w_{n+1} is a (hi, lo) sum with exact products
    // and two-sums, rounded to FP32 once (s_n u and the projection nearly
    // cancel, so a plain FP32 chain would leave rounding errors of the size of
    // s_n u, not of w_{n+1}, outside span(K)).
    const VT vsn = (VT)ssc[n];
    VT *wo = K + base + (int64_t)(n + 1) * MP;   // the next slot, unnormalised, zeros included
    // and, in global mode, its entries as the next product's input
    auto panel_at = [&](int p) {
        const int I = 8 * tord[(int64_t)c * ntile + (p >> 5)] + ((p >> 2) & 7);
        return panel + panel_pos(ntile, c, I) + (p & 3);
    };
#pragma unroll 1
    for (int v0 = group * SC; v0 < nch_u; v0 += G * SC) {
        PairAcc x[kF ? SC : 1][2];
        double xd[kF ? 1 : SC][4];
#pragma unroll 1
        for (int b = nb1 - 1; b >= 0; --b) {
            const int i0 = b * kB, nch = chunks(b);
            if (nch <= v0) break;   // the blocks before it have no larger support
            const int cnt = cnt_s[min(i0 + kB, n + 1)];
            VT cf[kB];
#pragma unroll
            for (int l = 0; l < kB; ++l) cf[l] = need_w && i0 + l <= n ? coef[i0 + l] : VT(0);
            PairAcc pa[kF ? kB : 1];
            DotAcc<VT> acc[kB];
            if constexpr (kF) {
#pragma unroll
                for (int q = 0; q < SC; ++q) {
                    if (v0 + q >= nch) break;
                    issue2();
                    copy_wait<R - 1>();
                    if (((v0 + q) * C + off) >> 5 < cnt) {
                        Quad<float> u, ul;
                        u.lds(piece(slot, 4, 0), 0);
                        ul.lds(piece(slot, 5, 0), 0);
                        const uint64_t nu2[2] = {neg_x2(u.p[0]), neg_x2(u.p[1])};
                        if (b == nb1 - 1) {
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                x[q][h] = PairAcc();
                                x[q][h].add(pair_of(vsn), u.p[h], nu2[h]);
                                x[q][h].lo = fma_x2(pair_of(vsn), ul.p[h], x[q][h].lo);
                            }
                        }
#pragma unroll
                        for (int l = 0; l < kB; ++l) {
                            if (i0 + l > n) break;
                            Quad<float> w;
                            w.lds(piece(slot, l, 0), 0);
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                pa[l].add(w.p[h], u.p[h], nu2[h]);
                                pa[l].lo = fma_x2(w.p[h], ul.p[h], pa[l].lo);
                                x[q][h].add(w.p[h], pair_of(-cf[l]), pair_of(cf[l]));
                            }
                        }
                    }
                    next();
                }
            } else {
                for_count<kB>(min(kB, n + 1 - i0), [&](auto nbk) {
#pragma unroll
                    for (int q = 0; q < SC; ++q) {
                        if (v0 + q >= nch) break;
                        const int k = ((v0 + q) * C + off) >> 5;
                        issue2();
                        copy_wait<R - 1>();
#pragma unroll
                        for (int h = 0; h < kH; ++h)
                            if (k + h * kHT < cnt) {
                                Quad<VT> w[nbk], u;
                                u.lds(piece(slot, 4, h), h);
#pragma unroll
                                for (int l = 0; l < nbk; ++l) w[l].lds(piece(slot, l, h), h);
#pragma unroll
                                for (int e = 2 * h; e < 2 * h + 2; ++e) {
                                    if (b == nb1 - 1) xd[q][e] = u.d[e] * vsn;
#pragma unroll
                                    for (int l = 0; l < nbk; ++l) {
                                        acc[l].add(w[l].d[e], u.d[e]);
                                        if (need_w) xd[q][e] = fma(-cf[l], w[l].d[e], xd[q][e]);
                                    }
                                }
                            }
                        next();
                    }
                });
            }
            if constexpr (kF) {
#pragma unroll
                for (int l = 0; l < kB; ++l) acc[l] = pa[l].joined();
            }
            // the warp's sums (slot lane / 8), added up over the passes (with
            // several groups at the end); every support holds tile 0, so the
            // first pass sets them all
            DotAcc<VT> r = warp_scatter(acc);
            const int i = i0 + (lane >> 3);
            if ((lane & 7) == 0 && i <= n) {
                double *ps = part + ((G > 1 ? v0 / SC * nu : 0) + i) * NW + warp;
                if (G == 1 && v0 > 0) {
                    DotAcc<VT> y;
                    y.unpack(*ps);
                    r.merge(y);
                }
                *ps = r.pack();
            }
        }
        if (need_w) {
#pragma unroll
            for (int q = 0; q < SC; ++q) {
                const int v = v0 + q;
                if (v >= nch_all) break;
                if constexpr (kF) {
                    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
                    if ((v * C + off) >> 5 < cnt_u)
                        r = make_float4(__fadd_rn(lane_x(x[q][0].hi), lane_x(x[q][0].lo)),
                                        __fadd_rn(lane_y(x[q][0].hi), lane_y(x[q][0].lo)),
                                        __fadd_rn(lane_x(x[q][1].hi), lane_x(x[q][1].lo)),
                                        __fadd_rn(lane_y(x[q][1].hi), lane_y(x[q][1].lo)));
                    *reinterpret_cast<float4 *>(wo + v * C + off) = r;
                    if (panel && (v * C + off) >> 5 < cnt_u) *reinterpret_cast<float4 *>(panel_at(v * C + off)) = r;
                } else {
#pragma unroll
                    for (int h = 0; h < kH; ++h) {
                        const int p = v * C + off + h * (C / 2);
                        const bool a = p >> 5 < cnt_u;
                        const double2 r = a ? make_double2(xd[q][2 * h], xd[q][2 * h + 1]) : make_double2(0.0, 0.0);
                        *reinterpret_cast<double2 *>(wo + p) = r;
                        if (panel && a) *reinterpret_cast<double2 *>(panel_at(p)) = r;
                    }
                }
            }
        }
    }
    if (need_w) {   // zeros past the last pass
        for (int v = (nch_u + SC - 1) / SC * SC + group; v < nch_all; v += G)
#pragma unroll
            for (int h = 0; h < kH; ++h)
                *reinterpret_cast<float4 *>(wo + v * C + off + h * (C / 2)) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    copy_wait<0>();
    __syncthreads();
    const double sn = ssc[n];
    for (int m = ta; m <= n; m += TA) {   // h_m of unit-norm vectors
        const int np = G > 1 ? (chunks(m / kB) + SC - 1) / SC : 1;
        auto sum_of = [&](int j) {   // warp j's, over the passes in order
            DotAcc<VT> y;
            y.unpack(part[m * NW + j]);
            for (int p = 1; p < np; ++p) {
                DotAcc<VT> z;
                z.unpack(part[(p * nu + m) * NW + j]);
                z.merge(y);
                y = z;
            }
            return y;
        };
        DotAcc<VT> s = sum_of(0);
#pragma unroll
        for (int j = 1; j < NW; ++j) s.merge(sum_of(j));
        const double h = s.value() * (ssc[m] * sn);
        Hsub[((int64_t)c * nu + m) * nu + n] = h;
        Hsub[((int64_t)c * nu + n) * nu + m] = h;
    }
}

template <typename VT, int C, int R, int G = 1, bool kPairs = false>
cudaError_t gs_dispatch(const KrylovBatch &b, int n, int need_w, double tau, cudaStream_t s)
{
    using Cfg = GsCfg<VT, C, R, G, kPairs>;
    if (b.shape.m_pad % C != 0 || (int64_t)b.ntile * 32 < b.shape.m_pad || !b.tcnt || !b.Lsub)
        return cudaErrorInvalidValue;
    const size_t smem = Cfg::smem(b.nu, (int)(b.shape.m_pad / C));
    cudaError_t e = allow_dynamic_smem((const void *)gs_kernel<VT, C, R, G, kPairs>, smem);
    if (e != cudaSuccess) return e;
    gs_kernel<VT, C, R, G, kPairs><<<b.nb, Cfg::TA, smem, s>>>(
        (VT *)b.K, (const VT *)b.SK, (const VT *)b.U, (const VT *)b.Ulo, b.Hsub, b.Lsub, b.scale, b.cn2,
        b.status, b.nu_eff, b.tcnt, b.tord, (VT *)b.panel, b.ntile, b.shape.m_pad, n, b.nu, need_w, tau * tau);
    return cudaGetLastError();
}

// A shape of `threads` entries per chunk and vpt chunks: C = threads chains of
// partial sums on a CTA of a quarter as many threads.  Ring stages: FP64 two
// (its arithmetic covers the copies).  FP32 two up to 1,024 entries, where the
// ring's shared memory would hold back the CTAs whose reductions cover each
// other (24,000 columns, nu = 30: 28.9 ms against 32.6 with three), three above
// (2,048 columns of 2,048 entries, nu = 100: 44.9 ms against 48.3 with two).
//
// At most one column per SM: as many groups of threads as make eight warps, for
// vectors of more than 1,024 entries.  One group's two (four) warps reach two of
// the SM's four schedulers, or hide little of each other's latency, where nothing
// else runs on the SM.  Gram-Schmidt of a solve with one group and with several
// (the Krylov vectors' bits are the same): FP64, 4,096 entries, nu = 200, 1 column
// 214 -> 90 ms, 150 columns 218 -> 92; nu = 30, 1 column 4.9 -> 2.4; mixed, 4,096
// entries, nu = 100, 1 column 21.7 -> 7.8; 8,192 entries, nu = 100, 1 column 20.9 ->
// 13.1, 150 columns 21.7 -> 14.0; 16,384 entries (256 pairs of chains), nu = 30, 1
// column 3.2 -> 2.1, 150 columns 3.6 -> 2.5.
// - Two CTAs per SM (at most 128 registers): solves of few columns also run side by
//   side on several streams.  Mixed, 4,096 entries, nu = 60, 150 columns: one CTA
//   per SM is 3 % faster alone, but eight streams take 46 ms per solve, with two
//   CTAs 41 (one group 42).  8,192 entries: sixteen warps are 17 % faster alone, but
//   four streams take 35 ms, with eight warps 31.5 (one group 31).
// - Up to 1,024 entries alone 1.78 -> 1.45 ms (FP64, nu = 30, 150 columns), but four
//   streams of such solves (nu = 60) 24.8 -> 26.7 ms per solve.
// - With more columns the CTAs run in turns: 300 columns, FP64, nu = 100, 4,096
//   entries 54.9 -> 46.8, but 340 columns 68.9 -> 69.7.
// FP64 shapes of 512 chains (only an autotuner's choice) keep one group.
constexpr int kGsFewColumns = 152;

template <typename VT>
cudaError_t gs_shape(const KrylovBatch &b, int n, int need_w, double tau, cudaStream_t s)
{
    constexpr int R = sizeof(VT) == 4 ? 3 : 2;
    if ((int64_t)b.shape.vpt * b.shape.threads != b.shape.m_pad) return cudaErrorInvalidValue;
    const bool few = b.nb <= kGsFewColumns;
    switch (b.shape.threads) {
    case 256:
        if (few && b.shape.m_pad > 1024) return gs_dispatch<VT, 256, R, 4>(b, n, need_w, tau, s);
        if (R == 3 && b.shape.m_pad <= 1024) return gs_dispatch<VT, 256, 2>(b, n, need_w, tau, s);
        return gs_dispatch<VT, 256, R>(b, n, need_w, tau, s);
    case 512:
        if constexpr (sizeof(VT) == 4)
            if (few) return gs_dispatch<VT, 512, R, 2>(b, n, need_w, tau, s);
        return gs_dispatch<VT, 512, R>(b, n, need_w, tau, s);
    case 1024: return gs_dispatch<VT, 1024, R>(b, n, need_w, tau, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

MARNOLDI_CHECK_TAKE(krylov)

cudaError_t launch_init(const DeviceMatrix &A, const KrylovBatch &b, cudaStream_t s)
{
    if (b.prec == 0)
        init_kernel<double><<<b.nb, 256, 0, s>>>(A.rp, A.ci, A.Sd, A.sdiag, b.cols, (double *)b.K,
                                                 (double *)b.SK, b.scale, b.status, b.nu_eff, b.nu,
                                                 b.shape.m_pad, b.tinv, b.nb, (double *)b.panel, b.ntile);
    else
        init_kernel<float><<<b.nb, 256, 0, s>>>(A.rp, A.ci, A.Sd, A.sdiag, b.cols, (float *)b.K,
                                                (float *)b.SK, b.scale, b.status, b.nu_eff, b.nu,
                                                b.shape.m_pad, b.tinv, b.nb, (float *)b.panel, b.ntile);
    return cudaGetLastError();
}

namespace {

constexpr int64_t kSpmmWarps = 152 * 8;   // fewest warps of a launch with several per CTA

template <typename VT, bool kS>
cudaError_t spmm_hs(const DeviceMatrix &A, const VT *Hv, const VT *Sv, const KrylovBatch &b, void *SY,
                    int64_t ldsy, int lim, cudaStream_t s)
{
    const int64_t ng = (b.nb + 63) / 64, ldu = b.shape.m_pad;
    auto go = [&](auto w, auto nc) {
        constexpr int W = decltype(w)::value, NC = decltype(nc)::value;
        const dim3 grid((unsigned)((A.nbr + W - 1) / W), (unsigned)((b.nb + 32 * NC - 1) / (32 * NC)));
        spmm_hs_kernel<VT, kS, W, NC><<<grid, 32 * W, 0, s>>>(
            (int)A.nbr, A.rp, A.ci, Hv, Sv, (const VT *)b.panel, b.ntile, (VT *)b.U, (VT *)b.Ulo, ldu, (VT *)SY, ldsy, b.nb,
            b.thop, b.tinv, lim);
    };
    // four rows per CTA; one when that leaves SMs without work, and then one FP64
    // column per lane (an FP64 instruction holds the warp's scheduler for 64
    // cycles): 64 atoms, 256 columns, nu = 30: FP64 0.79 ms against 1.30 with two
    // columns and 2.18 with eight rows per CTA, mixed 0.37 against 0.79
    if (A.nbr * ng >= kSpmmWarps) go(std::integral_constant<int, 4>(), std::integral_constant<int, 2>());
    else go(std::integral_constant<int, 1>(), std::integral_constant<int, sizeof(VT) == 4 ? 2 : 1>());
    return cudaGetLastError();
}
}  // namespace

cudaError_t launch_spmm_hs(const DeviceMatrix &A, const KrylovBatch &b, void *SY, int64_t ldsy, int lim,
                           cudaStream_t s)
{
    if (!b.thop || !b.tinv || !b.panel || b.ntile * 8 < A.nbr) return cudaErrorInvalidValue;
    if (b.prec == 0)
        return SY ? spmm_hs<double, true>(A, A.Hd, A.Sd, b, SY, ldsy, lim, s)
                  : spmm_hs<double, false>(A, A.Hd, A.Sd, b, SY, ldsy, lim, s);
    return SY ? spmm_hs<float, true>(A, A.Hf, A.Sf, b, SY, ldsy, lim, s)
              : spmm_hs<float, false>(A, A.Hf, A.Sf, b, SY, ldsy, lim, s);
}

cudaError_t launch_gs(const KrylovBatch &b, int n, int need_w, double tau, cudaStream_t s)
{
    if (gs_pair_shape(b.shape, b.prec)) {
        if (b.shape.threads == 288 && b.nb <= kGsFewColumns)   // see gs_shape
            return gs_dispatch<float, 512, 3, 2, true>(b, n, need_w, tau, s);
        return b.shape.threads == 288 ? gs_dispatch<float, 512, 3, 1, true>(b, n, need_w, tau, s)
                                      : gs_dispatch<float, 1024, 3, 1, true>(b, n, need_w, tau, s);
    }
    return b.prec == 0 ? gs_shape<double>(b, n, need_w, tau, s) : gs_shape<float>(b, n, need_w, tau, s);
}

}  // namespace marnoldi
