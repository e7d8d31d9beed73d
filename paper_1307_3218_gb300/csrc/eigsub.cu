// Subspace eigensolve of the multiple Arnoldi method on sm_103a.
//
// Each subspace L_nu^(j) gives a nu x nu standard eigenproblem
// H_sub v_a = eps_a v_a whose levels and vectors determine the Green's
// function (arXiv:1307.3218, Section 2).  The outputs need only
//   eps (ascending), V[0][:] and t = V^T q (q = K^T e_j), and P_j = K_pat V,
// i.e. the rows R = [e_1^T; q^T; K_pat] (n_pat + 2 rows) times V.
//
// H_sub is reduced to tridiagonal form T = Q^T H_sub Q by Householder
// reflections and T = Z Lambda Z^T by the implicit-shift QL algorithm
// (Bowdler, Martin, Reinsch & Wilkinson 1968), so R V = (R Q) Z.  Four
// kernels per chunk of subspaces:
//   eig_tridiag_kernel  one CTA per subspace: the reflections, applied to H_sub;
//                       writes d, e and the reflectors
//   eig_ql_kernel       one LANE per subspace: the QL recurrence, a serial chain
//                       of FP64 operations per subspace.  Every rotation is
//                       logged, as the two coefficients of a fast plane
//                       rotation, and every sweep's index range.
//   eig_rank_kernel     one CTA per subspace: the levels in ascending order
//   eig_apply_kernel    one warp per 32 rows of R, packed over the subspaces:
//                       L^-T, the reflectors, then the rotations of the log;
//                       w_a = sqrt(S_jj) (R V)[0][a] (R V)[1][a], t and P_j are
//                       written in ascending order of eps.
// All but the ranking are bound by FP64 instructions (64 cycles each on a warp's
// scheduler): their sum where many warps run, else the longest chain.  The
// reflections used to reach R in the first kernel, whose other threads waited and
// whose shared memory then held one CTA per SM (nu = 100), and a rotation took four
// FP64 instructions per row.  Per solve, then and now (tridiagonalisation, QL, rows):
// 24,000 subspaces of nu = 30: 13.9 + 2.1 + 12.0 -> 5.2 + 2.0 + 7.3 ms; 4,000 of
// nu = 100: 60.6 + 16.7 + 23.6 -> 16.5 + 9.8 + 13.9; 348 of nu = 300: 91.5 + 159.9 +
// 54.7 -> 36.8 + 77.0 + 37.7; 256 of nu = 30: 0.30 + 1.66 + 0.27 -> 0.24 + 1.02 + 0.25.
#include "internal.h"

#include <math_constants.h>

#include <algorithm>
#include <cfloat>

namespace marnoldi {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kTriThreads = 256;    // most threads of the tridiagonalisation
constexpr int kQlMaxIter = 30;      // QL iterations per eigenvalue
constexpr int kQlWarps = 152;       // one QL warp per SM
constexpr int kScaleBits = 930;     // a column scale below 2^-930 counts as no convergence

__device__ __forceinline__ double warp_sum(double s)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
    return s;
}

// ------------------------------------------------------------------ tridiagonalisation
// A = Q T Q^T with Q = P_0 P_1 ... P_{n-3}, P_k = I - tau_k v_k v_k^T on the
// entries k + 1 ...  A is symmetric and only its lower triangle is kept, row by
// row without gaps: entry (i, j <= i) at i (i + 1) / 2 + j.  Half the shared
// memory lets five CTAs share an SM at nu = 100 (two with the square), whose
// phases between barriers then overlap: 16.5 ms for 4,000 subspaces, 27.5 with
// the square.
// Shared memory: A, v, e, q; where eig_smem_bytes says so (nu above 145 for
// 12 blocks per row, 126 for 24) A lives in a global scratch per subspace (Ag)
// instead, which the CTA's sweeps keep in L2 (360 KB at nu = 300).  A thread per
// row of A: the CTA has as many threads as nu needs.
// Reflector k goes to V[sc][k][0 .. n - k - 2], tau_k to V[sc][k][nu - 1].
__device__ __forceinline__ int tri(int i) { return i * (i + 1) / 2; }

__global__ void __launch_bounds__(kTriThreads) eig_tridiag_kernel(
    const double *__restrict__ Hsub, const int *__restrict__ bnu_eff, int nu, int cofs,
    double *__restrict__ D, double *__restrict__ E, double *__restrict__ V, double *__restrict__ Ag,
    const double *__restrict__ Lsub)
{
    const int sc = blockIdx.x;
    const int c = cofs + sc;
    const int n = bnu_eff[c];
    const int tid = threadIdx.x, T = blockDim.x;
    extern __shared__ __align__(16) double sm[];
    double *A = Ag ? Ag + (size_t)sc * nu * (nu | 1) : sm;
    double *v = Ag ? sm : A + tri(nu);
    double *ev = v + nu;
    double *qv = ev + nu;
    double *Vc = V + (int64_t)sc * nu * nu;
    __shared__ double sc4[4];
    __shared__ double wpart[kTriThreads / 32];
    __shared__ int skip;

    for (int i = tid >> 5; i < n; i += T / 32)
        for (int l = tid & 31; l <= i; l += 32)
            A[tri(i) + l] = 0.5 * (Hsub[((int64_t)c * nu + i) * nu + l] + Hsub[((int64_t)c * nu + l) * nu + i]);
    __syncthreads();
    // The stored basis K~ has unit S-norms and S-Gram matrix G = L L^T, so the
    // S-orthonormal basis K = K~ L^-T carries the subspace problem
    // A = L^-1 H~ L^-T.  Lsub holds L^-1 (lower triangular).  First the lower
    // triangle of W = L^-1 A, row i from the last up: it reads rows m <= i of A
    // (and, by symmetry, their columns), which are not yet replaced.  Four
    // sums side by side keep the FP64 pipe supplied.
    const double *Lc = Lsub + (int64_t)c * nu * nu;
    constexpr int kPer = (kMaxNu + kTriThreads - 1) / kTriThreads;   // entries per thread
    for (int i = n - 1; i >= 0; --i) {
        const double *Li = Lc + (int64_t)i * nu;
        double x[kPer];
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const int col = tid + q * T;
            double s[4] = {0.0, 0.0, 0.0, 0.0};
            if (col <= i) {
                // row col left of the diagonal, then down column col, chosen per
                // lane: two loops would run every lane through both bounds
                const int r0 = tri(col);
                int m = 0, d = col;   // d = tri(m) + col
                for (; m + 3 <= i; m += 4)
#pragma unroll
                    for (int z = 0; z < 4; ++z) {
                        s[z] = fma(Li[m + z], A[m + z < col ? r0 + m + z : d], s[z]);
                        d += m + z + 1;
                    }
                for (; m <= i; ++m) {
                    s[0] = fma(Li[m], A[m < col ? r0 + m : d], s[0]);
                    d += m + 1;
                }
            }
            x[q] = (s[0] + s[1]) + (s[2] + s[3]);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kPer; ++q)
            if (tid + q * T <= i) A[tri(i) + tid + q * T] = x[q];
        __syncthreads();
    }
    // then W L^-T, column i from the last on, rows i ..: it reads columns m <= i
    // of W, not yet replaced
    for (int i = n - 1; i >= 0; --i) {
        const double *Li = Lc + (int64_t)i * nu;
        double x[kPer];
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const int row = tid + q * T;
            double s[4] = {0.0, 0.0, 0.0, 0.0};
            if (row >= i && row < n) {
                const double *Ar = A + tri(row);
                int m = 0;
                for (; m + 3 <= i; m += 4)
#pragma unroll
                    for (int z = 0; z < 4; ++z) s[z] = fma(Ar[m + z], Li[m + z], s[z]);
                for (; m <= i; ++m) s[0] = fma(Ar[m], Li[m], s[0]);
            }
            x[q] = (s[0] + s[1]) + (s[2] + s[3]);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kPer; ++q)
            if (tid + q * T >= i && tid + q * T < n) A[tri(tid + q * T) + i] = x[q];
        __syncthreads();
    }

    for (int k = 0; k + 2 < n; ++k) {
        const int L = n - k - 1;  // x = A[k+1 .. n-1][k]
        if (tid < 32) {
            double tail = 0.0;
            for (int l = 1 + tid; l < L; l += 32) {
                const double x = A[tri(k + 1 + l) + k];
                tail += x * x;
            }
            tail = warp_sum(tail);
            if (tid == 0) {
                const double x0 = A[tri(k + 1) + k];
                if (tail == 0.0) {
                    skip = 1;
                    ev[k] = x0;
                    Vc[(int64_t)k * nu + nu - 1] = 0.0;
                } else {
                    const double s = tail + x0 * x0;
                    const double alpha = -copysign(sqrt(s), x0);
                    const double v0 = x0 - alpha;
                    skip = 0;
                    ev[k] = alpha;
                    sc4[0] = 2.0 / (v0 * v0 + tail);   // reflector I - tau v v^T
                    sc4[1] = v0;
                    Vc[(int64_t)k * nu + nu - 1] = sc4[0];
                }
            }
        }
        __syncthreads();
        if (skip) {
            __syncthreads();
            continue;
        }
        const double tauh = sc4[0];
        for (int l = tid; l < L; l += T) {
            const double x = (l == 0) ? sc4[1] : A[tri(k + 1 + l) + k];
            v[l] = x;
            Vc[(int64_t)k * nu + l] = x;
        }
        __syncthreads();
        // p = tau A_sub v, one entry per thread; p goes to q
        double vp = 0.0;
        for (int col = tid; col < L; col += T) {
            const int r0 = tri(k + 1 + col) + (k + 1);
            double s[4] = {0.0, 0.0, 0.0, 0.0};
            int m = 0, d = tri(k + 1) + (k + 1 + col);
            for (; m + 3 < L; m += 4)
#pragma unroll
                for (int z = 0; z < 4; ++z) {
                    s[z] = fma(A[m + z < col ? r0 + m + z : d], v[m + z], s[z]);
                    d += k + m + z + 2;
                }
            for (; m < L; ++m) {
                s[0] = fma(A[m < col ? r0 + m : d], v[m], s[0]);
                d += k + m + 2;
            }
            const double pl = ((s[0] + s[1]) + (s[2] + s[3])) * tauh;
            qv[col] = pl;
            vp = fma(v[col], pl, vp);
        }
        // K = (tau/2) v . p
        vp = warp_sum(vp);
        if ((tid & 31) == 0) wpart[tid >> 5] = vp;
        __syncthreads();
        double kk = 0.0;
        for (int q = 0; q < T / 32; ++q) kk += wpart[q];
        kk *= 0.5 * tauh;
        __syncthreads();
        for (int col = tid; col < L; col += T) qv[col] = fma(-kk, v[col], qv[col]);   // q = p - K v
        __syncthreads();
        // A_sub -= v q^T + q v^T: a warp per row
        for (int a = tid >> 5; a < L; a += T / 32) {
            const double va = v[a], qa = qv[a];
            double *Ar = A + tri(k + 1 + a) + (k + 1);
            for (int b = tid & 31; b <= a; b += 32) Ar[b] = fma(-va, qv[b], fma(-qa, v[b], Ar[b]));
        }
        __syncthreads();
    }
    double *Dc = D + (int64_t)sc * nu, *Ec = E + (int64_t)sc * nu;
    for (int i = tid; i < n; i += T) {
        Dc[i] = A[tri(i) + i];
        Ec[i] = i + 2 < n ? ev[i] : (i + 2 == n ? A[tri(n - 1) + (n - 2)] : 0.0);
    }
}

// 1 / sqrt(a) and 1 / a of normal numbers (with normal results) from the
// hardware's 20-bit estimates by one step of third order (the binomial series of
// (1 - e)^(-1/2) and (1 - e)^(-1) in the estimate's defect e, cut after e^2): what
// is left is rounding, within 1.05 and 0.55 units of the last place.  Few FP64
// instructions (five and three) and no branch for special values.
__device__ __forceinline__ double series_rsqrt(double a)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
    const double e = fma(-(a * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ double series_rcp(double a)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
    const double e = fma(-a, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// ------------------------------------------------------------------ batched QL
// Lane = subspace (lanes < nl of a warp; nl shrinks with the chunk so that few
// subspaces still spread over the SMs).  d and e live in shared memory as
// [i][lane].  The lanes run their sweeps side by side, each at its own level l:
// a lane that finishes a level early goes on with the next one instead of
// waiting for the others.
//
// What bounds it: one warp's FP64 instruction holds its scheduler's FP64 unit
// for 64 cycles whatever the number of active lanes, and a subspace's rotations
// are one chain; so the time is that chain's count of FP64 instructions (19 per
// rotation, 1,216 cycles; about 1,500 are measured, the rest is the latency of the
// chain through f, g and the square root).  Tests that need no FP64 arithmetic (is e(m) negligible, which of
// |c|, |s| is larger) are made on the exponents, and what the chain does not
// wait for runs in the CTA's second warp, on another scheduler: it follows one
// sweep behind and turns each logged rotation into the form the rows use.
//
// Rotation (c, s) of the columns i, i + 1 of a row x takes
//   x_{i+1}' = s x_i + c x_{i+1},  x_i' = c x_i - s x_{i+1};
// the log holds it for x = diag(scale) y (the same for all rows) so that a row
// takes two multiply-adds instead of four FP64 instructions (fast plane
// rotations, W. M. Gentleman 1973).  With (p, q) = (y_{i+1}, y_i) when
// |c| >= |s|, else (y_i, y_{i+1}),
//   y_{i+1}' = p + alpha q,  y_i' = q + beta p,
// where alpha beta <= 0 and a rotation shrinks the two scales by no more than
// 0.7: over the rotations of nu <= 320 they stay far above underflow, and a
// scale below 1e-280 counts as no convergence.  rot = (alpha, |beta|), the
// second negative for the second form.
// Rotations go to rot[sc][0 .. rcap), sweeps (m, lo) to sweep[sc][0 .. scap);
// nsweep[sc] receives the sweep count, or -1 (no convergence in kQlMaxIter
// iterations for some level, or a full log).  Eigenvalues overwrite D,
// unsorted, the scales E.
__device__ __forceinline__ int exponent_of(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
// 2 x of a number far below overflow, on the integer pipe; no effect below the normal range
__device__ __forceinline__ double twice(double x)
{
    return __hiloint2double(__double2hiint(x) + (exponent_of(x) ? 0x100000 : 0), __double2loint(x));
}

template <int kLostBits>
__global__ void __launch_bounds__(64) eig_ql_kernel(const int *__restrict__ bnu_eff, int cofs,
                                                    int nb, int nu, int nl, double *__restrict__ D,
                                                    double *__restrict__ E,
                                                    double2 *__restrict__ rot, int64_t rcap,
                                                    int2 *__restrict__ sweep, int64_t scap,
                                                    int *__restrict__ nsweep)
{
    extern __shared__ __align__(16) double qsm[];
    __shared__ int4 trip[2][32];   // a lane's sweep: m, lo, rotations, -; double-buffered
    __shared__ int more[2];
    __shared__ int fail[32];
    const int lane = threadIdx.x & 31, sc = blockIdx.x * nl + lane;
    const bool mine = lane < nl && sc < nb, first = threadIdx.x < 32;
    double *d = qsm + (mine ? lane : 0);             // d[i] at d[i * nl]
    double *e = d + (size_t)nu * nl;
    double *w = e + (size_t)nu * nl;                 // the scales (second warp)
    const int n = mine ? bnu_eff[cofs + sc] : 0;
    double2 *rl = rot + (int64_t)(mine ? sc : 0) * rcap;
#define DD(i) d[(i) * nl]
#define EE(i) e[(i) * nl]
#define WW(i) w[(i) * nl]
    if (!first) {
        for (int i = 0; i < n; ++i) WW(i) = 1.0;
        for (int t = 0;; t ^= 1) {
            __syncthreads();   // sweep t is logged
            if (!more[t]) break;
            const int4 tr = trip[t][lane];
            double2 *r = rl;
            rl += mine ? tr.z : 0;
            double2 cs = tr.z > 0 ? r[0] : make_double2(1.0, 0.0);
            double wj = tr.z > 0 ? WW(tr.x) : 1.0;
            const int len = (int)__reduce_max_sync(kFull, (unsigned)tr.z);
            for (int q = 0; q < len; ++q)
                if (q < tr.z) {
                    const int i = tr.x - 1 - q;
                    const double cth = cs.x, s = cs.y, wi = WW(i);
                    if (q + 1 < tr.z) cs = r[q + 1];
                    const bool cf = (__double2hiint(cth) & 0x7fffffff) >= (__double2hiint(s) & 0x7fffffff);
                    const double num = cf ? s : cth, den = cf ? cth : s;
                    const double wp = cf ? wi : wj, wq = cf ? wj : wi;
                    const double alpha = (num * wp) * series_rcp(den * wq);
                    const double beta = fabs((num * wq) * series_rcp(den * wp));
                    r[q] = make_double2(alpha, cf ? beta : -beta);
                    WW(i + 1) = den * wq;
                    wj = cf ? den * wp : -(den * wp);
                }
            if (tr.z > 0) WW(tr.x - tr.z) = wj;
        }
        if (mine) {
            bool lost = false;   // rotations only shrink the scales: the last ones tell
            for (int i = 0; i < n; ++i) {
                const double wi = WW(i);
                E[(int64_t)sc * nu + i] = wi;
                lost |= exponent_of(wi) < 1023 - kLostBits;
            }
            fail[lane] = lost;
        }
        __syncthreads();
        return;
    }
    for (int i = 0; i < n; ++i) {
        d[i * nl] = D[(int64_t)sc * nu + i];
        e[i * nl] = E[(int64_t)sc * nu + i];
    }
    int2 *sl = sweep + (int64_t)(mine ? sc : 0) * scap;
    int64_t nrot = 0;
    int nsw = 0, l = 0, iter = 0;
    bool failed = false, done = n == 0;
    // every trip: each unfinished lane's next sweep; at most kQlMaxIter per level
    for (int t = 0;; t ^= 1) {
        int m = l;
        bool go = false;
        while (!done && !go) {
            for (m = l; m < n - 1; ++m) {
                // |e| > eps (|d| + |d'|) for sure when e's exponent is above the
                // larger of the others' less 50 and e is no zero or subnormal
                // number (whose exponent field, 0, says nothing)
                const double em = EE(m), d0 = DD(m), d1 = DD(m + 1);
                if (exponent_of(em) > max(max(exponent_of(d0), exponent_of(d1)) - 50, 0)) continue;
                if (fabs(em) <= DBL_EPSILON * (fabs(d0) + fabs(d1))) break;
            }
            if (m == l) {
                iter = 0;
                done = ++l >= n;
            } else if (++iter > kQlMaxIter || nrot + (m - l) > rcap || nsw >= scap) {
                failed = done = true;
            } else {
                go = true;
            }
        }
        const bool any = __any_sync(kFull, go);
        double g = 0.0, s = 1.0, cth = 1.0, p = 0.0;
        int i = -1, lo = 0;
        if (go) {
            g = (DD(l + 1) - DD(l)) / (2.0 * EE(l));
            g = DD(m) - DD(l) + EE(l) / (g + copysign(sqrt(fma(g, g, 1.0)), g));
            i = m - 1;
            lo = l;
        }
        // One straight block per rotation, so that the chain's waits are filled
        // with what does not hang on it: the next entries are read a rotation
        // ahead, and a rotation's results for d and e are worked out during the
        // next one (at first d(m) itself and a zero, to no effect).
        bool under = false;
        double dj = go ? DD(m) : 0.0;   // d(i + 1)
        double ei = go ? EE(i) : 0.0, di = go ? DD(i) : 0.0;
        double pe0 = 0.0, pe1 = 0.0, pd0 = dj, pd1 = 0.0;   // e(at) = pe0 * pe1, d(at) = pd0 + pd1
        int at = m;
        const int len = (int)__reduce_max_sync(kFull, go ? (unsigned)(m - l) : 0u);
        for (int q = 0; q < len; ++q) {
            if (i >= lo) {
                const int nx = max(i - 1, 0);
                const double en = EE(nx), dn = DD(nx);
                // r = |(f, g)| (the levels and couplings are bounded by the
                // spectrum's width, so f^2 + g^2 neither overflows nor
                // underflows unless both are as good as zero)
                const double f = s * ei, b = cth * ei;
                const double ss = fma(f, f, g * g);
                EE(at) = pe0 * pe1;
                DD(at) = pd0 + pd1;
                const double gd = dj - p, dd = di - gd;
                const double rinv = series_rsqrt(ss);
                const double sn = f * rinv, cn = g * rinv;
                const double r = fma(twice(cn), b, dd * sn);
                const double pn = sn * r, gn = fma(cn, r, -b);
                at = i + 1;
                pd0 = gd;
                if (exponent_of(ss) == 0) {
                    pe0 = 0.0;
                    pe1 = pd1 = 0.0;
                    under = true;
                    lo = i + 1;
                } else {
                    pe0 = ss;
                    pe1 = rinv;
                    pd1 = pn;
                    s = sn;
                    cth = cn;
                    rl[nrot++] = make_double2(cn, sn);
                    p = pn;
                    g = gn;
                    dj = di;
                    ei = en;
                    di = dn;
                    --i;
                }
            }
        }
        if (go) {
            sl[nsw++] = make_int2(m, lo);
            EE(at) = pe0 * pe1;
            DD(at) = pd0 + pd1;
            if (!under) {
                DD(l) = dj - p;
                EE(l) = g;
            }
            EE(m) = 0.0;
        }
        trip[t][lane] = make_int4(m, lo, go ? m - lo : 0, 0);
        if (lane == 0) more[t] = any;
        __syncthreads();
        if (!any) break;
    }
    __syncthreads();   // the second warp's last sweep
    if (!mine) return;
    for (int i = 0; i < n; ++i) D[(int64_t)sc * nu + i] = DD(i);
    nsweep[sc] = failed || fail[lane] ? -1 : nsw;
#undef DD
#undef EE
#undef WW
}

size_t ql_smem(int nu, int nl) { return (size_t)3 * nu * nl * sizeof(double); }

// Subspaces per warp: as few as leave one warp per SM (a sweep of the warp is
// as long as its longest lane's), 16 when 32 would not fit a CTA's shared
// memory beside the kernel's 1.2 KB of static arrays (nu above 300).
int ql_lanes(int nu, int nb2)
{
    int nl = ql_smem(nu, 32) + 2048 > (size_t)227 * 1024 ? 16 : 32;
    while (nl > 1 && (nb2 + nl / 2 - 1) / (nl / 2) <= kQlWarps) nl /= 2;
    return nl;
}

// ------------------------------------------------------------------ levels
// A CTA per subspace: eps in ascending order (ties by index; a NaN level, from
// non-finite input, ranks as +inf, so that the ranks always form a
// permutation) and the order, which takes the place of the levels in D.  The
// comparisons are of integers that order as the doubles do.
__global__ void __launch_bounds__(128) eig_rank_kernel(
    const int *__restrict__ bnu_eff, const int *__restrict__ bstatus, int cofs, int nu, int64_t col0,
    double *__restrict__ D, const int *__restrict__ nsweep, int *__restrict__ nu_eff_out,
    double *__restrict__ eps_out, int *__restrict__ eig_status)
{
    extern __shared__ __align__(16) double asm_[];
    double *d = asm_;
    uint64_t *key = reinterpret_cast<uint64_t *>(d + nu);
    const int sc = blockIdx.x, c = cofs + sc, n = bnu_eff[c];
    const int64_t g = col0 + c;
    double *Dc = D + (int64_t)sc * nu;
    int *order = reinterpret_cast<int *>(Dc);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double x = Dc[i];
        d[i] = x;
        const uint64_t u = (uint64_t)__double_as_longlong(x != x ? CUDART_INF : x + 0.0);   // -0 as 0
        key[i] = u >> 63 ? ~u : u | 0x8000000000000000ull;
    }
    __syncthreads();
    for (int a = threadIdx.x; a < nu; a += blockDim.x) {
        if (a >= n) {
            eps_out[g * nu + a] = 0.0;
            continue;
        }
        const uint64_t ka = key[a];
        int rank = 0;
        for (int b = 0; b < n; ++b) rank += key[b] < ka || (key[b] == ka && b < a);
        order[rank] = a;
        eps_out[g * nu + rank] = d[a];
    }
    if (threadIdx.x == 0) {
        nu_eff_out[g] = n;
        eig_status[g] = (nsweep[sc] < 0 ? 1 : 0) | (bstatus[c] == 2 ? 2 : 0);
    }
}

// ------------------------------------------------------------------ rows and outputs
// Rows of R = [e_1; q; K_pat; (v^T w_i)], one per lane: R L^-T, the
// reflectors, the rotations, the scales.  Bound by FP64 instructions, which
// cost as much for one lane as for 32, so the rows of all subspaces are packed
// without gaps: a CTA is one warp and takes the next `rows` of them, of one
// subspace or of several (a lane then follows its own subspace's log), in
// shared memory as [rows][ldr] (ldr odd).  Every subspace has an even number
// of rows, so its first two share a warp.  With a CTA per subspace, 75 rows
// took three warps and their CTAs filled an SM's four schedulers unevenly.
// 24,000 subspaces of nu = 30: 10.2 -> 7.3 ms; 4,000 of nu = 100: 22.7 -> 13.9;
// 348 of nu = 300: 55.3 -> 37.9.
constexpr int kLogAhead = 4;   // rotations held in registers ahead of their use

template <typename VT>
__global__ void __launch_bounds__(32) eig_apply_kernel(
    const int *__restrict__ bnu_eff, int cofs, int nb2, int nu, int rows, const double *__restrict__ bscale,
    const VT *__restrict__ K, int64_t m_pad, const uint16_t *__restrict__ tinv, int nb,
    const int64_t *__restrict__ bcols, const double *__restrict__ sdiag, const int64_t *__restrict__ rp,
    const int32_t *__restrict__ ci, const int *__restrict__ reg, int n_reg, int64_t col0,
    const double *__restrict__ D, const double *__restrict__ W, const double *__restrict__ V,
    const double *__restrict__ Lsub, const double *__restrict__ proj, const double2 *__restrict__ rot, int64_t rcap,
    const int2 *__restrict__ sweep, int64_t scap, const int *__restrict__ nsweep, double *__restrict__ w_out,
    double *__restrict__ t_out, double *__restrict__ P_out, const int64_t *__restrict__ p_off,
    double *__restrict__ proj_out)
{
    extern __shared__ __align__(16) double asm_[];
    const int lane = threadIdx.x;
    const int ldr = nu | 1;
    // first row of subspace s among all rows: its pattern rows start at
    // p_off / nu, and the others add two rows per subspace (four with a projection
    // row, the last of them unused)
    const int extra = proj ? 4 : 2;
    const int64_t g0 = col0 + cofs, p0 = p_off[g0];
    auto first = [&](int s) { return p_off[g0 + s] - p0 + (int64_t)extra * nu * s; };   // times nu
    const int64_t at = (int64_t)blockIdx.x * rows + lane;
    int lo = 0, hi = nb2;   // the last subspace whose first row is at or before `at`
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (first(mid) <= at * nu) lo = mid; else hi = mid;
    }
    const int sc = lo, c = cofs + sc;
    const int64_t j = bcols[c], J = j >> 2, kb = rp[J];
    const int npat = 4 * (int)(rp[J + 1] - kb);
    const int64_t r64 = at - first(sc) / nu;
    const int r = r64 < npat + 2 + (proj ? 1 : 0) ? (int)r64 : -1;   // -1: past the rows
    const bool own = lane < rows && r >= 0;
    const int n = bnu_eff[c];
    double *R = asm_ + 1;   // x[-1] is read ahead and not used
    double *x = R + (lane < rows ? lane : 0) * ldr;
    if (own) {
        // q = K^T e_j and K_pat (zero for atoms outside a region)
        const int *Rg = reg ? reg + (int64_t)c * n_reg : nullptr;
        int64_t pos = -1;   // the row's position in the column's vectors
        if (r == 1) {
            const int pJ = Rg ? find_sorted(Rg, n_reg, (int)J) : 0;
            pos = vpos(tinv, nb, c, Rg ? 4 * (int64_t)(pJ < 0 ? 0 : pJ) + (j & 3) : j);
        } else if (r >= 2 && r < npat + 2) {
            const int atom = ci[kb + ((r - 2) >> 2)];
            const int64_t lr = Rg ? find_sorted(Rg, n_reg, atom) : atom;
            if (lr >= 0) pos = vpos(tinv, nb, c, 4 * lr + ((r - 2) & 3));
        }
        const VT *Kc = K + (int64_t)c * nu * m_pad;
        const double *si = bscale + (int64_t)c * nu;
#pragma unroll 4
        for (int i = 0; i < n; ++i)
            x[i] = r == 0 ? (i == 0 ? 1.0 : 0.0)
                   : r == npat + 2 ? si[i] * proj[(int64_t)c * nu + i]
                   : pos >= 0 ? si[i] * (double)Kc[(int64_t)i * m_pad + pos] : 0.0;
        // rows 1..: R <- R L^-T (row 0, e_1^T, is unchanged: K^T S e_j =
        // sqrt(S_jj) e_1), four entries at a time from the last down
        const double *Lc = Lsub + (int64_t)c * nu * nu, *Vc = V + (int64_t)sc * nu * nu;
        if (r > 0) {
            for (int i = n - 1; i >= 0; i -= 4) {
                double s[4] = {0.0, 0.0, 0.0, 0.0};
                const double *L0 = Lc + (int64_t)i * nu;
                const int lo4 = i - 3;
                for (int m = 0; m <= lo4; ++m) {   // lo4 < 0: the general loop below
                    const double xm = x[m];
#pragma unroll
                    for (int z = 0; z < 4; ++z) s[z] = fma(xm, L0[m - (int64_t)z * nu], s[z]);
                }
                for (int m = lo4 < 0 ? 0 : lo4 + 1; m <= i; ++m) {
                    const double xm = x[m];
#pragma unroll
                    for (int z = 0; z < 4; ++z)
                        if (i - z >= m) s[z] = fma(xm, L0[m - (int64_t)z * nu], s[z]);
                }
#pragma unroll
                for (int z = 0; z < 4; ++z)
                    if (i - z >= 0) x[i - z] = s[z];
            }
        }
        for (int k = 0; k + 2 < n; ++k) {   // R <- R (I - tau v v^T) on columns k + 1 ..
            const int L = n - k - 1;
            const double *v = Vc + (int64_t)k * nu;
            const double tau = v[nu - 1];
            if (tau == 0.0) continue;
            double *row = x + k + 1;
            double s[4] = {0.0, 0.0, 0.0, 0.0};
            int m = 0;
            for (; m + 3 < L; m += 4)
#pragma unroll
                for (int z = 0; z < 4; ++z) s[z] = fma(row[m + z], v[m + z], s[z]);
            for (; m < L; ++m) s[0] = fma(row[m], v[m], s[0]);
            const double f = -tau * ((s[0] + s[1]) + (s[2] + s[3]));
#pragma unroll 4
            for (m = 0; m < L; ++m) row[m] = fma(f, v[m], row[m]);
        }
        // the next rotations and the next entry are fetched before the current
        // rotation's multiply-adds: the chain through carry is then one
        const int nsw = nsweep[sc];
        // multiply-add per rotation.  The log comes from DRAM, whose lines are
        // asked for 64 rotations early; no branches, which would add to the chain
        const double2 *rl = rot + (int64_t)sc * rcap;
        const int2 *sl = sweep + (int64_t)sc * scap;
        const int last = (int)rcap - 1;
        double2 ring[kLogAhead];
#pragma unroll
        for (int z = 0; z < kLogAhead; ++z) ring[z] = rl[min(z, last)];
        int ahead = kLogAhead;
        int2 sw = nsw > 0 ? sl[0] : make_int2(0, 0);
        for (int q = 0; q < nsw; ++q) {
            const int2 sn = q + 1 < nsw ? sl[q + 1] : make_int2(0, 0);
            double carry = x[sw.x];
            double yi = x[sw.x - 1];
            for (int i = sw.x - 1; i >= sw.y; --i) {
                const double al = ring[0].x, bs = ring[0].y, y = yi;
#pragma unroll
                for (int z = 0; z + 1 < kLogAhead; ++z) ring[z] = ring[z + 1];
                ring[kLogAhead - 1] = rl[min(ahead, last)];
                asm volatile("prefetch.global.L2 [%0];" ::"l"(rl + min(ahead + 64, last)));
                ++ahead;
                yi = x[i - 1];
                const bool sf = __double2hiint(bs) < 0;
                // beta = -sign(alpha) |bs|
                const double beta = __hiloint2double((__double2hiint(bs) & 0x7fffffff) |
                                                         (~__double2hiint(al) & 0x80000000),
                                                     __double2loint(bs));
                const double p = sf ? y : carry, qq = sf ? carry : y;
                carry = fma(beta, p, qq);
                x[i + 1] = fma(al, qq, p);
            }
            x[sw.y] = carry;
            sw = sn;
        }
    }
    __syncwarp();
    // a row's outputs, in ascending order of eps: the lanes run over the levels
    for (int l = 0; l < rows; ++l) {
        const int rr = __shfl_sync(kFull, own ? r : -1, l);
        const int s = __shfl_sync(kFull, sc, l);
        if (rr < 1) continue;   // row 0 goes with row 1
        const int np = __shfl_sync(kFull, npat, l), nn = __shfl_sync(kFull, n, l);
        const int64_t go = g0 + s;
        const int *order = reinterpret_cast<const int *>(D + (int64_t)s * nu);
        const double *wsc = W + (int64_t)s * nu, *xl = R + l * ldr;
        double *out = rr == 1 ? t_out + go * nu : rr == np + 2 ? proj_out + go * nu
                                                               : P_out + p_off[go] + (int64_t)(rr - 2) * nu;
        const double sq = rr == 1 ? sqrt(sdiag[bcols[cofs + s]]) : 0.0;
        for (int a = lane; a < nu; a += 32) {
            const int src = a < nn ? order[a] : 0;
            const double y = a < nn ? xl[src] * wsc[src] : 0.0;
            out[a] = y;
            if (rr == 1) w_out[go * nu + a] = a < nn ? sq * (xl[src - ldr] * wsc[src]) * y : 0.0;
        }
    }
}

// Rows per warp: 32, or fewer where that lets another warp share the SM and
// fewer than two per scheduler fit (nu above about 100): the most rows per
// turn of the fullest scheduler.
int apply_rows(int nu)
{
    int best = 32;
    double rate = 0.0;
    for (int rows = 32; rows >= 16; rows -= 2) {
        const int ctas = (int)((size_t)228 * 1024 / (((size_t)rows * (nu | 1) + 1) * sizeof(double) + 1024));
        const double x = (double)rows * ctas / ((ctas + 3) / 4);
        if (ctas > 0 && x > rate) {
            rate = x;
            best = rows;
        }
        if (ctas >= 8) break;
    }
    return best;
}

template <typename VT>
cudaError_t apply_dispatch(const DeviceMatrix &A, const KrylovBatch &b, const ColumnState &st, int64_t col0,
                           const RegionMaps *rm, const EigScratch &es, int cofs, int nb2, cudaStream_t s)
{
    const int rows = apply_rows(b.nu);
    const size_t smem = ((size_t)rows * (b.nu | 1) + 1) * sizeof(double);
    cudaError_t e = allow_dynamic_smem((const void *)eig_apply_kernel<VT>, smem);
    if (e != cudaSuccess) return e;
    // nr_max bounds a subspace's rows (odd; an even number is laid out)
    const unsigned grid = (unsigned)(((int64_t)nb2 * (es.nr_max + 1) + rows - 1) / rows);
    eig_apply_kernel<VT><<<grid, 32, smem, s>>>(
        b.nu_eff, cofs, nb2, b.nu, rows, b.scale, (const VT *)b.K, b.shape.m_pad, b.tinv, b.nb, b.cols, A.sdiag, A.rp,
        A.ci, rm ? rm->reg : nullptr, rm ? rm->n_reg : 0, col0, es.D, es.E, es.V, b.Lsub, es.proj, es.rot, es.rcap,
        es.sweep, es.scap, es.nsweep, st.w, st.t, st.P, st.p_off, es.proj ? es.proj_out : nullptr);
    return cudaGetLastError();
}

}  // namespace

// The measure that a solve is refused by and that decides where A lives: the
// full square of H_sub (unless a_global), all rows of R and three vectors in one
// CTA's shared memory.  No kernel holds as much (A is a triangle, which would fit
// up to nu = 237, and the rows go 32 at a time); which solves are accepted, and A's
// place, have stayed as they were.
size_t eig_smem_bytes(int nu, int nr_max, bool a_global)
{
    return ((size_t)((a_global ? 0 : nu) + nr_max) * (size_t)(nu | 1) + 3 * (size_t)nu) * sizeof(double);
}

cudaError_t launch_eig(const DeviceMatrix &A, const KrylovBatch &b, const ColumnState &st,
                       int64_t col0, const RegionMaps *rm, const EigScratch &es, cudaStream_t s)
{
    if ((es.proj == nullptr) != (es.proj_out == nullptr)) return cudaErrorInvalidValue;
    const int nu = b.nu;
    const size_t tsmem = ((es.Ag ? 0 : (size_t)nu * (nu + 1) / 2) + 3 * (size_t)nu) * sizeof(double);
    const int tthreads = std::min(kTriThreads, (nu + 31) / 32 * 32);
    cudaError_t e = allow_dynamic_smem((const void *)eig_tridiag_kernel, tsmem);
    if (e != cudaSuccess) return e;
    for (int cofs = 0; cofs < b.nb; cofs += es.chunk) {
        const int nb2 = b.nb - cofs < es.chunk ? b.nb - cofs : es.chunk;
        eig_tridiag_kernel<<<nb2, tthreads, tsmem, s>>>(b.Hsub, b.nu_eff, nu, cofs, es.D, es.E, es.V, es.Ag, b.Lsub);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        const int nl = ql_lanes(nu, nb2);
        const size_t qsmem = ql_smem(nu, nl);
        if ((e = allow_dynamic_smem((const void *)eig_ql_kernel<kScaleBits>, qsmem)) != cudaSuccess) return e;
        eig_ql_kernel<kScaleBits><<<(nb2 + nl - 1) / nl, 64, qsmem, s>>>(
            b.nu_eff, cofs, nb2, nu, nl, es.D, es.E, es.rot, es.rcap, es.sweep, es.scap, es.nsweep);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        const size_t rsmem = (size_t)2 * nu * sizeof(double);
        eig_rank_kernel<<<nb2, std::min(128, (nu + 31) / 32 * 32), rsmem, s>>>(
            b.nu_eff, b.status, cofs, nu, col0, es.D, es.nsweep, st.nu_eff, st.eps, st.eig_status);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        e = b.prec == 0 ? apply_dispatch<double>(A, b, st, col0, rm, es, cofs, nb2, s)
                        : apply_dispatch<float>(A, b, st, col0, rm, es, cofs, nb2, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace marnoldi
