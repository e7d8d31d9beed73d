// Device helpers of the Krylov build (krylov.cu, region.cu): packed and
// error-free FP32 dot accumulators, fixed-order warp reductions, and the FP64
// scalar step of one Krylov step (norm, breakdown test, the Gram matrix's new
// column, the new row of L^-1 and the projection coefficients).
#pragma once

#include "internal.h"

namespace marnoldi {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// ------------------------------------------------------------------ dot accumulators
// Per-thread partial inner products.  FP64 vectors: fused multiply-adds in
// FP64.  FP32 vectors (mixed precision): the product a*b of two floats is
// split exactly into p + e (p = fl(a*b), e = fma(a, b, -p)) and p is added to
// the running sum with an exact two-sum, so the pair (hi, lo) carries the sum
// to about 2^-48 relative.  The reduction across the CTA stays in such pairs
// and only the CTA total is converted to FP64, so the inner products are
// FP64-accurate on FP32 data with no per-element FP64 work (GB300 issues
// FP32 at about 64 times its FP64 rate).  The _rn intrinsics keep the
// compiler from contracting the error-free steps into FMAs.
__device__ __forceinline__ void df_add(float &hi, float &lo, float h2, float l2)
{
    const float s = __fadd_rn(hi, h2);
    const float bb = __fsub_rn(s, hi);
    const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(h2, bb));
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(l2, err));
}

template <typename VT> struct DotAcc;
template <> struct DotAcc<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double a, double b) { s = fma(a, b, s); }
    __device__ __forceinline__ double value() const { return s; }
    __device__ __forceinline__ void merge(const DotAcc &o) { s += o.s; }
    __device__ __forceinline__ DotAcc shfl_xor(int o) const
    {
        DotAcc r;
        r.s = __shfl_xor_sync(kFull, s, o);
        return r;
    }
    __device__ __forceinline__ double pack() const { return s; }
    __device__ __forceinline__ void unpack(double p) { s = p; }
};
template <> struct DotAcc<float> {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float a, float b)
    {
        const float p = __fmul_rn(a, b);
        const float e = __fmaf_rn(a, b, -p);
        df_add(hi, lo, p, e);
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
    __device__ __forceinline__ void merge(const DotAcc &o) { df_add(hi, lo, o.hi, o.lo); }
    __device__ __forceinline__ DotAcc shfl_xor(int o) const
    {
        DotAcc r;
        r.hi = __shfl_xor_sync(kFull, hi, o);
        r.lo = __shfl_xor_sync(kFull, lo, o);
        return r;
    }
    __device__ __forceinline__ double pack() const
    {
        union { float2 f; double d; } u;
        u.f = make_float2(hi, lo);
        return u.d;
    }
    __device__ __forceinline__ void unpack(double p)
    {
        union { float2 f; double d; } u;
        u.d = p;
        hi = u.f.x;
        lo = u.f.y;
    }
    __device__ __forceinline__ void set(float x)
    {
        hi = x;
        lo = 0.f;
    }
};


// Two adjacent FP32 values as one 64-bit register (lane x = the lower
// address), and the packed operations on such pairs (add/sub/mul/fma .rn.f32x2,
// sm_100 and later): each lane is rounded exactly as the scalar instruction
// would be, at half the instruction count.
__device__ __forceinline__ uint64_t pair_of(float x)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ uint64_t pack_x2(float x, float y)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ uint64_t fma_x2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t neg_x2(uint64_t a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ float lane_x(uint64_t a) { return __uint_as_float((unsigned)a); }
__device__ __forceinline__ float lane_y(uint64_t a) { return __uint_as_float((unsigned)(a >> 32)); }

// Two DotAcc<float> (one per lane) in packed registers: per lane the
// operations of DotAcc<float>::add.
struct PairAcc {
    uint64_t hi = 0, lo = 0;
    // += a b, with nb = -b given: fma(a, -b, p) is the exact negative of the
    // product's error e, and lo -= (-e - err) rounds as lo += (e + err), so no
    // integer instruction negates p
    __device__ __forceinline__ void add(uint64_t a, uint64_t b, uint64_t nb)
    {
        asm("{\n\t.reg .b64 p, e, s, bb, t, u, err;\n\t"
            "mul.rn.f32x2 p, %2, %3;\n\t"
            "fma.rn.f32x2 e, %2, %4, p;\n\t"
            "add.rn.f32x2 s, %0, p;\n\t"
            "sub.rn.f32x2 bb, s, %0;\n\t"
            "sub.rn.f32x2 t, s, bb;\n\t"
            "sub.rn.f32x2 t, %0, t;\n\t"
            "sub.rn.f32x2 u, p, bb;\n\t"
            "add.rn.f32x2 err, t, u;\n\t"
            "sub.rn.f32x2 e, e, err;\n\t"
            "sub.rn.f32x2 %1, %1, e;\n\t"
            "mov.b64 %0, s;\n\t}"
            : "+l"(hi), "+l"(lo)
            : "l"(a), "l"(b), "l"(nb));
    }
    // the two lanes' sums, joined by a two-sum
    __device__ __forceinline__ DotAcc<float> joined() const
    {
        DotAcc<float> r;
        r.hi = lane_x(hi);
        r.lo = lane_x(lo);
        DotAcc<float> y;
        y.hi = lane_y(hi);
        y.lo = lane_y(lo);
        r.merge(y);
        return r;
    }
};

// (hi, lo) += (h + l) x per lane of the pairs, nx = -x: p = h x, its error and
// l x (negated, so that no integer instruction negates p), and p added to hi
// with a two-sum.
__device__ __forceinline__ void spmm_add(uint64_t &hi, uint64_t &lo, uint64_t h, uint64_t l, uint64_t x, uint64_t nx)
{
    asm("{\n\t.reg .b64 p, e, s, bb, t, u, err;\n\t"
        "mul.rn.f32x2 p, %2, %4;\n\t"
        "fma.rn.f32x2 e, %2, %5, p;\n\t"
        "fma.rn.f32x2 e, %3, %5, e;\n\t"
        "add.rn.f32x2 s, %0, p;\n\t"
        "sub.rn.f32x2 bb, s, %0;\n\t"
        "sub.rn.f32x2 t, s, bb;\n\t"
        "sub.rn.f32x2 t, %0, t;\n\t"
        "sub.rn.f32x2 u, p, bb;\n\t"
        "add.rn.f32x2 err, t, u;\n\t"
        "sub.rn.f32x2 e, e, err;\n\t"
        "sub.rn.f32x2 %1, %1, e;\n\t"
        "mov.b64 %0, s;\n\t}"
        : "+l"(hi), "+l"(lo)
        : "l"(h), "l"(l), "l"(x), "l"(nx));
}

// Vectors per block of the Gram-Schmidt sweeps (one CTA reduction each).
constexpr int kGsBlock = 4;

// Sums of N <= 16 accumulators over a warp: a reduce-scatter butterfly over NP =
// 2^ceil(log2 N) slots; slot q (q < N) ends, summed over the warp, on lanes
// q (32 / NP) .. (q + 1) (32 / NP) - 1 (each lane sends half of its slots per
// round, so N values cost about as many shuffles as two).  Returns the lane's
// slot total.
template <typename VT, int N>
__device__ __forceinline__ DotAcc<VT> warp_scatter(const DotAcc<VT> (&in)[N])
{
    static_assert(N >= 1 && N <= 16, "1 <= N <= 16");
    constexpr int LOGN = N > 8 ? 4 : N > 4 ? 3 : N > 2 ? 2 : N > 1 ? 1 : 0;
    constexpr int NP = 1 << LOGN;
    const int lane = threadIdx.x & 31;
    DotAcc<VT> a[NP];
#pragma unroll
    for (int q = 0; q < N; ++q) a[q] = in[q];
#pragma unroll
    for (int r = 0; r < LOGN; ++r) {
        const int o = 16 >> r, half = NP >> (r + 1);
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int j = 0; j < half; ++j) {
            DotAcc<VT> keep = up ? a[j + half] : a[j];
            const DotAcc<VT> send = up ? a[j] : a[j + half];
            keep.merge(send.shfl_xor(o));
            a[j] = keep;
        }
    }
#pragma unroll
    for (int o = 16 >> LOGN; o > 0; o >>= 1) a[0].merge(a[0].shfl_xor(o));
    return a[0];
}

// sum over the warp of x (every lane holds the total)
__device__ __forceinline__ double warp_total(double x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    return x;
}

// Totals over the warp of eight values per lane: lane l gets that of x[l / 4].
// A reduce-scatter over lanes 16, 8, 4 apart, then 2 and 1: nine additions for
// eight totals, where eight calls of warp_total take forty (an FP64 addition
// holds the SM's two-lane FP64 pipe for 16 cycles per warp).  Each total is the
// sum of the same pairs in the same tree as warp_total's, so the bits are equal.
__device__ __forceinline__ double warp_total8(const double (&x)[8])
{
    const int lane = threadIdx.x & 31;
    double a[4], b[2];
    const bool u16 = (lane & 16) != 0, u8 = (lane & 8) != 0, u4 = (lane & 4) != 0;
#pragma unroll
    for (int j = 0; j < 4; ++j)
        a[j] = (u16 ? x[j + 4] : x[j]) + __shfl_xor_sync(kFull, u16 ? x[j] : x[j + 4], 16);
#pragma unroll
    for (int j = 0; j < 2; ++j) b[j] = (u8 ? a[j + 2] : a[j]) + __shfl_xor_sync(kFull, u8 ? a[j] : a[j + 2], 8);
    double c = (u4 ? b[1] : b[0]) + __shfl_xor_sync(kFull, u4 ? b[0] : b[1], 4);
    c += __shfl_xor_sync(kFull, c, 2);
    return c + __shfl_xor_sync(kFull, c, 1);
}

// Shared-memory arrays of the scalar step (length >= nu each).
template <typename VT>
struct GsScalarSmem {
    double *ssc;    // s_i (i < n) in, s_n set here
    double *tb;     // sweep totals b_i = (S w_i) . u
    double *tg;     // g_i = (S w_i) . w_n
    double *lrow;   // L^-1 G_{<n, n}
    double *nrow;   // the new row n of L^-1
    double *zc;     // L^-1 p
    VT *coef;       // subtraction coefficients c_i s_i
    int &stop;
    double &dinv;
};

// The FP64 scalar step of Krylov step n for column c, run by the T threads
// (thread index tid) that `sync` synchronises, after the sweep's totals are in
// tb, tg: beta_n and the breakdown test, s_n, G's column n, the new row of
// L^-1 (into Lsub), and, when need_w, the coefficients c = L^-T L^-1 p of
// s_n u into coef and |L^-1 p|^2 into cn2[c].  Returns false when the column
// stopped.  Lsub holds L^-1 (lower triangular), so every product is a
// matrix-vector product with no serial chain; a warp takes eight rows (or
// columns) at a time and reduces them together (warp_total8), and the two
// products with the same rows (L^-1 G_{<n,n} and L^-1 p) share one pass.  The
// step is bound by the FP64 pipe: one total per row and product spent 5 of
// about 6.5 FP64 instructions per row on its reduction at nu = 100.
template <typename VT, int T, typename Sync>
__device__ __forceinline__ bool gs_scalars(int c, int n, int nu, int need_w, double tau2, int tid,
                                           double *__restrict__ Lsub,
                                           double *__restrict__ scale, double *__restrict__ cn2,
                                           int *__restrict__ status, int *__restrict__ nu_eff,
                                           GsScalarSmem<VT> sm, Sync sync)
{
    const int warp = tid >> 5, lane = tid & 31;
    constexpr int NW = T / 32;
    double *Lc = Lsub + (int64_t)c * nu * nu;   // L^-1, row-major, lower triangle
    if (tid == 0) {
        double sn = 1.0;   // slot 0 is stored normalised (G_00 = 1)
        int stop = 0;
        if (n > 0) {
            const double beta2 = sm.tg[n];
            if (!(beta2 > 0.0) || beta2 <= tau2 * (beta2 + cn2[c])) {
                stop = 1;
                // a square norm below zero by no more than the threshold times the
                // projected part is rounding at breakdown (FP32 vectors near linear
                // dependence); further below, or NaN, it is not a norm (2)
                status[c] = (beta2 >= -sqrt(tau2) * cn2[c]) ? 1 : 2;
                nu_eff[c] = n;
            } else {
                sn = 1.0 / sqrt(beta2);
                scale[(int64_t)c * nu + n] = sn;
            }
        }
        sm.ssc[n] = sn;
        sm.stop = stop;
    }
    sync();
    if (sm.stop) return false;
    const double sn = sm.ssc[n];
    for (int m = tid; m <= n; m += T) {   // G_{mn} and p_m (of s_n u) of unit-norm vectors
        const double f = sm.ssc[m] * sn;
        sm.tg[m] *= f;
        sm.tb[m] *= f;
    }
    sync();
    // l = L^-1 G_{<n, n} and z = L^-1 p (rows below n)
    for (int r0 = 8 * warp; r0 < n; r0 += 8 * NW) {
        double x[8], y[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = y[j] = 0.0;
        const int mend = min(r0 + 8, n);
        for (int m = lane; m < mend; m += 32) {
            const double g = sm.tg[m], pm = need_w ? sm.tb[m] : 0.0;
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (m <= r0 + j && r0 + j < n) {
                    const double l = Lc[(int64_t)(r0 + j) * nu + m];
                    x[j] = fma(l, g, x[j]);
                    if (need_w) y[j] = fma(l, pm, y[j]);
                }
        }
        const int r = r0 + (lane >> 2);
        const double tx = warp_total8(x);
        if ((lane & 3) == 0 && r < n) sm.lrow[r] = tx;
        if (need_w) {
            const double ty = warp_total8(y);
            if ((lane & 3) == 0 && r < n) sm.zc[r] = ty;
        }
    }
    sync();
    // d = sqrt(G_nn - |l|^2), G_nn = 1; the new row of L^-1 is (-l^T L^-1, 1) / d
    if (warp == 0) {
        double x = 0.0;
        for (int r = lane; r < n; r += 32) x = fma(sm.lrow[r], sm.lrow[r], x);
        x = warp_total(x);
        if (lane == 0) {
            const double dd = 1.0 - x;
            if (!(dd > 0.0)) {   // the stored basis has lost its rank
                sm.stop = 1;
                status[c] = 1;
                nu_eff[c] = n;
            } else {
                sm.dinv = 1.0 / sqrt(dd);
            }
        }
    }
    sync();
    if (sm.stop) return false;
    const double dinv = sm.dinv;
    double *Ln = Lc + (int64_t)n * nu;
    for (int m0 = 8 * warp; m0 < n; m0 += 8 * NW) {
        double x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = 0.0;
        for (int o = lane; m0 + o < n; o += 32)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int r = m0 + j + o;
                if (r < n) x[j] = fma(sm.lrow[r], Lc[(int64_t)r * nu + m0 + j], x[j]);
            }
        const int m = m0 + (lane >> 2);
        const double tx = warp_total8(x);
        if ((lane & 3) == 0 && m < n) {
            sm.nrow[m] = -dinv * tx;
            Ln[m] = -dinv * tx;
        }
    }
    if (tid == 0) {
        sm.nrow[n] = dinv;
        Ln[n] = dinv;
    }
    sync();
    if (!need_w) return true;
    // z's last entry; then c = L^-T z and |z|^2 = |projection of s_n u|_S^2
    if (warp == 0) {
        double x = 0.0;
        for (int m = lane; m <= n; m += 32) x = fma(sm.nrow[m], sm.tb[m], x);
        x = warp_total(x);
        if (lane == 0) sm.zc[n] = x;
    }
    sync();
    for (int m0 = 8 * warp; m0 <= n; m0 += 8 * NW) {
        double x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = 0.0;
        for (int o = lane; m0 + o <= n; o += 32)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int r = m0 + j + o;
                if (r <= n) x[j] = fma(r == n ? sm.nrow[m0 + j] : Lc[(int64_t)r * nu + m0 + j], sm.zc[r], x[j]);
            }
        const int m = m0 + (lane >> 2);
        const double tx = warp_total8(x);
        if ((lane & 3) == 0 && m <= n) sm.coef[m] = (VT)(tx * sm.ssc[m]);
    }
    if (warp == NW - 1) {
        double x = 0.0;
        for (int r = lane; r <= n; r += 32) x = fma(sm.zc[r], sm.zc[r], x);
        x = warp_total(x);
        if (lane == 0) cn2[c] = x;
    }
    sync();
    return true;
}

}  // namespace
}  // namespace marnoldi
