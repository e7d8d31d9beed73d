// Host entries for the tests of the eigensolver's device code, one translation unit with it:
// eig_probe_ql runs the batched QL kernel on tridiagonal matrices given from the host,
// eig_probe_series the reciprocals of its rotations.
#include "eigsub.cu"

#include <vector>

namespace marnoldi {
cudaError_t allow_dynamic_smem(const void *kernel, size_t bytes)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
}  // namespace marnoldi

using namespace marnoldi;

template <int kLostBits>
static int ql(int nb, int n, int nl, double *d, double *e, int *nsweep)
{
    const int64_t rcap = (int64_t)8 * n * n, scap = (int64_t)40 * n;
    const size_t vals = (size_t)nb * n * sizeof(double);
    int *nu_eff = nullptr, *ns = nullptr;
    double *D = nullptr, *E = nullptr;
    double2 *rot = nullptr;
    int2 *sweep = nullptr;
    const std::vector<int> order(nb, n);
    cudaError_t err = cudaMalloc(&nu_eff, nb * sizeof(int));
    if (!err) err = cudaMalloc(&ns, nb * sizeof(int));
    if (!err) err = cudaMalloc(&D, vals);
    if (!err) err = cudaMalloc(&E, vals);
    if (!err) err = cudaMalloc(&rot, nb * rcap * sizeof(double2));
    if (!err) err = cudaMalloc(&sweep, nb * scap * sizeof(int2));
    if (!err) err = cudaMemcpy(nu_eff, order.data(), nb * sizeof(int), cudaMemcpyHostToDevice);
    if (!err) err = cudaMemcpy(D, d, vals, cudaMemcpyHostToDevice);
    if (!err) err = cudaMemcpy(E, e, vals, cudaMemcpyHostToDevice);
    const size_t smem = (size_t)3 * n * nl * sizeof(double);
    if (!err) err = allow_dynamic_smem((const void *)eig_ql_kernel<kLostBits>, smem);
    if (!err) {
        eig_ql_kernel<kLostBits><<<(nb + nl - 1) / nl, 64, smem>>>(nu_eff, 0, nb, n, nl, D, E, rot, rcap, sweep, scap,
                                                                   ns);
        err = cudaGetLastError();
    }
    if (!err) err = cudaMemcpy(d, D, vals, cudaMemcpyDeviceToHost);
    if (!err) err = cudaMemcpy(e, E, vals, cudaMemcpyDeviceToHost);
    if (!err) err = cudaMemcpy(nsweep, ns, nb * sizeof(int), cudaMemcpyDeviceToHost);
    for (void *p : {(void *)nu_eff, (void *)ns, (void *)D, (void *)E, (void *)rot, (void *)sweep}) cudaFree(p);
    return (int)err;
}

// nb matrices of order n: d [nb][n] (the levels on return), e [nb][n] (the column scales on
// return), nsweep [nb]; nl matrices per warp; a scale counts as lost below 2^-bits (0: the
// library's bound).  Returns a CUDA error code.
extern "C" int eig_probe_ql(int nb, int n, int nl, int bits, double *d, double *e, int *nsweep)
{
    switch (bits) {
    case 0: return ql<kScaleBits>(nb, n, nl, d, e, nsweep);
    case 2: return ql<2>(nb, n, nl, d, e, nsweep);
    case 4: return ql<4>(nb, n, nl, d, e, nsweep);
    case 8: return ql<8>(nb, n, nl, d, e, nsweep);
    default: return -1;
    }
}

static __global__ void series_kernel(int n, const double *x, double *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = x[i] > 0.0 ? series_rsqrt(x[i]) : 0.0;
    out[n + i] = x[i] > 0.0 ? rsqrt(x[i]) : 0.0;
    out[2 * n + i] = series_rcp(x[i]);
    out[3 * n + i] = 1.0 / x[i];
}

// out [4][n]: series_rsqrt and CUDA's rsqrt (0 for x <= 0), series_rcp and 1 / x.
extern "C" int eig_probe_series(int n, const double *x, double *out)
{
    double *X = nullptr, *Y = nullptr;
    cudaError_t err = cudaMalloc(&X, n * sizeof(double));
    if (!err) err = cudaMalloc(&Y, 4 * n * sizeof(double));
    if (!err) err = cudaMemcpy(X, x, n * sizeof(double), cudaMemcpyHostToDevice);
    if (!err) {
        series_kernel<<<(n + 255) / 256, 256>>>(n, X, Y);
        err = cudaGetLastError();
    }
    if (!err) err = cudaMemcpy(out, Y, 4 * n * sizeof(double), cudaMemcpyDeviceToHost);
    cudaFree(X);
    cudaFree(Y);
    return (int)err;
}

// Dynamic shared memory of the QL kernel for a chunk of nb subspaces (no GPU needed).
extern "C" int64_t eig_probe_ql_smem(int nu, int nb) { return (int64_t)ql_smem(nu, ql_lanes(nu, nb)); }
