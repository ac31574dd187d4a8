// FP64 reciprocals, roots and quotients of the kernels against the compiler's
// IEEE operations, value by value: what differs is counted on the device.
#include "wcc_halfstep.cuh"

using namespace wcc;

__device__ bool same(double a, double b) {
    return __double_as_longlong(a) == __double_as_longlong(b) || (a != a && b != b);
}

// a, b: operands.  bad[0..4]: recip, sqrt, sqrt_and_recip, quotient, cfl_quotients.
__global__ void compare(const double* a, const double* b, long long n, unsigned long long* bad) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double x = a[i], y = b[i];
        if (!same(recip(d3::reg(x)).v, __drcp_rn(x))) atomicAdd(&bad[0], 1ull);
        const double root = __dsqrt_rn(x);
        if (!same(wcc::sqrt(d3::reg(x)).v, root)) atomicAdd(&bad[1], 1ull);
        d3 ic;
        const d3 c = sqrt_and_recip(d3::reg(x), ic);
        if (!same(c.v, root) || !same(ic.v, __drcp_rn(root))) atomicAdd(&bad[2], 1ull);
        if (!same(quotient(d3::reg(x), d3::reg(y)).v, __ddiv_rn(x, y))) atomicAdd(&bad[3], 1ull);
        const double dx = fabs(y), inv_dx = __drcp_rn(dx);
        double dt, lam;
        cfl_quotients(0.25, dx, inv_dx, fabs(x), dt, lam);
        const double want = __ddiv_rn(0.25 * dx, fabs(x));
        if (!same(dt, want) || !same(lam, __ddiv_rn(want, dx))) atomicAdd(&bad[4], 1ull);
    }
}

extern "C" int fp64_ops_compare(const double* a, const double* b, long long n, unsigned long long* bad) {
    double *da = nullptr, *db = nullptr;
    unsigned long long* dbad = nullptr;
    const size_t bytes = (size_t)n * sizeof(double);
    cudaMalloc(&da, bytes);
    cudaMalloc(&db, bytes);
    cudaMalloc(&dbad, 5 * sizeof *dbad);
    cudaMemcpy(da, a, bytes, cudaMemcpyHostToDevice);
    cudaMemcpy(db, b, bytes, cudaMemcpyHostToDevice);
    cudaMemset(dbad, 0, 5 * sizeof *dbad);
    compare<<<152 * 8, 256>>>(da, db, n, dbad);
    cudaMemcpy(bad, dbad, 5 * sizeof *dbad, cudaMemcpyDeviceToHost);
    const cudaError_t e = cudaGetLastError();
    cudaFree(da);
    cudaFree(db);
    cudaFree(dbad);
    return (int)e;
}
