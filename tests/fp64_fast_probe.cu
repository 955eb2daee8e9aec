// Applies the functions of csrc/fp64_fast.cuh and CUDA's operators to arrays (test only).
#include "fp64_fast.cuh"

__global__ void k_apply(const double *__restrict__ a, const double *__restrict__ b, long long n, double *__restrict__ fast,
                        double *__restrict__ op) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double x = a[i], d = b[i];
    double y;
    fast[4 * i] = fp64_fast::divide(x, d);
    op[4 * i] = x / d;
    fast[4 * i + 1] = fp64_fast::reciprocal(x < 0 ? -1.0 : 1.0, d);
    op[4 * i + 1] = (x < 0 ? -1.0 : 1.0) / d;
    const double pos = fabs(d);
    const double s = fp64_fast::root(pos, y);
    fast[4 * i + 2] = s;
    op[4 * i + 2] = sqrt(pos);
    fast[4 * i + 3] = fp64_fast::reciprocal_near(s, y);
    op[4 * i + 3] = 1.0 / op[4 * i + 2];
}

extern "C" int fp64_fast_apply(const double *a, const double *b, long long n, double *fast, double *op) {
    k_apply<<<(unsigned)((n + 255) / 256), 256>>>(a, b, n, fast, op);
    const cudaError_t e = cudaGetLastError();
    return (int)(e ? e : cudaDeviceSynchronize());
}
