// C in fixed point for the split paths: C_int = round(C 2^{sh_C}), sh_C = top - e_C with
// max|C| < 2^{e_C} (top = W s - 3 for s digits of W bits: |C_int| < 2^{W s - 3} and
// |D_int| < 2^{W s - 2}, inside the range of s balanced digits; a complex vector counts as
// its 2n reals).  Two outputs: int64, or int32 signed pairs (C_int, -C_int) followed by one
// zero pair (the fused DAS kernel reads a move's value with its sign, or zero, in one load).
//
// Small vectors take one cluster of 8 blocks for all of it (clearing the scalars, the
// maximum, the conversion): the memset and the launch that it saves are a tenth of a split
// sigma of FCI(8e,8o) (36 -> 32 us).  The line is at 2^14 values: at 15,876 determinants the
// cluster still gains 2 us, at 48,400 it loses 4 and at 63,504 10 (eight SMs convert what
// the whole GPU would).
#include <cooperative_groups.h>

#include <algorithm>

#include "dependent.cuh"
#include "fci_internal.h"

namespace {

__device__ __forceinline__ unsigned long long abs_bits(double x) {
    return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}
__device__ __forceinline__ unsigned long long warp_max(unsigned long long m) {
    for (int o = 16; o; o >>= 1) m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
    return m;
}
// The shift of a vector whose largest |C| has the bits mb (0: the zero vector).
__device__ __forceinline__ int shift_of(unsigned long long mb, int top) {
    return top - (mb ? (int)((mb >> 52) & 0x7FF) - 1022 : 0);  // max|C| < 2^e (normal numbers)
}

template <bool PAIRS>
__device__ __forceinline__ void store(void *out, int64_t i, double c, int sh) {
    const int64_t v = __double2ll_rn(scalbn(c, sh));
    if (PAIRS) reinterpret_cast<int2 *>(out)[i] = make_int2((int)v, -(int)v);
    else reinterpret_cast<int64_t *>(out)[i] = v;
}

constexpr int SMALL_BLOCKS = 8, SMALL_THREADS = 512;
constexpr int64_t SMALL_VALUES = (int64_t)1 << 14;  // the line above
template <bool PAIRS>
__global__ void __cluster_dims__(SMALL_BLOCKS, 1, 1) __launch_bounds__(SMALL_THREADS)
    k_fixed_small(const double *__restrict__ C, int64_t n, int top, fci_split_scalars *__restrict__ sc,
                  void *__restrict__ out) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ unsigned long long warp_part[SMALL_THREADS / 32], block_part;
    await_previous();
    admit_next();
    const int64_t t0 = (int64_t)blockIdx.x * SMALL_THREADS + threadIdx.x;
    constexpr int64_t step = (int64_t)SMALL_BLOCKS * SMALL_THREADS;
    unsigned long long m = 0;
    for (int64_t i = t0; i < n; i += step) m = max(m, abs_bits(C[i]));
    m = warp_max(m);
    if ((threadIdx.x & 31) == 0) warp_part[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        m = warp_max(threadIdx.x < SMALL_THREADS / 32 ? warp_part[threadIdx.x] : 0ull);
        if (threadIdx.x == 0) block_part = m;
    }
    cluster.sync();
    m = 0;
#pragma unroll
    for (int b = 0; b < SMALL_BLOCKS; ++b) m = max(m, *cluster.map_shared_rank(&block_part, b));
    const int sh = shift_of(m, top);
    if (t0 == 0) {
        sc->maxbits = m;
        sc->shC = sh;
        sc->status = 0;
        if (PAIRS) reinterpret_cast<int2 *>(out)[n] = make_int2(0, 0);
    }
    for (int64_t i = t0; i < n; i += step) store<PAIRS>(out, i, C[i], sh);
    cluster.sync();  // no block leaves while another reads its maximum
}

__global__ void k_absmax_bits(const double *__restrict__ x, int64_t n, fci_split_scalars *__restrict__ sc) {
    await_previous();
    admit_next();
    unsigned long long m = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        m = max(m, abs_bits(x[i]));
    m = warp_max(m);
    if ((threadIdx.x & 31) == 0 && m) atomicMax(&sc->maxbits, m);
}

// Lets the next kernel in only when its blocks end: the blocks of the FCI digit image that
// started beside it stayed slow to their end (they live on L1, and an SM that is busy does
// not change its split between L1 and shared memory), which a grid of one wave never makes
// up.  us per sigma at s = 3, next kernel let in at the start / at the end: 364 x 3,432
// strings 1,118 / 874, 220 x 924 208 / 148, 462 x 462 146 / 139, 210 x 210 42 / 42,
// 924 x 924 443 / 443.
template <bool PAIRS>
__global__ void k_to_fixed(const double *__restrict__ C, int64_t n, int top, fci_split_scalars *__restrict__ sc,
                           void *__restrict__ out) {
    await_previous();
    const int sh = shift_of(sc->maxbits, top);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        sc->shC = sh;
        if (PAIRS) reinterpret_cast<int2 *>(out)[n] = make_int2(0, 0);
    }
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        store<PAIRS>(out, i, C[i], sh);
}

template <bool PAIRS>
cudaError_t launch(const double *C, int64_t n, int top, fci_split_scalars *sc, void *out, cudaStream_t st) {
    if (n <= SMALL_VALUES)
        return launch_dependent(true, k_fixed_small<PAIRS>, SMALL_BLOCKS, SMALL_THREADS, 0, st, C, n, top, sc, out);
    cudaError_t e = cudaMemsetAsync(sc, 0, sizeof *sc, st);
    if (e != cudaSuccess) return e;
    const unsigned nb = (unsigned)std::min<int64_t>(ceil_div(n, 256), 152 * 8);
    k_absmax_bits<<<nb, 256, 0, st>>>(C, n, sc);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return launch_dependent(true, k_to_fixed<PAIRS>, nb, 256, 0, st, C, n, top, sc, out);
}

}  // namespace

int fixed_point_launches(int64_t n) { return n <= SMALL_VALUES ? 1 : 2; }

cudaError_t launch_fixed_point(const double *C, int64_t n, int top, fci_split_scalars *sc, int64_t *Cint,
                               cudaStream_t st) {
    return launch<false>(C, n, top, sc, Cint, st);
}

cudaError_t launch_fixed_point_pairs(const double *C, int64_t n, int top, fci_split_scalars *sc, int32_t *Cint,
                                     cudaStream_t st) {
    return launch<true>(C, n, top, sc, Cint, st);
}
