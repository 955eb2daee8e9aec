// Complex (two-spinor) sigma build: one string of n spinors per determinant, complex
// Hermitian integrals (the relativistic case of the paper's Results; X2C two-spinors).
//   D[pq,K] = sum_J <K|E_pq|J> C_J      pq = p*n + q (no pair packing for complex g)
//   E = G D                             G = 1/2 g' ([n^2][n^2], complex FP64), over the
//                                       nonzero D and the E that the next step reads
//   sigma_I = e_core C_I + sum_{pq,K} <I|E_pq|K> E[pq,K]
// Single replacements are regenerated from the string masks (ranking by popc over the
// set bits) instead of being stored: at 24 spinors / 12 electrons the stored list
// would be 3.4 GB.
#include <algorithm>

#include "fci_internal.h"
#include "fp64_active.cuh"

namespace {

__device__ __forceinline__ uint32_t rank_serial(uint32_t T, const uint64_t *__restrict__ binom) {
    uint32_t r = 0;
    int j = 1;
    while (T) {
        const int p = __ffs(T) - 1;
        r += (uint32_t)__ldg(binom + p * FCI_BINOM_LD + j);
        ++j;
        T &= T - 1;
    }
    return r;
}

__device__ __forceinline__ int sign_between(uint32_t S, int a, int b) {
    const int lo = a < b ? a : b, hi = a < b ? b : a;
    const uint32_t between = (hi > lo + 1) ? (((1u << hi) - 1u) & ~((2u << lo) - 1u)) : 0u;
    return __popc(S & between) & 1;
}

__global__ void __launch_bounds__(256) k_scatter_spinor(int n, int64_t ns, const uint64_t *__restrict__ str,
                                                        const uint64_t *__restrict__ binom,
                                                        const double2 *__restrict__ E,
                                                        const double2 *__restrict__ C, double e_core,
                                                        double2 *__restrict__ sigma) {
    const int64_t I = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (I >= ns) return;
    const uint32_t S = (uint32_t)str[I];
    double sx = 0.0, sy = 0.0;
    for (int a = 0; a < n; ++a) {
        if (!((S >> a) & 1u)) continue;
        for (int b = 0; b < n; ++b) {
            if (b != a && ((S >> b) & 1u)) continue;
            const uint32_t T = (S & ~(1u << a)) | (1u << b);
            const double2 e = __ldg(E + (int64_t)(a * n + b) * ns + rank_serial(T, binom));
            if (sign_between(S, a, b)) { sx -= e.x; sy -= e.y; } else { sx += e.x; sy += e.y; }
        }
    }
    const double2 c = C[I];
    sigma[I] = make_double2(sx + e_core * c.x, sy + e_core * c.y);
}

// E = G D on the entries that carry anything (the scheme of fp64_active.cuh for one spinor
// string).  D[rs, K] is nonzero for r in K and s = r or s outside K, and E[pq, K] is read for
// q in K and p = q or p outside K: n_e (n - n_e + 1) entries each of the n^2 (110 of 400 at
// 20 spinors / 10 electrons, 156 of 576 at 24 / 12), so the dense product spent 93% of its
// FP64 multiply-adds on zeros and on rows that nothing reads.  A block lists the entries of T
// determinants (ascending rs, value of D and offset of the row of G^T), then deals the rows
// pq of all of them to its lanes; rows are taken p by p, so that neighbouring lanes read
// neighbouring columns q of a row of G^T.  Same terms in the same order as the dense
// product without its zero terms: the same bits.
constexpr int ZA_THREADS = 256;
constexpr int ZA_MAX_T = 32;

__global__ void __launch_bounds__(ZA_THREADS) k_contract_spinor(int n, int ne, int64_t ns, int T,
                                                                const uint64_t *__restrict__ str,
                                                                const uint64_t *__restrict__ binom,
                                                                const double2 *__restrict__ C,
                                                                const double2 *__restrict__ GT,
                                                                double2 *__restrict__ E) {
    extern __shared__ __align__(16) unsigned char za_smem[];
    const int nh = n - ne, m = ne * (nh + 1), n2 = n * n;
    double2 *val = reinterpret_cast<double2 *>(za_smem);     // [T][m]: D
    int *off = reinterpret_cast<int *>(val + T * m);         // [T][m]: rs n^2
    __shared__ unsigned char occ[ZA_MAX_T][32], emp[ZA_MAX_T][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int64_t k0 = (int64_t)blockIdx.x * T; k0 < ns; k0 += (int64_t)gridDim.x * T) {
        const int nt = (int)(ns - k0 < T ? ns - k0 : T);
        for (int t = warp; t < nt; t += ZA_THREADS / 32) {
            const uint32_t S = (uint32_t)str[k0 + t];
            if (lane < n) {
                const uint32_t below = (1u << lane) - 1u;
                if ((S >> lane) & 1u) occ[t][__popc(S & below)] = (unsigned char)lane;
                else emp[t][__popc(~S & below)] = (unsigned char)lane;
            }
            __syncwarp();
            for (int i = lane; i < m; i += 32) {
                // entry i: r = i / (nh + 1)-th electron, s the (i % (nh + 1))-th of the empty
                // spinors and r itself, ascending
                const int r = occ[t][i / (nh + 1)], x = i % (nh + 1);
                const int before = __popc(~S & ((1u << r) - 1u));  // empty spinors below r
                const int sp = x < before ? emp[t][x] : x == before ? r : emp[t][x - 1];
                const uint32_t target = (S & ~(1u << r)) | (1u << sp);
                const double2 c = __ldg(C + rank_serial(target, binom));
                val[t * m + i] = sign_between(S, r, sp) ? make_double2(-c.x, -c.y) : c;
                off[t * m + i] = (r * n + sp) * n2;
            }
        }
        __syncthreads();
        const int total = nt * m;
        for (int it = threadIdx.x; it < total; it += ZA_THREADS) {
            const int t = it / m, x = it - t * m;
            const int p = x < nh * ne ? emp[t][x / ne] : occ[t][x - nh * ne];
            const int q = x < nh * ne ? occ[t][x % ne] : p;
            const double2 *g = GT + (p * n + q);
            const double2 *v = val + t * m;
            const int *o = off + t * m;
            double2 acc = make_double2(0.0, 0.0);
#pragma unroll 4
            for (int i = 0; i < m; ++i) {
                const double2 a = __ldg(g + o[i]), b = v[i];
                acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
                acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
            }
            E[(int64_t)(p * n + q) * ns + (k0 + t)] = acc;
        }
        __syncthreads();
    }
}

__global__ void k_diag_spinor(int64_t ns, int n, const uint64_t *__restrict__ str, const double *__restrict__ hd,
                              const double *__restrict__ J, const double *__restrict__ K, double e_core,
                              double *__restrict__ diag) {
    for (int64_t I = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; I < ns; I += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t S = str[I];
        double e = e_core;
        for (int p = 0; p < n; ++p) {
            if (!((S >> p) & 1)) continue;
            e += hd[p];
            for (int q = 0; q < n; ++q)
                if ((S >> q) & 1) e += 0.5 * (J[p * n + q] - K[p * n + q]);
        }
        diag[I] = e;
    }
}

}  // namespace

cudaError_t launch_contract_spinor(const fci_context *h, const double *C, double *E, cudaStream_t s) {
    const int m = h->na * (h->n_orb - h->na + 1);
    if (m == 0) return cudaSuccess;  // no electron: the scatter reads nothing
    const int entry = (int)(sizeof(double2) + sizeof(int));
    const int T = fp64_active::batch_dets(m, h->nsa, entry);
    const int64_t blocks = std::min<int64_t>(ceil_div(h->nsa, T), 0x7FFFFFFF);
    k_contract_spinor<<<(unsigned)blocks, ZA_THREADS, (size_t)T * m * entry, s>>>(
        h->n_orb, h->na, h->nsa, T, h->d_str_a, h->d_binom, (const double2 *)C, (const double2 *)h->d_GT, (double2 *)E);
    return cudaGetLastError();
}

cudaError_t launch_scatter_spinor(const fci_context *h, const double *E, const double *C, double *sigma,
                                  cudaStream_t s) {
    k_scatter_spinor<<<(unsigned)ceil_div(h->nsa, 128), 128, 0, s>>>(h->n_orb, h->nsa, h->d_str_a, h->d_binom,
                                                                   (const double2 *)E, (const double2 *)C,
                                                                   h->e_core, (double2 *)sigma);
    return cudaGetLastError();
}

cudaError_t launch_diag_spinor(const fci_context *h, double *diag, cudaStream_t s) {
    unsigned blocks = (unsigned)std::min<int64_t>(ceil_div(h->nsa, 256), 152 * 32);
    k_diag_spinor<<<blocks, 256, 0, s>>>(h->nsa, h->n_orb, h->d_str_a, h->d_hd, h->d_J, h->d_K, h->e_core, diag);
    return cudaGetLastError();
}
