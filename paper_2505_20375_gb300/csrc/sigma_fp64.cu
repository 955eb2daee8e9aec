// FP64 sigma build for alpha/beta strings (real spin-free orbitals):
//   gather + contraction  D[pq,K] = sum_J <K|E_pq|J> C_J (pair-packed pq), E = G D,
//                         G = 1/2 g' packed, over the nonzero entries (fp64_active.cuh)
//   scatter               sigma_I = e_core C_I + sum_{pq,K} <I|E_pq|K> E[pq,K]
// (Methods, Eqs. sigmaL, sigmaL1e, sigmaL2e; the one-electron term is folded into g').
//
// Layouts: C and sigma are [N_alpha][N_beta] row-major; E is pair-major [n_pair][N_det] so
// that consecutive threads (consecutive beta strings) read consecutive addresses.  The
// dense pair tables are [n_pair][N_str]: entry (T << 1) | neg for the single replacement
// of the string that lands on pair pq, or -1.  Because a string's list never holds both
// (a,b) and (b,a) for a != b, each packed pair has at most one entry per string and spin,
// and the same pair leads back from T.
#include <algorithm>

#include "fci_internal.h"
#include "fp64_active.cuh"

namespace {

// The entries of K = (ia, ib): every pair on which the alpha or the beta string has a
// replacement; D is the signed sum of the (at most two) sources.
struct FciSource {
    int64_t nsa, nsb;
    const int32_t *pairA, *pairB;
    const double *C;
    struct Ctx {
        int64_t ia, ib;
    };
    __device__ __forceinline__ Ctx ctx(int64_t K) const {
        const int64_t ia = K / nsb;
        return {ia, K - ia * nsb};
    }
    __device__ __forceinline__ bool pair(const Ctx &c, int pp, double &v) const {
        const int32_t ea = __ldg(pairA + (int64_t)pp * nsa + c.ia), eb = __ldg(pairB + (int64_t)pp * nsb + c.ib);
        if (ea >= 0) {
            const double x = __ldg(C + (int64_t)(ea >> 1) * nsb + c.ib);
            v = (ea & 1) ? -x : x;
        }
        if (eb >= 0) {
            const double x = __ldg(C + c.ia * nsb + (eb >> 1));
            v += (eb & 1) ? -x : x;
        }
        return ea >= 0 || eb >= 0;
    }
};

__global__ void __launch_bounds__(256) k_scatter_fci_r64(int64_t nsa, int64_t nsb, int npair,
                                                         const int32_t *__restrict__ pairA,
                                                         const int32_t *__restrict__ pairB,
                                                         const double *__restrict__ E,
                                                         const double *__restrict__ C, double e_core,
                                                         double *__restrict__ sigma) {
    const int64_t ndet = nsa * nsb;
    const int64_t ib = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (ib >= nsb) return;
    for (int64_t ia = blockIdx.y; ia < nsa; ia += gridDim.y) {
        const int64_t det = ia * nsb + ib;
        double acc = 0.0;
        for (int pp = 0; pp < npair; ++pp) {
            const double *Ep = E + (int64_t)pp * ndet;
            const int32_t ea = __ldg(pairA + (int64_t)pp * nsa + ia);
            if (ea >= 0) {
                const double e = __ldg(Ep + (int64_t)(ea >> 1) * nsb + ib);
                acc += (ea & 1) ? -e : e;
            }
            const int32_t eb = __ldg(pairB + (int64_t)pp * nsb + ib);
            if (eb >= 0) {
                const double e = __ldg(Ep + ia * nsb + (eb >> 1));
                acc += (eb & 1) ? -e : e;
            }
        }
        sigma[det] = acc + e_core * C[det];
    }
}

// GT[c][r] = G[r][c] of the n x n operator (w = 1 real, 2 interleaved complex).
__global__ void k_transpose_operator(int n, int w, const double *__restrict__ G, double *__restrict__ GT) {
    const int64_t total = (int64_t)n * n;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t c = i / n, r = i - c * n;
        for (int k = 0; k < w; ++k) GT[i * w + k] = G[(r * n + c) * w + k];
    }
}

// H_II = sum_{p in a} h_pp + sum_{p in b} h_pp + 1/2 sum_{p,q in a} (J_pq - K_pq)
//      + 1/2 sum_{p,q in b} (J_pq - K_pq) + sum_{p in a, q in b} J_pq
// (Slater-Condon, the diagonal element).  The first four terms split into a per-string
// energy e(S) = sum_{p in S} h_pp + 1/2 sum_{p,q in S} (J_pq - K_pq), the last is the
// cross term X(a, b) = sum_{p in a} j_b(p) with j_S(p) = sum_{q in S} J_pq; both come from
// a table with one row per string (k_diag_strings), so a determinant costs O(n_el) adds.
// The cross term is taken as 1/2 (sum_{p in a} j_b(p) + sum_{p in b} j_a(p)) and the
// string energies are added as (e(a) + e(b)): H_II is then exactly symmetric under
// exchanging the alpha and beta strings, as the operator is.
__global__ void k_diag_strings(int64_t nsa, int64_t nsb, int n, const uint64_t *__restrict__ sa,
                               const uint64_t *__restrict__ sb, const double *__restrict__ hd,
                               const double *__restrict__ J, const double *__restrict__ K,
                               double *__restrict__ tab) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < nsa + nsb; s += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t S = s < nsa ? sa[s] : sb[s - nsa];
        double *row = tab + s * (n + 1);
        double e = 0.0;
        for (int p = 0; p < n; ++p) {
            double jp = 0.0;
            for (int q = 0; q < n; ++q)
                if ((S >> q) & 1) jp += J[p * n + q];
            row[1 + p] = jp;
            if (!((S >> p) & 1)) continue;
            e += hd[p];
            for (int q = 0; q < n; ++q)
                if ((S >> q) & 1) e += 0.5 * (J[p * n + q] - K[p * n + q]);
        }
        row[0] = e;
    }
}

__global__ void k_diag_fci(int64_t nsa, int64_t nsb, int n, const uint64_t *__restrict__ sa,
                           const uint64_t *__restrict__ sb, const double *__restrict__ tab, double e_core,
                           double *__restrict__ diag) {
    const int64_t ndet = nsa * nsb;
    for (int64_t det = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; det < ndet;
         det += (int64_t)gridDim.x * blockDim.x) {
        const int64_t ia = det / nsb, ib = det - ia * nsb;
        diag[det] = diag_from_strings(sa[ia], sb[ib], tab + ia * (n + 1), tab + (nsa + ib) * (n + 1), e_core);
    }
}

inline dim3 det_grid(int64_t nsa, int64_t nsb, int threads) {
    unsigned gx = (unsigned)ceil_div(nsb, threads);
    unsigned gy = (unsigned)(nsa < 65535 ? nsa : 65535);
    return dim3(gx, gy);
}

}  // namespace

cudaError_t launch_contract_fci_r64(const fci_context *h, const double *C, double *E, cudaStream_t s) {
    const FciSource src{h->nsa, h->nsb, h->d_pair_a, h->d_pair_b, C};
    return fp64_active::launch_real(src, h->ndet, h->npair, h->d_GT, E, h->ndet, s);
}

cudaError_t launch_scatter_fci_r64(const fci_context *h, const double *E, const double *C,
                                   double *sigma, cudaStream_t s) {
    const int threads = 128;
    k_scatter_fci_r64<<<det_grid(h->nsa, h->nsb, threads), threads, 0, s>>>(
        h->nsa, h->nsb, h->npair, h->d_pair_a, h->d_pair_b, E, C, h->e_core, sigma);
    return cudaGetLastError();
}

cudaError_t launch_transpose_operator(int n, int w, const double *G, double *GT, cudaStream_t s) {
    const int64_t total = (int64_t)n * n;
    k_transpose_operator<<<(unsigned)std::min<int64_t>(ceil_div(total, 256), 152 * 8), 256, 0, s>>>(n, w, G, GT);
    return cudaGetLastError();
}

cudaError_t launch_diag_strings(const fci_context *h, cudaStream_t s) {
    const int64_t ns = h->nsa + h->nsb;
    k_diag_strings<<<(unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(ns, 128), 152 * 8)), 128, 0, s>>>(
        h->nsa, h->nsb, h->n_orb, h->d_str_a, h->d_str_b, h->d_hd, h->d_J, h->d_K, h->d_dstr);
    return cudaGetLastError();
}

cudaError_t launch_diag_fci(const fci_context *h, double *diag, cudaStream_t s) {
    cudaError_t e = launch_diag_strings(h, s);
    if (e != cudaSuccess) return e;
    const int64_t ndet = h->nsa * h->nsb;
    unsigned blocks = (unsigned)std::min<int64_t>(ceil_div(ndet, 256), 152 * 32);
    k_diag_fci<<<blocks, 256, 0, s>>>(h->nsa, h->nsb, h->n_orb, h->d_str_a, h->d_str_b, h->d_dstr, h->e_core, diag);
    return cudaGetLastError();
}
