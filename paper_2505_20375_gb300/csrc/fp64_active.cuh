// FP64 contraction E = G D restricted to the entries that carry anything, with the gather of
// D inside (alpha/beta strings, DAS layout and spinor strings share this kernel body).
//
// An intermediate determinant K has a nonzero D[rs, K] only for the replacements rs that
// reach K from the vector's space, and E[pq, K] is read back only for the replacements pq
// that lead from K into it.  FCI(14e,14o): about 83 of 105 pairs; 16 orbitals with 8
// electrons on the DAS layout: 0 .. 90 of 136; 20 spinors with 10 electrons: 110 of 400.
// The FP64 pipe (about 2 multiply-adds per clock per SM on GB300, 1.25 TF/s) bounds this
// contraction so hard that a gather per multiply-add costs nothing beside it: the dense
// product spent its time on zeros.  The terms left are those of the dense product in its
// order (ascending rs, one fused multiply-add each), and a term G x 0 changes no bit of a
// sum, so E is the dense product's, bit for bit.
//
// A block takes T consecutive determinants at a time:
//   1. one warp per determinant lists its entries in shared memory, in ascending order, each
//      with its value of D and the offset of its row of G^T;
//   2. the (determinant, row pq) results of the batch are dealt to the lanes as one flat
//      list (full warps whatever the lists' lengths; a warp then spans at most a few
//      determinants).  A lane runs its determinant's list: one 16-byte shared load (the
//      same address across the lanes of a determinant), one load of G^T (neighbouring
//      lanes, neighbouring rows pq; 95% of the loads hit L1 at 11 orbitals, 61% at 16, the rest
//      L2) and one DFMA;
//   3. E goes out pair-major as before; rows that nothing reads are not written.
// One block per batch: five to eight resident blocks per SM overlap one block's lists with the
// others' multiply-adds, and the block scheduler levels the batches' uneven work (a
// persistent grid of 6 x 152 blocks ran its last 152 alone: 13% of FCI(12e,12o)'s time).
//
// Whole FP64 sigma, dense product before -> this: FCI(12e,12o) 14.9 -> 6.5 ms, 16 orbitals
// with 8 electrons (DAS, 655,360 target / 2.2 M intermediate determinants) 98.5 -> 7.5 ms,
// 20 spinors / 10 electrons 197 -> 15.6 ms.  The FP64 pipe is busy 95% of the contraction's cycles
// for FCI(11 orbitals, 5 + 5), 74% for the DAS layout and 99% for the spinors.
#pragma once

#include <algorithm>

#include "fci_internal.h"

namespace fp64_active {

constexpr int THREADS = 256;
constexpr int MAX_T = 32;

// First position of item `it` in the batch's flat list: the determinant t with
// off[t] <= it < off[t + 1].
__device__ __forceinline__ int find_det(const int *off, int T, int it) {
    int lo = 0, hi = T - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= it) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// off[t] = sum of cnt[0 .. t), t <= T <= 32; every thread of the first warp takes part.
__device__ __forceinline__ void scan_counts(const int *cnt, int T, int *off) {
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        int v = lane < T ? cnt[lane] : 0, s = v;
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xFFFFFFFFu, s, o);
            if (lane >= o) s += u;
        }
        if (lane == 0) off[0] = 0;
        off[lane + 1] = s;
    }
}

struct __align__(16) Entry {
    double v;   // D[rs, K]
    int off;    // rs * n_pair: the row of G^T
    int pair;   // rs
};

// Real, pair-packed.  Source: ctx(K) the determinant's strings, pair(ctx, pp, v) whether the
// pair connects K with the vector's space, and D[pp, K].
template <class Source>
__global__ void __launch_bounds__(THREADS) k_contract_real(const __grid_constant__ Source src, int64_t n, int npair, int T,
                                                           const double *__restrict__ GT, double *__restrict__ E,
                                                           int64_t ldE) {
    extern __shared__ __align__(16) unsigned char fa_smem[];
    Entry *list = reinterpret_cast<Entry *>(fa_smem);  // [T][npair]
    __shared__ int cnt[MAX_T], off[MAX_T + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int64_t k0 = (int64_t)blockIdx.x * T; k0 < n; k0 += (int64_t)gridDim.x * T) {
        const int nt = (int)(n - k0 < T ? n - k0 : T);
        for (int t = warp; t < nt; t += THREADS / 32) {
            const typename Source::Ctx c = src.ctx(k0 + t);
            Entry *row = list + t * npair;
            int m = 0;
            for (int p0 = 0; p0 < npair; p0 += 32) {
                const int pp = p0 + lane;
                double v = 0.0;
                const bool on = pp < npair && src.pair(c, pp, v);
                const unsigned mask = __ballot_sync(0xFFFFFFFFu, on);
                if (on) {
                    Entry e;
                    e.v = v;
                    e.off = pp * npair;
                    e.pair = pp;
                    row[m + __popc(mask & ((1u << lane) - 1u))] = e;
                }
                m += __popc(mask);
            }
            if (lane == 0) cnt[t] = m;
        }
        __syncthreads();
        scan_counts(cnt, nt, off);
        __syncthreads();
        const int total = off[nt];
        for (int it = threadIdx.x; it < total; it += THREADS) {
            const int t = find_det(off, nt, it);
            const Entry *row = list + t * npair;
            const int pq = row[it - off[t]].pair, m = cnt[t];
            const double *g = GT + pq;
            double acc = 0.0;
#pragma unroll 4
            for (int i = 0; i < m; ++i) {
                const Entry e = row[i];
                acc = fma(__ldg(g + e.off), e.v, acc);
            }
            E[(int64_t)pq * ldE + (k0 + t)] = acc;
        }
        __syncthreads();
    }
}

// Determinants per batch: about 1,000 results (four per thread) in a list of at most 17 KB,
// so that L1 keeps G^T beside the resident blocks' lists, and enough batches for every SM.
inline int batch_dets(int per_det, int64_t n, int entry_bytes) {
    const int64_t by_smem = 17408 / ((int64_t)per_det * entry_bytes);
    const int64_t by_grid = n / (152 * 4);
    return (int)std::max<int64_t>(1, std::min<int64_t>({(int64_t)MAX_T, by_smem, by_grid}));
}

template <class Source>
cudaError_t launch_real(const Source &src, int64_t n, int npair, const double *GT, double *E, int64_t ldE,
                        cudaStream_t s) {
    if (n <= 0 || npair <= 0) return cudaSuccess;
    const int T = batch_dets(npair, n, (int)sizeof(Entry));
    const size_t smem = (size_t)T * npair * sizeof(Entry);  // at most 17 KB (8.6 KB for one determinant of 32 orbitals)
    const int64_t blocks = std::min<int64_t>(ceil_div(n, T), 0x7FFFFFFF);
    k_contract_real<Source><<<(unsigned)blocks, THREADS, smem, s>>>(src, n, npair, T, GT, E, ldE);
    return cudaGetLastError();
}

}  // namespace fp64_active
