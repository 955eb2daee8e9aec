// Categorically compressed sigma on the STP-DAS layout (Results: categorical compression,
// the CI vector as a direct sum of per-category compressed vectors (V^B, A^B) holding only
// the nonzero coefficients and their addresses; Methods, Algorithm 1 and the compression-
// preservation argument: only nonzero coefficients contribute, and sigma comes out
// compressed as well).
//
// The paper's CPU algorithm intersects, for every intermediate determinant J, the sorted
// excitation list of J with the sorted addresses of the nonzero coefficients (exponential
// search), and accumulates sigma in per-category hash tables.  On the GPU the columns J
// are found from the other side (no scan over every J of the connected categories), D is
// gathered with that exponential search, and sigma is gathered on its support:
//   1. every nonzero C_K emits its single replacements J = E_sr K (alpha and beta moves
//      from the string tables), which are the only intermediate determinants whose
//      D[rs, J] = sum_K <J|E_rs|K> C_K can be nonzero; a hash table gives each distinct J a
//      column.  D[rs, J] is then gathered per column as Algorithm 1 does: the source K of
//      each move of J (one alpha, one beta) is looked up in the ascending nonzero addresses
//      of K's category by exponential search (galloping, then a binary search for the
//      lower bound), and the (at most two) values found are summed;
//   2. E = G D over those columns only, as the dense FP64 contraction computes it but
//      skipping the zero entries of D (the same multiply-adds in the same order);
//   3. every column J emits its single replacements L inside the target space: the
//      structural support of sigma, made distinct by a second hash table and sorted
//      (radix sort on the address), which is the compressed output order;
//   4. sigma_L = sum_pq <L|E_pq|J> E[pq, J] + e_core C_L for every L of the support, in pair
//      order (alpha then beta; absent J have E = 0): the arithmetic and its order are those
//      of the dense FP64 DAS path, so the result equals the dense sigma on the support and
//      the dense sigma is zero elsewhere.  The columns J that L reaches share its beta
//      string (an alpha move) or its alpha string (a beta move).  For a sparse vector
//      (cs_by_lists) they are found on lists of the columns per string: entries with short
//      lists (most: the alpha-beta doubles of a nonzero determinant) take one thread each,
//      those with long lists (its same-spin doubles and singles) one warp each.  Where the
//      columns crowd, and for entries with very long lists or many terms, a walk of L's
//      replacements looks each J up in the first table.
// The pair tables are read string-major (one string's row contiguous; copies built on the
// first call and kept by the handle).  Hash tables use open addressing with linear
// probing over a power-of-two capacity of at least twice the largest number of keys, so no
// probe sequence runs past a free slot; every probe loop is bounded by the capacity all
// the same and reports an overflow instead.
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <cooperative_groups.h>

#include <algorithm>
#include <vector>

#include "das_dev.cuh"

namespace {

using das_dev::das_addr;
using das_dev::das_strings;
using das_dev::DasDev;
using das_dev::make_dev;

constexpr unsigned long long HT_EMPTY = ~0ull;
constexpr int RS_THREADS = 256, RS_ITEMS = 32, RS_TILE = RS_THREADS * RS_ITEMS;  // radix sort tile (8192 keys)

inline size_t al(size_t b) { return (b + 255) & ~(size_t)255; }

// Home slot of key k in a table of mask + 1 (a power of two) slots: Fibonacci hashing, the
// top log2(capacity) bits of k times 2^64 / golden ratio (one multiply and a shift).
__device__ __forceinline__ uint64_t hslot(uint64_t k, uint64_t mask) {
    return (k * 0x9E3779B97F4A7C15ull) >> (64 - __popcll(mask));
}

// Insert key k (>= 0) once.  Returns false if every slot was probed (cannot happen at
// the capacities used; reported as an overflow).
__device__ bool ht_insert(unsigned long long *keys, uint64_t mask, uint64_t k) {
    uint64_t p = hslot(k, mask);
    for (uint64_t probe = 0; probe <= mask; ++probe) {
        const unsigned long long old = atomicCAS(keys + p, HT_EMPTY, (unsigned long long)k);
        if (old == HT_EMPTY || old == k) return true;
        p = (p + 1) & mask;
    }
    return false;
}

// Column of key k, or -1 if k is not in the table.
__device__ int64_t ht_find(const unsigned long long *__restrict__ keys, const int32_t *__restrict__ cols, uint64_t mask,
                           uint64_t k) {
    uint64_t p = hslot(k, mask);
    for (uint64_t probe = 0; probe <= mask; ++probe) {
        const unsigned long long v = keys[p];
        if (v == k) return cols[p];
        if (v == HT_EMPTY) return -1;
        p = (p + 1) & mask;
    }
    return -1;
}

struct CsArgs {
    DasDev d;
    int n_cat_int, nent_a, nent_b, npair;
    const uint64_t *rep_a, *rep_b;   // packed replacement lists [n_str][n_ent]
    const int32_t *pair_a, *pair_b;  // string-major pair tables [n_str][ldp]: (T << 1) | sign, or -1
    int ldp;                         // n_pair_pad
    const int64_t *c_addr;
    const double *c_val;
    int64_t nnz_c;
    int64_t *nz_lo;                  // [n_cat + 1]: first nonzero of each target category
    unsigned long long *hj;          // intermediate determinants J
    int32_t *hj_col;
    uint64_t hj_mask;
    int64_t *j_addr;                 // [n1]: the J of each column
    uint32_t *bm_a, *bm_b;           // bit A (B) set: some column has alpha (beta) string A (B)
    const uint64_t *str_a, *str_b;   // string masks
    // columns per string: entries off_a[S] .. off_a[S + 1] (off_b) of list hold the columns with
    // alpha (beta) string S, as (column, mask of its other string)
    uint32_t *off_a, *off_b;         // [n_str + 1] each, one after the other
    int2 *list;                      // [2 n1]: alpha, then beta
    bool by_lists;                   // the lists are built
    int64_t *work, *walk;            // support entries left to the warp form, and to the walk
    double *D, *E;                   // [n_pair][ldd]
    int64_t ldd;
    unsigned long long *hl;          // target determinants L of the support
    uint64_t hl_mask;
    int64_t *l_addr;                 // [n2]
    unsigned long long *counts;      // [0]: columns n1, [1]: support n2, [2]: overflow flag, [3]: entries in work, [4]: in walk
    double e_core;
};

// Step 1: every move of every nonzero C_K inserts its target J.
__global__ void __launch_bounds__(256) k_cs_expand(const __grid_constant__ CsArgs a) {
    const int nm = a.nent_a + a.nent_b;
    const int64_t total = a.nnz_c * nm;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / nm;
        const int m = (int)(t - i * nm);
        int32_t A, B;
        int pb;
        das_strings(a.d, a.d.n_cat, a.c_addr[i], A, B, pb);
        uint64_t e;
        int64_t J;
        if (m < a.nent_a) {
            e = a.rep_a[(int64_t)A * a.nent_a + m];
            J = das_addr(a.d, (int32_t)rep_target(e), B);
        } else {
            e = a.rep_b[(int64_t)B * a.nent_b + (m - a.nent_a)];
            J = das_addr(a.d, A, (int32_t)rep_target(e));
        }
        if (J >= 0 && !ht_insert(a.hj, a.hj_mask, (uint64_t)J)) atomicExch(a.counts + 2, 1ull);
    }
}

// Index of key in the ascending a[lo, hi), or -1: steps of 1, 2, 4, ... from lo bracket
// the key (Algorithm 1's exponentialSearch), then a binary search finds its lower bound.
__device__ int64_t exp_search(const int64_t *__restrict__ a, int64_t lo, int64_t hi, int64_t key) {
    if (lo >= hi) return -1;
    int64_t b = 1;
    while (lo + b < hi && a[lo + b] < key) b <<= 1;
    int64_t l = lo + (b >> 1), r = min(lo + b, hi - 1);
    while (l < r) {
        const int64_t m = (l + r) >> 1;
        if (a[m] < key) l = m + 1;
        else r = m;
    }
    return a[l] == key ? l : -1;
}

// nz_lo[c] = first index of a nonzero coefficient at or after the start of target category c
// (c = n_cat: the end of the target space), by binary search.
__global__ void k_cs_cat_ranges(const __grid_constant__ CsArgs a) {
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c <= a.d.n_cat; c += gridDim.x * blockDim.x) {
        const int64_t key = c < a.d.n_cat ? a.d.cat_off[c] : a.d.n_det;
        int64_t lo = 0, hi = a.nnz_c;
        while (lo < hi) {
            const int64_t m = (lo + hi) >> 1;
            if (a.c_addr[m] < key) lo = m + 1;
            else hi = m;
        }
        a.nz_lo[c] = lo;
    }
}

// The value of the target determinant K in the compressed C, or 0.
__device__ __forceinline__ bool cs_coef(const CsArgs &a, int64_t K, double &v) {
    if (K < 0 || K >= a.d.n_det) return false;
    const int c = das_dev::find_cat(a.d.cat_off, a.d.n_cat, K);
    const int64_t i = exp_search(a.c_addr, a.nz_lo[c], a.nz_lo[c + 1], K);
    if (i < 0) return false;
    v = a.c_val[i];
    return true;
}

// D[pair, column] for every column J and pair: the alpha source and the beta source of J
// under the pair, each looked up among the nonzero coefficients (Algorithm 1's
// intersection of J's excitation list with the compressed vector).  One warp per column, so
// that J is decoded once; its first lane marks J's strings in the bitmaps (a walk of the
// replacements looks a candidate column up only if both of its strings occur in some column)
// and counts the columns per string.
__global__ void __launch_bounds__(256) k_cs_gather(const __grid_constant__ CsArgs a, int64_t n1) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t j = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); j < n1; j += nw) {
        int32_t A, B;
        int pb;
        das_strings(a.d, a.n_cat_int, a.j_addr[j], A, B, pb);
        if (lane == 0) {
            atomicOr(a.bm_a + (A >> 5), 1u << (A & 31));
            atomicOr(a.bm_b + (B >> 5), 1u << (B & 31));
            if (a.by_lists) {
                atomicAdd(a.off_a + A, 1u);
                atomicAdd(a.off_b + B, 1u);
            }
        }
        for (int pp = lane; pp < a.npair; pp += 32) {
            double d = 0.0, v;
            const int32_t ea = __ldg(a.pair_a + (int64_t)A * a.ldp + pp);
            if (ea >= 0 && cs_coef(a, das_addr(a.d, ea >> 1, B), v)) d += (ea & 1) ? -v : v;
            const int32_t eb = __ldg(a.pair_b + (int64_t)B * a.ldp + pp);
            if (eb >= 0 && cs_coef(a, das_addr(a.d, A, eb >> 1), v)) d += (eb & 1) ? -v : v;
            a.D[(int64_t)pp * a.ldd + j] = d;
        }
    }
}

// Step 2: E[:, J] = G D[:, J] for every column, one warp per column: the warp walks the
// column 32 rows at a time, and for each nonzero D[rs, J] (ballot, ascending rs) every lane
// adds G[pq, rs] D[rs, J] to its rows pq = lane + 32 i with a fused multiply-add.  These
// are the multiply-adds of the dense product in the same order without its terms
// G[pq, rs] x 0 (which change no bit), so E equals the dense FP64 product; the columns hold
// only the moves into a sparse vector, so this is a small fraction of its work.
constexpr int CS_RPL = 17;  // rows per lane: n_pair <= 544 (32 orbitals)
__global__ void __launch_bounds__(256) k_cs_spmm(const double *__restrict__ G, int npair, const double *__restrict__ D,
                                                 int64_t ldd, int64_t n1, double *__restrict__ E) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t j = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); j < n1; j += nw) {
        double acc[CS_RPL];
#pragma unroll
        for (int i = 0; i < CS_RPL; ++i) acc[i] = 0.0;
        for (int r0 = 0; r0 < npair; r0 += 32) {
            const int rs = r0 + lane;
            const double d = rs < npair ? D[(int64_t)rs * ldd + j] : 0.0;
            unsigned nz = __ballot_sync(0xFFFFFFFFu, d != 0.0);
            while (nz) {
                const int b = __ffs(nz) - 1;
                nz &= nz - 1;
                const double v = __shfl_sync(0xFFFFFFFFu, d, b);
                const double *g = G + (r0 + b);
#pragma unroll
                for (int i = 0; i < CS_RPL; ++i) {
                    const int pq = lane + 32 * i;
                    if (pq < npair) acc[i] = fma(g[(int64_t)pq * npair], v, acc[i]);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < CS_RPL; ++i) {
            const int pq = lane + 32 * i;
            if (pq < npair) E[(int64_t)pq * ldd + j] = acc[i];
        }
    }
}

// dst[c][r] = src[r][c] for an R x C int32 table (32 x 32 tiles through shared memory, so
// that both the reads and the writes are coalesced).
__global__ void k_cs_transpose(const int32_t *__restrict__ src, int64_t R, int64_t C, int32_t *__restrict__ dst) {
    __shared__ int32_t t[32][33];
    const int64_t c0 = (int64_t)blockIdx.x * 32, r0 = (int64_t)blockIdx.y * 32;
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int64_t r = r0 + i, c = c0 + threadIdx.x;
        if (r < R && c < C) t[i][threadIdx.x] = src[r * C + c];
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int64_t c = c0 + i, r = r0 + threadIdx.x;
        if (r < R && c < C) dst[c * R + r] = t[threadIdx.x][i];
    }
}

// The lists of columns per string, after the gather has counted them (into off[S]) and the
// scan: written backwards from the end of each string's range, which leaves off[S] at its
// start (the order inside a list is free: the terms found on it are sorted).
__global__ void k_cs_lists(const __grid_constant__ CsArgs a, int64_t n1) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n1; j += (int64_t)gridDim.x * blockDim.x) {
        int32_t A, B;
        int pb;
        das_strings(a.d, a.n_cat_int, a.j_addr[j], A, B, pb);
        a.list[atomicSub(a.off_a + A, 1u) - 1u] = make_int2((int)j, (int)(uint32_t)a.str_b[B]);
        a.list[atomicSub(a.off_b + B, 1u) - 1u] = make_int2((int)j, (int)(uint32_t)a.str_a[A]);
    }
}

// Inclusive scan of c[0 .. m) in place (then c[S] is the end of string S's range), in two
// launches: block b adds up its 4,096 counts; then every block scans its own and adds the
// sums of the blocks before it.
constexpr int SCAN_TILE = 4096;
__device__ __forceinline__ uint32_t block_sum_256(uint32_t v, uint32_t *sh) {
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    uint32_t s = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) s += sh[w];
    __syncthreads();
    return s;
}
__global__ void __launch_bounds__(256) k_cs_scan_sums(const uint32_t *__restrict__ c, int64_t m, uint32_t *__restrict__ sums) {
    __shared__ uint32_t sh[8];
    uint32_t v = 0;
    for (int64_t i = (int64_t)blockIdx.x * SCAN_TILE + threadIdx.x; i < m && i < (int64_t)(blockIdx.x + 1) * SCAN_TILE; i += 256)
        v += c[i];
    v = block_sum_256(v, sh);
    if (threadIdx.x == 0) sums[blockIdx.x] = v;
}
__global__ void __launch_bounds__(256) k_cs_scan(uint32_t *__restrict__ c, int64_t m, const uint32_t *__restrict__ sums) {
    __shared__ uint32_t sh[8];
    uint32_t before = 0;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += 256) before += sums[b];
    uint32_t carry = block_sum_256(before, sh);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t b = (int64_t)blockIdx.x * SCAN_TILE; b < m && b < (int64_t)(blockIdx.x + 1) * SCAN_TILE; b += 256) {
        const int64_t i = b + threadIdx.x;
        const uint32_t v = i < m ? c[i] : 0u;
        uint32_t x = v;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) sh[warp] = x;
        __syncthreads();
        uint32_t ahead = 0, all = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            if (w < warp) ahead += sh[w];
            all += sh[w];
        }
        if (i < m) c[i] = carry + ahead + x;
        carry += all;
        __syncthreads();
    }
}

__device__ __forceinline__ bool bit(const uint32_t *__restrict__ bm, int32_t i) { return (__ldg(bm + (i >> 5)) >> (i & 31)) & 1u; }

// Distinct keys of a table get consecutive columns.  A block takes 2,048 slots at a time
// (8 per thread) and claims the columns of its keys with one addition to the counter (one
// per key, all to the same word, took ten times as long as reading the table).
__global__ void __launch_bounds__(256) k_cs_compact(const unsigned long long *__restrict__ keys, int32_t *__restrict__ cols,
                                                    uint64_t cap, int64_t *__restrict__ addr,
                                                    unsigned long long *__restrict__ counter) {
    __shared__ unsigned wsum[8];
    __shared__ unsigned long long base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (uint64_t p0 = blockIdx.x * (uint64_t)2048; p0 < cap; p0 += (uint64_t)gridDim.x * 2048) {
        unsigned long long k[8];  // the capacity is a power of two of at least 1,024
        unsigned n = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint64_t p = p0 + (uint64_t)i * 256 + threadIdx.x;
            k[i] = p < cap ? keys[p] : HT_EMPTY;
            n += k[i] != HT_EMPTY;
        }
        unsigned x = n;  // inclusive scan over the warp
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        unsigned before = 0, all = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            if (w < warp) before += wsum[w];
            all += wsum[w];
        }
        if (threadIdx.x == 0 && all) base = atomicAdd(counter, (unsigned long long)all);
        __syncthreads();
        unsigned long long c = base + before + x - n;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (k[i] == HT_EMPTY) continue;
            if (cols) cols[p0 + (uint64_t)i * 256 + threadIdx.x] = (int32_t)c;
            addr[c++] = (int64_t)k[i];
        }
        __syncthreads();  // wsum and base are rewritten by the next slots
    }
}

// Step 3: the target determinants one move away from a column J.
__global__ void __launch_bounds__(256) k_cs_support(const __grid_constant__ CsArgs a, int64_t n1) {
    const int nm = a.nent_a + a.nent_b;
    const int64_t total = n1 * nm;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = t / nm;
        const int m = (int)(t - j * nm);
        int32_t A, B;
        int pb;
        das_strings(a.d, a.n_cat_int, a.j_addr[j], A, B, pb);
        int64_t L;
        if (m < a.nent_a) L = das_addr(a.d, (int32_t)rep_target(a.rep_a[(int64_t)A * a.nent_a + m]), B);
        else L = das_addr(a.d, A, (int32_t)rep_target(a.rep_b[(int64_t)B * a.nent_b + (m - a.nent_a)]));
        if (L < 0 || L >= a.d.n_det) continue;
        if (!ht_insert(a.hl, a.hl_mask, (uint64_t)L)) atomicExch(a.counts + 2, 1ull);
    }
}

// Step 4: sigma on the sorted support, in the dense DAS path's order of terms.

// The key of the move between strings S and T that differ in two orbitals: pair, spin (alpha
// before beta), and the sign of <L|E|J> in the lowest bit.
__device__ __forceinline__ uint32_t cs_key(uint32_t S, uint32_t x, int spin) {
    const int hi = 31 - __clz(x), lo = __ffs(x) - 1;
    const uint32_t between = ((1u << hi) - 1u) & ~((2u << lo) - 1u);
    return ((uint32_t)(hi * (hi + 1) / 2 + lo) << 2) | (uint32_t)(spin << 1) | (__popc(S & between) & 1u);
}

// sigma_L from the sum of its terms: the coefficient C_L by binary search.  A nonzero
// determinant with electrons is a column itself (its diagonal replacements), so an L that is
// found not to be a column has C_L = 0 and no search.
__device__ __forceinline__ double cs_value(const CsArgs &a, int64_t L, double acc) {
    double cl = 0.0;
    int64_t lo = 0, hi = a.nnz_c - 1;
    while (lo <= hi) {
        const int64_t mid = (lo + hi) >> 1;
        const int64_t v = a.c_addr[mid];
        if (v == L) { cl = a.c_val[mid]; break; }
        if (v < L) lo = mid + 1; else hi = mid - 1;
    }
    return fma(a.e_core, cl, acc);  // as the dense FP64 scatter
}

// Appends o to a list, one addition to its count for the threads of a warp that come together.
__device__ __forceinline__ void cs_append(int64_t *list, unsigned long long *count, int64_t o) {
    const cooperative_groups::coalesced_group g = cooperative_groups::coalesced_threads();
    unsigned long long at = 0;
    if (g.thread_rank() == 0) at = atomicAdd(count, (unsigned long long)g.size());
    list[g.shfl(at, 0) + g.thread_rank()] = o;
}

// Thread form: entries whose two lists hold at most CS_SHORT columns, none of them L itself.
// The (at most CS_SHORT) terms go into ascending keys.  The others are left to the warp form,
// above CS_LIST columns to the walk.
constexpr int CS_SHORT = 8, CS_LIST = 400, CS_LONG = 64;
__global__ void __launch_bounds__(256) k_cs_sigma(const __grid_constant__ CsArgs a, const int64_t *__restrict__ l_sorted,
                                                  int64_t n2, double *__restrict__ out_val) {
    for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < n2; o += (int64_t)gridDim.x * blockDim.x) {
        const int64_t L = l_sorted[o];
        int32_t A, B;
        int pb;
        das_strings(a.d, a.d.n_cat, L, A, B, pb);
        const uint32_t b0 = __ldg(a.off_b + B), nb = __ldg(a.off_b + B + 1) - b0;
        const uint32_t a0 = __ldg(a.off_a + A), na = __ldg(a.off_a + A + 1) - a0;
        const bool walk = na + nb > CS_LIST;
        bool ok = na + nb <= CS_SHORT;
        uint32_t key[CS_SHORT];
        int32_t col[CS_SHORT];
#pragma unroll
        for (int i = 0; i < CS_SHORT; ++i) {
            key[i] = ~0u;
            col[i] = 0;
        }
        if (ok) {
            const uint32_t SA = (uint32_t)__ldg(a.str_a + A), SB = (uint32_t)__ldg(a.str_b + B);
            for (uint32_t c = 0; c < na + nb; ++c) {
                const bool alpha = c < nb;  // the columns with L's beta string are its alpha moves
                const int2 nd = __ldg(a.list + (alpha ? b0 + c : a0 + (c - nb)));
                const uint32_t S = alpha ? SA : SB, x = S ^ (uint32_t)nd.y;
                const int d = __popc(x);
                if (d == 0) ok = false;
                if (d != 2) continue;
                uint32_t k = cs_key(S, x, alpha ? 0 : 1);
                int32_t v = nd.x;
#pragma unroll
                for (int i = 0; i < CS_SHORT; ++i) {  // insertion; free places hold the largest key
                    if (k < key[i]) {
                        const uint32_t tk = key[i];
                        const int32_t tv = col[i];
                        key[i] = k;
                        col[i] = v;
                        k = tk;
                        v = tv;
                    }
                }
            }
        }
        if (!ok) {
            if (walk) cs_append(a.walk, a.counts + 4, o);
            else cs_append(a.work, a.counts + 3, o);
            continue;
        }
        double e[CS_SHORT], acc = 0.0;
#pragma unroll
        for (int i = 0; i < CS_SHORT; ++i)
            e[i] = key[i] != ~0u ? __ldg(a.E + (int64_t)(key[i] >> 2) * a.ldd + col[i]) : 0.0;
#pragma unroll
        for (int i = 0; i < CS_SHORT; ++i)
            if (key[i] != ~0u) acc += (key[i] & 1u) ? -e[i] : e[i];
        out_val[o] = fma(a.e_core, 0.0, acc);
    }
}

// Walk over the pairs of L's replacements, looking each J up in the first table: 32 pairs at a
// time by a warp while the entries are few, by a thread each once there are many.
constexpr int CS_WALK_WARPS = 1 << 14;  // entries up to which a warp takes one
__device__ __forceinline__ bool cs_look(const CsArgs &a, const uint32_t *__restrict__ bm, int32_t e, int32_t other, bool alpha,
                                        const double *__restrict__ Ep, double &v) {
    if (e < 0 || !bit(bm, e >> 1)) return false;
    const int64_t J = alpha ? das_addr(a.d, e >> 1, other) : das_addr(a.d, other, e >> 1);
    const int64_t c = J >= 0 ? ht_find(a.hj, a.hj_col, a.hj_mask, (uint64_t)J) : -1;
    if (c < 0) return false;
    v = (e & 1) ? -Ep[c] : Ep[c];
    return true;
}
template <bool WARP>
__device__ __forceinline__ void cs_walk(const CsArgs &a, int64_t L, double *__restrict__ out) {
    int32_t A, B;
    int pb;
    das_strings(a.d, a.d.n_cat, L, A, B, pb);
    const int32_t *ra = a.pair_a + (int64_t)A * a.ldp, *rb = a.pair_b + (int64_t)B * a.ldp;
    // an alpha move keeps B and a beta move keeps A: no column has them, no lookup
    const bool try_a = bit(a.bm_b, B), try_b = bit(a.bm_a, A);
    double acc = 0.0;
    if (WARP) {
        for (int p0 = 0; p0 < a.npair && (try_a || try_b); p0 += 32) {
            const int pp = p0 + (threadIdx.x & 31);
            const bool in = pp < a.npair;
            const double *Ep = a.E + (int64_t)pp * a.ldd;
            double va = 0.0, vb = 0.0;
            const bool fa = cs_look(a, a.bm_a, try_a && in ? __ldg(ra + pp) : -1, B, true, Ep, va);
            const bool fb = cs_look(a, a.bm_b, try_b && in ? __ldg(rb + pp) : -1, A, false, Ep, vb);
            const unsigned ma = __ballot_sync(0xFFFFFFFFu, fa), mb = __ballot_sync(0xFFFFFFFFu, fb);
            for (unsigned m = ma | mb; m; m &= m - 1) {  // the terms in pair order
                const int src = __ffs(m) - 1;
                const double ta = __shfl_sync(0xFFFFFFFFu, va, src), tb = __shfl_sync(0xFFFFFFFFu, vb, src);
                if ((ma >> src) & 1u) acc += ta;
                if ((mb >> src) & 1u) acc += tb;
            }
        }
        if ((threadIdx.x & 31) == 0) *out = cs_value(a, L, acc);
    } else {
        const int4 none = make_int4(-1, -1, -1, -1);
        for (int p4 = 0; p4 < a.npair && (try_a || try_b); p4 += 4) {  // rows past n_pair hold -1
            const int4 ia = try_a ? __ldg(reinterpret_cast<const int4 *>(ra + p4)) : none;
            const int4 ib = try_b ? __ldg(reinterpret_cast<const int4 *>(rb + p4)) : none;
            const int32_t ea[4] = {ia.x, ia.y, ia.z, ia.w}, eb[4] = {ib.x, ib.y, ib.z, ib.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const double *Ep = a.E + (int64_t)(p4 + k) * a.ldd;
                const int32_t xa = ea[k];
                if (xa >= 0 && bit(a.bm_a, xa >> 1)) {
                    const int64_t J = das_addr(a.d, xa >> 1, B);
                    const int64_t col = J >= 0 ? ht_find(a.hj, a.hj_col, a.hj_mask, (uint64_t)J) : -1;
                    if (col >= 0) {
                        const double e = Ep[col];
                        acc += (xa & 1) ? -e : e;
                    }
                }
                const int32_t xb = eb[k];
                if (xb >= 0 && bit(a.bm_b, xb >> 1)) {
                    const int64_t J = das_addr(a.d, A, xb >> 1);
                    const int64_t col = J >= 0 ? ht_find(a.hj, a.hj_col, a.hj_mask, (uint64_t)J) : -1;
                    if (col >= 0) {
                        const double e = Ep[col];
                        acc += (xb & 1) ? -e : e;
                    }
                }
            }
        }
        *out = cs_value(a, L, acc);
    }
}
// Every entry.
template <bool WARP>
__global__ void __launch_bounds__(256) k_cs_sigma_all(const __grid_constant__ CsArgs a, const int64_t *__restrict__ l_sorted,
                                                      int64_t n2, double *__restrict__ out_val) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
    for (int64_t o = WARP ? t >> 5 : t; o < n2; o += WARP ? nt >> 5 : nt) cs_walk<WARP>(a, l_sorted[o], out_val + o);
}
// The entries that the list forms have left.
__global__ void __launch_bounds__(256) k_cs_sigma_rest(const __grid_constant__ CsArgs a, const int64_t *__restrict__ l_sorted,
                                                       double *__restrict__ out_val) {
    const int64_t n = (int64_t)a.counts[4], t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
    if (n <= CS_WALK_WARPS)
        for (int64_t it = t >> 5; it < n; it += nt >> 5) cs_walk<true>(a, l_sorted[a.walk[it]], out_val + a.walk[it]);
    else
        for (int64_t it = t; it < n; it += nt) cs_walk<false>(a, l_sorted[a.walk[it]], out_val + a.walk[it]);
}

// Warp form.  The lanes check 32 columns of a list at a time; the terms (at most CS_LONG,
// the diagonal ones included if L itself is a column) are ranked by key in shared memory
// and added in that order.  Entries with more terms are left to the walk: a warp adds one
// term at a time, a walk by threads 32.
__global__ void __launch_bounds__(256) k_cs_sigma_warp(const __grid_constant__ CsArgs a, const int64_t *__restrict__ l_sorted,
                                                       double *__restrict__ out_val) {
    __shared__ uint32_t s_key[8][CS_LONG];
    __shared__ double s_val[8][CS_LONG], s_ord[8][CS_LONG];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n = (int64_t)a.counts[3], nw = (int64_t)gridDim.x * 8;
    for (int64_t it = (int64_t)blockIdx.x * 8 + warp; it < n; it += nw) {
        const int64_t o = a.work[it], L = l_sorted[o];
        int32_t A, B;
        int pb;
        das_strings(a.d, a.d.n_cat, L, A, B, pb);
        const uint32_t b0 = __ldg(a.off_b + B), nb = __ldg(a.off_b + B + 1) - b0;
        const uint32_t a0 = __ldg(a.off_a + A), na = __ldg(a.off_a + A + 1) - a0;
        double acc = 0.0;
        int terms = 0;
        bool itself = false;
        bool ok = true;
        {
            const uint32_t SA = (uint32_t)__ldg(a.str_a + A), SB = (uint32_t)__ldg(a.str_b + B);
            for (uint32_t c0 = 0; c0 < na + nb && ok; c0 += 32) {
                const uint32_t c = c0 + lane;
                const bool alpha = c < nb, live = c < na + nb;
                const int2 nd = live ? __ldg(a.list + (alpha ? b0 + c : a0 + (c - nb))) : make_int2(0, 0);
                const uint32_t S = alpha ? SA : SB, x = live ? S ^ (uint32_t)nd.y : ~0u;
                const bool hit = __popc(x) == 2;
                const unsigned hits = __ballot_sync(0xFFFFFFFFu, hit);
                if (terms + __popc(hits) > CS_LONG) {
                    ok = false;
                    break;
                }
                if (hit) {
                    const uint32_t k = cs_key(S, x, alpha ? 0 : 1);
                    const double e = __ldg(a.E + (int64_t)(k >> 2) * a.ldd + nd.x);
                    const int at = terms + __popc(hits & ((1u << lane) - 1u));
                    s_key[warp][at] = k;
                    s_val[warp][at] = (k & 1u) ? -e : e;
                }
                terms += __popc(hits);
                unsigned self = __ballot_sync(0xFFFFFFFFu, x == 0u);  // L itself: a term per electron
                itself |= self != 0;
                while (self) {
                    const int src = __ffs(self) - 1;
                    self &= self - 1;
                    const uint32_t T = __shfl_sync(0xFFFFFFFFu, S, src);
                    const int cl = __shfl_sync(0xFFFFFFFFu, nd.x, src), spin = __shfl_sync(0xFFFFFFFFu, alpha ? 0 : 1, src);
                    if (terms + __popc(T) > CS_LONG) {
                        ok = false;
                        break;
                    }
                    if ((T >> lane) & 1u) {
                        const uint32_t pp = (uint32_t)(lane * (lane + 1) / 2 + lane);
                        const int at = terms + __popc(T & ((1u << lane) - 1u));
                        s_key[warp][at] = (pp << 2) | (uint32_t)(spin << 1);
                        s_val[warp][at] = __ldg(a.E + (int64_t)pp * a.ldd + cl);
                    }
                    terms += __popc(T);
                }
            }
            __syncwarp();
            if (ok) {
                for (int i = lane; i < terms; i += 32) {  // keys differ: the rank is the place
                    const uint32_t k = s_key[warp][i];
                    int r = 0;
                    for (int q = 0; q < terms; ++q) r += s_key[warp][q] < k;
                    s_ord[warp][r] = s_val[warp][i];
                }
                __syncwarp();
                for (int i = 0; i < terms; ++i) acc += s_ord[warp][i];
                __syncwarp();
            }
        }
        if (!ok) {
            if (lane == 0) a.walk[atomicAdd(a.counts + 4, 1ull)] = o;
            continue;
        }
        if (lane == 0) out_val[o] = itself ? cs_value(a, L, acc) : fma(a.e_core, 0.0, acc);
    }
}

// ------------------------------------------------------------------ LSD radix sort
// 8-bit digits, ascending, stable; one tile = RS_TILE keys.  Histograms per tile and
// digit, an exclusive scan over (digit, tile), then a stable scatter: inside a tile the
// keys keep their order (rounds of 256 keys; within a round, warps in order and lanes in
// order, ranks from __match_any_sync).

__global__ void __launch_bounds__(RS_THREADS) k_rs_hist(const uint64_t *__restrict__ keys, int64_t n, int shift,
                                                        int64_t ntiles, unsigned long long *__restrict__ counts) {
    __shared__ unsigned int h[256];
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        h[threadIdx.x] = 0;
        __syncthreads();
        for (int r = 0; r < RS_ITEMS; ++r) {
            const int64_t idx = tile * RS_TILE + r * RS_THREADS + threadIdx.x;
            if (idx < n) atomicAdd(&h[(keys[idx] >> shift) & 255], 1u);
        }
        __syncthreads();
        counts[(int64_t)threadIdx.x * ntiles + tile] = h[threadIdx.x];
        __syncthreads();
    }
}

// Exclusive scan of each digit's counts over the tiles, one block per digit, and the digit's
// total; the scatter adds the totals of the smaller digits.
__global__ void __launch_bounds__(RS_THREADS) k_rs_scan(unsigned long long *__restrict__ counts, int64_t ntiles,
                                                        unsigned long long *__restrict__ totals) {
    __shared__ unsigned long long wsum[RS_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long *c = counts + (int64_t)blockIdx.x * ntiles;
    unsigned long long carry = 0;  // the same in every thread
    for (int64_t b = 0; b < ntiles; b += RS_THREADS) {
        const int64_t i = b + threadIdx.x;
        const unsigned long long v = i < ntiles ? c[i] : 0ull;
        unsigned long long x = v;  // inclusive scan inside the warp
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        unsigned long long before = 0, all = 0;
#pragma unroll
        for (int w = 0; w < RS_THREADS / 32; ++w) {
            if (w < warp) before += wsum[w];
            all += wsum[w];
        }
        if (i < ntiles) c[i] = carry + before + x - v;
        carry += all;
        __syncthreads();  // wsum is rewritten by the next tiles
    }
    if (threadIdx.x == 0) totals[blockIdx.x] = carry;
}

__global__ void __launch_bounds__(RS_THREADS) k_rs_scatter(const uint64_t *__restrict__ in, uint64_t *__restrict__ out,
                                                           int64_t n, int shift, int64_t ntiles,
                                                           const unsigned long long *__restrict__ base,
                                                           const unsigned long long *__restrict__ totals) {
    __shared__ unsigned int run[256];
    __shared__ unsigned int wc[RS_THREADS / 32][256];
    __shared__ unsigned long long dbase[256], dsum[RS_THREADS / 32];  // keys of smaller digits
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    {
        const unsigned long long v = totals[threadIdx.x];
        unsigned long long x = v;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) dsum[warp] = x;
        __syncthreads();
        x -= v;
        for (int w = 0; w < warp; ++w) x += dsum[w];
        dbase[threadIdx.x] = x;
        __syncthreads();
    }
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        run[threadIdx.x] = 0;
        for (int r = 0; r < RS_ITEMS; ++r) {
            for (int w = 0; w < RS_THREADS / 32; ++w) wc[w][threadIdx.x] = 0;
            __syncthreads();
            const int64_t idx = tile * RS_TILE + r * RS_THREADS + threadIdx.x;
            const bool valid = idx < n;
            const uint64_t key = valid ? in[idx] : 0;
            const unsigned dg = valid ? (unsigned)((key >> shift) & 255) : 256u + lane;  // invalid lanes match no one
            const unsigned peers = __match_any_sync(0xFFFFFFFFu, dg);
            const unsigned rank = __popc(peers & ((1u << lane) - 1u));
            if (valid && rank == 0) wc[warp][dg] = __popc(peers);
            __syncthreads();
            if (valid) {
                unsigned off = run[dg] + rank;
                for (int w = 0; w < warp; ++w) off += wc[w][dg];
                out[dbase[dg] + base[(int64_t)dg * ntiles + tile] + off] = key;
            }
            __syncthreads();
            unsigned add = 0;
            for (int w = 0; w < RS_THREADS / 32; ++w) add += wc[w][threadIdx.x];
            run[threadIdx.x] += add;
            __syncthreads();
        }
    }
}

unsigned grid_of(int64_t n) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, 256), 152 * 32)); }

uint64_t pow2_at_least(uint64_t x) {
    uint64_t c = 1024;
    while (c < x) c <<= 1;
    return c;
}

// Sizes of the compressed sigma's buffers for nnz_c nonzero coefficients: columns and
// support are bounded by the number of moves; hash tables hold twice their bound.
struct CsSizes {
    int64_t n1max, n2max;
    uint64_t capj, capl;
    int64_t ntiles;
    size_t bytes;
    size_t off_hj, off_hjc, off_jaddr, off_D, off_E, off_hl, off_laddr, off_tmp, off_cnt, off_hist, off_nzlo, off_bm, off_str,
        off_list, off_work;
    size_t bm_bytes, str_bytes;
    int64_t n_sums;  // scan blocks over the strings of both spins
};

// Whether sigma is found on the lists of columns per string, or by walking the replacements of
// every support entry.  Lists pay while they are short: for a sparse vector whose
// coefficients reach columns of their own.  The columns of neighbouring coefficients
// coincide (n1 below nnz times the moves of a determinant, the diagonal ones as one), and the
// lists of a nearly full space hold about as many as a walk has pairs; then a walk by
// threads, whose neighbours look up the same columns, is the faster one.  us per sigma,
// lists / walk:
//                                                       columns / moves   lists    walk
//   24 orbitals, 400 coefficients at random             1.00              6,596    20,652
//   24 orbitals, the first 200                          0.72              3,128    3,100
//   24 orbitals, the first 1,000                        0.66              16,786   11,486
//   16 orbitals, the first 4,000                        0.52              7,973    5,704
//   15 orbitals, 4,000 at random (lists of 0.6 n_pair)  0.99              18,378   24,140
//   12 orbitals, 1,000 at random (1.0 n_pair)           0.96              1,548    1,306
// FCI_CS_FORM=lists or walk overrides the rule (for tests).
bool cs_by_lists(const fci_context *h, int64_t nnz_c, int64_t n1) {
    if (const char *env = getenv("FCI_CS_FORM")) return strcmp(env, "lists") == 0;
    const int64_t moves = 1 + (h->nent_a - h->na) + (h->nent_b - h->nb);
    // half of the columns keep the alpha string of their coefficient, half the beta string: the
    // mean lists of a target determinant's two strings, at least
    const fci_das_layout &L = h->das;
    int64_t na = 0, nb = 0;  // strings of target determinants
    for (int p = 0; p < L.n_pat_a; ++p) na += L.exc_a[p] <= L.max_transfer ? L.pat_nstr_a[p] : 0;
    for (int p = 0; p < L.n_pat_b; ++p) nb += L.exc_b[p] <= L.max_transfer ? L.pat_nstr_b[p] : 0;
    const double lists = 0.5 * (double)n1 * (1.0 / (double)na + 1.0 / (double)nb);
    return 10 * n1 >= 7 * nnz_c * moves && lists < 0.8 * h->npair;
}

CsSizes cs_sizes(const fci_context *h, int64_t nnz_c) {
    CsSizes z;
    const int64_t nm = h->nent_a + h->nent_b;
    z.n1max = std::max<int64_t>(1, nnz_c * nm);
    z.n2max = std::max<int64_t>(1, z.n1max * nm);
    z.capj = pow2_at_least((uint64_t)(2 * z.n1max));
    z.capl = pow2_at_least((uint64_t)(2 * z.n2max));
    z.ntiles = ceil_div(z.n2max, RS_TILE);
    size_t o = 0;
    z.off_hj = o; o += al(z.capj * 8);
    z.off_hjc = o; o += al(z.capj * 4);
    z.off_jaddr = o; o += al((size_t)z.n1max * 8);
    z.off_D = o; o += al((size_t)h->npair * z.n1max * 8);
    z.off_E = o; o += al((size_t)h->npair * z.n1max * 8);
    z.off_hl = o; o += al(z.capl * 8);
    z.off_laddr = o; o += al((size_t)z.n2max * 8);
    z.off_tmp = o; o += al((size_t)z.n2max * 8);
    z.off_hist = o; o += al((size_t)256 * (z.ntiles + 1) * 8);  // counts, then the digits' totals
    z.off_nzlo = o; o += al((size_t)(h->das.n_cat + 1) * 8);
    z.bm_bytes = (size_t)((h->nsa + 31) / 32 + (h->nsb + 31) / 32) * 4;
    z.off_bm = o; o += al(z.bm_bytes);
    z.str_bytes = (size_t)(h->nsa + 1 + h->nsb + 1) * 4;
    z.n_sums = ceil_div(h->nsa + 1 + h->nsb + 1, SCAN_TILE);
    z.off_str = o; o += al(z.str_bytes + (size_t)z.n_sums * 4);
    z.off_list = o; o += al((size_t)z.n1max * 2 * sizeof(int2));
    z.off_work = z.off_hl;  // the support's hash table is done with by then (8 bytes per slot, two slots per entry)
    z.off_cnt = o; o += 256;
    z.bytes = o;
    return z;
}

}  // namespace

extern "C" {

int fci_sigma_compressed_workspace_bytes(fci_handle h, int64_t nnz_c, size_t *bytes) {
    if (!h || !bytes || nnz_c < 0) return fci_fail(h, FCI_ERR_ARG, "bad argument");
    if (!h->das_active) return fci_fail(h, FCI_ERR_STATE, "compressed sigma needs the DAS layout");
    *bytes = cs_sizes(h, nnz_c).bytes;
    return FCI_OK;
}

int fci_sigma_compressed(fci_handle h, const int64_t *c_addr, const double *c_val, int64_t nnz_c, int64_t *out_addr,
                         double *out_val, int64_t capacity, int64_t *nnz_sigma, void *ws, size_t ws_bytes,
                         fci_stream stream) {
    if (!h) return fci_fail(nullptr, FCI_ERR_ARG, "NULL handle");
    if (!h->das_active) return fci_fail(h, FCI_ERR_STATE, "compressed sigma needs the DAS layout");
    if (h->dtype != FCI_R64) return fci_fail(h, FCI_ERR_UNSUPPORTED, "compressed sigma is built for real integrals");
    if (!nnz_sigma || nnz_c < 0 || capacity < 0 || (nnz_c && (!c_addr || !c_val)) || (capacity && (!out_addr || !out_val)))
        return fci_fail(h, FCI_ERR_ARG, "bad compressed-vector arguments");
    const CsSizes z = cs_sizes(h, nnz_c);
    if (!ws || ws_bytes < z.bytes || ((uintptr_t)ws & 255))
        return fci_fail(h, FCI_ERR_ARG, "workspace %zu < %zu bytes or misaligned", ws_bytes, z.bytes);
    if (z.n1max >= ((int64_t)1 << 31)) return fci_fail(h, FCI_ERR_UNSUPPORTED, "too many nonzero coefficients");
    if (h->npair > 32 * CS_RPL) return fci_fail(h, FCI_ERR_UNSUPPORTED, "compressed sigma: %d orbital pairs", h->npair);
    FCI_CUDA(h, cudaSetDevice(h->device));
    cudaStream_t s = (cudaStream_t)stream;
    *nnz_sigma = 0;
    if (nnz_c == 0) return FCI_OK;
    // the addresses must be ascending target addresses (checked on the device copy)
    std::vector<int64_t> hc(nnz_c);
    FCI_CUDA(h, cudaMemcpyAsync(hc.data(), c_addr, nnz_c * 8, cudaMemcpyDeviceToHost, s));
    FCI_CUDA(h, cudaStreamSynchronize(s));
    for (int64_t i = 0; i < nnz_c; ++i)
        if (hc[i] < 0 || hc[i] >= h->das.n_det || (i && hc[i] <= hc[i - 1]))
            return fci_fail(h, FCI_ERR_ARG, "compressed C: addresses must be ascending target addresses");
    char *w = (char *)ws;
    CsArgs a;
    a.d = make_dev(h);
    a.n_cat_int = h->das.n_cat_int;
    a.nent_a = h->nent_a;
    a.nent_b = h->nent_b;
    a.npair = h->npair;
    a.rep_a = h->d_rep_a;
    a.rep_b = h->d_rep_b;
    if (!h->d_pair_a_t) {  // string-major copies of the pair tables: one string's row is contiguous
        const int64_t R = h->npair_pad;
        int rc = fci_dev_alloc(h, (void **)&h->d_pair_a_t, (size_t)R * h->nsa * 4);
        if (!rc) rc = fci_dev_alloc(h, (void **)&h->d_pair_b_t, (size_t)R * h->nsb * 4);
        if (rc) {
            fci_dev_free(h->d_pair_a_t);
            h->d_pair_a_t = nullptr;
            return rc;
        }
        const dim3 blk(32, 8);
        const unsigned gy = (unsigned)ceil_div(R, 32);
        k_cs_transpose<<<dim3((unsigned)ceil_div(h->nsa, 32), gy), blk, 0, s>>>(h->d_pair_a, R, h->nsa, h->d_pair_a_t);
        k_cs_transpose<<<dim3((unsigned)ceil_div(h->nsb, 32), gy), blk, 0, s>>>(h->d_pair_b, R, h->nsb, h->d_pair_b_t);
        FCI_CUDA(h, cudaGetLastError());
    }
    a.pair_a = h->d_pair_a_t;
    a.pair_b = h->d_pair_b_t;
    a.ldp = h->npair_pad;
    a.c_addr = c_addr;
    a.c_val = c_val;
    a.nnz_c = nnz_c;
    a.nz_lo = (int64_t *)(w + z.off_nzlo);
    a.bm_a = (uint32_t *)(w + z.off_bm);
    a.bm_b = a.bm_a + (h->nsa + 31) / 32;
    a.str_a = h->d_str_a;
    a.str_b = h->d_str_b;
    a.off_a = (uint32_t *)(w + z.off_str);
    a.off_b = a.off_a + h->nsa + 1;
    uint32_t *sums = a.off_b + h->nsb + 1;
    a.list = (int2 *)(w + z.off_list);
    a.work = (int64_t *)(w + z.off_work);
    a.walk = a.work + z.n2max;
    a.hj = (unsigned long long *)(w + z.off_hj);
    a.hj_col = (int32_t *)(w + z.off_hjc);
    a.hj_mask = z.capj - 1;
    a.j_addr = (int64_t *)(w + z.off_jaddr);
    a.D = (double *)(w + z.off_D);
    a.E = (double *)(w + z.off_E);
    a.ldd = z.n1max;
    a.hl = (unsigned long long *)(w + z.off_hl);
    a.hl_mask = z.capl - 1;
    a.l_addr = (int64_t *)(w + z.off_laddr);
    a.counts = (unsigned long long *)(w + z.off_cnt);
    a.e_core = h->e_core;
    unsigned long long cnt[3] = {0, 0, 0};
    // 1. the intermediate determinants one move from a nonzero coefficient, and D on them
    {
        phase_scope ps(h, s, FCI_PHASE_GATHER, 4);
        FCI_CUDA(h, cudaMemsetAsync(a.hj, 0xFF, z.capj * 8, s));
        FCI_CUDA(h, cudaMemsetAsync(a.counts, 0, 256, s));
        const int64_t moves = nnz_c * (a.nent_a + a.nent_b);
        k_cs_expand<<<grid_of(moves), 256, 0, s>>>(a);
        k_cs_cat_ranges<<<(unsigned)ceil_div(h->das.n_cat + 1, 256), 256, 0, s>>>(a);
        k_cs_compact<<<grid_of((int64_t)z.capj / 8), 256, 0, s>>>(a.hj, a.hj_col, z.capj, a.j_addr, a.counts);
        FCI_CUDA(h, cudaMemcpyAsync(cnt, a.counts, sizeof cnt, cudaMemcpyDeviceToHost, s));
        FCI_CUDA(h, cudaStreamSynchronize(s));
        if (cnt[2]) return fci_fail(h, FCI_ERR_CUDA, "compressed sigma: hash table overflow");
        a.by_lists = cs_by_lists(h, nnz_c, (int64_t)cnt[0]);
        FCI_CUDA(h, cudaMemsetAsync(a.bm_a, 0, (size_t)((char *)sums - (char *)a.bm_a), s));  // and the counts
        k_cs_gather<<<grid_of((int64_t)cnt[0] * 32), 256, 0, s>>>(a, (int64_t)cnt[0]);
        if (a.by_lists) {
            const int64_t m = h->nsa + 1 + h->nsb + 1;
            k_cs_scan_sums<<<(unsigned)z.n_sums, 256, 0, s>>>(a.off_a, m, sums);
            k_cs_scan<<<(unsigned)z.n_sums, 256, 0, s>>>(a.off_a, m, sums);
            k_cs_lists<<<grid_of((int64_t)cnt[0]), 256, 0, s>>>(a, (int64_t)cnt[0]);
            ps.launches += 3;
        }
        FCI_CUDA(h, cudaGetLastError());
    }
    const int64_t n1 = (int64_t)cnt[0];
    // 2. E = G D on the n1 columns
    {
        phase_scope ps(h, s, FCI_PHASE_CONTRACT, 1);
        k_cs_spmm<<<(unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n1, 8), 152 * 16)), 256, 0, s>>>(
            h->d_G, h->npair, a.D, z.n1max, n1, a.E);
        FCI_CUDA(h, cudaGetLastError());
    }
    // 3. the support of sigma, distinct and sorted
    {
        phase_scope ps(h, s, FCI_PHASE_OTHER, 2);
        FCI_CUDA(h, cudaMemsetAsync(a.hl, 0xFF, z.capl * 8, s));
        k_cs_support<<<grid_of(n1 * (a.nent_a + a.nent_b)), 256, 0, s>>>(a, n1);
        k_cs_compact<<<grid_of((int64_t)z.capl / 8), 256, 0, s>>>(a.hl, nullptr, z.capl, a.l_addr, a.counts + 1);
        FCI_CUDA(h, cudaMemcpyAsync(cnt, a.counts, sizeof cnt, cudaMemcpyDeviceToHost, s));
        FCI_CUDA(h, cudaStreamSynchronize(s));
        if (cnt[2]) return fci_fail(h, FCI_ERR_CUDA, "compressed sigma: hash table overflow");
    }
    const int64_t n2 = (int64_t)cnt[1];
    *nnz_sigma = n2;
    if (n2 > capacity)
        return fci_fail(h, FCI_ERR_ARG, "output capacity %lld < %lld support entries", (long long)capacity, (long long)n2);
    uint64_t *src = (uint64_t *)a.l_addr, *dst = (uint64_t *)(w + z.off_tmp);
    {
        int bits = 1;
        while (bits < 63 && ((uint64_t)1 << bits) < (uint64_t)h->das.n_det) ++bits;
        phase_scope ps(h, s, FCI_PHASE_OTHER, 3 * (int)ceil_div(bits, 8));
        const int64_t nt = ceil_div(n2, RS_TILE);
        unsigned long long *hist = (unsigned long long *)(w + z.off_hist);
        const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>(nt, 152 * 8));
        for (int shift = 0; shift < bits; shift += 8) {
            k_rs_hist<<<g, RS_THREADS, 0, s>>>(src, n2, shift, nt, hist);
            k_rs_scan<<<256, RS_THREADS, 0, s>>>(hist, nt, hist + 256 * nt);
            k_rs_scatter<<<g, RS_THREADS, 0, s>>>(src, dst, n2, shift, nt, hist, hist + 256 * nt);
            std::swap(src, dst);
        }
        FCI_CUDA(h, cudaGetLastError());
        FCI_CUDA(h, cudaMemcpyAsync(out_addr, src, n2 * 8, cudaMemcpyDeviceToDevice, s));
    }
    // 4. sigma on the support
    {
        phase_scope ps(h, s, FCI_PHASE_SCATTER, a.by_lists ? 3 : 1);
        if (a.by_lists) {
            k_cs_sigma<<<grid_of(n2), 256, 0, s>>>(a, out_addr, n2, out_val);
            k_cs_sigma_warp<<<152 * 8, 256, 0, s>>>(a, out_addr, out_val);
            k_cs_sigma_rest<<<152 * 8, 256, 0, s>>>(a, out_addr, out_val);
        } else if (n2 <= CS_WALK_WARPS) {
            k_cs_sigma_all<true><<<grid_of(32 * n2), 256, 0, s>>>(a, out_addr, n2, out_val);
        } else {
            k_cs_sigma_all<false><<<grid_of(n2), 256, 0, s>>>(a, out_addr, n2, out_val);
        }
        FCI_CUDA(h, cudaGetLastError());
    }
    FCI_CUDA(h, cudaStreamSynchronize(s));
    return FCI_OK;
}

}  // extern "C"
