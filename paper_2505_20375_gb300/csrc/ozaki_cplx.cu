// Split-precision sigma for complex spinor strings (the relativistic case of the paper's
// Results) with the contraction E = G D on the tcgen05 tensor cores, Ozaki style.
//
// The complex contraction over the n^2 spinor pairs is written as one real GEMM on the
// real embedding (index 2x = real part, 2x + 1 = imaginary part of complex index x):
//   [E_re; E_im] = [[G_re, -G_im]; [G_im, G_re]] [D_re; D_im],
// M = K = 2 n^2 rows (1,152 at 24 spinors), N = the determinants.  Neither operand fits in
// shared memory, so both are streamed from digit images in the shared-memory layout of the
// MMA operands: the G digit slices (prepared once) and the D digit slices (split from the
// fixed-point C by k_cz_split each sigma).
//
// A determinant has 156 of the 576 pairs at 24 spinors / 12 electrons, and 64 consecutive
// strings (one tile) share most of them: the pair index is cut into blocks of 8 pairs (16
// real rows or columns) by orbital ranges, L the 8 lowest spinors and U the others,
//   (a in U, 8 b of U) and (a in U, b of L): active if some string of the tile has a;
//   (8 a of L, b in U): active if some string of the tile lacks b;  (a in L, b of L): always,
// for column pairs (a, b) = (r, s) of D[rs, K] and, with the roles of the indices exchanged,
// (a, b) = (q, p) for the rows of E[pq, K], so one mask per tile serves both.  Inactive
// blocks are neither written nor multiplied nor stored (ozaki_blk.cu): 45 of 72 blocks are
// active on average at 24 / 12.
//
// Digits are balanced base-128 (7 bits, [-64, 63], exact in f16).  A D column has at
// most 2 n_e (n - n_e + 1) nonzero entries (312 at 24 spinors / 12 electrons), so a level
// sum S_L = sum_{i+j=L} G_i D_j stays an integer below s * 312 * 2^12 < 2^24 for s <= 13:
// every FP32 accumulation in TMEM is exact.  The top s levels (L >= s - 1) are formed;
// the epilogue combines them in int64 (levels below L0 = max(s - 1, 2s - 7) rounded
// away), and the scatter sums in int64:
//   sigma_I = 2^{7 L0 - sh_G - sh_C} sum <I|E_x|K> E_int[x, K] + e_core C_I.
//
// The GEMM itself is the block-sparse bulk-copy kernel (ozaki_blk.cu) with 7-bit digits, or,
// where that has too little to skip (cz_dense), the dense one (ozaki_gemm.cu) on images of all
// pairs; sigma has the same bits.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <complex>
#include <vector>

#include "fci_internal.h"
#include "oz_gemm.cuh"
#include "tc_ptx.cuh"

namespace {

using namespace tc;

constexpr int CZ_N = OZG_N;
constexpr int CZ_MAXS = OZG_MAXS;

// The blocks of 8 pairs (a, b) of n spinors, in the order of the header comment.
struct CzBlocks {
    int n, L, U, ubk;        // spinors, low and upper ones, blocks of 8 over U
    int ul, lu, ll, n_blk;   // first block of each later class, number of blocks
};
__host__ __device__ inline CzBlocks cz_blocks(int n) {
    CzBlocks c;
    c.n = n;
    c.L = n < 8 ? n : 8;
    c.U = n - c.L;
    c.ubk = (c.U + 7) / 8;
    c.ul = c.U * c.ubk;
    c.lu = c.ul + c.U;
    c.ll = c.lu + c.U;
    c.n_blk = c.ll + c.L;
    return c;
}
// Pair e (0 .. 7) of block k; false for a padding position.
__host__ __device__ inline bool cz_pair(const CzBlocks &c, int k, int e, int &a, int &b) {
    if (k < c.ul) {
        a = c.L + k / c.ubk;
        b = c.L + 8 * (k % c.ubk) + e;
        return b < c.n;
    }
    if (k < c.lu) {
        a = c.L + (k - c.ul);
        b = e;
    } else if (k < c.ll) {
        a = e;
        b = c.L + (k - c.lu);
    } else {
        a = k - c.ll;
        b = e;
    }
    return e < c.L;
}

// ------------------------------------------------------------- helper kernels

__device__ __forceinline__ uint32_t cz_rank(uint32_t T, const uint64_t *__restrict__ binom) {
    uint32_t r = 0;
    int j = 1;
    while (T) {
        const int q = __ffs(T) - 1;
        r += (uint32_t)__ldg(binom + q * FCI_BINOM_LD + j);
        ++j;
        T &= T - 1;
    }
    return r;
}

__device__ __forceinline__ int cz_sign(uint32_t S, int a, int b) {
    const int lo = a < b ? a : b, hi = a < b ? b : a;
    const uint32_t between = (hi > lo + 1) ? (((1u << hi) - 1u) & ~((2u << lo) - 1u)) : 0u;
    return __popc(S & between) & 1;
}

// Two balanced base-128 digits (bits 7j .. 7j+6 of the biased values) as an f16x2 word:
// 0x6400 | d encodes 1024 + d exactly, and one packed subtraction of 1024 + 64 leaves
// d - 64 in [-64, 63].
__device__ __forceinline__ uint32_t digits7_f16x2(uint64_t x, uint64_t y, int j) {
    const uint32_t lo = (uint32_t)(x >> (7 * j)) & 0x7Fu, hi = (uint32_t)(y >> (7 * j)) & 0x7Fu;
    const uint32_t w = (lo | (hi << 16)) | 0x64006400u;
    const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&w),
                              __halves2half2(__ushort_as_half(0x6440), __ushort_as_half(0x6440)));
    return *reinterpret_cast<const uint32_t *>(&h);
}

// D digit image and block masks, one CTA of 256 threads per tile of 64 determinants: the
// tile's union and intersection of occupations give the mask of active blocks; then the two
// halves of the CTA take the active blocks in turn, thread (row, core) writing the 8 digits
// of its 4 pairs (one core matrix row) per plane.
template <int S>
__global__ void __launch_bounds__(256) k_cz_split(const CzBlocks bl, int64_t ndet, const uint64_t *__restrict__ str,
                                                  const uint64_t *__restrict__ binom,
                                                  const int64_t *__restrict__ Cint, uint8_t *__restrict__ Dimg,
                                                  ulonglong2 *__restrict__ masks) {
    __shared__ uint32_t s_or[2], s_and[2], s_mask[4];
    uint64_t bias = 0;
#pragma unroll
    for (int j = 0; j < S; ++j) bias |= (uint64_t)64 << (7 * j);
    const int64_t nt = blockIdx.x;
    const int row = threadIdx.x & 63, core = (threadIdx.x >> 6) & 1, half = threadIdx.x >> 7;
    const int64_t K = nt * CZ_N + row;
    const bool live = K < ndet;
    const uint32_t Sm = live ? (uint32_t)__ldg(str + K) : 0u;
    if (threadIdx.x < 64) {
        const uint32_t o = __reduce_or_sync(0xFFFFFFFFu, Sm), a = __reduce_and_sync(0xFFFFFFFFu, live ? Sm : ~0u);
        if ((threadIdx.x & 31) == 0) {
            s_or[threadIdx.x >> 5] = o;
            s_and[threadIdx.x >> 5] = a;
        }
    }
    __syncthreads();
    if (threadIdx.x < OZG_MAX_BLK) {
        const uint32_t occ = s_or[0] | s_or[1], full = s_and[0] & s_and[1];  // in some string; in every string
        const int k = threadIdx.x;
        bool on = k < bl.n_blk;
        if (k < bl.ul) {
            const int a = bl.L + k / bl.ubk, b0 = bl.L + 8 * (k % bl.ubk);
            const uint32_t range = 0xFFu << b0;
            on = ((occ >> a) & 1u) && ((~full | (1u << a)) & range) != 0;
        } else if (k < bl.lu) {
            on = (occ >> (bl.L + (k - bl.ul))) & 1u;
        } else if (k < bl.ll) {
            on = !((full >> (bl.L + (k - bl.lu))) & 1u);
        }
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, on);
        if ((threadIdx.x & 31) == 0) s_mask[threadIdx.x >> 5] = m;
    }
    __syncthreads();
    if (threadIdx.x == 0)
        masks[nt] = make_ulonglong2(s_mask[0] | ((uint64_t)s_mask[1] << 32), s_mask[2] | ((uint64_t)s_mask[3] << 32));
    int turn = 0;
    for (int w = 0; w < 4; ++w) {
        for (uint32_t m = s_mask[w]; m; m &= m - 1, turn ^= 1) {
            if (turn != half) continue;
            const int k = 32 * w + __ffs(m) - 1;
            uint64_t y[8];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                int64_t vr = 0, vi = 0;
                int a, b;
                if (cz_pair(bl, k, 4 * core + e, a, b) && ((Sm >> a) & 1u) && (b == a || !((Sm >> b) & 1u))) {
                    const uint32_t T = (Sm & ~(1u << a)) | (1u << b);
                    const int64_t t = cz_rank(T, binom);
                    const int64_t cr = __ldg(Cint + 2 * t), ci = __ldg(Cint + 2 * t + 1);
                    const bool neg = cz_sign(Sm, a, b);
                    vr = neg ? -cr : cr;
                    vi = neg ? -ci : ci;
                }
                y[2 * e] = (uint64_t)vr + bias;
                y[2 * e + 1] = (uint64_t)vi + bias;
            }
            uint8_t *base = Dimg + ((size_t)nt * bl.n_blk + k) * S * 2048 + (row >> 3) * 256 + core * 128 + (row & 7) * 16;
#pragma unroll
            for (int j = 0; j < S; ++j) {
                uint4 d;
                d.x = digits7_f16x2(y[0], y[1], j);
                d.y = digits7_f16x2(y[2], y[3], j);
                d.z = digits7_f16x2(y[4], y[5], j);
                d.w = digits7_f16x2(y[6], y[7], j);
                __stcs((uint4 *)(base + j * 2048), d);  // streaming: keep C_int in L2
            }
        }
    }
}

// Dense form, digit image: block (N-tile nt, K-chunk kc) holds S planes of 64 determinants x 32
// real-embedded K, each in canonical K-major core matrices (8 rows x 16 bytes; core
// (row / 8, k / 8) at ((row / 8) * 4 + k / 8) * 128).  One CTA of 256 threads fills one
// block: thread t covers determinant t % 64 and core t / 64 (4 complex pairs = 8 reals).
template <int S>
__global__ void __launch_bounds__(256) k_cz_split_dense(int n, int64_t ndet, int n_kc, int64_t n_blocks,
                                                  const uint64_t *__restrict__ str,
                                                  const uint64_t *__restrict__ binom,
                                                  const int64_t *__restrict__ Cint, uint8_t *__restrict__ Dimg) {
    uint64_t bias = 0;
#pragma unroll
    for (int j = 0; j < S; ++j) bias |= (uint64_t)64 << (7 * j);
    const int row = threadIdx.x & 63, cc = threadIdx.x >> 6;
    const int n2 = n * n;
    for (int64_t blk = blockIdx.x; blk < n_blocks; blk += gridDim.x) {
        const int64_t nt = blk / n_kc;
        const int kc = (int)(blk - nt * n_kc);
        const int64_t K = nt * CZ_N + row;
        uint64_t y[8];
        const uint32_t Sm = K < ndet ? (uint32_t)__ldg(str + K) : 0u;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int x = (kc * 32 + cc * 8) / 2 + e;  // complex pair index
            int64_t vr = 0, vi = 0;
            if (K < ndet && x < n2) {
                const int a = x / n, b = x - a * n;
                if (((Sm >> a) & 1u) && (b == a || !((Sm >> b) & 1u))) {
                    const uint32_t T = (Sm & ~(1u << a)) | (1u << b);
                    const int64_t t = cz_rank(T, binom);
                    const int64_t cr = __ldg(Cint + 2 * t), ci = __ldg(Cint + 2 * t + 1);
                    const bool neg = cz_sign(Sm, a, b);
                    vr = neg ? -cr : cr;
                    vi = neg ? -ci : ci;
                }
            }
            y[2 * e] = (uint64_t)vr + bias;
            y[2 * e + 1] = (uint64_t)vi + bias;
        }
        uint8_t *base = Dimg + (size_t)blk * S * 4096 + ((row >> 3) * 4 + cc) * 128 + (row & 7) * 16;
#pragma unroll
        for (int j = 0; j < S; ++j) {
            uint4 w;
            w.x = digits7_f16x2(y[0], y[1], j);
            w.y = digits7_f16x2(y[2], y[3], j);
            w.z = digits7_f16x2(y[4], y[5], j);
            w.w = digits7_f16x2(y[6], y[7], j);
            __stcs((uint4 *)(base + j * 4096), w);  // streaming: keep C_int in L2
        }
    }
}

// sigma_I = scale * sum over the replacements of I of sign * E_int[x, T] (complex parts in
// rows 2x and 2x + 1 of the tile-major E image) + e_core C_I.
__global__ void __launch_bounds__(128) k_cz_scatter(int n, int64_t ndet, int M_pad, const uint64_t *__restrict__ str,
                                                    const uint64_t *__restrict__ binom,
                                                    const int64_t *__restrict__ E, const double *__restrict__ C,
                                                    double e_core, int ushift, const int *__restrict__ shC,
                                                    const int *__restrict__ status, int *__restrict__ sticky,
                                                    double *__restrict__ sigma) {
    const int64_t I = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (I >= ndet) return;
    const int u = ushift - *shC;
    const bool bad = *status != 0;
    if (bad && I == 0) atomicExch(sticky, *status);  // kept for fci_sync_status
    const uint32_t Sm = (uint32_t)str[I];
    int64_t ar = 0, ai = 0;
    for (int a = 0; a < n; ++a) {
        if (!((Sm >> a) & 1u)) continue;
        for (int b = 0; b < n; ++b) {
            if (b != a && ((Sm >> b) & 1u)) continue;
            const uint32_t T = (Sm & ~(1u << a)) | (1u << b);
            const int64_t t = cz_rank(T, binom);
            const int x = a * n + b;
            const int64_t *e = E + ((t / CZ_N) * M_pad + 2 * x) * CZ_N + (t % CZ_N);
            const int64_t er = __ldg(e), ei = __ldg(e + CZ_N);
            if (cz_sign(Sm, a, b)) { ar -= er; ai -= ei; } else { ar += er; ai += ei; }
        }
    }
    const double cr = C[2 * I], ci = C[2 * I + 1];
    if (bad) {
        sigma[2 * I] = sigma[2 * I + 1] = __longlong_as_double(0x7FF8000000000000ll);
    } else {
        sigma[2 * I] = scalbn(__ll2double_rn(ar), u) + e_core * cr;
        sigma[2 * I + 1] = scalbn(__ll2double_rn(ai), u) + e_core * ci;
    }
}

inline size_t al256(size_t b) { return (b + 255) & ~(size_t)255; }

uint16_t half_bits_of_small_int(int d) {  // IEEE binary16 of an integer |d| <= 1024 (exact)
    if (d == 0) return 0;
    const uint16_t sign = d < 0 ? 0x8000 : 0;
    unsigned m = (unsigned)(d < 0 ? -d : d);
    int e = 31 - __builtin_clz(m);
    const unsigned mant = (m << (10 - e)) & 0x3FF;
    return (uint16_t)(sign | ((unsigned)(e + 15) << 10) | mant);
}

// The dense form: all 2 n^2 rows and columns, M-tiles of 128, K-chunks of 32.
struct CzGeom {
    int M_real, n_mt, n_kc;
};
CzGeom cz_geom(const fci_context *h) {
    const int m = 2 * h->n_orb * h->n_orb;
    return {m, (int)ceil_div(m, OZG_M), (int)ceil_div(m, 32)};
}

// Work of the block-sparse GEMM over that of the dense one: the mean over sampled tiles of
// (units x active blocks), against M-tiles x K-chunks.  The masks are those of k_cz_split.
double cz_share(const fci_context *h) {
    if (h->cz_share >= 0.0) return h->cz_share;
    const CzBlocks c = cz_blocks(h->n_orb);
    const CzGeom g = cz_geom(h);
    const int64_t tiles = ceil_div(h->ndet, CZ_N), samples = std::min<int64_t>(tiles, 24);
    auto choose = [](int n, int k) {
        double r = 1.0;
        for (int i = 1; i <= k; ++i) r = r * (n - k + i) / i;
        return k > n ? 0.0 : r;  // below 2^53: exact
    };
    double sum = 0.0;
    for (int64_t i = 0; i < samples; ++i) {
        const int64_t first = (2 * i + 1) * tiles / (2 * samples) * CZ_N, last = std::min(first + CZ_N, h->ndet);
        uint64_t S = 0;  // the string of rank `first`: strings ascend by value
        double r = (double)first;
        for (int p = h->n_orb - 1, k = h->na; k > 0; --p)
            if (choose(p, k) <= r) {
                r -= choose(p, k--);
                S |= (uint64_t)1 << p;
            }
        uint64_t occ = 0, full = ~(uint64_t)0;
        for (int64_t t = first; t < last; ++t) {
            occ |= S;
            full &= S;
            const uint64_t low = S & (~S + 1), up = S + low;  // the next string with as many bits
            if (low) S = (((up ^ S) >> 2) / low) | up;
        }
        int on = c.L;
        for (int a = c.L; a < c.n; ++a) {
            if ((occ >> a) & 1)
                for (int b = 0; b < c.ubk; ++b)
                    on += ((~full | ((uint64_t)1 << a)) & ((uint64_t)0xFF << (c.L + 8 * b))) != 0;
            on += ((occ >> a) & 1) + !((full >> a) & 1);
        }
        sum += (double)ceil_div(on, 8) * on;
    }
    return h->cz_share = sum / (double)samples / ((double)g.n_mt * g.n_kc);
}

// Which form: the block-sparse GEMM skips half of the MMAs and more, but copies its operator
// block by block and costs about 3,000 cycles a unit, so it needs many MMAs per unit (slices),
// blocks to skip (cz_share; crowded or padded strings skip few) and tiles enough to fill the
// GPU.  us, dense / blocks:
//   spinors, electrons, share   s = 4           5               6               8
//   12, 6                       109/140         115/143         119/144         124/152
//   21, 5    1.09               598/648         710/767         845/784         1,164/972
//   19, 10   1.10               1,321/1,440     1,677/1,809     2,079/1,847     3,038/2,405
//   20, 10   1.08               2,710/2,566     3,607/3,331     4,624/3,402     7,031/4,521
//   22, 11   0.93               13,059/10,780   17,897/14,249   (s = 8 36,463/19,269)
//   22, 16   1.20               1,953/2,157     2,451/2,665     3,079/2,698     4,430/3,499
//   25, 20   1.37               2,448/3,279     3,010/4,063     3,677/4,095     5,254/5,388
// Up to 3 slices always take the dense form; above, FCI_SPLIT_FORM=dense or blocks overrides
// the rule (for tests).
bool cz_dense(const fci_context *h, int s) {
    if (s <= 3) return true;
    if (!oz_gemm_ring(s, 4, 0)) return false;
    if (const char *env = getenv("FCI_SPLIT_FORM")) return strcmp(env, "dense") == 0;
    if (h->n_orb < (s <= 5 ? 20 : 18) || h->ndet < ((int64_t)1 << (s <= 5 ? 16 : 14))) return true;
    return cz_share(h) > (s <= 5 ? 1.1 : s == 6 ? 1.26 : 1.36);
}

}  // namespace

int cz_check(fci_context *h, int s) {
    if (h->mode != FCI_MODE_SPINOR) return fci_fail(h, FCI_ERR_UNSUPPORTED, "complex split path needs spinor strings");
    if (s < 2 || s > CZ_MAXS) return fci_fail(h, FCI_ERR_UNSUPPORTED, "the complex split path takes 2..%d slices", CZ_MAXS);
    if (h->n_orb > 32) return fci_fail(h, FCI_ERR_UNSUPPORTED, "more than 32 spinors");
    const int64_t nnz = 2 * (int64_t)h->na * (h->n_orb - h->na + 1);  // nonzeros of a real-embedded D column
    if ((int64_t)s * nnz * 4096 >= ((int64_t)1 << 24))
        return fci_fail(h, FCI_ERR_UNSUPPORTED, "%d slices x %lld nonzero terms could exceed 2^24 in a level sum", s,
                        (long long)nnz);
    if (!(cz_dense(h, s) ? oz_gemm_ring(s, 4, 0) : oz_blk_ring(s)))
        return fci_fail(h, FCI_ERR_UNSUPPORTED, "%d slices do not fit two pipeline stages", s);
    return FCI_OK;
}

// Real-embedded G digit image in the A layout of the block-sparse GEMM, followed by the row
// map (row of E of each position of a row block).
static int cz_prepare_G(fci_context *h, int s, cudaStream_t st) {
    const bool dense = cz_dense(h, s);
    fci_image &image = h->img[dense][s];
    if (image.d) return FCI_OK;
    const CzBlocks bl = cz_blocks(h->n_orb);
    const CzGeom g = cz_geom(h);
    const int n = h->n_orb, n2 = n * n, np = bl.n_blk * 16;
    std::vector<double> G((size_t)n2 * n2 * 2);
    if (cudaMemcpy(G.data(), h->d_G, G.size() * 8, cudaMemcpyDeviceToHost) != cudaSuccess)
        return fci_cuda_check(h, cudaGetLastError(), "G download");
    double gmax = 0.0;
    for (double v : G) gmax = std::max(gmax, fabs(v));
    int eG = 0;
    if (gmax > 0) frexp(gmax, &eG);
    const int shG = 7 * s - 2 - eG;
    uint64_t bias = 0;
    for (int j = 0; j < s; ++j) bias |= (uint64_t)64 << (7 * j);
    // real-embedded index of each position as a column (r, s) = (a, b) and as a row (p, q) = (b, a)
    std::vector<int32_t> col(np, -1), row(np, -1);
    for (int k = 0; k < bl.n_blk; ++k)
        for (int e = 0; e < 8; ++e) {
            int a, b;
            if (!cz_pair(bl, k, e, a, b)) continue;
            for (int w = 0; w < 2; ++w) {
                col[16 * k + 2 * e + w] = 2 * (a * n + b) + w;
                row[16 * k + 2 * e + w] = 2 * (b * n + a) + w;
            }
        }
    const size_t map_off = (size_t)bl.n_blk * bl.n_blk * s * 512;
    std::vector<uint16_t> img;
    if (!dense) img.assign(map_off / 2 + (size_t)np * 2, 0);
    else img.assign((size_t)g.n_mt * g.n_kc * s * 4096, 0);
    for (int pr = 0; pr < np; ++pr)
        for (int pc = 0; pc < np; ++pc) {
            if (row[pr] < 0 || col[pc] < 0) continue;
            const int x = row[pr] >> 1, u = row[pr] & 1, y = col[pc] >> 1, w = col[pc] & 1;  // complex row x, column y
            const double gr = G[2 * ((size_t)x * n2 + y)], gi = G[2 * ((size_t)x * n2 + y) + 1];
            const int64_t gi64 = llrint(ldexp(u == w ? gr : (u == 0 ? -gi : gi), shG));
            const uint64_t yb = (uint64_t)gi64 + bias;
            size_t off, plane;
            if (dense) {  // [M-tile][K-chunk][plane][128 x 32]
                const int m = row[pr], k = col[pc], r = m % OZG_M, c = k % 32;
                off = ((size_t)(m / OZG_M) * g.n_kc + k / 32) * s * 8192 + ((r >> 3) * 4 + (c >> 3)) * 128 + (r & 7) * 16 +
                      (c & 7) * 2;
                plane = 8192;
            } else {
                const int r = pr & 15, c = pc & 15;
                off = ((size_t)(pr >> 4) * bl.n_blk + (pc >> 4)) * s * 512 + (size_t)(r >> 3) * s * 256 + (c >> 3) * 128 +
                      (r & 7) * 16 + (c & 7) * 2;
                plane = 256;
            }
            for (int j = 0; j < s; ++j)
                img[(off + (size_t)j * plane) / 2] = half_bits_of_small_int((int)((yb >> (7 * j)) & 0x7F) - 64);
        }
    if (!dense) memcpy(reinterpret_cast<char *>(img.data()) + map_off, row.data(), (size_t)np * 4);
    return fci_image_build(h, image, img.data(), img.size() * 2, shG, st);
}

// 2 KB units per slice of a tile's digit image.
static size_t cz_image_blocks(const fci_context *h, int s) {
    return cz_dense(h, s) ? 2 * (size_t)cz_geom(h).n_kc : (size_t)cz_blocks(h->n_orb).n_blk;
}

// C_int, the D digit image, E_int, the block masks, 256 bytes of scalars.
size_t cz_workspace_bytes(const fci_context *h, int s) {
    const size_t n_nt = (size_t)ceil_div(h->ndet, CZ_N), n2 = (size_t)h->n_orb * h->n_orb;
    return al256((size_t)h->ndet * 16) + al256(n_nt * cz_image_blocks(h, s) * s * 2048) +
           al256(n_nt * 2 * n2 * CZ_N * 8) + al256(n_nt * sizeof(ulonglong2)) + 256;
}

int cz_sigma(fci_context *h, const double *C, double *sigma, int s, void *ws, size_t ws_bytes, cudaStream_t st) {
    (void)ws_bytes;
    int rc = cz_check(h, s);
    if (!rc) rc = cz_prepare_G(h, s, st);
    if (rc) return rc;
    const CzBlocks bl = cz_blocks(h->n_orb);
    const int64_t n_nt = ceil_div(h->ndet, CZ_N);
    const int M_real = 2 * h->n_orb * h->n_orb;
    const bool dense = cz_dense(h, s);
    const fci_image &image = h->img[dense][s];
    const CzGeom g = cz_geom(h);
    char *p = (char *)ws;
    int64_t *Cint = (int64_t *)p;
    p += al256((size_t)h->ndet * 16);
    uint8_t *Dimg = (uint8_t *)p;
    p += al256((size_t)n_nt * cz_image_blocks(h, s) * s * 2048);
    int64_t *E = (int64_t *)p;
    p += al256((size_t)n_nt * M_real * CZ_N * 8);
    ulonglong2 *masks = (ulonglong2 *)p;
    p += al256((size_t)n_nt * sizeof(ulonglong2));
    fci_split_scalars *sc = (fci_split_scalars *)p;
    int *shC = &sc->shC, *status = &sc->status;
    {
        phase_scope ps(h, st, FCI_PHASE_GATHER, fixed_point_launches(2 * h->ndet) + 1);
        FCI_CUDA(h, launch_fixed_point(C, 2 * h->ndet, 7 * s - 3, sc, Cint, st));
        const int64_t n_img = n_nt * g.n_kc;  // dense form
        const unsigned gb = (unsigned)std::min<int64_t>(n_img, 152 * 16);
        switch (dense ? s : 10 + s) {
#define CZ_DENSE(S_) case S_: k_cz_split_dense<S_><<<gb, 256, 0, st>>>(h->n_orb, h->ndet, g.n_kc, n_img, h->d_str_a, h->d_binom, Cint, Dimg); break;
#define CZ_BLOCKS(S_) case 10 + S_: k_cz_split<S_><<<(unsigned)n_nt, 256, 0, st>>>(bl, h->ndet, h->d_str_a, h->d_binom, Cint, Dimg, masks); break;
            CZ_DENSE(2) CZ_DENSE(3) CZ_DENSE(4) CZ_DENSE(5) CZ_DENSE(6) CZ_DENSE(7) CZ_DENSE(8)
            CZ_BLOCKS(4) CZ_BLOCKS(5) CZ_BLOCKS(6) CZ_BLOCKS(7) CZ_BLOCKS(8)
#undef CZ_DENSE
#undef CZ_BLOCKS
        }
        FCI_CUDA(h, cudaGetLastError());
    }
    if (dense) {
        oz_gemm_args a;
        a.n_mt = g.n_mt;
        a.n_kc = g.n_kc;
        a.M_pad = M_real;
        a.M_real = M_real;
        a.n_nt = n_nt;
        a.Gimg = image.d;
        a.Dimg = Dimg;
        a.E = E;
        a.status = status;
        if ((rc = oz_gemm_launch(h, s, 7, 4, false, a, st))) return rc;
    } else {
        oz_blk_args a;
        a.n_blk = bl.n_blk;
        a.M_pad = M_real;
        a.n_nt = n_nt;
        a.Gimg = image.d;
        a.Dimg = Dimg;
        a.masks = masks;
        a.rowmap = (const int32_t *)((const char *)image.d + (size_t)bl.n_blk * bl.n_blk * s * 512);
        a.E = E;
        a.status = status;
        if ((rc = oz_blk_launch(h, s, 7, a, st))) return rc;
    }
    {
        phase_scope ps(h, st, FCI_PHASE_SCATTER, 1);
        const int L0 = oz_gemm_L0(s, 7);
        k_cz_scatter<<<(unsigned)ceil_div(h->ndet, 128), 128, 0, st>>>(h->n_orb, h->ndet, M_real, h->d_str_a,
                                                                        h->d_binom, E, C, h->e_core,
                                                                        7 * L0 - image.sh, shC, status, h->d_status,
                                                                        sigma);
        FCI_CUDA(h, cudaGetLastError());
    }
    return FCI_OK;
}
