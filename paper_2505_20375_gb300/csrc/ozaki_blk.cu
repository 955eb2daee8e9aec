// Block-sparse split GEMM on the tcgen05 tensor cores: E = G D where each tile of 64
// determinants has its own list of active 16-wide blocks of the pair index.
//
// On the DAS layout and for spinor strings most pairs do nothing for a given determinant K:
// D[rs, K] is zero and E[pq, K] is never read unless the replacement connects K with the
// vector's space.  Determinants next to each other share most of that pattern (a DAS
// category allows only some space-to-space moves; consecutive spinor strings share their
// upper orbitals), so the pair index is permuted into blocks of 16 that are active or not
// for a whole tile, and only active blocks are written to the digit image, multiplied and
// stored.  Skipped terms are products with zero digits and skipped rows are not read, so
// sigma keeps its bits.  Share of the dense MMA work left: 24 spinors / 12 electrons 0.42,
// DAS 4 x 4 orbitals with 12 electrons and one transfer 0.27, 16 electrons and two
// transfers 0.63.
//
// Operands (f16 digits, K-major core matrices of 8 rows x 16 bytes):
//   A (G): [row block][K block][row group of 8][plane i < s][K core][8 x 16 B]
//   B (D): [N-tile of 64][K block][plane j < s][row group][K core][8 x 16 B]
// Row blocks of a unit are packed next to each other in shared memory, which the layout
// of A allows with one copy per (row block, K block): row groups keep one stride (s x 256
// bytes), planes lie 256 bytes apart.  A work unit is (N-tile, up to 8 active row blocks =
// M 128); M rows past the last active block hold whatever shared memory held and are not
// stored.  Units are dealt round-robin to one persistent CTA per SM, the units of a tile
// next to each other so that its D blocks hit L2.
//
// Warps: 0 copies (one lane per bulk copy), 1 and 2 issue the MMAs of their share of the
// levels, the rest run the epilogue, exactly as in the dense kernel (ozaki_gemm.cu), whose
// comments on issue rate and accumulator hand-off apply.  Every wait is bounded in time
// (FCI_ERR_TIMEOUT; copies and MMAs in flight are waited for under a bound of their own).
#include <stdlib.h>

#include <algorithm>
#include <numeric>
#include <type_traits>

#include "oz_gemm.cuh"
#include "oz_pipe.cuh"
#include "tc_ptx.cuh"

namespace {

using namespace tc;
using namespace ozp;

// K blocks per pipeline stage: two where a stage of one would hold at most 10 MMAs.
__host__ __device__ constexpr int blk_nk(int s) { return s <= 4 ? 2 : 1; }
__host__ __device__ constexpr uint32_t blk_stage(int s) { return (uint32_t)blk_nk(s) * (uint32_t)s * 6144u; }
constexpr int BLK_MAX_STAGES = 6;
constexpr size_t BLK_SMEM_MAX = 232448 - 1024;

struct BlkParams {
    int n_mt, n_blk, M_pad, ring;
    int64_t n_nt;
    const uint8_t *Gimg, *Dimg;
    const ulonglong2 *masks;
    const int32_t *rowmap;
    int64_t *E;
    int *status;
    long long timeout_cycles;
    int stall_test;
};

struct BlkShared {
    uint64_t full[BLK_MAX_STAGES], empty[BLK_MAX_STAGES];
    uint64_t acc_full[2], acc_empty[OZG_MAXS];
    uint64_t drain;
    uint32_t tmem_base;
    int abort;
};

// Position of the k-th (from 0) set bit of x; x has more than k set bits.
__device__ __forceinline__ int select64(uint64_t x, int k) {
    int p = 0;
#pragma unroll
    for (int w = 32; w; w >>= 1) {
        const int c = __popcll(x & ((1ull << w) - 1ull));
        if (k >= c) {
            k -= c;
            p += w;
            x >>= w;
        }
    }
    return p;
}
// The k-th active block of a tile, or -1 past the last.
__device__ __forceinline__ int select_block(const ulonglong2 m, int k) {
    const int lo = __popcll(m.x);
    if (k < lo) return select64(m.x, k);
    k -= lo;
    return k < __popcll(m.y) ? 64 + select64(m.y, k) : -1;
}
__device__ __forceinline__ int blocks_of(const ulonglong2 m) { return __popcll(m.x) + __popcll(m.y); }
// The lowest active block, taken out of the mask.
__device__ __forceinline__ int pop_block(ulonglong2 &m) {
    if (m.x) {
        const int b = __ffsll((long long)m.x) - 1;
        m.x &= m.x - 1;
        return b;
    }
    const int b = __ffsll((long long)m.y) - 1;
    m.y &= m.y - 1;
    return 64 + b;
}

template <int S, int W>
__global__ void __launch_bounds__(ozg_threads(S), 1) k_oz_gemm_blk(const __grid_constant__ BlkParams p) {
    constexpr int NBUF = (2 * S * OZG_N <= 512) ? 2 : 1;
    constexpr int GH = 3;
    constexpr int NG = NBUF == 1 ? (S + GH - 1) / GH : 1;
    constexpr int NK = blk_nk(S);
    constexpr uint32_t A_BLK = S * 512, B_BLK = S * 2048;      // one (row block, K block); one (tile, K block)
    constexpr uint32_t STAGE_A = NK * 8 * A_BLK, STAGE = STAGE_A + NK * B_BLK;
    static_assert(STAGE == blk_stage(S), "stage size");
    extern __shared__ __align__(1024) uint8_t blk_smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)blk_smem_raw + 1023) & ~(uintptr_t)1023);
    const int R = p.ring;
    BlkShared *sh = (BlkShared *)(smem + (size_t)R * STAGE);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int r = 0; r < R; ++r) {
            mbar_init(smem_u32(&sh->full[r]), 1);
            mbar_init(smem_u32(&sh->empty[r]), OZG_ISSUERS);
        }
        for (int b = 0; b < 2; ++b) mbar_init(smem_u32(&sh->acc_full[b]), OZG_ISSUERS);
        for (int b = 0; b < OZG_MAXS; ++b) mbar_init(smem_u32(&sh->acc_empty[b]), ozg_epi_warps(S));
        mbar_init(smem_u32(&sh->drain), OZG_ISSUERS);
        sh->abort = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&sh->tmem_base), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh->tmem_base;
    volatile int *abort = &sh->abort;
    const int64_t n_units = p.n_nt * p.n_mt;

    if (warp == 0) {
        // ---------------------------------------------------------------- bulk copies
        // Lane 9 kk + i: row block i of the stage's K block kk (i < 8), or its D block (i = 8).
        const int kk = lane / 9, part = lane - 9 * kk;
        uint32_t q = 0, st = 0, ph = 0;  // stages filled, ring slot, the slot's use parity
        bool ok = true;
        for (int64_t u = blockIdx.x; u < n_units && ok; u += gridDim.x) {
            const int64_t nt = u / p.n_mt;
            const int mt = (int)(u - nt * p.n_mt);
            ulonglong2 m = p.masks[nt];
            const int nb = blocks_of(m);
            if (mt * 8 >= nb) continue;
            const int nrow = nb - mt * 8 < 8 ? nb - mt * 8 : 8;
            const int rb = part < nrow ? select_block(m, mt * 8 + part) : 0;
            const uint8_t *ga = p.Gimg + (size_t)rb * p.n_blk * A_BLK;
            const uint8_t *gb = p.Dimg + (size_t)nt * p.n_blk * B_BLK;
            for (int k0 = 0; k0 < nb; k0 += NK, ++q) {
                int kb[NK];
                const int nk = nb - k0 < NK ? nb - k0 : NK;
#pragma unroll
                for (int i = 0; i < NK; ++i) kb[i] = i < nk ? pop_block(m) : 0;
                if (q >= (uint32_t)R &&
                    !wait_warp<true>(smem_u32(&sh->empty[st]), ph ^ 1, abort, p.status, p.timeout_cycles)) {
                    ok = false;
                    break;
                }
                const uint32_t fb = smem_u32(&sh->full[st]);
                const uint32_t base = smem_u32(smem) + st * STAGE;
                if (lane == 0) mbar_expect_tx(fb, (uint32_t)nk * ((uint32_t)nrow * A_BLK + B_BLK));
                __syncwarp();
                if (kk < nk) {
                    const int b = NK == 2 && kk == 1 ? kb[NK - 1] : kb[0];
                    if (part < nrow)
                        bulk_g2s(base + (uint32_t)(kk * 8 + part) * A_BLK, ga + (size_t)b * A_BLK, A_BLK, fb);
                    else if (part == 8)
                        bulk_g2s(base + STAGE_A + (uint32_t)kk * B_BLK, gb + (size_t)b * B_BLK, B_BLK, fb);
                }
                if (++st == (uint32_t)R) {
                    st = 0;
                    ph ^= 1;
                }
            }
        }
        // every copy issued must land before the CTA leaves, also after an abort
        if (lane == 0) {
            const uint32_t used = q < (uint32_t)R ? q : (uint32_t)R;
            for (uint32_t k = 1; k <= used; ++k) {
                const uint32_t idx = q - k;
                drain_wait(smem_u32(&sh->full[idx % (uint32_t)R]), (idx / (uint32_t)R) & 1u, p.status, p.timeout_cycles);
            }
        }
    } else if (warp <= OZG_ISSUERS) {
        // ---------------------------------------------------------------- MMA issuers
        auto issuer = [&](auto me_c) {
            constexpr int ME = decltype(me_c)::value;
            auto wait = [&](uint32_t bar, uint32_t par) -> bool {
                return wait_one<true>(bar, par, abort, p.status, p.timeout_cycles);
            };
            const uint32_t idesc = idesc_f16(OZG_M, OZG_N);
            const uint64_t a0 = smem_desc(smem_u32(smem), 128, S * 256);
            const uint64_t b0 = smem_desc(smem_u32(smem) + STAGE_A, 128, 256);
            uint32_t st = 0, ph = 0, tau = 0;
            bool issued = false, ok = !p.stall_test;
            for (int64_t u = blockIdx.x; u < n_units && ok; u += gridDim.x) {
                const int64_t nt = u / p.n_mt;
                const int mt = (int)(u - nt * p.n_mt);
                const int nb = blocks_of(p.masks[nt]);
                if (mt * 8 >= nb) continue;
                const int buf = NBUF == 2 ? (int)(tau & 1) : 0;
                if (NBUF == 2 && tau >= 2) {
                    if (!wait(smem_u32(&sh->acc_empty[buf]), ((tau >> 1) - 1) & 1)) break;
                    tc_fence_after();
                }
                const uint32_t dbase = tmem + (uint32_t)(buf * S * OZG_N);
                for (int k0 = 0; k0 < nb; k0 += NK) {
                    if (!wait(smem_u32(&sh->full[st]), ph)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t as = a0 + (uint64_t)((st * STAGE) >> 4);
                    const uint64_t bs = b0 + (uint64_t)((st * STAGE) >> 4);
                    auto issue = [&](int lo, int hi) {
#pragma unroll
                        for (int kk = 0; kk < NK; ++kk) {
                            if (kk > 0 && k0 + kk >= nb) break;
#pragma unroll
                            for (int j = S - 1; j >= 0; --j) {
                                const uint64_t b = bs + (uint64_t)((kk * B_BLK + j * 2048) >> 4);
                                const uint32_t acc_in = (k0 != 0 || kk != 0 || j != S - 1) ? 1u : 0u;
#pragma unroll
                                for (int i = S - 1 - j; i < S; ++i) {
                                    const int lv = i + j - (S - 1);
                                    if (lv >= lo && lv < hi && ozg_issuer(S, lv) == ME)
                                        mma_f16(dbase + (uint32_t)(lv * OZG_N),
                                                as + (uint64_t)((kk * 8 * A_BLK + i * 256) >> 4), b, idesc, acc_in);
                                }
                            }
                        }
                    };
                    if (NBUF == 1 && k0 == 0 && tau >= 1) {
                        bool freed = true;
#pragma unroll
                        for (int g = 0; g < NG; ++g) {
                            if (!wait(smem_u32(&sh->acc_empty[g]), (tau - 1) & 1)) {
                                freed = false;
                                break;
                            }
                            tc_fence_after();
                            issue(g * GH, g * GH + GH);
                        }
                        if (!freed) {
                            ok = false;
                            break;
                        }
                    } else {
                        issue(0, S);
                    }
                    issued = true;
                    mma_commit(smem_u32(&sh->empty[st]));
                    if (++st == (uint32_t)R) {
                        st = 0;
                        ph ^= 1;
                    }
                }
                if (!ok) break;
                mma_commit(smem_u32(&sh->acc_full[buf]));
                ++tau;
            }
            if (issued) mma_commit(smem_u32(&sh->drain));
            else mbar_arrive(smem_u32(&sh->drain));
            if (!drain_wait(smem_u32(&sh->drain), 0, p.status, p.timeout_cycles))
                drain_wait(smem_u32(&sh->drain), 0, p.status, p.timeout_cycles);
        };
        if (lane == 0) {
            if (warp == 1) issuer(std::integral_constant<int, 0>{});
            else issuer(std::integral_constant<int, 1>{});
        }
    } else {
        // ---------------------------------------------------------------- epilogue
        const int qd = warp & 3;
        constexpr int NCOL = OZG_N / (ozg_epi_warps(S) / 4);  // columns per warp: 32 or 16
        const int sub = (warp - 1 - OZG_ISSUERS) >> 2;  // which part of the 64 columns
        const int row = 32 * qd + (NBUF == 1 ? lane : lane >> 2);  // the first this thread stores
        uint32_t tau = 0;
        for (int64_t u = blockIdx.x; u < n_units; u += gridDim.x) {
            const int64_t nt = u / p.n_mt;
            const int mt = (int)(u - nt * p.n_mt);
            const ulonglong2 m = p.masks[nt];
            if (mt * 8 >= blocks_of(m)) continue;
            auto natural_row = [&](int r) {  // the row of E at row r of this unit, -1: none
                const int rb = select_block(m, mt * 8 + (r >> 4));
                return rb >= 0 ? __ldg(p.rowmap + rb * 16 + (r & 15)) : -1;
            };
            const int nat = natural_row(row);
            const int buf = NBUF == 2 ? (int)(tau & 1) : 0;
            const uint32_t par = NBUF == 2 ? (tau >> 1) & 1 : tau & 1;
            if (!wait_warp(smem_u32(&sh->acc_full[buf]), par, abort, p.status, p.timeout_cycles)) break;
            tc_fence_after();
            const uint32_t tl = tmem + ((uint32_t)(32 * qd) << 16) + (uint32_t)(buf * S * OZG_N);
            if constexpr (NBUF == 1) {
                int64_t *dst = p.E + ((size_t)nt * p.M_pad + (size_t)(nat >= 0 ? nat : 0)) * OZG_N;
                ozg_epilogue_grouped<S, W, GH>(tl, NCOL * sub, dst, nat >= 0,
                                               [&](int g) { mbar_arrive(smem_u32(&sh->acc_empty[g])); });
            } else {
                EpiRows rows;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int n = i == 0 ? nat : natural_row(row + 8 * i);
                    rows.p[i] = n >= 0 ? p.E + ((size_t)nt * p.M_pad + (size_t)n) * OZG_N : nullptr;
                }
                ozg_epilogue_whole<S, W>(tl, NCOL * sub, NCOL, rows,
                                         [&]() { mbar_arrive(smem_u32(&sh->acc_empty[buf])); });
            }
            ++tau;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, 512);
}

template <int W>
void (*blk_kernel(int s))(const BlkParams) {
    switch (s) {  // 2 and 3 slices take the dense form or the fused DAS kernel
        case 4: return k_oz_gemm_blk<4, W>;
        case 5: return k_oz_gemm_blk<5, W>;
        case 6: return k_oz_gemm_blk<6, W>;
        case 7: return k_oz_gemm_blk<7, W>;
        case 8: return k_oz_gemm_blk<8, W>;
        default: return nullptr;
    }
}

size_t blk_fixed() { return 1024 + sizeof(BlkShared) + 64; }

}  // namespace

int oz_blk_ring(int s) {
    if (s < 4 || s > OZG_MAXS) return 0;
    const size_t r = (BLK_SMEM_MAX - blk_fixed()) / blk_stage(s);
    return r < 2 ? 0 : (int)std::min<size_t>(BLK_MAX_STAGES, r);
}

int oz_blk_launch(fci_context *h, int s, int w, const oz_blk_args &a, cudaStream_t st) {
    void (*kern)(const BlkParams) = w == 7 ? blk_kernel<7>(s) : w == 8 ? blk_kernel<8>(s) : nullptr;
    const int ring = oz_blk_ring(s);
    if (!kern || !ring || a.n_blk > OZG_MAX_BLK)
        return fci_fail(h, FCI_ERR_UNSUPPORTED, "block-sparse split GEMM: %d slices of %d bits, %d blocks", s, w, a.n_blk);
    BlkParams prm;
    prm.n_blk = a.n_blk;
    prm.n_mt = (a.n_blk + 7) / 8;
    prm.M_pad = a.M_pad;
    prm.ring = ring;
    prm.n_nt = a.n_nt;
    prm.Gimg = (const uint8_t *)a.Gimg;
    prm.Dimg = (const uint8_t *)a.Dimg;
    prm.masks = a.masks;
    prm.rowmap = a.rowmap;
    prm.E = a.E;
    prm.status = a.status;
    const char *to = getenv("FCI_WAIT_TIMEOUT_MS");
    prm.timeout_cycles = (long long)((to ? atof(to) : 2000.0) * 2.1e6);
    const char *stall = getenv("FCI_TEST_STALL_PRODUCER");
    prm.stall_test = stall ? atoi(stall) : 0;
    int nsm = 0;
    FCI_CUDA(h, cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, h->device));
    // Units are dealt round-robin and the last ones of a tile are often empty: a grid with no
    // common factor with the units per tile spreads them over every CTA (151 of 152 CTAs
    // when a tile has 2, 4 or 8 units).
    const int64_t units = a.n_nt * prm.n_mt;
    int64_t grid = std::max<int64_t>(1, std::min<int64_t>(nsm, units));
    while (grid > 1 && units > grid && std::gcd(grid, (int64_t)prm.n_mt) != 1) --grid;
    const size_t smem = blk_fixed() + (size_t)ring * blk_stage(s);
    FCI_CUDA(h, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    phase_scope ps(h, st, FCI_PHASE_CONTRACT, 1);
    kern<<<(unsigned)grid, ozg_threads(s), smem, st>>>(prm);
    FCI_CUDA(h, cudaGetLastError());
    return FCI_OK;
}
