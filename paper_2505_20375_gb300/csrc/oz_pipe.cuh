// Device parts shared by the two split GEMM kernels (ozaki_gemm.cu: dense; ozaki_blk.cu:
// block-sparse): warp roles, bulk copies, bounded mbarrier waits and the epilogue that turns
// the level sums of a tile into E_int.
#pragma once

#include "oz_gemm.cuh"
#include "tc_ptx.cuh"

namespace ozp {

using namespace tc;

// Epilogue warps: 8 (two per TMEM lane quadrant, 32 columns each) when the level
// accumulators are double-buffered, 16 (four per quadrant, 16 columns each) otherwise.
__host__ __device__ constexpr int ozg_epi_warps(int s) { return 2 * s * OZG_N <= 512 ? 8 : 16; }
constexpr int OZG_ISSUERS = 2;
__host__ __device__ constexpr int ozg_threads(int s) { return 32 * (1 + OZG_ISSUERS + ozg_epi_warps(s)); }
// The MMA issuer of level l of s (level l takes s - l products): levels in order of their
// product counts, each to the issuer with the fewest products so far.
__host__ __device__ constexpr int ozg_issuer(int s, int l) {
    int load[OZG_ISSUERS] = {};
    int who = 0;
    for (int k = 0; k <= l; ++k) {
        int m = 0;
        for (int e = 1; e < OZG_ISSUERS; ++e)
            if (load[e] < load[m]) m = e;
        load[m] += s - k;
        who = m;
    }
    return who;
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(bar),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// Bounded wait of one thread: false on timeout or when another role has aborted.
template <bool FAST = false>
__device__ __forceinline__ bool wait_one(uint32_t bar, uint32_t parity, volatile int *abort, int *status,
                                         long long timeout) {
    if (FAST && mbar_test_wait(bar, parity)) return true;
    const long long t0 = clock64();
    int spins = 0;
    while (!mbar_try_wait_sleep(bar, parity)) {
        if (((++spins) & 3) == 0) {
            if (*abort) return false;
            if (clock64() - t0 > timeout) {
                *abort = 1;
                atomicExch(status, FCI_ERR_TIMEOUT);
                return false;
            }
        }
    }
    return true;
}

// Wait for a phase that must complete (copies or MMAs already issued) before the CTA may
// leave: bounded like every other wait, but blind to the abort flag.
__device__ __forceinline__ bool drain_wait(uint32_t bar, uint32_t parity, int *status, long long timeout) {
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > timeout) {
            atomicExch(status, FCI_ERR_TIMEOUT);
            return false;
        }
    }
    return true;
}

// Warp-uniform form of wait_one: lane 0 waits, every lane gets the answer.
template <bool FAST = false>
__device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity, volatile int *abort, int *status,
                                          long long timeout) {
    int ok = 0;
    if ((threadIdx.x & 31) == 0) ok = wait_one<FAST>(bar, parity, abort, status, timeout) ? 1 : 0;
    return __shfl_sync(0xFFFFFFFFu, ok, 0) != 0;
}

// One warp's part of the epilogue: its 32 TMEM lanes (tl: the first level's accumulator at
// the warp's lane quadrant), the level sums combined in int64 and stored.
//
// Double-buffered accumulators (s <= 4) are read as 16x256b fragments: four neighbouring
// threads hold 8 consecutive columns of a row, so a store instruction writes 8 runs of 64
// bytes instead of 32 pieces of 16 bytes (one row per thread), each a pass of its own through
// L1.  Their units are short and their 8 epilogue warps bound them: a group of ten FCI
// problems of 6 to 12 orbitals at s = 3 went from 867 to 798 us.  With one buffer (s >= 5) the
// row form stays: fragments hold the accumulators longer (whole sigma, 14 orbitals, s = 6:
// 11.56 ms by rows, 11.80 by fragments; DAS, 16 orbitals, 12 electrons: 18.9 and 20.9).

// The rows of E that a thread writes: rows T / 4 + 8 i of the quadrant, i = 0 .. 3; nullptr:
// not stored.
struct EpiRows {
    int64_t *p[4];
};
// acc[8 h + 4 o + 2 k + e]: row T / 4 + 8 (2 h + k), column 8 o + 2 (T % 4) + e.
__device__ __forceinline__ void epi_store(const EpiRows &rows, int c0, const int64_t (&acc)[16]) {
    const int c = c0 + 2 * (threadIdx.x & 3);
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (rows.p[2 * h + k])
#pragma unroll
                for (int o = 0; o < 2; ++o)
                    __stcs((longlong2 *)(rows.p[2 * h + k] + c + 8 * o),
                           make_longlong2(acc[8 * h + 4 * o + 2 * k], acc[8 * h + 4 * o + 2 * k + 1]));
}

// Single-buffered accumulators (s >= 5): 16 columns from c0 to this lane's row of 64
// determinants at dst, if keep, read GH levels at a time; each group is handed back
// (release(g), one lane) as soon as it is in registers, so the next unit's first K step
// starts on it while the rest is read and combined.
template <int S, int W, int GH, class Release>
__device__ __forceinline__ void ozg_epilogue_grouped(uint32_t tl, int c0, int64_t *dst, bool keep, Release release) {
    constexpr int L0 = oz_gemm_L0(S, W), NG = (S + GH - 1) / GH, lowshift = W * (L0 - (S - 1));
    auto term = [](uint32_t x, int L) -> int64_t {
        const int64_t v = (int64_t)__float2int_rn(__uint_as_float(x));
        return L < L0 ? v * ((int64_t)1 << (W * (L - (S - 1)))) : v * ((int64_t)1 << (W * (L - L0)));
    };
    const uint32_t tl0 = tl + (uint32_t)c0;
    int64_t acc[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) acc[c] = 0;
#pragma unroll
    for (int g = 0; g < NG; ++g) {
        uint32_t v[GH][16];
#pragma unroll
        for (int l = g * GH; l < g * GH + GH && l < S; ++l) tmem_ld16(tl0 + (uint32_t)(l * OZG_N), v[l - g * GH]);
        tmem_ld_wait();
#pragma unroll
        for (int l = g * GH; l < g * GH + GH && l < S; ++l) tmem_regs_ready(v[l - g * GH]);
        tc_fence_before();
        __syncwarp();
        if ((threadIdx.x & 31) == 0) release(g);
#pragma unroll
        for (int l = g * GH; l < g * GH + GH && l < S; ++l) {
            const int L = S - 1 + l;
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                if (L == L0 && lowshift > 0) acc[c] = (acc[c] + ((int64_t)1 << (lowshift > 0 ? lowshift - 1 : 0))) >> lowshift;
                acc[c] += term(v[l - g * GH][c], L);
            }
        }
    }
    if (keep)
#pragma unroll
        for (int c = 0; c < 16; c += 2) __stcs((longlong2 *)(dst + c0 + c), make_longlong2(acc[c], acc[c + 1]));
}

// Double-buffered accumulators (s <= 4): ncol columns from c0 to the thread's four rows,
// combined level by level, the buffer released (release(), one lane) at the end.
template <int S, int W, class Release>
__device__ __forceinline__ void ozg_epilogue_whole(uint32_t tl, int c0, int ncol, const EpiRows &rows,
                                                   Release release) {
    constexpr int L0 = oz_gemm_L0(S, W), lowshift = W * (L0 - (S - 1));
#pragma unroll 1
    for (int cb = c0; cb < c0 + ncol; cb += 16) {
        int64_t acc[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) acc[c] = 0;
#pragma unroll
        for (int L = S - 1; L <= 2 * S - 2; ++L) {
            uint32_t v[16];
            tmem_ld_frag(tl + (uint32_t)((L - (S - 1)) * OZG_N + cb), v);
            tmem_ld_wait();
            tmem_regs_ready(v);
            if (L < L0) {
#pragma unroll
                for (int c = 0; c < 16; ++c)
                    acc[c] += (int64_t)__float2int_rn(__uint_as_float(v[c])) * ((int64_t)1 << (W * (L - (S - 1))));
            } else {
                if (L == L0 && lowshift > 0) {
#pragma unroll
                    for (int c = 0; c < 16; ++c) acc[c] = (acc[c] + ((int64_t)1 << (lowshift > 0 ? lowshift - 1 : 0))) >> lowshift;
                }
#pragma unroll
                for (int c = 0; c < 16; ++c)
                    acc[c] += (int64_t)__float2int_rn(__uint_as_float(v[c])) * ((int64_t)1 << (W * (L - L0)));
            }
        }
        epi_store(rows, cb, acc);
    }
    tc_fence_before();
    __syncwarp();
    if ((threadIdx.x & 31) == 0) release();
}

}  // namespace ozp
