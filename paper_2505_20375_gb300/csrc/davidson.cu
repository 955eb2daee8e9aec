// Davidson eigensolver on the device (Results: the Ritz residual r = H C - E C is
// preconditioned and appended as the next expansion vector; Eq. sparsePreconditioner).
//
// Every vector operation runs here in FP64 (complex vectors as interleaved pairs):
// subspace projections V^H w, Ritz combinations, the residual, the preconditioner with
// its 1e-12 guard and eps * ||s|| threshold, two rounds of classical Gram-Schmidt and
// the projected eigenproblem (a cluster of eight thread blocks; complex Hermitian matrices
// through their real symmetric embedding [[A, -B], [B, A]]).  The host reads back a handful of scalars per
// iteration to decide convergence.  On small spaces the vector work is a chain of short
// launches, so every reduction ends inside its own kernel: the last block to finish adds
// the block partials in a fixed order and applies what follows (a sign, the new column of
// the projected matrix, a norm).
#include <math.h>
#include <string.h>

#include <cooperative_groups.h>

#include <algorithm>
#include <chrono>
#include <new>
#include <vector>

#include "fci_internal.h"
#include "fp64_fast.cuh"

namespace {

constexpr int RED_BLOCKS = 608;  // 4 x 152 SMs
constexpr int RED_THREADS = 256;
constexpr int KMAX = 32;
constexpr int JAC_THREADS = 256;  // the projected eigensolver's blocks, and how many share it
constexpr int JAC_CLUSTER = 8;

struct dav_scalars {      // device-resident scalars, read back each iteration
    double lam;           // lowest Ritz value (sigma carries e_core C, so e_core is included)
    double rnorm2, snorm2, maxdc;
};

// Butterfly over the lanes (exchange distances 16, 8, 4, 2, 1) that adds K per-lane values at
// once: each of the first log2 K steps halves the values a lane carries, so K values cost
// about K + 5 additions in place of 5 K (on small spaces the FP64 additions of the
// reductions took longer than the multiply-adds of the dot products).  The sums are those
// of K plain butterflies, bit for bit.  Lane l ends with value many_index<K>(l) in v[0];
// lanes with many_writer<K>(l) cover every value once.  K: a power of two up to 32.
template <int K>
__device__ __forceinline__ void warp_sum_many(double (&v)[K]) {
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int n = K; n > 1; n >>= 1, o >>= 1) {  // lanes that differ in bit o split the n values
#pragma unroll
        for (int i = 0; i < n / 2; ++i) {
            const double keep = (lane & o) ? v[2 * i + 1] : v[2 * i], give = (lane & o) ? v[2 * i] : v[2 * i + 1];
            v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, o);
        }
    }
#pragma unroll
    for (; o; o >>= 1) v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], o);
}
template <int K>
__device__ __forceinline__ int many_index(int lane) { return (int)(__brev((unsigned)lane) >> 27) & (K - 1); }
template <int K>
__device__ __forceinline__ bool many_writer(int lane) { return (lane & (32 / K - 1)) == 0; }

// True in every thread of the last block of the grid to arrive at *counter (which it leaves
// at zero for the next kernel); that block then sees the partials every block has written.
__device__ __forceinline__ bool last_block(unsigned *counter) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(counter, 1u) == gridDim.x - 1;
        if (last) *counter = 0;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// Sums over the nb block partials of a reduction in a fixed order (lane l adds blocks l,
// l + 32, ..., then a butterfly over the lanes), so every result is reproducible: NI results
// at p, p + step, ... side by side, eight loads of each in flight (one after another, the
// loads of the last block took longer than the reduction itself).
template <int NI>
__device__ __forceinline__ void warp_sum_blocks(const double *p, int64_t stride, int nb, int step, double (&a)[NI]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < NI; ++q) a[q] = 0.0;
    for (int b0 = lane; b0 < nb; b0 += 256) {
        double v[NI][8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
            for (int q = 0; q < NI; ++q)
                v[q][u] = b0 + 32 * u < nb ? __ldcg(p + (int64_t)(b0 + 32 * u) * stride + q * step) : 0.0;
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (b0 + 32 * u < nb)
#pragma unroll
                for (int q = 0; q < NI; ++q) a[q] += v[q][u];
    }
    for (int o = 16; o; o >>= 1)
#pragma unroll
        for (int q = 0; q < NI; ++q) a[q] += __shfl_xor_sync(0xFFFFFFFFu, a[q], o);
}
__device__ __forceinline__ double warp_sum_blocks(const double *p, int64_t stride, int nb) {
    double a[1];
    warp_sum_blocks<1>(p, stride, nb, 0, a);
    return a[0];
}

// What the last block does with <V_i|x>, i = i0 .. i0 + k - 1.
enum { DOT_PLAIN = 0,   // out[i] = the sum (complex)
       DOT_NEGATE = 1,  // out[i] = minus the sum: the coefficients of a Gram-Schmidt update
       DOT_COLUMN = 2   // the new column (and row) `col` of the projected matrix `out`
};

// <V_i|x> for i0 <= i < i0 + k (k <= KB): KB (a power of two) sizes the accumulator arrays, so
// a call with few vectors keeps few registers and many warps resident.
template <bool CPLX, int KB>
__global__ void __launch_bounds__(RED_THREADS) k_multidot(const double *__restrict__ V, int64_t ldv, int i0, int k,
                                                          const double *__restrict__ x, int64_t n,
                                                          double *__restrict__ partial, unsigned *__restrict__ counter,
                                                          int mode, int col, double *__restrict__ out) {
    constexpr int NV = CPLX ? 2 * KB : KB;  // real values reduced: re, im interleaved if complex
    __shared__ double red[RED_THREADS / 32][NV];
    double acc[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) acc[i] = 0.0;
    const double *Vb = V + (int64_t)i0 * (CPLX ? 2 : 1) * ldv;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        if (CPLX) {
            const double xr = x[2 * j], xi = x[2 * j + 1];
#pragma unroll
            for (int i = 0; i < KB; ++i) {
                if (i < k) {
                    const double vr = Vb[i * 2 * ldv + 2 * j], vi = Vb[i * 2 * ldv + 2 * j + 1];
                    acc[(2 * i) % NV] = fma(vr, xr, fma(vi, xi, acc[(2 * i) % NV]));
                    acc[(2 * i + 1) % NV] = fma(vr, xi, fma(-vi, xr, acc[(2 * i + 1) % NV]));
                }
            }
        } else {
            const double xr = x[j];
#pragma unroll
            for (int i = 0; i < KB; ++i)
                if (i < k) acc[i] = fma(Vb[i * ldv + j], xr, acc[i]);
        }
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    warp_sum_many<NV>(acc);
    if (many_writer<NV>(lane)) red[wid][many_index<NV>(lane)] = acc[0];
    __syncthreads();
    if (threadIdx.x < NV) {
        double s = 0.0;
        for (int w = 0; w < RED_THREADS / 32; ++w) s += red[w][threadIdx.x];
        partial[(int64_t)blockIdx.x * NV + threadIdx.x] = s;
    }
    if (!last_block(counter)) return;
    // warp wid takes results wid, wid + 8, ...
    constexpr int NW = RED_THREADS / 32, NI = (KB + NW - 1) / NW;
    if (wid >= k) return;
    double sum[CPLX ? 2 * NI : NI];  // complex: re, im of each
    if (CPLX) {
#pragma unroll
        for (int q = 0; q < NI; ++q) {
            double two[2];
            warp_sum_blocks<2>(partial + 2 * min(wid + NW * q, KB - 1), NV, gridDim.x, 1, two);
            sum[CPLX ? 2 * q : 0] = two[0];
            sum[CPLX ? 2 * q + 1 : 0] = two[1];
        }
    } else {
        double all[NI];
        warp_sum_blocks<NI>(partial + wid, NV, gridDim.x, NW, all);
#pragma unroll
        for (int q = 0; q < NI; ++q) sum[q] = all[q];
    }
    if (lane) return;
#pragma unroll
    for (int q = 0; q < NI; ++q) {
        const int i = wid + NW * q, g = i0 + i;
        if (i >= k) break;
        double re = sum[CPLX ? 2 * q : q], im = CPLX ? sum[CPLX ? 2 * q + 1 : 0] : 0.0;
        if (mode == DOT_COLUMN) {
            if (g == col) im = 0.0;
            out[2 * (g * KMAX + col)] = re;
            out[2 * (g * KMAX + col) + 1] = im;
            out[2 * (col * KMAX + g)] = re;
            out[2 * (col * KMAX + g) + 1] = g == col ? 0.0 : -im;
        } else {
            if (mode == DOT_NEGATE) {
                re = -re;
                im = -im;
            }
            out[2 * g] = re;
            out[2 * g + 1] = im;
        }
    }
}

// out_b = sum_i y_i V_b,i  (+ out_b when accumulate) for the vectors V0 (and V1 if out1), y
// complex as 2 doubles per entry.  NORM (real vectors): also *n2 = ||out_0||^2,
// added in the order of k_norm2.
template <bool CPLX, bool NORM>
__global__ void __launch_bounds__(RED_THREADS) k_lincomb(const double *__restrict__ V0, const double *__restrict__ V1,
                                                         int64_t ldv, int k, const double *__restrict__ y, int64_t n,
                                                         double *__restrict__ out0, double *__restrict__ out1,
                                                         int accumulate, double *__restrict__ partial,
                                                         unsigned *__restrict__ counter, double *__restrict__ n2) {
    __shared__ double sy[2 * KMAX];
    if (threadIdx.x < 2 * k) sy[threadIdx.x] = y[threadIdx.x];
    __syncthreads();
    double norm = 0.0;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        for (int b = 0; b < (out1 ? 2 : 1); ++b) {
            const double *V = b ? V1 : V0;
            double *out = b ? out1 : out0;
            if (CPLX) {
                double re = accumulate ? out[2 * j] : 0.0, im = accumulate ? out[2 * j + 1] : 0.0;
#pragma unroll 4
                for (int i = 0; i < k; ++i) {
                    const double vr = V[i * 2 * ldv + 2 * j], vi = V[i * 2 * ldv + 2 * j + 1];
                    re = fma(sy[2 * i], vr, fma(-sy[2 * i + 1], vi, re));
                    im = fma(sy[2 * i], vi, fma(sy[2 * i + 1], vr, im));
                }
                out[2 * j] = re;
                out[2 * j + 1] = im;
            } else {
                double acc = accumulate ? out[j] : 0.0;
#pragma unroll 4
                for (int i = 0; i < k; ++i) acc = fma(sy[2 * i], V[i * ldv + j], acc);
                out[j] = acc;
                if (NORM && b == 0) norm = fma(acc, acc, norm);
            }
        }
    }
    if (NORM) {
        __shared__ double red[RED_THREADS / 32];
        for (int o = 16; o; o >>= 1) norm += __shfl_xor_sync(0xFFFFFFFFu, norm, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = norm;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0;
            for (int w = 0; w < RED_THREADS / 32; ++w) s += red[w];
            partial[blockIdx.x] = s;
        }
        if (!last_block(counter)) return;
        if (threadIdx.x < 32) {
            const double a = warp_sum_blocks(partial, 1, gridDim.x);
            if (threadIdx.x == 0) *n2 = a;
        }
    }
}

// Phase-align (c, sc) to c_prev by the scalar ph = conj(ov)/|ov|, then
//   r = sc - lam c;  s_i = r_i / (lam - H_ii) if |lam - H_ii| >= 1e-12 else 0;  t = s.
// ov = <c_prev|c>.  Into scal: ||r||^2, ||s||^2, max |c - c_prev|.
template <bool CPLX>
__global__ void __launch_bounds__(RED_THREADS) k_residual(double *__restrict__ c, double *__restrict__ sc,
                                                          const double *__restrict__ cprev, int have_prev,
                                                          const double *__restrict__ diag,
                                                          const double *__restrict__ ov, dav_scalars *__restrict__ scal,
                                                          int64_t n, double *__restrict__ t,
                                                          double *__restrict__ partial, unsigned *__restrict__ counter) {
    const double lam = scal->lam;
    double pr = 1.0, pi = 0.0;
    if (have_prev) {
        const double ore = ov[0], oim = ov[1], m = sqrt(ore * ore + oim * oim);
        if (m > 0) { pr = ore / m; pi = -oim / m; }
    }
    double r2 = 0.0, s2 = 0.0, mdc = 0.0;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        const double den = lam - diag[j];
        const bool ok = fabs(den) >= 1e-12;
        if (CPLX) {
            double cr = c[2 * j], ci = c[2 * j + 1], sr = sc[2 * j], si = sc[2 * j + 1];
            double a = cr * pr - ci * pi, b = cr * pi + ci * pr;
            cr = a; ci = b;
            a = sr * pr - si * pi; b = sr * pi + si * pr;
            sr = a; si = b;
            c[2 * j] = cr; c[2 * j + 1] = ci; sc[2 * j] = sr; sc[2 * j + 1] = si;
            const double rr = sr - lam * cr, ri = si - lam * ci;
            r2 += rr * rr + ri * ri;
            const double tr = ok ? rr / den : 0.0, ti = ok ? ri / den : 0.0;
            s2 += tr * tr + ti * ti;
            t[2 * j] = tr; t[2 * j + 1] = ti;
            if (have_prev) {
                const double dr = cr - cprev[2 * j], di = ci - cprev[2 * j + 1];
                mdc = fmax(mdc, sqrt(dr * dr + di * di));
            }
        } else {
            double cr = c[j] * pr, sr = sc[j] * pr;
            c[j] = cr; sc[j] = sr;
            const double rr = sr - lam * cr;
            r2 += rr * rr;
            const double tr = ok ? rr / den : 0.0;
            s2 += tr * tr;
            t[j] = tr;
            if (have_prev) mdc = fmax(mdc, fabs(cr - cprev[j]));
        }
    }
    __shared__ double red[3][RED_THREADS / 32];
    for (int o = 16; o; o >>= 1) {
        r2 += __shfl_xor_sync(0xFFFFFFFFu, r2, o);
        s2 += __shfl_xor_sync(0xFFFFFFFFu, s2, o);
        mdc = fmax(mdc, __shfl_xor_sync(0xFFFFFFFFu, mdc, o));
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) { red[0][wid] = r2; red[1][wid] = s2; red[2][wid] = mdc; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0, b = 0, m = 0;
        for (int w = 0; w < RED_THREADS / 32; ++w) { a += red[0][w]; b += red[1][w]; m = fmax(m, red[2][w]); }
        partial[blockIdx.x * 4 + 0] = a;
        partial[blockIdx.x * 4 + 1] = b;
        partial[blockIdx.x * 4 + 2] = m;
    }
    if (!last_block(counter) || wid != 0) return;
    double ab[2];
    warp_sum_blocks<2>(partial, 4, gridDim.x, 1, ab);
    const double a = ab[0], b = ab[1];
    double m = 0;
    for (int i = lane; i < (int)gridDim.x; i += 32) m = fmax(m, __ldcg(partial + i * 4 + 2));
    for (int o = 16; o; o >>= 1) m = fmax(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
    if (lane == 0) {
        scal->rnorm2 = a;
        scal->snorm2 = b;
        scal->maxdc = m;
    }
}

// Compression-compatible threshold: t_i = 0 where |t_i| < eps ||s||.
template <bool CPLX>
__global__ void k_threshold(double *__restrict__ t, int64_t n, const dav_scalars *__restrict__ s, double eps) {
    const double thr = eps * sqrt(s->snorm2);
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        if (CPLX) {
            const double a = t[2 * j], b = t[2 * j + 1];
            if (sqrt(a * a + b * b) < thr) { t[2 * j] = 0.0; t[2 * j + 1] = 0.0; }
        } else if (fabs(t[j]) < thr) {
            t[j] = 0.0;
        }
    }
}

// *n2 = ||x||^2 (complex counted as 2n reals).
__global__ void __launch_bounds__(RED_THREADS) k_norm2(const double *__restrict__ x, int64_t nreal,
                                                       double *__restrict__ partial, unsigned *__restrict__ counter,
                                                       double *__restrict__ n2) {
    double a = 0.0;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nreal; j += (int64_t)gridDim.x * blockDim.x)
        a = fma(x[j], x[j], a);
    __shared__ double red[RED_THREADS / 32];
    for (int o = 16; o; o >>= 1) a += __shfl_xor_sync(0xFFFFFFFFu, a, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0;
        for (int w = 0; w < RED_THREADS / 32; ++w) s += red[w];
        partial[blockIdx.x] = s;
    }
    if (!last_block(counter)) return;
    if (threadIdx.x < 32) {
        const double s = warp_sum_blocks(partial, 1, gridDim.x);
        if (threadIdx.x == 0) *n2 = s;
    }
}

// out = x / sqrt(*n2) (out may be x)
__global__ void k_scale(const double *x, double *out, int64_t nreal, const double *__restrict__ n2) {
    const double f = 1.0 / sqrt(*n2);
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nreal; j += (int64_t)gridDim.x * blockDim.x)
        out[j] = x[j] * f;
}

// One rotation: (a, b) of a row (or column) pair becomes (c a - s b, s a + c b).
__device__ __forceinline__ double rot_p(double c, double sn, double ap, double aq) { return fma(c, ap, -sn * aq); }
__device__ __forceinline__ double rot_q(double c, double sn, double ap, double aq) { return fma(sn, ap, c * aq); }
// Either of the two.
__device__ __forceinline__ double rot_one(bool q, double c, double sn, double ap, double aq) {
    return fma(q ? sn : c, ap, (q ? c : -sn) * aq);
}

// Pair t of round r (round-robin over M indices, M even): (M - 1, r), then (r + t, r - t) modulo
// M - 1; and the pair of index x, with is_q telling which of the two x is.
__device__ __forceinline__ void jac_pair(int M, int r, int t, int &p, int &q) {
    if (t == 0) {
        p = M - 1;
        q = r;
    } else {
        p = r + t < M - 1 ? r + t : r + t - (M - 1);
        q = r - t >= 0 ? r - t : r - t + (M - 1);
    }
}
__device__ __forceinline__ int jac_find(int M, int r, int x, bool &is_q) {
    if (x == M - 1 || x == r) {
        is_q = x == r;
        return 0;
    }
    const int d = x - r >= 0 ? x - r : x - r + (M - 1);
    is_q = d > M / 2 - 1;
    return is_q ? M - 1 - d : d;
}

// A low eigenpair of the k x k Hermitian Hs (leading dimension KMAX, complex entries) by
// Jacobi on the real symmetric embedding of size m = k (real) or 2k (complex), with the
// rotations of a sweep in round-robin order: each of the M - 1 rounds (M = m rounded up to
// even) pairs every index with one other, so the M / 2 rotations of a round touch disjoint
// rows and columns and run at once: angles from the current A (the classical formula, tan
// of the angle the smaller root of t^2 + 2 theta t - 1 = 0, theta = (A_qq - A_pp) / (2 A_pq)),
// then the columns of A and Q, then the rows of A.  Sweeps stop once the off-diagonal mass is
// below 1e-30 of the total.  Writes y (complex, k entries) and lam.
//
// A 32 x 32 round is 6,144 FP64 operations, and one SM does two per clock: on one block the
// projected eigenproblem took 360 us, half of a Davidson iteration on 63,504 determinants.
// A cluster of JAC_CLUSTER blocks shares a round:
//   - a 2 x 2 block (pair i, pair j) takes its column and its row rotation on its own, so a
//     thread owns such a block, without a barrier between the two phases;
//   - every block keeps a full copy of A (two buffers) and writes its results to all copies
//     through distributed shared memory, one cluster barrier per round;
//   - the rows of Q stay with one block each;
//   - the angles of the next round are computed while the others rotate, by three warps of
//     each block, from the old A: three elements of the new A per pair, then the angle (37
//     FP64 instructions by fp64_fast.cuh, 64 cycles each: what bounds a round).
// The operations on each element are those of the one-block form in the same order (the same
// bits): 360 -> 228 us on average over a solve (10 electrons in 10 orbitals, up to 32 vectors).
// root: 0 = lowest Ritz pair, 1 = second lowest (the real embedding of a complex Hermitian
// matrix has every eigenvalue twice, so there the selected entry is the (2 root)-th).
__global__ void __cluster_dims__(JAC_CLUSTER, 1, 1) __launch_bounds__(JAC_THREADS)
    k_jacobi(const double *__restrict__ Hs, int k, int cplx, int root, double *__restrict__ y,
             dav_scalars *__restrict__ out) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ double jac_smem[];  // A (two buffers, m x (m + 1)), own rows of Q
    constexpr int QROWS = 2 * KMAX / JAC_CLUSTER;
    __shared__ double cs[2][KMAX][2], el[2][KMAX];
    __shared__ double red[2][JAC_THREADS / 32];
    __shared__ double ycol[2 * KMAX];
    __shared__ int stop, best;
    const int m = cplx ? 2 * k : k;
    const int ld = m + 1;
    const int M = m + (m & 1), half = M / 2;
    const int rank = (int)cluster.block_rank();
    double *Ab = jac_smem, *Qb = jac_smem + 2 * m * ld;
    const int t = threadIdx.x, nt = blockDim.x;
    if (t == 0) best = 0;  // stays if NaN leaves no entry with the wanted rank (the host sees lam)
    for (int i = t; i < m * m; i += nt) {
        const int r = i / m, c = i % m;
        double v;
        if (!cplx) {
            v = Hs[2 * (r * KMAX + c)];
        } else {
            const int rb = r / k, cb = c / k, rr = r % k, cc = c % k;
            const double re = Hs[2 * (rr * KMAX + cc)], im = Hs[2 * (rr * KMAX + cc) + 1];
            v = (rb == cb) ? re : (rb == 1 ? im : -im);
        }
        Ab[r * ld + c] = v;
    }
    for (int i = t; i < QROWS * m; i += nt) {  // row rank + JAC_CLUSTER * (i / m)
        const int r = rank + JAC_CLUSTER * (i / m), c = i % m;
        Qb[(i / m) * ld + c] = (r == c) ? 1.0 : 0.0;
    }
    __syncthreads();
    // angle of the pair (p, q) from its three elements (comparisons on the bits: every FP64
    // instruction of this chain costs 64 cycles)
    auto angle = [&](double apq, double app, double aqq, double &c, double &sn) {
        c = 1.0;
        sn = 0.0;
        const int ex = fp64_fast::exponent(apq);
        if (ex > 30 ? ex < 2046 : fabs(apq) > 1e-300) {  // 2^-993 > 1e-300
            const double theta = fp64_fast::divide(aqq - app, fp64_fast::twice(apq));
            double y0, y1;
            const double den = fabs(theta) + fp64_fast::root(theta * theta + 1.0, y0);
            const double tt = fp64_fast::reciprocal(theta >= 0 ? 1.0 : -1.0, den);
            const double s = fp64_fast::root(tt * tt + 1.0, y1);  // in [1, sqrt 2]
            c = fp64_fast::reciprocal_near(s, y1);
            sn = tt * c;
        }
    };
    int buf = 0;  // current buffer of A and of the angles
    if (t < half) {
        int p, q;
        jac_pair(M, 0, t, p, q);
        double c = 1.0, sn = 0.0;
        if (p < m && q < m) angle(Ab[p * ld + q], Ab[p * ld + p], Ab[q * ld + q], c, sn);
        cs[0][t][0] = c;
        cs[0][t][1] = sn;
    }
    cluster.sync();  // every copy of A is loaded before a neighbour writes to it
    for (int sweep = 0; sweep < 60 && m > 1; ++sweep) {
        const double *A0 = Ab + buf * m * ld;
        double off = 0.0, tot = 0.0;
        for (int i = t; i < m * m; i += nt) {
            const int r = i / m, c = i % m;
            const double a2 = A0[r * ld + c] * A0[r * ld + c];
            tot += a2;
            if (r != c) off += a2;
        }
        for (int o = 16; o; o >>= 1) {
            off += __shfl_xor_sync(0xFFFFFFFFu, off, o);
            tot += __shfl_xor_sync(0xFFFFFFFFu, tot, o);
        }
        if ((t & 31) == 0) {
            red[0][t >> 5] = off;
            red[1][t >> 5] = tot;
        }
        __syncthreads();
        if (t == 0) {
            double o = 0.0, a = 0.0;
            for (int w = 0; w < nt / 32; ++w) {
                o += red[0][w];
                a += red[1][w];
            }
            stop = (o <= 1e-30 * a) || o == 0.0;
        }
        __syncthreads();
        if (stop) break;  // every block of the cluster has the same A and decides the same
        for (int r = 0; r < M - 1; ++r, buf ^= 1) {
            const double *A = Ab + buf * m * ld;
            double *An = Ab + (buf ^ 1) * m * ld;
            const double(*rot)[2] = cs[buf];
            if (t < 96) {
                // angles of the next round's pairs (round 0 after the last of a sweep), on one SM
                // sub-partition per element: warp 0 takes A_pq, warp 1 A_pp, warp 2 A_qq of A after
                // this round, then warp 0 the angle.  An identity rotation (1, 0) keeps its values,
                // and the padding index of a pair reads as zero.
                const int rn = r + 1 < M - 1 ? r + 1 : 0, warp = t >> 5, lane = t & 31;
                int p = 0, q = 0;
                bool on = lane < half;
                if (on) jac_pair(M, rn, lane, p, q);
                on = on && p < m && q < m;
                double v = 0.0;
                if (on) {
                    const int row = warp == 2 ? q : p, col = warp == 1 ? p : q;
                    bool row_q, col_q;
                    const int i = jac_find(M, r, row, row_q), j = jac_find(M, r, col, col_q);
                    int pi, qi, pj, qj;
                    jac_pair(M, r, i, pi, qi);
                    jac_pair(M, r, j, pj, qj);
                    const double ci = rot[i][0], si = rot[i][1], cj = rot[j][0], sj = rot[j][1];
                    const bool rp = pi < m, cp = pj < m;
                    const double a00 = rp && cp ? A[pi * ld + pj] : 0.0, a01 = rp ? A[pi * ld + qj] : 0.0;
                    const double a10 = cp ? A[qi * ld + pj] : 0.0, a11 = A[qi * ld + qj];
                    v = rot_one(row_q, ci, si, rot_one(col_q, cj, sj, a00, a01), rot_one(col_q, cj, sj, a10, a11));
                    if (warp) el[warp - 1][lane] = v;
                }
                asm volatile("bar.sync 1, 96;" ::: "memory");
                if (warp == 0 && lane < half) {
                    double c = 1.0, sn = 0.0;
                    if (on) angle(v, el[0][lane], el[1][lane], c, sn);
                    cs[buf ^ 1][lane][0] = c;
                    cs[buf ^ 1][lane][1] = sn;
                }
            } else {
                const int w = t - 96, nw = nt - 96;
                // own share of the 2 x 2 blocks
                for (int b = rank + JAC_CLUSTER * w; b < half * half; b += JAC_CLUSTER * nw) {
                    const int i = b / half, j = b - i * half;
                    int pi, qi, pj, qj;
                    jac_pair(M, r, i, pi, qi);
                    jac_pair(M, r, j, pj, qj);
                    const double ci = rot[i][0], si = rot[i][1], cj = rot[j][0], sj = rot[j][1];
                    const bool rp = pi < m, cp = pj < m;  // only p can be the padding index
                    double a00 = rp && cp ? A[pi * ld + pj] : 0.0, a01 = rp ? A[pi * ld + qj] : 0.0;
                    double a10 = cp ? A[qi * ld + pj] : 0.0, a11 = A[qi * ld + qj];
                    if (sj != 0.0) {
                        const double b00 = rot_p(cj, sj, a00, a01), b01 = rot_q(cj, sj, a00, a01);
                        const double b10 = rot_p(cj, sj, a10, a11), b11 = rot_q(cj, sj, a10, a11);
                        a00 = b00; a01 = b01; a10 = b10; a11 = b11;
                    }
                    if (si != 0.0) {
                        const double b00 = rot_p(ci, si, a00, a10), b10 = rot_q(ci, si, a00, a10);
                        const double b01 = rot_p(ci, si, a01, a11), b11 = rot_q(ci, si, a01, a11);
                        a00 = b00; a01 = b01; a10 = b10; a11 = b11;
                    }
#pragma unroll
                    for (int g = 0; g < JAC_CLUSTER; ++g) {
                        double *R = cluster.map_shared_rank(An, g);
                        if (rp && cp) R[pi * ld + pj] = a00;
                        if (rp) R[pi * ld + qj] = a01;
                        if (cp) R[qi * ld + pj] = a10;
                        R[qi * ld + qj] = a11;
                    }
                }
                // own rows of Q
                for (int b = w; b < QROWS * half; b += nw) {
                    const int i = b / half, j = b - i * half;
                    const double sj = rot[j][1], cj = rot[j][0];
                    if (rank + JAC_CLUSTER * i >= m || sj == 0.0) continue;
                    int pj, qj;
                    jac_pair(M, r, j, pj, qj);
                    const double qp = Qb[i * ld + pj], qq = Qb[i * ld + qj];
                    Qb[i * ld + pj] = rot_p(cj, sj, qp, qq);
                    Qb[i * ld + qj] = rot_q(cj, sj, qp, qq);
                }
            }
            cluster.sync();
        }
    }
    // the (root * (cplx ? 2 : 1))-th smallest diagonal entry (ties: lowest index)
    const double *A = Ab + buf * m * ld;
    const int want = root * (cplx ? 2 : 1);
    if (t < m) {
        int before = 0;  // entries before t in the ascending order
        for (int j = 0; j < m; ++j)
            if (A[j * ld + j] < A[t * ld + t] || (A[j * ld + j] == A[t * ld + t] && j < t)) ++before;
        if (before == want) best = t;
    }
    __syncthreads();
    {
        double *col = cluster.map_shared_rank(ycol, 0);
        for (int i = t; i < QROWS; i += nt)
            if (rank + JAC_CLUSTER * i < m) col[rank + JAC_CLUSTER * i] = Qb[i * ld + best];
    }
    cluster.sync();
    if (rank == 0 && t == 0) {
        out->lam = A[best * ld + best];
        double nrm = 0.0;
        for (int i = 0; i < k; ++i) {
            const double re = ycol[i], im = cplx ? ycol[k + i] : 0.0;
            y[2 * i] = re;
            y[2 * i + 1] = im;
            nrm += re * re + im * im;
        }
        nrm = 1.0 / sqrt(nrm);
        for (int i = 0; i < 2 * k; ++i) y[i] *= nrm;
    }
}

// argmin of diag (lowest index on ties) -> unit vector
// Index of the smallest diagonal element (the lowest index among equal ones), in two
// passes: per block (value, index) into part, then one block over the nb block results.
__device__ __forceinline__ void argmin_merge(double &v, int64_t &i, double v2, int64_t i2) {
    if (v2 < v || (v2 == v && i2 < i)) { v = v2; i = i2; }
}
__device__ void argmin_block(double v, int64_t idx, double *bv, int64_t *bi) {
    for (int o = 16; o; o >>= 1)
        argmin_merge(v, idx, __shfl_xor_sync(0xFFFFFFFFu, v, o), __shfl_xor_sync(0xFFFFFFFFu, idx, o));
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) { bv[wid] = v; bi[wid] = idx; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) argmin_merge(v, idx, bv[w], bi[w]);
        bv[0] = v;
        bi[0] = idx;
    }
}
__global__ void __launch_bounds__(256) k_argmin_part(const double *__restrict__ d, int64_t n, double *__restrict__ part) {
    __shared__ double bv[8];
    __shared__ int64_t bi[8];
    double v = INFINITY;
    int64_t idx = INT64_MAX;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
        if (d[j] < v) { v = d[j]; idx = j; }
    argmin_block(v, idx, bv, bi);
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = bv[0];
        part[2 * blockIdx.x + 1] = __longlong_as_double((long long)bi[0]);
    }
}
__global__ void __launch_bounds__(256) k_argmin_final(const double *__restrict__ part, int nb, int64_t *__restrict__ out) {
    __shared__ double bv[8];
    __shared__ int64_t bi[8];
    double v = INFINITY;
    int64_t idx = INT64_MAX;
    for (int b = threadIdx.x; b < nb; b += blockDim.x)
        argmin_merge(v, idx, part[2 * b], (int64_t)__double_as_longlong(part[2 * b + 1]));
    argmin_block(v, idx, bv, bi);
    if (threadIdx.x == 0) *out = bi[0] == INT64_MAX ? 0 : bi[0];
}

// splitmix64 (Steele, Lea and Flood 2014, "Fast splittable pseudorandom number
// generators"): the published finaliser of a 64-bit counter.
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Start vector: the unit vector at idx plus, if mix > 0, mix times a pseudo-random vector
// of norm about one (entries uniform in [-1, 1) from splitmix64 of the index, scaled by
// sqrt(3 / nreal)).  The admixture gives the start a component in every symmetry sector
// (a closed-shell unit vector alone is symmetric under alpha <-> beta exchange, and the
// iteration would stay in that sector).
__global__ void k_set_start(double *__restrict__ x, int64_t nreal, int cplx, const int64_t *__restrict__ idx,
                            double mix) {
    const int64_t at = (cplx ? 2 : 1) * (*idx);
    const double scale = mix * sqrt(3.0 / (double)nreal);
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nreal; j += (int64_t)gridDim.x * blockDim.x) {
        double v = (j == at) ? 1.0 : 0.0;
        if (mix > 0.0) v += scale * (2.0 * (double)(splitmix64((uint64_t)j) >> 11) * 0x1.0p-53 - 1.0);
        x[j] = v;
    }
}

// Shared memory of k_jacobi at size m: two buffers of A, this block's rows of Q.
inline size_t jac_smem_bytes(int m) { return (size_t)(2 * m + 2 * KMAX / JAC_CLUSTER) * (m + 1) * sizeof(double); }

inline size_t al(size_t b) { return (b + 255) & ~(size_t)255; }

}  // namespace

// Davidson as a state machine: run_until_sigma() advances the iteration until the next
// sigma product is needed (it then exposes x and y = H x to the caller) or until the
// solve ends.  davidson_solve drives it with the library's own sigma; the step-wise C ABI
// (davidson_begin/advance/finish) lets a scheduler compute the sigma products of many
// solves together.
struct fci_davidson_state {
    enum { REQ_NONE = 0, REQ_INIT, REQ_SWITCH, REQ_APPEND };
    fci_context *h = nullptr;
    fci_davidson_opts o{};
    cudaStream_t s = nullptr;
    int64_t n = 0, nreal = 0, ldv = 0;
    bool cplx = false;
    size_t esz = 8, vec = 0;
    int ms = 0;
    double *V = nullptr, *S = nullptr, *c = nullptr, *sc = nullptr, *cp = nullptr, *scp = nullptr, *t = nullptr,
           *diag = nullptr;
    void *sig_ws = nullptr;
    size_t sig_bytes = 0;
    double *partial = nullptr, *Hs = nullptr, *dots = nullptr, *y = nullptr, *nrm = nullptr, *ov = nullptr;
    unsigned *counter = nullptr;  // blocks done in the running reduction (zero between kernels)
    double *ritz = nullptr;       // the current Ritz vector (c, or c_prev after the exchange)
    dav_scalars *scal = nullptr;
    int64_t *argmin = nullptr;
    unsigned vb = 1;
    // iteration state
    int k = 0, it = 0, it_rec = 0, phase1_iters = 0, n_sigma = 0;
    int prec = FCI_PREC_FP64, slices = 0;
    bool final_phase = true, have_prev = false, converged = false, done = false;
    double E_prev = 0.0, lam_pending = 0.0;
    int request = REQ_NONE;
    double *req_x = nullptr, *req_y = nullptr;
    double *stage_x = nullptr, *stage_y = nullptr, *real_y = nullptr;  // staged sigma requests
    // gap bound (Results, Eq. gammaLowerBound): after convergence, the second Ritz pair
    bool gap_phase = false;
    int gap_iters = 0;
    double E1 = NAN, r1n = NAN, r0n = NAN, gap_lower = NAN, err_bound = NAN;
    std::chrono::steady_clock::time_point t_iter;
    std::vector<fci_davidson_iter> log;
    int status = FCI_OK;

    double *Vk(int i) { return (double *)((char *)V + (size_t)i * vec); }
    double *Sk(int i) { return (double *)((char *)S + (size_t)i * vec); }

    template <int KB>
    void multidot_kb(const double *Vb, int i0, int kk, const double *x, int mode, int col, double *out) {
        if (cplx) k_multidot<true, (KB <= 16 ? KB : 16)><<<vb, RED_THREADS, 0, s>>>(Vb, ldv, i0, kk, x, n, partial, counter, mode, col, out);
        else k_multidot<false, KB><<<vb, RED_THREADS, 0, s>>>(Vb, ldv, i0, kk, x, n, partial, counter, mode, col, out);
    }
    // <V_i|x> for i < kk: one pass (real, and complex up to 16 vectors), else 16 vectors per pass
    cudaError_t multidot(const double *Vb, int kk, const double *x, double *out, int mode = DOT_PLAIN, int col = 0) {
        if (kk <= 1) multidot_kb<1>(Vb, 0, kk, x, mode, col, out);
        else if (kk <= 4) multidot_kb<4>(Vb, 0, kk, x, mode, col, out);
        else if (kk <= 8) multidot_kb<8>(Vb, 0, kk, x, mode, col, out);
        else if (kk <= 16) multidot_kb<16>(Vb, 0, kk, x, mode, col, out);
        else if (!cplx) multidot_kb<32>(Vb, 0, kk, x, mode, col, out);
        else {
            multidot_kb<16>(Vb, 0, 16, x, mode, col, out);
            multidot_kb<16>(Vb, 16, kk - 16, x, mode, col, out);
        }
        return cudaGetLastError();
    }
    // out0 (and out1) = sum_i yy_i V0_i (V1_i), added to what is there if acc; n2 = ||out0||^2 if given
    cudaError_t lincomb(const double *V0, int kk, const double *yy, double *out0, int acc, double *n2 = nullptr,
                        const double *V1 = nullptr, double *out1 = nullptr) {
        if (cplx) {  // the norm of a complex vector adds its 2n reals in k_norm2's order
            k_lincomb<true, false><<<vb, RED_THREADS, 0, s>>>(V0, V1, ldv, kk, yy, n, out0, out1, acc, partial, counter, n2);
            if (n2) norm2(out0, n2);
        } else if (n2) {
            k_lincomb<false, true><<<vb, RED_THREADS, 0, s>>>(V0, V1, ldv, kk, yy, n, out0, out1, acc, partial, counter, n2);
        } else {
            k_lincomb<false, false><<<vb, RED_THREADS, 0, s>>>(V0, V1, ldv, kk, yy, n, out0, out1, acc, partial, counter, n2);
        }
        return cudaGetLastError();
    }
    void norm2(const double *x, double *n2) { k_norm2<<<vb, RED_THREADS, 0, s>>>(x, nreal, partial, counter, n2); }
    void scale(const double *x, double *out, const double *n2) { k_scale<<<vb, RED_THREADS, 0, s>>>(x, out, nreal, n2); }
    cudaError_t normalize(double *x, double *n2out) {
        norm2(x, n2out);
        scale(x, x, n2out);
        return cudaGetLastError();
    }
    // Ritz pair `root` of the projected matrix: y and scal->lam
    void ritz_pair(int root) {
        const int m = cplx ? 2 * k : k;
        k_jacobi<<<JAC_CLUSTER, JAC_THREADS, jac_smem_bytes(m), s>>>(Hs, k, cplx ? 1 : 0, root, y, scal);
    }
    void residual(bool with_prev) {
        if (cplx) k_residual<true><<<vb, RED_THREADS, 0, s>>>(c, sc, cp, with_prev, diag, ov, scal, n, t, partial, counter);
        else k_residual<false><<<vb, RED_THREADS, 0, s>>>(c, sc, cp, with_prev, diag, ov, scal, n, t, partial, counter);
    }
    // New subspace column kk: Hs[:, kk] = V^H S_kk.
    int add_column(int kk) {
        FCI_CUDA(h, multidot(V, kk + 1, Sk(kk), Hs, DOT_COLUMN, kk));
        return FCI_OK;
    }
    int ask(int kind, double *x, double *yv) {
        request = kind;
        req_x = x;
        req_y = yv;
        ++n_sigma;
        if (o.staged_sigma) {  // the caller always sees the same two vectors
            FCI_CUDA(h, cudaMemcpyAsync(stage_x, x, (size_t)n * esz, cudaMemcpyDeviceToDevice, s));
            req_x = stage_x;
            req_y = stage_y;
            real_y = yv;
        }
        return FCI_OK;
    }

    int init(fci_context *hh, const fci_davidson_opts *oo, const void *guess, void *ws, cudaStream_t st) {
        h = hh;
        o = *oo;
        s = st;
        n = h->das_active ? h->das.n_det : h->ndet;
        cplx = h->dtype == FCI_C128;
        esz = cplx ? 16 : 8;
        nreal = cplx ? 2 * n : n;
        vec = al((size_t)n * esz);
        ms = o.max_subspace;
        char *p = (char *)ws;
        V = (double *)p; p += ms * vec;
        S = (double *)p; p += ms * vec;
        c = (double *)p; p += vec;
        sc = (double *)p; p += vec;
        cp = (double *)p; p += vec;
        scp = (double *)p; p += vec;
        t = (double *)p; p += vec;
        diag = (double *)p; p += al((size_t)n * 8);
        if (o.staged_sigma) {
            stage_x = (double *)p; p += vec;
            stage_y = (double *)p; p += vec;
        }
        sig_ws = p;
        size_t sig = sigma_ws_bytes(h, o.precision, o.n_slices);
        if (o.precision != FCI_PREC_FP64) sig = std::max(sig, sigma_ws_bytes(h, o.final_precision, o.final_slices));
        sig_bytes = al(sig);
        ldv = (int64_t)(vec / esz);
        double *small = h->d_small;
        partial = small;                           // RED_BLOCKS * 2 * KMAX
        Hs = partial + RED_BLOCKS * 2 * KMAX;      // 2 * KMAX * KMAX
        dots = Hs + 2 * KMAX * KMAX;               // 2 * KMAX
        y = dots + 2 * KMAX;                       // 2 * KMAX
        nrm = y + 2 * KMAX;                        // 4
        ov = nrm + 4;                              // 2
        scal = (dav_scalars *)(ov + 2);
        argmin = (int64_t *)(scal + 1);
        counter = (unsigned *)(argmin + 1);
        vb = (unsigned)std::min<int64_t>(RED_BLOCKS, std::max<int64_t>(1, ceil_div(n, RED_THREADS)));
        ritz = c;
        FCI_CUDA(h, cudaMemsetAsync(counter, 0, sizeof(unsigned), s));
        prec = o.precision;
        slices = o.n_slices;
        if (o.eps < 0.0) o.eps = 10.0 / sqrt((double)n);  // the paper's eps <~ 10 / sqrt(N_dets) rule
        final_phase = o.precision == FCI_PREC_FP64 || (o.precision == o.final_precision && o.n_slices == o.final_slices);
        FCI_CUDA(h, cudaFuncSetAttribute(k_jacobi, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)jac_smem_bytes(2 * KMAX)));
        if (h->das_active) FCI_CUDA(h, launch_diag_das(h, diag, s));
        else if (h->mode == FCI_MODE_SPINOR) FCI_CUDA(h, launch_diag_spinor(h, diag, s));
        else FCI_CUDA(h, launch_diag_fci(h, diag, s));
        if (guess) {
            FCI_CUDA(h, cudaMemcpyAsync(Vk(0), guess, (size_t)n * esz, cudaMemcpyDeviceToDevice, s));
        } else {
            k_argmin_part<<<vb, 256, 0, s>>>(diag, n, partial);
            k_argmin_final<<<1, 256, 0, s>>>(partial, (int)vb, argmin);
            k_set_start<<<vb, RED_THREADS, 0, s>>>(Vk(0), nreal, cplx, argmin, o.start_mix);
        }
        FCI_CUDA(h, normalize(Vk(0), nrm));
        return ask(REQ_INIT, Vk(0), Sk(0));
    }

    // The caller has written y = H x for the pending request.
    int consume_sigma() {
        int rc;
        if (o.staged_sigma && request != REQ_NONE)
            FCI_CUDA(h, cudaMemcpyAsync(real_y, stage_y, (size_t)n * esz, cudaMemcpyDeviceToDevice, s));
        switch (request) {
            case REQ_INIT:
                FCI_CUDA(h, cudaMemsetAsync(Hs, 0, 2 * KMAX * KMAX * 8, s));
                if ((rc = add_column(0))) return rc;
                k = 1;
                break;
            case REQ_SWITCH:
                FCI_CUDA(h, cudaMemsetAsync(Hs, 0, 2 * KMAX * KMAX * 8, s));
                if ((rc = add_column(0))) return rc;
                k = 1;
                FCI_CUDA(h, cudaMemcpyAsync(cp, c, (size_t)n * esz, cudaMemcpyDeviceToDevice, s));
                have_prev = true;
                E_prev = lam_pending;
                break;
            case REQ_APPEND:
                if ((rc = add_column(k))) return rc;
                ++k;
                break;
            default:
                return fci_fail(h, FCI_ERR_STATE, "no sigma product was requested");
        }
        request = REQ_NONE;
        return FCI_OK;
    }

    // Advance until the next sigma request (returns FCI_OK with request != REQ_NONE) or
    // until the solve ends (done = true).
    int run_until_sigma() {
        int rc;
        dav_scalars hs{};
        while (!done) {
            if (!gap_phase && it >= o.max_iter) {
                done = true;
                break;
            }
            if (!gap_phase) ++it;  // second-root passes have their own limit (max_iter of them)
            t_iter = std::chrono::steady_clock::now();
            ritz_pair(gap_phase ? 1 : 0);
            FCI_CUDA(h, lincomb(V, k, y, c, 0, nullptr, S, sc));
            ritz = c;
            if (have_prev) FCI_CUDA(h, multidot(cp, 1, c, ov));  // <c_prev|c>
            residual(have_prev);
            FCI_CUDA(h, cudaGetLastError());
            FCI_CUDA(h, cudaMemcpyAsync(&hs, scal, sizeof hs, cudaMemcpyDeviceToHost, s));
            FCI_CUDA(h, cudaStreamSynchronize(s));
            const double lam = hs.lam, rn = sqrt(hs.rnorm2);
            const double dE = it > 1 ? lam - E_prev : 0.0;
            const auto t1 = std::chrono::steady_clock::now();
            fci_davidson_iter r;
            r.iteration = it;
            r.precision = prec;
            r.energy = lam;  // sigma carries e_core C
            r.delta_energy = dE;
            r.max_delta_c = have_prev ? hs.maxdc : 0.0;
            r.residual_norm = rn;
            r.seconds = std::chrono::duration<double>(t1 - t_iter).count();
            if (!gap_phase) log.push_back(r);
            if (!isfinite(lam) || !isfinite(rn)) return fci_fail(h, FCI_ERR_CUDA, "Davidson produced a non-finite value");
            if (!final_phase) {
                ++phase1_iters;
                if (rn <= o.switch_residual || phase1_iters >= o.max_iter / 2) {
                    // Residual correction: restart from the Ritz vector with the final precision.
                    final_phase = true;
                    prec = o.final_precision;
                    slices = o.final_slices;
                    FCI_CUDA(h, cudaMemcpyAsync(Vk(0), c, (size_t)n * esz, cudaMemcpyDeviceToDevice, s));
                    FCI_CUDA(h, normalize(Vk(0), nrm));
                    lam_pending = lam;
                    return ask(REQ_SWITCH, Vk(0), Sk(0));
                }
            } else if (gap_phase) {
                ++gap_iters;
                E1 = lam;
                r1n = rn;
                if (rn <= std::max(o.tol_residual, 0.25 * (lam - E_prev)) || gap_iters >= o.max_iter ||
                    (k >= ms && ms < 3)) {
                    if ((rc = finish_gap())) return rc;
                    done = true;
                    break;
                }
            } else if (rn <= o.tol_residual && it > 1 && fabs(dE) <= o.tol_energy) {
                converged = true;
                E_prev = lam;
                if (o.gap_bound && k >= 2) {
                    // keep the subspace and steer it to the second Ritz pair (root 0 stays in it)
                    gap_phase = true;
                    have_prev = false;
                    r0n = rn;
                    continue;  // the next pass re-diagonalises for root 1
                }
                done = true;
                break;
            }
            if (o.eps > 0.0) {
                if (cplx) k_threshold<true><<<vb, RED_THREADS, 0, s>>>(t, n, scal, o.eps);
                else k_threshold<false><<<vb, RED_THREADS, 0, s>>>(t, n, scal, o.eps);
            }
            if (k >= ms && !gap_phase) {
                // collapse to the current and previous Ritz vectors (sigma by linearity)
                // V_0 = c / ||c||, S_0 = sc / ||c||
                norm2(c, nrm);
                scale(c, Vk(0), nrm);
                scale(sc, Sk(0), nrm);
                int knew = 1;
                if (have_prev && ms > 2) {
                    // p = c_prev - <c|c_prev> c, S_p = sc_prev - <c|c_prev> sc, both / ||p||.
                    // Two Gram-Schmidt passes: c and c_prev are nearly parallel near
                    // convergence, and one pass leaves an orthogonality error of eps / ||p||
                    // that compounds over successive collapses.
                    FCI_CUDA(h, cudaMemcpyAsync(Vk(1), cp, (size_t)n * esz, cudaMemcpyDeviceToDevice, s));
                    FCI_CUDA(h, cudaMemcpyAsync(Sk(1), scp, (size_t)n * esz, cudaMemcpyDeviceToDevice, s));
                    for (int pass = 0; pass < 2; ++pass) {
                        FCI_CUDA(h, multidot(Vk(0), 1, Vk(1), dots, DOT_NEGATE));
                        FCI_CUDA(h, lincomb(Vk(0), 1, dots, Vk(1), 1, nullptr, Sk(0), Sk(1)));
                    }
                    norm2(Vk(1), nrm);
                    double pn2 = 0.0;
                    FCI_CUDA(h, cudaMemcpyAsync(&pn2, nrm, 8, cudaMemcpyDeviceToHost, s));
                    FCI_CUDA(h, cudaStreamSynchronize(s));
                    if (sqrt(pn2) > 1e-10) {
                        scale(Vk(1), Vk(1), nrm);
                        scale(Sk(1), Sk(1), nrm);
                        knew = 2;
                    }
                }
                FCI_CUDA(h, cudaMemsetAsync(Hs, 0, 2 * KMAX * KMAX * 8, s));
                for (int jj = 0; jj < knew; ++jj)
                    if ((rc = add_column(jj))) return rc;
                k = knew;
            }
            if (k >= ms && gap_phase) {
                // collapse to the ground-state Ritz vector (it must stay in the subspace for
                // the final E_0) and the current second Ritz vector orthogonalised against it;
                // c_prev / sc_prev are free in this phase and hold the ground state meanwhile
                ritz_pair(0);
                FCI_CUDA(h, lincomb(V, k, y, cp, 0, nrm, S, scp));
                scale(cp, Vk(0), nrm);
                scale(scp, Sk(0), nrm);
                FCI_CUDA(h, cudaMemcpyAsync(Vk(1), c, (size_t)n * esz, cudaMemcpyDeviceToDevice, s));
                FCI_CUDA(h, cudaMemcpyAsync(Sk(1), sc, (size_t)n * esz, cudaMemcpyDeviceToDevice, s));
                for (int pass = 0; pass < 2; ++pass) {
                    FCI_CUDA(h, multidot(Vk(0), 1, Vk(1), dots, DOT_NEGATE));
                    FCI_CUDA(h, lincomb(Vk(0), 1, dots, Vk(1), 1, nullptr, Sk(0), Sk(1)));
                }
                norm2(Vk(1), nrm);
                scale(Vk(1), Vk(1), nrm);
                scale(Sk(1), Sk(1), nrm);
                FCI_CUDA(h, cudaGetLastError());
                FCI_CUDA(h, cudaMemsetAsync(Hs, 0, 2 * KMAX * KMAX * 8, s));
                for (int jj = 0; jj < 2; ++jj)
                    if ((rc = add_column(jj))) return rc;
                k = 2;
            }
            // two rounds of classical Gram-Schmidt against V[0..k)
            for (int round = 0; round < 2; ++round) {
                FCI_CUDA(h, multidot(V, k, t, dots, DOT_NEGATE));
                FCI_CUDA(h, lincomb(V, k, dots, t, 1, round ? nrm : nullptr));
            }
            double tn2 = 0.0;
            FCI_CUDA(h, cudaMemcpyAsync(&tn2, nrm, 8, cudaMemcpyDeviceToHost, s));
            FCI_CUDA(h, cudaStreamSynchronize(s));
            if (!gap_phase) {
                have_prev = true;
                E_prev = lam;
            }
            if (!(sqrt(tn2) >= 1e-10)) {  // new direction linearly dependent on the subspace
                if (gap_phase && (rc = finish_gap())) return rc;
                done = true;
                break;
            }
            if (!gap_phase) {  // this Ritz pair is the next step's previous one
                std::swap(c, cp);
                std::swap(sc, scp);
            }
            scale(t, Vk(k), nrm);
            FCI_CUDA(h, cudaGetLastError());
            return ask(REQ_APPEND, Vk(k), Sk(k));
        }
        return FCI_OK;
    }

    // Root 0 on the final subspace (its Ritz vector goes back to c), then the gap bound:
    // gamma_0^- = (E_1 - ||r_1||) - E_0 and |dE| <= ||r_0||^2 / gamma_0^- (gap theorem).
    int finish_gap() {
        dav_scalars hs{};
        ritz_pair(0);
        FCI_CUDA(h, lincomb(V, k, y, c, 0, nullptr, S, sc));
        ritz = c;
        residual(false);
        FCI_CUDA(h, cudaGetLastError());
        FCI_CUDA(h, cudaMemcpyAsync(&hs, scal, sizeof hs, cudaMemcpyDeviceToHost, s));
        FCI_CUDA(h, cudaStreamSynchronize(s));
        E_prev = hs.lam;
        r0n = sqrt(hs.rnorm2);
        gap_lower = (E1 - r1n) - E_prev;
        err_bound = gap_lower > 0.0 ? r0n * r0n / gap_lower : INFINITY;
        return FCI_OK;
    }

    int finish(void *C_out, double *energy, fci_davidson_log *lg) {
        if (C_out) FCI_CUDA(h, cudaMemcpyAsync(C_out, ritz, (size_t)n * esz, cudaMemcpyDeviceToDevice, s));
        FCI_CUDA(h, cudaStreamSynchronize(s));
        if (energy) *energy = E_prev;
        if (lg) {
            const int m = std::min<int>((int)log.size(), lg->capacity);
            if (lg->iters)
                for (int i = 0; i < m; ++i) lg->iters[i] = log[i];
            lg->n_iter = lg->iters ? m : 0;
            lg->converged = converged ? 1 : 0;
            lg->n_sigma = n_sigma;
            lg->e1 = E1;
            lg->r1_norm = r1n;
            lg->r0_norm = r0n;
            lg->gap_lower = gap_lower;
            lg->error_bound = err_bound;
            lg->gap_iterations = gap_iters;
        }
        if (!converged)
            return fci_fail(h, FCI_ERR_NOT_CONVERGED, "Davidson did not converge in %d iterations", o.max_iter);
        return FCI_OK;
    }
};

size_t davidson_ws_bytes(const fci_context *h, const fci_davidson_opts *o) {
    const int64_t n = h->das_active ? h->das.n_det : h->ndet;
    const size_t esz = h->dtype == FCI_C128 ? 16 : 8;
    const size_t vec = al((size_t)n * esz);
    size_t sig = sigma_ws_bytes(h, o->precision, o->n_slices);
    if (o->precision != FCI_PREC_FP64) sig = std::max(sig, sigma_ws_bytes(h, o->final_precision, o->final_slices));
    return 2 * (size_t)o->max_subspace * vec + (o->staged_sigma ? 7 : 5) * vec + al((size_t)n * 8) + al(sig);
}

int davidson_run(fci_context *h, const fci_davidson_opts *o, double *C_io, double *energy, fci_davidson_log *log,
                 void *ws, size_t ws_bytes, cudaStream_t s) {
    (void)ws_bytes;
    fci_davidson_state st;
    int rc = st.init(h, o, o->use_guess ? C_io : nullptr, ws, s);
    while (!rc) {
        rc = sigma_dispatch(h, st.req_x, st.req_y, st.prec, st.slices, st.sig_ws, st.sig_bytes, s);
        if (rc) break;
        if ((rc = st.consume_sigma())) break;
        if ((rc = st.run_until_sigma())) break;
        if (st.done) break;
    }
    if (rc) return rc;
    return st.finish(C_io, energy, log);
}

// ------------------------------------------------------------------ step-wise ABI

int davidson_state_begin(fci_context *h, const fci_davidson_opts *o, const void *guess, void *ws, cudaStream_t s,
                         fci_davidson_state **out) {
    fci_davidson_state *st = new (std::nothrow) fci_davidson_state();
    if (!st) return fci_fail(h, FCI_ERR_OOM, "host allocation failed");
    int rc = st->init(h, o, guess, ws, s);
    if (rc) {
        delete st;
        return rc;
    }
    *out = st;
    return FCI_OK;
}

int davidson_state_advance(fci_davidson_state *st, int *done) {
    int rc = st->consume_sigma();
    if (!rc) rc = st->run_until_sigma();
    *done = st->done ? 1 : 0;
    return rc;
}

void davidson_state_request(const fci_davidson_state *st, const void **x, void **y, int *prec, int *slices,
                            void **sig_ws, size_t *sig_bytes) {
    if (x) *x = st->req_x;
    if (y) *y = st->req_y;
    if (prec) *prec = st->prec;
    if (slices) *slices = st->slices;
    if (sig_ws) *sig_ws = st->sig_ws;
    if (sig_bytes) *sig_bytes = st->sig_bytes;
}

int davidson_state_finish(fci_davidson_state *st, void *C_out, double *energy, fci_davidson_log *log) {
    const int rc = st->finish(C_out, energy, log);
    delete st;
    return rc;
}

fci_context *davidson_state_handle(const fci_davidson_state *st) { return st->h; }
