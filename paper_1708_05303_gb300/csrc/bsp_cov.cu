// bsp_cov.cu -- FP64 mean and covariance of the mocks' multipoles.
//
//   C[i][j] = sum_m (X[m][i] - mean[i]) (X[m][j] - mean[j]) / (M - 1).
//
// Two paths.  The direct one (k_cov) multiplies in FP64; GB300 has two FP64
// multiply-adds per SM and clock, so 512 x 4 962 values take 11.3 ms there and the
// unit is the bound.  With a workspace the products run on the tensor cores (the
// error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012):
//   * k_cov_split centres each column, scales it by the power of two 2^e above its
//     largest magnitude, rounds to a 63-bit integer and cuts that into eight
//     balanced base-256 digits (-128 .. 128), each exact in FP16;
//   * k_cov_tc forms the products of digits p and q, p + q < 8 (from 0), with
//     tcgen05.mma in FP32 accumulators, one per level p + q.  A level adds at most
//     8 x 128 products of at most 2^14 between drains, so every partial sum is an
//     integer up to 2^24: exact.  The levels are joined in 64-bit integers, divided by
//     M - 1 with a 64-bit reciprocal and rounded to FP64 once.
// What is lost per mock is at most 9.1 x 2^-64 of 2^(e_i + e_j) (the digit products
// left out 7.1, the two values' rounding 1 each): below 2^-58 of the product of the two
// columns' LARGEST magnitudes, whatever the values of that mock.  Where a column's
// values are mostly far below its largest one (an outlying mock) that could exceed the
// rounding of an FP64 sum, which is relative to the products themselves; columns whose
// values lie more than CV_GAP = 7 bits below the largest on (geometric) average are
// therefore multiplied directly, in k_cov_direct.  Up to there the digits are the more
// accurate ones entry by entry.  Against exact sums, largest error over the sum of the
// products' magnitudes, digits and direct: 512 Gaussian mocks 1.0e-16 and 1.7e-15, products of
// three Gaussians 1.1e-16 and 1.4e-15, two opposite outliers of 2^7 in each of
// 100 mocks 3.1e-16 and 1.2e-15 (seven-bit digits, before: 4.6e-14; outliers of 2^20: 7e-10,
// now direct).  So are columns that are not finite, or so large or small that a product
// could leave the normal range.
#include <cuda_runtime.h>

#include <algorithm>

#include "../../include/bsp.h"
#include "bsp_internal.h"
#include "bsp_ptx.h"

namespace bsp {

namespace {

__global__ void k_col_mean(const double* __restrict__ X, int m, int d, double* __restrict__ mean) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= d) return;
    double s = 0.0;
    for (int i = 0; i < m; ++i) s += X[(size_t)i * d + j];
    mean[j] = s / m;
}

// One 32 x 32 tile of the products in FP64, the 32 rows listed in ri (-1: none), columns
// from j0: 16 x 16 threads, 2 x 2 outputs each; fixed summation order.
struct CovTile {
    double A[16][33], B[16][33];
    int ri[32];
};
__device__ __forceinline__ void cov_tile(CovTile& S, const double* __restrict__ X, const double* __restrict__ mean, int m,
                                         int d, int j0, double (&acc)[2][2]) {
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    acc[0][0] = acc[0][1] = acc[1][0] = acc[1][1] = 0.0;
    for (int k0 = 0; k0 < m; k0 += 16) {
        for (int e = threadIdx.x; e < 16 * 32; e += 256) {
            const int kk = e / 32, c = e % 32, i = S.ri[c], k = k0 + kk;
            double a = 0.0, b = 0.0;
            if (k < m && i >= 0) a = X[(size_t)k * d + i] - mean[i];
            if (k < m && j0 + c < d) b = X[(size_t)k * d + j0 + c] - mean[j0 + c];
            S.A[kk][c] = a;
            S.B[kk][c] = b;
        }
        __syncthreads();
#pragma unroll 4
        for (int kk = 0; kk < 16; ++kk)
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int v = 0; v < 2; ++v) acc[u][v] = fma(S.A[kk][ty * 2 + u], S.B[kk][tx * 2 + v], acc[u][v]);
        __syncthreads();
    }
}

// Direct: the tiles of the upper triangle, mirrored.
__global__ void __launch_bounds__(256) k_cov(const double* __restrict__ X, const double* __restrict__ mean, int m,
                                             int d, double* __restrict__ C) {
    const int bi = blockIdx.y, bj = blockIdx.x;
    if (bj < bi) return;
    __shared__ CovTile S;
    if (threadIdx.x < 32) S.ri[threadIdx.x] = bi * 32 + (int)threadIdx.x < d ? bi * 32 + (int)threadIdx.x : -1;
    __syncthreads();
    double acc[2][2];
    cov_tile(S, X, mean, m, d, bj * 32, acc);
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    for (int u = 0; u < 2; ++u)
        for (int v = 0; v < 2; ++v) {
            const int i = S.ri[ty * 2 + u], j = bj * 32 + tx * 2 + v;
            if (i >= 0 && j < d) {
                const double c = acc[u][v] / (m - 1);
                C[(size_t)i * d + j] = c;
                C[(size_t)j * d + i] = c;
            }
        }
}

// The entries of the columns that the digits do not take, after k_cov_tc.  dmask: a bit
// per column, set for those (and past d), a word per 32 columns.  A few of them are
// gathered, 32 to a tile, against all columns; from half of all columns on, the tiles of
// the upper triangle that hold one, as k_cov (a mock that is not finite takes every column:
// 600 x 2 000 values 2.9 ms, the direct path alone 2.4; in the tiles of k_cov_tc, one
// thread an entry, 8.4 ms).
__global__ void __launch_bounds__(256) k_cov_direct(const double* __restrict__ X, const double* __restrict__ mean, int m,
                                                    int d, const uint32_t* __restrict__ dmask, double* __restrict__ C) {
    __shared__ CovTile S;
    __shared__ int total;
    const int nb = (d + 31) / 32, tid = threadIdx.x, lane = tid & 31;
    auto word = [&](int w) {   // direct columns of block w
        const int live = d - 32 * w;
        return w < nb ? dmask[w] & (live < 32 ? (1u << live) - 1u : ~0u) : 0u;
    };
    if (tid == 0) total = 0;
    __syncthreads();
    int n = 0;
    for (int w = tid; w < nb; w += 256) n += __popc(word(w));
    for (int o = 16; o; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
    if (lane == 0 && n) atomicAdd(&total, n);
    __syncthreads();
    n = total;
    if (n == 0) return;
    const bool all = n > d / 2;
    const int nr = all ? nb : (n + 31) / 32;
    for (long long t = blockIdx.x; t < (long long)nr * nb; t += gridDim.x) {
        const int r = (int)(t / nb), bj = (int)(t % nb);
        if (all && (bj < r || (word(r) | word(bj)) == 0u)) continue;
        if (tid < 32) {   // the tile's rows: block r, or direct columns 32 r .. 32 r + 31 in order
            S.ri[lane] = all && r * 32 + lane < d ? r * 32 + lane : -1;
            __syncwarp();
            for (int w0 = 0, before = 0; !all && w0 < nb && before < 32 * (r + 1); w0 += 32) {
                const uint32_t bits = word(w0 + lane);
                int upto = __popc(bits);
                for (int o = 1; o < 32; o <<= 1) {
                    const int x = __shfl_up_sync(0xffffffffu, upto, o);
                    if (lane >= o) upto += x;
                }
                int at = before + upto - __popc(bits) - 32 * r;
                for (uint32_t b = bits; b; b &= b - 1, ++at)
                    if (at >= 0 && at < 32) S.ri[at] = 32 * (w0 + lane) + __ffs((int)b) - 1;
                before += __shfl_sync(0xffffffffu, upto, 31);
            }
        }
        __syncthreads();
        double acc[2][2];
        cov_tile(S, X, mean, m, d, bj * 32, acc);
        const int tx = tid % 16, ty = tid / 16;
        for (int u = 0; u < 2; ++u)
            for (int v = 0; v < 2; ++v) {
                const int i = S.ri[ty * 2 + u], j = bj * 32 + tx * 2 + v;
                if (i < 0 || j >= d) continue;
                if (all && !((dmask[i >> 5] >> (i & 31) | dmask[j >> 5] >> (j & 31)) & 1u)) continue;
                const double c = acc[u][v] / (m - 1);
                C[(size_t)i * d + j] = c;
                C[(size_t)j * d + i] = c;
            }
        __syncthreads();   // before the next tile's rows
    }
}

constexpr int CV_S = 8;                    // digits
constexpr int CV_K = 32;                   // mocks per chunk: a 64-byte row of FP16 digits
constexpr int CV_GROUP = 4;                // chunks (128 mocks) between drains: sums stay within 2^24
constexpr int CV_GAP = 7;                  // bits below a column's largest value that its values may lie on average
constexpr int CV_TM = 128, CV_TN = 64;     // tile (MMA M x N)
constexpr int CV_EMAX = 400;               // |exponent| of a column that the digits take

// Layout of the digits: chunk kc, digit s, column j: 64 bytes at ((kc * 8 + s) * dp + j) * 64,
// 16-byte piece c (8 mocks) at piece c ^ ((j >> 1) & 3): the 64-byte swizzle of the
// tensor-core operand, so that plain copies give the shared-memory image.
// 1024 threads per 32 columns: sums, then the largest magnitude, then the digits;
// the strip (256 bytes a mock) is read three times, from L2 after the first.  89 us for
// 512 x 4 962 values, set by the FP64 unit (five operations a value) and latency.
__global__ void __launch_bounds__(1024) k_cov_split(const double* __restrict__ X, int m, int d, int dp, int nkc,
                                                    double* __restrict__ mean, int* __restrict__ ecol,
                                                    uint32_t* __restrict__ dmask, uint4* __restrict__ digits) {
    __shared__ double red[32][33];
    __shared__ double smean[32], sscale[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, j = blockIdx.x * 32 + lane;
    const bool live = j < d;
    const double* x = X + (live ? j : 0);
    double s = 0.0;
    if (live)
        for (int k = wid; k < m; k += 32) s += x[(size_t)k * d];
    red[wid][lane] = s;
    __syncthreads();
    if (wid == 0) {
        s = red[0][lane];
        for (int w = 1; w < 32; ++w) s += red[w][lane];
        smean[lane] = s / m;
        if (live) mean[j] = s / m;
    }
    __syncthreads();
    const double mu = smean[lane];
    // largest |x - mean| as bits (ordered like the values; infinities and NaN above all numbers)
    unsigned long long mx = 0;
    if (live)
        for (int k = wid; k < m; k += 32)
            mx = max(mx, (unsigned long long)__double_as_longlong(x[(size_t)k * d] - mu) & 0x7fffffffffffffffull);
    red[wid][lane] = __longlong_as_double((long long)mx);
    __syncthreads();
    if (wid == 0) {
        for (int w = 1; w < 32; ++w) mx = max(mx, (unsigned long long)__double_as_longlong(red[w][lane]));
        // 2^e above the largest magnitude: |x - mean| 2^(63 - e) < 2^63 (and 2^10 below it: 53 bits)
        const int ex = (int)(mx >> 52);
        int e = mx == 0 ? 0 : ex - 1022;
        const bool direct = mx != 0 && (ex == 0 || e < -CV_EMAX || e > CV_EMAX);
        if (direct) e = 0;
        sscale[lane] = direct ? 0.0 : __longlong_as_double((long long)(1023 + 63 - e) << 52);
        ecol[j] = e;
    }
    __syncthreads();
    const double sc = sscale[lane];
    int gap = 0, cnt = 0;   // bits that the values lie below the largest (up to 63), and how many are not 0
    for (int o = wid; o < nkc * (CV_K / 8); o += 32) {   // eight mocks of one column
        uint32_t q[CV_S][4];
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) {
            long long v[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int k = o * 8 + 2 * k2 + u;
                v[u] = 0;
                if (live && k < m && sc != 0.0) {
                    const double y = x[(size_t)k * d] - mu;
                    v[u] = __double2ll_rn(y * sc);
                    if (v[u] != 0 || (__double_as_longlong(y) << 1) != 0) {
                        gap += min(63, __clzll(llabs(v[u])) - 1);
                        ++cnt;
                    }
                }
            }
#pragma unroll
            for (int t = CV_S - 1; t >= 0; --t) {   // balanced digits, the lowest first; what is left is the top one
                int g[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    g[u] = t == 0 ? (int)v[u] : (int)((v[u] + 128) & 255) - 128;
                    v[u] = (v[u] - g[u]) >> 8;
                }
                asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(q[t][k2]) : "f"((float)g[1]), "f"((float)g[0]));
            }
        }
        const int kc = o >> 2, c = o & 3;
#pragma unroll
        for (int t = 0; t < CV_S; ++t)
            digits[((size_t)(kc * CV_S + t) * dp + j) * 4 + (c ^ ((j >> 1) & 3))] =
                make_uint4(q[t][0], q[t][1], q[t][2], q[t][3]);
    }
    red[wid][lane] = __hiloint2double(gap, cnt);   // the bits (red was last read before the barrier above)
    __syncthreads();
    if (wid == 0) {
        for (int w = 1; w < 32; ++w) {
            gap += __double2hiint(red[w][lane]);
            cnt += __double2loint(red[w][lane]);
        }
        const bool direct = sc == 0.0 || gap > (long long)CV_GAP * cnt;
        const uint32_t bits = __ballot_sync(0xffffffffu, direct || !live);
        if (lane == 0) dmask[blockIdx.x] = bits;
    }
}

struct CvSmem {
    uint8_t a[2][CV_S][CV_TM * 64];   // [stage][digit][row]
    uint8_t b[2][CV_S][CV_TN * 64];
    uint64_t full[2], empty[2], acc_full, acc_empty;
    uint32_t tmem_base;
    volatile int abort;
};

// K-major operand, 8-row x 64-byte atoms with the 64-byte swizzle, 512 bytes apart.
__device__ __forceinline__ uint64_t sw64_desc(uint32_t saddr) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | (uint64_t)1 << 16 | (uint64_t)(512 >> 4) << 32 | (uint64_t)1 << 46 |
           (uint64_t)4 << 61;
}
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

// 1 / (M - 1) as rec 2^-(63 + sh), rec in [2^63, 2^64).
struct CvRecip {
    unsigned long long rec;
    int sh;
};
CvRecip cov_recip(int m) {
    const unsigned long long q = (unsigned long long)m - 1;
    int sh = 0;
    while ((1ull << sh) < q) ++sh;
    return CvRecip{(unsigned long long)(((unsigned __int128)1 << (63 + sh)) / q), sh};
}

// (hi 2^32 + lo) 2^e / (M - 1) rounded to FP64 (nearest; the quotient is truncated to
// 63 bits or more before, 2^-10 of a last place); the result is a normal number or 0.
__device__ __forceinline__ double join_round(long long hi, long long lo, int e, CvRecip r) {
    const __int128 t = ((__int128)hi << 32) + lo;
    if (t == 0) return 0.0;
    const unsigned long long sign = t < 0 ? 0x8000000000000000ull : 0ull;
    const unsigned __int128 u = t < 0 ? (unsigned __int128)(-t) : (unsigned __int128)t;
    const unsigned long long uh = (unsigned long long)(u >> 64), ul = (unsigned long long)u;
    const int n = uh ? 127 - __clzll((long long)uh) : 63 - __clzll((long long)ul);   // top bit, up to 95
    const unsigned long long top = n > 63 ? (unsigned long long)(u >> (n - 63)) : ul << (63 - n);
    unsigned long long p = __umul64hi(top, r.rec);   // [2^62, 2^64): the value is p 2^(n - 62 - sh + e)
    const int s = (int)(~p >> 63);
    p <<= s;
    const unsigned long long rem = p & 2047;
    unsigned long long q = p >> 11;
    if (rem > 1024 || (rem == 1024 && (q & 1))) ++q;
    // q in [2^52, 2^53]: a carry out of the mantissa moves into the exponent
    return __longlong_as_double((long long)(sign | (((unsigned long long)(n + e - r.sh - s + 1023) << 52) + q)));
}

// One 128 x 64 tile per CTA: eight levels of 64 columns fill tensor memory, so A and B
// both come from shared memory, 96 KB for 32 mocks, two stages.  The MMAs read 6 KB
// of shared memory per 32 cycles of tensor work, which bounds them at 48; 572 us for
// 1 560 tiles of 512 mocks (52 us a tile, 27 us of that the MMAs' operand reads and four
// drains of ~2 us, which nothing overlaps).
constexpr int CV_THREADS = 320;   // warp 0 copies, warp 1 MMAs, warps 2 .. 9 drain (quadrant warp % 4, 32 columns each)

__global__ void __launch_bounds__(CV_THREADS, 1) k_cov_tc(const uint8_t* __restrict__ digits, int dp, int nkc,
                                                          const int* __restrict__ ecol,
                                                          const uint32_t* __restrict__ dmask, CvRecip recip, int d,
                                                          double* __restrict__ C, long long wlim) {
    extern __shared__ uint8_t cv_raw[];
    CvSmem& S = *reinterpret_cast<CvSmem*>((reinterpret_cast<uintptr_t>(cv_raw) + 1023) & ~(uintptr_t)1023);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // tiles (I, J) of 128 rows x 64 columns that reach the upper triangle: J >= 2 I
    const int nJ = (d + CV_TN - 1) / CV_TN;
    int I = 0, J = blockIdx.x;
    while (J >= nJ - 2 * I) {
        J -= nJ - 2 * I;
        ++I;
    }
    J += 2 * I;
    // no row or no column of the tile's is the digits': k_cov_direct has all of it
    if ((dmask[4 * I] & dmask[4 * I + 1] & dmask[4 * I + 2] & dmask[4 * I + 3]) == ~0u ||
        (dmask[2 * J] & dmask[2 * J + 1]) == ~0u)
        return;
    if (tid == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(&S.full[s], 1);
            mbar_init(&S.empty[s], 1);
        }
        mbar_init(&S.acc_full, 1);
        mbar_init(&S.acc_empty, 8);
        S.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem_base)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem_base;

    if (warp == 0) {
        if (lane == 0) {
            int issued = 0;
            for (int k = 0; k < nkc && !S.abort; ++k) {
                const int s = k & 1, u = k >> 1;
                if (u > 0 && !mbar_wait(&S.empty[s], (u - 1) & 1, wlim)) {
                    S.abort = 1;
                    break;
                }
                mbar_expect_tx(&S.full[s], CV_S * (CV_TM + CV_TN) * 64);
                for (int t = 0; t < CV_S; ++t) {
                    const uint8_t* src = digits + (size_t)(k * CV_S + t) * dp * 64;
                    bulk_load(S.a[s][t], src + (size_t)I * CV_TM * 64, CV_TM * 64, &S.full[s]);
                    bulk_load(S.b[s][t], src + (size_t)J * CV_TN * 64, CV_TN * 64, &S.full[s]);
                }
                issued = k + 1;
            }
            for (int k = max(0, issued - 2); k < issued; ++k)   // copies in flight land before the CTA ends (the long limit)
                if (!mbar_wait(&S.full[k & 1], (k >> 1) & 1)) S.abort = 1;
        }
    } else if (warp == 1) {
        // FP16 operands, FP32 accumulators, both K-major, M = 128, N = 64
        const uint32_t idesc = (1u << 4) | ((uint32_t)(CV_TN >> 3) << 17) | ((uint32_t)(CV_TM >> 4) << 24);
        int done = 0;
        for (int k = 0; k < nkc; ++k) {
            const int s = k & 1, g = k / CV_GROUP, kg = k % CV_GROUP;
            // the chunk's copies, and where it starts a group the accumulators read out: one barrier per lane
            const bool acc = kg == 0 && g > 0 && (lane & 1);
            if (!warp_wait<128>(smem_u32(acc ? &S.acc_empty : &S.full[s]), (uint32_t)((acc ? g - 1 : k >> 1) & 1), wlim, &S.abort)) {
                S.abort = 1;
                break;
            }
            tc_fence_after();
            if (elect_one()) {
                const uint64_t a0 = sw64_desc(smem_u32(S.a[s][0])), b0 = sw64_desc(smem_u32(S.b[s][0]));
#pragma unroll 1
                for (int p = 0; p < CV_S; ++p)
#pragma unroll 1
                    for (int q = 0; q < CV_S - p; ++q)
#pragma unroll
                        for (int kk = 0; kk < CV_K / 16; ++kk)
                            mma_ss(tmem + (uint32_t)(p + q) * CV_TN, a0 + (uint64_t)(p * (CV_TM * 64 / 16) + 2 * kk),
                                   b0 + (uint64_t)(q * (CV_TN * 64 / 16) + 2 * kk), idesc,
                                   kg == 0 && p == 0 && kk == 0 ? 0u : 1u);
                mma_commit(&S.empty[s]);
                if (kg == CV_GROUP - 1 || k == nkc - 1) mma_commit(&S.acc_full);
            }
            __syncwarp();
            done = k + 1;
        }
        // the last MMAs finish before tensor memory is released (the long limit)
        if (done > 0 && !warp_wait<1>(smem_u32(&S.empty[(done - 1) & 1]), (uint32_t)(((done - 1) >> 1) & 1), WAIT_CYCLES, nullptr)) S.abort = 1;
    } else {
        const int c0 = 32 * ((warp - 2) >> 2);
        const uint32_t lanebase = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + c0;
        long long hi[32], lo[32];   // levels 0 .. 3 and 4 .. 7, in units of 2^-38 and 2^-70
#pragma unroll
        for (int c = 0; c < 32; ++c) hi[c] = lo[c] = 0;
        const int ng = (nkc + CV_GROUP - 1) / CV_GROUP;
        // the whole warp waits and decides together: the loads of tensor memory below are .aligned
        bool bad = false;   // a wait gave up: no numbers
        for (int g = 0; g < ng; ++g) {
            if (!warp_wait<1>(smem_u32(&S.acc_full), (uint32_t)(g & 1), wlim, &S.abort)) {
                S.abort = 1;
                bad = true;
                break;
            }
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < 32; c += 4) {
                uint32_t r[CV_S][4];
#pragma unroll
                for (int t = 0; t < CV_S; ++t)
                    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(r[t][0]), "=r"(r[t][1]), "=r"(r[t][2]), "=r"(r[t][3])
                                 : "r"(lanebase + (uint32_t)(t * CV_TN + c)));
                // the registers pass through the wait, so that nothing reads them before it
#pragma unroll
                for (int t = 0; t < CV_S; ++t)
                    asm volatile("tcgen05.wait::ld.sync.aligned;"
                                 : "+r"(r[t][0]), "+r"(r[t][1]), "+r"(r[t][2]), "+r"(r[t][3])::"memory");
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    int v[CV_S];
#pragma unroll
                    for (int t = 0; t < CV_S; ++t) v[t] = __float2int_rn(__uint_as_float(r[t][u]));
                    hi[c + u] += ((((((long long)v[0] << 8) + v[1]) << 8) + v[2]) << 8) + v[3];
                    lo[c + u] += ((((((long long)v[4] << 8) + v[5]) << 8) + v[6]) << 8) + v[7];
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.acc_empty);
        }
        const int i = I * CV_TM + 32 * (warp & 3) + lane;
        const int ei = ecol[i];
        const uint32_t di = dmask[i >> 5] >> lane & 1u, dj = dmask[(J * CV_TN + c0) >> 5];   // direct (or past d)
        if (!bad) {
            double* stage = reinterpret_cast<double*>(S.a[0]) + (size_t)(warp - 2) * (32 * 33);   // the operands are used up
#pragma unroll
            for (int c = 0; c < 32; ++c) {
                const int j = J * CV_TN + c0 + c;
                double v = 0.0;
                if (!di && !(dj >> c & 1u) && j >= i) {
                    v = join_round(hi[c], lo[c], ei + ecol[j] - 70, recip);
                    C[(size_t)j * d + i] = v;   // lanes: consecutive i
                }
                stage[lane * 33 + c] = v;
            }
            __syncwarp();
            for (int r = 0; r < 32; ++r) {      // lanes: consecutive j
                const int ir = I * CV_TM + 32 * (warp & 3) + r, j = J * CV_TN + c0 + lane;
                if (!(__shfl_sync(0xffffffffu, di, r) | (dj >> lane & 1u)) && j > ir) C[(size_t)ir * d + j] = stage[r * 33 + lane];
            }
        } else {   // (copies may still land in shared memory: nothing passes through it)
            for (int c = 0; c < 32; ++c) {
                const int j = J * CV_TN + c0 + c;
                if (di || (dj >> c & 1u) || j < i) continue;
                C[(size_t)j * d + i] = C[(size_t)i * d + j] = __longlong_as_double(0x7ff8000000000000ll);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

struct CovLayout {
    int dp, nkc;
    size_t mask, digits, end;   // offsets: the columns' exponents at 0
};
CovLayout cov_layout(int m, int d) {
    CovLayout L{};
    L.dp = (d + CV_TM - 1) / CV_TM * CV_TM;
    L.nkc = (m + CV_K - 1) / CV_K;
    L.mask = (size_t)L.dp * sizeof(int);
    L.digits = (L.mask + (size_t)L.dp / 8 + 255) / 256 * 256;
    L.end = L.digits + (size_t)L.nkc * CV_S * L.dp * 64;
    return L;
}

// The tensor-core path from where it is the faster one.  The direct one takes 0.36 us
// per mock where its tiles fit the SMs at once (100 x 50 values: 47 us on both; 160 x
// 128: 66 against 50) and m d^2 / 1.1e6 us beyond (64 x 400: 51 against 39; 512 x 1 000:
// 747 against 99; 512 x 4 962: 11 329 against 666).  Not where few columns, padded to 128, would
// take far more digits than the matrix itself (16 x 128 bytes a mock; up to 1 GiB is let pass:
// 400 000 x 3 values), nor past 2^22 mocks, up to which the 64-bit level sums hold
// (2^40.4 a mock).
bool cov_use_tc(int m, int d) {
    if (m > (1 << 22) || !(m >= 100 || (double)m * d * d >= 1.0e7)) return false;
    const CovLayout L = cov_layout(m, d);
    return L.end <= (size_t)1 << 30 || L.dp <= 4ll * d;
}

// The digits' path; wlim: limit of the pipeline's waits in clock cycles (an entry of a tile
// whose wait runs out is NaN).
cudaError_t launch_cov_digits(int m, int d, const double* rows, double* mean, double* cov, void* ws, long long wlim,
                              cudaStream_t st) {
    const CovLayout L = cov_layout(m, d);
    int* ecol = (int*)ws;
    uint32_t* dmask = (uint32_t*)((char*)ws + L.mask);
    uint8_t* digits = (uint8_t*)ws + L.digits;
    const size_t smem = sizeof(CvSmem) + 1024;
    static SmemLimit limit;
    const cudaError_t e = raise_smem(limit, smem, k_cov_tc);
    if (e != cudaSuccess) return e;
    const int nJ = (d + CV_TN - 1) / CV_TN, nI = (d + CV_TM - 1) / CV_TM;
    int tiles = 0;
    for (int I = 0; I < nI; ++I) tiles += nJ - 2 * I;
    k_cov_split<<<L.dp / 32, 1024, 0, st>>>(rows, m, d, L.dp, L.nkc, mean, ecol, dmask, (uint4*)digits);
    k_cov_tc<<<tiles, CV_THREADS, smem, st>>>(digits, L.dp, L.nkc, ecol, dmask, cov_recip(m), d, cov, wlim);
    const long long nb = (d + 31) / 32;
    k_cov_direct<<<(int)std::min<long long>(nb * nb, 152 * 8), 256, 0, st>>>(rows, mean, m, d, dmask, cov);
    return cudaGetLastError();
}

}  // namespace

}  // namespace bsp

using namespace bsp;

extern "C" {

bsp_status bsp_covariance(int m, int d, const double* rows, double* mean, double* cov, void* stream) {
    if (m < 2 || d < 1 || !rows || !mean || !cov) return BSP_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    k_col_mean<<<(d + 255) / 256, 256, 0, st>>>(rows, m, d, mean);
    dim3 grid((d + 31) / 32, (d + 31) / 32);
    k_cov<<<grid, 256, 0, st>>>(rows, mean, m, d, cov);
    return cudaGetLastError() == cudaSuccess ? BSP_OK : BSP_ECUDA;
}

bsp_status bsp_covariance_workspace_size(int m, int d, size_t* bytes) {
    if (m < 2 || d < 1 || !bytes) return BSP_EINVAL;
    *bytes = cov_use_tc(m, d) ? cov_layout(m, d).end : 0;
    return BSP_OK;
}

bsp_status bsp_covariance_ws(int m, int d, const double* rows, double* mean, double* cov, void* ws, size_t ws_bytes,
                             void* stream) {
    if (m < 2 || d < 1 || !rows || !mean || !cov) return BSP_EINVAL;
    if (!cov_use_tc(m, d)) return bsp_covariance(m, d, rows, mean, cov, stream);
    if (!ws || ((uintptr_t)ws & 255u)) return BSP_EINVAL;
    if (ws_bytes < cov_layout(m, d).end) return BSP_ENOMEM;
    const cudaError_t e = launch_cov_digits(m, d, rows, mean, cov, ws, WAIT_CYCLES, (cudaStream_t)stream);
    return e == cudaSuccess ? BSP_OK : record_cuda_error(e, "covariance");
}

}  // extern "C"
