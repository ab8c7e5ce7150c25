// bsp_cov.cu -- FP64 mean and covariance of the mocks' multipoles.
//
//   C[i][j] = sum_m (X[m][i] - mean[i]) (X[m][j] - mean[j]) / (M - 1).
//
// Two paths.  The direct one (k_cov) multiplies in FP64; GB300 has two FP64
// multiply-adds per SM and clock, so 512 x 4 962 values take 11.3 ms there and the
// unit is the bound.  With a workspace the products run on the tensor cores
// without losing a bit of what FP64 would keep (the error-free splitting of
// Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012):
//   * k_cov_split centres each column, scales it by the power of two above its
//     largest magnitude, rounds to a 55-bit integer and cuts that into eight
//     balanced base-128 digits (-64 .. 64), each exact in FP16;
//   * k_cov_tc forms the products of digits p and q, p + q <= 9, with tcgen05.mma in
//     FP32 accumulators, one per level p + q.  A level adds at most 8 x 512 products
//     of at most 2^12, so every partial sum is an integer up to 2^24: exact.
//     The levels are joined in 64-bit integers and rounded to FP64 once.
// What is left out is below 2^-54 of the two columns' largest magnitudes per
// mock, less than the rounding of an FP64 product sum (the measured error against
// 64 bits is no larger than the direct path's).
// Columns that are not finite, or so large or small that a product could leave
// the normal range, are multiplied directly.
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

// Direct: 32 x 32 tiles, upper triangle computed and mirrored; fixed summation order.
__global__ void __launch_bounds__(256) k_cov(const double* __restrict__ X, const double* __restrict__ mean, int m,
                                             int d, double* __restrict__ C) {
    const int bi = blockIdx.y, bj = blockIdx.x;
    if (bj < bi) return;
    __shared__ double A[16][33], Bt[16][33];
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;   // 16 x 16 threads, 2 x 2 outputs each
    double acc[2][2] = {{0, 0}, {0, 0}};
    const int i0 = bi * 32, j0 = bj * 32;
    for (int k0 = 0; k0 < m; k0 += 16) {
        for (int e = threadIdx.x; e < 16 * 32; e += 256) {
            const int kk = e / 32, c = e % 32;
            const int k = k0 + kk;
            double a = 0.0, b = 0.0;
            if (k < m && i0 + c < d) a = X[(size_t)k * d + i0 + c] - mean[i0 + c];
            if (k < m && j0 + c < d) b = X[(size_t)k * d + j0 + c] - mean[j0 + c];
            A[kk][c] = a;
            Bt[kk][c] = b;
        }
        __syncthreads();
#pragma unroll 4
        for (int kk = 0; kk < 16; ++kk)
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int v = 0; v < 2; ++v) acc[u][v] = fma(A[kk][ty * 2 + u], Bt[kk][tx * 2 + v], acc[u][v]);
        __syncthreads();
    }
    for (int u = 0; u < 2; ++u)
        for (int v = 0; v < 2; ++v) {
            const int i = i0 + ty * 2 + u, j = j0 + tx * 2 + v;
            if (i < d && j < d) {
                const double c = acc[u][v] / (m - 1);
                C[(size_t)i * d + j] = c;
                C[(size_t)j * d + i] = c;
            }
        }
}

constexpr int CV_S = 8;                    // digits
constexpr int CV_K = 32;                   // mocks per chunk: a 64-byte row of FP16 digits
constexpr int CV_GROUP = 16;               // chunks (512 mocks) between drains: sums stay below 2^24
constexpr int CV_TM = 128, CV_TN = 64;     // tile (MMA M x N)
constexpr int CV_EMAX = 400;               // |exponent| of a column that the digits take
constexpr int CV_DIRECT = 1 << 20;         // "exponent" of a column that is multiplied directly

// Layout of the digits: chunk kc, digit s, column j: 64 bytes at ((kc * 8 + s) * dp + j) * 64,
// 16-byte piece c (8 mocks) at piece c ^ ((j >> 1) & 3): the 64-byte swizzle of the
// tensor-core operand, so that plain copies give the shared-memory image.
// 1024 threads per 32 columns: sums, then the largest magnitude, then the digits;
// the strip (256 bytes a mock) is read three times, from L2 after the first.  85 us for
// 512 x 4 962 values, set by the FP64 unit (five operations a value) and latency.
__global__ void __launch_bounds__(1024) k_cov_split(const double* __restrict__ X, int m, int d, int dp, int nkc,
                                                    double* __restrict__ mean, int* __restrict__ ecol,
                                                    uint4* __restrict__ digits) {
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
        // 2^e above the largest magnitude: |x - mean| 2^(55 - e) < 2^55
        const int ex = (int)(mx >> 52);
        int e = mx == 0 ? 0 : ex - 1022;
        const bool direct = mx != 0 && (ex == 0 || e < -CV_EMAX || e > CV_EMAX);
        if (direct) e = 0;
        sscale[lane] = direct ? 0.0 : __longlong_as_double((long long)(1023 + 55 - e) << 52);
        if (blockIdx.x * 32 + lane < dp) ecol[j] = direct ? CV_DIRECT : e;
    }
    __syncthreads();
    const double sc = sscale[lane];
    for (int o = wid; o < nkc * (CV_K / 8); o += 32) {   // eight mocks of one column
        uint32_t q[CV_S][4];
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) {
            long long v[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int k = o * 8 + 2 * k2 + u;
                v[u] = live && k < m && sc != 0.0 ? __double2ll_rn((x[(size_t)k * d] - mu) * sc) : 0ll;
            }
#pragma unroll
            for (int t = CV_S - 1; t >= 0; --t) {   // balanced digits, the lowest first; what is left is the top one
                int g[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    g[u] = t == 0 ? (int)v[u] : (int)((v[u] + 64) & 127) - 64;
                    v[u] = (v[u] - g[u]) >> 7;
                }
                asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(q[t][k2]) : "f"((float)g[1]), "f"((float)g[0]));
            }
        }
        const int kc = o >> 2, c = o & 3;
        if (j < dp)
#pragma unroll
            for (int t = 0; t < CV_S; ++t)
                digits[((size_t)(kc * CV_S + t) * dp + j) * 4 + (c ^ ((j >> 1) & 3))] =
                    make_uint4(q[t][0], q[t][1], q[t][2], q[t][3]);
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

// (hi 2^28 + lo) 2^e rounded to FP64 (nearest, ties to even); the result is a normal number or 0.
__device__ __forceinline__ double join_round(long long hi, long long lo, int e) {
    __int128 t = ((__int128)hi << 28) + lo;
    if (t == 0) return 0.0;
    const unsigned long long sign = t < 0 ? 0x8000000000000000ull : 0ull;
    const unsigned __int128 u = t < 0 ? (unsigned __int128)(-t) : (unsigned __int128)t;
    const unsigned long long uh = (unsigned long long)(u >> 64), ul = (unsigned long long)u;
    const int n = uh ? 127 - __clzll((long long)uh) : 63 - __clzll((long long)ul);   // top bit
    unsigned long long q;
    if (n <= 52) {
        q = ul << (52 - n);
    } else {
        const int s = n - 52;   // 1 .. 40
        q = (unsigned long long)(u >> s);
        const unsigned long long rem = ul & ((1ull << s) - 1), half = 1ull << (s - 1);
        if (rem > half || (rem == half && (q & 1))) ++q;
    }
    // q in [2^52, 2^53]: a carry out of the mantissa moves into the exponent
    return __longlong_as_double((long long)(sign | (((unsigned long long)(n + e + 1022) << 52) + q)));
}

// One 128 x 64 tile per CTA: eight levels of 64 columns fill tensor memory, so A and B
// both come from shared memory, 96 KB for 32 mocks, two stages.  The MMAs read 6 KB
// of shared memory per 32 cycles of tensor work, which bounds them at 48; 580 us for
// 1 560 tiles of 512 mocks (52 us a tile, 27 us of that the MMAs' operand reads).
constexpr int CV_THREADS = 320;   // warp 0 copies, warp 1 MMAs, warps 2 .. 9 drain (quadrant warp % 4, 32 columns each)

__global__ void __launch_bounds__(CV_THREADS, 1) k_cov_tc(const uint8_t* __restrict__ digits, int dp, int nkc,
                                                          const int* __restrict__ ecol, const double* __restrict__ X,
                                                          const double* __restrict__ mean, int m, int d,
                                                          double* __restrict__ C) {
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
                if (u > 0 && !mbar_wait(&S.empty[s], (u - 1) & 1)) {
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
            for (int k = max(0, issued - 2); k < issued; ++k)   // copies in flight land before the CTA ends
                if (!mbar_wait(&S.full[k & 1], (k >> 1) & 1)) S.abort = 1;
        }
    } else if (warp == 1) {
        // FP16 operands, FP32 accumulators, both K-major, M = 128, N = 64
        const uint32_t idesc = (1u << 4) | ((uint32_t)(CV_TN >> 3) << 17) | ((uint32_t)(CV_TM >> 4) << 24);
        int done = 0;
        for (int k = 0; k < nkc; ++k) {
            const int s = k & 1, g = k / CV_GROUP, kg = k % CV_GROUP;
            bool ok = kg != 0 || g == 0 || mbar_wait(&S.acc_empty, (g - 1) & 1);
            ok = ok && mbar_wait(&S.full[s], (k >> 1) & 1);
            if (!__all_sync(0xffffffffu, ok)) {
                S.abort = 1;
                break;
            }
            if (__shfl_sync(0xffffffffu, S.abort, 0)) break;
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
        if (done > 0 && !__all_sync(0xffffffffu, mbar_wait(&S.empty[(done - 1) & 1], ((done - 1) >> 1) & 1))) S.abort = 1;
    } else {
        const int c0 = 32 * ((warp - 2) >> 2);
        const uint32_t lanebase = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + c0;
        long long hi[32], lo[32];   // levels 2 .. 5 and 6 .. 9, in units of 2^-33 and 2^-61
#pragma unroll
        for (int c = 0; c < 32; ++c) hi[c] = lo[c] = 0;
        const int ng = (nkc + CV_GROUP - 1) / CV_GROUP;
        for (int g = 0; g < ng && !S.abort; ++g) {
            if (!mbar_wait(&S.acc_full, g & 1)) {
                S.abort = 1;
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
                    hi[c + u] += ((((((long long)v[0] << 7) + v[1]) << 7) + v[2]) << 7) + v[3];
                    lo[c + u] += ((((((long long)v[4] << 7) + v[5]) << 7) + v[6]) << 7) + v[7];
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.acc_empty);
        }
        const int i = I * CV_TM + 32 * (warp & 3) + lane;
        const double inv = 1.0 / (double)(m - 1);
        const int ei = i < d ? ecol[i] : 0;
        const bool bad = S.abort != 0;   // a wait gave up: no number
        double* stage = reinterpret_cast<double*>(S.a[0]) + (size_t)(warp - 2) * (32 * 33);   // the operands are used up
#pragma unroll
        for (int c = 0; c < 32; ++c) {
            const int j = J * CV_TN + c0 + c;
            double v = 0.0;
            if (i < d && j < d && j >= i) {
                const int ej = ecol[j];
                if (bad) {
                    v = __longlong_as_double(0x7ff8000000000000ll);
                } else if (ei == CV_DIRECT || ej == CV_DIRECT) {
                    for (int k = 0; k < m; ++k)
                        v = fma(X[(size_t)k * d + i] - mean[i], X[(size_t)k * d + j] - mean[j], v);
                    v /= (m - 1);
                } else {
                    v = join_round(hi[c], lo[c], ei + ej - 61) * inv;
                }
                C[(size_t)j * d + i] = v;   // lanes: consecutive i
            }
            stage[lane * 33 + c] = v;
        }
        __syncwarp();
        for (int r = 0; r < 32; ++r) {      // lanes: consecutive j
            const int ir = I * CV_TM + 32 * (warp & 3) + r, j = J * CV_TN + c0 + lane;
            if (ir < d && j < d && j > ir) C[(size_t)ir * d + j] = stage[r * 33 + lane];
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
    size_t digits, end;   // offsets: the columns' exponents at 0
};
CovLayout cov_layout(int m, int d) {
    CovLayout L{};
    L.dp = (d + CV_TM - 1) / CV_TM * CV_TM;
    L.nkc = (m + CV_K - 1) / CV_K;
    L.digits = ((size_t)L.dp * sizeof(int) + 255) / 256 * 256;
    L.end = L.digits + (size_t)L.nkc * CV_S * L.dp * 64;
    return L;
}

// The tensor-core path from where it is the faster one.  The direct one takes 0.36 us
// per mock where its tiles fit the SMs at once (100 x 50 values: 47 us on both; 160 x
// 128: 66 against 50) and m d^2 / 1.1e6 us beyond (64 x 400: 51 against 39; 512 x 1 000:
// 747 against 99; 512 x 4 962: 11 329 against 662).
bool cov_use_tc(int m, int d) { return m >= 100 || (double)m * d * d >= 1.0e7; }

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
    const CovLayout L = cov_layout(m, d);
    if (ws_bytes < L.end) return BSP_ENOMEM;
    cudaStream_t st = (cudaStream_t)stream;
    int* ecol = (int*)ws;
    uint8_t* digits = (uint8_t*)ws + L.digits;
    const size_t smem = sizeof(CvSmem) + 1024;
    static bool attr = false;   // once, never inside a graph capture
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_cov_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return record_cuda_error(e, "covariance");
        attr = true;
    }
    const int nJ = (d + CV_TN - 1) / CV_TN, nI = (d + CV_TM - 1) / CV_TM;
    int tiles = 0;
    for (int I = 0; I < nI; ++I) tiles += nJ - 2 * I;
    k_cov_split<<<L.dp / 32, 1024, 0, st>>>(rows, m, d, L.dp, L.nkc, mean, ecol, (uint4*)digits);
    k_cov_tc<<<tiles, CV_THREADS, smem, st>>>(digits, L.dp, L.nkc, ecol, rows, mean, m, d, cov);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? BSP_OK : record_cuda_error(e, "covariance");
}

}  // extern "C"
