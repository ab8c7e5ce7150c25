// bsp_contract.cu -- CUDA-core contraction of filtered fields and the FP64
// reduction / normalisation of its partial sums.
//
// The x-integral of Eq. Standard_ell_Estim (Sec. 3.1),
//   T^l[a; b, c] = sum_x F^l_a(x) F^0_b(x) F^0_c(x),
// is organised as a matrix product over x: rows r = (l, a), columns
// p = pairs (b, c), T[r][p] = sum_x A_r(x) P_p(x) with P_p = F^0_b F^0_c formed
// once per x and shared by the rows.  A CTA owns one work item (a set of pairs
// times a set of rows) and one contiguous x-segment, keeps its sums on chip and
// writes them once to its own FP64 slot.  FP32 sums run over at most 64 points;
// each such block sum is folded into a compensated (TwoSum hi + lo) FP32 pair, so
// the segment sum is accurate to ~eps times the block error.  The reduction
// sums the per-segment partials in a fixed order in FP64 (deterministic),
// then normalises: B = T / (V n^3 N_abc) or N_abc = rint(T / n^3).
#include <algorithm>

#include "bsp_internal.h"

namespace bsp {

namespace {

constexpr int CC_THREADS = 256;
constexpr int CC_ROWS = 64;
constexpr int CC_COLS = 64;
constexpr int CC_OUT = CC_ROWS * CC_COLS;

// FP64 contraction (the counts): a CTA owns a tile of <= 64 pairs times <= 64
// rows and one x-segment, 4 x 4 outputs per thread.
constexpr int F64_XC = 16;   // points staged per step
__global__ void __launch_bounds__(CC_THREADS) k_contract_f64(const double* __restrict__ rows,
                                                             const double* __restrict__ px, size_t fstride,
                                                             const Work* __restrict__ works,
                                                             const int2* __restrict__ pair_fields,
                                                             const int* __restrict__ row_fields, size_t npts,
                                                             size_t seg, double* __restrict__ partial) {
    constexpr int XC = F64_XC;
    constexpr int AS = CC_ROWS + 4;         // padded row strides (multiples of 16 bytes)
    constexpr int PS = CC_COLS + 4;
    __shared__ __align__(16) double As[XC][AS];
    __shared__ __align__(16) double Ps[XC][PS];
    __shared__ __align__(16) double Fz[64][XC];
    __shared__ int2 pf[CC_COLS];
    __shared__ int rf[CC_ROWS];

    const Work w = works[blockIdx.x];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ty = (warp & 1) * 8 + (lane >> 2);     // rows 4*ty .. 4*ty+3
    const int tx = (warp >> 1) * 4 + (lane & 3);     // cols 4*tx .. 4*tx+3
    for (int i = tid; i < CC_COLS; i += CC_THREADS) {
        int2 v = {-1, -1};
        if (i < w.npairs) {
            v = pair_fields[w.pair0 + i];
            v.x -= w.shell_lo;
            v.y -= w.shell_lo;
        }
        pf[i] = v;
    }
    for (int i = tid; i < CC_ROWS; i += CC_THREADS) rf[i] = i < w.nrows ? row_fields[w.rowbase + i] : -1;

    const size_t x_begin = (size_t)blockIdx.y * seg;
    const size_t x_end = min(npts, x_begin + seg);

    double acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
    __syncthreads();

    for (size_t x0 = x_begin; x0 < x_end; x0 += XC) {
        const int nx = (int)min((size_t)XC, x_end - x0);
        for (int e = tid; e < w.nshell * XC; e += CC_THREADS) {
            const int s = e / XC, x = e % XC;
            Fz[s][x] = x < nx ? px[(size_t)(w.shell_lo + s) * fstride + x0 + x] : 0.0;
        }
        for (int e = tid; e < CC_ROWS * XC; e += CC_THREADS) {
            const int r = e / XC, x = e % XC;
            const int f = rf[r];
            As[x][r] = (f >= 0 && x < nx) ? rows[(size_t)f * fstride + x0 + x] : 0.0;
        }
        __syncthreads();
        for (int e = tid; e < CC_COLS * XC; e += CC_THREADS) {
            const int p = e % CC_COLS, x = e / CC_COLS;
            const int2 bc = pf[p];
            Ps[x][p] = bc.x >= 0 ? Fz[bc.x][x] * Fz[bc.y][x] : 0.0;
        }
        __syncthreads();
#pragma unroll 4
        for (int x = 0; x < XC; ++x) {
            const double2 a0 = *reinterpret_cast<const double2*>(&As[x][ty * 4]);
            const double2 a1 = *reinterpret_cast<const double2*>(&As[x][ty * 4 + 2]);
            const double2 p0 = *reinterpret_cast<const double2*>(&Ps[x][tx * 4]);
            const double2 p1 = *reinterpret_cast<const double2*>(&Ps[x][tx * 4 + 2]);
            const double a[4] = {a0.x, a0.y, a1.x, a1.y}, p[4] = {p0.x, p0.y, p1.x, p1.y};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], p[j], acc[i][j]);
        }
        __syncthreads();
    }
    double* slot = partial + ((size_t)blockIdx.x * gridDim.y + blockIdx.y) * CC_OUT;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) slot[(size_t)(ty * 4 + i) * CC_COLS + tx * 4 + j] = acc[i][j];
}

// ---------------------------------------------------------------------------
// FP32 contraction.  A work item has 16 slots; a slot is one shell b with an
// octet of eight consecutive shells c and its own list of rows (l, a), those
// that can close a triangle with (b, c).  128 threads: a warp has four slots,
// lane = 8 x slot + row slot; a thread owns rows rs + 8 i (i < TR) times the eight
// pairs of its slot.  Per point it forms the eight products
// F_b F_c itself (they never pass through shared memory) and does 8 TR
// multiply-adds, two pairs per fma.rn.f32x2.  The fields of 32 points are
// staged by cp.async, two stages deep, in rows of 36 floats: a quarter warp
// reads eight consecutive rows (all 32 banks) or one pair-factor row (broadcast).
// Sums keep their order: 64 points of one output are one FP32 chain, folded
// into a compensated (TwoSum hi + lo) pair, so the split of the work does not
// show in the result beyond ~2^-48.  The pairs are touched once in 64 points and
// would take twice the registers of the sums: they live in tensor memory (the
// thread's own lane, 16 TR of its columns), which leaves room for 12 warps an SM.
//
// Bound: the FP32 pipe, 67 % busy with 12 warps (192^3, 32 shells), then shared
// memory (TR + 4.5 wavefronts per warp and point for 8 TR + 8 multiply-add slots a
// thread).  The kernel before this one -- tiles of 64 pairs x 64 rows, the products
// staged through shared memory, 4 x 4 scalar multiply-adds a thread -- was bound by
// those loads and its issue slots: shot noise on 256^3 (four contractions, 32
// shells) 138 -> 88 ms, 160^3 with 24 shells 4.45 -> 2.3 ms.
// ---------------------------------------------------------------------------
constexpr int OCT_THREADS = 8 * OCT_SLOTS;
constexpr int OCT_XS = 32;                         // points per stage
constexpr int OCT_RB = (OCT_XS + 4) * 4;           // bytes per staged row
// the most any work stages: 192 fields as rows, 8 octets and 16 shells b twice over
constexpr int OCT_SMEM_MAX = (192 + 2 * 80) * (2 * OCT_RB + 8);
constexpr uint32_t OCT_TMEM = 128;                 // tensor-memory columns: hi at 0, lo at 64
static_assert(8 * OCT_TRMAX <= 64, "hi and lo fit their columns");

__device__ __forceinline__ void cp_async16(void* dst, const void* src, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pk2(float a, float b) {
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ void unpk2(f32x2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float4 lds4(const char* p) { return *reinterpret_cast<const float4*>(p); }

// Eight columns each of hi and lo, of the calling warp's lanes: v[k] = columns 2 k, 2 k + 1.
__device__ __forceinline__ void tmem_ld8x2(uint32_t ah, uint32_t al, f32x2 (&h)[4], f32x2 (&l)[4]) {
    uint32_t r[8], s[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(ah));
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(s[0]), "=r"(s[1]), "=r"(s[2]), "=r"(s[3]), "=r"(s[4]), "=r"(s[5]), "=r"(s[6]), "=r"(s[7])
                 : "r"(al));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(s[0]), "+r"(s[1]), "+r"(s[2]), "+r"(s[3]), "+r"(s[4]), "+r"(s[5]), "+r"(s[6]), "+r"(s[7])
                 ::"memory");
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        h[k] = pk2(__uint_as_float(r[2 * k]), __uint_as_float(r[2 * k + 1]));
        l[k] = pk2(__uint_as_float(s[2 * k]), __uint_as_float(s[2 * k + 1]));
    }
}
__device__ __forceinline__ void tmem_st8(uint32_t addr, const f32x2 (&v)[4]) {
    float f[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) unpk2(v[k], f[2 * k], f[2 * k + 1]);
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(addr), "f"(f[0]),
                 "f"(f[1]), "f"(f[2]), "f"(f[3]), "f"(f[4]), "f"(f[5]), "f"(f[6]), "f"(f[7])
                 : "memory");
}
template <bool SYM, int TR>
__device__ __forceinline__ void oct_body(char* sm, const float* const* src, int nrow, uint32_t stage_bytes, uint32_t tmem,
                                         const OctWork* __restrict__ w, size_t npts, size_t seg,
                                         double* __restrict__ partial) {
    const int tid = threadIdx.x, lane = tid & 31, oct = 4 * (tid >> 5) + (lane >> 3), rs = lane & 7;
    const size_t x_begin = (size_t)blockIdx.y * seg;
    const size_t x_end = min(npts, x_begin + seg);
    const int nst = x_end > x_begin ? (int)((x_end - x_begin + OCT_XS - 1) / OCT_XS) : 0;
    uint32_t ao[TR];
#pragma unroll
    for (int i = 0; i < TR; ++i) ao[i] = (uint32_t)w->arow[oct][rs + 8 * i] * OCT_RB;
    const uint32_t bo = (uint32_t)(w->nA + w->brow[oct]) * OCT_RB, co = (uint32_t)(w->nA + w->crow[oct]) * OCT_RB;
    const uint32_t yo = SYM ? (uint32_t)w->nX * OCT_RB : 0u;   // Y rows follow the X rows
    const uint32_t tm = tmem + ((uint32_t)(tid & 96) << 16);   // this warp's lane quadrant

    // stage s -> buffer b: 16-byte chunk ch of every staged row, zero-filled past x_end
    const int ch = tid & 7;
    auto load = [&](int st, int b) {
        const size_t x = x_begin + (size_t)st * OCT_XS + 4 * ch;
        const int bytes = x < x_end ? (int)min((size_t)4, x_end - x) * 4 : 0;
        char* dst = sm + (uint32_t)b * stage_bytes + 16 * ch;
        for (int r = tid >> 3; r < nrow; r += OCT_THREADS / 8) cp_async16(dst + r * OCT_RB, src[r] + (bytes ? x : 0), bytes);
    };

    f32x2 acc[TR][4];
#pragma unroll
    for (int i = 0; i < TR; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
    if (nst > 0) load(0, 0);
    cp_async_commit();
    for (int st = 0; st < nst; ++st) {
        cp_async_wait<0>();
        __syncthreads();   // stage st has landed, and everyone is done with the other buffer
        if (st + 1 < nst) load(st + 1, (st + 1) & 1);
        cp_async_commit();
        const char* s = sm + (uint32_t)(st & 1) * stage_bytes;
#pragma unroll 1
        for (int x = 0; x < OCT_XS * 4; x += 16) {
            f32x2 p[4][4];   // [point][pair of pairs]
            const float4 b = lds4(s + bo + x);
            float4 yb;
            if (SYM) yb = lds4(s + bo + yo + x);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 c0 = lds4(s + co + (2 * j) * OCT_RB + (SYM ? yo : 0u) + x);
                const float4 c1 = lds4(s + co + (2 * j + 1) * OCT_RB + (SYM ? yo : 0u) + x);
                if (SYM) {
                    const float4 d0 = lds4(s + co + (2 * j) * OCT_RB + x), d1 = lds4(s + co + (2 * j + 1) * OCT_RB + x);
                    p[0][j] = pk2(fmaf(yb.x, d0.x, b.x * c0.x), fmaf(yb.x, d1.x, b.x * c1.x));
                    p[1][j] = pk2(fmaf(yb.y, d0.y, b.y * c0.y), fmaf(yb.y, d1.y, b.y * c1.y));
                    p[2][j] = pk2(fmaf(yb.z, d0.z, b.z * c0.z), fmaf(yb.z, d1.z, b.z * c1.z));
                    p[3][j] = pk2(fmaf(yb.w, d0.w, b.w * c0.w), fmaf(yb.w, d1.w, b.w * c1.w));
                } else {
                    p[0][j] = pk2(b.x * c0.x, b.x * c1.x);
                    p[1][j] = pk2(b.y * c0.y, b.y * c1.y);
                    p[2][j] = pk2(b.z * c0.z, b.z * c1.z);
                    p[3][j] = pk2(b.w * c0.w, b.w * c1.w);
                }
            }
#pragma unroll
            for (int i = 0; i < TR; ++i) {
                const float4 a = lds4(s + ao[i] + x);
                const f32x2 a0 = pk2(a.x, a.x), a1 = pk2(a.y, a.y), a2 = pk2(a.z, a.z), a3 = pk2(a.w, a.w);
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma2(a0, p[0][j], acc[i][j]);
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma2(a1, p[1][j], acc[i][j]);
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma2(a2, p[2][j], acc[i][j]);
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma2(a3, p[3][j], acc[i][j]);
            }
        }
        if (st & 1) {   // every 64 points: fold the block sums into the compensated pairs (TwoSum)
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");   // the last fold's stores
#pragma unroll
            for (int i = 0; i < TR; ++i) {
                f32x2 h[4] = {0ull, 0ull, 0ull, 0ull}, l[4] = {0ull, 0ull, 0ull, 0ull};
                if (st > 1) tmem_ld8x2(tm + 8u * i, tm + 64u + 8u * i, h, l);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const f32x2 v = acc[i][j], t = add2(h[j], v), bb = sub2(t, h[j]);
                    l[j] = add2(l[j], add2(sub2(h[j], sub2(t, bb)), sub2(v, bb)));
                    h[j] = t;
                    acc[i][j] = 0ull;
                }
                tmem_st8(tm + 8u * i, h);
                tmem_st8(tm + 64u + 8u * i, l);
            }
        }
    }
    cp_async_wait<0>();
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    double* slot = partial + ((size_t)blockIdx.x * gridDim.y + blockIdx.y) * (OCT_ROWS * OCT_COLS) + oct * 8;
#pragma unroll
    for (int i = 0; i < TR; ++i) {
        f32x2 h[4] = {0ull, 0ull, 0ull, 0ull}, l[4] = {0ull, 0ull, 0ull, 0ull};
        if (nst > 1) tmem_ld8x2(tm + 8u * i, tm + 64u + 8u * i, h, l);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float a0, a1, h0, h1, l0, l1;
            unpk2(acc[i][j], a0, a1);
            unpk2(h[j], h0, h1);
            unpk2(l[j], l0, l1);
            double2 d;
            d.x = (double)a0 + (double)h0 + (double)l0;
            d.y = (double)a1 + (double)h1 + (double)l1;
            *reinterpret_cast<double2*>(slot + (size_t)(rs + 8 * i) * OCT_COLS + 2 * j) = d;
        }
    }
}

template <bool SYM>
__global__ void __launch_bounds__(OCT_THREADS, 3) k_contract_oct(const float* __restrict__ rows,
                                                                 const float* __restrict__ px,
                                                                 const float* __restrict__ py, size_t fstride,
                                                                 const OctWork* __restrict__ works,
                                                                 const int* __restrict__ stage, uint32_t stage_bytes,
                                                                 size_t npts, size_t seg, double* __restrict__ partial) {
    extern __shared__ __align__(16) char oct_smem[];
    __shared__ uint32_t tmem_base;
    const OctWork* w = works + blockIdx.x;
    const float** src = reinterpret_cast<const float**>(oct_smem + 2 * stage_bytes);   // staged rows in global memory
    const int nA = w->nA, nX = w->nX, nrow = nA + (SYM ? 2 : 1) * nX;
    for (int r = threadIdx.x; r < nrow; r += OCT_THREADS) {
        const int k = r < nA + nX ? r : r - nX;
        src[r] = (r < nA ? rows : r < nA + nX ? px : py) + (size_t)stage[w->stage0 + k] * fstride;
    }
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(&tmem_base)),
                     "r"(OCT_TMEM)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tm = tmem_base;
    switch (w->tr) {   // uniform over the CTA
        case 1: oct_body<SYM, 1>(oct_smem, src, nrow, stage_bytes, tm, w, npts, seg, partial); break;
        case 2: oct_body<SYM, 2>(oct_smem, src, nrow, stage_bytes, tm, w, npts, seg, partial); break;
        case 3: oct_body<SYM, 3>(oct_smem, src, nrow, stage_bytes, tm, w, npts, seg, partial); break;
        case 4: oct_body<SYM, 4>(oct_smem, src, nrow, stage_bytes, tm, w, npts, seg, partial); break;
        case 5: oct_body<SYM, 5>(oct_smem, src, nrow, stage_bytes, tm, w, npts, seg, partial); break;
        case 6: oct_body<SYM, 6>(oct_smem, src, nrow, stage_bytes, tm, w, npts, seg, partial); break;
        default: oct_body<SYM, 7>(oct_smem, src, nrow, stage_bytes, tm, w, npts, seg, partial); break;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm), "r"(OCT_TMEM) : "memory");
    }
}

// One output per lane; the eight warps of a CTA sum every eighth partial each,
// then their sums in order (fixed order on every run).  A thread per output
// walking all partials alone took 9 to 60 us (58 us for 410 segments).
constexpr int RED_WARPS = 8;
__global__ void __launch_bounds__(32 * RED_WARPS) k_reduce(
    const double* __restrict__ partial, int nsplit, size_t unit, int row_stride, const BinLoc* __restrict__ loc,
    int nout, int nbins, const double* __restrict__ counts, double scale, int mode, double* __restrict__ T_out,
    double* __restrict__ out, ShotTerms shot, const int* __restrict__ err) {
    __shared__ double red[4][RED_WARPS][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    const int nset = 1 + shot.n;
    // the contraction's error word: after a wait that gave up, slots may hold an earlier call's sums
    const bool gave_up = err != nullptr && *err != 0;
    if (i < nout) {
        const BinLoc L = loc[i];
        // nsplit > 0: slots work*nsplit .. +nsplit; else slots L.work .. L.work + L.pad
        const int nsum = nsplit > 0 ? nsplit : L.pad;
        const size_t off = (size_t)L.work * (nsplit > 0 ? nsplit : 1) * unit + (size_t)L.row * row_stride + L.col;
        for (int t = 0; t < nset; ++t) {
            const double* q = (t == 0 ? partial : shot.partial[t - 1]) + off;
            double s = 0.0;
#pragma unroll 4
            for (int k = wid; k < nsum; k += RED_WARPS) s += q[(size_t)k * unit];
            red[t][wid][lane] = s;
        }
    }
    __syncthreads();
    if (wid != 0 || i >= nout) return;
    double u[4];
    for (int t = 0; t < nset; ++t) {
        u[t] = red[t][0][lane];
        for (int k = 1; k < RED_WARPS; ++k) u[t] += red[t][k][lane];
    }
    if (gave_up) u[0] = __longlong_as_double(0x7ff8000000000000ll);
    if (T_out) T_out[i] = u[0];
    if (mode == 0) {
        out[i] = rint(u[0] * scale);
        return;
    }
    double v = u[0] * scale;
    if (mode == 2) {   // raw sums, scaled
        out[i] = v;
        return;
    }
    for (int t = 0; t < shot.n; ++t) v -= shot.coef[t] * u[1 + t];   // the shot-noise contractions
    out[i] = v / counts[i % nbins];
}

// Unit fields on the orbit representatives: w_r I_a(x_r) and I_a(x_r) for
// every shell a (grid-stride over a * nrep + r).
__global__ void k_gather_reps(const double* __restrict__ fields, size_t npts, int nsh,
                              const uint32_t* __restrict__ idx, const double* __restrict__ w, size_t nrep,
                              double* __restrict__ wrows, double* __restrict__ urows) {
    const size_t total = (size_t)nsh * nrep;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const size_t a = i / nrep, r = i - a * nrep;
        const double v = fields[a * npts + idx[r]];
        urows[i] = v;
        wrows[i] = v * w[r];
    }
}

}  // namespace

cudaError_t launch_gather_reps(const double* fields, size_t npts, int nsh, const uint32_t* idx, const double* w,
                               size_t nrep, double* wrows, double* urows, cudaStream_t st) {
    if (nsh <= 0 || nrep == 0) return cudaSuccess;
    const size_t total = (size_t)nsh * nrep;
    const unsigned blocks = (unsigned)std::min<size_t>((total + 255) / 256, 152 * 16);
    k_gather_reps<<<blocks, 256, 0, st>>>(fields, npts, nsh, idx, w, nrep, wrows, urows);
    return cudaGetLastError();
}

cudaError_t launch_contract_f64(const double* rows, const double* pf, size_t fstride, const Work* works, int nwork,
                                const int2* pair_fields, const int* row_fields, size_t npts, int nsplit,
                                double* partial, cudaStream_t st) {
    size_t seg = (npts + nsplit - 1) / nsplit;
    seg = (seg + F64_XC - 1) / F64_XC * F64_XC;
    k_contract_f64<<<dim3(nwork, nsplit), CC_THREADS, 0, st>>>(rows, pf, fstride, works, pair_fields, row_fields, npts,
                                                               seg, partial);
    return cudaGetLastError();
}

cudaError_t launch_contract_oct(const float* rows, const float* px, const float* py, int sym, size_t fstride,
                                const OctWork* works, int nwork, const int* stage, int max_a, int max_x, size_t npts,
                                int nsplit, double* partial, cudaStream_t st) {
    size_t seg = (npts + nsplit - 1) / nsplit;
    seg = (seg + 2 * OCT_XS - 1) / (2 * OCT_XS) * (2 * OCT_XS);   // whole 64-point blocks
    const int nrow = max_a + (sym ? 2 : 1) * max_x;
    const uint32_t stage_bytes = (uint32_t)nrow * OCT_RB;
    const size_t smem = 2 * (size_t)stage_bytes + (size_t)nrow * sizeof(float*);
    static SmemLimit limit[2];
    auto kern = sym ? k_contract_oct<true> : k_contract_oct<false>;
    const cudaError_t e = raise_smem(limit[sym != 0], OCT_SMEM_MAX, kern);
    if (e != cudaSuccess) return e;
    kern<<<dim3(nwork, nsplit), OCT_THREADS, smem, st>>>(rows, px, py, fstride, works, stage, stage_bytes, npts, seg,
                                                         partial);
    return cudaGetLastError();
}

cudaError_t launch_reduce(const double* partial, int nsplit, size_t unit, int row_stride, const BinLoc* loc,
                          int nout, int nbins, const double* counts, double scale, int mode, double* T_out,
                          double* out, cudaStream_t st, const ShotTerms* shot, const int* err) {
    ShotTerms none{};
    none.n = 0;
    if (nout <= 0) return cudaSuccess;
    if (unit == 0) unit = CC_OUT;
    if (row_stride == 0) row_stride = CC_COLS;
    k_reduce<<<(nout + 31) / 32, 32 * RED_WARPS, 0, st>>>(partial, nsplit, unit, row_stride, loc, nout, nbins, counts, scale,
                                                          mode, T_out, out, shot ? *shot : none, err);
    return cudaGetLastError();
}

}  // namespace bsp
