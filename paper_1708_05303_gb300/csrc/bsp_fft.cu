// bsp_fft.cu -- shell/Legendre filter fused into a pruned, batched inverse
// 3-D FFT (complex along x, complex along y, complex-to-real along z).
//
// Computes, for each requested field f (Sec. 3.1: the filtered real-space
// fields D^{(l)}_k(x) = int_k d^3q e^{iq.x} delta^{(l)}(q) under
// Eq. Standard_ell_Estim; Sec. 3.5: M^{(l)}_n(x) of Eq. betaEst),
//
//   F_f(x) = sum_n W_f(n) S_f(n) e^{+2 pi i n.x / N},
//   W_f(n) = w_l(mu) x {1[n in shell] | R_p[|n|^2]},  w_l = (2l+1) L_l,
//   S_f(n) = delta(n) | 1 | |delta(n)|^2,
//
// over the Hermitian half spectrum delta[N][N][N/2+1].  No 1/N^3 factor.
//
// Pruning: all weights vanish for |n| >= the last shell edge, so only
// frequencies |f| <= K on x and y and 0 <= f_z < nKz are carried:
//   pass 1: per (f_y, f_z) pencil, filter + inverse DFT along x
//           -> T1[f_y (compact)][x][f_z]
//   pass 2: per (x, f_z) pencil, inverse DFT along y -> T2[x][y][f_z]
//   pass 3: per (x, y) pencil, real inverse DFT along z -> F[x][y][z]
// Each CTA holds a few lines side by side, so global reads and writes are
// contiguous runs: n = 512 in registers (k_pass1r, k_pass2r), the z pass of every
// compile-time size likewise (k_pass3v), the rest as mixed-radix stages through
// shared memory whose first and last stage touch global memory directly (k_col1,
// k_col2, k_pass3g); FP64 (the unit fields of the counts) as Stockham stages on
// batches of lines (k_pass1, k_pass2, k_pass3).  T1 and T2 rows are padded to 64 bytes.  Twiddles come from a
// host table of exp(+2 pi i t/N) computed in FP64.
#include <algorithm>
#include <type_traits>

#include "bsp_cic.h"
#include "bsp_internal.h"

namespace bsp {

namespace {

constexpr int NTHR = 256;

template <typename R>
__device__ __forceinline__ cx<R> cmul(cx<R> a, cx<R> b) {
    return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
template <typename R>
__device__ __forceinline__ cx<R> cadd(cx<R> a, cx<R> b) { return {a.re + b.re, a.im + b.im}; }
template <typename R>
__device__ __forceinline__ cx<R> csub(cx<R> a, cx<R> b) { return {a.re - b.re, a.im - b.im}; }
template <typename R>
__device__ __forceinline__ cx<R> cmuli(cx<R> a) { return {-a.im, a.re}; }   // i * a
template <typename R>
__device__ __forceinline__ cx<R> cscale(cx<R> a, R s) { return {a.re * s, a.im * s}; }

// Inverse (sign +1) DFT of RADIX values in registers: y_q = sum_r v_r e^{+2 pi i r q / RADIX}.
template <typename R, int RADIX>
__device__ __forceinline__ void butterfly(cx<R>* v) {
    if constexpr (RADIX == 2) {
        cx<R> a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    } else if constexpr (RADIX == 4) {
        cx<R> s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]);
        cx<R> s13 = cadd(v[1], v[3]), d13 = cmuli(csub(v[1], v[3]));
        v[0] = cadd(s02, s13);
        v[2] = csub(s02, s13);
        v[1] = cadd(d02, d13);
        v[3] = csub(d02, d13);
    } else if constexpr (RADIX == 8) {
        cx<R> e[4] = {v[0], v[2], v[4], v[6]};
        cx<R> o[4] = {v[1], v[3], v[5], v[7]};
        butterfly<R, 4>(e);
        butterfly<R, 4>(o);
        const R h = (R)0.70710678118654752440;   // 1/sqrt(2)
        cx<R> w1o = {(o[1].re - o[1].im) * h, (o[1].re + o[1].im) * h};     // e^{i pi/4} o1
        cx<R> w2o = cmuli(o[2]);                                             // e^{i pi/2} o2
        cx<R> w3o = {-(o[3].re + o[3].im) * h, (o[3].re - o[3].im) * h};    // e^{3i pi/4} o3
        v[0] = cadd(e[0], o[0]);
        v[4] = csub(e[0], o[0]);
        v[1] = cadd(e[1], w1o);
        v[5] = csub(e[1], w1o);
        v[2] = cadd(e[2], w2o);
        v[6] = csub(e[2], w2o);
        v[3] = cadd(e[3], w3o);
        v[7] = csub(e[3], w3o);
    } else if constexpr (RADIX == 16) {
        // 16 = 4 x 4: X[k1 + 4 k2] = sum_j2 W4^{j2 k2} W16^{j2 k1} sum_j1 x[j2 + 4 j1] W4^{j1 k1}
        const R c1 = (R)0.92387953251128675613, s1 = (R)0.38268343236508977173;   // cos, sin 2pi/16
        const R h = (R)0.70710678118654752440;
        const cx<R> w[10] = {{(R)1, (R)0}, {c1, s1}, {h, h}, {s1, c1}, {(R)0, (R)1},
                             {-s1, c1}, {-h, h}, {-c1, s1}, {(R)-1, (R)0}, {-c1, -s1}};   // W16^m, m = 0..9
        cx<R> a[4][4];
#pragma unroll
        for (int j2 = 0; j2 < 4; ++j2) {
            cx<R> t[4] = {v[j2], v[j2 + 4], v[j2 + 8], v[j2 + 12]};
            butterfly<R, 4>(t);
#pragma unroll
            for (int k1 = 0; k1 < 4; ++k1) a[j2][k1] = (j2 * k1 == 0) ? t[k1] : cmul(t[k1], w[j2 * k1]);
        }
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            cx<R> u[4] = {a[0][k1], a[1][k1], a[2][k1], a[3][k1]};
            butterfly<R, 4>(u);
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = u[k2];
        }
    } else if constexpr (RADIX == 3) {
        const R s3 = (R)0.86602540378443864676;  // sqrt(3)/2
        cx<R> t = cadd(v[1], v[2]), d = csub(v[1], v[2]);
        cx<R> m = {v[0].re - (R)0.5 * t.re, v[0].im - (R)0.5 * t.im};
        cx<R> id = cmuli(cscale(d, s3));
        v[0] = cadd(v[0], t);
        v[1] = cadd(m, id);
        v[2] = csub(m, id);
    } else if constexpr (RADIX == 5) {
        const R c1 = (R)0.30901699437494742410, c2 = (R)-0.80901699437494742410;   // cos 2pi/5, cos 4pi/5
        const R s1 = (R)0.95105651629515357212, s2 = (R)0.58778525229247312917;    // sin 2pi/5, sin 4pi/5
        cx<R> t1 = cadd(v[1], v[4]), d1 = csub(v[1], v[4]);
        cx<R> t2 = cadd(v[2], v[3]), d2 = csub(v[2], v[3]);
        cx<R> a1 = {v[0].re + c1 * t1.re + c2 * t2.re, v[0].im + c1 * t1.im + c2 * t2.im};
        cx<R> a2 = {v[0].re + c2 * t1.re + c1 * t2.re, v[0].im + c2 * t1.im + c1 * t2.im};
        cx<R> b1 = cmuli(cx<R>{s1 * d1.re + s2 * d2.re, s1 * d1.im + s2 * d2.im});
        cx<R> b2 = cmuli(cx<R>{s2 * d1.re - s1 * d2.re, s2 * d1.im - s1 * d2.im});
        v[0] = cadd(v[0], cadd(t1, t2));
        v[1] = cadd(a1, b1);
        v[4] = csub(a1, b1);
        v[2] = cadd(a2, b2);
        v[3] = csub(a2, b2);
    }
}

// FP32 arithmetic with every rounding written out.  Which product of a sum the
// multiply-add takes is a choice of the compiler's that changes with the code
// around it (by 1e-7 of a field); here it is fixed, so a transform has the same
// bits whatever kernel it runs in.
__device__ __forceinline__ cx<float> radd(cx<float> a, cx<float> b) { return {__fadd_rn(a.re, b.re), __fadd_rn(a.im, b.im)}; }
__device__ __forceinline__ cx<float> rsub(cx<float> a, cx<float> b) { return {__fsub_rn(a.re, b.re), __fsub_rn(a.im, b.im)}; }
__device__ __forceinline__ cx<float> rmul(cx<float> a, cx<float> b) {
    return {__fmaf_rn(a.re, b.re, -__fmul_rn(a.im, b.im)), __fmaf_rn(a.im, b.re, __fmul_rn(a.re, b.im))};
}
// Inverse DFT of RADIX values in registers (as butterfly).
template <int RADIX>
__device__ __forceinline__ void dft(cx<float>* v) {
    if constexpr (RADIX == 2) {
        const cx<float> a = v[0], b = v[1];
        v[0] = radd(a, b);
        v[1] = rsub(a, b);
    } else if constexpr (RADIX == 4) {
        const cx<float> s02 = radd(v[0], v[2]), d02 = rsub(v[0], v[2]), s13 = radd(v[1], v[3]), d = rsub(v[1], v[3]);
        const cx<float> d13 = {-d.im, d.re};
        v[0] = radd(s02, s13);
        v[2] = rsub(s02, s13);
        v[1] = radd(d02, d13);
        v[3] = rsub(d02, d13);
    } else if constexpr (RADIX == 8) {
        cx<float> e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
        dft<4>(e);
        dft<4>(o);
        const float h = 0.70710678118654752440f;
        const cx<float> u1 = {__fsub_rn(o[1].re, o[1].im), __fadd_rn(o[1].re, o[1].im)};
        const cx<float> u3 = {-__fadd_rn(o[3].re, o[3].im), __fsub_rn(o[3].re, o[3].im)};
        const cx<float> w2o = {-o[2].im, o[2].re};
        v[0] = radd(e[0], o[0]);
        v[4] = rsub(e[0], o[0]);
        v[1] = {__fmaf_rn(u1.re, h, e[1].re), __fmaf_rn(u1.im, h, e[1].im)};
        v[5] = {__fmaf_rn(-u1.re, h, e[1].re), __fmaf_rn(-u1.im, h, e[1].im)};
        v[2] = radd(e[2], w2o);
        v[6] = rsub(e[2], w2o);
        v[3] = {__fmaf_rn(u3.re, h, e[3].re), __fmaf_rn(u3.im, h, e[3].im)};
        v[7] = {__fmaf_rn(-u3.re, h, e[3].re), __fmaf_rn(-u3.im, h, e[3].im)};
    } else if constexpr (RADIX == 16) {
        const float c1 = 0.92387953251128675613f, s1 = 0.38268343236508977173f, h = 0.70710678118654752440f;
        const cx<float> w[10] = {{1.f, 0.f}, {c1, s1}, {h, h}, {s1, c1}, {0.f, 1.f}, {-s1, c1}, {-h, h}, {-c1, s1}, {-1.f, 0.f}, {-c1, -s1}};
        cx<float> a[4][4];
#pragma unroll
        for (int j2 = 0; j2 < 4; ++j2) {
            cx<float> t[4] = {v[j2], v[j2 + 4], v[j2 + 8], v[j2 + 12]};
            dft<4>(t);
#pragma unroll
            for (int k1 = 0; k1 < 4; ++k1) {
                const int m = j2 * k1;
                const cx<float> x = t[k1];
                if (m == 0) a[j2][k1] = x;
                else if (m == 4) a[j2][k1] = {-x.im, x.re};
                else if (m == 2)
                    a[j2][k1] = {__fmaf_rn(x.re, h, -__fmul_rn(x.im, h)), __fmaf_rn(x.re, h, __fmul_rn(x.im, h))};
                else if (m == 6)
                    a[j2][k1] = {__fmaf_rn(x.re, -h, -__fmul_rn(x.im, h)), __fmaf_rn(x.im, -h, __fmul_rn(x.re, h))};
                else a[j2][k1] = rmul(x, w[m]);
            }
        }
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            cx<float> u[4] = {a[0][k1], a[1][k1], a[2][k1], a[3][k1]};
            dft<4>(u);
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = u[k2];
        }
    } else if constexpr (RADIX == 3) {
        const float s3 = 0.86602540378443864676f;
        const cx<float> t = radd(v[1], v[2]), d = rsub(v[1], v[2]);
        const cx<float> m = {__fmaf_rn(-0.5f, t.re, v[0].re), __fmaf_rn(-0.5f, t.im, v[0].im)};
        v[0] = radd(v[0], t);
        v[1] = {__fmaf_rn(-d.im, s3, m.re), __fmaf_rn(d.re, s3, m.im)};
        v[2] = {__fmaf_rn(d.im, s3, m.re), __fmaf_rn(-d.re, s3, m.im)};
    } else if constexpr (RADIX == 5) {
        const float c1 = 0.30901699437494742410f, c2 = -0.80901699437494742410f;
        const float s1 = 0.95105651629515357212f, s2 = 0.58778525229247312917f;
        const cx<float> t1 = radd(v[1], v[4]), d1 = rsub(v[1], v[4]), t2 = radd(v[2], v[3]), d2 = rsub(v[2], v[3]);
        const cx<float> a1 = {__fmaf_rn(c2, t2.re, __fmaf_rn(c1, t1.re, v[0].re)), __fmaf_rn(c2, t2.im, __fmaf_rn(c1, t1.im, v[0].im))};
        const cx<float> a2 = {__fmaf_rn(c1, t2.re, __fmaf_rn(c2, t1.re, v[0].re)), __fmaf_rn(c1, t2.im, __fmaf_rn(c2, t1.im, v[0].im))};
        const cx<float> b1 = {-__fmaf_rn(s1, d1.im, __fmul_rn(s2, d2.im)), __fmaf_rn(s1, d1.re, __fmul_rn(s2, d2.re))};
        const cx<float> b2 = {-__fmaf_rn(s2, d1.im, -__fmul_rn(s1, d2.im)), __fmaf_rn(s2, d1.re, -__fmul_rn(s1, d2.re))};
        v[0] = radd(v[0], radd(t1, t2));
        v[1] = radd(a1, b1);
        v[4] = rsub(a1, b1);
        v[2] = radd(a2, b2);
        v[3] = rsub(a2, b2);
    }
}

// Shared-memory layouts of P pencils of length M (one element = one complex):
//   pencil-fast (passes 1, 2):  (p, i) -> i P + p + i/8
//   index-fast  (pass 3):       (p, i) -> p PS + i + i/8,  PS = M + M/8 + 1
// The i/8 padding spreads the strided Stockham accesses over all banks.
template <bool PF, int P>
__device__ __forceinline__ int sidx(int p, int i, int M) {
    return PF ? i * P + p + (i >> 3) : p * (M + (M >> 3) + 1) + i + (i >> 3);
}
template <bool PF, int P>
__host__ __device__ constexpr int smem_elems(int M) {
    return PF ? M * P + (M >> 3) + 1 : P * (M + (M >> 3) + 1);
}

// One Stockham stage of radix RADIX over P pencils of length M, out of
// place from src to dst.  Butterfly j reads x[j + r M/RADIX], twiddles by
// W_M^{r (j mod Ns) M/(Ns RADIX)} and writes y[(j/Ns) Ns RADIX + j mod Ns + r Ns]
// (autosort: natural order after the last stage).  With M and Ns compile-time
// constants (the specialised kernels) all index arithmetic folds to shifts.
template <typename R, int RADIX, bool PF, int P>
__device__ __forceinline__ void fft_stage(const cx<R>* __restrict__ src, cx<R>* __restrict__ dst, int M, int Ns,
                                          const cx<R>* tw, int twmul) {
    const int nbf = M / RADIX;
    const int total = nbf * P;
    for (int b = threadIdx.x; b < total; b += NTHR) {
        int p, j;
        if (PF) { p = b % P; j = b / P; } else { j = b % nbf; p = b / nbf; }
        const int k = j % Ns;
        const int tstep = k * (M / (Ns * RADIX)) * twmul;
        cx<R> v[RADIX];
#pragma unroll
        for (int r = 0; r < RADIX; ++r) {
            const cx<R> x = src[sidx<PF, P>(p, j + r * nbf, M)];
            v[r] = r == 0 ? x : cmul(x, tw[r * tstep]);
        }
        butterfly<R, RADIX>(v);
        const int o = (j / Ns) * Ns * RADIX + k;
#pragma unroll
        for (int r = 0; r < RADIX; ++r) dst[sidx<PF, P>(p, o + r * Ns, M)] = v[r];
    }
    __syncthreads();
}

// Runtime radix list (any supported length).  Returns the result buffer.
template <typename R, bool PF, int P>
__device__ cx<R>* fft_pingpong(cx<R>* a, cx<R>* b, int M, const int* rad, int nrad, const cx<R>* tw, int twmul) {
    int Ns = 1;
    for (int s = 0; s < nrad; ++s) {
        switch (rad[s]) {
            case 8: fft_stage<R, 8, PF, P>(a, b, M, Ns, tw, twmul); break;
            case 4: fft_stage<R, 4, PF, P>(a, b, M, Ns, tw, twmul); break;
            case 2: fft_stage<R, 2, PF, P>(a, b, M, Ns, tw, twmul); break;
            case 3: fft_stage<R, 3, PF, P>(a, b, M, Ns, tw, twmul); break;
            case 5: fft_stage<R, 5, PF, P>(a, b, M, Ns, tw, twmul); break;
        }
        Ns *= rad[s];
        cx<R>* t = a; a = b; b = t;
    }
    return a;
}

// Compile-time radix list: 16s for the power of two (with one 8 and/or 4 for
// the leftover; 2^9 = 16 x 8 x 4), then 3s and 5s.  The host's plan for the
// run-time kernels uses radices up to 8; both give the same transform.
struct RadixList {
    int n;
    int r[8];
};
__host__ __device__ constexpr RadixList radix_list(int m) {
    RadixList L{0, {0, 0, 0, 0, 0, 0, 0, 0}};
    int a = 0;
    while (m % 2 == 0) { m /= 2; ++a; }
    int n16 = a / 4, rem = a % 4;
    if (rem == 1 && n16 > 0) { --n16; }
    for (int i = 0; i < n16; ++i) L.r[L.n++] = 16;
    if (rem == 3) L.r[L.n++] = 8;
    else if (rem == 2) L.r[L.n++] = 4;
    else if (rem == 1 && a >= 5) { L.r[L.n++] = 8; L.r[L.n++] = 4; }
    else if (rem == 1) L.r[L.n++] = 2;
    while (m % 3 == 0) { m /= 3; L.r[L.n++] = 3; }
    while (m % 5 == 0) { m /= 5; L.r[L.n++] = 5; }
    return L;
}

template <typename R, bool PF, int P, int M, int S = 0, int NS = 1>
__device__ __forceinline__ cx<R>* fft_ct(cx<R>* a, cx<R>* b, const cx<R>* tw, int twmul) {
    constexpr RadixList L = radix_list(M);
    if constexpr (S >= L.n) {
        return a;
    } else {
        constexpr int RADIX = L.r[S];
        fft_stage<R, RADIX, PF, P>(a, b, M, NS, tw, twmul);
        return fft_ct<R, PF, P, M, S + 1, NS * RADIX>(b, a, tw, twmul);
    }
}

__device__ __forceinline__ int freq_of(int idx, int n) { return idx < n / 2 ? idx : idx - n; }

// Largest |frequency component| where the field can be nonzero (its shell's
// outer edge, at most K).  Every pass uses the same bound: pass 1 skips the
// pencils beyond it (f_y or f_z), pass 2 skips the f_z beyond it and reads no
// f_y beyond it, pass 3 reads no f_z beyond it, so nothing unwritten is read.
__device__ __forceinline__ int field_ext(const FieldDesc& fd, const FftGeom& g) {
    return fd.kext > 0 ? min(fd.kext, g.K) : g.K;
}

// W_f(n): the field's radial factor times w_l(mu), mu^2 = n_z^2/|n|^2.
template <typename R>
__device__ __forceinline__ R filter_weight(const FieldDesc& fd, int n2, int fz, const int16_t* shell_of,
                                           const float* radial, int n2max) {
    if (n2 <= 0 || n2 > n2max) return (R)0;
    R base;
    if (fd.kind == FIELD_RAW) return (R)1;
    if (fd.kind == FIELD_RADIAL) base = (R)radial[(size_t)fd.shell * (n2max + 1) + n2];
    else base = (shell_of[n2] == fd.shell) ? (R)1 : (R)0;
    if (base == (R)0 || fd.ell == 0) return base;
    const R mu2 = (R)(fz * fz) / (R)n2;
    if (fd.ell == 2) return base * (R)2.5 * ((R)3 * mu2 - (R)1);                       // 5 L_2
    return base * (R)1.125 * (((R)35 * mu2 - (R)30) * mu2 + (R)3);                     // 9 L_4
}

// Input of pass 1: the filtered spectrum W_f(n) S_f(n) at (f_x of ix, f_y of
// iy, k_z), zero outside the pruned range.
template <typename R>
__device__ __forceinline__ cx<R> pass1_input(const FftGeom& g, const FieldDesc& fd, const cx<float>* __restrict__ delta,
                                             const int16_t* __restrict__ shell_of, const float* __restrict__ radial,
                                             int N, int ix, int fy, int iy, int kz) {
    const int fx = freq_of(ix, N);
    cx<R> val = {(R)0, (R)0};
    if (kz < g.nKz && (!g.pruned || (fx >= -g.K && fx <= g.K))) {
        const int fz = (kz == N / 2) ? -(N / 2) : kz;
        const int n2 = fx * fx + fy * fy + fz * fz;
        const R w = filter_weight<R>(fd, n2, fz, shell_of, radial, g.n2max);
        if (w != (R)0) {
            if (fd.kind == FIELD_UNIT) {
                val.re = w;
            } else {
                const cx<float> d = delta[((size_t)ix * N + iy) * (N / 2 + 1) + kz];
                if (fd.kind == FIELD_POWER) {
                    // |delta|^2 of the Hermitian part: on the n_z = 0 and n/2 planes the
                    // half spectrum holds both n and -n, (delta(n) + conj delta(-n)) / 2
                    R re = (R)d.re, im = (R)d.im;
                    if (kz == 0 || kz == N / 2) {
                        const cx<float> m = delta[((size_t)((N - ix) % N) * N + (N - iy) % N) * (N / 2 + 1) + kz];
                        re = (R)0.5 * (re + (R)m.re);
                        im = (R)0.5 * (im - (R)m.im);
                    }
                    val.re = w * (re * re + im * im);
                } else {
                    val.re = w * (R)d.re;
                    val.im = w * (R)d.im;
                }
            }
        }
    }
    return val;
}

// Pass 1: filter + inverse DFT along x for P consecutive f_z of one f_y.
template <typename R, int P, int NN>
__global__ void __launch_bounds__(NTHR) k_pass1(FftGeom g, const cx<float>* __restrict__ delta,
                                                const int16_t* __restrict__ shell_of,
                                                const float* __restrict__ radial,
                                                const FieldDesc* __restrict__ fields,
                                                const cx<R>* __restrict__ twg, cx<R>* __restrict__ t1,
                                                size_t t1_stride) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = NN ? NN : g.n;
    cx<R>* tw = reinterpret_cast<cx<R>*>(smem_raw);
    cx<R>* buf = tw + N;
    cx<R>* scr = buf + smem_elems<true, P>(N);
    const FieldDesc fd = fields[blockIdx.y];
    const int nkzb = (g.nKz + P - 1) / P;
    const int cy = blockIdx.x / nkzb, kz0 = (blockIdx.x % nkzb) * P;
    const int fy = g.pruned ? cy - g.K : freq_of(cy, N);
    const int iy = (fy + N) % N;
    const int ke = field_ext(fd, g);
    if (fy > ke || fy < -ke || kz0 > ke) return;   // zero there, and pass 2 reads none of it
    for (int t = threadIdx.x; t < N; t += NTHR) tw[t] = twg[t];
    for (int e = threadIdx.x; e < N * P; e += NTHR) {
        const int p = e % P, ix = e / P, kz = kz0 + p;
        const cx<R> val = pass1_input<R>(g, fd, delta, shell_of, radial, N, ix, fy, iy, kz);
        buf[sidx<true, P>(p, ix, N)] = val;
    }
    __syncthreads();
    const cx<R>* res;
    if constexpr (NN > 0) res = fft_ct<R, true, P, NN>(buf, scr, tw, 1);
    else res = fft_pingpong<R, true, P>(buf, scr, N, g.rad, g.nrad, tw, 1);
    cx<R>* dst = t1 + (size_t)blockIdx.y * t1_stride;
    for (int e = threadIdx.x; e < N * P; e += NTHR) {
        const int p = e % P, x = e / P, kz = kz0 + p;
        if (kz < g.nKz) dst[((size_t)cy * N + x) * g.ldz + kz] = res[sidx<true, P>(p, x, N)];
    }
}

// Pass 2: inverse DFT along y for P consecutive f_z of one x.
__device__ __forceinline__ void block_max_to(unsigned* dst, float m) {
    // m >= 0: the float bit patterns order like the values
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(dst, __float_as_uint(m));
}

// Power of two s with bound * s in [2^(t-1), 2^t): t = 15 keeps 16-bit
// values below the FP16 maximum; t = 7 keeps a product of two scaled pair
// factors below 2^14.  Exact, so dividing by s afterwards is exact.
__device__ __forceinline__ float pow2_scale(float bound, int t = 15) {
    if (!(bound > 0.f)) return 1.f;
    int e;
    frexpf(bound, &e);
    return ldexpf(1.f, t - e);
}

template <typename R, int P, int NN>
__global__ void __launch_bounds__(NTHR) k_pass2(FftGeom g, const cx<R>* __restrict__ t1,
                                                size_t t1_stride, const cx<R>* __restrict__ twg,
                                                cx<R>* __restrict__ t2, size_t t2_stride,
                                                const FieldDesc* __restrict__ fields) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = NN ? NN : g.n;
    cx<R>* tw = reinterpret_cast<cx<R>*>(smem_raw);
    cx<R>* buf = tw + N;
    cx<R>* scr = buf + smem_elems<true, P>(N);
    const int nkzb = (g.nKz + P - 1) / P;
    const int x = blockIdx.x / nkzb, kz0 = (blockIdx.x % nkzb) * P;
    const int ke = field_ext(fields[blockIdx.y], g);
    if (kz0 > ke) return;   // zero there, and pass 3 reads none of it
    const cx<R>* src = t1 + (size_t)blockIdx.y * t1_stride;
    for (int t = threadIdx.x; t < N; t += NTHR) tw[t] = twg[t];
    for (int e = threadIdx.x; e < N * P; e += NTHR) {
        const int p = e % P, iy = e / P, kz = kz0 + p;
        const int fy = freq_of(iy, N);
        cx<R> val = {(R)0, (R)0};
        if (kz < g.nKz && fy >= -ke && fy <= ke) {
            const int cy = g.pruned ? fy + g.K : iy;
            val = src[((size_t)cy * N + x) * g.ldz + kz];
        }
        buf[sidx<true, P>(p, iy, N)] = val;
    }
    __syncthreads();
    const cx<R>* res;
    if constexpr (NN > 0) res = fft_ct<R, true, P, NN>(buf, scr, tw, 1);
    else res = fft_pingpong<R, true, P>(buf, scr, N, g.rad, g.nrad, tw, 1);
    cx<R>* dst = t2 + (size_t)blockIdx.y * t2_stride;
    for (int e = threadIdx.x; e < N * P; e += NTHR) {
        const int p = e % P, y = e / P, kz = kz0 + p;
        if (kz < g.nKz) dst[((size_t)x * N + y) * g.ldz + kz] = res[sidx<true, P>(p, y, N)];
    }
}

// Pass 2 for n = 512 with the y-lines in registers: 8 lines (consecutive
// f_z of one x) per CTA, 32 threads per line, k_z fastest across the lanes so
// that every global load and store is a run of 8 consecutive f_z (64 bytes).
// With k = k1 + 32 k2 (thread k1 holds k2 = 0..15) and m = m1 + 16 m2,
//   z_m = sum_k1 W32^{k1 m2} [ W512^{k1 m1} sum_k2 X_{k1 + 32 k2} W16^{k2 m1} ],
// W_L = e^{2 pi i / L}; after one shared-memory transpose the outer 32-point
// DFT over k1 = j1 + 2 j2 is a 16-point DFT over j2 in each of two threads
// (j1 = 0, 1) and a radix-2 step between them through a shuffle:
//   z_{m1 + 16 (n + 16 q)} = U_0[n] + (-1)^q W32^n U_1[n].
constexpr int P2R = 8;
__host__ __device__ constexpr int p2r_idx(int row, int p) { return row * P2R + p + (row >> 4) * 8; }   // row = k1 * 16 + m1
constexpr size_t p2r_smem_bytes() { return sizeof(cx<float>) * (512 + (size_t)p2r_idx(511, P2R - 1) + 1); }

// The 512-point inverse DFT of the CTA's 8 lines.  On entry thread (k1 = 4 warp
// + c, line p) holds X_{k1 + 32 k2} in v[k2] and the twiddles are in tw; on
// return thread (m1 = 2 warp + (c >> 1), j1 = c & 1, line p) holds
// z_{m1 + 16 (n + 16 j1)} in v[n].  tr: the transpose buffer.
__device__ __forceinline__ void line512(cx<float> (&v)[16], const cx<float>* tw, cx<float>* tr, int warp, int c,
                                        int p) {
    const int k1 = 4 * warp + c;
    butterfly<float, 16>(v);   // v[m1] = sum_k2 X_{k1 + 32 k2} W16^{k2 m1}
#pragma unroll
    for (int m1 = 0; m1 < 16; ++m1) tr[p2r_idx(k1 * 16 + m1, p)] = m1 == 0 ? v[0] : cmul(v[m1], tw[k1 * m1]);
    __syncthreads();
    const int m1 = 2 * warp + (c >> 1), j1 = c & 1;
#pragma unroll
    for (int j2 = 0; j2 < 16; ++j2) v[j2] = tr[p2r_idx((j1 + 2 * j2) * 16 + m1, p)];
    butterfly<float, 16>(v);   // U_j1[n]
#pragma unroll
    for (int n = 0; n < 16; ++n) {
        cx<float> u = v[n];
        if (j1) u = cmul(u, tw[16 * n]);   // W32^n U_1[n]
        const cx<float> o = {__shfl_xor_sync(0xffffffffu, u.re, 8), __shfl_xor_sync(0xffffffffu, u.im, 8)};
        // j1 = 0 keeps U_0 + W U_1 (m2 = n), j1 = 1 keeps U_0 - W U_1 (m2 = n + 16)
        v[n] = j1 ? csub(o, u) : cadd(u, o);
    }
}

// Pass 1 for n = 512 with the x-lines in registers: 8 lines (consecutive
// f_z of one f_y) per CTA, laid out and transformed as in k_pass2r.
__global__ void __launch_bounds__(NTHR) k_pass1r(FftGeom g, const cx<float>* __restrict__ delta,
                                                 const int16_t* __restrict__ shell_of,
                                                 const float* __restrict__ radial,
                                                 const FieldDesc* __restrict__ fields,
                                                 const cx<float>* __restrict__ twg, cx<float>* __restrict__ t1,
                                                 size_t t1_stride) {
    constexpr int N = 512;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cx<float>* tw = reinterpret_cast<cx<float>*>(smem_raw);
    cx<float>* tr = tw + N;
    const FieldDesc fd = fields[blockIdx.y];
    const int nkzb = (g.nKz + P2R - 1) / P2R;
    const int cy = blockIdx.x / nkzb, kz0 = (blockIdx.x % nkzb) * P2R;
    const int fy = g.pruned ? cy - g.K : freq_of(cy, N);
    const int iy = (fy + N) % N;
    const int ke = field_ext(fd, g);
    if (fy > ke || fy < -ke || kz0 > ke) return;   // zero there, and pass 2 reads none of it
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int p = lane & 7, c = lane >> 3;
    const int kz = kz0 + p;
    for (int i = threadIdx.x; i < N; i += NTHR) tw[i] = twg[i];
    const int k1 = 4 * warp + c;
    cx<float> v[16];
#pragma unroll
    for (int k2 = 0; k2 < 16; ++k2) v[k2] = pass1_input<float>(g, fd, delta, shell_of, radial, N, k1 + 32 * k2, fy, iy, kz);
    __syncthreads();   // twiddles
    line512(v, tw, tr, warp, c, p);
    const int m1 = 2 * warp + (c >> 1), j1 = c & 1;
    if (kz < g.nKz) {
        cx<float>* dst = t1 + (size_t)blockIdx.y * t1_stride;
#pragma unroll
        for (int n = 0; n < 16; ++n) dst[((size_t)cy * N + m1 + 16 * (n + 16 * j1)) * g.ldz + kz] = v[n];
    }
}

__global__ void __launch_bounds__(NTHR) k_pass2r(FftGeom g, const cx<float>* __restrict__ t1, size_t t1_stride,
                                                 const cx<float>* __restrict__ twg, cx<float>* __restrict__ t2,
                                                 size_t t2_stride, const FieldDesc* __restrict__ fields,
                                                 unsigned* __restrict__ fmax2) {
    constexpr int N = 512;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cx<float>* tw = reinterpret_cast<cx<float>*>(smem_raw);
    cx<float>* tr = tw + N;
    const int nkzb = (g.nKz + P2R - 1) / P2R;
    const int x = blockIdx.x / nkzb, kz0 = (blockIdx.x % nkzb) * P2R;
    const int ke = field_ext(fields[blockIdx.y], g);
    if (kz0 > ke) return;   // zero there, and pass 3 reads none of it
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int p = lane & 7, c = lane >> 3;   // line (f_z offset) and lane group
    const int kz = kz0 + p;
    const bool live = kz < g.nKz;
    for (int i = threadIdx.x; i < N; i += NTHR) tw[i] = twg[i];
    const cx<float>* src = t1 + (size_t)blockIdx.y * t1_stride;
    // step A: thread k1 = 4 warp + c
    const int k1 = 4 * warp + c;
    cx<float> v[16];
#pragma unroll
    for (int k2 = 0; k2 < 16; ++k2) {
        const int iy = k1 + 32 * k2, fy = iy < N / 2 ? iy : iy - N;
        cx<float> val = {0.f, 0.f};
        if (live && fy >= -ke && fy <= ke) {
            const int cy = g.pruned ? fy + g.K : iy;
            val = src[((size_t)cy * N + x) * g.ldz + kz];
        }
        v[k2] = val;
    }
    __syncthreads();   // twiddles
    line512(v, tw, tr, warp, c, p);
    const int m1 = 2 * warp + (c >> 1), j1 = c & 1;
    cx<float>* dst = t2 + (size_t)blockIdx.y * t2_stride;
    float mx = 0.f;
#pragma unroll
    for (int n = 0; n < 16; ++n) {
        const int y = m1 + 16 * (n + 16 * j1);
        if (live) {
            dst[((size_t)x * N + y) * g.ldz + kz] = v[n];
            mx = fmaxf(mx, fabsf(v[n].re) + fabsf(v[n].im));
        }
    }
    if (fmax2) {
        const int f = fields[blockIdx.y].out16;
        if (f >= 0) block_max_to(fmax2 + f, mx);
    }
}

// Pass 3: real inverse DFT along z for P consecutive y of one x, through a
// complex DFT of length M = N/2:  Z_k = (H_k + conj H_{M-k})
//   + i (H_k - conj H_{M-k}) e^{2 pi i k/N},  F[2m] = Re z_m, F[2m+1] = Im z_m,
// with Im H_0 = Im H_M = 0 (the Hermitian part of the n_z = 0, N/2 planes).
template <typename R, int P, int NN>
__global__ void __launch_bounds__(NTHR) k_pass3(FftGeom g, const cx<R>* __restrict__ t2,
                                                size_t t2_stride, const cx<R>* __restrict__ twg,
                                                const FieldDesc* __restrict__ fields, R* __restrict__ out,
                                                size_t out_stride) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = NN ? NN : g.n, M = N / 2;
    cx<R>* tw = reinterpret_cast<cx<R>*>(smem_raw);
    cx<R>* buf = tw + N;
    cx<R>* scr = buf + smem_elems<false, P>(M);
    const int nyb = (N + P - 1) / P;
    const int x = blockIdx.x / nyb, y0 = (blockIdx.x % nyb) * P;
    const cx<R>* src = t2 + (size_t)blockIdx.y * t2_stride;
    const int nk = field_ext(fields[blockIdx.y], g) + 1;   // f_z read: 0 .. nk - 1
    for (int t = threadIdx.x; t < N; t += NTHR) tw[t] = twg[t];
    __syncthreads();
    for (int e = threadIdx.x; e < M * P; e += NTHR) {
        const int k = e % M, p = e / M, y = y0 + p;
        cx<R> z = {(R)0, (R)0};
        if (y < N) {
            const cx<R>* h = src + ((size_t)x * N + y) * g.ldz;
            cx<R> a = {(R)0, (R)0}, b = {(R)0, (R)0};
            if (k < nk) a = h[k];
            if (M - k < nk) b = h[M - k];
            if (k == 0) { a.im = (R)0; b.im = (R)0; }   // H_0 and H_M: real parts only
            const cx<R> bc = {b.re, -b.im};
            const cx<R> s = cadd(a, bc), d = csub(a, bc);
            z = cadd(s, cmuli(cmul(d, tw[k])));
        }
        buf[sidx<false, P>(p, k, M)] = z;
    }
    __syncthreads();
    const cx<R>* res;
    if constexpr (NN > 0) res = fft_ct<R, false, P, NN / 2>(buf, scr, tw, 2);
    else res = fft_pingpong<R, false, P>(buf, scr, M, g.rad_h, g.nrad_h, tw, 2);
    cx<R>* dst = reinterpret_cast<cx<R>*>(out + (size_t)fields[blockIdx.y].out32 * out_stride);
    for (int e = threadIdx.x; e < M * P; e += NTHR) {
        const int m = e % M, p = e / M, y = y0 + p;
        if (y < N) dst[((size_t)x * N + y) * M + m] = res[sidx<false, P>(p, m, M)];
    }
}

// Pass 3 for the sizes known at compile time, FP32, with the z-lines in registers:
// M = n/2 = R1 x R2, the two stages of the Stockham list (16 x 3, 16 x 4, 16 x 5,
// 16 x 8, 16 x 16, 8 x 4).  P consecutive lines (of all n^2: T2 and the output are
// both linear in the line) per CTA.  Thread (line, j < R2) forms its R1 inputs
// Z_{j + R2 r} straight from T2 (the same Z_k as k_pass3) and takes the R1-point
// DFT; the lines pass once through shared memory, and thread (line, j < R1)
// takes the R2-point DFTs and stores from registers: 16 lanes hold 16
// consecutive complex values, a whole 128-byte run of FP32 or 64 bytes of each
// 16-bit plane row.  One barrier.  Eight lines a CTA through one shared-memory
// stage after another, as before, kept a few dozen of 256 threads busy in the
// radix-16 stage.  Fields and time before -> now: 288 FP32 fields of 256^3 14.2 ->
// 4.9 ms (4.4 at the copy rate), 72 of 160^3 1.33 -> 0.27 ms, 150 operand sets of 256^3
// 8.9 -> 4.0 ms, 96 of 512^3 (16 x 16 in registers before, staged for 16-byte stores)
// 20.5 -> 18.8 ms.  Bound for FP32 fields of 256^3: L1, 77 % busy, then DRAM at 77 % of the
// copy rate (36 fields 533 us); the planes of 512^3 are written at 67 % of it.
template <int NN>
struct P3V {
    static constexpr int M = NN / 2;
    static constexpr RadixList L = radix_list(M);
    static constexpr int R1 = L.r[0], R2 = L.r[1];
    static_assert(L.n == 2 && R1 * R2 == M, "two stages");
    static constexpr int P = M >= 256 ? 16 : M >= 80 ? 32 : 64;   // divides n^2
    static constexpr int T = P * R2;
    // element i of a line at i + i / R1: stage 1 writes rows of R1 (odd row stride) and stage 2 reads columns
    static constexpr int PS = M + R2;
    __device__ static int idx(int p, int i) { return p * PS + i + i / R1; }
    static constexpr size_t smem() { return sizeof(cx<float>) * ((size_t)P * PS + M); }
};

enum { P3_FIELD, P3_F16, P3_BF16 };   // FP32 fields, or the K-block-major operands with FP16 or BF16 planes

// Two consecutive z values (x0 in the low half) -> 16-bit hi and lo words.
template <int MODE>
__device__ __forceinline__ void split_pair(float x0, float x1, uint32_t& hw, uint32_t& lw) {
    float h0, h1;
    if (MODE == P3_F16) {
        asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(hw) : "f"(x1), "f"(x0));
        unsigned short a = (unsigned short)(hw & 0xFFFFu), b = (unsigned short)(hw >> 16);
        asm("cvt.f32.f16 %0, %1;" : "=f"(h0) : "h"(a));
        asm("cvt.f32.f16 %0, %1;" : "=f"(h1) : "h"(b));
        asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(lw) : "f"(x1 - h1), "f"(x0 - h0));
    } else {
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(hw) : "f"(x1), "f"(x0));
        h0 = __uint_as_float(hw << 16);
        h1 = __uint_as_float(hw & 0xFFFF0000u);
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(lw) : "f"(x1 - h1), "f"(x0 - h0));
    }
}

template <int NN, int MODE>
__global__ void __launch_bounds__(P3V<NN>::T, 1024 / P3V<NN>::T) k_pass3v(FftGeom g, const cx<float>* __restrict__ t2, size_t t2_stride,
                                                       const cx<float>* __restrict__ tw,
                                                       const FieldDesc* __restrict__ fields, float* __restrict__ out,
                                                       size_t out_stride, uint32_t* __restrict__ hi, int split,
                                                       const unsigned* __restrict__ fmax2, FieldLayout lay) {
    using V = P3V<NN>;
    constexpr int M = V::M, R1 = V::R1, R2 = V::R2, P = V::P;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cx<float>* buf = reinterpret_cast<cx<float>*>(smem_raw);
    cx<float>* tw2 = buf + P * V::PS;   // [r][j] = W_M^{r j}: consecutive across the lanes (gathered from global
                                        // memory at each use, they took most of the L1 wavefronts)
    const FieldDesc fd = fields[blockIdx.y];
    const int nKz = g.nKz, nk = field_ext(fd, g) + 1;   // f_z read: 0 .. nk - 1
    const size_t line0 = (size_t)blockIdx.x * P;
    for (int i = threadIdx.x; i < M; i += V::T) tw2[i] = tw[2 * (i / R1) * (i % R1)];
    {
        const int j = threadIdx.x % R2, p = threadIdx.x / R2;
        const cx<float>* h = t2 + (size_t)blockIdx.y * t2_stride + (line0 + p) * g.ldz;
        cx<float> v[R1];
#pragma unroll
        for (int r = 0; r < R1; ++r) {
            const int k = j + R2 * r;
            cx<float> a = {0.f, 0.f}, b = {0.f, 0.f};
            if (k < nk) a = h[k];
            if (M - k < nk) b = h[M - k];
            if (k == 0) { a.im = 0.f; b.im = 0.f; }   // H_0 and H_M: real parts only
            const cx<float> bc = {b.re, -b.im};
            const cx<float> s = radd(a, bc), d = rsub(a, bc), dw = rmul(d, tw[k]);
            v[r] = radd(s, cx<float>{-dw.im, dw.re});
        }
        dft<R1>(v);
#pragma unroll
        for (int r = 0; r < R1; ++r) buf[V::idx(p, j * R1 + r)] = v[r];
    }
    __syncthreads();
    // the power-of-two scales of the tensor-core operands (|F(x,y,z)| <= sum_kz 2 |H_kz| <=
    // 2 nKz max|T2|): 16-bit planes below 2^15, FP32 pair factors below 2^7
    float sc = 1.f, s7 = 1.f;
    if (MODE != P3_FIELD) {
        const float bound = 2.f * (float)nKz * __uint_as_float(fmax2[fd.out16]);
        sc = pow2_scale(bound);
        s7 = pow2_scale(bound, 7);
    }
#pragma unroll 1
    for (int e = threadIdx.x; e < P * R1; e += V::T) {
        const int j = e % R1, p = e / R1;
        cx<float> v[R2];
#pragma unroll
        for (int r = 0; r < R2; ++r) {
            const cx<float> x = buf[V::idx(p, j + R1 * r)];
            v[r] = r == 0 ? x : rmul(x, tw2[r * R1 + j]);
        }
        dft<R2>(v);
        const size_t pos0 = (line0 + p) * M + j;   // complex values: pairs of consecutive z
        if (MODE == P3_FIELD) {
            cx<float>* d = reinterpret_cast<cx<float>*>(out + (size_t)fd.out32 * out_stride) + pos0;
#pragma unroll
            for (int r = 0; r < R2; ++r) d[R1 * r] = v[r];
            continue;
        }
        // Value r is pair w = pos % 32 of K-block pos / 32 (points 2 w, 2 w + 1).  pos0 - j is a
        // multiple of R1; where a line is whole K-blocks (M = 32, 64, ...), w depends on r
        // through r R1 % 32 only.
        const size_t kb0 = pos0 >> 5;
        const int w0 = (int)(pos0 & 31);
        auto at = [&](int r, size_t& kb, int& w) {
            if (M % 32 == 0) {
                kb = kb0 + (R1 * r) / 32;
                w = j + (R1 * r) % 32;
            } else {
                kb = kb0 + ((w0 + R1 * r) >> 5);
                w = (w0 + R1 * r) & 31;
            }
        };
        if (fd.out32 >= 0) {   // FP32 row: 16-byte chunk J of 256 bytes, swizzled in halves
            const int r32 = fd.out32 & 7;
            cx<float>* d = reinterpret_cast<cx<float>*>(out) + (size_t)fd.out32 * 32;
#pragma unroll
            for (int r = 0; r < R2; ++r) {
                size_t kb;
                int w;
                at(r, kb, w);
                d[kb * (size_t)(lay.rows32 * 32) + (w ^ (2 * r32))] = cx<float>{v[r].re * s7, v[r].im * s7};
            }
        }
        uint32_t* q = hi + (size_t)(fd.out16 >> 3) * 512 + (size_t)(fd.out16 & 7) * 32;
        const int r16 = fd.out16 & 7;
#pragma unroll
        for (int r = 0; r < R2; ++r) {   // plane rows: 16-byte chunks swizzled; the lo row 1024 bytes further
            size_t kb;
            int w;
            at(r, kb, w);
            uint32_t* d = q + kb * (size_t)(lay.groups16 * 512) + (w ^ (4 * r16));
            uint32_t hw, lw;
            split_pair<MODE>(v[r].re * sc, v[r].im * sc, hw, lw);
            d[0] = hw;
            if (split) d[256] = lw;
        }
    }
}

// ---------------------------------------------------------------------------
// Passes 1 and 2 (FP32) for every size but 512, and pass 3 for the sizes not known at
// compile time.  CP lines side by side in shared memory, element i of line p at
// i SP + p: the lanes run over the lines, so every access is a row of consecutive
// lines (no conflicts, no index division), and a stage has (length / radix) CP
// butterflies for the CTA's threads.  Passes 1 and 2 take their first stage straight
// from global memory and store the last one there, in runs of CP consecutive f_z
// (128 bytes, in rows padded to 64).  Bound by issue slots and latency: at 150^3 pass 2 has 64 %
// of its slots busy, pass 3 78 %; two to four stages with a barrier each.  Eight lines on 256 threads with run-time divisions in
// every index, before, left most threads idle.  Before -> now, microseconds: 42 fields
// of 150^3 pass 1 107 -> 70, 2 302 -> 190, 3 1 331 -> 630; 150 of 256^3 pass 2 3 159 -> 2 000;
// 72 of 160^3 pass 2 160 -> 130; 32^3 with 8 shells, all three 50 -> 30.
// ---------------------------------------------------------------------------
constexpr int CP = 16;

// NSC: the product of the radices before (0: known at run time; magic = ceil(2^32 / Ns)).
template <int RADIX, bool FIRST, bool LAST, int NSC, int SP, int P, class Ld, class St>
__device__ __forceinline__ void col_stage(const cx<float>* src, cx<float>* dst, int M, int Ns_, unsigned magic, int twmul,
                                          const cx<float>* __restrict__ tw, Ld ld, St st) {
    const int nbf = M / RADIX, Ns = NSC ? NSC : Ns_;
    const int tmul = nbf / Ns * twmul;   // M / (Ns RADIX) twiddle steps
#pragma unroll 1
    for (int b = threadIdx.x; b < nbf * P; b += blockDim.x) {
        const int p = b % P, j = b / P;
        const int k = Ns == 1 ? 0 : j - Ns * (NSC ? j / NSC : (int)__umulhi((unsigned)j, magic));
        cx<float> v[RADIX];
#pragma unroll
        for (int r = 0; r < RADIX; ++r) {
            v[r] = FIRST ? ld(j + r * nbf, p) : src[(j + r * nbf) * SP + p];
            if (!FIRST && r > 0 && Ns > 1) v[r] = rmul(v[r], tw[r * k * tmul]);
        }
        dft<RADIX>(v);
        const int o = (j - k) * RADIX + k;
#pragma unroll
        for (int r = 0; r < RADIX; ++r) {
            if (LAST) st(o + r * Ns, p, v[r]);
            else dst[(o + r * Ns) * SP + p] = v[r];
        }
    }
    if (!LAST) __syncthreads();
}

// Compile-time radix list, through the buffers a and b.  IO: the first stage loads
// through ld and the last stores through st; otherwise the lines are in a, and the
// buffer they end in is returned.
template <int M, bool IO, int SP, int P, int S, int NS, class Ld, class St>
__device__ __forceinline__ cx<float>* col_ct(cx<float>* a, cx<float>* b, int twmul, const cx<float>* tw, Ld ld, St st) {
    constexpr RadixList L = radix_list(M);
    if constexpr (S < L.n) {
        col_stage<L.r[S], IO && S == 0, IO && S == L.n - 1, NS, SP, P>(a, b, M, NS, 0u, twmul, tw, ld, st);
        return col_ct<M, IO, SP, P, S + 1, NS * L.r[S]>(b, a, twmul, tw, ld, st);
    } else {
        return a;
    }
}

// Run-time radix list (8, 4, 2, 3, 5).
template <bool FIRST, bool LAST, int SP, int P, class Ld, class St>
__device__ __forceinline__ void col_rt1(int rad, const cx<float>* a, cx<float>* b, int M, int Ns, int twmul,
                                        const cx<float>* tw, Ld ld, St st) {
    const unsigned magic = Ns > 1 ? (unsigned)((0x100000000ull + Ns - 1) / Ns) : 0u;
    switch (rad) {
        case 8: col_stage<8, FIRST, LAST, 0, SP, P>(a, b, M, Ns, magic, twmul, tw, ld, st); break;
        case 4: col_stage<4, FIRST, LAST, 0, SP, P>(a, b, M, Ns, magic, twmul, tw, ld, st); break;
        case 2: col_stage<2, FIRST, LAST, 0, SP, P>(a, b, M, Ns, magic, twmul, tw, ld, st); break;
        case 3: col_stage<3, FIRST, LAST, 0, SP, P>(a, b, M, Ns, magic, twmul, tw, ld, st); break;
        default: col_stage<5, FIRST, LAST, 0, SP, P>(a, b, M, Ns, magic, twmul, tw, ld, st); break;
    }
}
template <bool IO, int SP, int P, class Ld, class St>
__device__ __forceinline__ cx<float>* col_rt(cx<float>* a, cx<float>* b, int M, const int* rad, int nrad, int twmul,
                                             const cx<float>* tw, Ld ld, St st) {
    if (IO && nrad == 1) {
        col_rt1<true, true, SP, P>(rad[0], a, b, M, 1, twmul, tw, ld, st);
        return a;
    }
    int Ns = 1;
    for (int s = 0; s < nrad; ++s) {
        if (IO && s == 0) col_rt1<true, false, SP, P>(rad[s], a, b, M, Ns, twmul, tw, ld, st);
        else if (IO && s == nrad - 1) col_rt1<false, true, SP, P>(rad[s], a, b, M, Ns, twmul, tw, ld, st);
        else col_rt1<false, false, SP, P>(rad[s], a, b, M, Ns, twmul, tw, ld, st);
        Ns *= rad[s];
        cx<float>* t = a;
        a = b;
        b = t;
    }
    return a;
}

// Pass 1: filter + inverse DFT along x for CP consecutive f_z of one f_y.
template <int NN>
__global__ void __launch_bounds__(256) k_col1(FftGeom g, const cx<float>* __restrict__ delta,
                                              const int16_t* __restrict__ shell_of, const float* __restrict__ radial,
                                              const FieldDesc* __restrict__ fields, const cx<float>* __restrict__ tw,
                                              cx<float>* __restrict__ t1, size_t t1_stride) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = NN ? NN : g.n;
    cx<float>* buf = reinterpret_cast<cx<float>*>(smem_raw);
    const FieldDesc fd = fields[blockIdx.y];
    const int nkzb = (g.nKz + CP - 1) / CP;
    const int cy = blockIdx.x / nkzb, kz0 = (blockIdx.x % nkzb) * CP;
    const int fy = g.pruned ? cy - g.K : freq_of(cy, N);
    const int iy = fy < 0 ? fy + N : fy;
    const int ke = field_ext(fd, g);
    if (fy > ke || fy < -ke || kz0 > ke) return;   // zero there, and pass 2 reads none of it
    cx<float>* dst = t1 + (size_t)blockIdx.y * t1_stride + (size_t)cy * N * g.ldz + kz0;
    auto ld = [&](int i, int p) { return pass1_input<float>(g, fd, delta, shell_of, radial, N, i, fy, iy, kz0 + p); };
    auto st = [&](int i, int p, cx<float> v) {
        if (kz0 + p < g.nKz) dst[(size_t)i * g.ldz + p] = v;
    };
    if constexpr (NN > 0) col_ct<NN, true, CP, CP, 0, 1>(buf + NN * CP, buf, 1, tw, ld, st);   // two stages use buf only
    else col_rt<true, CP, CP>(buf + N * CP, buf, N, g.rad, g.nrad, 1, tw, ld, st);
}

// Pass 2: inverse DFT along y for CP consecutive f_z of one x.
template <int NN>
__global__ void __launch_bounds__(256) k_col2(FftGeom g, const cx<float>* __restrict__ t1, size_t t1_stride,
                                              const cx<float>* __restrict__ tw, cx<float>* __restrict__ t2,
                                              size_t t2_stride, const FieldDesc* __restrict__ fields,
                                              unsigned* __restrict__ fmax2) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = NN ? NN : g.n;
    cx<float>* buf = reinterpret_cast<cx<float>*>(smem_raw);
    const int nkzb = (g.nKz + CP - 1) / CP;
    const int x = blockIdx.x / nkzb, kz0 = (blockIdx.x % nkzb) * CP;
    const FieldDesc fd = fields[blockIdx.y];
    const int ke = field_ext(fd, g);
    if (kz0 > ke) return;   // zero there, and pass 3 reads none of it
    const cx<float>* src = t1 + (size_t)blockIdx.y * t1_stride + (size_t)x * g.ldz + kz0;
    cx<float>* dst = t2 + (size_t)blockIdx.y * t2_stride + (size_t)x * N * g.ldz + kz0;
    float m = 0.f;
    auto ld = [&](int i, int p) {
        const int f = freq_of(i, N);
        cx<float> v = {0.f, 0.f};
        if (kz0 + p < g.nKz && f >= -ke && f <= ke) v = src[(size_t)(g.pruned ? f + g.K : i) * N * g.ldz + p];
        return v;
    };
    auto st = [&](int i, int p, cx<float> v) {
        if (kz0 + p < g.nKz) {
            dst[(size_t)i * g.ldz + p] = v;
            m = fmaxf(m, fabsf(v.re) + fabsf(v.im));
        }
    };
    if constexpr (NN > 0) col_ct<NN, true, CP, CP, 0, 1>(buf + NN * CP, buf, 1, tw, ld, st);   // two stages use buf only
    else col_rt<true, CP, CP>(buf + N * CP, buf, N, g.rad, g.nrad, 1, tw, ld, st);
    if (fmax2 && fd.out16 >= 0) block_max_to(fmax2 + fd.out16, m);
}

// Pass 3 for run-time sizes: CP consecutive lines (of all n^2), lanes along k for the
// loads and along m for the stores (row stride CP + 1: no conflicts either way).
template <int MODE>
__global__ void __launch_bounds__(256) k_pass3g(FftGeom g, const cx<float>* __restrict__ t2, size_t t2_stride,
                                                const cx<float>* __restrict__ tw, const FieldDesc* __restrict__ fields,
                                                float* __restrict__ out, size_t out_stride, uint32_t* __restrict__ hi,
                                                int split, const unsigned* __restrict__ fmax2, FieldLayout lay) {
    constexpr int SP = CP + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = g.n, M = N / 2, nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    cx<float>* buf = reinterpret_cast<cx<float>*>(smem_raw);
    const FieldDesc fd = fields[blockIdx.y];
    const int nKz = g.nKz, nk = field_ext(fd, g) + 1;   // f_z read: 0 .. nk - 1
    const size_t line0 = (size_t)blockIdx.x * CP, lines = (size_t)N * N;
    for (int p = warp; p < CP; p += nw) {
        const cx<float>* h = t2 + (size_t)blockIdx.y * t2_stride + (line0 + p) * g.ldz;
        for (int k = lane; k < M; k += 32) {
            cx<float> z = {0.f, 0.f};
            if (line0 + p < lines) {
                cx<float> a = {0.f, 0.f}, b = {0.f, 0.f};
                if (k < nk) a = h[k];
                if (M - k < nk) b = h[M - k];
                if (k == 0) { a.im = 0.f; b.im = 0.f; }   // H_0 and H_M: real parts only
                const cx<float> bc = {b.re, -b.im};
                const cx<float> s = radd(a, bc), d = rsub(a, bc), dw = rmul(d, tw[k]);
                z = radd(s, cx<float>{-dw.im, dw.re});
            }
            buf[k * SP + p] = z;
        }
    }
    __syncthreads();
    auto none_ld = [](int, int) { return cx<float>{0.f, 0.f}; };
    auto none_st = [](int, int, cx<float>) {};
    const cx<float>* res = col_rt<false, SP, CP>(buf, buf + M * SP, M, g.rad_h, g.nrad_h, 2, tw, none_ld, none_st);
    float sc = 1.f, s7 = 1.f;   // as in k_pass3v
    if (MODE != P3_FIELD) {
        const float bound = 2.f * (float)nKz * __uint_as_float(fmax2[fd.out16]);
        sc = pow2_scale(bound);
        s7 = pow2_scale(bound, 7);
    }
    const int r32 = fd.out32 & 7, r16 = fd.out16 & 7;
    uint32_t* q = MODE != P3_FIELD ? hi + (size_t)(fd.out16 >> 3) * 512 + (size_t)r16 * 32 : nullptr;
    for (int p = warp; p < CP; p += nw) {
        if (line0 + p >= lines) break;
        for (int m = lane; m < M; m += 32) {
            const cx<float> v = res[m * SP + p];
            const size_t pos = (line0 + p) * M + m;   // complex values: pairs of consecutive z
            if (MODE == P3_FIELD) {
                reinterpret_cast<cx<float>*>(out + (size_t)fd.out32 * out_stride)[pos] = v;
                continue;
            }
            const size_t kb = pos >> 5;
            const int w = (int)(pos & 31);
            if (fd.out32 >= 0)
                (reinterpret_cast<cx<float>*>(out) + (size_t)fd.out32 * 32)[kb * (size_t)(lay.rows32 * 32) + (w ^ (2 * r32))] =
                    cx<float>{v.re * s7, v.im * s7};
            uint32_t hw, lw;
            split_pair<MODE>(v.re * sc, v.im * sc, hw, lw);
            uint32_t* d = q + kb * (size_t)(lay.groups16 * 512) + (w ^ (4 * r16));
            d[0] = hw;
            if (split) d[256] = lw;
        }
    }
}

// FP64 (the unit fields of the counts): the shared-memory kernels above.
template <int NN>
cudaError_t launch_n(const FftGeom& g, const cx<float>* delta, const int16_t* shell_of, const float* radial,
                     const FieldDesc* d_fields, int nfields, const cx<double>* tw, cx<double>* t1, cx<double>* t2,
                     double* out, size_t out_stride, uint32_t*, uint32_t*, int, unsigned*, cudaStream_t st, FieldLayout) {
    constexpr int P = 4, P3 = 8;
    const int N = g.n, M = N / 2;
    const size_t t1_stride = (size_t)g.nK * N * g.ldz, t2_stride = (size_t)N * N * g.ldz;
    const size_t sm12 = sizeof(cx<double>) * ((size_t)N + 2 * (size_t)smem_elems<true, P>(N));
    const size_t sm3 = sizeof(cx<double>) * ((size_t)N + 2 * (size_t)smem_elems<false, P3>(M));
    static SmemLimit limit12, limit3;
    cudaError_t e;
    if ((e = raise_smem(limit12, sm12, k_pass1<double, P, NN>, k_pass2<double, P, NN>)) != cudaSuccess ||
        (e = raise_smem(limit3, sm3, k_pass3<double, P3, NN>)) != cudaSuccess)
        return e;
    const int nkzb = (g.nKz + P - 1) / P;
    k_pass1<double, P, NN><<<dim3(g.nK * nkzb, nfields), NTHR, sm12, st>>>(g, delta, shell_of, radial, d_fields, tw, t1,
                                                                           t1_stride);
    k_pass2<double, P, NN><<<dim3(N * nkzb, nfields), NTHR, sm12, st>>>(g, t1, t1_stride, tw, t2, t2_stride,
                                                                        d_fields);
    k_pass3<double, P3, NN><<<dim3(N * ((N + P3 - 1) / P3), nfields), NTHR, sm3, st>>>(g, t2, t2_stride, tw, d_fields, out,
                                                                                       out_stride);
    return cudaGetLastError();
}

// Threads for `items` butterflies of a CTA's largest stage, 64 .. 256.
inline int col_threads(int items) { return std::min(256, std::max(64, (items + 31) / 32 * 32)); }

template <int NN>
cudaError_t launch_n(const FftGeom& g, const cx<float>* delta, const int16_t* shell_of, const float* radial,
                     const FieldDesc* d_fields, int nfields, const cx<float>* tw, cx<float>* t1, cx<float>* t2, float* out,
                     size_t out_stride, uint32_t* hi, uint32_t* lo, int f16, unsigned* fmax2, cudaStream_t st,
                     FieldLayout lay) {
    const int N = g.n, M = N / 2;
    const size_t t1_stride = (size_t)g.nK * N * g.ldz, t2_stride = (size_t)N * N * g.ldz;
    cudaError_t e;
    if constexpr (NN == 512) {
        static SmemLimit limit;
        if ((e = raise_smem(limit, p2r_smem_bytes(), k_pass1r, k_pass2r)) != cudaSuccess) return e;
        const int nkzb = (g.nKz + P2R - 1) / P2R;
        k_pass1r<<<dim3(g.nK * nkzb, nfields), NTHR, p2r_smem_bytes(), st>>>(g, delta, shell_of, radial, d_fields, tw, t1,
                                                                             t1_stride);
        k_pass2r<<<dim3(N * nkzb, nfields), NTHR, p2r_smem_bytes(), st>>>(g, t1, t1_stride, tw, t2, t2_stride, d_fields,
                                                                          fmax2);
    } else {
        const int nrad = NN ? radix_list(NN).n : g.nrad, rad0 = NN ? radix_list(NN).r[0] : g.rad[0];
        const size_t sm = sizeof(cx<float>) * (size_t)N * CP * (nrad > 2 ? 2 : 1);   // two stages: one buffer
        static SmemLimit limit;
        if ((e = raise_smem(limit, sm, k_col1<NN>, k_col2<NN>)) != cudaSuccess) return e;
        const int nkzb = (g.nKz + CP - 1) / CP, thr = col_threads(N / rad0 * CP);
        k_col1<NN><<<dim3(g.nK * nkzb, nfields), thr, sm, st>>>(g, delta, shell_of, radial, d_fields, tw, t1, t1_stride);
        k_col2<NN><<<dim3(N * nkzb, nfields), thr, sm, st>>>(g, t1, t1_stride, tw, t2, t2_stride, d_fields, fmax2);
    }
    const bool kbm = lay.groups16 > 0;
    if constexpr (NN > 0) {
        using V = P3V<NN>;
        auto kern = !kbm ? k_pass3v<NN, P3_FIELD> : f16 ? k_pass3v<NN, P3_F16> : k_pass3v<NN, P3_BF16>;
        kern<<<dim3((unsigned)((size_t)N * N / V::P), nfields), V::T, V::smem(), st>>>(
            g, t2, t2_stride, tw, d_fields, out, out_stride, hi, lo != nullptr, fmax2, lay);
    } else {
        auto kern = !kbm ? k_pass3g<P3_FIELD> : f16 ? k_pass3g<P3_F16> : k_pass3g<P3_BF16>;
        const size_t sm = sizeof(cx<float>) * 2 * (size_t)M * (CP + 1);
        static SmemLimit limit[3];
        if ((e = raise_smem(limit[!kbm ? 0 : f16 ? 1 : 2], sm, kern)) != cudaSuccess) return e;
        kern<<<dim3((unsigned)(((size_t)N * N + CP - 1) / CP), nfields), col_threads(M * CP / 4), sm, st>>>(
            g, t2, t2_stride, tw, d_fields, out, out_stride, hi, lo != nullptr, fmax2, lay);
    }
    return cudaGetLastError();
}


// ---------------------------------------------------------------------------
// Density input stage: cloud-in-cell with interlacing, then a forward
// real-to-complex 3-D FFT of both grids, combined into delta(k).  The
// forward transforms reuse the inverse Stockham stages through
// FFT(x) = conj(IFFT(conj x)).
// ---------------------------------------------------------------------------

// Two consecutive z cells, g[i] += w0 and g[i + 1] += w1, as one 16-byte reduction unless
// they straddle a 16-byte boundary (the other two words get + 0).
__device__ __forceinline__ void cic_add2(float* g, size_t i, float w0, float w1) {
    const int q = (int)(i & 3);
    if (q == 3) {
        atomicAdd(g + i, w0);
        atomicAdd(g + i + 1, w1);
        return;
    }
    const float a = q == 0 ? w0 : 0.f, b = q == 1 ? w0 : q == 0 ? w1 : 0.f, c = q == 2 ? w0 : q == 1 ? w1 : 0.f,
                d = q == 2 ? w1 : 0.f;
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(g + (i - q)), "f"(a), "f"(b), "f"(c), "f"(d)
                 : "memory");
}

__device__ __forceinline__ void cic_deposit(float* g, int n, const int (&b)[3], const float (&t)[3]) {
    const int ix[2] = {b[0], b[0] + 1 == n ? 0 : b[0] + 1}, iy[2] = {b[1], b[1] + 1 == n ? 0 : b[1] + 1};
    const float wx[2] = {1.f - t[0], t[0]}, wy[2] = {1.f - t[1], t[1]}, wz0 = 1.f - t[2], wz1 = t[2];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float w = wx[c >> 1] * wy[c & 1];
        const size_t row = ((size_t)ix[c >> 1] * n + iy[c & 1]) * n;
        if (b[2] + 1 < n) {
            cic_add2(g, row + b[2], w * wz0, w * wz1);
        } else {
            atomicAdd(g + row + b[2], w * wz0);
            atomicAdd(g + row, w * wz1);
        }
    }
}

// CIC weights of every particle on grid 1 (cells at j H) and grid 2 (cells at
// (j + 1/2) H).  Cell units u = p n / box to ~2^-46 as an FP32 pair (p times the pair
// sh + sl), far below the 2^-25 to which the weights round their fraction; positions
// outside [0, box) take FP64 and the wrap.  4 Mi particles on 256^3: 172 us, bound by the
// way of the reductions, 4 to 8 a particle and grid, through L1 (77 % busy) and L2 (60 %) (FP64 with two divisions a coordinate and
// 16 scalar additions a particle: 722 us).
__global__ void k_cic(const float* __restrict__ pos, long long np, int n, double scale, float sh, float sl,
                      float* __restrict__ g1, float* __restrict__ g2) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < np;
         i += (long long)gridDim.x * blockDim.x) {
        int b1[3], b2[3];
        float t1[3], t2[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float p = pos[3 * i + a];
            const float h = __fmul_rn(p, sh);
            if (h >= 0.f && h < (float)n) {
                const float l = __fmaf_rn(p, sl, __fmaf_rn(p, sh, -h));   // u = h + l
                const float fl = floorf(h), f = __fsub_rn(h, fl);
                // grid 1: cell fl and fraction f + l, one cell back or on where l crosses it
                float t = __fadd_rn(f, l);
                int c = (int)fl;
                if (t < 0.f) {
                    t = __fadd_rn(__fadd_rn(f, 1.f), l);
                    --c;
                } else if (t > 1.f) {
                    t = __fadd_rn(__fsub_rn(f, 1.f), l);
                    ++c;
                }
                b1[a] = c < 0 ? c + n : c >= n ? c - n : c;
                t1[a] = t;
                // grid 2: u - 1/2
                c = (int)fl;
                t = __fadd_rn(__fsub_rn(f, 0.5f), l);
                if (t < 0.f) {
                    t = __fadd_rn(__fadd_rn(f, 0.5f), l);
                    --c;
                }
                b2[a] = c < 0 ? c + n : c;
                t2[a] = t;
            } else {
#pragma unroll
                for (int gs = 0; gs < 2; ++gs)
                    cic_wrap((double)p * scale - 0.5 * gs, n, (gs ? b2 : b1)[a], (gs ? t2 : t1)[a]);
            }
        }
        cic_deposit(g1, n, b1, t1);
        cic_deposit(g2, n, b2, t2);
    }
}

// exp(+2 pi i t / n), t < n, from FP64 sincospi.
__global__ void k_twiddles(int n, cx<float>* __restrict__ tw) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    double s, c;
    sincospi(2.0 * (double)t / (double)n, &s, &c);
    tw[t] = cx<float>{(float)c, (float)s};
}

// z pass: P real lines (x fixed, y0 .. y0 + P - 1) of grid blockIdx.y (or,
// with msub > 0, of the sub-cube blockIdx.y of side n of a grid of side
// nfull cut into msub^3 cubes), with
// delta = a g + b applied on load, packed as z_m = d_{2m} + i d_{2m+1}; an
// M = n/2-point FFT gives Z; X_k = E_k + e^{-2 pi i k/n} O_k with
// E_k = (Z_k + conj Z_{M-k})/2, O_k = (Z_k - conj Z_{M-k})/(2i), k = 0 .. M.
// Lines side by side as in k_col1 (P consecutive of all n^2; lanes along z for the
// loads, along k for the stores; 64 lines of 32 points, 16 of 128, so that a stage has
// work for every thread).  Eight lines on 256 threads before: 512 sub-cubes of 64^3 z
// 550 -> 377 us, y and x 1 064 -> 349 together (the x pass takes its lines (y, k_z) from
// one run, so 33 k_z leave no idle lanes there); two grids of 256^3 y and x 224 -> 92.
template <int NN>
constexpr int fwd_lines() { return NN == 0 || NN >= 256 ? CP : NN >= 128 ? 32 : 64; }

template <int NN, bool SQ = false>
__global__ void __launch_bounds__(256) k_fwd_z(FftGeom g, const float* __restrict__ grid, size_t gstride, float a,
                                               float b, const cx<float>* __restrict__ tw, cx<float>* __restrict__ T,
                                               size_t tstride, int msub = 0, int nfull = 0) {
    constexpr int P = fwd_lines<NN>(), SP = P + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = NN ? NN : g.n, M = N / 2, H = M + 1;
    const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    cx<float>* buf = reinterpret_cast<cx<float>*>(smem_raw);
    const size_t line0 = (size_t)blockIdx.x * P, lines = (size_t)N * N;
    const float* src = grid + (size_t)blockIdx.y * gstride;
    size_t sx = (size_t)N * N, sy = (size_t)N;   // element strides of x and y in the source
    if (msub > 0) {
        const int c = blockIdx.y, cx_ = c / (msub * msub), cy = (c / msub) % msub, cz = c % msub;
        sx = (size_t)nfull * nfull;
        sy = (size_t)nfull;
        src = grid + (size_t)cx_ * N * sx + (size_t)cy * N * sy + (size_t)cz * N;
    }
    for (int p = warp; p < P; p += nw) {
        const int l = (int)(line0 + p), x = l / N, y = l - x * N;
        const bool live = line0 + p < lines;
        const float* row = src + (size_t)x * sx + (size_t)y * sy;
        for (int m = lane; m < M; m += 32) {
            cx<float> v = {0.f, 0.f};
            if (live) {
                const float2 r = *reinterpret_cast<const float2*>(row + 2 * m);
                const float r0 = SQ ? r.x * r.x : r.x, r1 = SQ ? r.y * r.y : r.y;
                v = cx<float>{a * r0 + b, -(a * r1 + b)};   // conjugated
            }
            buf[m * SP + p] = v;
        }
    }
    __syncthreads();
    auto none_ld = [](int, int) { return cx<float>{0.f, 0.f}; };
    auto none_st = [](int, int, cx<float>) {};
    const cx<float>* res;
    if constexpr (NN > 0) res = col_ct<NN / 2, false, SP, P, 0, 1>(buf, buf + M * SP, 2, tw, none_ld, none_st);
    else res = col_rt<false, SP, CP>(buf, buf + M * SP, M, g.rad_h, g.nrad_h, 2, tw, none_ld, none_st);
    cx<float>* dst = T + (size_t)blockIdx.y * tstride + line0 * H;
    for (int p = warp; p < P; p += nw) {
        if (line0 + p >= lines) break;
        for (int k = lane; k < H; k += 32) {
            const cx<float> rk = res[(k == M ? 0 : k) * SP + p], rm = res[(k == 0 ? 0 : M - k) * SP + p];
            const cx<float> zk = {rk.re, -rk.im}, czm = {rm.re, rm.im};   // Z_k, conj Z_{M-k}
            const cx<float> E = cscale(cadd(zk, czm), 0.5f);
            const cx<float> D = cscale(csub(zk, czm), 0.5f);
            const cx<float> O = {D.im, -D.re};                               // D / i
            const cx<float> w = {tw[k].re, -tw[k].im};                       // e^{-2 pi i k/n}
            dst[(size_t)p * H + k] = cadd(E, cmul(w, O));
        }
    }
}

// y or x pass, in place: P consecutive of the L lines of row o of grid blockIdx.y,
// element j of line l at o * so + j * sj + l (y: the n/2 + 1 lines k_z of one x; x: all
// the lines (y, k_z)).
template <int NN, int P>
__global__ void __launch_bounds__(256) k_fwd_axis(FftGeom g, const cx<float>* __restrict__ tw, cx<float>* T,
                                                  size_t tstride, size_t so, size_t sj, int L) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = NN ? NN : g.n;
    cx<float>* buf = reinterpret_cast<cx<float>*>(smem_raw);
    const int nlb = (L + P - 1) / P;
    const int o = blockIdx.x / nlb, l0 = (blockIdx.x % nlb) * P;
    cx<float>* t = T + (size_t)blockIdx.y * tstride + (size_t)o * so + l0;
    auto ld = [&](int i, int p) {
        cx<float> v = {0.f, 0.f};
        if (l0 + p < L) {
            const cx<float> u = t[(size_t)i * sj + p];
            v = cx<float>{u.re, -u.im};
        }
        return v;
    };
    auto st = [&](int i, int p, cx<float> v) {
        if (l0 + p < L) t[(size_t)i * sj + p] = cx<float>{v.re, -v.im};
    };
    if constexpr (NN > 0) col_ct<NN, true, P, P, 0, 1>(buf + NN * P, buf, 1, tw, ld, st);
    else col_rt<true, P, P>(buf + N * P, buf, N, g.rad, g.nrad, 1, tw, ld, st);
}

// y and x passes, P lines a CTA.
template <int NN, int P>
cudaError_t launch_fwd_axes(const FftGeom& g, const cx<float>* tw, cx<float>* T, int nb, cudaStream_t st) {
    const int N = g.n, H = N / 2 + 1;
    const size_t tstride = (size_t)N * N * H;
    const int nrad = NN ? radix_list(NN).n : g.nrad, rad0 = NN ? radix_list(NN).r[0] : g.rad[0];
    const size_t sm = sizeof(cx<float>) * (size_t)N * P * (nrad > 2 ? 2 : 1);   // two stages: one buffer
    static SmemLimit limit;
    const cudaError_t e = raise_smem(limit, sm, k_fwd_axis<NN, P>);
    if (e != cudaSuccess) return e;
    const int t = col_threads(N / rad0 * P);
    k_fwd_axis<NN, P><<<dim3(N * ((H + P - 1) / P), nb), t, sm, st>>>(g, tw, T, tstride, (size_t)N * H, (size_t)H, H);
    k_fwd_axis<NN, P><<<dim3((N * H + P - 1) / P, nb), t, sm, st>>>(g, tw, T, tstride, 0, (size_t)N * H, N * H);
    return cudaGetLastError();
}

// The three forward passes of nb grids (z with a g + b on load, or of a g^2).
template <int NN, bool SQ>
cudaError_t launch_fwd(const FftGeom& g, const float* grid, size_t gstride, float a, float b, const cx<float>* tw,
                       cx<float>* T, int nb, int msub, int nfull, cudaStream_t st) {
    constexpr int P = fwd_lines<NN>();
    const int N = g.n, M = N / 2, H = M + 1;
    const size_t smz = sizeof(cx<float>) * 2 * (size_t)M * (P + 1);
    static SmemLimit limitz;
    const cudaError_t e = raise_smem(limitz, smz, k_fwd_z<NN, SQ>);
    if (e != cudaSuccess) return e;
    const int rz = NN ? radix_list(NN / 2).r[0] : 4;
    k_fwd_z<NN, SQ><<<dim3((unsigned)(((size_t)N * N + P - 1) / P), nb), col_threads(M / rz * P), smz, st>>>(
        g, grid, gstride, a, b, tw, T, (size_t)N * N * H, msub, nfull);
    // 16 lines of more than 896 points and three stages do not fit shared memory twice
    if (NN == 0 && N > 896) return launch_fwd_axes<NN, NN ? CP : CP / 2>(g, tw, T, nb, st);
    return launch_fwd_axes<NN, CP>(g, tw, T, nb, st);
}

// delta(k) = (V/n^3) [X1(k) + e^{-i pi (n_x+n_y+n_z)/n} X2(k)] / (2 W(k)),
// W = prod_a sinc^2(pi n_a / n).
__global__ void k_fwd_combine(int N, const cx<float>* __restrict__ T1, const cx<float>* __restrict__ T2, float scale,
                              cx<float>* __restrict__ out) {
    const int H = N / 2 + 1;
    const size_t total = (size_t)N * N * H;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int kz = (int)(i % H), y = (int)((i / H) % N), x = (int)(i / ((size_t)H * N));
        const int fx = x < N / 2 ? x : x - N, fy = y < N / 2 ? y : y - N, fz = kz == N / 2 ? -(N / 2) : kz;
        float s, c;
        sincospif(-(float)(fx + fy + fz) / (float)N, &s, &c);
        float W = 1.f;
        const int f3[3] = {fx, fy, fz};
#pragma unroll
        for (int a = 0; a < 3; ++a)
            if (f3[a] != 0) {
                const float u = (float)f3[a] / (float)N;
                const float sc = sinpif(u) / (3.14159265358979f * u);
                W *= sc * sc;
            }
        const cx<float> a1 = T1[i], a2 = T2[i];
        const cx<float> ph = {c, s};
        out[i] = cscale(cadd(a1, cmul(ph, a2)), 0.5f * scale / W);
    }
}

template <int NN>
cudaError_t launch_density_n(const FftGeom& g, const float* pos, long long np, double box, char* ws,
                             cx<float>* out, cudaStream_t st) {
    const int N = g.n, H = N / 2 + 1;
    const DensityLayout L = density_layout(N);
    cx<float>* tw = reinterpret_cast<cx<float>*>(ws + L.tw);
    float* grids = reinterpret_cast<float*>(ws + L.grids);
    cx<float>* T = reinterpret_cast<cx<float>*>(ws + L.spec);
    const size_t gstride = (size_t)N * N * N, tstride = (size_t)N * N * H;
    cudaError_t e;
    if ((e = cudaMemsetAsync(grids, 0, 2 * gstride * sizeof(float), st)) != cudaSuccess) return e;
    k_twiddles<<<(N + 255) / 256, 256, 0, st>>>(N, tw);
    const int cic_blocks = (int)std::min<long long>(4096, (np + 255) / 256);
    const double scale = (double)N / box;
    const float sh = (float)scale, sl = (float)(scale - (double)sh);
    k_cic<<<cic_blocks, 256, 0, st>>>(pos, np, N, scale, sh, sl, grids, grids + gstride);
    // delta_g = count / (N_p / n^3) - 1
    const float a = (float)((double)gstride / (double)np);
    if ((e = launch_fwd<NN, false>(g, grids, gstride, a, -1.f, tw, T, 2, 0, 0, st)) != cudaSuccess) return e;
    const double V = box * box * box;
    k_fwd_combine<<<4096, 256, 0, st>>>(N, T, T + tstride, (float)(V / (double)gstride), out);
    return cudaGetLastError();
}
}  // namespace

// Sizes of the workloads get kernels specialised at compile time; any other
// supported size runs the same kernels with run-time radix lists.
template <typename R>
cudaError_t launch_fft_fields(const FftGeom& g, const cx<float>* delta, const int16_t* shell_of,
                              const float* radial, const FieldDesc* d_fields, int nfields,
                              const cx<R>* tw, cx<R>* t1, cx<R>* t2, R* out, size_t out_stride,
                              uint32_t* hi, uint32_t* lo, int f16, unsigned* fmax2, cudaStream_t st,
                              FieldLayout lay) {
#define BSP_FFT_CASE(NV) \
    case NV:             \
        return launch_n<NV>(g, delta, shell_of, radial, d_fields, nfields, tw, t1, t2, out, out_stride, hi, lo, f16, \
                            fmax2, st, lay);
    switch (g.n) {
        BSP_FFT_CASE(64)
        BSP_FFT_CASE(96)
        BSP_FFT_CASE(128)
        BSP_FFT_CASE(160)
        BSP_FFT_CASE(256)
        BSP_FFT_CASE(512)
        default:
            return launch_n<0>(g, delta, shell_of, radial, d_fields, nfields, tw, t1, t2, out, out_stride, hi, lo, f16,
                               fmax2, st, lay);
    }
#undef BSP_FFT_CASE
}

template cudaError_t launch_fft_fields<float>(const FftGeom&, const cx<float>*, const int16_t*, const float*,
                                              const FieldDesc*, int, const cx<float>*, cx<float>*,
                                              cx<float>*, float*, size_t, uint32_t*, uint32_t*, int, unsigned*,
                                              cudaStream_t, FieldLayout);
DensityLayout density_layout(int n) {
    auto r256 = [](size_t b) { return (b + 255) / 256 * 256; };
    DensityLayout L{};
    const size_t n3 = (size_t)n * n * n, nh = (size_t)n * n * (n / 2 + 1);
    L.tw = 0;
    L.grids = r256(sizeof(cx<float>) * (size_t)n);
    L.spec = L.grids + r256(2 * n3 * sizeof(float));
    L.end = L.spec + r256(2 * nh * sizeof(cx<float>));
    return L;
}

cudaError_t launch_forward_square(const FftGeom& g, const float* x, float a, const cx<float>* tw, cx<float>* T,
                                  cudaStream_t st) {
    switch (g.n) {
        case 64: return launch_fwd<64, true>(g, x, 0, a, 0.f, tw, T, 1, 0, 0, st);
        case 96: return launch_fwd<96, true>(g, x, 0, a, 0.f, tw, T, 1, 0, 0, st);
        case 128: return launch_fwd<128, true>(g, x, 0, a, 0.f, tw, T, 1, 0, 0, st);
        case 160: return launch_fwd<160, true>(g, x, 0, a, 0.f, tw, T, 1, 0, 0, st);
        case 256: return launch_fwd<256, true>(g, x, 0, a, 0.f, tw, T, 1, 0, 0, st);
        case 512: return launch_fwd<512, true>(g, x, 0, a, 0.f, tw, T, 1, 0, 0, st);
        default: return launch_fwd<0, true>(g, x, 0, a, 0.f, tw, T, 1, 0, 0, st);
    }
}

cudaError_t launch_forward_subcubes(const FftGeom& g, int nfull, int m, const float* x, float a, cx<float>* tw,
                                    cx<float>* T, cudaStream_t st) {
    if (m < 1 || m * g.n != nfull || m * m * m > 65535) return cudaErrorInvalidValue;
    const int nc = m * m * m;
    k_twiddles<<<(g.n + 255) / 256, 256, 0, st>>>(g.n, tw);
    switch (g.n) {
        case 64: return launch_fwd<64, false>(g, x, 0, a, 0.f, tw, T, nc, m, nfull, st);
        case 128: return launch_fwd<128, false>(g, x, 0, a, 0.f, tw, T, nc, m, nfull, st);
        default: return launch_fwd<0, false>(g, x, 0, a, 0.f, tw, T, nc, m, nfull, st);
    }
}

cudaError_t launch_density(const FftGeom& g, const float* pos, long long np, double box, void* ws,
                           cx<float>* out, cudaStream_t st) {
    char* w = reinterpret_cast<char*>(ws);
    switch (g.n) {
        case 64: return launch_density_n<64>(g, pos, np, box, w, out, st);
        case 96: return launch_density_n<96>(g, pos, np, box, w, out, st);
        case 128: return launch_density_n<128>(g, pos, np, box, w, out, st);
        case 160: return launch_density_n<160>(g, pos, np, box, w, out, st);
        case 256: return launch_density_n<256>(g, pos, np, box, w, out, st);
        case 512: return launch_density_n<512>(g, pos, np, box, w, out, st);
        default: return launch_density_n<0>(g, pos, np, box, w, out, st);
    }
}

template cudaError_t launch_fft_fields<double>(const FftGeom&, const cx<float>*, const int16_t*, const float*,
                                               const FieldDesc*, int, const cx<double>*, cx<double>*,
                                               cx<double>*, double*, size_t, uint32_t*, uint32_t*, int,
                                               unsigned*, cudaStream_t, FieldLayout);

}  // namespace bsp
