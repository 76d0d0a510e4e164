// segment.cu -- overlap-save transforms for lags and kernels much shorter than
// the image.
//
// The build needs circular correlations of the weighted images only at lags
// |rho| <= 2w, and the subtraction convolves with kernels of half-width w.
// Both are sums over short segments: with a(x) restricted to a core of C
// samples and b taken on a window of C + 2h samples around it, the circular
// correlation of window length equals the image's at every |rho| <= h, for any
// image length (the window wraps around the image edge).
//   * k_lagx: the lag sums along x of every spectrum product, at one frequency
//     column.  The window's DFT (length 128) of every sequence is formed per
//     segment, the products are summed over the segments in the frequency
//     domain, and one short inverse DFT per product gives all lags: no
//     transform of the whole column, and no stored column spectra.
//   * k_rows_seg, k_rows_inv_seg: the row transforms (along y) of a row length
//     that is not a power of two, as transforms of length 256 over segments of
//     the row.  A segment's frequencies are further columns of the row
//     transform table: column c = segment * 129 + m.
#include <cuda_runtime.h>

#include <type_traits>
#include <utility>

#include "common.cuh"
#include "fft.cuh"
#include "fft16.cuh"
#include "internal.h"

namespace sfft {

// ---------------------------------------------------------------------------
// Lag sums along x.  One block per frequency column c.
//
// For n_K = NK kernel terms the sequences are NK "core" ones (a: the weighted
// column on the segment's core, zero outside) and NK + 1 "window" ones (b:
// the terms and S on the whole window).  A warp transforms four segments of
// one sequence, eight lanes of 16 values per transform: a radix-16 pass in
// registers, an exchange through the transform's own row of shared memory
// (rows of 9, transform stride 152: no bank conflicts) and two radix-8 passes.
// Then thread (k, role) adds the products of bin k over its segments to
// register sums.  At the end Z_p(k), k < 128, of product p is inverted in two
// steps, k = c + 16 r: Y_c(s) = sum_r Z(c + 16 r) e^(2 pi i r s / 8), and
// Q(rho) = sum_c e^(2 pi i c rho / 128) Y_c(rho mod 8).
//
// Accuracy, FP32 (error of the difference image against 64 bits; the column FFT
// and the direct lag sums that these took the place of are "before"):
//   * Roundings of the inverse are white over the bins and so hide the weak high
//     frequencies, where M's small eigenvalues are.  It is taken in integers (30
//     bits of Z, 64-bit sums) and leaves one rounding, that of the stored Q.
//   * Rounded twiddles and constants act like one filter in every column and
//     segment, so their effect does not average out.  Columns take turns in eight
//     roundings of each (LagTab) whose mean is right; what is left of the error
//     alternates with the column and lands at lags of an eighth of the row.
//     Without it the coefficients' error doubles (1024 x 1024, 3 terms, w = 6: 5.6e-6
//     and 1.1e-5; before 5.6e-6).
//   * In each bin the sum over segments runs over terms of that bin's own size:
//     compensated sums changed no error by more than 2 %.
// 4096 x 4096, w = 8: 8.8e-6 before, 7.9e-6 with an FP32 inverse and rounded twiddles,
// 6.9e-6 (342 -> 357 us, most of it the integer inverse); 1501 x 1024, w = 5: 2.4e-6
// before, 3.8e-6, 2.5e-6.
//
// The core's halos are zero and the window's hold the wrapped image, so the
// segments need no special case at the image edge and any n0 serves.  The
// windows of a batch come by asynchronous copies that run during the product
// sums of the batch before.  Bound by shared-memory traffic and instruction issue
// (73 % of the shared-memory data pipe, 65 % of the issue slots, 25 warps per
// multiprocessor), not by HBM (the row transforms are read once).  Against the column FFT and gather it
// replaced (w0 = 8, 6 terms, 4096 x 4096, FP32): 630 -> 357 us; against direct
// lag sums (2046 columns of x, w0 = 6): 2250 -> 230 us.
// Window 128: a longer one (256) has fewer halo samples but twice the
// exchange per transform; the lags need 4 w0 < 128.
//
// The DC bin of column m = 0 (the sky's square, which cancels in every
// difference of Eq. B5/B7/B13) is removed by centring both sequences there.
constexpr int kLagL = kLagLen;  // window length
constexpr int kLagRow = 152;  // elements of shared memory per transform (16 rows of 9, 8 mod 16)
constexpr int kLagWin = 136;  // elements per staged window (8 mod 16)

// Per block: segments per batch, threads (8 per transform), and three roles of
// 128 threads for the product sums.  With 6 terms the 27 products are split
// over the roles, 9 each (18 registers of sums; all 27 in one thread would
// spill at two blocks per SM); with fewer terms a thread takes all products
// and the roles split the segments.
template <int NK>
struct LagShape {
    static constexpr int kSeg = NK == 1 ? 16 : 4;
    static constexpr int kSeq = 2 * NK + 1;
    static constexpr int kThreads = kSeg * kSeq * 8;
    static constexpr int kRoles = NK == 3 ? 1 : 3;
    static constexpr int kPairs = NK * (NK + 1) / 2 + NK;
    static constexpr bool kSplitPairs = NK == 6;
    static constexpr int kOwn = kSplitPairs ? kPairs / kRoles : kPairs;  // products per thread
    static_assert(kThreads >= kRoles * kLagL, "a thread per bin and role");
};

// products (a, q), q = NK: Theta, in the order a = 0: q = 0..NK, a = 1: q = 1..NK, ...
template <int NK>
__host__ __device__ constexpr int lag_pair_a(int p) {
    int a = 0;
    while (p >= NK + 1 - a) {
        p -= NK + 1 - a;
        ++a;
    }
    return a;
}
template <int NK>
__host__ __device__ constexpr int lag_pair_q(int p) {
    int a = 0;
    while (p >= NK + 1 - a) {
        p -= NK + 1 - a;
        ++a;
    }
    return a + p;
}

// acc[i] += the products FIRST + i of one bin of one segment (sp: the bin in
// the first core sequence; sequences are `stride` apart).  Every index is a
// template argument, so that the sums stay in registers.
template <typename T, int NK, int FIRST, int OWN, int... I>
__device__ __forceinline__ void lag_products(cpx<T> (&acc)[OWN], const cpx<T> *sp, size_t stride,
                                             std::integer_sequence<int, I...>) {
    constexpr int a0 = lag_pair_a<NK>(FIRST), a1 = lag_pair_a<NK>(FIRST + OWN - 1);
    cpx<T> a[NK], b[NK + 1];
#pragma unroll
    for (int q = a0; q <= NK; ++q) b[q] = sp[(NK + q) * stride];
#pragma unroll
    for (int q = a0; q <= a1; ++q) a[q] = conj(sp[q * stride]);
    ((acc[I] = cfma(acc[I], a[std::integral_constant<int, lag_pair_a<NK>(FIRST + I)>::value],
                    b[std::integral_constant<int, lag_pair_q<NK>(FIRST + I)>::value])),
     ...);
}

// Forward dft8 and dft16 (fft.cuh, fft16.cuh) with given cos(pi / 4), cos(pi /
// 8) and sin(pi / 8)
template <typename T>
struct LagConst {
    T c4, c8, s8;
};
template <typename T>
__device__ __forceinline__ void dft8c(cpx<T> (&v)[8], const LagConst<T> &k) {
    cpx<T> a[4], b[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        a[i] = v[i] + v[i + 4];
        b[i] = v[i] - v[i + 4];
    }
    b[1] = cmul(b[1], mk(k.c4, -k.c4));
    b[2] = mul_i(b[2], -1);
    b[3] = cmul(b[3], mk(-k.c4, -k.c4));
    dft4(a[0], a[1], a[2], a[3], -1);
    dft4(b[0], b[1], b[2], b[3], -1);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[2 * i] = a[i];
        v[2 * i + 1] = b[i];
    }
}
template <typename T>
__device__ __forceinline__ void dft16c(cpx<T> (&v)[16], const LagConst<T> &k) {
#pragma unroll
    for (int r = 0; r < 4; ++r) dft4(v[r], v[r + 4], v[r + 8], v[r + 12], -1);
    v[5] = cmul(v[5], mk(k.c8, -k.s8));
    v[9] = cmul(v[9], mk(k.c4, -k.c4));
    v[13] = cmul(v[13], mk(k.s8, -k.c8));
    v[6] = cmul(v[6], mk(k.c4, -k.c4));
    v[10] = mul_i(v[10], -1);
    v[14] = cmul(v[14], mk(-k.c4, -k.c4));
    v[7] = cmul(v[7], mk(k.s8, -k.c8));
    v[11] = cmul(v[11], mk(-k.c4, -k.c4));
    v[15] = cmul(v[15], mk(-k.c8, k.s8));
#pragma unroll
    for (int r = 0; r < 4; ++r) dft4(v[4 * r], v[4 * r + 1], v[4 * r + 2], v[4 * r + 3], -1);
}

// 8-point inverse DFT of integers up to 2^30 in magnitude, exact but for the
// products with cos(pi / 4) (30 bits); outputs up to 2^33.5, in the order 0, 2,
// 4, 6, 1, 3, 5, 7
using i64 = long long;
__device__ __forceinline__ void idft4(i64 (&re)[8], i64 (&im)[8], int o) {
    const i64 ar = re[o] + re[o + 2], ai = im[o] + im[o + 2], br = re[o] - re[o + 2], bi = im[o] - im[o + 2];
    const i64 cr = re[o + 1] + re[o + 3], ci = im[o + 1] + im[o + 3];
    const i64 er = re[o + 1] - re[o + 3], ei = im[o + 1] - im[o + 3];
    re[o] = ar + cr, im[o] = ai + ci;
    re[o + 1] = br - ei, im[o + 1] = bi + er;
    re[o + 2] = ar - cr, im[o + 2] = ai - ci;
    re[o + 3] = br + ei, im[o + 3] = bi - er;
}
__device__ __forceinline__ void idft8(i64 (&re)[8], i64 (&im)[8]) {
    auto cos4 = [](i64 v) { return (v * 759250125LL + (1LL << 29)) >> 30; };  // 2^30 cos(pi / 4)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const i64 ar = re[k], ai = im[k], br = re[k + 4], bi = im[k + 4];
        re[k] = ar + br, im[k] = ai + bi;
        re[k + 4] = ar - br, im[k + 4] = ai - bi;
    }
    i64 r = re[5], i = im[5];
    re[5] = cos4(r - i), im[5] = cos4(i + r);
    r = re[6], i = im[6];
    re[6] = -i, im[6] = r;
    r = re[7], i = im[7];
    re[7] = cos4(-r - i), im[7] = cos4(r - i);
    idft4(re, im, 0);
    idft4(re, im, 4);
}

template <int BYTES>
__device__ __forceinline__ void cp_async(void *smem, const void *gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)),
                 "l"(gmem), "n"(BYTES));
}

template <typename T, int NK>
__global__ void __launch_bounds__(LagShape<NK>::kThreads, sizeof(T) == 4 ? (NK == 3 ? 4 : 2) : 1)
    k_lagx(int n0, int hc, int ncol, int w0, int offb, int nfy, const cpx<T> *__restrict__ F,
           const T *__restrict__ fx, const LagTab<T> *__restrict__ tab, int norm, cpx<T> *__restrict__ Q) {
    using Sh = LagShape<NK>;
    constexpr int NP = Sh::kPairs, NSEQ = Sh::kSeq, SEG = Sh::kSeg;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cpx<T> *spec = reinterpret_cast<cpx<T> *>(smem_raw);     // [NSEQ * SEG][kLagRow]
    cpx<T> *raw = spec + (size_t)NSEQ * SEG * kLagRow;       // [row-transform sequences][SEG][kLagWin]
    const int nraw = offb + nfy + 1;
    T *wraw = reinterpret_cast<T *>(raw + (size_t)nraw * SEG * kLagWin);  // [nfy - 1][SEG][kLagWin]: xt^i, i >= 1
    __shared__ cpx<T> stp[kLagL];                         // exp(-2 pi i j g / 128) at 8 j + g (no bank conflicts)
    __shared__ T mean[NSEQ];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c = blockIdx.x;
    const int h = 2 * w0, core = kLagL - 2 * h;
    const size_t seqstride = (size_t)ncol * n0;
    const int dither = (c % hc) % LagTab<T>::kNum;
    for (int q = tid; q < kLagL; q += Sh::kThreads) stp[q] = tab->fwd[dither][(q >> 3) * (q & 7)];
    const LagConst<T> lc{tab->fwd[dither][16].re, tab->fwd[dither][8].re, -tab->fwd[dither][8].im};
    // Sequence q < NK: core ones, then NK + 1 window ones; its power of xt and
    // its row-transform sequence.
    auto sequence = [&](int q, int &ti, int &fsq) {
        const int t = q < NK ? q : q - NK;  // kernel term (t = NK: S)
        int tj = nfy;
        ti = 0;
        if (t < NK) term_ij(t, &ti, &tj);
        fsq = q < NK ? tj : offb + tj;
    };
    const int nseg = (n0 + core - 1) / core;
    // this thread's sequence and segment: eight threads a transform, the
    // segments of a sequence side by side.  In FP64, whose instructions take a
    // warp 64 cycles whatever the number of its lanes at work, a column of fewer
    // segments than a batch has packs its transforms (build
    // of 64 x 2000, 6 terms, w = 8: 1187 -> 963 us)
    const int per = sizeof(T) == 8 ? min(SEG, nseg) : SEG;
    const int sq = (tid >> 3) / per, sub = (tid >> 3) % per, g = lane & 7;
    const bool has = sq < NSEQ, is_core = sq < NK;
    int ti = 0, fsq = 0;
    if (has) sequence(sq, ti, fsq);
    cpx<T> *row = spec + (size_t)(sq * SEG + sub) * kLagRow;
    const bool centre = c % hc == 0;
    if (centre) {  // means of the sequences (real at m = 0), a warp each
        constexpr int kWarpsPerSeq = SEG / 4;
        if (warp % kWarpsPerSeq == 0) {
            const int q = warp / kWarpsPerSeq;
            int ti, fsq;
            sequence(q, ti, fsq);
            const cpx<T> *col = F + (size_t)fsq * seqstride + (size_t)c * n0;
            const T *wx = fx + (size_t)ti * n0;
            double a = 0.0;
            for (int x = lane; x < n0; x += 32) {
                const T v = col[x].re;
                a += (double)(ti > 0 ? v * wx[x] : v);
            }
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (lane == 0) mean[q] = (T)(a / n0);
        }
    }
    __syncthreads();
    const T mu = centre && has ? mean[sq] : (T)0;
    const int k = tid & (kLagL - 1), role = tid / kLagL;  // product sums: bin and role
    cpx<T> acc[Sh::kOwn];
#pragma unroll
    for (int p = 0; p < Sh::kOwn; ++p) acc[p] = mk((T)0, (T)0);
    const bool small = n0 < 2 * kLagL;  // windows may wrap more than once
    // asynchronous copies of a batch's windows (and the weights xt^i along
    // them) into shared memory, one window per warp and turn
    auto fetch = [&](int s0) {
        const int cnt = min(SEG, nseg - s0);
        for (int w = warp; w < (nraw + nfy - 1) * cnt; w += Sh::kThreads / 32) {
            const int sq = w / cnt, sb = w - sq * cnt;
            const int x0 = (s0 + sb) * core - h;
            const bool is_f = sq < nraw;
            const cpx<T> *src = F + (size_t)sq * seqstride + (size_t)c * n0;
            const T *wsrc = fx + (size_t)(sq - nraw + 1) * n0;
            cpx<T> *dst = raw + sq * (SEG * kLagWin) + sb * kLagWin + lane;
            T *wdst = wraw + (sq - nraw) * (SEG * kLagWin) + sb * kLagWin + lane;
            if (x0 >= 0 && x0 + kLagL <= n0) {  // the window inside the image
                src += x0 + lane;
                wsrc += x0 + lane;
#pragma unroll
                for (int i = 0; i < kLagL / 32; ++i) {
                    if (is_f) cp_async<sizeof(cpx<T>)>(dst + 32 * i, src + 32 * i);
                    else cp_async<sizeof(T)>(wdst + 32 * i, wsrc + 32 * i);
                }
            } else {
                for (int i = 0; i < kLagL / 32; ++i) {
                    int x = x0 + lane + 32 * i;
                    x = small ? imod(x, n0) : (x < 0 ? x + n0 : (x >= n0 ? x - n0 : x));
                    if (is_f) cp_async<sizeof(cpx<T>)>(dst + 32 * i, src + x);
                    else cp_async<sizeof(T)>(wdst + 32 * i, wsrc + x);
                }
            }
        }
        asm volatile("cp.async.commit_group;\n" ::);
    };
    fetch(0);
    const cpx<T> *win = raw + (size_t)fsq * SEG * kLagWin + sub * kLagWin + g;
    const T *wwin = wraw + (size_t)(ti - 1) * SEG * kLagWin + sub * kLagWin + g;
    for (int s0 = 0; s0 < nseg; s0 += SEG) {
        asm volatile("cp.async.wait_group 0;\n" ::);
        __syncthreads();  // this batch's windows are staged; the sums of the one before are done
        const int seg = s0 + sub;
        if (has && seg < nseg) {
            const int x0 = seg * core;
            cpx<T> v[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = win[8 * i];
            if (ti > 0) {
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] = scale(v[i], wwin[8 * i]);
            }
            if (centre) {
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i].re -= mu;
            }
            if (is_core) {  // the halos are h <= 32 wide
                const int hi = h + min(core, n0 - x0);
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (g + 8 * i < h) v[i] = mk((T)0, (T)0);
                if (hi >= kLagL - 32) {
#pragma unroll
                    for (int i = 12; i < 16; ++i)
                        if (g + 8 * i >= hi) v[i] = mk((T)0, (T)0);
                } else {
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (g + 8 * i >= hi) v[i] = mk((T)0, (T)0);
                }
            }
            dft16c(v, lc);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const cpx<T> y = v[slot16(j)];
                row[j * 9 + g] = j == 0 ? y : cmul(y, stp[j * 8 + g]);
            }
            __syncwarp(0xffu << (lane & 24));
            cpx<T> u[2][8];
#pragma unroll
            for (int b = 0; b < 2; ++b) {
#pragma unroll
                for (int q = 0; q < 8; ++q) u[b][q] = row[(g + 8 * b) * 9 + q];
            }
            __syncwarp(0xffu << (lane & 24));
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                dft8c(u[b], lc);
#pragma unroll
                for (int q = 0; q < 8; ++q) row[16 * q + 8 * b + g] = u[b][q];
            }
        }
        __syncthreads();
        if (s0 + SEG < nseg) fetch(s0 + SEG);  // in flight during the product sums
        const int cnt = min(SEG, nseg - s0);
        constexpr size_t kStride = (size_t)SEG * kLagRow;
        constexpr auto own = std::make_integer_sequence<int, Sh::kOwn>{};
        if constexpr (Sh::kSplitPairs) {
            constexpr int OWN = Sh::kOwn;
            for (int s = 0; s < cnt; ++s) {
                const cpx<T> *sp = spec + (size_t)s * kLagRow + k;
                if (role == 0) lag_products<T, NK, 0>(acc, sp, kStride, own);
                else if (role == 1) lag_products<T, NK, OWN>(acc, sp, kStride, own);
                else if (role == 2) lag_products<T, NK, 2 * OWN>(acc, sp, kStride, own);
            }
        } else if (role < Sh::kRoles) {
            for (int s = role; s < cnt; s += Sh::kRoles)
                lag_products<T, NK, 0>(acc, spec + (size_t)s * kLagRow + k, kStride, own);
        }
    }
    __syncthreads();
    // Z_p(k); where the roles split the segments, their sums added in order
    cpx<T> *Z = spec;  // [NP][kLagL]
    if constexpr (Sh::kSplitPairs) {
        if (role < Sh::kRoles) {
#pragma unroll
            for (int p = 0; p < Sh::kOwn; ++p) Z[(role * Sh::kOwn + p) * kLagL + k] = acc[p];
        }
        __syncthreads();
    } else {
        for (int r = 0; r < Sh::kRoles; ++r) {
            if (role == r) {
#pragma unroll
                for (int p = 0; p < NP; ++p) Z[p * kLagL + k] = r == 0 ? acc[p] : Z[p * kLagL + k] + acc[p];
            }
            __syncthreads();
        }
    }
    // Y_c(s) at row s, and the outer twiddles e^(2 pi i c rho / 128), in rows
    // that lanes of consecutive rho read without bank conflicts.  In FP32 both
    // are integers: Z in units of 2^-30 of its product's largest value (up to a
    // power of two), Y of 2^-27, the twiddles of 2^-28.
    constexpr bool kInt = sizeof(T) == 4;
    constexpr int kYRow = 17, kYLen = 8 * kYRow;
    using E = typename std::conditional<kInt, int2, cpx<T>>::type;
    E *Y = reinterpret_cast<E *>(Z + NP * kLagL);  // [NP][8][kYRow]
    E *tq = Y + NP * kYLen;                        // [16][2 h + 1]
    const int nl = 2 * h + 1;
    __shared__ unsigned zmax[NP];  // bits of the largest magnitude (of a NaN where there is one)
    if constexpr (kInt) {
        for (int p = warp; p < NP; p += Sh::kThreads / 32) {
            unsigned m = 0;
#pragma unroll
            for (int i = 0; i < kLagL / 32; ++i) {
                const cpx<T> z = Z[p * kLagL + lane + 32 * i];
                m = max(m, max(__float_as_uint(fabsf(z.re)), __float_as_uint(fabsf(z.im))));
            }
            m = __reduce_max_sync(0xffffffffu, m);
            if (lane == 0) zmax[p] = max(m, 32u << 23);
        }
        __syncthreads();
    }
    for (int e = tid; e < NP * 16; e += Sh::kThreads) {
        const cpx<T> *z = Z + (e >> 4) * kLagL + (e & 15);
        E *y = Y + (e >> 4) * kYLen + (e & 15);
        if constexpr (kInt) {
            const float up = __uint_as_float((283u - (zmax[e >> 4] >> 23)) << 23);  // the largest to 2^29 .. 2^30
            i64 re[8], im[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const cpx<T> v = z[16 * r];
                re[r] = __float2int_rn(v.re * up);
                im[r] = __float2int_rn(v.im * up);
            }
            idft8(re, im);
            auto part = [](i64 v) { return (int)((v + 4) >> 3); };
#pragma unroll
            for (int r = 0; r < 8; ++r)
                y[kYRow * r] = make_int2(part(re[(r & 1) * 4 + r / 2]), part(im[(r & 1) * 4 + r / 2]));
        } else {
            cpx<T> v[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) v[r] = z[16 * r];
            dft8(v, 1);
#pragma unroll
            for (int r = 0; r < 8; ++r) y[kYRow * r] = v[r];
        }
    }
    for (int e = tid; e < 16 * nl; e += Sh::kThreads) {
        const int cc = e / nl, rho = e - cc * nl - h, q = (cc * rho) & (kLagL - 1);
        if constexpr (kInt) tq[e] = tab->inv[q];
        else tq[e] = conj(tab->fwd[0][q]);
    }
    __syncthreads();
    // norm times the lag sums, in the row order of the stage-1 table: the Omega
    // products (a, q) first, then the Theta products
    const int nom = NK * (NK + 1) / 2 * nl, nq = nom + NK * (2 * w0 + 1);
    for (int e = tid; e < nq; e += Sh::kThreads) {
        int p, rho;
        if (e < nom) {
            const int o = e / nl;
            rho = e - o * nl - h;
            int a = 0, q = o;  // o-th pair a <= q of the Omega list
            while (q >= NK - a) {
                q -= NK - a;
                ++a;
            }
            p = o + a;  // each earlier a also has a Theta product
        } else {
            const int a = (e - nom) / (2 * w0 + 1);
            rho = (e - nom) - a * (2 * w0 + 1) - w0;
            // products before (a, NK): sum over a' <= a of (NK + 1 - a'), minus 1
            p = (a + 1) * (NK + 1) - a * (a + 1) / 2 - 1;
        }
        const E *y = Y + p * kYLen + kYRow * (rho & 7), *w = tq + rho + h;
        cpx<T> out;
        if constexpr (kInt) {
            i64 re = 0, im = 0;
#pragma unroll 4
            for (int cc = 0; cc < 16; ++cc) {
                const int2 a = w[cc * nl], b = y[cc];
                re += (i64)a.x * b.x - (i64)a.y * b.y;
                im += (i64)a.x * b.y + (i64)a.y * b.x;
            }
            // norm times the sums, from their bits 20 and up (the rest is below Y's
            // roundings) in one rounding; NaN where Z is not finite
            const unsigned m = zmax[p];
            const float unit = (m < 0x7f800000u ? __uint_as_float(((m >> 23) - 29u) << 23) * 0x1p-12f
                                                : __uint_as_float(0x7fffffffu)) * norm;
            auto value = [&](i64 v) {
                return fmaf((float)(int)(v >> 42), unit * 0x1p22f, (float)(int)((v >> 20) & 0x3fffff) * unit);
            };
            out = mk(value(re), value(im));
        } else {
            CAcc<T> s;
            s.zero();
#pragma unroll 4
            for (int cc = 0; cc < 16; cc += 2) s.add(cmul(w[cc * nl], y[cc]) + cmul(w[(cc + 1) * nl], y[cc + 1]));
            out = scale(mk((T)s.re.value(), (T)s.im.value()), (T)norm / kLagL);
        }
        Q[(size_t)e * ncol + c] = out;
    }
}

template <typename T, int NK>
static cudaError_t lagx_nk(Plan *p, cudaStream_t s) {
    using Sh = LagShape<NK>;
    const RowForm &f = p->build;
    const size_t smem = (size_t)Sh::kSeg * ((Sh::kSeq * kLagRow + (f.offb + p->nfy + 1) * kLagWin) * sizeof(cpx<T>) +
                                            (p->nfy - 1) * kLagWin * sizeof(T));
    // the epilogue's tables lie over the transforms and windows
    const size_t epi = (size_t)(Sh::kPairs * (kLagL + 136) + 16 * (4 * p->cfg.w0 + 1)) * sizeof(cpx<T>);
    if (epi > smem) return cudaErrorInvalidConfiguration;
    auto kern = k_lagx<T, NK>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    kern<<<f.ncol, Sh::kThreads, smem, s>>>(p->n0, f.hc, f.ncol, p->cfg.w0, f.offb, p->nfy,
                                             (const cpx<T> *)p->F, ftab_of<T>(p).fx, (const LagTab<T> *)p->tw128, lag_norm(p),
                                             (cpx<T> *)p->Q);
    p->launches++;
    return cudaGetLastError();
}

template <typename T>
static cudaError_t lagx_t(Plan *p, cudaStream_t s) {
    switch (p->nk) {
        case 1: return lagx_nk<T, 1>(p, s);
        case 3: return lagx_nk<T, 3>(p, s);
        case 6: return lagx_nk<T, 6>(p, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t lag_sums_x(Plan *p, cudaStream_t s) { return p->fp64 ? lagx_t<double>(p, s) : lagx_t<float>(p, s); }

// ---------------------------------------------------------------------------
// Row transforms by segments.  Block: 16 rows of one segment, 8 groups of 16
// threads; group q transforms rows 2q and 2q + 1 together (real and imaginary
// part), each thread 16 values: a radix-16 pass, an exchange through shared
// memory and a second radix-16 pass.  The pixels of R are read once and kept
// in registers for the nfy core sequences yt^j R (zero outside the core) and
// the nfy window ones, then S.
constexpr int kSegRows = 16;
constexpr int kSegL = kSegLen;                // 256
constexpr int kSegStride = 16 * 17 + 2;       // per row pair: rows of 17, 2 mod 16

// X = DFT of v (values g + 16 i of a group's 256) left in z[k], k < 256
template <typename T>
__device__ __forceinline__ void seg_fft(cpx<T> (&v)[16], cpx<T> *z, const cpx<T> *stw, int g, int sgn) {
    const unsigned grp = 0xffffu << (threadIdx.x & 16);
    dft16(v, sgn);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const cpx<T> y = v[slot16(j)];
        if (j == 0) {
            z[g] = y;
        } else {
            const cpx<T> w = stw[j * g];
            z[j * 17 + g] = cmul(y, sgn < 0 ? w : conj(w));
        }
    }
    __syncwarp(grp);
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = z[g * 17 + q];
    __syncwarp(grp);
    dft16(v, sgn);
}

template <typename T, typename I>
__global__ void __launch_bounds__(128) k_rows_seg(int n0, int n1, int hop, int halo, int nfy, int with_core,
                                                  const I *__restrict__ R, const I *__restrict__ S,
                                                  const uint8_t *__restrict__ mask, const T *__restrict__ fy,
                                                  const cpx<T> *__restrict__ tw256, cpx<T> *__restrict__ F,
                                                  size_t seqstride) {
    __shared__ cpx<T> Z[kSegRows / 2][kSegStride];
    __shared__ cpx<T> stw[kSegL];
    __shared__ T yt[kSegL];
    __shared__ int ys[kSegL];
    const int tid = threadIdx.x, g = tid & 15, q = tid >> 4;
    const int x0 = blockIdx.x * kSegRows, seg = blockIdx.y;
    const int y0 = seg * hop, len = min(hop, n1 - y0);
    for (int e = tid; e < kSegL; e += 128) {
        const int y = imod(y0 - halo + e, n1);
        ys[e] = y;
        yt[e] = nfy > 1 ? fy[n1 + y] : (T)0;  // the y-function 1: yt
        stw[e] = tw256[e];
    }
    __syncthreads();
    const int xa = x0 + 2 * q, xb = xa + 1;
    cpx<T> *z = Z[q];
    T ra[16], rb[16];
    auto load = [&](const I *img) {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int y = ys[g + 16 * i];
            ra[i] = xa < n0 ? (T)img[(size_t)xa * n1 + y] : (T)0;
            rb[i] = xb < n0 ? (T)img[(size_t)xb * n1 + y] : (T)0;
        }
        if (mask != nullptr) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const int y = ys[g + 16 * i];
                if (xa < n0 && mask[(size_t)xa * n1 + y] == 0) ra[i] = (T)0;
                if (xb < n0 && mask[(size_t)xb * n1 + y] == 0) rb[i] = (T)0;
            }
        }
    };
    // transform of the values in registers (on the core only, or everywhere)
    // into sequence `sq` of F
    auto emit = [&](int sq, bool on_core) {
        cpx<T> v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int e = g + 16 * i;
            const bool in = !on_core || (e >= halo && e < halo + len);
            v[i] = in ? mk(ra[i], rb[i]) : mk((T)0, (T)0);
        }
        seg_fft(v, z, stw, g, -1);
#pragma unroll
        for (int r = 0; r < 16; ++r) z[g + 16 * r] = v[slot16(r)];
        __syncthreads();
        // separate the two rows and write x-contiguous
        constexpr int H = kSegL / 2 + 1;
        const int r = tid & 15;
        if (x0 + r < n0) {
            const cpx<T> *zz = Z[r >> 1];
            cpx<T> *out = F + (size_t)sq * seqstride + ((size_t)seg * H) * n0 + x0 + r;
            for (int m = tid >> 4; m < H; m += 8) {
                const cpx<T> a = zz[m], b = conj(zz[(kSegL - m) & (kSegL - 1)]);
                out[(size_t)m * n0] = (r & 1) ? mul_i(scale(a - b, (T)0.5), -1) : scale(a + b, (T)0.5);
            }
        }
        __syncthreads();
    };
    load(R);
    const int offb = nfy;
    for (int j = 0; j < nfy; ++j) {
        if (j > 0) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const T w = yt[g + 16 * i];
                ra[i] *= w;
                rb[i] *= w;
            }
        }
        if (with_core) emit(j, true);
        emit(offb + j, false);
    }
    load(S);
    emit(offb + nfy, false);
}

// Inverse of the rows: the segment's core of D from D~(x, c).
template <typename T, typename I>
__global__ void __launch_bounds__(128) k_rows_inv_seg(int n0, int n1, int hop, int halo, const cpx<T> *__restrict__ Dt,
                                                      const cpx<T> *__restrict__ tw256, I *__restrict__ D) {
    constexpr int H = kSegL / 2 + 1;
    __shared__ cpx<T> Z[kSegRows / 2][kSegStride];
    __shared__ cpx<T> stw[kSegL];
    const int tid = threadIdx.x, g = tid & 15, q = tid >> 4;
    const int x0 = blockIdx.x * kSegRows, seg = blockIdx.y;
    const int y0 = seg * hop, len = min(hop, n1 - y0);
    for (int e = tid; e < kSegL; e += 128) stw[e] = tw256[e];
    const int r = tid & 15;
    cpx<T> *zz = Z[r >> 1];
    // rows a = 2 (r / 2), b = a + 1: row a's thread stores a + i b, m <= 128,
    // row b's thread the mirror conj(a) + i conj(b); the other row's value
    // comes from the neighbouring lane
    const cpx<T> *src = Dt + (size_t)seg * H * n0 + x0 + r;
    for (int m = tid >> 4; m < H + 7; m += 8) {  // every lane takes part in the shuffle
        cpx<T> v = mk((T)0, (T)0), o;
        if (m < H && x0 + r < n0) v = src[(size_t)m * n0];
        o.re = __shfl_xor_sync(0xffffffffu, v.re, 1);
        o.im = __shfl_xor_sync(0xffffffffu, v.im, 1);
        if (m < H) {
            if (!(r & 1)) zz[m] = v + mul_i(o, 1);
            else if (m > 0 && m < kSegL / 2) zz[kSegL - m] = conj(o) + mul_i(conj(v), 1);
        }
    }
    __syncthreads();
    cpx<T> *z = Z[q];
    cpx<T> v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = z[g + 16 * i];
    __syncwarp(0xffffu << (threadIdx.x & 16));
    seg_fft(v, z, stw, g, 1);
    const T inv = (T)1 / (T)kSegL;
    const int xa = x0 + 2 * q, xb = xa + 1;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const int e = g + 16 * k - halo;
        if (e >= 0 && e < len) {
            const cpx<T> o = v[slot16(k)];
            if (xa < n0) D[(size_t)xa * n1 + y0 + e] = (I)(o.re * inv);
            if (xb < n0) D[(size_t)xb * n1 + y0 + e] = (I)(o.im * inv);
        }
    }
}

template <typename T, typename I>
static cudaError_t rows_seg_t(Plan *p, const void *ref, const void *sci, const uint8_t *mask, bool core,
                              cudaStream_t s) {
    const RowForm &f = core ? p->build : p->own;
    const dim3 grid((p->n0 + kSegRows - 1) / kSegRows, f.nsy);
    k_rows_seg<T, I><<<grid, 128, 0, s>>>(p->n0, p->n1, f.hop, f.halo, p->nfy, core ? 1 : 0, (const I *)ref,
                                          (const I *)sci, mask, ftab_of<T>(p).fy, (const cpx<T> *)f.twy,
                                          (cpx<T> *)p->F, (size_t)f.ncol * p->n0);
    p->launches++;
    return cudaGetLastError();
}

cudaError_t rows_segments(Plan *p, const void *ref, const void *sci, const uint8_t *mask, bool core,
                          cudaStream_t s) {
    const bool img64 = p->cfg.dtype == SFFT_F64;
    if (p->fp64)
        return img64 ? rows_seg_t<double, double>(p, ref, sci, mask, core, s)
                     : rows_seg_t<double, float>(p, ref, sci, mask, core, s);
    return img64 ? rows_seg_t<float, double>(p, ref, sci, mask, core, s)
                 : rows_seg_t<float, float>(p, ref, sci, mask, core, s);
}

template <typename T, typename I>
static cudaError_t rows_inv_seg_t(Plan *p, const RowForm &f, void *diff, cudaStream_t s) {
    const dim3 grid((p->n0 + kSegRows - 1) / kSegRows, f.nsy);
    k_rows_inv_seg<T, I><<<grid, 128, 0, s>>>(p->n0, p->n1, f.hop, f.halo, (const cpx<T> *)p->U,
                                              (const cpx<T> *)f.twy, (I *)diff);
    return cudaGetLastError();
}

cudaError_t rows_inv_segments(Plan *p, const RowForm &f, void *diff, cudaStream_t s) {
    const bool img64 = p->cfg.dtype == SFFT_F64;
    if (p->fp64) return img64 ? rows_inv_seg_t<double, double>(p, f, diff, s) : rows_inv_seg_t<double, float>(p, f, diff, s);
    return img64 ? rows_inv_seg_t<float, double>(p, f, diff, s) : rows_inv_seg_t<float, float>(p, f, diff, s);
}

}  // namespace sfft
