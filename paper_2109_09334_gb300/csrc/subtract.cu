// subtract.cu -- difference image of Eq. 12-13 from the solved coefficients.
//
// D = S - sum_t sum_(a,b) c_t(a,b) g_t(x - a, y - b) - sum_s b_s T^s, with
// g_t = xt^i yt^j R (Eq. 10-11) or B_i(xt) B_j(yt) R (Eq. 8), T^s the
// background basis, and the per-term kernel c_t of the delta basis (Eq. 3-4):
// c_t(a,b) = a_t,ab for (a,b) != 0 and c_t(0,0) = a_t,00 - sum_(a,b)!=0 a_t,ab.
// Along y the convolution is taken in Fourier space (Eq. 13): with the row
// transforms G~_t(x, m) of the build, the row transform of D is
//   D~(x, m) = S~(x, m) - sum_t sum_a kap_t(a, m) G~_t(x - a, m) - B~(x, m),
//   kap_t(a, m) = sum_b c_t(a, b) exp(-2 pi i m b / N1),
// an L0-tap circular stencil along x per frequency column m; one inverse
// real FFT per row then gives D.
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"
#include "fft.cuh"
#include "fft16.cuh"
#include "internal.h"

namespace sfft {

// kap[t][a + w0][m] = sum_b k_t(a, b) exp(-2 pi i m b / ylen), one block per
// (t, a) and 256 frequencies.  The row's coefficients are read and rounded to
// the compute type once; in the centre row the (0, 0) value also loses the sum
// of the term's other coefficients (FP64).  Bound by the twiddle reads, b words
// apart across the lanes: one serves b and -b.  (A sum kernel before, and per
// output 2 w1 + 1 reads of the FP64 coefficients, of twiddles and as many
// moduli: 4.7 + 17.9 -> 8.2 us at 4096 x 4096, w = 8, 6 terms.)
template <typename T>
__global__ void __launch_bounds__(256) k_kernel_table(int ylen, BasisView bv, const double *__restrict__ x,
                                                      const cpx<T> *__restrict__ tw1, cpx<T> *__restrict__ kap) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *c = reinterpret_cast<T *>(smem_raw);  // [2 w1 + 1]
    const int w0 = bv.w0, w1 = bv.w1, L0 = 2 * w0 + 1, L1 = 2 * w1 + 1;
    const int h1c = ylen / 2 + 1, t = blockIdx.y / L0, a = (int)blockIdx.y % L0 - w0;
    double ksum = 0.0;  // in thread 0 of a centre row
    if (a == 0) {
        double s = 0.0;
        for (int off = threadIdx.x; off < L0 * L1; off += blockDim.x) {
            const int oa = off / L1 - w0, ob = off % L1 - w1;
            if (oa == 0 && ob == 0) continue;
            const int u = bv.unknown(t, oa, ob);
            if (u >= 0) s += x[u];
        }
        __shared__ double red[32];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x == 0)
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) ksum += red[w];
    }
    for (int b = threadIdx.x; b < L1; b += blockDim.x) {
        if (a == 0 && b == w1) continue;
        const int u = bv.unknown(t, a, b - w1);
        c[b] = u >= 0 ? (T)x[u] : (T)0;
    }
    if (a == 0 && threadIdx.x == 0) {
        const int u = bv.unknown(t, 0, 0);
        c[w1] = (T)((u >= 0 ? x[u] : 0.0) - ksum);
    }
    __syncthreads();
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= h1c) return;
    T re = c[w1], im = (T)0;
    int idx = m;  // m b mod ylen
    for (int b = 1; b <= w1; ++b) {
        const cpx<T> w = tw1[idx];  // exp(-2 pi i m b / ylen)
        const T cp = c[w1 + b], cm = c[w1 - b];
        re += cp * w.re;
        im += cp * w.im;
        re += cm * w.re;
        im -= cm * w.im;
        idx += m;
        if (idx >= ylen) idx -= ylen;
    }
    kap[(size_t)blockIdx.y * h1c + m] = mk(re, im);
}

// D~(x, m) into Dt[m][x]: one block per column m and segment of x.  For each
// kernel term (i, j) the weighted column W(x) = xt^i F_j(x, m) is staged in
// shared memory over the segment and w0 values on either side, wrapped at the
// image edge (one pad element after every Q, so that the threads' strided
// reads hit distinct banks); thread t slides a window of Q values over it for
// its outputs Q t .. Q t + Q - 1: per tap a read of the kernel value, one of W,
// and Q complex multiply-adds.  In FP32 these run in packed pairs (real and
// imaginary part), with the kernel values kept as the pairs (-re, -re) and
// (im, -im) that acc - k w = acc + (-re) (w.re, w.im) + (im, -im) (w.im, w.re)
// takes: the roundings of four scalar ones.  Global memory is read and written
// with consecutive x in consecutive threads; the sums' start S - B and their
// result pass through shared memory.  Segments of 256 threads: several blocks
// on a multiprocessor cover each other's loads.  A block for a whole column
// (1024 threads, scalar multiply-adds) spent half of its time waiting:
// 257 -> 219 us at 4096 x 4096, w = 8, 6 terms, FP32 (2322 columns of 2046, w =
// 6: 124 -> 109 us).
template <typename T>
__host__ __device__ constexpr int sub_q() { return sizeof(T) == 4 ? 4 : 8; }
constexpr int kSubThreads = 256;
// Launch shape.  Where the kernel values leave no room for both pairs each
// (n_K L0 above some 12000 values), they are kept once and the pairs made at
// every tap (223 instead of 176 us at 4093 x 256, w0 = 100, w1 = 0, 6 terms,
// where both fit).  Where they leave none for the segments of 256 threads
// either, these are halved: whatever fits beside a whole column fits so.
struct SubShape {
    int threads;
    bool two;  // both pairs kept
    size_t smem;
};
template <typename T>
static SubShape sub_shape(const Plan *p) {
    constexpr int q = sub_q<T>(), most = sizeof(T) == 4 ? kSubThreads : 64;
    constexpr size_t room = 227 * 1024 - kMaxFun * sizeof(cpx<T>);  // (bp)
    SubShape h;
    h.threads = std::min((p->n0 + q - 1) / q, most);
    auto size = [&](int copies) {
        const int len = q * h.threads + 2 * p->cfg.w0;
        return ((size_t)copies * p->nk * p->L0 + 2 * (size_t)(len + len / q + q + 1)) * sizeof(cpx<T>);
    };
    h.two = sizeof(T) == 4 && size(2) <= room;
    if (!h.two)
        while (h.threads > 1 && size(1) > room) h.threads = (h.threads + 1) / 2;
    h.smem = size(h.two ? 2 : 1);
    return h;
}

// W0 >= 0: the kernel half-width is the compile-time W0 (the tap loop unrolls
// completely, so the window shifts are register renames); W0 < 0: w0 at run time.
// TWO: both pairs of a kernel value in shared memory (FP32).
template <typename T, int W0, bool TWO>
__global__ void __launch_bounds__(kSubThreads, sizeof(T) == 4 ? 4 : 1)
    k_sub_cols(int n0, int hc, int ncol, int offb, BasisView bv, FTab<T> ft, int w0, int nbkg_off,
               const cpx<T> *__restrict__ F, const cpx<T> *__restrict__ kap, const cpx<T> *__restrict__ yhat,
               const double *__restrict__ x, cpx<T> *__restrict__ Dt) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr bool PK = sizeof(T) == 4;
    constexpr int Q = sub_q<T>(), KS = TWO ? 2 : 1;
    const int nk = bv.nk, nbt = bv.nb;
    if (W0 >= 0) w0 = W0;
    const int L0 = 2 * w0 + 1;
    auto padq = [](int v) { return v + v / Q; };
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int col = blockIdx.x, m = col % hc, xb = blockIdx.y * (Q * nthr);
    const int len = min(Q * nthr, n0 - xb), ext = len + 2 * w0;  // outputs; staged values
    cpx<T> *kp = reinterpret_cast<cpx<T> *>(smem_raw);  // nk * L0 (TWO: two pairs each)
    cpx<T> *Wb = kp + KS * nk * L0;  // two buffers, alternating by term
    const int wlen = padq(Q * nthr + 2 * w0) + Q + 1;
    for (int e = tid; e < nk * L0; e += nthr) {
        const cpx<T> v = kap[(size_t)e * hc + m];
        if constexpr (TWO) {
            kp[2 * e] = mk(-v.re, -v.re);
            kp[2 * e + 1] = mk(v.im, -v.im);
        } else {
            kp[e] = v;
        }
    }
    // S~ minus the background B~(x, m) = sum_p bx_p(x) sum_q b_pq Y_q(m)
    const cpx<T> *Sc = F + ((size_t)(offb + bv.nfy) * ncol + col) * n0 + xb;
    cpx<T> v[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) v[q] = tid + q * nthr < len ? Sc[tid + q * nthr] : mk((T)0, (T)0);
    __shared__ cpx<T> bp[kMaxFun];
    for (int p = tid; p < bv.nbx; p += nthr) {
        cpx<T> b = mk((T)0, (T)0);
        for (int s = 0; s < nbt; ++s)
            if (bv.sp(s) == p) b = cadd(b, scale(yhat[(size_t)bv.sq(s) * ncol + col], (T)x[nbkg_off + s]));
        bp[p] = b;
    }
    __syncthreads();
    for (int p = 0; p < bv.nbx; ++p) {
        const T *wx = ft.bx + (size_t)p * n0 + xb + tid;
        const cpx<T> b = bp[p];
#pragma unroll
        for (int q = 0; q < Q; ++q)
            if (tid + q * nthr < len) v[q] = csub(v[q], scale(b, wx[q * nthr]));
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) Wb[wlen + padq(tid + q * nthr)] = v[q];
    __syncthreads();
    cpx<T> acc[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) acc[q] = Wb[wlen + padq(Q * tid) + q];
    // terms grouped by their y-function j: F_j is loaded once per group.  The
    // weighted columns alternate between two buffers, so one barrier per term
    // separates a buffer's fill from its reads and from its refill two terms on.
    constexpr int NF = Q + 1;  // staged values per thread (2 w0 <= nthr, or the rest below)
    auto wrapx = [&](int e) {  // image column of staged value e
        const int u = xb - w0 + e;
        return u < 0 ? u + n0 : (u >= n0 ? u - n0 : u);
    };
    int xi[NF];
#pragma unroll
    for (int q = 0; q < NF; ++q) xi[q] = tid + q * nthr < ext ? wrapx(tid + q * nthr) : -1;
    int nterm = 0;
    for (int j = 0; j < bv.nfy; ++j) {
        const int ncj = bv.jcnt(j);
        if (ncj == 0) continue;
        const cpx<T> *Fj = F + ((size_t)(offb + j) * ncol + col) * n0;
        cpx<T> f[NF];
#pragma unroll
        for (int q = 0; q < NF; ++q) f[q] = xi[q] >= 0 ? Fj[xi[q]] : mk((T)0, (T)0);
        for (int k = 0; k < ncj; ++k) {
            const int t = bv.jterm(j, k);
            const T *wx = ft.fx + (size_t)bv.ti(t) * n0;
            cpx<T> *W = Wb + (size_t)(nterm++ & 1) * wlen;
#pragma unroll
            for (int q = 0; q < NF; ++q)
                if (xi[q] >= 0) W[padq(tid + q * nthr)] = scale(f[q], wx[xi[q]]);
            for (int e = tid + NF * nthr; e < ext; e += nthr)  // (few threads, wide kernels)
                W[padq(e)] = scale(Fj[wrapx(e)], wx[wrapx(e)]);
            __syncthreads();  // this buffer is filled; the other one's reads (two terms ago) are done
            const cpx<T> *kt = kp + KS * t * L0;
            const cpx<T> *Wt = W + padq(Q * tid);
            if constexpr (PK) {
                pair32 pa[Q], win[Q], swp[Q];  // sums; window values (re, im) and (im, re)
                auto get = [&](int e, pair32 &v, pair32 &w) {
                    const cpx<T> c = Wt[padq(e)];
                    v = pack2(c.re, c.im);
                    w = pack2(c.im, c.re);
                };
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    pa[q] = pack2(acc[q].re, acc[q].im);
                    get(q, win[q], swp[q]);
                }
#pragma unroll
                for (int c = 0; c <= 2 * (W0 >= 0 ? W0 : w0); ++c) {  // tap a = w0 - c
                    pair32 kr, ki;
                    if constexpr (TWO) {
                        const float4 kv = *reinterpret_cast<const float4 *>(kt + 2 * (L0 - 1 - c));
                        kr = pack2(kv.x, kv.y), ki = pack2(kv.z, kv.w);
                    } else {
                        const cpx<T> kv = kt[L0 - 1 - c];
                        kr = pack2(-kv.re, -kv.re), ki = pack2(kv.im, -kv.im);
                    }
#pragma unroll
                    for (int q = 0; q < Q; ++q) fma2(pa[q], kr, win[q]);
#pragma unroll
                    for (int q = 0; q < Q; ++q) fma2(pa[q], ki, swp[q]);
#pragma unroll
                    for (int q = 0; q + 1 < Q; ++q) {
                        win[q] = win[q + 1];
                        swp[q] = swp[q + 1];
                    }
                    get(Q + c, win[Q - 1], swp[Q - 1]);
                }
#pragma unroll
                for (int q = 0; q < Q; ++q) acc[q] = unpack2(pa[q]);
            } else {
                cpx<T> win[Q];
#pragma unroll
                for (int q = 0; q < Q; ++q) win[q] = Wt[padq(q)];
#pragma unroll
                for (int c = 0; c <= 2 * (W0 >= 0 ? W0 : w0); ++c) {
                    const cpx<T> kv = kt[L0 - 1 - c];
#pragma unroll
                    for (int q = 0; q < Q; ++q) acc[q] = cfms(acc[q], kv, win[q]);
#pragma unroll
                    for (int q = 0; q + 1 < Q; ++q) win[q] = win[q + 1];
                    win[Q - 1] = Wt[padq(Q + c)];
                }
            }
        }
    }
    cpx<T> *W = Wb + (size_t)(nterm & 1) * wlen;  // (last read two terms ago)
#pragma unroll
    for (int q = 0; q < Q; ++q) W[padq(Q * tid) + q] = acc[q];
    __syncthreads();
    cpx<T> *out = Dt + (size_t)col * n0 + xb;
#pragma unroll
    for (int q = 0; q < Q; ++q)
        if (tid + q * nthr < len) out[tid + q * nthr] = W[padq(tid + q * nthr)];
}

// two consecutive complex values from global memory (16-byte aligned for
// float: one 16-byte load)
__device__ __forceinline__ void load_pair(const cpx<float> *p, cpx<float> &a, cpx<float> &b) {
    const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
    a = mk(v.x, v.y);
    b = mk(v.z, v.w);
}
__device__ __forceinline__ void load_pair(const cpx<double> *p, cpx<double> &a, cpx<double> &b) {
    a = p[0];
    b = p[1];
}

// Inverse real FFT of rows: NG groups of G = n1/16 threads per block, each
// group transforms two rows at once (real and imaginary part of one complex
// FFT of the Hermitian-extended row spectra).
template <typename T, typename I>
__global__ void __launch_bounds__(sizeof(T) == 4 ? 512 : 256) k_rows_inv(int n0, int n1, int NG, const cpx<T> *__restrict__ Dt,
                                                   const cpx<T> *__restrict__ tw1g, I *__restrict__ D) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int G = n1 / 16;
    const int np = padded_len(n1);
    cpx<T> *Z = reinterpret_cast<cpx<T> *>(smem_raw);  // NG * np
    const int tid = threadIdx.x;
    const int grp = tid / G, gt = tid - grp * G;
    const int half = n1 / 2;
    const T inv = (T)1 / (T)n1;
    const int xa = (blockIdx.x * NG + grp) * 2, xb = xa + 1;
    const cpx<T> *tw = tw1g;  // pass-ordered twiddles, read through L1
    cpx<T> *zr = Z + (size_t)grp * np;
    {
        // 16 frequencies per thread, all loads in flight; rows xa, xb are
        // adjacent, so with an even n0 both come in one 2-element load
        cpx<T> A[16], B[16];
        if (xb < n0 && (n0 & 1) == 0) {
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                const int mm = gt + c * G;
                const int mr = (mm <= half) ? mm : n1 - mm;
                load_pair(Dt + (size_t)mr * n0 + xa, A[c], B[c]);
            }
        } else {
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                const int mm = gt + c * G;
                const int mr = (mm <= half) ? mm : n1 - mm;
                A[c] = xa < n0 ? Dt[(size_t)mr * n0 + xa] : mk((T)0, (T)0);
                B[c] = xb < n0 ? Dt[(size_t)mr * n0 + xb] : mk((T)0, (T)0);
            }
        }
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            const int mm = gt + c * G;
            const cpx<T> a = (mm <= half) ? A[c] : conj(A[c]);
            const cpx<T> b = (mm <= half) ? B[c] : conj(B[c]);
            zr[pad16(mm)] = a + mul_i(b, 1);
        }
    }
    __syncthreads();
    group_fft(zr, n1, 1, tw, gt, G);
    for (int y = gt; y < n1; y += G) {
        const cpx<T> z = zr[pad16(y)];
        if (xa < n0) D[(size_t)xa * n1 + y] = (I)(z.re * inv);
        if (xb < n0) D[(size_t)xb * n1 + y] = (I)(z.im * inv);
    }
}

// Inverse real transform of rows for a row length n1 that is not a power of
// two: as k_rows_inv, with Bluestein DFTs of length n1 (FFTs of length m1).
template <typename T, typename I>
__global__ void __launch_bounds__(sizeof(T) == 4 ? 1024 : 512) k_rows_inv_blu(int n0, int n1, int m1, int NG,
                                                       const cpx<T> *__restrict__ Dt,
                                                       const cpx<T> *__restrict__ chirp,
                                                       const cpx<T> *__restrict__ bfilt,
                                                       const cpx<T> *__restrict__ twpm, I *__restrict__ D) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int G = m1 / 16;
    const int np = padded_len(m1);
    cpx<T> *Z = reinterpret_cast<cpx<T> *>(smem_raw);  // NG * np
    const int tid = threadIdx.x;
    const int grp = tid / G, gt = tid - grp * G;
    const int half = n1 / 2;
    const T inv = (T)1 / (T)n1;
    const int xa = (blockIdx.x * NG + grp) * 2, xb = xa + 1;
    cpx<T> *zr = Z + (size_t)grp * np;
    for (int mm = gt; mm < n1; mm += G) {
        const int mr = (mm <= half) ? mm : n1 - mm;
        cpx<T> a = xa < n0 ? Dt[(size_t)mr * n0 + xa] : mk((T)0, (T)0);
        cpx<T> b = xb < n0 ? Dt[(size_t)mr * n0 + xb] : mk((T)0, (T)0);
        if (mm > half) {
            a = conj(a);
            b = conj(b);
        }
        zr[pad16(mm)] = a + mul_i(b, 1);
    }
    __syncthreads();
    bluestein(zr, n1, m1, 1, chirp, bfilt, twpm, gt, G);
    for (int y = gt; y < n1; y += G) {
        const cpx<T> z = zr[pad16(y)];
        if (xa < n0) D[(size_t)xa * n1 + y] = (I)(z.re * inv);
        if (xb < n0) D[(size_t)xb * n1 + y] = (I)(z.im * inv);
    }
}

// D from its row transforms in p->U (layout [m][x]): the inverse real FFT of
// every row, two rows per complex transform.
template <typename T>
static cudaError_t launch_rows_inv(Plan *p, void *diff, cudaStream_t s) {
    if (p->gen1) {
        const int G = p->m1 / 16;
        int NG = (sizeof(T) == 4 ? 1024 : 512) / G;
        if (NG < 1) NG = 1;
        if (NG > 4) NG = 4;
        if (NG > (p->n0 + 1) / 2) NG = (p->n0 + 1) / 2;
        size_t smem = (size_t)NG * padded_len(p->m1) * sizeof(cpx<T>);
        while (NG > 1 && smem > 200 * 1024) {
            NG /= 2;
            smem = (size_t)NG * padded_len(p->m1) * sizeof(cpx<T>);
        }
        if (p->tune_ng > 0 && p->tune_ng < NG) {
            NG = p->tune_ng;
            smem = (size_t)NG * padded_len(p->m1) * sizeof(cpx<T>);
        }
        const int blocks = (p->n0 + 2 * NG - 1) / (2 * NG);
        const cpx<T> *ch = (const cpx<T> *)p->chirp1, *bf = (const cpx<T> *)p->bfilt1, *tw = (const cpx<T> *)p->twpm1;
        if (p->cfg.dtype == SFFT_F64) {
            cudaFuncSetAttribute(k_rows_inv_blu<T, double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            k_rows_inv_blu<T, double><<<blocks, NG * G, smem, s>>>(p->n0, p->n1, p->m1, NG, (const cpx<T> *)p->U,
                                                                    ch, bf, tw, (double *)diff);
        } else {
            cudaFuncSetAttribute(k_rows_inv_blu<T, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            k_rows_inv_blu<T, float><<<blocks, NG * G, smem, s>>>(p->n0, p->n1, p->m1, NG, (const cpx<T> *)p->U,
                                                                   ch, bf, tw, (float *)diff);
        }
    } else {
        const int G = p->n1 / 16;
        // at most 512 (FP32) / 256 (FP64) threads and about 100 KB of shared
        // memory per block, so that two blocks share an SM
        int NG = (sizeof(T) == 4 ? 512 : 256) / G;
        if (NG < 1) NG = 1;
        if (NG > 4) NG = 4;
        if (NG > (p->n0 + 1) / 2) NG = (p->n0 + 1) / 2;
        size_t smem = (size_t)NG * padded_len(p->n1) * sizeof(cpx<T>);
        while (NG > 1 && smem > 110 * 1024) {
            NG /= 2;
            smem = (size_t)NG * padded_len(p->n1) * sizeof(cpx<T>);
        }
        if (p->tune_ng > 0 && p->tune_ng < NG) {
            NG = p->tune_ng;
            smem = (size_t)NG * padded_len(p->n1) * sizeof(cpx<T>);
        }
        const int blocks = (p->n0 + 2 * NG - 1) / (2 * NG);
        if (p->cfg.dtype == SFFT_F64) {
            cudaFuncSetAttribute(k_rows_inv<T, double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            k_rows_inv<T, double><<<blocks, NG * G, smem, s>>>(p->n0, p->n1, NG, (const cpx<T> *)p->U,
                                                                (const cpx<T> *)p->twp1, (double *)diff);
        } else {
            cudaFuncSetAttribute(k_rows_inv<T, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            k_rows_inv<T, float><<<blocks, NG * G, smem, s>>>(p->n0, p->n1, NG, (const cpx<T> *)p->U,
                                                               (const cpx<T> *)p->twp1, (float *)diff);
        }
    }
    return cudaGetLastError();
}

template <typename T>
static cudaError_t sub_t(Plan *p, const RowForm &f, const double *x, void *diff, cudaStream_t s) {
    cudaError_t err;
    p->launches += 3;
    const size_t csmem = (size_t)p->L1 * sizeof(T);
    k_kernel_table<T><<<dim3((f.hc + 255) / 256, p->nk * p->L0), 256, csmem, s>>>(
        f.ylen, p->bv, x, (const cpx<T> *)f.twy, (cpx<T> *)p->kap);
    if ((err = cudaGetLastError())) return err;
    {
        const SubShape h = sub_shape<T>(p);
        const int seg = sub_q<T>() * h.threads;
        const int nbkg_off = p->n - p->nb;
        constexpr bool two = sizeof(T) == 4;
        auto kern = h.two ? k_sub_cols<T, -1, two> : k_sub_cols<T, -1, false>;
        if (h.two || !two) {
            switch (p->cfg.w0) {  // the half-widths of the workloads, unrolled
                case 4: kern = k_sub_cols<T, 4, two>; break;
                case 5: kern = k_sub_cols<T, 5, two>; break;
                case 6: kern = k_sub_cols<T, 6, two>; break;
                case 7: kern = k_sub_cols<T, 7, two>; break;
                case 8: kern = k_sub_cols<T, 8, two>; break;
                default: break;
            }
        }
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)h.smem);
        kern<<<dim3(f.ncol, (p->n0 + seg - 1) / seg), h.threads, h.smem, s>>>(
            p->n0, f.hc, f.ncol, f.offb, p->bv, ftab_of<T>(p), p->cfg.w0, nbkg_off, (const cpx<T> *)p->F,
            (const cpx<T> *)p->kap, (const cpx<T> *)f.yhat, x, (cpx<T> *)p->U);
        if ((err = cudaGetLastError())) return err;
    }
    if (f.seg) return rows_inv_segments(p, f, diff, s);
    return launch_rows_inv<T>(p, diff, s);
}

// ---------------------------------------------------------------------------
// Noise decorrelation (App. C, Eq. 21-24) for one pair.  The spatial
// variation of the kernel is ignored there, so the matching kernel of Eq. 6
// is taken at one normalised position (xt0, yt0):
//     K(a, b) = sum_t xt0^i yt0^j c_t(a, b)            (kernel image, FP64)
// and the real filter of Eq. 24, normalised to unit kernel sum,
//     Q(l, m) = sqrt((s_S^2 + s_R^2 K^(0,0)^2) / (s_S^2 + s_R^2 |K^(l, m)|^2)),
// multiplies the 2-D transform of D:  D_dc = D (*) Q.  K^ is separable in the
// same way as the subtraction: kappa(a, m) = sum_b K(a, b) exp(-2 pi i m b / N1)
// and K^(l, m) = sum_a kappa(a, m) exp(-2 pi i l a / N0).

// Term weights at one normalised position (host-computed): xt0^i yt0^j,
// B_i(xt0) B_j(yt0), or 1 for the constant term.
struct TermWeights {
    double w[kMaxKTerms];
};

__global__ void k_kernel_image(BasisView bv, TermWeights tw, const double *__restrict__ x, double *__restrict__ kimg) {
    const int w0 = bv.w0, w1 = bv.w1;
    const int L1 = 2 * w1 + 1, L = (2 * w0 + 1) * L1;
    for (int e = threadIdx.x; e < L; e += blockDim.x) {
        const int a = e / L1 - w0, b = e % L1 - w1;
        double v = 0.0;
        for (int t = 0; t < bv.nk; ++t) {
            const double wt = tw.w[t];
            if (a != 0 || b != 0) {
                const int u = bv.unknown(t, a, b);
                if (u >= 0) v += wt * x[u];
            } else {
                const int u0 = bv.unknown(t, 0, 0);
                double c = u0 >= 0 ? x[u0] : 0.0;
                for (int o = 0; o < L; ++o) {
                    const int aa = o / L1 - w0, bb = o % L1 - w1;
                    if (aa == 0 && bb == 0) continue;
                    const int u = bv.unknown(t, aa, bb);
                    if (u >= 0) c -= x[u];
                }
                v += wt * c;
            }
        }
        kimg[e] = v;
    }
}

// kap[a + w0][m] = sum_b K(a, b) exp(-2 pi i m b / N1)
// for nkern centred kernels of half-widths w0, w1 (kernel c at kimg_a for
// c < na, else kimg_b): kap[c][a + w0][m] = sum_b k_c(a, b) exp(-2 pi i m b / N1)
template <typename T>
__global__ void k_decorr_kappa(int n1, int nkern, int na, int w0, int w1, const double *__restrict__ kimg_a,
                               const double *__restrict__ kimg_b, const cpx<T> *__restrict__ tw1,
                               cpx<T> *__restrict__ kap) {
    const int h1c = n1 / 2 + 1, L0 = 2 * w0 + 1, L1 = 2 * w1 + 1;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < nkern * L0 * h1c; e += gridDim.x * blockDim.x) {
        const int ca = e / h1c, m = e - ca * h1c;
        const int c = ca / L0, a = ca - c * L0;
        const double *k = c < na ? kimg_a + (size_t)c * L0 * L1 : kimg_b + (size_t)(c - na) * L0 * L1;
        cpx<T> v = mk((T)0, (T)0);
        for (int bi = 0; bi < L1; ++bi) v = cadd(v, scale(tw1[imod(m * (bi - w1), n1)], (T)k[a * L1 + bi]));
        kap[e] = v;
    }
}

// The co-added form of Eq. 21: ns science kernels G_j then nr reference
// kernels H_i (half-widths g0 along x), their noise variances s2[0 .. ns+nr).
struct CoaddDesc {
    int ns, nr, g0;
    double s2[2 * kMaxCoadd];
};

// Forward real transform of the rows of D, two rows per complex transform,
// written as Dt[m][x] (m < N1/2 + 1): pow2 n1 by the radix-16 FFT, other n1
// by Bluestein.
template <typename T, typename I, bool BLU>
__global__ void __launch_bounds__(sizeof(T) == 4 ? 1024 : 512) k_decorr_rows(int n0, int n1, int mlen, int NG,
                                                      const I *__restrict__ D, const cpx<T> *__restrict__ twg,
                                                      const cpx<T> *__restrict__ chirp,
                                                      const cpx<T> *__restrict__ bfilt, cpx<T> *__restrict__ Dt) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int G = mlen / 16;
    const int np = padded_len(mlen);
    const cpx<T> *tw = twg;                              // pass table (pow2), read through L1
    cpx<T> *Z = reinterpret_cast<cpx<T> *>(smem_raw);   // NG * np
    const int tid = threadIdx.x;
    const int grp = tid / G, gt = tid - grp * G;
    const int xa = (blockIdx.x * NG + grp) * 2, xb = xa + 1;
    cpx<T> *zr = Z + (size_t)grp * np;
    for (int y = gt; y < n1; y += G) {
        const T a = xa < n0 ? (T)D[(size_t)xa * n1 + y] : (T)0;
        const T b = xb < n0 ? (T)D[(size_t)xb * n1 + y] : (T)0;
        zr[pad16(y)] = mk(a, b);
    }
    __syncthreads();
    if (BLU) bluestein(zr, n1, mlen, -1, chirp, bfilt, twg, gt, G);
    else group_fft(zr, n1, -1, tw, gt, G);
    // the block's 2 NG rows (a power of two) side by side along x
    const int h1c = n1 / 2 + 1;
    const int nr = 2 * NG, total = h1c * nr;
    for (int e = tid; e < total; e += NG * G) {
        const int r = e & (nr - 1), m = e / nr, x = blockIdx.x * nr + r;
        if (x >= n0) continue;
        const cpx<T> *zz = Z + (size_t)(r >> 1) * np;
        const cpx<T> z = zz[pad16(m)];
        const cpx<T> zc = conj(zz[pad16(m == 0 ? 0 : n1 - m)]);
        Dt[(size_t)m * n0 + x] = (r & 1) ? mul_i(scale(z - zc, (T)0.5), -1) : scale(z + zc, (T)0.5);
    }
}

// Per frequency column m: transform along x, multiply by Q(l, m), transform
// back (scaled by 1/N0), in place in Dt[m][x].
template <typename T, bool BLU>
__global__ void __launch_bounds__(512) k_decorr_cols(int n0, int n1, int mlen, int w0,
                                                      double sigma_ref, double sigma_sci,
                                                      const cpx<T> *__restrict__ kap, const cpx<T> *__restrict__ tw0,
                                                      const cpx<T> *__restrict__ twg, const cpx<T> *__restrict__ chirp,
                                                      const cpx<T> *__restrict__ bfilt, cpx<T> *__restrict__ Dt,
                                                      CoaddDesc cd, const cpx<T> *__restrict__ gam) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int G = mlen / 16;
    const int L0 = 2 * w0 + 1;
    const int nc = cd.ns + cd.nr, Lg = 2 * cd.g0 + 1;  // nc = 0: the one-pair form
    const cpx<T> *tw = twg;                               // pass table (pow2), read through L1
    cpx<T> *kp = reinterpret_cast<cpx<T> *>(smem_raw);   // L0: kappa(a, m)
    cpx<T> *gp = kp + L0;                                // nc * Lg: gamma_c(a, m)
    cpx<T> *zr = gp + nc * Lg;                           // padded mlen
    const int tid = threadIdx.x, m = blockIdx.x;
    const int h1c = n1 / 2 + 1;
    for (int a = tid; a < L0; a += G) kp[a] = kap[(size_t)a * h1c + m];
    for (int e = tid; e < nc * Lg; e += G) gp[e] = gam[(size_t)e * h1c + m];
    // K^(0, 0) (kernel nc) and the sums of the homogenisation kernels, one
    // thread each: FP64 sums in every thread took as long as the transforms
    __shared__ double ksums[2 * kMaxCoadd + 1];
    __shared__ double numer;  // the filter's numerator: its denominator at frequency 0
    for (int c = tid; c <= nc; c += G) {
        double v = 0.0;
        if (c == nc) {
            for (int a = 0; a < L0; ++a) v += (double)kap[(size_t)a * h1c].re;
        } else {
            for (int a = 0; a < Lg; ++a) v += (double)gam[((size_t)c * Lg + a) * h1c].re;
        }
        ksums[c] = v;
    }
    cpx<T> *col = Dt + (size_t)m * n0;
    for (int x = tid; x < n0; x += G) zr[pad16(x)] = col[x];
    __syncthreads();
    if (tid == 0) {
        const double k00 = ksums[nc];
        if (nc == 0) {
            const double ss2 = sigma_sci * sigma_sci, sr2 = sigma_ref * sigma_ref;
            numer = ss2 + sr2 * k00 * k00;
        } else {
            double ds = 0.0, dr = 0.0;
            for (int c = 0; c < nc; ++c) {
                const double g00 = ksums[c];
                (c < cd.ns ? ds : dr) += cd.s2[c] * g00 * g00;
            }
            numer = ds + k00 * k00 * dr;
        }
    }
    if (BLU) bluestein(zr, n0, mlen, -1, chirp, bfilt, twg, tid, G);
    else group_fft(zr, n0, -1, tw, tid, G);
    // K^(l, m) = sum_a kappa(a, m) e^(-2 pi i l a / N0): the twiddle index steps by l
    auto khat = [&](int l) {
        cpx<T> kh = mk((T)0, (T)0);
        int idx = imod(-l * w0, n0);
        for (int a = 0; a < L0; ++a) {
            kh = cadd(kh, cmul(kp[a], tw0[idx]));
            idx += l;
            if (idx >= n0) idx -= n0;
        }
        return kh;
    };
    if (nc == 0) {
        const double ss2 = sigma_sci * sigma_sci, sr2 = sigma_ref * sigma_ref;
        const T num = (T)numer;
        for (int l = tid; l < n0; l += G) {
            const cpx<T> kh = khat(l);
            const T q = sqrt(num / ((T)ss2 + (T)sr2 * (kh.re * kh.re + kh.im * kh.im)));
            zr[pad16(l)] = scale(zr[pad16(l)], q);
        }
    } else {
        // Eq. 23-24 in full: den = sum_j s_Sj^2 |G^_j|^2 + |K^|^2 sum_i s_Ri^2 |H^_i|^2,
        // normalised by its value at frequency 0 (unit kernel sum).  Eight
        // kernels at a time share each twiddle.
        const T num = (T)numer;
        constexpr int kC = 8;
        for (int l = tid; l < n0; l += G) {
            const cpx<T> kh = khat(l);
            T es = (T)0, er = (T)0;
            const int idx0 = imod(-l * cd.g0, n0);
            for (int c0 = 0; c0 < nc; c0 += kC) {
                cpx<T> gh[kC];
#pragma unroll
                for (int j = 0; j < kC; ++j) gh[j] = mk((T)0, (T)0);
                int idx = idx0;
                for (int a = 0; a < Lg; ++a) {
                    const cpx<T> w = tw0[idx];
#pragma unroll
                    for (int j = 0; j < kC; ++j)
                        if (c0 + j < nc) gh[j] = cadd(gh[j], cmul(gp[(c0 + j) * Lg + a], w));
                    idx += l;
                    if (idx >= n0) idx -= n0;
                }
#pragma unroll
                for (int j = 0; j < kC; ++j) {
                    if (c0 + j >= nc) break;
                    const T e2 = (T)cd.s2[c0 + j] * (gh[j].re * gh[j].re + gh[j].im * gh[j].im);
                    if (c0 + j < cd.ns) es += e2;
                    else er += e2;
                }
            }
            const T q = sqrt(num / (es + (kh.re * kh.re + kh.im * kh.im) * er));
            zr[pad16(l)] = scale(zr[pad16(l)], q);
        }
    }
    __syncthreads();
    if (BLU) bluestein(zr, n0, mlen, 1, chirp, bfilt, twg, tid, G);
    else group_fft(zr, n0, 1, tw, tid, G);
    const T inv = (T)1 / (T)n0;
    for (int x = tid; x < n0; x += G) col[x] = scale(zr[pad16(x)], inv);
}

template <typename T>
static cudaError_t decorr_t(Plan *p, const double *x, double xt0, double yt0, double sr, double ss,
                            const void *diff, void *out, const Coadd *co, cudaStream_t s) {
    cudaError_t err;
    const int w0 = p->cfg.w0, w1 = p->cfg.w1;
    TermWeights tw;
    basis_term_weights(p, xt0, yt0, tw.w);
    k_kernel_image<<<1, 256, 0, s>>>(p->bv, tw, x, p->kimg);
    const int tot = p->L0 * p->h1c;
    k_decorr_kappa<T><<<(tot + 255) / 256, 256, 0, s>>>(p->n1, 1, 1, w0, w1, p->kimg, nullptr,
                                                        (const cpx<T> *)p->tw1, (cpx<T> *)p->kap);
    p->launches += 2;
    CoaddDesc cd{};
    if (co) {  // row spectra of the homogenisation kernels, science then reference
        cd.ns = co->ns;
        cd.nr = co->nr;
        cd.g0 = co->g0;
        for (int c = 0; c < co->ns + co->nr; ++c) cd.s2[c] = co->sigma2[c];
        const int totc = (co->ns + co->nr) * (2 * co->g0 + 1) * p->h1c;
        k_decorr_kappa<T><<<(totc + 255) / 256, 256, 0, s>>>(p->n1, co->ns + co->nr, co->ns, co->g0, co->g1,
                                                             co->G, co->H, (const cpx<T> *)p->tw1,
                                                             (cpx<T> *)p->gam);
        p->launches++;
    }
    if ((err = cudaGetLastError())) return err;
    {  // rows
        const int G = p->m1 / 16;
        int NG = (sizeof(T) == 4 ? 1024 : 512) / G;
        if (NG < 1) NG = 1;
        if (NG > 4) NG = 4;
        if (NG > (p->n0 + 1) / 2) NG = (p->n0 + 1) / 2;
        auto smem_of = [&](int ng) { return (size_t)ng * padded_len(p->m1) * sizeof(cpx<T>); };
        while (NG > 1 && smem_of(NG) > 200 * 1024) NG /= 2;
        const size_t smem = smem_of(NG);
        const int blocks = (p->n0 + 2 * NG - 1) / (2 * NG);
        const cpx<T> *twg = (const cpx<T> *)(p->gen1 ? p->twpm1 : p->twp1);
        const cpx<T> *ch = (const cpx<T> *)p->chirp1, *bf = (const cpx<T> *)p->bfilt1;
        cpx<T> *Dt = (cpx<T> *)p->U;
#define SFFT_DROWS(I, BLU)                                                                                    \
    do {                                                                                                      \
        cudaFuncSetAttribute(k_decorr_rows<T, I, BLU>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); \
        k_decorr_rows<T, I, BLU><<<blocks, NG * G, smem, s>>>(p->n0, p->n1, p->m1, NG, (const I *)diff, twg, ch, \
                                                              bf, Dt);                                        \
    } while (0)
        if (p->cfg.dtype == SFFT_F64) {
            if (p->gen1) SFFT_DROWS(double, true);
            else SFFT_DROWS(double, false);
        } else {
            if (p->gen1) SFFT_DROWS(float, true);
            else SFFT_DROWS(float, false);
        }
#undef SFFT_DROWS
        p->launches++;
        if ((err = cudaGetLastError())) return err;
    }
    {  // columns
        const int G = p->m0 / 16;
        const int ncg = (cd.ns + cd.nr) * (2 * cd.g0 + 1);
        const size_t smem = ((size_t)p->L0 + ncg + padded_len(p->m0)) * sizeof(cpx<T>);
        auto kern = p->gen0 ? k_decorr_cols<T, true> : k_decorr_cols<T, false>;
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        kern<<<p->h1c, G, smem, s>>>(p->n0, p->n1, p->m0, w0, sr, ss, (const cpx<T> *)p->kap, (const cpx<T> *)p->tw0,
                                     (const cpx<T> *)(p->gen0 ? p->twpm0 : p->twp0), (const cpx<T> *)p->chirp0,
                                     (const cpx<T> *)p->bfilt0, (cpx<T> *)p->U, cd, (const cpx<T> *)p->gam);
        p->launches++;
        if ((err = cudaGetLastError())) return err;
    }
    p->launches++;
    return launch_rows_inv<T>(p, out, s);
}

cudaError_t decorrelate(Plan *p, const double *x, double xt0, double yt0, double sigma_ref, double sigma_sci,
                        const void *diff, void *out, const Coadd *co, cudaStream_t s) {
    return p->fp64 ? decorr_t<double>(p, x, xt0, yt0, sigma_ref, sigma_sci, diff, out, co, s)
                   : decorr_t<float>(p, x, xt0, yt0, sigma_ref, sigma_sci, diff, out, co, s);
}

cudaError_t subtract_from_rows(Plan *p, const RowForm &f, const double *x, void *diff, cudaStream_t s) {
    return p->fp64 ? sub_t<double>(p, f, x, diff, s) : sub_t<float>(p, f, x, diff, s);
}

}  // namespace sfft
