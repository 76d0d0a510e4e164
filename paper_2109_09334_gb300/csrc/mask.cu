// mask.cu -- crowded-flavor masking (Sec. 3.1): the pixels affected by
// saturated sources, for the mask argument of the build.
//
// A pixel is masked (0) when R or S reaches its saturation level anywhere in
// the square of half-width `grow` around it (Chebyshev distance, clipped at
// the image edges) or when the input mask masks it; else kept (1).
// One block per tile of ROWS rows by 256 columns.  The flags of the tile and
// its halo become bits, a warp's comparison of 32 pixels one word, so that the
// dilation along y is a shift of words and the one along x an OR of words.
// Bound by the reads of R and S (1.25 times the image with the halos); the
// comparisons are in the images' type (FP64 compares at 1/64 of the FP32 rate
// took most of an earlier, byte-wise form: 167 us at 2046 x 4094, halo 5).
#include <cuda_runtime.h>
#include <math.h>

#include "internal.h"

namespace sfft {

constexpr int kMaskWords = 8;  // words of 32 columns
constexpr int kMaxGrow = 16;
constexpr int kMaskBlocks = 200;

__host__ __device__ constexpr int mask_threads(int rows) { return rows == 64 ? 256 : 512; }
// Resident blocks per SM.  Tall tiles run where the image makes many of them:
// 8 blocks of 256 threads (32 registers) take the 1024 tiles of 4096 x 4096 in
// one wave, 6 (40 registers) leave a second, nearly empty one: 54 -> 45 us,
// halo 0.  FP64 at 6 instead of 5: 3500 x 4000 98 -> 70 us.
template <typename I>
__host__ __device__ constexpr int mask_blocks(int rows) {
    return rows == 64 ? (sizeof(I) == 4 ? 8 : 6) : 2;
}
template <typename I, int ROWS>
__global__ void __launch_bounds__(mask_threads(ROWS), mask_blocks<I>(ROWS))
    k_sat_mask(int n0, int n1, const I *__restrict__ R, const I *__restrict__ S, I sat_r, I sat_s, int grow, bool vec,
               const uint8_t *mask_in, uint8_t *mask_out) {
    constexpr int kMaskThreads = mask_threads(ROWS);
    constexpr int E = ROWS + 2 * kMaxGrow, kW = kMaskWords + 2;
    __shared__ uint32_t flag[E][kW];          // rows of tile + halo; words 0 and kW - 1 the halo along y
    __shared__ uint32_t ydil[E][kMaskWords];  // dilated along y
    __shared__ uint32_t dil[ROWS][kMaskWords];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = kMaskThreads / 32;
    const int x0 = blockIdx.y * ROWS, y0 = blockIdx.x * 32 * kMaskWords;
    const int rows = min(ROWS, n0 - x0) + 2 * grow;
    const int ylo = max(0, y0 - grow), yhi = y0 + min(n1 - y0, 32 * kMaskWords + grow);  // pixels that matter
    // Rows and words to read: all of them in tall tiles; in the others, where a
    // turn of the loads is most of the time, only those with such pixels (the
    // rest of the flags is 0).
    constexpr bool kAll = ROWS == 64;
    const int i0 = kAll ? 0 : max(0, grow - x0), ni = kAll ? rows : min(rows, n0 - x0 + grow) - i0;
    const int j0 = kAll || ylo < y0 ? 0 : 1, nj = kAll ? kW : (yhi - y0 + 31) / 32 + 1 - j0, nword = ni * nj;
    const int inv = (65535 + nj) / nj;  // t / nj = t inv >> 16 for t < 6553 and nj <= 10
    if (!kAll) {
        for (int t = tid; t < rows * kW; t += kMaskThreads) flag[0][t] = 0;
        __syncthreads();
    }
    constexpr int kU = 4;  // words in flight per warp
    for (int t0 = warp; t0 < nword; t0 += kU * nw) {
        I r[kU], s[kU];
        bool ok[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int t = t0 + u * nw, q = kAll ? t / kW : (t * inv) >> 16;
            const int x = x0 - grow + i0 + q, y = y0 - 32 + 32 * (j0 + t - q * nj) + lane;
            ok[u] = t < nword && x >= 0 && x < n0 && y >= ylo && y < yhi;
            const size_t k = ok[u] ? (size_t)x * n1 + y : 0;
            r[u] = R[k];
            s[u] = S[k];
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int t = t0 + u * nw, q = kAll ? t / kW : (t * inv) >> 16;
            const uint32_t w = __ballot_sync(0xffffffffu, ok[u] && (r[u] >= sat_r || s[u] >= sat_s));
            if (lane == 0 && t < nword) flag[i0 + q][j0 + t - q * nj] = w;
        }
    }
    __syncthreads();
    for (int t = tid; t < rows * kMaskWords; t += kMaskThreads) {
        const int i = t / kMaskWords, j = t % kMaskWords;
        const uint32_t p = flag[i][j], c = flag[i][j + 1], n = flag[i][j + 2];
        uint32_t o = c;
        for (int d = 1; d <= grow; ++d) o |= (c << d) | (p >> (32 - d)) | (c >> d) | (n << (32 - d));
        ydil[i][j] = o;
    }
    __syncthreads();
    for (int t = tid; t < (rows - 2 * grow) * kMaskWords; t += kMaskThreads) {
        const int i = t / kMaskWords, j = t % kMaskWords;
        uint32_t o = 0;
        for (int d = 0; d <= 2 * grow; ++d) o |= ydil[i + d][j];
        dil[i][j] = o;
    }
    __syncthreads();
    // four columns per thread and turn (one 4-byte store where rows and
    // pointers are 4-byte aligned)
    for (int t = tid; t < (rows - 2 * grow) * kMaskWords * 8; t += kMaskThreads) {
        const int i = t / (kMaskWords * 8), q = t % (kMaskWords * 8);
        const uint32_t bits = dil[i][q >> 3] >> (4 * (q & 7));
        const int y = y0 + 4 * q;
        const size_t k = (size_t)(x0 + i) * n1 + y;
        if (vec) {
            if (y >= n1) continue;
            uchar4 m = make_uchar4(1, 1, 1, 1);
            if (mask_in != nullptr) m = *reinterpret_cast<const uchar4 *>(mask_in + k);
            uchar4 o;
            o.x = (m.x != 0 && !(bits & 1u)) ? 1 : 0;
            o.y = (m.y != 0 && !(bits & 2u)) ? 1 : 0;
            o.z = (m.z != 0 && !(bits & 4u)) ? 1 : 0;
            o.w = (m.w != 0 && !(bits & 8u)) ? 1 : 0;
            *reinterpret_cast<uchar4 *>(mask_out + k) = o;
        } else {
            for (int e = 0; e < 4; ++e)
                if (y + e < n1)
                    mask_out[k + e] = ((mask_in == nullptr || mask_in[k + e] != 0) && !((bits >> e) & 1u)) ? 1 : 0;
        }
    }
}

// Rows per tile.  Tall tiles read less of their halos of 2 grow rows, but a
// small image makes few of them, and each waits for its loads turn by turn: the
// tallest of 64, 32, 16 and 8 that makes kMaskBlocks blocks, where blocks of a
// tall halo count for more ((rows + 2 grow) / rows).  512 x 512, halo 5: 20.7 -> 8 us
// (64 rows -> 8), FP64 24.8 -> 10.4; 1000 x 1000 FP64, halo 0: 20.7 -> 10.5 (16).
template <typename I>
static cudaError_t sat_mask(int n0, int n1, const void *R, const void *S, I sat_r, I sat_s, int grow, bool vec,
                            const uint8_t *mask_in, uint8_t *mask_out, cudaStream_t s) {
    const int cols = (n1 + 32 * kMaskWords - 1) / (32 * kMaskWords);
    int rows = 64;
    while (rows > 8 && (int64_t)cols * ((n0 + rows - 1) / rows) * (rows + 2 * grow) < (int64_t)kMaskBlocks * rows)
        rows /= 2;
    const dim3 grid(cols, (n0 + rows - 1) / rows);
    auto kern = rows == 64   ? k_sat_mask<I, 64>
                : rows == 32 ? k_sat_mask<I, 32>
                : rows == 16 ? k_sat_mask<I, 16>
                             : k_sat_mask<I, 8>;
    kern<<<grid, mask_threads(rows), 0, s>>>(n0, n1, (const I *)R, (const I *)S, sat_r, sat_s, grow, vec, mask_in,
                                             mask_out);
    return cudaGetLastError();
}

// the least float t with (double)v >= sat exactly where v >= t, for every float v
static float float_level(double sat) {
    float t = (float)sat;
    if ((double)t < sat) t = nextafterf(t, INFINITY);
    return t;
}

}  // namespace sfft

using namespace sfft;

extern "C" int sfft_saturation_mask(int32_t n0, int32_t n1, int32_t dtype, const void *d_ref, const void *d_sci,
                                    double sat_ref, double sat_sci, int32_t grow, const uint8_t *d_mask_in,
                                    uint8_t *d_mask_out, sfft_stream_t stream) {
    if (!d_ref || !d_sci || !d_mask_out) return SFFT_ERR_INVALID;
    if (n0 < 1 || n1 < 1 || grow < 0 || grow > kMaxGrow) return SFFT_ERR_INVALID;
    if (dtype != SFFT_F32 && dtype != SFFT_F64) return SFFT_ERR_INVALID;
    const bool vec = n1 % 4 == 0 && (((uintptr_t)d_mask_in | (uintptr_t)d_mask_out) & 3u) == 0;
    cudaStream_t s = (cudaStream_t)stream;
    return status_of(dtype == SFFT_F32 ? sat_mask<float>(n0, n1, d_ref, d_sci, float_level(sat_ref),
                                                         float_level(sat_sci), grow, vec, d_mask_in, d_mask_out, s)
                                       : sat_mask<double>(n0, n1, d_ref, d_sci, sat_ref, sat_sci, grow, vec, d_mask_in,
                                                          d_mask_out, s));
}
