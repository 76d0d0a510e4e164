// solve.cu -- solution of the normal equations M theta = rhs (Eq. 18).
//
// The paper names no solver.  M = C^T C is symmetric positive semidefinite;
// we factor the Jacobi-scaled matrix A = D M D (D = diag(M)^-1/2) by Cholesky
// in the plan's compute type (FP32 for the mixed path, FP64 for the plain
// path), form W = L^-1 explicitly, and refine with FP64 residuals:
//     r = rhs - M x (FP64),  x += D W^T W D r,
// until ||r|| / ||rhs|| <= 1e-12.
//
// Everything runs in one cooperative (grid-synchronised) kernel.  The
// factorisation and the inverse are one in-place sweep over an array X of
// TS x TS tiles (TS = 64 in FP32, 32 in FP64; rows padded to whole tiles, so
// that every load is a whole vector): at step k the lower triangle of X holds
// W in the block columns before k and the trailing A from there on.  A
// step is
//   * phase P: the panel of this step, TS rows over all columns c:
//       P(:, c) = Dk X(k, c)          (c before block k: row block k of W),
//       P(:, k) = Dk = L_kk^-1,
//       P(:, c) = Dk X(c, k)^T        (c after block k: L_ck^T);
//     row block k of X becomes its final W;
//   * phase U: X(i, j) -= P(:, i)^T P(:, j) for every tile j <= i, i > k (the
//     old values of block column k count as zero).  The same product updates
//     the trailing A (j > k) and W (j <= k).
// The arithmetic is that of 32-wide steps whatever TS: with TS = 64 a step is
// two of them, Dk = [D1 0; * D2] stays in its 32 x 32 parts D1, D2 and L21,
//     P1 = D1 X1,  P2 = D2 (X2 - L21 P1),
// and phase U subtracts the products of the two halves one after the other.
// Half the barriers and passes over X, the same roundings.
// Meanwhile one block per system, which takes no tasks, forms the next
// diagonal block from the tiles as the step found them: L_{k+1,k}, the last
// update of X(k+1, k+1), its factor and the inverses of that.  It arrives at
// the barrier between P and U as soon as it has read its two tiles and waits
// there only when it is done, so that its chain runs beside both phases.
//
// What bounds it (n = 1735, 27 steps): one system alone by the step's latency
// (the chain, or P, one to three rounds of tiles and two grid barriers);
// eight systems by the tiles' FP32 products and their shared-memory reads.
// One system 907 -> 515 us, eight of 507 to 1735 unknowns 1510 -> 913 us against
// 32-wide steps with two whole-grid barriers, the chain inside phase U.
//   * refinement: residual GEMV in FP64 and two GEMVs with W.
// Every control decision after a barrier uses values written before it, so
// all blocks execute the same sequence of barriers.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>


#include "common.cuh"
#include "internal.h"

namespace cg = cooperative_groups;

namespace sfft {

constexpr int kDB = 32;         // order of a block factored by one warp
constexpr int kKC = 32;         // k chunk of a tensor-core tile product
constexpr int kTile = 64;       // FP32 tile
constexpr int kMaxIters = 12;   // refinement iterations
constexpr double kTol = 1e-12;  // ||r|| / ||rhs||
constexpr int kThreads = 256;
constexpr int kBlocksPerSM = 2;  // resident FP32 solve blocks per SM (more loads in flight); FP64 takes 1
constexpr int kSeg = 8;        // row segments of the W^T y product
constexpr int kWDepth32 = 16;   // FP32 loads in flight per lane in the products with W
constexpr int kMaxBatch = kMaxSolveBatch;  // systems solved together by one launch

// Tile edge TS (also the width of a step); R x R outputs per thread of a tile
// product; KV values per 16-byte vector.  FP64 tiles are smaller because the FP64 units set their time: more
// blocks share it.
template <typename T>
struct Shape {
    static constexpr int TS = sizeof(T) == 4 ? kTile : kDB;
    static constexpr int R = TS / 16;
    static constexpr int KV = 16 / sizeof(T);
    static constexpr int LDD = kDB + KV;  // pitch of a 32 x 32 block in shared memory
    static constexpr int LDT = TS + KV;   // pitch of a TS x TS tile held by the chain
    static constexpr int kDiag = TS == kDB ? 1 : 3;  // blocks of a diagonal block: D1, D2, L21
};

template <typename T>
struct SolveArgs {
    int n, ld;  // unknowns; rows and columns of X in whole tiles
    const double *M, *rhs;
    double *dsc, *x, *r, *stats;  // stats[0..3]
    T *X, *P, *D;  // [ld][ld]; [TS][ld]; two buffers of a diagonal block, [kDiag][32][32]
    T *z, *y, *wseg;
    // [0] status (0 running, 1 converged, <0 failure), [1] iterations, [2]
    // first diagonal block with a pivot that is not positive (INT_MAX: none)
    int *flag;
    double *xout;
    sfft_solve_info *info;
};

// 16 bytes of T
template <typename T>
struct alignas(16) Vec {
    T v[Shape<T>::KV];
};
template <typename T>
__device__ __forceinline__ Vec<T> ldv(const T *p) {
    return *reinterpret_cast<const Vec<T> *>(p);
}
template <typename T>
__device__ __forceinline__ void stv(T *p, const Vec<T> &v) {
    *reinterpret_cast<Vec<T> *>(p) = v;
}
// from global memory, past L1 (other blocks wrote it in this launch)
__device__ __forceinline__ Vec<float> ldg_cg(const float *p) {
    const float4 f = __ldcg(reinterpret_cast<const float4 *>(p));
    return {{f.x, f.y, f.z, f.w}};
}
__device__ __forceinline__ Vec<double> ldg_cg(const double *p) {
    const double2 f = __ldcg(reinterpret_cast<const double2 *>(p));
    return {{f.x, f.y}};
}
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)),
                 "l"(gmem));
}

// The thread's R x R outputs of a TS x TS tile start at (tile_row, tile_col):
// a warp covers 8 x 4 threads, row and column bits interleaved in the lane
// number, so that lanes 2 apart share their column vector and lanes 1 apart
// their row vector.  Shared memory then delivers a half-warp's vectors in one
// pass.
template <typename T>
__device__ __forceinline__ int tile_row() {
    const int w = threadIdx.x >> 5, l = threadIdx.x;
    return Shape<T>::R * ((w & 1) * 8 + (((l >> 1) & 1) | ((l >> 2) & 6)));
}
template <typename T>
__device__ __forceinline__ int tile_col() {
    const int w = threadIdx.x >> 5, l = threadIdx.x;
    return Shape<T>::R * ((w >> 1) * 4 + ((l & 1) | ((l >> 1) & 2)));
}

// acc(u, v) = sum_p a[p][tile_row + u] b[p][tile_col + v], p < 32 in order, both
// operands k-major with pitch TS
template <typename T>
__device__ __forceinline__ void tile_mul(T (&acc)[Shape<T>::R][Shape<T>::R], const T *a, const T *b) {
    using S = Shape<T>;
    const T *pa = a + tile_row<T>(), *pb = b + tile_col<T>();
#pragma unroll
    for (int u = 0; u < S::R; ++u)
#pragma unroll
        for (int v = 0; v < S::R; ++v) acc[u][v] = (T)0;
#pragma unroll 8
    for (int p = 0; p < kDB; ++p) {
        const Vec<T> av = ldv(pa + p * S::TS), bv = ldv(pb + p * S::TS);
#pragma unroll
        for (int u = 0; u < S::R; ++u)
#pragma unroll
            for (int v = 0; v < S::R; ++v) acc[u][v] += av.v[u] * bv.v[v];
    }
}

// 32 x 32 product by a team of threads (t: number in it): out(i, j) = or -=
// sum_p a[p][i] b[p][j], p < 32 in order; out is kept as out[j][i].  Four rows
// and CU columns per thread: 64 threads of 4 x 4 wait for shared memory (1500
// cycles), 256 of 4 x 1 for its throughput (1260; a 16-byte read costs four
// cycles even where lanes share it); 128 of 4 x 2 lie between.  FP64 is bound
// by its units, which all threads share.  Not inlined: the chain calls it ten
// times a step and finds its code in the cache.
template <typename T, bool SUB, int TEAM>
__device__ __noinline__ void unit(const T *a, int pa, const T *b, int pb, T *out, int po, int t) {
    using S = Shape<T>;
    constexpr int KV = S::KV, CU = kDB * kDB / 4 / TEAM;
    a += 4 * (t & 7);
    b += CU * (t >> 3);
    T acc[4][CU] = {};
#pragma unroll 8
    for (int p = 0; p < kDB; ++p) {
        T av[4], bv[CU];
#pragma unroll
        for (int u = 0; u < 4; u += KV) {
            const Vec<T> w = ldv(a + p * pa + u);
#pragma unroll
            for (int i = 0; i < KV; ++i) av[u + i] = w.v[i];
        }
        if constexpr (CU == 1) {
            bv[0] = b[p * pb];
        } else if constexpr (CU == 2) {
            const cpx<T> w = *reinterpret_cast<const cpx<T> *>(b + p * pb);
            bv[0] = w.re;
            bv[1] = w.im;
        } else {
#pragma unroll
            for (int v = 0; v < CU; v += KV) {
                const Vec<T> w = ldv(b + p * pb + v);
#pragma unroll
                for (int i = 0; i < KV; ++i) bv[v + i] = w.v[i];
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < CU; ++v) acc[u][v] += av[u] * bv[v];
    }
    out += CU * (t >> 3) * po + 4 * (t & 7);
#pragma unroll
    for (int v = 0; v < CU; ++v)
#pragma unroll
        for (int u = 0; u < 4; u += KV) {
            Vec<T> w, o;
            if (SUB) o = ldv(out + v * po + u);
#pragma unroll
            for (int i = 0; i < KV; ++i) w.v[i] = SUB ? o.v[i] - acc[u + i][v] : acc[u + i][v];
            stv(out + v * po + u, w);
        }
}

// ---- the FP32 tile GEMM on the tensor cores (tcgen05, sm_100 family) --------
// The tile products of phase U run, in chunks of 32 panel rows, as tcgen05.mma of
// kind::tf32 (M = N = 64, K = 8 per instruction) with the accumulator in
// tensor memory.  TF32 keeps 10 mantissa bits, too few for a factor that
// must seed the FP64 refinement at a Jacobi-scaled condition number near
// 3e6, so each operand is split as v = hi + lo with hi = tf32(v) and
// lo = tf32(v - hi) (both rounded to nearest) and the tile product is
// accumulated as hi*hi + hi*lo + lo*hi ("3xTF32"): the dropped lo*lo term and
// the rounding of lo are below 2^-21 of each product, close to FP32.
// Operands are staged through registers into shared memory in the canonical
// K-major layout without swizzle: core matrices of 8 rows x 16 bytes, the
// next core matrix along K at +128 bytes (leading byte offset), the next
// 8-row group at +1024 bytes (stride byte offset, 32 K values per row).  One
// elected thread issues the 12 MMAs of a chunk and commits them to an
// mbarrier; the block waits on it (bounded by a clock limit), reads the
// accumulator back with tcgen05.ld and hands it to the caller in the
// register layout of tile_mul, through a shared transpose.  In tensor
// memory an M = 64 accumulator holds row 16 q + l in lane 32 q + l (q < 4,
// l < 16) and column j in column j.
constexpr int kTcCols = 64;                    // tensor-memory columns per block
constexpr long long kTcWaitCycles = 2000000000LL;  // bounded wait on the MMA barrier (~1 s)

struct __align__(1024) TcSmem {
    float op[4][kTile * kKC];  // a_hi, a_lo, b_hi, b_lo in the canonical K-major layout
};

// block-wide tensor-core state: the mbarrier, the accumulator's tensor-memory
// address, the phase of the next completion, and a sticky failure
struct TcState {
    uint64_t *mbar;
    uint32_t tmem;
    uint32_t phase;
    bool dead;
};

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// canonical K-major position (floats) of element (row i, k) in a 64 x 32 tile
__device__ __forceinline__ int tc_pos(int i, int k) { return (((i >> 3) * 8 + (k >> 2)) << 5) + ((i & 7) << 2) + (k & 3); }

__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46);
}

__device__ __forceinline__ float tf32_rn(float v) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(v));
    return __uint_as_float(r);
}

__device__ __forceinline__ void tc_mma(uint32_t tmem, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(da), "l"(db), "r"(idesc), "r"(acc));
}

// wait for completion `phase` of the mbarrier, at most kTcWaitCycles
__device__ __forceinline__ bool tc_wait(uint64_t *mbar, uint32_t phase) {
    const long long t0 = clock64();
    uint32_t done = 0;
    while (!done) {
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(smem_addr(mbar)), "r"(phase));
        if (!done && clock64() - t0 > kTcWaitCycles) return false;
    }
    return true;
}

__device__ void tc_init(TcState &st, uint64_t *mbar, uint32_t *slot) {
    if ((threadIdx.x >> 5) == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(slot)),
                     "n"(kTcCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(mbar)));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    st.mbar = mbar;
    st.tmem = *slot;
    st.phase = 0;
    st.dead = false;
}

__device__ void tc_release(TcState &st) {
    if (st.dead) tc_wait(st.mbar, st.phase);  // a commit still outstanding: one more bounded wait
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if ((threadIdx.x >> 5) == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(st.tmem), "n"(kTcCols));
}

// One chunk of kKC panel rows of a 64x64 tile product on the tensor cores:
// acc(i, j) = sum_k P[k][i0 + i] P[k][j0 + j], k0 <= k < k0 + kKC, in the
// thread layout of tile_mul.  Returns false if the MMAs did not complete
// within the wait limit (acc is then not valid).
__device__ bool tile_mul_tc(float (&acc)[4][4], TcSmem &tc, TcState &st, const float *P, int ld, int i0, int j0,
                            int k0) {
    constexpr int kLd = kTile * kKC / kThreads;
    const int tid = threadIdx.x;
    // element e = tid + q * kThreads of a 64 x 32 operand is (row, k) with
    // the lane choosing (row mod 8, k mod 4) and the rest (row / 8, k / 4):
    // a warp then stores one whole core matrix (32 consecutive words, no
    // bank conflict) and reads 4 k-rows x 32 bytes
    float ra[kLd], rb[kLd];
    int ri[kLd], rk[kLd];
#pragma unroll
    for (int q = 0; q < kLd; ++q) {
        const int e = tid + q * kThreads, l = e & 31, hi = e >> 5;
        ri[q] = (hi & 7) * 8 + (l >> 2);
        rk[q] = (hi >> 3) * 4 + (l & 3);
    }
#pragma unroll
    for (int q = 0; q < kLd; ++q) {
        const float *row = P + (size_t)(k0 + rk[q]) * ld + ri[q];
        ra[q] = __ldcg(row + i0);
        rb[q] = __ldcg(row + j0);
    }
#pragma unroll
    for (int q = 0; q < kLd; ++q) {
        const int pos = tc_pos(ri[q], rk[q]);
        const float ah = tf32_rn(ra[q]);
        tc.op[0][pos] = ah;
        tc.op[1][pos] = tf32_rn(ra[q] - ah);
        const float bh = tf32_rn(rb[q]);
        tc.op[2][pos] = bh;
        tc.op[3][pos] = tf32_rn(rb[q] - bh);
    }
    // the generic-proxy stores must be visible to the tensor core's reads
    asm volatile("fence.proxy.async.shared::cta;");
    __syncthreads();
    if (tid == 0 && !st.dead) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        constexpr uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(kTile >> 3) << 17) |
                                   ((uint32_t)(kTile >> 4) << 24);
        const uint32_t a0 = smem_addr(tc.op[0]), a1 = smem_addr(tc.op[1]);
        const uint32_t b0 = smem_addr(tc.op[2]), b1 = smem_addr(tc.op[3]);
#pragma unroll
        for (int ks = 0; ks < kKC / 8; ++ks) {
            const uint32_t off = ks * 256;  // two core matrices along K per MMA
            tc_mma(st.tmem, tc_desc(a0 + off), tc_desc(b0 + off), idesc, ks > 0);
            tc_mma(st.tmem, tc_desc(a0 + off), tc_desc(b1 + off), idesc, 1);
            tc_mma(st.tmem, tc_desc(a1 + off), tc_desc(b0 + off), idesc, 1);
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            smem_addr(st.mbar)));
    }
    bool ok = !st.dead;
    if (ok) {
        ok = tc_wait(st.mbar, st.phase);
        st.phase ^= 1u;
    }
    // every thread takes the same decision (a timeout is seen by all but is
    // not guaranteed to be simultaneous): agree before touching the result
    ok = __syncthreads_and(ok);
    if (!ok) {
        st.dead = true;
        return false;
    }
    asm volatile("tcgen05.fence::after_thread_sync;");
    // accumulator -> shared transpose (over the operand tiles, whose reads
    // are complete) -> this thread's 4x4 entries
    float *Cs = &tc.op[0][0];  // 64 x 65
    const int warp = tid >> 5, lane = tid & 31, q = warp & 3, h = warp >> 2;
    uint32_t v[32];
    const uint32_t taddr = st.tmem + ((uint32_t)(32 * q) << 16) + 32 * h;
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
        "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;");
    if (lane < 16) {
        float *row = Cs + (16 * q + lane) * (kTile + 1) + 32 * h;
#pragma unroll
        for (int c = 0; c < 32; ++c) row[c] = __uint_as_float(v[c]);
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int w = 0; w < 4; ++w) acc[u][w] = Cs[(tile_row<float>() + u) * (kTile + 1) + tile_col<float>() + w];
    __syncthreads();  // the shared tiles are refilled by the next call
    return true;
}
// 1 / sqrt(d): the FP32 factor only seeds the FP64 refinement, so the
// hardware approximation serves; FP64 takes the correctly rounded path.
__device__ __forceinline__ float inv_sqrt(float d) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
    return r;
}
__device__ __forceinline__ double inv_sqrt(double d) { return 1.0 / sqrt(d); }

// named barriers: 1..8 pass the steps of a factorisation from warp 0 to warp
// 1, kBarHelp joins the helper warps of the chain; 0 is __syncthreads
constexpr int kBarHelp = 9;
__device__ __forceinline__ void bar_sync(int id, int threads) {
    asm volatile("barrier.cta.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
    asm volatile("barrier.cta.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Two warps factor the 32x32 block A (lower triangle at s, pitch lds) and
// invert its factor, four columns per step.  Warp 0: lane r holds row r of A;
// every lane factors the 4x4 pivot block itself, and the four L entries of
// each row pass through shared memory (ex: a vector per row, then the four
// reciprocal pivots).  Warp 1 follows a step behind with the forward
// elimination of the identity, column r of Y in lane r (L Y = I); Y(r, c) goes
// to dt[c * ldd + r], zeros above the diagonal included.  Rows nb and up are
// the identity's (the caller sets them); a pivot that is not positive sets
// bad; minpiv takes the smallest of the rest.  Bound by the chain of pivots.
// (About 4.5 k cycles; a whole block taking four columns a step, with a
// barrier and an exchange each, took 12 k.)
// The steps are a loop of short code (the columns move down by four registers
// a step; 28 columns are updated in each of the first four steps and 12 in
// each of the last four, dead ones among them): unrolled, the code ran once a
// call and waited for its instructions.  In FP64 the updates take 64 cycles an
// instruction, so there the loop is unrolled and the dead columns left out.
constexpr int kExRows = kDB + 12;  // rows of ex: those of dead columns are read, not used
constexpr int kExStep = kExRows * 4 + 4;
template <typename T>
__device__ __forceinline__ void get4(const T *p, T (&o)[4]) {
#pragma unroll
    for (int v = 0; v < 4; v += Shape<T>::KV) {
        const Vec<T> w = ldv(p + v);
#pragma unroll
        for (int i = 0; i < Shape<T>::KV; ++i) o[v + i] = w.v[i];
    }
}
template <typename T>
__device__ __forceinline__ void put4(T *p, const T (&o)[4]) {
#pragma unroll
    for (int v = 0; v < 4; v += Shape<T>::KV) {
        Vec<T> w;
#pragma unroll
        for (int i = 0; i < Shape<T>::KV; ++i) w.v[i] = o[v + i];
        stv(p + v, w);
    }
}
// L entries in columns jb..jb+3 of a row from its entries r there, by the
// pivot block's L entries and reciprocal pivots
template <typename T>
__device__ __forceinline__ void lrow(const T (&r)[4], T i0, T i1, T i2, T i3, T l10, T l20, T l21, T l30, T l31, T l32,
                                     T (&l)[4]) {
    l[0] = r[0] * i0;
    l[1] = (r[1] - l[0] * l10) * i1;
    l[2] = (r[2] - l[0] * l20 - l[1] * l21) * i2;
    l[3] = (r[3] - l[0] * l30 - l[1] * l31 - l[2] * l32) * i3;
}

template <typename T, int N>
__device__ __forceinline__ void factor_steps(T (&a)[N], int jb0, T *ex, int nb, bool &bad, T &low) {
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    constexpr int U = sizeof(T) == 4 ? 1 : 4;
#pragma unroll U
    for (int jb = jb0; jb < jb0 + 16; jb += 4) {
        T pv[4][4];  // rows jb..jb+3 of the pivot block
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c <= r; ++c) pv[r][c] = __shfl_sync(kAll, a[c], jb + r);
        const T d0 = pv[0][0];
        const T i0 = inv_sqrt(d0);
        const T l10 = pv[1][0] * i0, l20 = pv[2][0] * i0, l30 = pv[3][0] * i0;
        const T d1 = pv[1][1] - l10 * l10;
        const T i1 = inv_sqrt(d1);
        const T l21 = (pv[2][1] - l20 * l10) * i1, l31 = (pv[3][1] - l30 * l10) * i1;
        const T d2 = pv[2][2] - l20 * l20 - l21 * l21;
        const T i2 = inv_sqrt(d2);
        const T l32 = (pv[3][2] - l30 * l20 - l31 * l21) * i2;
        const T d3 = pv[3][3] - l30 * l30 - l31 * l31 - l32 * l32;
        const T i3 = inv_sqrt(d3);
        const T r[4] = {a[0], a[1], a[2], a[3]};
        T lt[4];
        lrow(r, i0, i1, i2, i3, l10, l20, l21, l30, l31, l32, lt);
        T *e = ex + (jb >> 2) * kExStep;
        put4(e + lane * 4, lt);
        if (lane == 0) {
            const T iv[4] = {i0, i1, i2, i3};
            put4(e + kExRows * 4, iv);
        }
        __syncwarp();
        bar_arrive(1 + (jb >> 2), 64);
        e += (jb + 4) * 4;
#pragma unroll
        for (int c = 4; c < N; ++c) {
            if (sizeof(T) == 8 && c >= N - (jb - jb0)) continue;
            T lc[4];
            get4(e + (c - 4) * 4, lc);
            a[c - 4] = a[c] - (lt[0] * lc[0] + lt[1] * lc[1] + lt[2] * lc[2] + lt[3] * lc[3]);
        }
        const T dp[4] = {d0, d1, d2, d3};
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            if (!(dp[p] > (T)0)) bad = true;
            if (jb + p < nb && dp[p] < low) low = dp[p];
        }
    }
}
// (s: the block by columns, pitch lds)
template <typename T>
__device__ __noinline__ void factor_rows(const T *s, int lds, T *ex, int nb, bool &bad, T &minpiv) {
    const int lane = threadIdx.x & 31;
    T a[kDB], low = (T)1e30;
#pragma unroll
    for (int c = 0; c < kDB; ++c) a[c] = s[c * lds + lane];
    bool neg = bad;
    factor_steps(a, 0, ex, nb, neg, low);
    T a2[kDB / 2];
#pragma unroll
    for (int c = 0; c < kDB / 2; ++c) a2[c] = a[c];
    factor_steps(a2, 16, ex, nb, neg, low);
    bad = neg;
    if (!neg && low < minpiv) minpiv = low;
}
template <typename T, int N>
__device__ __forceinline__ void invert_steps(T (&y)[N], int jb0, const T *ex, T *dt) {
    constexpr int U = sizeof(T) == 4 ? 1 : 4;
#pragma unroll U
    for (int jb = jb0; jb < jb0 + 16; jb += 4) {
        const T *e = ex + (jb >> 2) * kExStep;
        bar_sync(1 + (jb >> 2), 64);
        T iv[4], l1[4], l2[4], l3[4], x[4];
        get4(e + kExRows * 4, iv);
        e += jb * 4;
        get4(e + 4, l1);
        get4(e + 8, l2);
        get4(e + 12, l3);
        const T r[4] = {y[0], y[1], y[2], y[3]};
        lrow(r, iv[0], iv[1], iv[2], iv[3], l1[0], l2[0], l2[1], l3[0], l3[1], l3[2], x);
        put4(dt + jb, x);
#pragma unroll
        for (int c = 4; c < N; ++c) {
            if (sizeof(T) == 8 && c >= N - (jb - jb0)) continue;
            T lc[4];
            get4(e + c * 4, lc);
            y[c - 4] = y[c] - (lc[0] * x[0] + lc[1] * x[1] + lc[2] * x[2] + lc[3] * x[3]);
        }
    }
}
template <typename T>
__device__ __noinline__ void invert_rows(const T *ex, T *dt, int ldd) {
    const int lane = threadIdx.x & 31;
    T y[kDB], y2[kDB / 2];
#pragma unroll
    for (int c = 0; c < kDB; ++c) y[c] = c == lane ? (T)1 : (T)0;
    invert_steps(y, 0, ex, dt + lane * ldd);
#pragma unroll
    for (int c = 0; c < kDB / 2; ++c) y2[c] = y[c];
    invert_steps(y2, 16, ex, dt + lane * ldd);
}

// Shared memory of the block that forms the diagonal blocks of its system.
// d is kept from step to step: [q][p] of D1(p, q), and for TS = 64 of
// D2(p, q) and L21(p, q).
template <typename T>
struct ChainSmem {
    using S = Shape<T>;
    T d[S::kDiag][kDB * S::LDD];
    T d1[kDB * S::LDD];    // the new D1 while the old one is in use
    T xt[S::TS * S::LDT];  // X(k+1, k) by columns
    T lt[S::TS * S::LDT];  // L_{k+1,k} by columns
    T s[S::TS * S::LDT];   // X(k+1, k+1) by columns
    T ex[8 * kExStep];
};

// The 32 rows a..a+31 of a panel from those of X = [X1 X2] (by columns, pitch
// px): L1 = X1 D1^T; X2 -= L1 L21^T; L2 = X2 D2^T into l1 and l2 (by columns,
// pitch pl), each followed by sync()
template <typename T, int TEAM, typename F>
__device__ __forceinline__ void panel_rows(T *x, int px, const T (*d)[kDB * Shape<T>::LDD], T *l1, T *l2, int pl,
                                           int t, F sync) {
    using S = Shape<T>;
    unit<T, false, TEAM>(x, px, d[0], S::LDD, l1, pl, t);
    sync();
    if constexpr (S::kDiag == 3) {
        unit<T, true, TEAM>(l1, pl, d[2], S::LDD, x + kDB * px, px, t);
        sync();
        unit<T, false, TEAM>(x + kDB * px, px, d[1], S::LDD, l2, pl, t);
        sync();
    }
}

// Forms diagonal block kb: with `update` its last update from step kb - 1
// (whose blocks are in c.d) first; then its own blocks into c.d and
// s.D[kb & 1].  arrive() is called once both tiles have been read.  For TS =
// 64 warps 0, 1, 4 and 5 take the first 32 rows and the first two factor them,
// while warps 2, 3, 6 and 7 (on the other schedulers) update the rest.
constexpr int kBarTeam = 10, kBarFirst = 11;  // named barriers of the chain
template <typename T, typename F>
__device__ __forceinline__ void chain_block(const SolveArgs<T> &s, ChainSmem<T> &c, int kb, bool update, bool &bad,
                                            T &minpiv, F arrive) {
    using S = Shape<T>;
    constexpr int TS = S::TS, KV = S::KV, LDD = S::LDD, LDT = S::LDT, NV = TS * TS / KV / kThreads, RG = TS / 8;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int k0 = kb * TS, nb = min(TS, s.n - k0), ld = s.ld;
    // tiles by columns: a warp reads 64 bytes of 8 rows
    Vec<T> sv[NV], xv[NV];
    auto row = [&](int q) { return ((warp + 8 * q) % RG) * 8 + (lane & 7); };
    auto col = [&](int q) { return (((warp + 8 * q) / RG) * 4 + (lane >> 3)) * KV; };
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        const T *X = s.X + (size_t)(k0 + row(q)) * ld + k0 + col(q);
        if (update) xv[q] = ldg_cg(X - TS);
        sv[q] = ldg_cg(X);
    }
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        const int r = row(q), j = col(q);
#pragma unroll
        for (int v = 0; v < KV; ++v) {
            if (update) c.xt[(j + v) * LDT + r] = xv[q].v[v];
            c.s[(j + v) * LDT + r] = r < nb ? sv[q].v[v] : (r == j + v ? (T)1 : (T)0);
        }
    }
    __syncthreads();
    arrive();
    if constexpr (TS == kDB) {
        if (update) {
            panel_rows<T, kThreads>(c.xt, LDT, c.d, c.lt, c.lt, LDT, tid, [] { __syncthreads(); });
            unit<T, true, kThreads>(c.lt, LDT, c.lt, LDT, c.s, LDT, tid);
            __syncthreads();
        }
        if (warp == 0) factor_rows<T>(c.s, LDT, c.ex, nb, bad, minpiv);
        else if (warp == 1) invert_rows<T>(c.ex, c.d[0], LDD);
        __syncthreads();
    } else {
        T *l2 = c.lt + kDB * LDT;
        const int t = (warp >> 2) * 64 + (tid & 63);  // number in the team
        if (!(warp & 2)) {
            if (update) {
                panel_rows<T, 128>(c.xt, LDT, c.d, c.lt, l2, LDT, t, [] { bar_sync(kBarTeam, 128); });
                bar_arrive(kBarFirst, 256);
                unit<T, true, 128>(c.lt, LDT, c.lt, LDT, c.s, LDT, t);
                unit<T, true, 128>(l2, LDT, l2, LDT, c.s, LDT, t);
                bar_sync(kBarTeam, 128);
            }
            if (warp == 0) factor_rows<T>(c.s, LDT, c.ex, nb, bad, minpiv);
            else if (warp == 1) invert_rows<T>(c.ex, c.d1, LDD);
        } else if (update) {
            bar_sync(kBarFirst, 256);  // the first rows' panel
            panel_rows<T, 128>(c.xt + kDB, LDT, c.d, c.lt + kDB, l2 + kDB, LDT, t, [] { bar_sync(kBarHelp, 128); });
#pragma unroll 1
            for (int j0 = 0; j0 < TS; j0 += kDB) {  // S21, S22
                T *out = c.s + j0 * LDT + kDB;
                unit<T, true, 128>(c.lt + kDB, LDT, c.lt + j0, LDT, out, LDT, t);
                unit<T, true, 128>(l2 + kDB, LDT, l2 + j0, LDT, out, LDT, t);
            }
        }
        __syncthreads();
        if (!(warp & 2)) {
            T *s22 = c.s + kDB * LDT + kDB;
            unit<T, false, 128>(c.s + kDB, LDT, c.d1, LDD, c.d[2], LDD, t);  // L21 = A21 D1^T
            bar_sync(kBarTeam, 128);
            unit<T, true, 128>(c.d[2], LDD, c.d[2], LDD, s22, LDT, t);  // A22 -= L21 L21^T
            bar_sync(kBarTeam, 128);
            if (warp == 0) factor_rows<T>(s22, LDT, c.ex, nb - kDB, bad, minpiv);
            else if (warp == 1) invert_rows<T>(c.ex, c.d[1], LDD);
        } else {
            for (int e = t; e < kDB * LDD / KV; e += 128) stv(c.d[0] + e * KV, ldv(c.d1 + e * KV));
        }
        __syncthreads();
    }
    T *D = s.D + (size_t)(kb & 1) * S::kDiag * kDB * kDB;
    for (int e = tid; e < S::kDiag * kDB * kDB / KV; e += kThreads) {
        const int q = e / (kDB / KV), g = e % (kDB / KV);
        stv(D + q * kDB + g * KV, ldv(c.d[0] + q * LDD + g * KV));
    }
    if (tid == 0 && bad && s.flag[2] > kb) s.flag[2] = kb;
    __syncthreads();
}

// Phase P task: 32 columns of the panel of step kb.
template <typename T>
struct PanelSmem {
    using S = Shape<T>;
    T d[S::kDiag][kDB * S::LDD];
    T x[S::TS * S::LDD];  // [q][c]: the chunk's columns of X(k, :), or its rows of X(:, k)
    T p[S::TS * S::LDD];  // [p][c]
};
template <typename T>
__device__ __forceinline__ void panel_task(const SolveArgs<T> &s, PanelSmem<T> &sm, int kb, int task) {
    using S = Shape<T>;
    constexpr int TS = S::TS, KV = S::KV, LDD = S::LDD, VR = kDB / KV;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, ld = s.ld;
    const int k0 = kb * TS, c0 = task * kDB;
    const T *D = s.D + (size_t)(kb & 1) * S::kDiag * kDB * kDB;
    constexpr int ND = S::kDiag * kDB * kDB / KV / kThreads, NX = TS * kDB / KV / kThreads;
    Vec<T> dv[ND], xv[NX];
#pragma unroll
    for (int q = 0; q < ND; ++q) dv[q] = ldg_cg(D + (size_t)(tid + q * kThreads) * KV);
    const bool diag = c0 >= k0 && c0 < k0 + TS, upper = c0 < k0;
    const int h0 = c0 - k0;  // (diag) first of the chunk's columns in the block
    // after block k the rows of X(:, k), transposed: a warp reads 64 bytes of 8 rows
    auto row = [&](int q) { return ((warp + 8 * q) & 3) * 8 + (lane & 7); };
    auto col = [&](int q) { return (((warp + 8 * q) >> 2) * 4 + (lane >> 3)) * KV; };
    if (!diag) {
#pragma unroll
        for (int q = 0; q < NX; ++q) {
            const int e = tid + q * kThreads;
            xv[q] = upper ? ldg_cg(s.X + (size_t)(k0 + e / VR) * ld + c0 + (e % VR) * KV)
                          : ldg_cg(s.X + (size_t)(c0 + row(q)) * ld + k0 + col(q));
        }
    }
    __syncthreads();  // the reads of the task before are done
#pragma unroll
    for (int q = 0; q < ND; ++q) {
        const int e = tid + q * kThreads;
        stv(sm.d[0] + (e / VR) * LDD + (e % VR) * KV, dv[q]);
    }
    if (!diag) {
#pragma unroll
        for (int q = 0; q < NX; ++q) {
            const int e = tid + q * kThreads;
            if (upper) {
                stv(sm.x + (e / VR) * LDD + (e % VR) * KV, xv[q]);
            } else {
#pragma unroll
                for (int v = 0; v < KV; ++v) sm.x[(col(q) + v) * LDD + row(q)] = xv[q].v[v];
            }
        }
    }
    __syncthreads();
    // P1 = D1 X1, P2 = D2 (X2 - L21 P1); in the diagonal block's own columns
    // [D1; -D2 L21 D1] and [0; D2]
    if (diag) {
        for (int e = tid; e < TS * kDB; e += kThreads) {
            const int p = e / kDB, c = e % kDB;
            if (p / kDB == h0 / kDB) sm.p[p * LDD + c] = sm.d[h0 / kDB][c * LDD + p % kDB];
            else if (h0 > 0) sm.p[p * LDD + c] = (T)0;
            else sm.x[p * LDD + c] = (T)0;  // X2
        }
        __syncthreads();
    }
    auto sync = [] { __syncthreads(); };
    if (!diag) {
        panel_rows<T, kThreads>(sm.x, LDD, sm.d, sm.p, sm.p + kDB * LDD, LDD, tid, sync);
    } else if constexpr (S::kDiag == 3) {
        if (h0 == 0) {
            T *x2 = sm.x + kDB * LDD;
            unit<T, true, kThreads>(sm.p, LDD, sm.d[2], LDD, x2, LDD, tid);
            sync();
            unit<T, false, kThreads>(x2, LDD, sm.d[1], LDD, sm.p + kDB * LDD, LDD, tid);
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NX; ++q) {
        const int e = tid + q * kThreads, p = e / VR, g = (e % VR) * KV;
        const Vec<T> v = ldv(sm.p + p * LDD + g);
        stv(s.P + (size_t)p * ld + c0 + g, v);
        if (upper || diag) stv(s.X + (size_t)(k0 + p) * ld + c0 + g, v);
    }
}

// Phase U: the tiles (i, j), kb < i < blocks, j <= i, in row order, without
// the next diagonal block (kb + 1, kb + 1), which its chain forms.
__device__ __forceinline__ int tile_count(int blocks, int kb) {
    return blocks * (blocks + 1) / 2 - (kb + 1) * (kb + 2) / 2 - 1;
}
__device__ __forceinline__ void tile_of(int kb, int task, int &i, int &j) {
    const int t = task + (kb + 1) * (kb + 2) / 2 + (task > kb ? 1 : 0);  // index in the whole lower triangle
    i = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
    if (i * (i + 1) / 2 > t) --i;
    if ((i + 1) * (i + 2) / 2 <= t) ++i;
    j = t - i * (i + 1) / 2;
}

template <typename T>
struct UpdateSmem {
    T a[2][Shape<T>::TS * Shape<T>::TS];  // P(:, i) and P(:, j) of a tile, two tiles
    T b[2][Shape<T>::TS * Shape<T>::TS];
};

template <typename T>
union __align__(1024) SolveSmem {
    ChainSmem<T> chain;
    PanelSmem<T> panel;
    UpdateSmem<T> upd;
    TcSmem tc;  // FP32 only (the tensor-core tile product)
    T red[kThreads / 32][32];
};

template <typename T>
__device__ __forceinline__ void tile_old(const SolveArgs<T> &s, int kb, int i, int j,
                                         T (&old)[Shape<T>::R][Shape<T>::R]) {
    using S = Shape<T>;
    const T *C = s.X + (size_t)(i * S::TS + tile_row<T>()) * s.ld + j * S::TS + tile_col<T>();
#pragma unroll
    for (int u = 0; u < S::R; ++u)
#pragma unroll
        for (int v = 0; v < S::R; v += S::KV) {
            Vec<T> t = {};
            if (j != kb) t = ldg_cg(C + (size_t)u * s.ld + v);
#pragma unroll
            for (int q = 0; q < S::KV; ++q) old[u][v + q] = t.v[q];
        }
}
// old -= the product of the panel rows, 32 at a time
template <typename T>
__device__ __forceinline__ void tile_update(T (&old)[Shape<T>::R][Shape<T>::R], const T *a, const T *b) {
    using S = Shape<T>;
#pragma unroll
    for (int h = 0; h < S::TS / kDB; ++h) {
        T acc[S::R][S::R];
        tile_mul(acc, a + h * kDB * S::TS, b + h * kDB * S::TS);
#pragma unroll
        for (int u = 0; u < S::R; ++u)
#pragma unroll
            for (int v = 0; v < S::R; ++v) old[u][v] -= acc[u][v];
    }
}
template <typename T>
__device__ __forceinline__ void tile_store(const SolveArgs<T> &s, int i, int j,
                                           const T (&val)[Shape<T>::R][Shape<T>::R]) {
    using S = Shape<T>;
    T *C = s.X + (size_t)(i * S::TS + tile_row<T>()) * s.ld + j * S::TS + tile_col<T>();
#pragma unroll
    for (int u = 0; u < S::R; ++u)
#pragma unroll
        for (int v = 0; v < S::R; v += S::KV) {
            Vec<T> t;
#pragma unroll
            for (int q = 0; q < S::KV; ++q) t.v[q] = val[u][v + q];
            stv(C + (size_t)u * s.ld + v, t);
        }
}

// asynchronous copies of the operands of tile (i, j) into shared memory
template <typename T>
__device__ __forceinline__ void tile_fetch(const SolveArgs<T> &s, T *a, T *b, int i, int j) {
    using S = Shape<T>;
    constexpr int VR = S::TS / S::KV;  // vectors per row
#pragma unroll
    for (int q = 0; q < S::TS * VR / kThreads; ++q) {
        const int e = threadIdx.x + q * kThreads, p = e / VR, g = (e % VR) * S::KV;
        const T *row = s.P + (size_t)p * s.ld + g;
        cp_async16(a + p * S::TS + g, row + i * S::TS);
        cp_async16(b + p * S::TS + g, row + j * S::TS);
    }
}

// pairwise sum of D partial sums (D a power of two) in a fixed order:
// neighbours first, ((a0 + a1) + (a2 + a3)) + ... 
template <typename T, int D>
__device__ __forceinline__ T tree_sum(T (&acc)[D]) {
#pragma unroll
    for (int s = 1; s < D; s *= 2)
#pragma unroll
        for (int q = 0; q + s < D; q += 2 * s) acc[q] = acc[q] + acc[q + s];
    return acc[0];
}

// sum_{j < len} a[j] b[j] by one warp (lane = this thread's lane): D partial
// sums per lane over its elements in rounds of D, what is left of an
// incomplete round in the first, added pairwise and across the warp (every
// lane returns it).  The loads of the next round are in flight during the
// products of one (the residual at n = 1735: 14.8 -> 11.6 us).
template <typename T, typename V, int D = 8>
__device__ __forceinline__ T dot_warp(const T *a, const V *b, int lane, int len) {
    T acc[D], av[D], bv[D];
#pragma unroll
    for (int q = 0; q < D; ++q) acc[q] = (T)0;
    auto fetch = [&](int j, T (&x)[D], T (&y)[D]) {
#pragma unroll
        for (int q = 0; q < D; ++q) {
            const bool in = j + 32 * q < len;
            x[q] = in ? a[j + 32 * q] : (T)0;
            y[q] = in ? (T)b[j + 32 * q] : (T)0;
        }
    };
    fetch(lane, av, bv);
    for (int j = lane; j - lane < len; j += D * 32) {
        T an[D], bn[D];
        fetch(j + D * 32, an, bn);
        if (j + (D - 1) * 32 < len) {
#pragma unroll
            for (int q = 0; q < D; ++q) acc[q] += av[q] * bv[q];
        } else {
#pragma unroll
            for (int q = 0; q < D; ++q)
                if (j + 32 * q < len) acc[0] += av[q] * bv[q];
        }
#pragma unroll
        for (int q = 0; q < D; ++q) {
            av[q] = an[q];
            bv[q] = bn[q];
        }
    }
    T r = tree_sum<T, D>(acc);
    for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    return r;
}

// sum_{k0 <= k < k1} W[k][i] y[k] by the block for 32 columns i (one per
// lane): D partial sums over the rows k = q mod D, the remaining rows in the
// first, added pairwise in a fixed order.  The warps share the partial sums,
// eight rows of each in flight.  Valid in warp 0.
template <typename T, int D>
__device__ __forceinline__ T col_dot(const T *W, const T *y, int ld, int i, int k0, int k1, T (*red)[32]) {
    constexpr int NW = kThreads / 32, P = D / NW;  // partial sums per warp
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int len = max(0, k1 - k0), m = len / D;
    T acc[P];
#pragma unroll
    for (int q = 0; q < P; ++q) acc[q] = (T)0;
    const T *Wc = W + (size_t)(k0 + P * warp) * ld + i, *yc = y + k0 + P * warp;
    for (int j = 0; j < m; j += 8) {
        T wv[8][P], yv[8][P];
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int q = 0; q < P; ++q) {
                const int k = (j + r) * D + q;
                wv[r][q] = j + r < m ? Wc[(size_t)k * ld] : (T)0;
                yv[r][q] = j + r < m ? yc[k] : (T)0;
            }
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int q = 0; q < P; ++q)
                if (j + r < m) acc[q] += wv[r][q] * yv[r][q];
    }
    if (warp == 0)
        for (int k = k0 + m * D; k < k1; ++k) acc[0] += W[(size_t)k * ld + i] * y[k];
    red[warp][lane] = tree_sum<T, P>(acc);
    __syncthreads();
    T r = (T)0;
    if (warp == 0) {
        T part[NW];
#pragma unroll
        for (int q = 0; q < NW; ++q) part[q] = red[q][lane];
        r = tree_sum<T, NW>(part);
    }
    __syncthreads();
    return r;
}

// loads in flight per lane in the refinement's products with W (compute type)
template <typename T>
__host__ __device__ constexpr int w_depth() { return sizeof(T) == 4 ? kWDepth32 : 8; }

// row i of A = D M D up to the diagonal, eight loads of each operand in flight per lane
template <typename T>
__device__ __forceinline__ void scale_row(const SolveArgs<T> &s, int i, int lane) {
    const int n = s.n;
    const double di = s.dsc[i];
    const double *Mi = s.M + (size_t)i * n;
    T *Ai = s.X + (size_t)i * s.ld;
    for (int j0 = lane; j0 <= i; j0 += 8 * 32) {
        double m[8], d[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int j = j0 + 32 * q;
            m[q] = j <= i ? Mi[j] : 0.0;
            d[q] = j <= i ? s.dsc[j] : 0.0;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int j = j0 + 32 * q;
            if (j <= i) Ai[j] = (T)(m[q] * di * d[q]);
        }
    }
}

// Up to kMaxBatch systems, of equal or different sizes, solved together:
// every phase spreads the tasks of all systems over the grid, and block b
// forms the diagonal blocks of system b, so the serial chains of the
// systems run side by side.  Each system sees the operations of a solve on
// its own, in the same order.
template <typename T>
struct BatchArgs {
    int nsys;
    long long wait;  // limit of a wait on the grid barrier, in cycles
    SolveArgs<T> sys[kMaxBatch];
};

// system of a flat task index, from the prefix sums offs[0..nsys]
__device__ __forceinline__ int sys_of(const int *offs, int nsys, int task) {
    int b = 0;
    while (b + 1 < nsys && task >= offs[b + 1]) ++b;
    return b;
}

// sum of squares of the n values of v by the whole block, in an order that
// depends on n alone; valid in thread 0
__device__ __forceinline__ double block_norm2(const double *v, int n, double *red) {
    double a = 0.0;
    for (int i0 = threadIdx.x; i0 < n; i0 += 8 * kThreads) {
        double u[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) u[q] = i0 + q * kThreads < n ? v[i0 + q * kThreads] : 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) a += u[q] * u[q];
    }
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < kThreads / 32; ++w) r += red[w];
    return r;
}

// Barrier of the whole grid after a first grid.sync (which orders the reset of
// its counter).  Unlike that of the cooperative groups an arrival does not
// wait for the counter's value, and the thread that makes it can be any.
// Waits are bounded.  One that runs out replaces a count below its target by
// kBarDead, in one atomic step: a barrier is complete for every block or for
// none, and no later one completes.  A late block may then still be writing what
// the others read, so alive() is false from then on, to all threads of a block
// alike, and the block leaves the kernel before every step whose loops and
// branches follow values in memory; what runs in between works on meaningless
// values, within its bounds.  (These checks: 471 -> 478 us for one system of 1732
// unknowns; at every barrier, 482.)  The limit (kSolveWaitCycles) is far above any
// step.
constexpr int kBarDead = 1 << 30;
struct GridBar {
    int *cnt;
    volatile int *dead;  // in shared memory
    int target;
    long long limit;
    __device__ __forceinline__ void arrive(int thread) {  // after the block's work: every thread calls it
        __syncthreads();
        if ((int)threadIdx.x == thread) {
            asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(cnt) : "memory");
        }
        target += gridDim.x;
    }
    __device__ __forceinline__ void wait() {
        if (threadIdx.x == 0) {
            const long long t0 = clock64();
            int v;
            do {
                asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(cnt) : "memory");
                // (a count that moved meanwhile is read again: at most one turn per block)
                if (v < target && clock64() - t0 > limit && atomicCAS(cnt, v, kBarDead) == v) v = kBarDead;
            } while (v < target);
            if (v >= kBarDead) *dead = 1;
        }
        __syncthreads();
    }
    __device__ __forceinline__ void sync() {
        arrive(0);
        wait();
    }
    __device__ __forceinline__ bool alive() { return *dead == 0; }  // after a wait, before the next arrive
};

__device__ __forceinline__ int multiprocessor() {
    int id;
    asm volatile("mov.u32 %0, %smid;" : "=r"(id));
    return id;
}

// The end of a launch whose barrier ran out: zero coefficients, the status, tensor
// memory released.  Every thread of the block calls it and does not return.
template <typename T, bool TC>
__device__ __noinline__ void leave(const BatchArgs<T> *ba, TcState st) {
    for (int b = 0; b < ba->nsys; ++b) {
        const SolveArgs<T> &s = ba->sys[b];
        for (int i = blockIdx.x * kThreads + threadIdx.x; i < s.n; i += gridDim.x * kThreads) s.xout[i] = 0.0;
    }
    if (blockIdx.x == 0 && (int)threadIdx.x < ba->nsys) {
        const SolveArgs<T> &s = ba->sys[threadIdx.x];
        if (s.info) {
            s.info->status = SFFT_ERR_TIMEOUT;
            s.info->iters = s.flag[1];
            s.info->rel_residual = (s.stats[1] > 0.0) ? sqrt(s.stats[2] / s.stats[1]) : sqrt(s.stats[2]);
            s.info->min_pivot = s.stats[0];
        }
    }
    if constexpr (TC) tc_release(st);
    asm volatile("exit;");
}

template <typename T, bool TC>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 4 ? kBlocksPerSM : 1)
    k_solve_coop(const __grid_constant__ BatchArgs<T> ba) {
    using S = Shape<T>;
    constexpr int TS = S::TS;
    cg::grid_group grid = cg::this_grid();
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    SolveSmem<T> &sm = *reinterpret_cast<SolveSmem<T> *>(smem_raw);
    __shared__ double red[kThreads / 32];
    __shared__ __align__(8) uint64_t tc_mbar;
    __shared__ uint32_t tc_slot;
    TcState st{};
    if constexpr (TC) tc_init(st, &tc_mbar, &tc_slot);
    const int tid = threadIdx.x, bid = blockIdx.x, nbk = gridDim.x;
    const int gtid = bid * kThreads + tid, gthreads = nbk * kThreads;
    // warp tasks: consecutive ones on different blocks, so that every
    // multiprocessor gets its share of a short list (its FP64 units bound the
    // residual and the scaling)
    const int warp = tid >> 5, lane = tid & 31, nw = kThreads / 32;
    const int wtask = warp * nbk + bid, wstep = nbk * nw;
    const int nsys = ba.nsys;
    // sizes may differ between systems: rows of all systems as one flat range
    int nrow[kMaxBatch + 1];
    int wofs[kMaxBatch + 1];  // flat W^T y tasks of all systems
    int yofs[kMaxBatch + 1];  // flat row-pair tasks (k, n - 1 - k) of all systems
    nrow[0] = wofs[0] = yofs[0] = 0;
    int nblk_max = 0;
    for (int b = 0; b < nsys; ++b) {
        const int n = ba.sys[b].n;
        nrow[b + 1] = nrow[b] + n;
        wofs[b + 1] = wofs[b] + ((n + 31) / 32) * kSeg;
        yofs[b + 1] = yofs[b] + (n + 1) / 2;
        nblk_max = max(nblk_max, ba.sys[b].ld / TS);
    }
    const int nrows_all = nrow[nsys];

    __shared__ int rank_s;
    int *workers = reinterpret_cast<int *>(ba.sys[0].stats + 4);
    // ---- status reset; Jacobi scaling, zero x and the padding rows of X ------
    if (bid == 0 && tid < nsys) {
        const SolveArgs<T> &s = ba.sys[tid];
        s.flag[0] = s.flag[1] = s.flag[3] = 0;
        s.flag[2] = INT_MAX;
        s.stats[0] = 1e300;
        s.stats[1] = s.stats[2] = s.stats[3] = 0.0;
        if (tid == 0) *workers = 0;
    }
    // A block that shares its multiprocessor with one that forms diagonal
    // blocks takes no tasks of the factorisation: the chain would wait for its
    // instructions.  The others draw their numbers.
    if (bid < nsys && tid == 0) reinterpret_cast<int *>(ba.sys[bid].stats + 5)[0] = multiprocessor();
    grid.sync();
    __shared__ int dead_s;
    if (tid == 0) dead_s = 0;
    GridBar bar{&ba.sys[0].flag[3], &dead_s, 0, ba.wait};
    if (bid >= nsys && tid == 0) {
        bool own = true;
        for (int b = 0; b < nsys; ++b)
            own = own && reinterpret_cast<const int *>(ba.sys[b].stats + 5)[0] != multiprocessor();
        rank_s = own ? atomicAdd(workers, 1) : -1;
    }
    for (int b = 0; b < nsys; ++b) {
        const SolveArgs<T> &s = ba.sys[b];
        const int n = s.n;
        for (int i = gtid; i < n; i += gthreads) {
            const double d = s.M[(size_t)i * n + i];
            if (!(d > 0.0)) s.flag[0] = SFFT_ERR_SINGULAR;
            s.dsc[i] = (d > 0.0) ? 1.0 / sqrt(d) : 0.0;
            s.x[i] = 0.0;
        }
        for (int e = gtid; e < (s.ld - n) * s.ld; e += gthreads) s.X[(size_t)n * s.ld + e] = (T)0;
    }
    bar.sync();
    // A = D M D on the lower triangle (nothing reads the upper one), one warp
    // per row pair (k, n - 1 - k)
    for (int task = wtask; task < yofs[nsys]; task += wstep) {
        const int b = sys_of(yofs, nsys, task), k = task - yofs[b];
        const SolveArgs<T> &s = ba.sys[b];
        scale_row(s, k, lane);
        if (s.n - 1 - k != k) scale_row(s, s.n - 1 - k, lane);
    }
    bar.sync();

    // ---- Cholesky and W = L^-1 ----------------------------------------------
    // A system whose status turned negative is skipped from then on, and one
    // whose steps are done waits for the larger ones.  The task counts must be
    // the same in every block: a chain that fails while step kb runs records
    // block kb + 1, which the test of step kb reads the same way before and
    // after.
    // (no worker left: a small grid set by hand; then all share the tasks)
    const int nown = *workers, nwork = nown > 0 ? nown : nbk - nsys;
    const int rank = bid < nsys ? -1 : (nown > 0 ? rank_s : bid - nsys);
    bool bad = false;  // of the chain of system bid (thread 0)
    T minpiv = (T)1e30;
    const bool first = bid < nsys && ba.sys[bid].flag[0] == 0;
    if (!bar.alive()) leave<T, TC>(&ba, st);
    if (first) chain_block(ba.sys[bid], sm.chain, 0, false, bad, minpiv, [] {});
    bar.sync();
    for (int kb = 0; kb < nblk_max; ++kb) {
        unsigned live = 0;
        bool more = false;
        int poff[kMaxBatch + 1], uoff[kMaxBatch + 1];
        poff[0] = uoff[0] = 0;
        for (int b = 0; b < nsys; ++b) {
            const SolveArgs<T> &s = ba.sys[b];
            const int blocks = s.ld / TS;
            int np = 0, nu = 0;
            if (kb < blocks && s.flag[0] == 0 && s.flag[2] > kb) {
                live |= 1u << b;
                np = s.ld / kDB;
                if (kb + 1 < blocks) {
                    more = true;
                    nu = tile_count(blocks, kb);
                }
            }
            poff[b + 1] = poff[b] + np;
            uoff[b + 1] = uoff[b] + nu;
        }
        if (!bar.alive()) leave<T, TC>(&ba, st);
        const bool chain = bid < nsys && (live & (1u << bid)) && kb + 1 < ba.sys[bid].ld / TS;
        if (chain) {
            chain_block(ba.sys[bid], sm.chain, kb + 1, true, bad, minpiv, [&] { bar.arrive(kThreads - 1); });
            bar.wait();
        } else {
            if (rank >= 0) {
                for (int task = rank; task < poff[nsys]; task += nwork) {
                    const int b = sys_of(poff, nsys, task);
                    panel_task(ba.sys[b], sm.panel, kb, task - poff[b]);
                }
            }
            bar.sync();
        }
        if (!more) break;  // every system's steps are done (same in every block)
        if (rank >= 0) {
            const int step = nwork, total = uoff[nsys];
            if constexpr (TC && sizeof(T) == 4) {
                for (int task = rank; task < total; task += step) {
                    const int b = sys_of(uoff, nsys, task);
                    const SolveArgs<T> &s = ba.sys[b];
                    int i, j;
                    tile_of(kb, task - uoff[b], i, j);
                    T old[4][4];
                    tile_old(s, kb, i, j, old);
                    bool ok = true;
                    for (int kk = 0; kk < TS && ok; kk += kKC) {
                        T part[4][4];
                        ok = tile_mul_tc(part, sm.tc, st, s.P, s.ld, i * TS, j * TS, kk);
#pragma unroll
                        for (int u = 0; u < 4; ++u)
#pragma unroll
                            for (int v = 0; v < 4; ++v) old[u][v] -= part[u][v];
                    }
                    if (!ok) {  // a wait that timed out: flag the system, redo the tile on the CUDA cores
                        if (tid == 0) s.flag[0] = SFFT_ERR_TIMEOUT;
                        tile_old(s, kb, i, j, old);
                        tile_fetch(s, sm.upd.a[0], sm.upd.b[0], i, j);
                        asm volatile("cp.async.wait_all;\n" ::: "memory");
                        __syncthreads();
                        tile_update(old, sm.upd.a[0], sm.upd.b[0]);
                        __syncthreads();
                    }
                    tile_store(s, i, j, old);
                }
            } else {
                // the operands of the next tile arrive while this one's product runs
                int task = rank, b = 0, i = 0, j = 0, buf = 0;
                auto fetch = [&](int t, int &fb, int &fi, int &fj, int to) {
                    fb = sys_of(uoff, nsys, t);
                    tile_of(kb, t - uoff[fb], fi, fj);
                    tile_fetch(ba.sys[fb], sm.upd.a[to], sm.upd.b[to], fi, fj);
                    asm volatile("cp.async.commit_group;\n" ::: "memory");
                };
                __syncthreads();  // phase P's shared memory is free
                if (task < total) fetch(task, b, i, j, 0);
                while (task < total) {
                    const SolveArgs<T> &s = ba.sys[b];
                    const int next = task + step;
                    int nb_ = 0, ni = 0, nj = 0;
                    T old[S::R][S::R];
                    tile_old(s, kb, i, j, old);
                    if (next < total) {
                        fetch(next, nb_, ni, nj, buf ^ 1);
                        asm volatile("cp.async.wait_group 1;\n" ::: "memory");
                    } else {
                        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
                    }
                    __syncthreads();
                    tile_update(old, sm.upd.a[buf], sm.upd.b[buf]);
                    tile_store(s, i, j, old);
                    __syncthreads();  // before this buffer is filled again
                    task = next;
                    b = nb_;
                    i = ni;
                    j = nj;
                    buf ^= 1;
                }
            }
        }
        bar.sync();
    }

    if (bid < nsys && tid == 0 && (double)minpiv < ba.sys[bid].stats[0]) ba.sys[bid].stats[0] = (double)minpiv;

    // ---- refinement ---------------------------------------------------------
    // done: bit b set once system b has converged, failed or run out of
    // iterations; every block derives it from the same values.  The norms
    // are sums over the rows in one fixed order, so the decisions do not depend
    // on the grid or the batch.
    unsigned done = 0;
    for (int b = 0; b < nsys; ++b)
        if (ba.sys[b].flag[0] != 0 || ba.sys[b].flag[2] != INT_MAX) done |= 1u << b;
    if (!bar.alive()) leave<T, TC>(&ba, st);
    const unsigned all = (1u << nsys) - 1u;
    for (int it = 0; it <= kMaxIters && done != all; ++it) {
        // r = rhs - M x (FP64); z = D r
        for (int row = wtask; row < nrows_all; row += wstep) {
            const int b = sys_of(nrow, nsys, row), i = row - nrow[b];
            if (done & (1u << b)) continue;
            const SolveArgs<T> &s = ba.sys[b];
            const double a = dot_warp<double>(s.M + (size_t)i * s.n, s.x, lane, s.n);
            const double ri = s.rhs[i] - a;
            if (lane == 0) {
                s.r[i] = ri;
                s.z[i] = (T)(s.dsc[i] * ri);
            }
        }
        bar.sync();
        // ||r||^2 (and first ||rhs||^2) of system b by block b, beside the
        // product y = W z of the others: the next barrier serves both
        if (bid < nsys && !(done & (1u << bid))) {
            const SolveArgs<T> &s = ba.sys[bid];
            const double rr = block_norm2(s.r, s.n, red);
            if (it == 0) {
                const double bb = block_norm2(s.rhs, s.n, red);
                if (tid == 0) s.stats[1] = bb;
            }
            if (tid == 0) s.stats[2] = rr;
        }
        // y = W z  (W lower triangular; row i has i + 1 entries).  A warp task
        // takes rows k and n - 1 - k, n + 1 entries together, so that every
        // task has the same length.
        for (int task = bid < nsys ? yofs[nsys] : warp * (nbk - nsys) + bid - nsys; task < yofs[nsys];
             task += (nbk - nsys) * nw) {
            const int b = sys_of(yofs, nsys, task), k = task - yofs[b];
            if (done & (1u << b)) continue;
            const SolveArgs<T> &s = ba.sys[b];
            const int i2 = s.n - 1 - k;
            const T a = dot_warp<T, T, w_depth<T>()>(s.X + (size_t)k * s.ld, s.z, lane, k + 1);
            if (lane == 0) s.y[k] = a;
            if (i2 != k) {
                const T a2 = dot_warp<T, T, w_depth<T>()>(s.X + (size_t)i2 * s.ld, s.z, lane, i2 + 1);
                if (lane == 0) s.y[i2] = a2;
            }
        }
        bar.sync();
        for (int b = 0; b < nsys; ++b) {
            if (done & (1u << b)) continue;
            const SolveArgs<T> &s = ba.sys[b];
            const double bb = s.stats[1], rr = s.stats[2];
            if (rr <= kTol * kTol * (bb > 0.0 ? bb : 1.0) || rr == 0.0) {
                if (bid == 0 && tid == 0) s.flag[0] = 1;
                done |= 1u << b;
            } else if (it == kMaxIters) {
                if (bid == 0 && tid == 0) s.flag[0] = SFFT_ERR_NOT_CONVERGED;
                done |= 1u << b;
            }
        }
        if (!bar.alive()) leave<T, TC>(&ba, st);
        if (done == all) break;
        // w = W^T y in kSeg row segments (coalesced rows of W), summed in a fixed order
        for (int task = bid; task < wofs[nsys]; task += nbk) {
            const int b = sys_of(wofs, nsys, task), q = task - wofs[b];
            if (done & (1u << b)) continue;
            const SolveArgs<T> &s = ba.sys[b];
            const int n = s.n;
            const int segrows = (n + kSeg - 1) / kSeg;
            const int ch = q / kSeg, sg = q % kSeg;
            const int i = ch * 32 + lane;
            const int k0 = max(ch * 32, sg * segrows), k1 = min(n, (sg + 1) * segrows);
            // (columns n and up of the last chunk are padding; their sums are not stored)
            const T a = col_dot<T, w_depth<T>()>(s.X, s.y, s.ld, i, k0, k1, sm.red);
            if (warp == 0 && i < n) s.wseg[(size_t)sg * n + i] = a;
        }
        bar.sync();
        for (int e = gtid; e < nrows_all; e += gthreads) {
            const int b = sys_of(nrow, nsys, e), i = e - nrow[b];
            if (done & (1u << b)) continue;
            const SolveArgs<T> &s = ba.sys[b];
            T a = (T)0;
#pragma unroll
            for (int sg = 0; sg < kSeg; ++sg) a += s.wseg[(size_t)sg * s.n + i];
            s.x[i] += s.dsc[i] * (double)a;
        }
        if (bid == 0 && tid < nsys && !(done & (1u << tid))) ba.sys[tid].flag[1] += 1;
        bar.sync();
    }
    // ---- results ------------------------------------------------------------
    for (int e = gtid; e < nrows_all; e += gthreads) {
        const int b = sys_of(nrow, nsys, e), i = e - nrow[b];
        ba.sys[b].xout[i] = ba.sys[b].x[i];
    }
    __syncthreads();  // (block 0: its first thread wrote the statuses)
    if (bid == 0 && tid < nsys) {
        const SolveArgs<T> &s = ba.sys[tid];
        if (s.info) {
            int f = s.flag[0];
            if (f == 0) f = s.flag[2] != INT_MAX ? SFFT_ERR_SINGULAR : SFFT_ERR_NOT_CONVERGED;
            s.info->status = (f == 1) ? SFFT_OK : f;
            s.info->iters = s.flag[1];
            s.info->rel_residual = (s.stats[1] > 0.0) ? sqrt(s.stats[2] / s.stats[1]) : sqrt(s.stats[2]);
            s.info->min_pivot = s.stats[0];
        }
    }
    if constexpr (TC) tc_release(st);
}

static size_t solve_dyn_smem(bool fp64) { return fp64 ? sizeof(SolveSmem<double>) : sizeof(SolveSmem<float>); }

// Arguments of one system: the caller's M, rhs, x, info and the workspace.
template <typename T>
static SolveArgs<T> system_args(int n, const double *M, const double *rhs, double *x, sfft_solve_info *info,
                                double *dsc, double *xw, double *r, void *A, void *zv, int *flag) {
    constexpr int TS = Shape<T>::TS;
    SolveArgs<T> a;
    a.n = n;
    a.ld = (n + TS - 1) / TS * TS;
    a.M = M;
    a.rhs = rhs;
    a.dsc = dsc;
    a.x = xw;
    a.r = r;
    a.stats = xw + n;
    a.X = (T *)A;
    a.P = a.X + (size_t)a.ld * a.ld;
    a.D = a.P + (size_t)TS * a.ld;
    a.z = (T *)zv;
    a.y = (T *)zv + n;
    a.wseg = (T *)zv + 2 * (size_t)n;
    a.flag = flag;
    a.xout = x;
    a.info = info;
    return a;
}

size_t solve_matrix_elems(int n, bool fp64) {
    const size_t ts = fp64 ? Shape<double>::TS : Shape<float>::TS, ld = (n + ts - 1) / ts * ts;
    return ld * ld + ts * ld + 2 * 3 * kDB * kDB;
}

// the kernel variant: tile products on the tensor cores (FP32 only) or not
static const void *solve_kernel(bool fp64, bool tc) {
    if (fp64) return (const void *)k_solve_coop<double, false>;
    return tc ? (const void *)k_solve_coop<float, true> : (const void *)k_solve_coop<float, false>;
}

template <typename T>
static cudaError_t launch_batch(const BatchArgs<T> &ba, int grid, cudaStream_t st, bool tc = false) {
    if (grid <= ba.nsys) return cudaErrorInvalidConfiguration;  // blocks >= nsys take the shared tasks
    void *args[] = {(void *)&ba};
    const void *kern = solve_kernel(sizeof(T) == 8, tc);
    return cudaLaunchCooperativeKernel(kern, grid, kThreads, args, solve_dyn_smem(sizeof(T) == 8), st);
}

template <typename T>
static cudaError_t solve_batch_t(Plan *const *plans, int count, const double *const *M, const double *const *rhs,
                                 double *const *x, sfft_solve_info *const *info, cudaStream_t st) {
    BatchArgs<T> ba;
    ba.nsys = count;
    ba.wait = plans[0]->solve_wait;
    for (int b = 0; b < count; ++b) {
        Plan *p = plans[b];
        ba.sys[b] = system_args<T>(p->n, M[b], rhs[b], x[b], info[b], p->dscale, p->xw, p->r, p->A, p->zv, p->flag);
    }
    // the tensor-core tile variant (tune_tc = 2, FP32 only) allocates tensor
    // memory, which limits it to one block per SM: its own grid
    const bool tc = sizeof(T) == 4 && plans[0]->tune_tc == 2 && plans[0]->solve_grid_tc > count;
    const int full = tc ? plans[0]->solve_grid_tc : plans[0]->solve_grid;
    const int sg = plans[0]->tune_sgrid;
    int grid = full;
    if (sg > count && sg <= full) {
        grid = sg;  // set by hand
    } else if (count == 1 && !tc && sizeof(T) == 4 && full >= 2 * kMaxSolveBatch) {
        // one system alone: one block per SM (the step's latency, not the
        // tile throughput, sets its time; us on 152 and on 304 blocks: 70 and 75 at
        // n = 84, 156 and 163 at 508, 471 and 515 at 1732, 1137 and 1154 at 2884; only
        // systems far above those of the fits in use are the other way round, 4851
        // and 4143 at 5284); several: every resident block
        grid = full / kBlocksPerSM;
    }
    const cudaError_t err = launch_batch(ba, grid, st, tc);
    plans[0]->launches += 1;
    return err;
}

cudaError_t solve_batch(Plan *const *plans, int count, const double *const *M, const double *const *rhs,
                        double *const *x, sfft_solve_info *const *info, cudaStream_t s) {
    if (count < 1 || count > kMaxBatch) return cudaErrorInvalidValue;
    for (int b = 1; b < count; ++b)  // sizes may differ
        if (plans[b]->fp64 != plans[0]->fp64 || (!plans[0]->fp64 && plans[b]->solve_panel != plans[0]->solve_panel))
            return cudaErrorInvalidValue;
    return plans[0]->fp64 ? solve_batch_t<double>(plans, count, M, rhs, x, info, s)
                          : solve_batch_t<float>(plans, count, M, rhs, x, info, s);
}

cudaError_t solve_system(Plan *p, const double *M, const double *rhs, double *x, sfft_solve_info *info,
                         cudaStream_t s) {
    return solve_batch(&p, 1, &M, &rhs, &x, &info, s);
}

int solve_grid_size(bool fp64, bool tc) {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const size_t dsm = solve_dyn_smem(fp64);
    // all of the unified L1/shared storage as shared memory, so that two FP32
    // blocks (76.8 KB of shared memory each) fit on an SM
    const void *kern = solve_kernel(fp64, tc);
    cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dsm);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, kThreads, dsm);
    if (per < 1 || sms < 1) return 0;
    const int g = sms * (per < kBlocksPerSM ? per : kBlocksPerSM);
    return g <= kMaxSolveGrid ? g : 0;
}

size_t solve_vec_elems(int n) { return (size_t)(2 + kSeg) * n; }

template <typename T>
static cudaError_t solve_buf_t(const SolveBuffers &b, const double *M, const double *rhs, double *x,
                               sfft_solve_info *info, cudaStream_t st) {
    BatchArgs<T> ba;
    ba.nsys = 1;
    ba.wait = kSolveWaitCycles;
    ba.sys[0] = system_args<T>(b.n, M, rhs, x, info, b.dsc, b.xw, b.r, b.A, b.zv, b.flag);
    return launch_batch(ba, b.grid, st);
}

cudaError_t solve_on_buffers(const SolveBuffers &b, const double *M, const double *rhs, double *x,
                             sfft_solve_info *info, cudaStream_t s) {
    return b.fp64 ? solve_buf_t<double>(b, M, rhs, x, info, s) : solve_buf_t<float>(b, M, rhs, x, info, s);
}

}  // namespace sfft
