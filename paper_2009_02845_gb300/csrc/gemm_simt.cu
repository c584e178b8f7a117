// Binary32 CUDA-core GEMM used by the FP32 precision form of the sketched
// products (A = M S, B = V^T S, R = A B^T; Section 3.3 eq. def_A_B and the
// gradient terms of eq. gradient_descent), with operand layouts and optional
// row gathers so the same kernel serves the Gaussian, subsampling and
// identity sketches without copies.
//
// Each output is one FMA chain in increasing l whatever the tile, so results are
// deterministic and do not depend on the tile chosen.  Two tiles:
//   64 x 64   4 x 4 outputs per thread, the next tile's loads in flight (a 128 x 128 tile
//             of 8 x 8, staged without prefetch, was slower at every size: 65,536 x 64 from
//             2,048 450 against 1,170 us, 13,500 x 500 from 5,000 1.87 against 3.24 ms);
//   16 x 16   one output per thread, for results with too few large tiles and a long K
//             (256 x 256 from 8,192 rows: 142 us, 347 on 16 of the large tiles, 1,590 on
//             four of 128 x 128): operands K-contiguous in shared memory, so four steps of
//             a chain take two 16-byte loads.  Bound by shared-memory wavefronts (two
//             per K and warp).
#include "common.cuh"
#include "kernels.cuh"

namespace dsanls {

// ---- 64 x 64 tile -----------------------------------------------------------
constexpr int MT = 64, MK = 16;

template <bool AK, bool BKC>
__global__ void __launch_bounds__(256)
    k_sgemm_mid(int64_t M, int64_t N, int64_t K, const float *__restrict__ A, int64_t lda,
                const int32_t *__restrict__ ga, const float *__restrict__ B, int64_t ldb,
                const int32_t *__restrict__ gb, float *__restrict__ C, int64_t ldc, float alpha, int64_t kchunk,
                int64_t c_split_stride, int avec, int bvec) {
    __shared__ __align__(16) float As[2][MK][MT + 4], Bs[2][MK][MT + 4];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int64_t ntn = ceil_div(N, MT), m0 = (blockIdx.x / ntn) * MT, n0 = (blockIdx.x % ntn) * MT;
    const int64_t kbeg = (int64_t)blockIdx.y * kchunk, kend = min(K, kbeg + kchunk);
    C += (int64_t)blockIdx.y * c_split_stride;
    // four elements of a 64 x 16 operand tile per thread: K contiguous (row, 4 K) or rows contiguous (K, 4 rows)
    auto load = [&](const float *P, int64_t ld, const int32_t *g, bool kc, bool vec, int64_t r0, int64_t rows,
                    int64_t k0, float (&v)[4]) {
        if (kc) {
            const int64_t r = r0 + (tid >> 2), k = k0 + 4 * (tid & 3);
            if (vec && r < rows && k + 4 <= kend) {
                const float4 x = *reinterpret_cast<const float4 *>(P + r * ld + k);
                v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = (r < rows && k + e < kend) ? P[r * ld + k + e] : 0.0f;
            }
        } else {
            const int64_t k = k0 + (tid >> 4), r = r0 + 4 * (tid & 15);
            const float *q = k < kend ? P + (g ? (int64_t)g[k] : k) * ld + r : P;
            if (vec && k < kend && r + 4 <= rows) {
                const float4 x = *reinterpret_cast<const float4 *>(q);
                v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = (k < kend && r + e < rows) ? q[e] : 0.0f;
            }
        }
    };
    auto store = [&](float (*T)[MT + 4], bool kc, const float (&v)[4]) {
        if (kc) {
#pragma unroll
            for (int e = 0; e < 4; ++e) T[4 * (tid & 3) + e][tid >> 2] = v[e];
        } else {
            *reinterpret_cast<float4 *>(&T[tid >> 4][4 * (tid & 15)]) = make_float4(v[0], v[1], v[2], v[3]);
        }
    };
    float acc[4][4], va[4], vb[4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.0f;
    load(A, lda, ga, AK, avec, m0, M, kbeg, va);
    load(B, ldb, gb, BKC, bvec, n0, N, kbeg, vb);
    int cur = 0;
    for (int64_t k0 = kbeg; k0 < kend; k0 += MK, cur ^= 1) {
        store(As[cur], AK, va);
        store(Bs[cur], BKC, vb);
        __syncthreads();  // (the other buffer was last read before this barrier)
        if (k0 + MK < kend) {
            load(A, lda, ga, AK, avec, m0, M, k0 + MK, va);
            load(B, ldb, gb, BKC, bvec, n0, N, k0 + MK, vb);
        }
#pragma unroll
        for (int l = 0; l < MK; ++l) {
            const float4 x = *reinterpret_cast<const float4 *>(&As[cur][l][4 * ty]);
            const float4 y = *reinterpret_cast<const float4 *>(&Bs[cur][l][4 * tx]);
            const float xa[4] = {x.x, x.y, x.z, x.w}, yb[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = __fmaf_rn(xa[a], yb[b], acc[a][b]);
        }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int64_t i = m0 + 4 * ty + a;
        if (i >= M) continue;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int64_t j = n0 + 4 * tx + b;
            if (j < N) C[i * ldc + j] = __fmul_rn(alpha, acc[a][b]);
        }
    }
}

// ---- 16 x 16 tile -----------------------------------------------------------
constexpr int ST = 16, SK = 64;

template <bool AK, bool BKC>
__global__ void __launch_bounds__(256)
    k_sgemm_small(int64_t M, int64_t N, int64_t K, const float *__restrict__ A, int64_t lda,
                  const int32_t *__restrict__ ga, const float *__restrict__ B, int64_t ldb,
                  const int32_t *__restrict__ gb, float *__restrict__ C, int64_t ldc, float alpha, int64_t kchunk,
                  int64_t c_split_stride) {
    // [row][K]: rows 68 floats apart, so the 8 rows of a 16-byte phase fall on different banks
    __shared__ __align__(16) float As[2][ST][SK + 4], Bs[2][ST][SK + 4];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int64_t ntn = ceil_div(N, ST), m0 = (blockIdx.x / ntn) * ST, n0 = (blockIdx.x % ntn) * ST;
    const int64_t kbeg = (int64_t)blockIdx.y * kchunk, kend = min(K, kbeg + kchunk);
    C += (int64_t)blockIdx.y * c_split_stride;
    // four elements of a 16 x 64 operand tile per thread
    auto load = [&](const float *P, int64_t ld, const int32_t *g, bool kc, int64_t r0, int64_t rows, int64_t k0,
                    float (&v)[4]) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int u = tid + 256 * e;
            const int64_t r = r0 + (kc ? u >> 6 : u & 15), k = k0 + (kc ? u & 63 : u >> 4);
            float x = 0.0f;
            if (r < rows && k < kend) x = kc ? P[r * ld + k] : P[(g ? (int64_t)g[k] : k) * ld + r];
            v[e] = x;
        }
    };
    auto store = [&](float (*T)[SK + 4], bool kc, const float (&v)[4]) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int u = tid + 256 * e;
            T[kc ? u >> 6 : u & 15][kc ? u & 63 : u >> 4] = v[e];
        }
    };
    float acc = 0.0f, va[2][4], vb[2][4];  // two tiles in flight: one step of 64 K is shorter than a load
    load(A, lda, ga, AK, m0, M, kbeg, va[0]);
    load(B, ldb, gb, BKC, n0, N, kbeg, vb[0]);
    load(A, lda, ga, AK, m0, M, kbeg + SK, va[1]);
    load(B, ldb, gb, BKC, n0, N, kbeg + SK, vb[1]);
    for (int64_t k0 = kbeg; k0 < kend; k0 += 2 * SK) {
#pragma unroll
        for (int cur = 0; cur < 2; ++cur) {
            if (k0 + cur * SK >= kend) break;
            store(As[cur], AK, va[cur]);
            store(Bs[cur], BKC, vb[cur]);
            __syncthreads();
            load(A, lda, ga, AK, m0, M, k0 + (cur + 2) * SK, va[cur]);
            load(B, ldb, gb, BKC, n0, N, k0 + (cur + 2) * SK, vb[cur]);
#pragma unroll
            for (int l = 0; l < SK; l += 4) {
                const float4 x = *reinterpret_cast<const float4 *>(&As[cur][ty][l]);
                const float4 y = *reinterpret_cast<const float4 *>(&Bs[cur][tx][l]);
                acc = __fmaf_rn(x.x, y.x, acc);
                acc = __fmaf_rn(x.y, y.y, acc);
                acc = __fmaf_rn(x.z, y.z, acc);
                acc = __fmaf_rn(x.w, y.w, acc);
            }
        }
    }
    const int64_t i = m0 + ty, j = n0 + tx;
    if (i < M && j < N) C[i * ldc + j] = __fmul_rn(alpha, acc);
}

template <bool AK, bool BKC>
static void dispatch(const GemmArgs &g, int tile, cudaStream_t s) {
    const int splits = g.splits < 1 ? 1 : g.splits;
    const int64_t kchunk = ceil_div(ceil_div(g.K, splits), 8) * 8;
    const dim3 grid((unsigned)(ceil_div(g.N, tile) * ceil_div(g.M, tile)), (unsigned)splits);
    if (tile == MT) {
        const int avec = g.lda % 4 == 0 && ((uintptr_t)g.A & 15) == 0 && (!AK || kchunk % 4 == 0);
        const int bvec = g.ldb % 4 == 0 && ((uintptr_t)g.B & 15) == 0 && (!BKC || kchunk % 4 == 0);
        k_sgemm_mid<AK, BKC><<<grid, 256, 0, s>>>(g.M, g.N, g.K, g.A, g.lda, g.ga, g.B, g.ldb, g.gb, g.C, g.ldc, g.alpha,
                                                  kchunk, g.c_split_stride, avec, bvec);
    } else {
        k_sgemm_small<AK, BKC><<<grid, 256, 0, s>>>(g.M, g.N, g.K, g.A, g.lda, g.ga, g.B, g.ldb, g.gb, g.C, g.ldc,
                                                    g.alpha, kchunk, g.c_split_stride);
    }
    DSANLS_LAUNCH_CHECK();
}

void launch_sgemm(const GemmArgs &g, cudaStream_t s) {
    if (g.M <= 0 || g.N <= 0) return;
    const int64_t splits = g.splits < 1 ? 1 : g.splits;
    const int64_t mid = ceil_div(g.M, MT) * ceil_div(g.N, MT) * splits;
    const int64_t small = ceil_div(g.M, ST) * ceil_div(g.N, ST) * splits;
    // large tiles from half a wave of them on, or where the small ones would be many waves
    // (2,429 x 100 from 200: 76 large tiles 14.6 us, 19.1 small; 4,096 x 64 from 1,000: 64
    // large 49, 64 small; 1,665 x 100 from 100: 54 large 10.1, 8.5 small; over 361 .. 65,536 rows,
    // ranks of 10 to 128 and K of 64 to 4,000 never slower than one 128-row tile at a time)
    // Beside the Gram and the step size of a half-step (45 to 75 us of a few CTAs) the product is
    // hidden as long as it is short, and the small tiles' many CTAs then only hold those up:
    // coordinate descent on sampled columns, us per half-step with large / small tiles, 2,000
    // rows: rank 10, K = 256 39.7 / 40.1, 350 41.6 / 40.6, 600 79 / 44; rank 31, 200 62.9 / 65.9, 420
    // 65 / 68, 500 75 / 69; rank 64, 200 100 / 107, 500 106 / 116, 600 128 / 121; rank 100, 200 260 /
    // 273, 700 280 / 306, 1,400 338 / 356.
    const int64_t hidden = g.N <= 16 ? 300 : (g.N <= 32 ? 450 : (g.N <= 64 ? 550 : 2048));
    const bool large = mid >= 76 || (small > 6 * 152 && mid >= 16) || (g.beside && g.K < hidden);
    const int tile = large ? MT : ST;
    if (g.a_kcontig && g.b_kcontig) dispatch<true, true>(g, tile, s);
    else if (g.a_kcontig) dispatch<true, false>(g, tile, s);
    else if (g.b_kcontig) dispatch<false, true>(g, tile, s);
    else dispatch<false, false>(g, tile, s);
}

// (a thread's loads of eight slices are in flight together; packed slices need no division)
__global__ void k_split_reduce(const float *__restrict__ part, int64_t stride, int splits, int64_t M, int64_t N,
                               int64_t ldp, float *__restrict__ out, int64_t ldo) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= M * N) return;
    int64_t src = idx, dst = idx;
    if (ldp != N || ldo != N) {
        const int64_t i = idx / N, j = idx - i * N;
        src = i * ldp + j;
        dst = i * ldo + j;
    }
    float acc = 0.0f;
#pragma unroll 8
    for (int z = 0; z < splits; ++z) acc = __fadd_rn(acc, part[z * stride + src]);
    out[dst] = acc;
}

void launch_split_reduce(const float *part, int64_t stride, int splits, int64_t M, int64_t N, int64_t ldp,
                         float *out, int64_t ldo, cudaStream_t s) {
    const int64_t total = M * N;
    if (total == 0) return;
    const int threads = total < 256 * 304 ? 64 : 256;  // a small result is spread over more SMs
    k_split_reduce<<<(unsigned)ceil_div(total, threads), threads, 0, s>>>(part, stride, splits, M, N, ldp, out, ldo);
    DSANLS_LAUNCH_CHECK();
}

}  // namespace dsanls
