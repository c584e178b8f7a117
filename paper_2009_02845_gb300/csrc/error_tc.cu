// Squared residual ||M - U V^T||_F^2 of dense M (Section 5.1) with the inner products on
// tensor cores.
//
// The CUDA-core form (error.cu) is bound by the FP64 pipe (two operations per clock and
// SM): a conversion, a subtraction and an FMA per entry of M are 11.6 ms for 65,536 x
// 16,384 where reading M takes 0.64.  Here the inner products come from three bf16 parts of
// each row of U and of V on the row's own fixed grid (error-free slicing, Ozaki, Ogita,
// Oishi, Rump 2012): multiples of 2^-8, 2^-17 and 2^-26 of a power of two above the row's
// largest entry, at most 256 of them each (exact in bf16), so a product of parts is an
// integer of at most 2^16 in its unit and the sums of k <= 128 of them, D0 = hh and
// D1 = hm + mh, are exact in the fp32 accumulator (D2 = hl + mm + lh to its last bit) -- the
// tensor cores' rounding toward zero, a bias of 1e-7 of the result with the plain split,
// has nothing to round.  They are added rounding to nearest; the parts' remainders are
// 2^-27 of the largest entry, of either sign.  The residual is a binary32 subtraction (its error is relative to the
// residual), and its square is summed in pairs of binary32 (two-product and two-sum, Dekker
// 1971 and Knuth: 2^-48 of the sum), which a thread turns into FP64 once.
//
// Persistent CTAs take contiguous ranges of 128 x 64 tiles in row order.  Warps by role:
//   epilogue (16)  a thread owns a row and 16 columns: residual of the tile of M in shared
//                  memory (TMA, 32-column boxes, 128-byte swizzle: no bank conflicts)
//                  against the accumulators;
//   mma            one thread: per K step A_h x [B_h | B_m | B_l], A_m x [B_h | B_m],
//                  A_l x B_h into one of two sets of accumulators;
//   tma M          the tile of M, a ring of 32-column chunks;
//   tma U, V       U's parts when the row tile changes, V's parts of every tile (from L2).
// What bounds it: HBM needs 1,515 cycles per tile, the products 832 (k <= 64), the
// epilogue's issue slots about 1,300.  Measured, with the parts and the final sum, 65,536 x
// 16,384 with k = 64: 1.24 ms (11.6 in FP64) = 3.5 TB/s; the result's distance from FP64
// arithmetic 5e-14 to 3e-9 relative over random and fitted factors of five shapes, where
// the FP64 form with binary32 chains had 2e-13 to 6e-10.
#include <cuda.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "tc_gemm.cuh"
#include "tc_ptx.cuh"

namespace dsanls {

namespace {

constexpr int RT_BM = 128, RT_BN = 64, RT_CHUNK = 32;
constexpr int RT_EW = 16;                            // epilogue warps
constexpr int RT_THREADS = 32 * (RT_EW + 3);
constexpr int RT_CHUNK_BYTES = RT_BM * RT_CHUNK * 4;
constexpr int RT_DSET = 3 * RT_BN;
constexpr int RT_MAX_M = 6, RT_BST = 2;
constexpr unsigned long long RT_WAIT_NS = 2000000000ull;

struct __align__(16) RtTail {
    uint64_t mfull[RT_MAX_M], mempty[RT_MAX_M];
    uint64_t bfull[RT_BST], bempty[RT_BST];
    uint64_t afull, aempty;
    uint64_t dfull[2], dempty[2];
    uint64_t fin;
    double red[RT_EW];
    uint32_t tmem_base;
    int abort;
};

// KB: K blocks of 64 (1 for k <= 64, 2 above)
template <int KB>
struct RtCfg {
    static constexpr int ABYTES = KB * 3 * RT_BM * 128;   // U's parts of a row tile
    static constexpr int BBYTES = KB * 3 * RT_BN * 128;   // V's parts of a tile
    static constexpr int MST = KB == 1 ? 6 : 2;           // chunks of M in the ring
    static constexpr size_t SMEM = 1024 + ABYTES + RT_BST * BBYTES + MST * RT_CHUNK_BYTES + sizeof(RtTail);
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

DSANLS_DEV bool rt_wait(uint64_t *bar, uint32_t parity, volatile int *abort) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = globaltimer_ns();
    while (!mbar_try_wait(bar, parity)) {
        if (*abort) return false;
        if (globaltimer_ns() - t0 > RT_WAIT_NS) {
            *abort = 1;
            return false;
        }
    }
    return true;
}

// power of two near 1 / rms(M): the squares then neither overflow nor vanish against M's
__host__ __device__ inline int rt_exponent(double mm, double count) {
    int e = 0;
    const double rms = sqrt(mm / count);
    if (rms > 0.0 && rms < 1e300) frexp(rms, &e);
    return e < -120 ? -120 : (e > 120 ? 120 : e);
}

template <int KB>
__global__ void __launch_bounds__(RT_THREADS, 1)
    k_residual_tc(const __grid_constant__ CUtensorMap map_m, const __grid_constant__ CUtensorMap map_u,
                  const __grid_constant__ CUtensorMap map_v, int64_t m, int64_t n, int k, int64_t urows, int64_t vrows,
                  const double *__restrict__ mm, double *__restrict__ part, int *__restrict__ err) {
    using Cfg = RtCfg<KB>;
    constexpr int MST = Cfg::MST, APART = RT_BM * 128, BPART = RT_BN * 128;
    extern __shared__ __align__(1024) uint8_t rt_raw[];
    uint8_t *base = rt_raw + ((1024u - (smem_u32(rt_raw) & 1023u)) & 1023u);
    uint8_t *ap = base, *bp = ap + Cfg::ABYTES, *mp = bp + RT_BST * Cfg::BBYTES;
    RtTail *tail = reinterpret_cast<RtTail *>(mp + MST * RT_CHUNK_BYTES);
    volatile int *abort = &tail->abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int i = 0; i < MST; ++i) {
            mbar_init(&tail->mfull[i], 1);
            mbar_init(&tail->mempty[i], RT_EW / 2);
        }
        for (int i = 0; i < RT_BST; ++i) {
            mbar_init(&tail->bfull[i], 1);
            mbar_init(&tail->bempty[i], 1);
        }
        mbar_init(&tail->afull, 1);
        mbar_init(&tail->aempty, 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(&tail->dfull[i], 1);
            mbar_init(&tail->dempty[i], RT_EW);
        }
        mbar_init(&tail->fin, 1);
        tail->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == RT_EW) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tail->tmem_base)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = tail->tmem_base;
    const int64_t ntn = ceil_div(n, (int64_t)RT_BN), tiles = ceil_div(m, (int64_t)RT_BM) * ntn;
    const int64_t t0 = tiles * blockIdx.x / gridDim.x, t1 = tiles * (blockIdx.x + 1) / gridDim.x;
    const int nt = (int)(t1 - t0);
    float hi = 0.0f, lo = 0.0f;  // epilogue: the thread's sum
    if (warp < RT_EW) {
        const int q = warp & 3, cg = warp >> 2, r = 32 * q + lane;  // columns 16 cg .. of the tile
        const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16) + 16 * cg;
        const float scale = __int_as_float((127 - rt_exponent(*mm, (double)m * (double)n)) << 23);
        for (int i = 0; i < nt; ++i) {
            const int c = 2 * i + (cg >> 1), slot = c % MST, buf = i & 1;
            const bool ok = rt_wait(&tail->mfull[slot], (c / MST) & 1, abort) &&
                            rt_wait(&tail->dfull[buf], (i >> 1) & 1, abort);
            if (!__all_sync(0xffffffffu, ok)) break;
            fence_after();
            uint32_t d[16];
            float x[16];
            tmem_ld16(tl + buf * RT_DSET + RT_BN, d);
            {
                uint32_t d2[16];
                tmem_ld16(tl + buf * RT_DSET + 2 * RT_BN, d2);
                tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 16; ++e) x[e] = __fadd_rn(__uint_as_float(d[e]), __uint_as_float(d2[e]));
            }
            tmem_ld16(tl + buf * RT_DSET, d);
            const float4 *row = reinterpret_cast<const float4 *>(mp + slot * RT_CHUNK_BYTES) + r * (RT_CHUNK / 4);
            float4 v[4];
#pragma unroll
            for (int p = 0; p < 4; ++p) v[p] = row[(4 * (cg & 1) + p) ^ (r & 7)];
            tmem_ld_wait();
            fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&tail->dempty[buf]);
                mbar_arrive(&tail->mempty[slot]);
            }
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const float4 w = v[e >> 2];
                const float me = (e & 3) == 0 ? w.x : ((e & 3) == 1 ? w.y : ((e & 3) == 2 ? w.z : w.w));
                const float uv = __fadd_rn(__uint_as_float(d[e]), x[e]);
                const float res = __fmul_rn(__fsub_rn(me, uv), scale);
                const float p = __fmul_rn(res, res), pe = __fmaf_rn(res, res, -p);
                // (hi, lo) += p + pe: columns past n and rows past m have a residual of zero
                const float s = __fadd_rn(hi, p), t = __fsub_rn(s, hi);
                const float se = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, t)), __fsub_rn(p, t));
                hi = s;
                lo = __fadd_rn(lo, __fadd_rn(se, pe));
            }
        }
    } else if (warp == RT_EW) {
        if (lane == 0) {
            // ---- mma ----
            const uint32_t id1 = idesc_bf16(RT_BM, RT_BN), id2 = idesc_bf16(RT_BM, 2 * RT_BN),
                           id3 = idesc_bf16(RT_BM, 3 * RT_BN);
            int64_t rt = -1;
            int na = 0;  // row tiles so far
            const int steps = (k + 15) / 16;
            for (int i = 0; i < nt; ++i) {
                const int64_t row = (t0 + i) / ntn;
                const int sb = i % RT_BST, buf = i & 1;
                if (row != rt) {
                    if (na > 0) mma_commit(&tail->aempty);
                    if (!rt_wait(&tail->afull, na & 1, abort)) break;
                    rt = row;
                    ++na;
                }
                if (i >= 2 && !rt_wait(&tail->dempty[buf], ((i >> 1) - 1) & 1, abort)) break;
                if (!rt_wait(&tail->bfull[sb], (i / RT_BST) & 1, abort)) break;
                fence_after();
                const uint32_t d = tmem + buf * RT_DSET;
                for (int ks = 0; ks < steps; ++ks) {
                    const uint32_t o = (ks & 3) * 32;
                    const uint32_t ah = smem_u32(ap) + (ks >> 2) * 3 * APART + o, am = ah + APART, al = am + APART;
                    const uint64_t bh = sw128_desc(smem_u32(bp) + sb * Cfg::BBYTES + (ks >> 2) * 3 * BPART + o);
                    mma_bf16(d, sw128_desc(ah), bh, id3, ks > 0);
                    mma_bf16(d + RT_BN, sw128_desc(am), bh, id2, 1);
                    mma_bf16(d + 2 * RT_BN, sw128_desc(al), bh, id1, 1);
                }
                mma_commit(&tail->bempty[sb]);
                mma_commit(&tail->dfull[buf]);
            }
            // every product this thread issued has retired before the tensor memory is freed
            mma_commit(&tail->fin);
            mbar_wait(&tail->fin, 0, RT_WAIT_NS);
        }
    } else if (warp == RT_EW + 1) {
        if (lane == 0) {
            // ---- tma M ----
            int issued = 0;
            for (int c = 0; c < 2 * nt; ++c) {
                const int slot = c % MST;
                if (c >= MST && !rt_wait(&tail->mempty[slot], ((c / MST) - 1) & 1, abort)) break;
                const int64_t t = t0 + (c >> 1);
                mbar_expect_tx(&tail->mfull[slot], RT_CHUNK_BYTES);
                tma_load_2d(mp + slot * RT_CHUNK_BYTES, &map_m, (int)((t % ntn) * RT_BN + (c & 1) * RT_CHUNK),
                            (int)((t / ntn) * RT_BM), &tail->mfull[slot]);
                issued = c + 1;
            }
            if (*abort)  // nobody may be waiting for the last copies any more
                for (int c = max(0, issued - MST); c < issued; ++c)
                    mbar_wait(&tail->mfull[c % MST], (c / MST) & 1, RT_WAIT_NS);
        }
    } else if (lane == 0) {
        // ---- tma U, V (parts p of K block kb: rows p urows + i, columns 64 kb ..) ----
        int64_t rt = -1;
        int na = 0, issued = 0;
        for (int i = 0; i < nt; ++i) {
            const int64_t row = (t0 + i) / ntn;
            const int sb = i % RT_BST;
            if (row != rt) {
                if (na > 0 && !rt_wait(&tail->aempty, (na - 1) & 1, abort)) break;
                mbar_expect_tx(&tail->afull, Cfg::ABYTES);
                for (int x = 0; x < 3 * KB; ++x)
                    tma_load_2d(ap + x * APART, &map_u, (x / 3) * 64, (int)((x % 3) * urows + row * RT_BM), &tail->afull);
                rt = row;
                ++na;
            }
            if (i >= RT_BST && !rt_wait(&tail->bempty[sb], ((i / RT_BST) - 1) & 1, abort)) break;
            mbar_expect_tx(&tail->bfull[sb], Cfg::BBYTES);
            for (int x = 0; x < 3 * KB; ++x)
                tma_load_2d(bp + sb * Cfg::BBYTES + x * BPART, &map_v, (x / 3) * 64,
                            (int)((x % 3) * vrows + ((t0 + i) % ntn) * RT_BN), &tail->bfull[sb]);
            issued = i + 1;
        }
        if (*abort) {
            if (na > 0) mbar_wait(&tail->afull, (na - 1) & 1, RT_WAIT_NS);
            for (int i = max(0, issued - RT_BST); i < issued; ++i)
                mbar_wait(&tail->bfull[i % RT_BST], (i / RT_BST) & 1, RT_WAIT_NS);
        }
    }
    double v = (double)hi + (double)lo;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (warp < RT_EW && lane == 0) tail->red[warp] = v;
    fence_before();
    __syncthreads();
    fence_after();
    if (tid == 0) {
        double tot = 0.0;
        for (int i = 0; i < RT_EW; ++i) tot += tail->red[i];
        part[blockIdx.x] = ldexp(tot, 2 * rt_exponent(*mm, (double)m * (double)n));
        if (tail->abort) atomicOr(err, 2);
    }
    if (warp == RT_EW)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

// The three parts of the rows of X (rows x k) on each row's grid, out[p][row][ldk], prows
// rows per part (zero past the last); one warp per row.  A row whose largest entry is not in
// [2^-90, 2^100], or not finite, becomes NaN: the caller's result is then not finite.
__global__ void __launch_bounds__(256) k_parts_grid(const float *__restrict__ X, int64_t rows, int k, int64_t ldk,
                                                    int64_t prows, __nv_bfloat16 *__restrict__ out) {
    const int lane = threadIdx.x & 31;
    for (int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); r < prows; r += (int64_t)gridDim.x * 8) {
        float z[4], mx = 0.0f;
        bool finite = true;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = lane + 32 * u;
            z[u] = r < rows && c < k ? X[r * k + c] : 0.0f;
            finite = finite && fabsf(z[u]) <= 3.402823466e38f;
            mx = fmaxf(mx, fabsf(z[u]));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const bool bad = !__all_sync(0xffffffffu, finite) || (mx > 0.0f && (mx < 0x1p-90f || mx > 0x1p100f));
        // e: 2^e above every entry; rounding to a multiple of q by adding and subtracting 1.5 2^23 q
        const int e = mx > 0.0f && !bad ? (int)((__float_as_uint(mx) >> 23) & 255) - 126 : 0;
        const float c1 = __int_as_float((127 + e + 15) << 23) * 1.5f, c2 = c1 * 0x1p-9f, c3 = c1 * 0x1p-18f;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = lane + 32 * u;
            if (c >= k) break;
            const float h = __fsub_rn(__fadd_rn(z[u], c1), c1), r1 = __fsub_rn(z[u], h);
            const float m = __fsub_rn(__fadd_rn(r1, c2), c2), r2 = __fsub_rn(r1, m);
            const float l = __fsub_rn(__fadd_rn(r2, c3), c3);
            const float nan = __int_as_float(0x7fc00000);
            __nv_bfloat16 *o = out + r * ldk + c;
            o[0] = __float2bfloat16_rn(bad ? nan : h);
            o[prows * ldk] = __float2bfloat16_rn(bad ? nan : m);
            o[2 * prows * ldk] = __float2bfloat16_rn(bad ? nan : l);
        }
    }
}

void launch_parts_grid(const float *X, int64_t rows, int k, int64_t ldk, int64_t prows, __nv_bfloat16 *out,
                       cudaStream_t s) {
    k_parts_grid<<<(unsigned)std::min<int64_t>(ceil_div(prows, 8), 152 * 16), 256, 0, s>>>(X, rows, k, ldk, prows, out);
    DSANLS_LAUNCH_CHECK();
}

int64_t pad_rows(int64_t r, int64_t t) { return ceil_div(r, t) * t; }

template <int KB>
void residual_launch(const CUtensorMap &mm_map, const CUtensorMap &mu, const CUtensorMap &mv, int64_t m, int64_t n, int k,
                     const double *mm, double *work, int grid, int *err, cudaStream_t s) {
    k_residual_tc<KB><<<grid, RT_THREADS, RtCfg<KB>::SMEM, s>>>(mm_map, mu, mv, m, n, k, pad_rows(m, RT_BM),
                                                                pad_rows(n, RT_BN), mm, work, err);
    DSANLS_LAUNCH_CHECK();
}

}  // namespace

bool residual_tc_supported(int64_t ld, int64_t m, int64_t n, int k) {
    // whole 16-byte rows for TMA; rows and columns in a tensor map's coordinates
    return ld % 4 == 0 && k >= 1 && k <= 128 && 3 * pad_rows(m, RT_BM) < (1ll << 31) && 3 * pad_rows(n, RT_BN) < (1ll << 31);
}

int64_t residual_tc_parts(int64_t m, int64_t n, int k) {
    return 3 * (pad_rows(m, RT_BM) + pad_rows(n, RT_BN)) * split_parts_ld(k);
}

void launch_dense_residual_tc(const float *M, int64_t ld, const float *U, const float *V, int64_t m, int64_t n, int k,
                              const double *mm, __nv_bfloat16 *parts, double *work, int64_t work_elems, double *out,
                              int *err, cudaStream_t s) {
    if (!residual_tc_supported(ld, m, n, k)) throw ArgError{"residual on tensor cores: unsupported size"};
    const int64_t ldk = split_parts_ld(k), ur = pad_rows(m, RT_BM), vr = pad_rows(n, RT_BN);
    __nv_bfloat16 *up = parts, *vp = parts + 3 * ur * ldk;
    launch_parts_grid(U, m, k, ldk, ur, up, s);
    launch_parts_grid(V, n, k, ldk, vr, vp, s);
    CUtensorMap mm_map, mu, mv;
    encode_f32_map(&mm_map, M, m, n, ld, RT_CHUNK, RT_BM, true);
    encode_bf16_map_ld(&mu, up, 3 * ur, k, ldk, RT_BM);
    encode_bf16_map_ld(&mv, vp, 3 * vr, k, ldk, RT_BN);
    const int64_t tiles = ceil_div(m, RT_BM) * ceil_div(n, RT_BN);
    const int grid = (int)std::min<int64_t>({tiles, 152, work_elems});  // one CTA per SM (tensor memory)
    if (k <= 64)
        residual_launch<1>(mm_map, mu, mv, m, n, k, mm, work, grid, err, s);
    else
        residual_launch<2>(mm_map, mu, mv, m, n, k, mm, work, grid, err, s);
    launch_sum_parts(work, grid, out, s);
}

void prime_residual_attributes(int max_smem) {
    allow_max_dynamic_smem(k_residual_tc<1>, max_smem);
    allow_max_dynamic_smem(k_residual_tc<2>, max_smem);
}

}  // namespace dsanls
