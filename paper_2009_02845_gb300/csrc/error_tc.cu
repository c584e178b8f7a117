// Squared residual ||M - U V^T||_F^2 of dense M (Section 5.1) with the inner products on
// tensor cores.
//
// The CUDA-core form (error.cu) is bound by the FP64 pipe (two operations per clock and
// SM): a conversion, a subtraction and an FMA per entry of M are 11.6 ms for 65,536 x
// 16,384 where reading M takes 0.64.  Here the inner products come from four bf16 parts of
// each row of U and of V on the row's own fixed grid (error-free slicing, Ozaki, Ogita,
// Oishi, Rump 2012): multiples of 2^-8, 2^-17, 2^-26 and 2^-35 of a power of two above the
// row's largest entry, at most 256 of them each (exact in bf16), so a product of parts is an
// integer of at most 2^16 in its unit and the sums of k <= 128 of them, D0 = hh and
// D1 = hm + mh, are exact in the fp32 accumulator (D2 = hl + mm + lh and D3 = hq + ml + lm +
// qh to their last bits) -- the tensor cores' rounding toward zero, a bias of 1e-7 of the
// result with the plain split, has nothing to round.  The residual is ((M - D0) - D1) - (D2 +
// D3) in binary32: M - D0 is exact where the product fits M, and what it rounds otherwise is
// relative to a difference.  Its square is summed in pairs of binary32 (two-product and
// two-sum, Dekker 1971 and Knuth: 2^-48 of the sum), which a thread adds to FP64 every
// RT_CARRY tiles.
//
// What the slicing drops is absolute: each of the at most min(nz_i, nz_j) products of nonzeros
// of rows i of U and j of V loses up to 5.1 2^-36 2^(e_i + e_j), 2^e above a row's largest entry
// (the remainders, 2^-36 of that against an entry of the other row, and the products of parts
// beyond D3).  That is nothing beside the residual as long as a large entry of one row does not
// meet the dropped tail of the other (columns of U and V of opposite scales, a component dead
// in one factor and large in the other).  So k_parts_grid also sums nz_i 4^e_i over the rows, and
//     E^2 = 26 2^-72 (sum over U) (sum over V) + m n (k 2^-125)^2
// (the last term for products that underflow) bounds the sum of the squares of what is dropped:
// the caller takes the result only if E^2 is at most 1e-12 of it or 2^-58 ||M||^2
// (residual_tc_holds).  Whatever the signs, ||M - U V^T||_F is then within 1e-6 of itself or, for
// factors that fit M closely, within 2^-29 ||M||, an eighth of what rounding each product
// to binary32 once would move.  Otherwise the columns are
// balanced first -- column c of U times a power of two and column c of V by its inverse, from
// the largest entry of both; exact, and the product is the same -- and if that does not meet
// the bound either, the FP64 form answers.  Over random, planted and fitted factors of seven
// shapes (the last ones within 1e-4 of M) the result is 1e-13 to 1.6e-10 of itself away from
// FP64 arithmetic, where the binary32 chains of error.cu are 4e-13 to 9e-7 away.  Three parts
// and a bound were not enough: the tails dropped at 2^-27 are the same along a whole row of M
// and average out less than a chain's roundings (1.2e-9 where the chains have 4e-10).
//
// Persistent CTAs take contiguous ranges of 128 x 64 tiles in row order.  Warps by role:
//   epilogue (16)  a thread owns a row and 16 columns: residual of the tile of M in shared
//                  memory (TMA, 32-column boxes, 128-byte swizzle: no bank conflicts)
//                  against the accumulators;
//   mma            one thread: per K step A_h x [B_h | B_m | B_l | B_q], A_m x [B_h | B_m |
//                  B_l], A_l x [B_h | B_m], A_q x B_h into one of two sets of accumulators
//                  (all of tensor memory);
//   tma M          the tile of M, a ring of 32-column chunks;
//   tma U, V       U's parts when the row tile changes, V's parts of every tile and K block of
//                  64 (from L2).
// What bounds it: HBM needs 1,515 cycles per tile, the products 1,280 (k <= 64), the
// epilogue's issue slots about 1,400.  Measured, with the parts and the final sum, 65,536 x
// 16,384 with k = 64: 1.17 ms (11.6 in FP64) = 3.7 TB/s, about twice that where the columns are
// balanced in a second pass; k = 100, whose products take 2,560 cycles a tile, 1.81.  The
// epilogue's arithmetic and the latency of its loads bound it: it runs two columns to an
// instruction (1.46 ms with one), reads M before it waits for the products and its
// accumulators with one wait (1.35 otherwise).
#include <cuda.h>

#include <algorithm>
#include <cmath>

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
constexpr int RT_PARTS = 4;
constexpr int RT_DSET = RT_PARTS * RT_BN;
constexpr int RT_MAX_M = 6, RT_BST = 2;
constexpr int RT_BSTAGE = RT_PARTS * RT_BN * 128;    // V's parts of a tile and K block
constexpr int RT_CARRY = 16;                         // tiles between carries into FP64
constexpr int64_t RT_GRID_SUMS = 512;                // doubles of `work` before k_parts_grid's sums

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
    static constexpr int ABYTES = KB * RT_PARTS * RT_BM * 128;  // U's parts of a row tile
    static constexpr int MST = KB == 1 ? 6 : 2;           // chunks of M in the ring
    static constexpr size_t SMEM = 1024 + ABYTES + RT_BST * RT_BSTAGE + MST * RT_CHUNK_BYTES + sizeof(RtTail);
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

// Two binary32 operations, rounded to nearest, in one instruction.
DSANLS_DEV uint64_t rt_pair(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
DSANLS_DEV uint64_t rt_pair(uint32_t a, uint32_t b) { return rt_pair(__uint_as_float(a), __uint_as_float(b)); }
DSANLS_DEV uint64_t rt_add(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
DSANLS_DEV uint64_t rt_sub(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
DSANLS_DEV uint64_t rt_mul(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
DSANLS_DEV uint64_t rt_fma(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
DSANLS_DEV double rt_total(uint64_t hi, uint64_t lo) {
    float h0, h1, l0, l1;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(h0), "=f"(h1) : "l"(hi));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(l0), "=f"(l1) : "l"(lo));
    return ((double)h0 + (double)l0) + ((double)h1 + (double)l1);
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
                  const double *__restrict__ mm, double *__restrict__ part, int *__restrict__ err, WaitSwitch wait) {
    using Cfg = RtCfg<KB>;
    constexpr int MST = Cfg::MST, APART = RT_BM * 128, BPART = RT_BN * 128;
    extern __shared__ __align__(1024) uint8_t rt_raw[];
    uint8_t *base = rt_raw + ((1024u - (smem_u32(rt_raw) & 1023u)) & 1023u);
    uint8_t *ap = base, *bp = ap + Cfg::ABYTES, *mp = bp + RT_BST * RT_BSTAGE;
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
    uint64_t hi = 0, lo = 0;  // epilogue: the thread's sums (even and odd columns) since the last carry
    double sum = 0.0;
    if (warp < RT_EW) {
        const int q = warp & 3, cg = warp >> 2, r = 32 * q + lane;  // columns 16 cg .. of the tile
        const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16) + 16 * cg;
        const float sc = __int_as_float((127 - rt_exponent(*mm, (double)m * (double)n)) << 23);
        const uint64_t scale = rt_pair(sc, sc);
        // (a loop of its own for the carry: under a condition in this one its FP64 conversions and
        // additions run for every tile, 2,000 cycles of the FP64 pipe: 1.21 ms, k = 31 17 % more)
        bool ok = true;
        for (int i0 = 0; ok && i0 < nt; i0 += RT_CARRY) {
            const int i1 = min(nt, i0 + RT_CARRY);
            for (int i = i0; i < i1; ++i) {
                const int c = 2 * i + (cg >> 1), slot = c % MST, buf = i & 1;
                ok = role_wait(&tail->mfull[slot], (c / MST) & 1, abort, wait.ns);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                const float4 *row = reinterpret_cast<const float4 *>(mp + slot * RT_CHUNK_BYTES) + r * (RT_CHUNK / 4);
                float4 v[4];
#pragma unroll
                for (int p = 0; p < 4; ++p) v[p] = row[(4 * (cg & 1) + p) ^ (r & 7)];
                __syncwarp();  // (the next copy runs under these products: with a ring of one tile, k = 100,
                if (lane == 0) mbar_arrive(&tail->mempty[slot]);  // 2.44 ms when released below, 1.79 here)
                ok = role_wait(&tail->dfull[buf], (i >> 1) & 1, abort, wait.ns);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                fence_after();
                uint32_t d[16], d1[16], d2[16], d3[16];
                uint64_t x[8];
                tmem_ld16(tl + buf * RT_DSET, d);
                tmem_ld16(tl + buf * RT_DSET + RT_BN, d1);
                tmem_ld16(tl + buf * RT_DSET + 2 * RT_BN, d2);
                tmem_ld16(tl + buf * RT_DSET + 3 * RT_BN, d3);
                tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    x[e] = rt_add(rt_pair(d2[2 * e], d2[2 * e + 1]), rt_pair(d3[2 * e], d3[2 * e + 1]));
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&tail->dempty[buf]);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float4 w = v[e >> 1];
                    const uint64_t me = (e & 1) ? rt_pair(w.z, w.w) : rt_pair(w.x, w.y);
                    const uint64_t r1 = rt_sub(rt_sub(me, rt_pair(d[2 * e], d[2 * e + 1])), rt_pair(d1[2 * e], d1[2 * e + 1]));
                    const uint64_t res = rt_mul(rt_sub(r1, x[e]), scale);
                    const uint64_t p = rt_mul(res, res), pe = rt_fma(res, res, p ^ 0x8000000080000000ull);
                    // (hi, lo) += p + pe: columns past n and rows past m have a residual of zero
                    const uint64_t s = rt_add(hi, p), t = rt_sub(s, hi);
                    const uint64_t se = rt_add(rt_sub(hi, rt_sub(s, t)), rt_sub(p, t));
                    hi = s;
                    lo = rt_add(lo, rt_add(se, pe));
                }
            }
            sum += rt_total(hi, lo);
            hi = lo = 0;
        }
    } else if (warp == RT_EW) {
        if (lane == 0) {
            // ---- mma ----
            uint32_t id[RT_PARTS];  // N = 1 .. 4 parts of V
            for (int p = 0; p < RT_PARTS; ++p) id[p] = idesc_bf16(RT_BM, (p + 1) * RT_BN);
            int64_t rt = -1;
            int na = 0;  // row tiles so far
            const int steps = (k + 15) / 16;
            for (int i = 0; i < nt; ++i) {
                const int64_t row = (t0 + i) / ntn;
                const int buf = i & 1;
                if (row != rt) {
                    if (na > 0) mma_commit(&tail->aempty);
                    if (!role_wait(&tail->afull, na & 1, abort, wait.ns)) break;
                    rt = row;
                    ++na;
                }
                if (i >= 2 && !role_wait(&tail->dempty[buf], ((i >> 1) - 1) & 1, abort, wait.ns)) break;
                const uint32_t d = tmem + buf * RT_DSET;
                bool ok = true;
                for (int kb = 0; kb < KB; ++kb) {
                    const int b = i * KB + kb, sb = b % RT_BST;
                    ok = role_wait(&tail->bfull[sb], (b / RT_BST) & 1, abort, wait.ns);
                    if (!ok) break;
                    fence_after();
                    const int nks = min(4, steps - 4 * kb);
                    for (int ks = 0; ks < nks; ++ks) {
                        const uint32_t a = smem_u32(ap) + kb * RT_PARTS * APART + ks * 32;
                        const uint64_t bh = sw128_desc(smem_u32(bp) + sb * RT_BSTAGE + ks * 32);
                        // part p of U times the parts 0 .. 3 - p of V, into D_p .. D_3
#pragma unroll
                        for (int p = 0; p < RT_PARTS; ++p)
                            mma_bf16(d + p * RT_BN, sw128_desc(a + p * APART), bh, id[RT_PARTS - 1 - p],
                                     p > 0 || kb > 0 || ks > 0);
                    }
                    mma_commit(&tail->bempty[sb]);
                }
                if (!ok) break;
                mma_commit(&tail->dfull[buf]);
            }
            // every product this thread issued has retired before the tensor memory is freed
            mma_commit(&tail->fin);
            mbar_wait(&tail->fin, 0, wait.ns);
        }
    } else if (warp == RT_EW + 1) {
        if (lane == 0 && !wait.starve) {
            // ---- tma M ----
            int issued = 0;
            for (int c = 0; c < 2 * nt; ++c) {
                const int slot = c % MST;
                if (c >= MST && !role_wait(&tail->mempty[slot], ((c / MST) - 1) & 1, abort, wait.ns)) break;
                const int64_t t = t0 + (c >> 1);
                mbar_expect_tx(&tail->mfull[slot], RT_CHUNK_BYTES);
                tma_load_2d(mp + slot * RT_CHUNK_BYTES, &map_m, (int)((t % ntn) * RT_BN + (c & 1) * RT_CHUNK),
                            (int)((t / ntn) * RT_BM), &tail->mfull[slot]);
                issued = c + 1;
            }
            if (*abort)  // nobody may be waiting for the last copies any more
                for (int c = max(0, issued - MST); c < issued; ++c)
                    mbar_wait(&tail->mfull[c % MST], (c / MST) & 1, wait.ns);
        }
    } else if (lane == 0) {
        // ---- tma U, V (part p of K block kb: rows p urows + i, columns 64 kb ..) ----
        int64_t rt = -1;
        int na = 0, issued = 0;
        bool ok = true;
        for (int i = 0; ok && i < nt; ++i) {
            const int64_t row = (t0 + i) / ntn;
            if (row != rt) {
                if (na > 0 && !role_wait(&tail->aempty, (na - 1) & 1, abort, wait.ns)) break;
                mbar_expect_tx(&tail->afull, Cfg::ABYTES);
                for (int x = 0; x < RT_PARTS * KB; ++x)
                    tma_load_2d(ap + x * APART, &map_u, (x / RT_PARTS) * 64,
                                (int)((x % RT_PARTS) * urows + row * RT_BM), &tail->afull);
                rt = row;
                ++na;
            }
            for (int kb = 0; kb < KB; ++kb) {
                const int b = i * KB + kb, sb = b % RT_BST;
                ok = b < RT_BST || role_wait(&tail->bempty[sb], ((b / RT_BST) - 1) & 1, abort, wait.ns);
                if (!ok) break;
                mbar_expect_tx(&tail->bfull[sb], RT_BSTAGE);
                for (int p = 0; p < RT_PARTS; ++p)
                    tma_load_2d(bp + sb * RT_BSTAGE + p * BPART, &map_v, kb * 64,
                                (int)(p * vrows + ((t0 + i) % ntn) * RT_BN), &tail->bfull[sb]);
                issued = b + 1;
            }
        }
        if (*abort) {
            if (na > 0) mbar_wait(&tail->afull, (na - 1) & 1, wait.ns);
            for (int b = max(0, issued - RT_BST); b < issued; ++b)
                mbar_wait(&tail->bfull[b % RT_BST], (b / RT_BST) & 1, wait.ns);
        }
    }
    double v = sum;
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

// Scratch ahead of the parts: the largest entry (bits) of every column of U, then of V.
constexpr int64_t RT_COLS = 128;
constexpr int64_t RT_COL_BYTES = 2 * RT_COLS * sizeof(uint32_t);

// Largest |entry| of every column of U (blockIdx.y = 0) and V (1), into the zeroed cmax.
__global__ void __launch_bounds__(256) k_column_max(const float *__restrict__ U, const float *__restrict__ V, int64_t m,
                                                    int64_t n, int k, uint32_t *__restrict__ cmax) {
    const float *X = blockIdx.y ? V : U;
    const int64_t rows = blockIdx.y ? n : m;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t mx[4] = {0, 0, 0, 0};
    for (int64_t r = (int64_t)blockIdx.x * 8 + warp; r < rows; r += (int64_t)gridDim.x * 8)
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (lane + 32 * u < k) mx[u] = max(mx[u], __float_as_uint(fabsf(X[r * k + lane + 32 * u])));
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (lane + 32 * u < k) atomicMax(&cmax[blockIdx.y * RT_COLS + lane + 32 * u], mx[u]);
}

// The four parts of the rows of U (blocks 0 .. ublocks-1) and V (the rest) on each row's grid,
// out[p][row][ldk], prows rows per part (zero past the last); one warp per row, the next row's
// entries on their way.  A row whose largest entry is not in [2^-90, 2^100], or not finite,
// becomes NaN: the result is then not finite.  Each block's sum of (nonzeros) 4^e goes to
// sums[b]; a warp keeps its own as acc 4^ref (in FP64 the row's few operations were two thirds
// of the kernel).  With cmax the columns are balanced first (a column that is zero in either
// factor is dropped).  NC: columns per lane, k <= 32 NC.
template <int NC>
__global__ void __launch_bounds__(256)
    k_parts_grid(const float *__restrict__ U, const float *__restrict__ V, int64_t m, int64_t n, int k, int64_t ldk,
                 int64_t ur, int64_t vr, __nv_bfloat16 *__restrict__ parts, int ublocks,
                 const uint32_t *__restrict__ cmax, double *__restrict__ sums) {
    __shared__ double red[8];
    const bool is_v = (int)blockIdx.x >= ublocks;
    const float *X = is_v ? V : U;
    const int64_t rows = is_v ? n : m, prows = is_v ? vr : ur;
    __nv_bfloat16 *out = parts + (is_v ? RT_PARTS * ur * ldk : 0);
    const int blk = (int)blockIdx.x - (is_v ? ublocks : 0), nblk = is_v ? (int)gridDim.x - ublocks : ublocks;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float f[NC], f2[NC];  // the column's factor in two steps
#pragma unroll
    for (int u = 0; u < NC; ++u) {
        const int c = lane + 32 * u;
        f[u] = f2[u] = 1.0f;
        if (!cmax || c >= k) continue;
        const uint32_t a = cmax[c], b = cmax[RT_COLS + c];
        const int t = ((int)(b >> 23) - (int)(a >> 23)) >> 1, e = is_v ? -t : t;  // |t| <= 127
        f[u] = a && b ? __int_as_float((127 + (e >> 1)) << 23) : 0.0f;
        f2[u] = __int_as_float((127 + e - (e >> 1)) << 23);
    }
    const int64_t step = (int64_t)nblk * 8;
    float acc = 0.0f, next[NC];
    int ref = -128;
    auto load = [&](int64_t r) {
#pragma unroll
        for (int u = 0; u < NC; ++u) next[u] = r < rows && lane + 32 * u < k ? X[r * k + lane + 32 * u] : 0.0f;
    };
    load((int64_t)blk * 8 + warp);
    for (int64_t r = (int64_t)blk * 8 + warp; r < prows; r += step) {
        float z[NC];
        unsigned bits = 0, nz = 0;
#pragma unroll
        for (int u = 0; u < NC; ++u) {
            z[u] = cmax ? __fmul_rn(__fmul_rn(next[u], f[u]), f2[u]) : next[u];
            bits = max(bits, __float_as_uint(z[u]) & 0x7fffffffu);  // (NaN above Inf above all numbers)
            nz += z[u] != 0.0f;
        }
        load(r + step);
        bits = __reduce_max_sync(0xffffffffu, bits);
        nz = __reduce_add_sync(0xffffffffu, nz);
        const float mx = __uint_as_float(bits);
        const bool bad = bits && !(mx >= 0x1p-90f && mx <= 0x1p100f);
        // e: 2^e above every entry; rounding to a multiple of q by adding and subtracting 1.5 2^23 q
        const int e = bits && !bad ? (int)(bits >> 23) - 126 : 0;
        if (bits) {
            if (e > ref) {
                acc = ref - e < -63 ? 0.0f : acc * __int_as_float((127 + 2 * (ref - e)) << 23);
                ref = e;
            }
            if (e - ref >= -63) acc += (float)nz * __int_as_float((127 + 2 * (e - ref)) << 23);
        }
        const float c1 = __int_as_float((127 + e + 15) << 23) * 1.5f;
#pragma unroll
        for (int u = 0; u < NC; ++u) {
            const int c = lane + 32 * u;
            if (c >= k) break;
            __nv_bfloat16 *o = out + r * ldk + c;
            float x = z[u], q = c1;
#pragma unroll
            for (int p = 0; p < RT_PARTS; ++p) {
                const float h = __fsub_rn(__fadd_rn(x, q), q);
                o[p * prows * ldk] = __float2bfloat16_rn(bad ? __int_as_float(0x7fc00000) : h);
                x = __fsub_rn(x, h);
                q *= 0x1p-9f;
            }
        }
    }
    if (lane == 0) red[warp] = ldexp((double)acc, 2 * ref);
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[w];
        sums[blockIdx.x] = t;
    }
}

// out[0] = the squared residual, out[1] = E^2 (the head of this file): three sums in fixed
// orders, eight warps each (one warp's shuffles for all three took 2 us more)
__global__ void __launch_bounds__(768)
    k_residual_sum(const double *__restrict__ part, int np, const double *__restrict__ sums, int ublocks, int vblocks,
                   double m, double n, double k, double *__restrict__ out) {
    __shared__ double red[24];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = warp >> 3;  // the residual, U's and V's nz 4^e
    const double *x = q == 0 ? part : (q == 1 ? sums : sums + ublocks);
    const int len = q == 0 ? np : (q == 1 ? ublocks : vblocks);
    double v = 0.0;
#pragma unroll 4
    for (int i = threadIdx.x & 255; i < len; i += 256) v += x[i];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (warp > 0) return;
    v = lane < 24 ? red[lane] : 0.0;
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);  // eight lanes to a sum
    const double u4 = __shfl_sync(0xffffffffu, v, 8), v4 = __shfl_sync(0xffffffffu, v, 16);
    if (lane == 0) {
        const double under = k * 0x1p-125;
        out[0] = v;
        out[1] = 26.0 * 0x1p-72 * u4 * v4 + m * n * under * under;
    }
}

int64_t pad_rows(int64_t r, int64_t t) { return ceil_div(r, t) * t; }

template <int KB>
void residual_launch(const CUtensorMap &mm_map, const CUtensorMap &mu, const CUtensorMap &mv, int64_t m, int64_t n, int k,
                     const double *mm, double *work, int grid, int *err, cudaStream_t s) {
    k_residual_tc<KB><<<grid, RT_THREADS, RtCfg<KB>::SMEM, s>>>(mm_map, mu, mv, m, n, k, pad_rows(m, RT_BM),
                                                                pad_rows(n, RT_BN), mm, work, err, wait_switch());
    DSANLS_LAUNCH_CHECK();
}

}  // namespace

bool residual_tc_supported(int64_t ld, int64_t m, int64_t n, int k) {
    // whole 16-byte rows for TMA; rows and columns in a tensor map's coordinates
    return ld % 4 == 0 && k >= 1 && k <= 128 && RT_PARTS * pad_rows(m, RT_BM) < (1ll << 31) &&
           RT_PARTS * pad_rows(n, RT_BN) < (1ll << 31);
}

int64_t residual_tc_parts(int64_t m, int64_t n, int k) {
    return RT_COL_BYTES / (int64_t)sizeof(__nv_bfloat16) +
           RT_PARTS * (pad_rows(m, RT_BM) + pad_rows(n, RT_BN)) * split_parts_ld(k);
}

bool residual_tc_holds(double mm, double residual, double dropped) {
    // (below 2^-90 of ||M||^2 the squares themselves would leave binary32's range)
    return std::isfinite(residual) && residual >= 0x1p-90 * mm && dropped <= std::max(1e-12 * residual, 0x1p-58 * mm);
}

void launch_dense_residual_tc(const float *M, int64_t ld, const float *U, const float *V, int64_t m, int64_t n, int k,
                              bool balance, const double *mm, __nv_bfloat16 *parts, double *work, int64_t work_elems,
                              double *out, int *err, cudaStream_t s) {
    if (!residual_tc_supported(ld, m, n, k)) throw ArgError{"residual on tensor cores: unsupported size"};
    const int64_t ldk = split_parts_ld(k), ur = pad_rows(m, RT_BM), vr = pad_rows(n, RT_BN);
    const int ublocks = (int)std::min<int64_t>(ceil_div(ur, 8), 152 * 8);
    const int vblocks = (int)std::min<int64_t>(ceil_div(vr, 8), 152 * 8);
    if (work_elems < RT_GRID_SUMS + ublocks + vblocks) throw ArgError{"residual: workspace too small"};
    uint32_t *cmax = reinterpret_cast<uint32_t *>(parts);
    __nv_bfloat16 *up = parts + RT_COL_BYTES / sizeof(__nv_bfloat16), *vp = up + RT_PARTS * ur * ldk;
    double *sums = work + RT_GRID_SUMS;
    if (balance) {
        DSANLS_CUDA(cudaMemsetAsync(cmax, 0, RT_COL_BYTES, s));
        k_column_max<<<dim3((unsigned)std::max(ublocks, vblocks), 2), 256, 0, s>>>(U, V, m, n, k, cmax);
        DSANLS_LAUNCH_CHECK();
    }
    const auto parts_kernel = k <= 32 ? k_parts_grid<1> : (k <= 64 ? k_parts_grid<2> : k_parts_grid<4>);
    parts_kernel<<<(unsigned)(ublocks + vblocks), 256, 0, s>>>(U, V, m, n, k, ldk, ur, vr, up, ublocks,
                                                               balance ? cmax : nullptr, sums);
    DSANLS_LAUNCH_CHECK();
    CUtensorMap mm_map, mu, mv;
    encode_f32_map(&mm_map, M, m, n, ld, RT_CHUNK, RT_BM, true);
    encode_bf16_map_ld(&mu, up, RT_PARTS * ur, k, ldk, RT_BM);
    encode_bf16_map_ld(&mv, vp, RT_PARTS * vr, k, ldk, RT_BN);
    const int64_t tiles = ceil_div(m, RT_BM) * ceil_div(n, RT_BN);
    const int grid = (int)std::min<int64_t>(tiles, 152);  // one CTA per SM (tensor memory)
    if (k <= 64)
        residual_launch<1>(mm_map, mu, mv, m, n, k, mm, work, grid, err, s);
    else
        residual_launch<2>(mm_map, mu, mv, m, n, k, mm, work, grid, err, s);
    k_residual_sum<<<1, 768, 0, s>>>(work, grid, sums, ublocks, vblocks, (double)m, (double)n, (double)k, out);
    DSANLS_LAUNCH_CHECK();
}

void prime_residual_attributes(int max_smem) {
    allow_max_dynamic_smem(k_residual_tc<1>, max_smem);
    allow_max_dynamic_smem(k_residual_tc<2>, max_smem);
}


}  // namespace dsanls
