// Fused row update on tensor cores: Z <- max(0, Z - eta (Z G - R)) (eq.
// gradient_descent, one projected-gradient step) for 32 < k <= 128.
//
// Z G is taken on tcgen05 from a three-way bf16 split of both operands, z = z_h + z_m +
// z_l (split3): the six products z_i g_j with i + j <= 2 accumulate in fp32 in tensor
// memory, and the dropped terms are of order 2^-24 |z| |g|, the rounding level of a
// binary32 product.  With bf16 factors z is a bf16 value (z_m = z_l = 0): three products,
// and the step's binary32 result is rounded to bf16 when it is stored.
//
// Sparse subsampled data (SPR): the right-hand side of a row of at most SubCsr::warp_rows()
// sub-CSR entries is formed here, r = alpha * sum over the row's entries (ascending) of
// val * Y[col][.], one fused multiply-add per entry and column -- the arithmetic of
// launch_subcsr_rows bit for bit -- so R is neither written nor read for it; longer rows
// come precomputed in R (launch_subcsr_long_rows).
//
// Persistent, one CTA per SM; the CTA splits G once into the three B operands in shared
// memory (N = k rounded up to 16 rows, K = k rounded up to 64, 128-byte swizzled K-major)
// and walks 128-row tiles of Z.  A tile is nr x k contiguous elements.  Its path crosses
// four roles that work on different tiles at the same time, joined by mbarriers:
//   copy   (1 warp)    bulk copies of the tile's 32-row pieces into a ring of NZ buffers (a
//                      piece whose bytes are not a multiple of 16 by plain loads);
//   split  (4 warps)   a thread reads a row of the tile and writes its parts to tensor
//                      memory, row i in lane i, as the MMAs' A operand;
//   mma    (1 warp)    the products of a tile into the accumulators of the tile's group;
//   step   (2 or 3 groups, 24 warps; tile j to group j mod NG)  a thread owns a row and
//                      every few 16-column chunks of it: forms or loads r (nothing of which
//                      waits for the products), then takes the step with the exact z of
//                      the piece and stores the row's chunk.
// The groups are there for the gather of r: its chain of loads (entry range, entries, rows
// of Y) is microseconds per tile whatever the bandwidth, and the next tiles' chains run
// beside it.  One 512-thread CTA that did the four in turn took 10.4 us per tile of k = 100.
// Now, per SM and tile of k = 100 in binary32, 7.5 us: the split 1.7 and the products 1.4 of
// it, one after the other on the one set of A parts; the rest of the step's 17,500 clk is
// the gather and the uncoalesced row accesses of its 24 warps.  HBM needs 2.3.
// 2e6 x 5e5, 1.4e6 sampled entries, k = 100, U / V half: binary32 1,069 / 310 us before,
// 770 / 176 now (floor 235 / 59); bf16 800 / 210 before, 486 / 111 now.
// Also tried: r gathered row by row by its own warps into shared memory, and the step in
// coalesced rows (1,155 us: three instructions for each of these; and any register spill
// there costs an L2 round trip each time, for the shared memory leaves almost no L1).
#include <algorithm>

#include "bounds.cuh"
#include "common.cuh"
#include "kernels.cuh"
#include "tc_gemm.cuh"
#include "tc_ptx.cuh"

namespace dsanls {

namespace {

constexpr int UPD_BM = 128;    // rows of a tile; a piece is 32 of them
constexpr int UPD_SPLIT = 4;   // warps of the split
constexpr int UPD_STEPS = 24;  // warps of all step groups
constexpr int UPD_MAX_NG = 3, UPD_MAX_NZ = 16;
constexpr int UPD_THREADS = 32 * (UPD_SPLIT + UPD_STEPS + 2);
// Step groups: as many as hold their tiles in shared memory with a piece or two to spare.
// Binary32 at k = 100 keeps 11 pieces: two groups of 12 warps 770 us against 839 for three
// of 8 (the third waits for its tile); bf16 keeps 16: three 486 us, two 533.
template <typename ZT>
__host__ __device__ constexpr int upd_groups() {
    return sizeof(ZT) == 2 ? 3 : 2;
}

struct __align__(8) UpdTail {
    uint64_t zfull[UPD_MAX_NZ], zempty[UPD_MAX_NZ];  // pieces of Z
    uint64_t afull, aempty;                          // the split parts of a tile
    uint64_t dfull[UPD_MAX_NG], dempty[UPD_MAX_NG];  // accumulators
    uint64_t fin;
    uint32_t tmem_base;
    int abort;
};

DSANLS_DEV float upd_project(float v, float bound, int *flag) {
    if (!(fabsf(v) <= 3.402823466e38f)) {  // NaN or Inf
        *flag = 1;
        return 0.0f;
    }
    return fminf(fmaxf(v, 0.0f), bound);
}

// Shared memory by its own address space: through the 64-bit pointers that the aligned
// start of dynamic shared memory gives, the compiler keeps every access behind the stores
// to Z before it.
DSANLS_DEV float4 lds4(uint32_t a) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(a));
    return v;
}
DSANLS_DEV float lds1(uint32_t a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
// Four consecutive elements of a row in global memory, `n` of them valid (the rest 0).
template <bool VEC>
DSANLS_DEV void load4(const float *p, int n, float *y) {
    if (VEC) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (n > 0) v = *reinterpret_cast<const float4 *>(p);
        y[0] = v.x, y[1] = v.y, y[2] = v.z, y[3] = v.w;
    } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) y[u] = u < n ? p[u] : 0.0f;
    }
}
template <bool VEC>
DSANLS_DEV void load4(const __nv_bfloat16 *p, int n, float *y) {
    if (VEC) {
        uint2 w = make_uint2(0u, 0u);
        if (n > 0) w = *reinterpret_cast<const uint2 *>(p);
        y[0] = __uint_as_float(w.x << 16), y[1] = __uint_as_float(w.x & 0xffff0000u);
        y[2] = __uint_as_float(w.y << 16), y[3] = __uint_as_float(w.y & 0xffff0000u);
    } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) y[u] = u < n ? __bfloat162float(p[u]) : 0.0f;
    }
}
template <bool VEC>
DSANLS_DEV void store4(float *p, int n, const float *v) {
    if (VEC) {
        if (n > 0) *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (u < n) p[u] = v[u];
    }
}
template <bool VEC>
DSANLS_DEV void store4(__nv_bfloat16 *p, int n, const float *v) {
    if (VEC) {
        if (n > 0) *reinterpret_cast<uint2 *>(p) = make_uint2(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]));
    } else {
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (u < n) p[u] = __float2bfloat16_rn(v[u]);
    }
}

// Four consecutive elements of a row in shared memory, `n` of them valid (the rest 0).
template <bool VEC>
DSANLS_DEV void lds_row(uint32_t p, int n, float *y, float) {
    if (VEC) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (n > 0) v = lds4(p);
        y[0] = v.x, y[1] = v.y, y[2] = v.z, y[3] = v.w;
    } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) y[u] = u < n ? lds1(p + 4 * u) : 0.0f;
    }
}
template <bool VEC>
DSANLS_DEV void lds_row(uint32_t p, int n, float *y, __nv_bfloat16) {
    if (VEC) {
        uint32_t a = 0u, b = 0u;
        if (n > 0) asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(a), "=r"(b) : "r"(p));
        y[0] = __uint_as_float(a << 16), y[1] = __uint_as_float(a & 0xffff0000u);
        y[2] = __uint_as_float(b << 16), y[3] = __uint_as_float(b & 0xffff0000u);
    } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            uint16_t h = 0;
            if (u < n) asm volatile("ld.shared.b16 %0, [%1];" : "=h"(h) : "r"(p + 2 * u));
            y[u] = __uint_as_float((uint32_t)h << 16);
        }
    }
}

template <typename ZT>
struct UpdSub {
    const int64_t *ptr;
    const int32_t *col;
    const float *val;
    const ZT *Y;
    int64_t yrows;
    float alpha;
    int most;  // entries of a row whose r is formed here; a longer row's is in R
};

struct UpdShape {
    int k, N, katoms;        // N: k up to 16; katoms: K atoms of 64 columns
    int na;                  // accumulators
    int nz, zbytes;          // pieces of Z in shared memory and their size
    int bulk;                // Z starts on 16 bytes: its pieces can come by bulk copies
    int acol;                // tensor-memory column of the A parts
    uint32_t tmem_cols;
};

// One product issued by one lane of a warp that runs converged: the operands stay in uniform
// registers.  Under a lane test each of them is moved there first, 148 clk a product beside
// 19 busy warps instead of the 56 that the tensor core takes.
DSANLS_DEV void upd_mma(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
        "r"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}

DSANLS_DEV void upd_commit(uint64_t *bar) {
    asm volatile(
        "{\n\t.reg .pred e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(smem_u32(bar))
        : "memory");
}

// The products of a tile, in the order of the parts: z_h (g_h, g_m, g_l), z_m (g_h, g_m),
// z_l g_h.  Descriptor steps in units of 16 bytes: part of G, K atom of 64, 16 columns.
template <int KS, int ZPARTS>
DSANLS_DEV void upd_products(uint32_t d, uint32_t a, uint64_t b, int part, int atom, uint32_t idesc) {
#pragma unroll
    for (int i = 0; i < ZPARTS; ++i)
#pragma unroll
        for (int p = 0; i + p < 3; ++p)
#pragma unroll
            for (int ks = 0; ks < KS; ++ks)
                upd_mma(d, a + (i * KS + ks) * 8, b + (uint64_t)(p * part + (ks >> 2) * atom + (ks & 3) * 2), idesc,
                                (i | p | ks) != 0);
}

template <typename ZT, bool SPR, bool VEC>
__global__ void __launch_bounds__(UPD_THREADS)
    k_update_tc(ZT *__restrict__ Z, const float *__restrict__ R, int64_t rows, UpdShape sh,
                const float *__restrict__ Gf, int kp, const double *__restrict__ scal, float bound,
                int *__restrict__ flag, UpdSub<ZT> sub, WaitSwitch wait) {
    constexpr bool ZBF = sizeof(ZT) == 2;
    constexpr int UPD_STEP = UPD_STEPS / upd_groups<ZT>();  // warps of a step group
    constexpr int ZPARTS = ZBF ? 1 : 3;  // nonzero parts of the split of z
    extern __shared__ uint8_t upd_smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(upd_smem_raw) + 1023) & ~uintptr_t(1023));
    const int k = sh.k, N = sh.N, KC = sh.katoms * 64;
    const int b_part = sh.katoms * N * 128;
    uint8_t *Bp = base;  // 3 parts x katoms x N rows x 128 B
    uint8_t *zb = Bp + 3 * b_part;
    UpdTail *tail = reinterpret_cast<UpdTail *>(zb + sh.nz * sh.zbytes);
    volatile int *abort = &tail->abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int w_step = UPD_SPLIT, w_mma = w_step + sh.na * UPD_STEP, w_copy = w_mma + 1;
    const int KS = (k + 15) >> 4;  // K steps (and output chunks) of 16 that hold data
    const int64_t ntiles = (rows + UPD_BM - 1) / UPD_BM;
    const int nt = (int)((ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x);  // tiles of this CTA
    auto tile_of = [&](int j) { return (int64_t)blockIdx.x + (int64_t)j * gridDim.x; };
    // piece p = 4 j + q: rows 32 q.. of tile j; its first row and how many there are (<= 0: none)
    auto row_of = [&](int p) { return tile_of(p >> 2) * UPD_BM + 32 * (p & 3); };
    auto nrows = [&](int p) { return (int)min((int64_t)32, rows - row_of(p)); };
    auto zpiece = [&](int p) { return reinterpret_cast<ZT *>(zb + (p % sh.nz) * sh.zbytes); };
    auto full_wait = [&](uint64_t *bars, int p, int n) { return role_wait(&bars[p % n], (p / n) & 1, abort, wait.ns); };
    auto free_wait = [&](uint64_t *bars, int p, int n) {
        return p < n || role_wait(&bars[p % n], ((p / n) - 1) & 1, abort, wait.ns);
    };

    // R given: the first tile, when it is whole, is asked for while G is split, 1 us of the 7
    // that a CTA with one tile takes.  (SPR goes without: the same lines cost the code of its
    // step 11 % of 2e6 rows in bf16, 484 -> 530 us.)
    const bool early = !SPR && sh.bulk && ((int64_t)blockIdx.x + 1) * UPD_BM <= rows && !wait.starve;
    if (warp == w_copy) {
        if (lane == 0) {
            for (int i = 0; i < sh.nz; ++i) {
                mbar_init(&tail->zfull[i], 1);
                mbar_init(&tail->zempty[i], UPD_STEP / 4);
            }
            mbar_init(&tail->afull, UPD_SPLIT);
            mbar_init(&tail->aempty, 1);
            for (int i = 0; i < sh.na; ++i) {
                mbar_init(&tail->dfull[i], 1);
                mbar_init(&tail->dempty[i], UPD_STEP);
            }
            mbar_init(&tail->fin, 1);
            tail->abort = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            if (early) {
                const uint32_t bytes = 32 * k * (int)sizeof(ZT);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                for (int q = 0; q < 4; ++q) {
                    mbar_expect_tx(&tail->zfull[q], bytes);
                    bulk_load(zb + q * sh.zbytes, Z + ((int64_t)blockIdx.x * UPD_BM + 32 * q) * k, bytes,
                              &tail->zfull[q]);
                }
            }
        }
    }
    if (warp == w_mma) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tail->tmem_base)),
                     "r"(sh.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // the three parts of G: B row n, K column c holds G[n][c] (G is symmetric)
    for (int e = tid; e < N * KC; e += blockDim.x) {
        const int n = e >> (5 + sh.katoms), c = e & (KC - 1);
        const float g = (n < k && c < k) ? Gf[n * kp + c] : 0.0f;
        __nv_bfloat16 h, m, l;
        split3_one(g, h, m, l);
        const int off = sw128_off(n, c, N);
        *reinterpret_cast<__nv_bfloat16 *>(Bp + off) = h;
        *reinterpret_cast<__nv_bfloat16 *>(Bp + b_part + off) = m;
        *reinterpret_cast<__nv_bfloat16 *>(Bp + 2 * b_part + off) = l;
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = tail->tmem_base;
    if (warp < w_step) {
        // ---- split ----
        const uint32_t ta = tmem + ((uint32_t)(32 * warp) << 16) + sh.acol;
        for (int j = 0; j < nt; ++j) {
            const int p = 4 * j + warp, nv = lane < nrows(p) ? k : 0;  // valid columns of the row
            // (the parts are free: every piece of the tiles before has landed, so the parity
            // of zfull, nz >= 4, cannot be two phases behind)
            const bool ok = free_wait(&tail->aempty, j, 1) && full_wait(tail->zfull, p, sh.nz);
            if (!__all_sync(0xffffffffu, ok)) break;
            fence_after();
            const uint32_t z = smem_u32(zpiece(p) + lane * k);
            for (int c = 0; c < 16 * KS; c += 8) {
                float v[8];
                lds_row<VEC>(z + c * (int)sizeof(ZT), nv - c, v, ZT());
                lds_row<VEC>(z + (c + 4) * (int)sizeof(ZT), nv - c - 4, v + 4, ZT());
                uint32_t h[4], m[4], l[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    h[e] = pack_bf16(v[2 * e], v[2 * e + 1]);
                    if (!ZBF) {
                        const float a0 = __fsub_rn(v[2 * e], __uint_as_float(h[e] << 16));
                        const float a1 = __fsub_rn(v[2 * e + 1], __uint_as_float(h[e] & 0xffff0000u));
                        m[e] = pack_bf16(a0, a1);
                        l[e] = pack_bf16(__fsub_rn(a0, __uint_as_float(m[e] << 16)),
                                         __fsub_rn(a1, __uint_as_float(m[e] & 0xffff0000u)));
                    }
                }
                tmem_st(ta + c / 2, h);
                if (!ZBF) {
                    tmem_st(ta + 8 * KS + c / 2, m);
                    tmem_st(ta + 16 * KS + c / 2, l);
                }
            }
            tmem_st_wait();
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tail->afull);
        }
    } else if (warp < w_mma) {
        // ---- step ----
        const int g = (warp - w_step) / UPD_STEP, q = warp & 3, part = (warp - w_step) % UPD_STEP / 4;
        const uint32_t td = tmem + ((uint32_t)(32 * q) << 16) + g * N;
        const float eta = (float)scal[2], bnd = bound > 0.0f ? bound : 3.402823466e38f;
        int64_t e0 = 0, n0 = 0;  // the row's entries: first and number, this tile's and the next one's
        int en = 0, nn = 0;
        auto range = [&](int j, int64_t &a, int &n) {
            a = 0, n = 0;
            if (SPR && j < nt && lane < nrows(4 * j + q)) {
                const int64_t row = row_of(4 * j + q) + lane;
                a = sub.ptr[row];
                n = (int)min(sub.ptr[row + 1] - a, (int64_t)sub.most + 1);
            }
        };
        range(g, e0, en);
        for (int j = g; j < nt; j += sh.na, e0 = n0, en = nn) {
            const int p = 4 * j + q, kv = lane < nrows(p) ? k : 0;
            const int64_t off = (row_of(p) + lane) * (int64_t)k;
            range(j + sh.na, n0, nn);
            const bool given = !SPR || en > sub.most;  // r comes in R
            // the first two entries, read once for every chunk
            float v0 = 0.0f, v1 = 0.0f;
            int32_t y0 = 0, y1 = 0;
            if (SPR && !given) {
                if (en > 0) {
                    v0 = sub.val[e0];
                    y0 = sub.col[e0];
                }
                if (en > 1) {
                    v1 = sub.val[e0 + 1];
                    y1 = sub.col[e0 + 1];
                }
            }
            const uint32_t z = smem_u32(zpiece(p) + lane * k);
            bool ok = true;
            for (int ci = part; ci < KS; ci += UPD_STEP / 4) {
                const int c0 = 16 * ci, nv = kv - c0;
                float rv[16];
                if (given) {
#pragma unroll
                    for (int e = 0; e < 16; e += 4) load4<VEC>(R + off + c0 + e, nv - e, rv + e);
                } else {
#pragma unroll
                    for (int e = 0; e < 16; ++e) rv[e] = 0.0f;
                    float vn = v0;
                    int32_t yn = y0;
                    float vm = v1;
                    int32_t ym = y1;
                    for (int i = 0; i < en; ++i) {
                        const float v = vn;
                        const int32_t y = yn;
                        vn = vm, yn = ym;
                        if (i + 2 < en) {  // two entries ahead of the row of Y
                            vm = sub.val[e0 + i + 2];
                            ym = sub.col[e0 + i + 2];
                        }
                        if (!DSANLS_IN(y, sub.yrows, 301)) continue;
                        const ZT *yr = sub.Y + (int64_t)y * k + c0;
                        float a[16];
#pragma unroll
                        for (int e = 0; e < 16; e += 4) load4<VEC>(yr + e, nv - e, a + e);
#pragma unroll
                        for (int e = 0; e < 16; ++e) rv[e] = __fmaf_rn(v, a[e], rv[e]);
                    }
#pragma unroll
                    for (int e = 0; e < 16; ++e) rv[e] = __fmul_rn(sub.alpha, rv[e]);
                }
                __syncwarp();
                if (ci == part) {  // the tile's products, and with them its z
                    ok = __all_sync(0xffffffffu, full_wait(tail->dfull, j, sh.na) && full_wait(tail->zfull, p, sh.nz));
                    if (!ok) break;
                    fence_after();
                }
#pragma unroll
                for (int hh = 0; hh < 16; hh += 8) {
                    uint32_t d[8];
                    tmem_ld8(td + c0 + hh, d);
                    float zv[8];
                    lds_row<VEC>(z + (c0 + hh) * (int)sizeof(ZT), nv - hh, zv, ZT());
                    lds_row<VEC>(z + (c0 + hh + 4) * (int)sizeof(ZT), nv - hh - 4, zv + 4, ZT());
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const float grad = __fsub_rn(__uint_as_float(d[e]), rv[hh + e]);
                        zv[e] = upd_project(__fmaf_rn(-eta, grad, zv[e]), bnd, flag);
                    }
                    store4<VEC>(Z + off + c0 + hh, nv - hh, zv);
                    store4<VEC>(Z + off + c0 + hh + 4, nv - hh - 4, zv + 4);
                }
            }
            if (!ok) break;
            fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&tail->dempty[g]);
                mbar_arrive(&tail->zempty[p % sh.nz]);
            }
        }
    } else if (warp == w_mma) {
        // ---- mma ----
        const uint32_t idesc = idesc_bf16(UPD_BM, N);
        const uint64_t bdesc = sw128_desc(smem_u32(Bp));
        const uint32_t tbase = __shfl_sync(0xffffffffu, tmem, 0);
        const int b16 = b_part >> 4, n8 = N * 8;
        for (int j = 0; j < nt; ++j) {
            const int g = j % sh.na;
            const bool ok = free_wait(tail->dempty, j, sh.na) && full_wait(&tail->afull, j, 1);
            if (!__all_sync(0xffffffffu, ok)) break;
            fence_after();
            const uint32_t d = tbase + g * N, a = tbase + sh.acol;
            switch (KS) {
                case 3: upd_products<3, ZPARTS>(d, a, bdesc, b16, n8, idesc); break;
                case 4: upd_products<4, ZPARTS>(d, a, bdesc, b16, n8, idesc); break;
                case 5: upd_products<5, ZPARTS>(d, a, bdesc, b16, n8, idesc); break;
                case 6: upd_products<6, ZPARTS>(d, a, bdesc, b16, n8, idesc); break;
                case 7: upd_products<7, ZPARTS>(d, a, bdesc, b16, n8, idesc); break;
                default: upd_products<8, ZPARTS>(d, a, bdesc, b16, n8, idesc); break;
            }
            upd_commit(&tail->aempty);
            upd_commit(&tail->dfull[g]);
        }
        // every product of this warp has retired before the tensor memory is freed
        upd_commit(&tail->fin);
        mbar_wait(&tail->fin, 0, wait.ns);
    } else if (warp == w_copy) {
        // ---- copy ----
        int issued = early ? 4 : 0;
        for (int p = issued; p < 4 * nt && !wait.starve; ++p) {
            const int nr = max(0, nrows(p));
            const uint32_t bytes = (uint32_t)(nr * k * (int)sizeof(ZT));
            if (!__all_sync(0xffffffffu, free_wait(tail->zempty, p, sh.nz))) break;
            uint64_t *full = &tail->zfull[p % sh.nz];
            const ZT *src = Z + row_of(p) * (int64_t)k;
            if (sh.bulk && bytes > 0 && (bytes & 15) == 0) {
                if (lane == 0) {
                    mbar_expect_tx(full, bytes);
                    bulk_load(zpiece(p), src, bytes, full);
                }
            } else {
                ZT *dst = zpiece(p);
                for (int e = lane; e < nr * k; e += 32) dst[e] = src[e];
                __syncwarp();
                if (lane == 0) mbar_arrive(full);
            }
            issued = p + 1;
        }
        if (*abort && lane == 0)  // nobody may be waiting for the last copies any more
            for (int p = max(0, issued - sh.nz); p < issued; ++p)
                mbar_wait(&tail->zfull[p % sh.nz], (p / sh.nz) & 1, wait.ns);
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (tid == 0 && tail->abort) atomicOr(flag, 2);
    if (warp == w_mma)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(sh.tmem_cols) : "memory");
}

template <typename ZT, bool SPR>
void launch_update_tc_any(ZT *Z, const float *R, int64_t rows, int k, const float *Gf, int kp, const double *scal,
                          float bound, int *flag, UpdSub<ZT> sub, cudaStream_t s) {
    if (!update_tc_supported(k)) throw ArgError{"launch_update_tc: needs 32 < k <= 128"};
    if (rows <= 0) return;
    int dev = 0, sms = 152;
    DSANLS_CUDA(cudaGetDevice(&dev));
    DSANLS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    UpdShape sh{};
    sh.k = k;
    sh.N = (k + 15) / 16 * 16;
    sh.katoms = k <= 64 ? 1 : 2;
    const int acols = (sizeof(ZT) == 2 ? 1 : 3) * sh.N / 2;
    sh.na = std::min(upd_groups<ZT>(), (512 - acols) / sh.N);  // accumulators that fit beside the A parts
    sh.bulk = (reinterpret_cast<uintptr_t>(Z) & 15) == 0 && (32 * (size_t)k * sizeof(ZT)) % 16 == 0;
    sh.acol = sh.na * sh.N;
    sh.tmem_cols = 32;
    while ((int)sh.tmem_cols < sh.acol + acols) sh.tmem_cols <<= 1;
    sh.zbytes = (int)((32 * (size_t)k * sizeof(ZT) + 127) / 128 * 128);
    const size_t fixed = 1024 + 3 * (size_t)sh.katoms * sh.N * 128 + sizeof(UpdTail);
    sh.nz = std::min(UPD_MAX_NZ, (int)((227 * 1024 - fixed) / sh.zbytes));  // 8 at k = 128 in binary32, 11 at 100
    const int64_t ntiles = (rows + UPD_BM - 1) / UPD_BM;
    const int64_t grid = std::min<int64_t>(ntiles, sms);  // one CTA per SM (shared memory and TMEM)
    if (ntiles / grid >= (1ll << 28)) throw ArgError{"launch_update_tc: too many rows"};
    const size_t smem = fixed + sh.nz * (size_t)sh.zbytes;
    const auto kern = k % 4 == 0 ? k_update_tc<ZT, SPR, true> : k_update_tc<ZT, SPR, false>;
    const int threads = 32 * (UPD_SPLIT + sh.na * (UPD_STEPS / upd_groups<ZT>()) + 2);
    kern<<<(unsigned)grid, threads, smem, s>>>(Z, R, rows, sh, Gf, kp, scal, bound, flag, sub, wait_switch());
    DSANLS_LAUNCH_CHECK();
}

}  // namespace

bool update_tc_supported(int k) { return k > 32 && k <= 128; }

template <typename ZT>
void launch_update_tc(ZT *Z, const float *R, int64_t rows, int k, const float *Gf, int kp, const double *scal,
                      float bound, int *flag, cudaStream_t s) {
    launch_update_tc_any<ZT, false>(Z, R, rows, k, Gf, kp, scal, bound, flag, UpdSub<ZT>{}, s);
}
template void launch_update_tc<float>(float *, const float *, int64_t, int, const float *, int, const double *, float,
                                      int *, cudaStream_t);
template void launch_update_tc<__nv_bfloat16>(__nv_bfloat16 *, const float *, int64_t, int, const float *, int,
                                              const double *, float, int *, cudaStream_t);

template <typename ZT>
void launch_update_tc_subcsr(ZT *Z, const float *R, const SubCsr &sc, const ZT *Y, int64_t yrows, float alpha,
                             int64_t rows, int k, const float *Gf, int kp, const double *scal, float bound, int *flag,
                             cudaStream_t s) {
    if (sc.rows != rows) throw ArgError{"launch_update_tc_subcsr: the sub-CSR has other rows"};
    const UpdSub<ZT> sub{sc.ptr, sc.col[sc.cur], sc.val[sc.cur], Y, yrows, alpha, (int)sc.warp_rows()};
    launch_update_tc_any<ZT, true>(Z, R, rows, k, Gf, kp, scal, bound, flag, sub, s);
}
template void launch_update_tc_subcsr<float>(float *, const float *, const SubCsr &, const float *, int64_t, float,
                                             int64_t, int, const float *, int, const double *, float, int *,
                                             cudaStream_t);
template void launch_update_tc_subcsr<__nv_bfloat16>(__nv_bfloat16 *, const float *, const SubCsr &,
                                                     const __nv_bfloat16 *, int64_t, float, int64_t, int,
                                                     const float *, int, const double *, float, int *, cudaStream_t);

void bounds_report_tc(int reset, int64_t out[3]) {
#ifdef DSANLS_BOUNDS
    bounds_read_tu(reset, out);
#else
    (void)reset;
    out[0] = out[1] = out[2] = 0;
#endif
}

void prime_update_attributes(int max_smem) {
    allow_max_dynamic_smem(k_update_tc<float, false, true>, max_smem);
    allow_max_dynamic_smem(k_update_tc<float, false, false>, max_smem);
    allow_max_dynamic_smem(k_update_tc<float, true, true>, max_smem);
    allow_max_dynamic_smem(k_update_tc<float, true, false>, max_smem);
    allow_max_dynamic_smem(k_update_tc<__nv_bfloat16, false, true>, max_smem);
    allow_max_dynamic_smem(k_update_tc<__nv_bfloat16, false, false>, max_smem);
    allow_max_dynamic_smem(k_update_tc<__nv_bfloat16, true, true>, max_smem);
    allow_max_dynamic_smem(k_update_tc<__nv_bfloat16, true, false>, max_smem);
}


}  // namespace dsanls
