// Binary32-accurate GEMM on tcgen05 tensor cores from a binary32 first operand (the
// FP32 form's products: A = X S, R = A B^T, the sampled R = c^2 X[:, J] Y[J, :],
// B = Y^T S, and the wide products of the warm start's prediction).
//
// Every element is three bf16 parts, z = h + m + l (split3), and the six products
// whose parts' orders add to at most 2 are taken; the dropped ones are of order 2^-24
// of the product.  (The parts are bf16 values: below about 1e-33 an entry's third one is
// rounded or lost, between 3.39e38 and the largest binary32 its first is infinite.)  The
// second operand's parts are made beforehand (it is small or used by every row tile); the
// first operand's on its way to tensor memory, so a large matrix is read once, as binary32,
// and no split copy of it is kept.  The parts
// of the second operand lie side by side (BN columns each), so one K step takes the
// MMAs A_h x [B_h | B_m | B_l], A_m x [B_h | B_m], A_l x B_h (N = 3, 2, 1 BN; an MMA of
// N < 96 costs as much as one of 96) into three column blocks of tensor memory by
// order of magnitude: D0 = hh, D1 = hm + mh, D2 = hl + mm + lh.  A second operand of
// one part (bf16 values) takes A_h, A_m and A_l times it into D0, D1 and D2.
//
// The tensor cores' fp32 sums round toward zero, which drifts over a chain of
// additions of one sign.  So a chain lasts only FLUSH K blocks: the accumulating
// warps then add D0 + (D1 + D2) to binary32 registers, rounding to nearest, while the
// products fill the other set of accumulators (BN <= 64; with BN = 128 there is one
// set, and longer chains).
//
// One CTA per 128 x BN tile (and K split), warps by role, joined by mbarriers, in steps
// of 32 K:
//   conv   read 8 consecutive K of a row of the first operand's binary32 tile (a ring of
//          steps in shared memory), split them and store the parts to tensor memory, from
//          where the MMAs take A (row i in lane i).  Two groups take alternate steps.
//          Gathered K rows and rows that are not 16-byte aligned are copied by these
//          warps too, by cp.async, a ring ahead;
//   acc    accumulate (one row and half of the columns per thread), store the tile;
//   gate   one thread waits for a step's operands and accumulators and counts it ready;
//   mma    one thread issues the products.  It only polls the gate's count: an mbarrier
//          wait between MMAs costs it 195 cycles even when the phase is complete, which
//          the few MMAs queued do not cover (a step of 32 K is 384 cycles of products);
//   tma A  otherwise one tile copy per step; elements outside the matrix arrive as zeros;
//   tma B  copies the second operand's parts of each K block of 64.
// Measured (SM clock 2.0 GHz; the CUDA-core kernel in brackets): R of 65,536 x 64 from
// 2,048 K rows 149 us, gathered from 16,384 rows 181 us [1,017], of which HBM needs 79;
// from 16,384 K 948 us [11,000], HBM 635; A = X S of 13,500 x 500 x 5,000 317 us [3,150] =
// 213 TFLOP/s of binary32 work, 67% of the bf16 peak / 6.  A K block of 64 takes about
// 2,150 cycles against 832 of products (BN = 64) and 1,480 of HBM time: the chain split ->
// products -> next split through the two steps of A that fit in tensor memory next to the
// accumulators bounds it.  Forms tried on the same shape: eight warps that copy by
// cp.async, split both operands and meet at a barrier per step, 271 us (half of it the
// second operand and the copies' addresses); these roles with A's parts in shared memory,
// 148 us but 352 for A = X S (232 KB of shared-memory traffic per block); one group of
// splitting warps 166; without the gate 156; D1 and D2 in one block and four steps of A,
// 162 (five MMAs a K step instead of three).  Gathered rows by TMA (rows or
// tile::gather4) take the copy engine 80-110 cycles per row of 512 bytes: 264 us.
// Every wait is bounded and gives up together; the copies and MMAs in flight complete
// before the CTA leaves.
#include <cuda.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "tc_gemm.cuh"
#include "tc_ptx.cuh"

namespace dsanls {

namespace {

constexpr int SG_BM = 128, SG_BK = 64;
constexpr int SG_RK = 32;     // K of one step
constexpr int SG_RAW_BYTES = SG_BM * SG_RK * 4;
constexpr int SG_MAX_RAW = 8, SG_MAX_BST = 3, SG_MAX_AST = 4;
constexpr int SG_ACOLS = 3 * SG_RK / 2;  // tensor-memory columns of the parts of one step of A

template <int BN>
struct SgCfg {
    static constexpr int CW = BN <= 64 ? 16 : 8;     // splitting warps
    static constexpr int AW = 8;                     // accumulating warps
    static constexpr int THREADS = 32 * (CW + AW + 4);
    static constexpr int RAW = BN <= 64 ? 8 : 6;     // steps of the binary32 ring
    static constexpr int BST = BN <= 64 ? 3 : 2;     // K blocks of the second operand's ring
    static constexpr int NSET = BN <= 64 ? 2 : 1;    // accumulator sets
    static constexpr int FLUSH = BN <= 64 ? 2 : 4;   // K blocks per accumulator chain
    static constexpr int AST = BN <= 32 ? 4 : 2;     // steps of A in tensor memory
    static constexpr int BBYTES = 3 * BN * SG_BK * 2;
    static constexpr uint32_t DSET = 3 * BN;
    static constexpr uint32_t ACOL = NSET * DSET;    // A's parts after the accumulators
    static_assert(ACOL + AST * SG_ACOLS <= 512, "tensor memory");
    static constexpr uint32_t TCOLS = 512;
};

struct __align__(16) SgTail {
    uint64_t afull[SG_MAX_AST], aempty[SG_MAX_AST];  // A's parts of a step
    uint64_t bfull[SG_MAX_BST], bempty[SG_MAX_BST];  // B's parts of a K block
    uint64_t rfull[SG_MAX_RAW], rempty[SG_MAX_RAW];  // binary32 steps
    uint64_t dfull[2], dempty[2];
    uint64_t fin;
    uint32_t tmem_base;
    int abort;
    int ready;  // steps whose operands and accumulators are ready (gate -> mma)
};

template <int BN>
constexpr size_t sg_smem() {
    return 1024 + SgCfg<BN>::BST * (size_t)SgCfg<BN>::BBYTES + SgCfg<BN>::RAW * SG_RAW_BYTES + sizeof(SgTail);
}

// wait (bounded) for the gate's count of ready steps to exceed st; the count, or <= st when giving up
DSANLS_DEV int sg_poll(const int *count, int st, volatile int *abort, unsigned long long limit) {
    int n = 0;
    unsigned long long t0 = 0;
    for (int spin = 1;; ++spin) {
        asm volatile("ld.acquire.cta.shared::cta.b32 %0, [%1];" : "=r"(n) : "r"(smem_u32(count)) : "memory");
        if (n > st || *abort) return n;
        if ((spin & 255) == 0) {
            const unsigned long long t = globaltimer_ns();
            if (t0 == 0) t0 = t;
            if (t - t0 > limit) {
                *abort = 1;
                return n;
            }
        }
    }
}

// 16- and 4-byte copies of which `bytes` are read and the rest zero
DSANLS_DEV void sg_copy16(void *dst, const float *src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes)
                 : "memory");
}
DSANLS_DEV void sg_copy4(void *dst, const float *src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes)
                 : "memory");
}
// arrive on the barrier (which counts this thread) once its copies so far have landed
DSANLS_DEV void sg_copies_arrive(uint64_t *bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// the parts of 8 consecutive K, two bf16 per word
DSANLS_DEV void sg_split8(const float (&v)[8], uint32_t *h, uint32_t *m, uint32_t *l) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float z0 = v[2 * e], z1 = v[2 * e + 1];
        h[e] = pack_bf16(z0, z1);
        const float a0 = __fsub_rn(z0, __uint_as_float(h[e] << 16));
        const float a1 = __fsub_rn(z1, __uint_as_float(h[e] & 0xffff0000u));
        m[e] = pack_bf16(a0, a1);
        l[e] = pack_bf16(__fsub_rn(a0, __uint_as_float(m[e] << 16)),
                         __fsub_rn(a1, __uint_as_float(m[e] & 0xffff0000u)));
    }
}

// 8 K elements (chunk c of the step) of row r from the step's binary32 tile: [row][32]
// with the 16-byte pieces of a row swizzled by TMA (KC), or [K][128].  A warp's lanes are
// 32 rows: no bank conflicts in either.
template <bool KC>
DSANLS_DEV void sg_read(float (&v)[8], const float *raw, int r, int c) {
    if (KC) {
        const float4 *q = reinterpret_cast<const float4 *>(raw + r * SG_RK);
        const float4 x = q[(2 * c) ^ (r & 7)], y = q[(2 * c + 1) ^ (r & 7)];
        v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w, v[4] = y.x, v[5] = y.y, v[6] = y.z, v[7] = y.w;
    } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = raw[(8 * c + e) * SG_BM + r];
    }
}

template <int BN, bool AK, int NPB>
__global__ void __launch_bounds__(SgCfg<BN>::THREADS, 1)
    k_split_gemm(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, int64_t M,
                 int64_t N, int64_t K, const float *__restrict__ A, int64_t lda, const int32_t *__restrict__ gather,
                 int tma, int avec, WaitSwitch wait, float *__restrict__ C, int64_t ldm, int64_t ldn, float alpha,
                 int kb_per_split, int64_t c_split_stride, int *__restrict__ err) {
    using Cfg = SgCfg<BN>;
    constexpr int CW = Cfg::CW, AW = Cfg::AW, NSET = Cfg::NSET, FLUSH = Cfg::FLUSH, RAW = Cfg::RAW;
    constexpr int BST = Cfg::BST, AST = Cfg::AST, BPART = BN * 128;
    constexpr int GW = CW / 2;   // warps of a splitting group: one takes the even steps, the other the odd ones
    constexpr int NU = 16 / GW;  // 8-K chunks of a splitting thread's row per step
    static_assert(RAW % 2 == 0 && AST % 2 == 0, "a step's slots belong to one group");
    extern __shared__ __align__(1024) uint8_t sg_raw[];
    uint8_t *base = sg_raw + ((1024u - (smem_u32(sg_raw) & 1023u)) & 1023u);
    float *raw = reinterpret_cast<float *>(base);
    uint8_t *bst = base + RAW * SG_RAW_BYTES;  // BST x NPB parts of BN x 64
    SgTail *tail = reinterpret_cast<SgTail *>(bst + BST * Cfg::BBYTES);
    volatile int *abort = &tail->abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t ntn = ceil_div(N, BN);
    const int64_t m0 = (int64_t)(blockIdx.x / ntn) * SG_BM, n0 = (int64_t)(blockIdx.x % ntn) * BN;
    const int64_t kb0 = (int64_t)blockIdx.y * kb_per_split;
    const int nkb = (int)min((int64_t)kb_per_split, ceil_div(K, SG_BK) - kb0);
    const int nst = 2 * nkb;
    const int64_t kbeg = kb0 * SG_BK;
    if (tid == 0) {
        for (int s = 0; s < AST; ++s) {
            mbar_init(&tail->afull[s], GW);
            mbar_init(&tail->aempty[s], 1);
        }
        for (int s = 0; s < BST; ++s) {
            mbar_init(&tail->bfull[s], 1);
            mbar_init(&tail->bempty[s], 1);
        }
        for (int r = 0; r < RAW; ++r) {
            mbar_init(&tail->rfull[r], tma ? 1 : 32 * GW);
            mbar_init(&tail->rempty[r], GW);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tail->dfull[b], 1);
            mbar_init(&tail->dempty[b], 32 * AW);
        }
        mbar_init(&tail->fin, 1);
        tail->abort = 0;
        tail->ready = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == CW + AW) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tail->tmem_base)),
                     "r"(Cfg::TCOLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = tail->tmem_base;

    if (warp < CW) {
        // ---- conv: group gr, rows of lane quarter q, chunks NU j .. NU j + NU - 1 of its steps ----
        const int gr = warp / GW, wl = warp % GW, q = wl & 3, j = wl >> 2, r = 32 * q + lane;
        const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + Cfg::ACOL + 4 * NU * j;
        // without tile copies (gathered K rows, rows of any alignment) the group copies its own steps,
        // RAW steps ahead: rows RPW wl .. of K, or tile rows TPW wl .. with the lanes along K
        constexpr int RPW = SG_RK / GW, TPW = SG_BM / GW;
        auto row_index = [&](int st) -> int {  // lane i < RPW: the matrix row of the i-th K row
            const int64_t k = kbeg + st * SG_RK + RPW * wl + lane;
            return !AK && lane < RPW && st < nst && k < K ? (gather ? __ldg(gather + k) : (int)k) : -1;
        };
        auto copy_step = [&](int st, int idx) {
            float *dst = raw + (st % RAW) * (SG_RAW_BYTES / 4);
            if (AK) {
                const int64_t k = kbeg + st * SG_RK + lane;
#pragma unroll 4
                for (int i = 0; i < TPW; ++i) {
                    const int t = TPW * wl + i;
                    const bool in = k < K && m0 + t < M;
                    sg_copy4(dst + t * SG_RK + (((lane >> 2) ^ (t & 7)) << 2) + (lane & 3),
                             in ? A + (m0 + t) * lda + k : A, in ? 4 : 0);
                }
            } else {
#pragma unroll
                for (int i = 0; i < RPW; ++i) {
                    const int row = __shfl_sync(0xffffffffu, idx, i);
                    const float *src = A + (int64_t)max(row, 0) * lda + m0;
                    float *d = dst + (RPW * wl + i) * SG_BM;
                    if (avec) {
                        const int64_t left = row >= 0 ? M - m0 - 4 * lane : 0;
                        sg_copy16(d + 4 * lane, left > 0 ? src + 4 * lane : A,
                                  left >= 4 ? 16 : (left > 0 ? 4 * (int)left : 0));
                    } else {
#pragma unroll
                        for (int u = 0; u < SG_BM; u += 32) {
                            const bool in = row >= 0 && m0 + u + lane < M;
                            sg_copy4(d + u + lane, in ? src + u + lane : A, in ? 4 : 0);
                        }
                    }
                }
            }
            sg_copies_arrive(&tail->rfull[st % RAW]);
        };
        int next = -1;  // row_index of step st + RAW
        if (!tma && !wait.starve) {
            for (int st = gr; st < RAW; st += 2)
                if (st < nst) copy_step(st, row_index(st));
            next = row_index(RAW + gr);
        }
        for (int st = gr; st < nst; st += 2) {
            const int slot = st % RAW, sa = st % AST;
            bool ok = role_wait(&tail->rfull[slot], (st / RAW) & 1, abort, wait.ns);
            if (ok && st >= AST) ok = role_wait(&tail->aempty[sa], ((st / AST) - 1) & 1, abort, wait.ns);
            if (!__all_sync(0xffffffffu, ok)) break;
            fence_after();
#pragma unroll
            for (int i = 0; i < NU; ++i) {
                float v[8];
                uint32_t h[4], m[4], l[4];
                sg_read<AK>(v, raw + slot * (SG_RAW_BYTES / 4), r, NU * j + i);
                sg_split8(v, h, m, l);
                tmem_st(ta + sa * SG_ACOLS + 4 * i, h);
                tmem_st(ta + sa * SG_ACOLS + SG_RK / 2 + 4 * i, m);
                tmem_st(ta + sa * SG_ACOLS + SG_RK + 4 * i, l);
            }
            tmem_st_wait();
            fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&tail->afull[sa]);
                mbar_arrive(&tail->rempty[slot]);
            }
            if (!tma && st + RAW < nst) {  // the slot is free once the group has read it
                const bool free = role_wait(&tail->rempty[slot], (st / RAW) & 1, abort, wait.ns);
                if (!__all_sync(0xffffffffu, free)) break;
                copy_step(st + RAW, next);
                next = row_index(st + RAW + 2);
            }
        }
        if (!tma) asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (warp < CW + AW) {
        // ---- acc ----
        constexpr int NC = BN / 2;  // columns of this thread
        const int q = warp & 3, half = (warp - CW) >> 2;
        const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16) + half * NC;
        float acc[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c] = 0.0f;
        const int niv = (nkb + FLUSH - 1) / FLUSH;
        bool ok = true;
        for (int iv = 0; iv < niv; ++iv) {
            const int buf = iv % NSET;
            ok = __all_sync(0xffffffffu, role_wait(&tail->dfull[buf], (iv / NSET) & 1, abort, wait.ns));
            if (!ok) break;
            fence_after();
#pragma unroll
            for (int c = 0; c < NC; c += 8) {
                uint32_t d0[8], d1[8], d2[8];
                tmem_ld8(tl + buf * Cfg::DSET + c, d0);
                tmem_ld8(tl + buf * Cfg::DSET + BN + c, d1);
                tmem_ld8(tl + buf * Cfg::DSET + 2 * BN + c, d2);
                tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    acc[c + e] = __fadd_rn(
                        acc[c + e], __fadd_rn(__uint_as_float(d0[e]),
                                              __fadd_rn(__uint_as_float(d1[e]), __uint_as_float(d2[e]))));
            }
            fence_before();
            mbar_arrive(&tail->dempty[buf]);
        }
        const int64_t r = m0 + q * 32 + lane, c0 = n0 + half * NC;
        if (ok && r < M) {
            float *dst = C + (int64_t)blockIdx.y * c_split_stride + r * ldm + c0 * ldn;
            const bool vec = ldn == 1 && (ldm & 3) == 0 && (reinterpret_cast<uintptr_t>(dst) & 15) == 0;
#pragma unroll
            for (int c = 0; c < NC; c += 4) {
                float x[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) x[e] = __fmul_rn(alpha, acc[c + e]);
                if (vec && c0 + c + 4 <= N) {
                    *reinterpret_cast<float4 *>(dst + c) = make_float4(x[0], x[1], x[2], x[3]);
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (c0 + c + e < N) dst[(c + e) * ldn] = x[e];
                }
            }
        }
    } else if (warp == CW + AW) {
        if (lane == 0) {
            // ---- mma ----
            const uint32_t id1 = idesc_bf16(SG_BM, BN), id2 = idesc_bf16(SG_BM, 2 * BN);
            const uint32_t id3 = idesc_bf16(SG_BM, BN <= 64 ? 3 * BN : BN);
            int ready = 0;
            for (int st = 0; st < nst; ++st) {
                const int kb = st >> 1, sb = kb % BST, sa = st % AST, iv = kb / FLUSH, buf = iv % NSET;
                const bool first = st % (2 * FLUSH) == 0;
                if (ready <= st) ready = sg_poll(&tail->ready, st, abort, wait.ns);
                if (ready <= st) break;
                fence_after();
                const uint32_t ah = tmem + Cfg::ACOL + sa * SG_ACOLS, am = ah + SG_RK / 2, al = am + SG_RK / 2;
                const uint32_t bb = smem_u32(bst + sb * Cfg::BBYTES) + (st & 1) * 64, d = tmem + buf * Cfg::DSET;
#pragma unroll
                for (int kk = 0; kk < SG_RK / 16; ++kk) {
                    const uint32_t on = !first || kk > 0, o = 8 * kk;
                    const uint64_t bh = sw128_desc(bb + kk * 32);
                    if (NPB == 1) {
                        mma_bf16_tmem_a(d, ah + o, bh, id1, on);
                        mma_bf16_tmem_a(d + BN, am + o, bh, id1, on);
                        mma_bf16_tmem_a(d + 2 * BN, al + o, bh, id1, on);
                    } else if (BN <= 64) {
                        mma_bf16_tmem_a(d, ah + o, bh, id3, on);
                        mma_bf16_tmem_a(d + BN, am + o, bh, id2, 1);
                        mma_bf16_tmem_a(d + 2 * BN, al + o, bh, id1, 1);
                    } else {
                        mma_bf16_tmem_a(d, ah + o, bh, id2, on);
                        mma_bf16_tmem_a(d + 2 * BN, ah + o, sw128_desc(bb + 2 * BPART + kk * 32), id1, on);
                        mma_bf16_tmem_a(d + BN, am + o, bh, id2, 1);
                        mma_bf16_tmem_a(d + 2 * BN, al + o, bh, id1, 1);
                    }
                }
                mma_commit(&tail->aempty[sa]);
                if (st & 1) {
                    mma_commit(&tail->bempty[sb]);
                    if ((kb + 1) % FLUSH == 0 || kb + 1 == nkb) mma_commit(&tail->dfull[buf]);
                }
            }
            // every product this thread issued has retired before the tensor memory is freed
            mma_commit(&tail->fin);
            mbar_wait(&tail->fin, 0, wait.ns);
        }
    } else if (warp == CW + AW + 3) {
        if (lane == 0) {
            // ---- gate ----
            for (int st = 0; st < nst; ++st) {
                const int kb = st >> 1, iv = kb / FLUSH;
                if (st % (2 * FLUSH) == 0 && iv >= NSET &&
                    !role_wait(&tail->dempty[iv % NSET], ((iv / NSET) - 1) & 1, abort, wait.ns))
                    break;
                if ((st & 1) == 0 && !role_wait(&tail->bfull[kb % BST], (kb / BST) & 1, abort, wait.ns)) break;
                if (!role_wait(&tail->afull[st % AST], (st / AST) & 1, abort, wait.ns)) break;
                fence_after();
                fence_before();
                asm volatile("st.release.cta.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tail->ready)), "r"(st + 1)
                             : "memory");
            }
        }
    } else if (warp == CW + AW + 1) {
        if (tma && lane == 0 && !wait.starve) {
            // ---- tma A ----
            int issued = 0;
            for (int st = 0; st < nst; ++st) {
                const int slot = st % RAW;
                if (st >= RAW && !role_wait(&tail->rempty[slot], ((st / RAW) - 1) & 1, abort, wait.ns)) break;
                float *dst = raw + slot * (SG_RAW_BYTES / 4);
                const int k0 = (int)(kbeg + st * SG_RK);
                mbar_expect_tx(&tail->rfull[slot], SG_RAW_BYTES);
                if (AK)
                    tma_load_2d(dst, &map_a, k0, (int)m0, &tail->rfull[slot]);
                else
                    tma_load_2d(dst, &map_a, (int)m0, k0, &tail->rfull[slot]);
                issued = st + 1;
            }
            if (*abort)  // nobody may be waiting for the last copies any more
                for (int st = max(0, issued - RAW); st < issued; ++st)
                    mbar_wait(&tail->rfull[st % RAW], (st / RAW) & 1, wait.ns);
        }
    } else if (lane == 0) {
        // ---- tma B ----
        int issued = 0;
        for (int kb = 0; kb < nkb; ++kb) {
            const int s = kb % BST;
            if (kb >= BST && !role_wait(&tail->bempty[s], ((kb / BST) - 1) & 1, abort, wait.ns)) break;
            uint8_t *dst = bst + s * Cfg::BBYTES;
            mbar_expect_tx(&tail->bfull[s], NPB * BPART);
            for (int p = 0; p < NPB; ++p)
                tma_load_2d(dst + p * BPART, &map_b, (int)(kbeg + kb * SG_BK), (int)(p * N + n0), &tail->bfull[s]);
            issued = kb + 1;
        }
        if (*abort)
            for (int kb = max(0, issued - BST); kb < issued; ++kb)
                mbar_wait(&tail->bfull[kb % BST], (kb / BST) & 1, wait.ns);
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (tid == 0 && tail->abort) atomicOr(err, 2);
    if (warp == CW + AW)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(Cfg::TCOLS) : "memory");
}

// Parts of a second operand: out[p][n][ldk], ldk = K rounded up to 8.
// K contiguous in B (row n at B + n ldb): blockDim.x along K, blockDim.y and the grid along the rows.
__global__ void k_parts_rows(const float *__restrict__ B, int64_t ldb, int64_t N, int64_t K, int64_t ldk,
                             __nv_bfloat16 *__restrict__ out) {
    for (int64_t n = (int64_t)blockIdx.x * blockDim.y + threadIdx.y; n < N; n += (int64_t)gridDim.x * blockDim.y)
        for (int64_t k = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; k < K; k += (int64_t)gridDim.y * blockDim.x) {
            __nv_bfloat16 *o = out + n * ldk + k;
            split3_one(B[n * ldb + k], o[0], o[N * ldk], o[2 * N * ldk]);
        }
}

// N contiguous in B (element (n, k) at B[row(k) ldb + n], row(k) = gather[k] or k)
__global__ void k_parts_cols(const float *__restrict__ B, int64_t ldb, const int32_t *__restrict__ gather, int64_t N,
                             int64_t K, int64_t ldk, __nv_bfloat16 *__restrict__ out) {
    __shared__ float tile[32][33];
    const int64_t k0 = (int64_t)blockIdx.x * 32;
    for (int64_t n0 = (int64_t)blockIdx.y * 32; n0 < N; n0 += (int64_t)gridDim.y * 32) {
        for (int y = threadIdx.y; y < 32; y += blockDim.y) {
            const int64_t k = k0 + y, n = n0 + threadIdx.x;
            if (k < K && n < N) tile[y][threadIdx.x] = B[(gather ? (int64_t)gather[k] : k) * ldb + n];
        }
        __syncthreads();
        for (int y = threadIdx.y; y < 32; y += blockDim.y) {
            const int64_t n = n0 + y, k = k0 + threadIdx.x;
            if (k < K && n < N) {
                __nv_bfloat16 *o = out + n * ldk + k;
                split3_one(tile[threadIdx.x][y], o[0], o[N * ldk], o[2 * N * ldk]);
            }
        }
        __syncthreads();  // the tile is free again
    }
}

template <int BN, int NPB>
void sg_launch(const SplitGemm &g, float *dst, int64_t ldm, int64_t ldn, const SplitPlan &p, int *err,
               cudaStream_t s) {
    const int64_t tiles = ceil_div(g.M, SG_BM) * ceil_div(g.N, BN);
    const dim3 grid((unsigned)tiles, (unsigned)p.splits);
    const int64_t ldk = split_parts_ld(g.K);
    CUtensorMap mb, ma;
    encode_bf16_map_ld(&mb, g.Bp, NPB * g.N, g.K, ldk, BN);
    const int avec = g.lda % 4 == 0 && ((uintptr_t)g.A & 15) == 0;  // tensor maps want 16-byte rows
    const int tma = avec && !g.gather;
    ma = mb;
    if (tma && g.a_kcontig)
        encode_f32_map(&ma, g.A, g.M, g.K, g.lda, SG_RK, SG_BM, true);
    else if (tma)
        encode_f32_map(&ma, g.A, g.K, g.M, g.lda, SG_BM, SG_RK, false);
    const auto kernel = g.a_kcontig ? k_split_gemm<BN, true, NPB> : k_split_gemm<BN, false, NPB>;
    kernel<<<grid, SgCfg<BN>::THREADS, sg_smem<BN>(), s>>>(ma, mb, g.M, g.N, g.K, g.A, g.lda, g.gather, tma, avec,
                                                           wait_switch(), dst, ldm, ldn, g.alpha, p.kb_per_split,
                                                           g.M * g.N, err);
    DSANLS_LAUNCH_CHECK();
}

int sg_bn(int64_t N) { return N <= 32 ? 32 : (N <= 64 ? 64 : 128); }

}  // namespace

int64_t split_parts_ld(int64_t K) { return ceil_div(K, 8) * 8; }

void launch_split_parts(const float *B, int64_t ldb, bool kcontig, const int32_t *gather, int64_t N, int64_t K,
                        __nv_bfloat16 *out, cudaStream_t s) {
    if (N <= 0 || K <= 0) return;
    const int64_t ldk = split_parts_ld(K);
    if (kcontig) {
        const int tx = K <= 32 ? 32 : (K <= 64 ? 64 : (K <= 128 ? 128 : 256)), ty = 256 / tx;
        const dim3 grid((unsigned)std::min<int64_t>(ceil_div(N, ty), 152 * 16),
                        (unsigned)std::min<int64_t>(ceil_div(K, tx), 64));
        k_parts_rows<<<grid, dim3(tx, ty), 0, s>>>(B, ldb, N, K, ldk, out);
    } else {
        const dim3 grid((unsigned)ceil_div(K, 32), (unsigned)std::min<int64_t>(ceil_div(N, 32), 65535));
        k_parts_cols<<<grid, dim3(32, 8), 0, s>>>(B, ldb, gather, N, K, ldk, out);
    }
    DSANLS_LAUNCH_CHECK();
}

SplitPlan split_gemm_plan(int64_t M, int64_t N, int64_t K, int max_splits) {
    const int bn = sg_bn(N);
    const int64_t tiles = ceil_div(M, SG_BM) * ceil_div(N, bn);
    const int nk = (int)ceil_div(K, SG_BK);
    // The unit is a K block of one CTA (about 0.6 us): whole waves of one CTA per SM, a CTA
    // costs about four blocks besides its own, and splits one more launch and a write and a
    // read of their partial sums (8 bytes each at HBM rate), of which at most 256 MB are kept.
    int best = 1;
    double best_t = 1e30;
    for (int sp = 1; sp <= std::min(nk, max_splits); ++sp) {
        const int kb = (int)ceil_div(nk, sp), real = (int)ceil_div(nk, kb);
        const double out = (double)sp * (double)M * (double)N;
        if (real != sp || (sp > 1 && out > 64.0e6)) continue;
        const double waves = (double)ceil_div(tiles * sp, 152);
        const double t = waves * (kb + 4.0) + (sp > 1 ? 4.0 + 8.0 * out / 4.1e6 : 0.0);
        if (t < best_t * 0.999) {
            best_t = t;
            best = sp;
        }
    }
    SplitPlan p;
    p.kb_per_split = (int)ceil_div(nk, best);
    p.splits = (int)ceil_div(nk, p.kb_per_split);
    p.part_elems = p.splits > 1 ? (int64_t)p.splits * M * N : 0;
    return p;
}

bool split_gemm_supported(int64_t M, int64_t N, int64_t K) {
    // coordinates of tensor maps (the three parts lie one below the other)
    return M < (1ll << 31) && K < (1ll << 31) && 3 * N < (1ll << 31);
}

void launch_split_gemm(const SplitGemm &g, int *err, cudaStream_t s) {
    if (g.M <= 0 || g.N <= 0) return;
    if (g.K <= 0) throw ArgError{"split GEMM: K must be >= 1"};
    if (g.gather && g.a_kcontig) throw ArgError{"split GEMM: a gather needs K rows"};
    if (!split_gemm_supported(g.M, g.N, g.K)) throw ArgError{"sizes too large"};
    const SplitPlan p = split_gemm_plan(g.M, g.N, g.K, g.max_splits);
    float *dst = p.splits > 1 ? g.part : g.C;
    // partials keep C's orientation, so the reduction below is a plain sum of slices
    const int64_t rows = g.c_trans ? g.N : g.M, cols = g.c_trans ? g.M : g.N;
    const int64_t ld = p.splits > 1 ? cols : g.ldc;
    const int64_t ldm = g.c_trans ? 1 : ld, ldn = g.c_trans ? ld : 1;
    const int bn = sg_bn(g.N);
    if (g.parts == 1) {
        if (bn == 32) sg_launch<32, 1>(g, dst, ldm, ldn, p, err, s);
        else if (bn == 64) sg_launch<64, 1>(g, dst, ldm, ldn, p, err, s);
        else sg_launch<128, 1>(g, dst, ldm, ldn, p, err, s);
    } else {
        if (bn == 32) sg_launch<32, 3>(g, dst, ldm, ldn, p, err, s);
        else if (bn == 64) sg_launch<64, 3>(g, dst, ldm, ldn, p, err, s);
        else sg_launch<128, 3>(g, dst, ldm, ldn, p, err, s);
    }
    if (p.splits > 1) launch_split_reduce(g.part, g.M * g.N, p.splits, rows, cols, cols, g.C, g.ldc, s);
}

namespace {
template <int BN, int NPB>
void prime_sg(int max_smem) {
    allow_max_dynamic_smem(k_split_gemm<BN, true, NPB>, max_smem);
    allow_max_dynamic_smem(k_split_gemm<BN, false, NPB>, max_smem);
}
}  // namespace

void prime_split_gemm_attributes(int max_smem) {
    prime_sg<32, 1>(max_smem);
    prime_sg<64, 1>(max_smem);
    prime_sg<128, 1>(max_smem);
    prime_sg<32, 3>(max_smem);
    prime_sg<64, 3>(max_smem);
    prime_sg<128, 3>(max_smem);
}


}  // namespace dsanls
