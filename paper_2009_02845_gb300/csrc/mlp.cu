// Learned warm start for the proximal row subproblem of a half-step:
//     f(x) = 1/2 x^T (G + mu I) x - (r + mu u)^T x,  x >= 0     (eq. reg_sub)
// A small MLP maps the normalised (G, b = r + mu u) to a starting point, a
// few projected-gradient steps on f correct it, and the plain projected
// gradient step of eq. gradient_descent is kept whenever its objective is
// lower (fallback).
//
// Network (k <= 32, hidden h <= 256), parameters theta in this order:
//   W1g (h x k*k), W1b (h x k), b1 (h), W2 (h x h), b2 (h), W3 (k x h), b3 (k)
//   h1 = GELU(W1g vec(Gn) + W1b bn + b1), h2 = GELU(W2 h1 + b2),
//   y  = ReLU(W3 h2 + b3)
//   Gn = (G + mu I) / s, s = tr(G + mu I) / k; bn = b / beta, beta = ||b|| / sqrt(k)
// The weights used by the forward and backward passes are the fp32 master
// weights rounded to bf16 (bf16 weights, fp32 accumulation); Adam updates the
// fp32 masters.  Prediction's products run on tensor cores at binary32 accuracy
// (gemm_split.cu: three-way bf16 splits; the weights are bf16 values, one part) but for the
// one over the k columns of bn, too short for it.
// Training's stay binary32 chains in the order of the rows (gemm_simt.cu, k_colsum): Adam
// divides by the gradient's own size and the weights are rounded to bf16 after every step,
// so a rounding difference of 1e-7 in a gradient moves the weights by 1e-5 to 1e-4 within
// 30 steps -- as far as the chain's own error, but a run would no longer repeat an earlier
// one.  (Split products took 0.31 ms per step of 8,192 rows where these take 0.56; the
// first form, one thread per column sum and 128 x 128 tiles, 6.5.)
// Everything is deterministic; GELU is the exact x Phi(x) (normcdff).
// Rows are grouped by subproblem: rows group_off[g] .. group_off[g+1]-1 share
// G_g and mu_g.
#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "common.cuh"
#include "kernels.cuh"
#include "mlp.cuh"

namespace dsanls {

namespace {

DSANLS_DEV float gelu_f(float x) { return x * normcdff(x); }
DSANLS_DEV float gelu_grad_f(float x) { return normcdff(x) + x * 0.3989422804014327f * __expf(-0.5f * x * x); }

// A weight matrix (rows x cols at `off` of the parameters) as the second operand of
// prediction's products: bf16 rows of split_parts_ld(cols).
struct WeightParts {
    int64_t off;
    int rows, cols;
    __nv_bfloat16 *n;
};

DSANLS_DEV void put_parts(const WeightParts &w, int64_t i, __nv_bfloat16 q) {
    const int64_t e = i - w.off;
    if (e < 0 || e >= (int64_t)w.rows * w.cols) return;
    const int64_t r = e / w.cols, c = e - r * w.cols;
    w.n[r * ((w.cols + 7) / 8 * 8) + c] = q;
}

// wq = theta rounded to bf16, and the weights' operand copies.  With lr > 0 one Adam step
// on theta first (the step and the rounding share one pass over the parameters).
__global__ void k_adam_round(float *__restrict__ theta, float *__restrict__ m, float *__restrict__ v,
                             const float *__restrict__ g, int64_t n, float lr, float b1, float b2, float c1, float c2,
                             float eps, float *__restrict__ wq, WeightParts w0, WeightParts w1, WeightParts w2) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float x = theta[i];
    if (lr > 0.0f) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        x -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        theta[i] = x;
    }
    const __nv_bfloat16 q = __float2bfloat16_rn(x);
    wq[i] = __bfloat162float(q);
    put_parts(w0, i, q);
    put_parts(w1, i, q);
    put_parts(w2, i, q);
}

// per group: s_g and Gn_g; the first kernel of a pass clears the word that the pass's products raise
__global__ void k_norm_groups(const float *__restrict__ G, const float *__restrict__ mu, int k, int ngroups,
                              float *__restrict__ Gn, float *__restrict__ s_out, int *__restrict__ clear) {
    const int g = blockIdx.x;
    if (clear && g == 0 && threadIdx.x == 0) *clear = 0;
    if (g >= ngroups) return;
    __shared__ float s_sh;
    const float *Gg = G + (int64_t)g * k * k;
    if (threadIdx.x == 0) {
        float tr = 0.0f;
        for (int i = 0; i < k; ++i) tr += Gg[i * k + i];
        s_sh = (tr + k * mu[g]) / k;
        s_out[g] = s_sh;
    }
    __syncthreads();
    const float inv = 1.0f / s_sh;
    for (int e = threadIdx.x; e < k * k; e += blockDim.x) {
        const int i = e / k, j = e % k;
        Gn[(int64_t)g * k * k + e] = (Gg[e] + (i == j ? mu[g] : 0.0f)) * inv;
    }
}

// the subproblem of row r, from group_off
DSANLS_DEV int group_of(const int64_t *off, int ngroups, int64_t r) {
    int lo = 0, hi = ngroups;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= r)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

// W lanes per row, one per column (k <= W <= 32); the sum of squares in column order.  (A whole
// warp for a row of 8 took 29 us for 57,556 rows, one thread 8.)
template <int W>
__global__ void __launch_bounds__(256) k_norm_rows(const float *__restrict__ b, int64_t rows, int k,
                                                   float *__restrict__ bn, float *__restrict__ beta) {
    const int lane = threadIdx.x % W;
    const int64_t r = (int64_t)blockIdx.x * (256 / W) + threadIdx.x / W;
    const float x = r < rows && lane < k ? b[r * k + lane] : 0.0f;
    float ss = 0.0f;
#pragma unroll
    for (int j = 0; j < W; ++j) {
        const float y = __shfl_sync(0xffffffffu, x, j, W);
        ss = fmaf(y, y, ss);  // (zeros past k)
    }
    if (r >= rows) return;
    float bt = sqrtf(ss / k);
    if (!(bt > 0.0f)) bt = 1.0f;
    if (lane == 0) beta[r] = bt;
    const float inv = 1.0f / bt;
    if (lane < k) bn[r * k + lane] = x * inv;
}

// The activations: a CTA takes ACT_ROWS rows, threads the columns, so no element divides
// for its row and column and a row's group is looked up once.
constexpr int ACT_ROWS = 4;

// z1 += zg[group] + b1 (in place), h1 = GELU(z1)
__global__ void __launch_bounds__(256)
    k_layer1_finish(float *__restrict__ z1, float *__restrict__ h1, const float *__restrict__ zg,
                    const float *__restrict__ b1, const int64_t *__restrict__ off, int ngroups, int64_t rows, int h) {
    __shared__ int grp[ACT_ROWS];
    const int64_t r0 = (int64_t)blockIdx.x * ACT_ROWS;
    if (threadIdx.x < ACT_ROWS) grp[threadIdx.x] = group_of(off, ngroups, min(rows - 1, r0 + threadIdx.x));
    __syncthreads();
    for (int j = threadIdx.x; j < h; j += blockDim.x) {
        const float bj = b1[j];
#pragma unroll
        for (int i = 0; i < ACT_ROWS; ++i) {
            if (r0 + i >= rows) break;
            const int64_t idx = (r0 + i) * h + j;
            const float z = z1[idx] + zg[(int64_t)grp[i] * h + j] + bj;
            z1[idx] = z;
            h1[idx] = gelu_f(z);
        }
    }
}

// z += bias (per column), act = GELU(z) or ReLU(z)
__global__ void __launch_bounds__(256)
    k_bias_act(float *__restrict__ z, float *__restrict__ act, const float *__restrict__ bias, int64_t rows, int cols,
               int relu) {
    const int64_t r0 = (int64_t)blockIdx.x * ACT_ROWS * blockDim.y + threadIdx.y * ACT_ROWS;
    for (int j = threadIdx.x; j < cols; j += blockDim.x) {
        const float bj = bias[j];
#pragma unroll
        for (int i = 0; i < ACT_ROWS; ++i) {
            if (r0 + i >= rows) break;
            const int64_t idx = (r0 + i) * cols + j;
            const float v = z[idx] + bj;
            z[idx] = v;
            act[idx] = relu ? fmaxf(v, 0.0f) : gelu_f(v);
        }
    }
}

// The loss of a row against y* = x* s_g / beta_r: e = o - y* where y* > 0, max(o, 0)
// where y* = 0 (o before the ReLU); do = e / N; 1/2 ||e||^2 to rowloss.  Equal to the squared
// error of the ReLU output except where o < 0 < y*, where it keeps a gradient.  One warp
// per row, one lane per column (k <= 32).
__global__ void __launch_bounds__(256)
    k_out_grad(const float *__restrict__ o, const float *__restrict__ xstar, const float *__restrict__ s_g,
               const float *__restrict__ beta, const int64_t *__restrict__ off, int ngroups, int64_t rows, int k,
               float invN, float *__restrict__ dout, double *__restrict__ rowloss) {
    const int lane = threadIdx.x & 31;
    const int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (r >= rows) return;
    double l = 0.0;
    if (lane < k) {
        const float oj = o[r * k + lane], t = xstar[r * k + lane] * s_g[group_of(off, ngroups, r)] / beta[r];
        const float e = t > 0.0f ? oj - t : fmaxf(oj, 0.0f);
        l = 0.5 * (double)e * (double)e;
        dout[r * k + lane] = e * invN;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) l += __shfl_xor_sync(0xffffffffu, l, d);
    if (lane == 0) rowloss[r] = l;
}

// dh *= GELU'(z) in place (the backward pass through the activation)
__global__ void __launch_bounds__(256) k_gelu_back(const float *__restrict__ z, float *__restrict__ dh, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dh[i] *= gelu_grad_f(z[i]);
}

// out[g * cols + j] = sum over rows off[g] <= r < off[g+1] of X[r * cols + j], one chain per
// column in row order (off null: one segment of all rows).  A CTA takes 32 columns of a
// segment: seven warps copy tiles of CS_ROWS rows ahead by cp.async, the first one adds.
// Bound by the chain, four cycles per row (a thread that loaded each row itself took 1 ms
// for 8,192 rows).
constexpr int CS_ROWS = 112, CS_STAGES = 3;
__global__ void __launch_bounds__(256) k_colsum(const float *__restrict__ X, const int64_t *__restrict__ off,
                                                int64_t rows, int cols, float *__restrict__ out) {
    __shared__ float tile[CS_STAGES][CS_ROWS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, ctiles = (cols + 31) / 32;
    const int64_t g = blockIdx.x / ctiles;
    const int j = (int)(blockIdx.x % ctiles) * 32 + lane;
    const int64_t r0 = off ? off[g] : 0, r1 = off ? off[g + 1] : rows;
    const int64_t nt = r1 > r0 ? (r1 - r0 + CS_ROWS - 1) / CS_ROWS : 0;
    auto fetch = [&](int64_t t) {
        if (w == 0) return;
#pragma unroll
        for (int i = 0; i < CS_ROWS / 7; ++i) {
            const int q = w - 1 + 7 * i;
            const int64_t r = r0 + t * CS_ROWS + q;
            const bool in = t < nt && r < r1 && j < cols;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                             (uint32_t)__cvta_generic_to_shared(&tile[t % CS_STAGES][q][lane])),
                         "l"(in ? X + r * cols + j : X), "r"(in ? 4 : 0)
                         : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int t = 0; t < CS_STAGES - 1; ++t) fetch(t);
    float acc = 0.0f;
    for (int64_t t = 0; t < nt; ++t) {
        asm volatile("cp.async.wait_group %0;" ::"n"(CS_STAGES - 2) : "memory");
        __syncthreads();  // tile t has landed, tile t - 1 has been added
        fetch(t + CS_STAGES - 1);
        if (w == 0) {
            const float(*x)[32] = tile[t % CS_STAGES];
            const int n = (int)min((int64_t)CS_ROWS, r1 - r0 - t * CS_ROWS);
            if (n == CS_ROWS) {
#pragma unroll
                for (int q = 0; q < CS_ROWS; q += 16) {
                    float v[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) v[e] = x[q + e][lane];
#pragma unroll
                    for (int e = 0; e < 16; ++e) acc = __fadd_rn(acc, v[e]);
                }
            } else {
                for (int r = 0; r < n; ++r) acc = __fadd_rn(acc, x[r][lane]);
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (w == 0 && j < cols) out[g * cols + j] = acc;
}

__global__ void __launch_bounds__(1024) k_sum_doubles(const double *__restrict__ x, int64_t n, double scale,
                                                      double *__restrict__ out) {
    __shared__ double red[32];
    double v = 0.0;
#pragma unroll 8
    for (int64_t i = threadIdx.x; i < n; i += 1024) v += x[i];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        v = red[threadIdx.x];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (threadIdx.x == 0) *out = v * scale;
    }
}

__global__ void k_g_to_float(const double *__restrict__ G64, int k, const double *__restrict__ scal,
                             float *__restrict__ gf, float *__restrict__ mu, int64_t *__restrict__ off, int64_t rows) {
    for (int e = threadIdx.x; e < k * k; e += blockDim.x) gf[e] = (float)G64[e];
    if (threadIdx.x == 0) {
        mu[0] = (float)scal[1];
        off[0] = 0;
        off[1] = rows;
    }
}

__global__ void k_rhs_b(const float *__restrict__ R, const float *__restrict__ Z, const double *__restrict__ scal,
                        int64_t n, float *__restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = __fmaf_rn((float)scal[1], Z[i], R[i]);
}

unsigned nblk(int64_t n) { return (unsigned)ceil_div(n, 256); }

// C (M x N) = A W^T at binary32 accuracy on tensor cores, W's bf16 rows as parts (no split
// of K: C holds as many rows as the batch)
void times_weights(int64_t M, int64_t N, int64_t K, const float *A, const __nv_bfloat16 *W, float *C, int *err,
                   cudaStream_t s) {
    launch_split_gemm(SplitGemm{M, N, K, A, K, true, nullptr, W, 1, C, N, false, 1.0f, nullptr, 1}, err, s);
}

// one binary32 chain per output
void chain(int64_t M, int64_t N, int64_t K, const float *A, int64_t lda, bool ak, const float *B, int64_t ldb, bool bk,
           float *C, int64_t ldc, cudaStream_t s) {
    launch_sgemm(GemmArgs{M, N, K, A, lda, nullptr, ak, B, ldb, nullptr, bk, C, ldc, 1.0f, 1, 0}, s);
}

void column_sums(const float *X, const int64_t *off, int nseg, int64_t rows, int cols, float *out, cudaStream_t s) {
    k_colsum<<<(unsigned)(ceil_div(cols, 32) * nseg), 256, 0, s>>>(X, off, rows, cols, out);
    DSANLS_LAUNCH_CHECK();
}

// The Gram layer's product: most slices of its K, for batches of at most so many subproblems
constexpr int MLP_MAX_SPLITS = 64, MLP_SPLIT_GROUPS = 19456;

}  // namespace

int64_t mlp_param_count(int k, int h) { return (int64_t)h * k * k + (int64_t)h * k + h + (int64_t)h * h + h + (int64_t)k * h + k; }

MlpOffsets mlp_offsets(int k, int h) {
    MlpOffsets o;
    o.W1g = 0;
    o.W1b = o.W1g + (int64_t)h * k * k;
    o.b1 = o.W1b + (int64_t)h * k;
    o.W2 = o.b1 + h;
    o.b2 = o.W2 + (int64_t)h * h;
    o.W3 = o.b2 + h;
    o.b3 = o.W3 + (int64_t)k * h;
    o.total = o.b3 + k;
    return o;
}

void mlp_alloc(MlpState &st, int k, int h, int64_t max_rows, int max_groups) {
    st.k = k;
    st.h = h;
    st.max_rows = max_rows;
    st.max_groups = max_groups;
    const int64_t P = mlp_param_count(k, h);
    auto al = [](auto *&p, int64_t n) {
        if (cudaMalloc((void **)&p, (size_t)std::max<int64_t>(n, 1) * sizeof(*p)) != cudaSuccess) {
            cudaGetLastError();
            throw std::bad_alloc();
        }
    };
    al(st.theta, P); al(st.wq, P); al(st.grad, P); al(st.m, P); al(st.v, P);
    al(st.Gn, (int64_t)max_groups * k * k); al(st.s, max_groups); al(st.zg, (int64_t)max_groups * h);
    al(st.dzg, (int64_t)max_groups * h);
    al(st.bn, max_rows * k); al(st.beta, max_rows);
    al(st.z1, max_rows * h); al(st.h1, max_rows * h); al(st.z2, max_rows * h); al(st.h2, max_rows * h);
    al(st.o, max_rows * k); al(st.y, max_rows * k); al(st.dout, max_rows * k); al(st.rowloss, max_rows);
    al(st.loss, 2);  // the loss, then the error words
    st.err = reinterpret_cast<int *>(st.loss + 1);
    al(st.gf1, (int64_t)k * k); al(st.mu1, 1); al(st.off1, 2);
    al(st.W1g, h * split_parts_ld((int64_t)k * k)); al(st.W2, h * split_parts_ld(h));
    al(st.W3, k * split_parts_ld(h));
    // split-K partials of the Gram layer: the most that its plan takes for any number of groups
    // (at most 10 MB: from 9,728 groups on it does not split)
    int64_t most = 0;
    for (int64_t g = 1; g <= std::min<int64_t>(max_groups, MLP_SPLIT_GROUPS); ++g)
        most = std::max(most, split_gemm_plan(g, h, (int64_t)k * k, MLP_MAX_SPLITS).part_elems);
    al(st.part, most);
    DSANLS_CUDA(cudaMemset(st.loss, 0, 2 * sizeof(double)));
    DSANLS_CUDA(cudaMemset(st.m, 0, P * sizeof(float)));
    DSANLS_CUDA(cudaMemset(st.v, 0, P * sizeof(float)));
}

void mlp_reserve_training(MlpState &st) {
    if (!st.dz2 && cudaMalloc((void **)&st.dz2, (size_t)(st.max_rows * st.h) * sizeof(float)) != cudaSuccess) {
        cudaGetLastError();
        st.dz2 = nullptr;
        throw std::bad_alloc();
    }
    for (cudaStream_t &t : st.side)
        if (!t) DSANLS_CUDA(cudaStreamCreateWithFlags(&t, cudaStreamNonBlocking));
    for (cudaEvent_t *e : {&st.ev[0], &st.ev[1], &st.ev[2], &st.done[0], &st.done[1], &st.done[2]})
        if (!*e) DSANLS_CUDA(cudaEventCreateWithFlags(e, cudaEventDisableTiming));
}

void mlp_free(MlpState &st) {
    for (void *p : {(void *)st.theta, (void *)st.wq, (void *)st.grad, (void *)st.m, (void *)st.v, (void *)st.Gn,
                    (void *)st.s, (void *)st.zg, (void *)st.dzg, (void *)st.bn, (void *)st.beta, (void *)st.z1,
                    (void *)st.h1, (void *)st.z2, (void *)st.h2, (void *)st.o, (void *)st.y, (void *)st.dout,
                    (void *)st.rowloss, (void *)st.loss, (void *)st.gf1, (void *)st.mu1, (void *)st.off1,
                    (void *)st.W1g, (void *)st.W2, (void *)st.W3, (void *)st.part,
                    (void *)st.dz2})
        if (p) cudaFree(p);
    for (cudaStream_t t : st.side)
        if (t) cudaStreamDestroy(t);
    for (cudaEvent_t e : {st.ev[0], st.ev[1], st.ev[2], st.done[0], st.done[1], st.done[2]})
        if (e) cudaEventDestroy(e);
    st = MlpState{};
}

// Adam step (lr > 0) and the rounded weights
static void adam_round(MlpState &st, float lr, cudaStream_t s) {
    const int k = st.k, h = st.h;
    const MlpOffsets O = mlp_offsets(k, h);
    float c1 = 1.0f, c2 = 1.0f;
    const float b1 = 0.9f, b2 = 0.999f;
    if (lr > 0.0f) {
        st.adam_t += 1;
        c1 = 1.0f - std::pow(b1, (float)st.adam_t);
        c2 = 1.0f - std::pow(b2, (float)st.adam_t);
    }
    k_adam_round<<<nblk(O.total), 256, 0, s>>>(st.theta, st.m, st.v, st.grad, O.total, lr, b1, b2, c1, c2, 1e-8f, st.wq,
                                               WeightParts{O.W1g, h, k * k, st.W1g},
                                               WeightParts{O.W2, h, h, st.W2},
                                               WeightParts{O.W3, k, h, st.W3});
    DSANLS_LAUNCH_CHECK();
}

void mlp_quantise(MlpState &st, cudaStream_t s) { adam_round(st, 0.0f, s); }
void mlp_adam(MlpState &st, float lr, cudaStream_t s) { adam_round(st, lr, s); }

static void bias_act(float *z, float *act, const float *bias, int64_t rows, int cols, int relu, cudaStream_t s) {
    const unsigned tx = (unsigned)std::min(256, (cols + 31) / 32 * 32), ty = 256 / tx;
    k_bias_act<<<(unsigned)ceil_div(rows, ACT_ROWS * ty), dim3(tx, ty), 0, s>>>(z, act, bias, rows, cols, relu);
    DSANLS_LAUNCH_CHECK();
}

// Forward pass: y (rows x k, normalised output) in st.y; o, z1, h1, z2, h2 kept.
void mlp_forward(MlpState &st, const float *G, const float *mu, const int64_t *off, int ngroups, const float *b,
                 int64_t rows, bool training, int *err, cudaStream_t s) {
    const int k = st.k, h = st.h;
    const int64_t kk = (int64_t)k * k;
    const MlpOffsets O = mlp_offsets(k, h);
    const float *W = st.wq;
    k_norm_groups<<<ngroups, 128, 0, s>>>(G, mu, k, ngroups, st.Gn, st.s, err == st.err ? err : nullptr);
    DSANLS_LAUNCH_CHECK();
    if (training)
        chain(ngroups, h, kk, st.Gn, kk, true, W + O.W1g, kk, true, st.zg, h, s);
    else
        launch_split_gemm(SplitGemm{ngroups, h, kk, st.Gn, kk, true, nullptr, st.W1g, 1, st.zg, h, false, 1.0f, st.part,
                                    ngroups <= MLP_SPLIT_GROUPS ? MLP_MAX_SPLITS : 1},
                          err, s);
    if (k <= 8)
        k_norm_rows<8><<<(unsigned)ceil_div(rows, 32), 256, 0, s>>>(b, rows, k, st.bn, st.beta);
    else if (k <= 16)
        k_norm_rows<16><<<(unsigned)ceil_div(rows, 16), 256, 0, s>>>(b, rows, k, st.bn, st.beta);
    else
        k_norm_rows<32><<<(unsigned)ceil_div(rows, 8), 256, 0, s>>>(b, rows, k, st.bn, st.beta);
    DSANLS_LAUNCH_CHECK();
    // (K = k <= 32: the CTAs of the split product have a block or two each; 57,556 x 64 from 8
    // 52 us there, 20 here, and 1,000 .. 57,556 x 256 from 32 the same)
    chain(rows, h, k, st.bn, k, true, W + O.W1b, k, true, st.z1, h, s);
    k_layer1_finish<<<(unsigned)ceil_div(rows, ACT_ROWS), (unsigned)std::min(256, (h + 31) / 32 * 32), 0, s>>>(
        st.z1, st.h1, st.zg, W + O.b1, off, ngroups, rows, h);
    DSANLS_LAUNCH_CHECK();
    if (training)
        chain(rows, h, h, st.h1, h, true, W + O.W2, h, true, st.z2, h, s);
    else
        times_weights(rows, h, h, st.h1, st.W2, st.z2, err, s);
    bias_act(st.z2, st.h2, W + O.b2, rows, h, 0, s);
    if (training)
        chain(rows, k, h, st.h2, h, true, W + O.W3, h, true, st.o, k, s);
    else
        times_weights(rows, k, h, st.h2, st.W3, st.o, err, s);
    bias_act(st.o, st.y, W + O.b3, rows, k, 1, s);
}

// Loss and gradient (into st.grad) of the one-sided squared error (k_out_grad) after mlp_forward.
void mlp_backward(MlpState &st, const int64_t *off, int ngroups, const float *xstar, int64_t rows, cudaStream_t s) {
    const int k = st.k, h = st.h;
    const int64_t kk = (int64_t)k * k;
    const MlpOffsets O = mlp_offsets(k, h);
    const float *W = st.wq;
    float *dG = st.grad;
    k_out_grad<<<(unsigned)ceil_div(rows, 8), 256, 0, s>>>(st.o, xstar, st.s, st.beta, off, ngroups, rows, k,
                                                          1.0f / (float)rows, st.dout, st.rowloss);
    DSANLS_LAUNCH_CHECK();
    k_sum_doubles<<<1, 1024, 0, s>>>(st.rowloss, rows, 1.0 / (double)rows, st.loss);  // mean over rows
    DSANLS_LAUNCH_CHECK();
    const unsigned eb = (unsigned)std::min<int64_t>(ceil_div(rows * h, 256), 152 * 16);
    // The weight gradients and the column sums are long chains on few SMs: they run beside the
    // path to the lower layer on the side streams (0: dW3, 1: the column sums, 2: dW2), each
    // from the event after its input, and join it at the end.  That path writes buffers whose
    // last reader is behind it: dz2 has its own, dz1 takes z2's.
    auto fork = [&](int e) { DSANLS_CUDA(cudaEventRecord(st.ev[e], s)); };
    auto after = [&](int t, int e) { DSANLS_CUDA(cudaStreamWaitEvent(st.side[t], st.ev[e], 0)); };
    fork(0);  // do
    after(0, 0);
    chain(k, h, rows, st.dout, k, false, st.h2, h, false, dG + O.W3, h, st.side[0]);  // dW3 = do^T h2
    after(1, 0);
    column_sums(st.dout, nullptr, 1, rows, k, dG + O.b3, st.side[1]);
    chain(rows, h, k, st.dout, k, true, W + O.W3, h, false, st.dz2, h, s);  // dh2 = do W3 -> dz2
    k_gelu_back<<<eb, 256, 0, s>>>(st.z2, st.dz2, rows * h);
    DSANLS_LAUNCH_CHECK();
    fork(1);  // dz2
    after(2, 1);
    chain(h, h, rows, st.dz2, h, false, st.h1, h, false, dG + O.W2, h, st.side[2]);  // dW2 = dz2^T h1
    after(1, 1);
    column_sums(st.dz2, nullptr, 1, rows, h, dG + O.b2, st.side[1]);
    float *dz1 = st.z2;
    chain(rows, h, h, st.dz2, h, true, W + O.W2, h, false, dz1, h, s);  // dh1 = dz2 W2 -> dz1
    k_gelu_back<<<eb, 256, 0, s>>>(st.z1, dz1, rows * h);
    DSANLS_LAUNCH_CHECK();
    fork(2);  // dz1
    after(1, 2);
    column_sums(dz1, nullptr, 1, rows, h, dG + O.b1, st.side[1]);
    // per-group dzg and dW1g = dzg^T Gn, dW1b = dz1^T bn
    column_sums(dz1, off, ngroups, rows, h, st.dzg, s);
    chain(h, kk, ngroups, st.dzg, h, false, st.Gn, kk, false, dG + O.W1g, kk, s);
    chain(h, k, rows, dz1, h, false, st.bn, k, false, dG + O.W1b, k, s);
    for (int t = 0; t < 3; ++t) {
        DSANLS_CUDA(cudaEventRecord(st.done[t], st.side[t]));
        DSANLS_CUDA(cudaStreamWaitEvent(s, st.done[t], 0));
    }
}

__global__ void k_init_segment(float *__restrict__ theta, int64_t off, int64_t n, float a) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) theta[off + i] = a * (2.0f * theta[off + i] - 1.0f);
}

void mlp_init(MlpState &st, uint64_t seed, cudaStream_t s) {
    const int k = st.k, h = st.h;
    const MlpOffsets O = mlp_offsets(k, h);
    launch_uniform_field(seed, 0x20, 0, O.total, 1, st.theta, s);
    struct Seg {
        int64_t off, n;
        float fan_in;
    };
    const Seg segs[7] = {{O.W1g, (int64_t)h * k * k, (float)(k * k + k)}, {O.W1b, (int64_t)h * k, (float)(k * k + k)},
                         {O.b1, h, 0.0f}, {O.W2, (int64_t)h * h, (float)h}, {O.b2, h, 0.0f},
                         {O.W3, (int64_t)k * h, (float)h}, {O.b3, k, 0.0f}};
    for (const Seg &g : segs) {
        const float a = g.fan_in > 0.0f ? std::sqrt(3.0f / g.fan_in) : 0.0f;
        k_init_segment<<<nblk(g.n), 256, 0, s>>>(st.theta, g.off, g.n, a);
        DSANLS_LAUNCH_CHECK();
    }
    mlp_quantise(st, s);
}

__global__ void k_unscale(const float *__restrict__ y, const float *__restrict__ s_g, const float *__restrict__ beta,
                          const int64_t *__restrict__ off, int ngroups, int64_t rows, int k, int *__restrict__ err,
                          float *__restrict__ x) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= rows * k) return;
    const int64_t r = idx / k;
    // a product gave up: no number that could pass for a prediction, and the handle is told
    const bool failed = err[0] != 0;
    if (failed && idx == 0) err[1] = 1;
    x[idx] = failed ? __int_as_float(0x7fc00000) : y[idx] * beta[r] / s_g[group_of(off, ngroups, r)];
}

void mlp_unscale(MlpState &st, const int64_t *off, int ngroups, int64_t rows, float *x_out, cudaStream_t s) {
    k_unscale<<<nblk(rows * st.k), 256, 0, s>>>(st.y, st.s, st.beta, off, ngroups, rows, st.k, st.err, x_out);
    DSANLS_LAUNCH_CHECK();
}

// ---------------------------------------------------------------------------
// learned update of one half-step (k <= 32): one warp per row, lane c owns
// column c of the row; (x G)_c = sum_l x_l G[l][c] with x_l broadcast from
// lane l (an FMA chain in increasing l)
// ---------------------------------------------------------------------------
constexpr int LF_THREADS = 256;

DSANLS_DEV float row_times_g(float x, float init, const float (*gs)[33], int lane) {
    float acc = init;
#pragma unroll
    for (int l = 0; l < 32; ++l) acc = __fmaf_rn(__shfl_sync(0xffffffffu, x, l), gs[l][lane], acc);
    return acc;
}

DSANLS_DEV float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__global__ void __launch_bounds__(LF_THREADS)
    k_learned_finish(float *__restrict__ Z, const float *__restrict__ R, const float *__restrict__ y,
                     const float *__restrict__ beta, const float *__restrict__ s_g, const float *__restrict__ Gf,
                     int kp, const double *__restrict__ scal, int64_t rows, int k, int pg_iters, int plain_iters,
                     unsigned long long *__restrict__ kept, int *__restrict__ flag) {
    __shared__ float gs[32][33];
    for (int e = threadIdx.x; e < 32 * 32; e += blockDim.x) {
        const int a = e / 32, c = e % 32;
        gs[a][c] = (a < k && c < k) ? Gf[a * kp + c] : 0.0f;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const bool on = lane < k;
    const float mu = (float)scal[1], eta = (float)scal[2];
    const float inv_s = 1.0f / s_g[0];
    unsigned long long nkept = 0;
    const int64_t nwarps = (int64_t)gridDim.x * (LF_THREADS / 32);
    for (int64_t r = (int64_t)blockIdx.x * (LF_THREADS / 32) + (threadIdx.x >> 5); r < rows; r += nwarps) {
        const float u = on ? Z[r * k + lane] : 0.0f;
        const float rc = on ? R[r * k + lane] : 0.0f;
        const float bb = __fmaf_rn(mu, u, rc);
        float x = on ? y[r * k + lane] * (beta[r] * inv_s) : 0.0f;
        // the plain path's update from u: one step of eq. gradient_descent, or
        // plain_iters steps on f from u
        float xp;
        if (plain_iters <= 1) {
            const float v = __fmaf_rn(-eta, row_times_g(u, 0.0f, gs, lane) - rc, u);
            xp = (on && v > 0.0f) ? v : 0.0f;
        } else {
            xp = u;
            for (int it = 0; it < plain_iters; ++it) {
                const float v = __fmaf_rn(-eta, row_times_g(xp, mu * xp, gs, lane) - bb, xp);
                xp = (on && v > 0.0f) ? v : 0.0f;
            }
        }
        // correction: pg_iters projected-gradient steps on f from the network's point
        for (int it = 0; it < pg_iters; ++it) {
            const float v = __fmaf_rn(-eta, row_times_g(x, mu * x, gs, lane) - bb, x);
            x = (on && v > 0.0f) ? v : 0.0f;
        }
        // objectives f(x) = 1/2 x^T (G + mu I) x - b^T x
        const float fx = warp_sum(x * (0.5f * row_times_g(x, mu * x, gs, lane) - bb));
        const float fp = warp_sum(xp * (0.5f * row_times_g(xp, mu * xp, gs, lane) - bb));
        const bool use_mlp = fx <= fp;
        nkept += use_mlp ? 1 : 0;
        float v = use_mlp ? x : xp;
        if (!(fabsf(v) <= 3.402823466e38f)) {
            *flag = 1;
            v = 0.0f;
        }
        if (on) Z[r * k + lane] = v;
    }
    if (lane == 0 && nkept) atomicAdd(kept, nkept);
}

void mlp_learned_update(MlpState &st, float *Z, const float *R, int64_t rows, const double *G64, const float *Gf,
                        int kp, const double *scal, int pg_iters, int plain_iters, unsigned long long *kept, int *flag,
                        cudaStream_t s) {
    const int k = st.k;
    // one group: G (fp32) and mu from the half-step
    k_g_to_float<<<1, 256, 0, s>>>(G64, k, scal, st.gf1, st.mu1, st.off1, rows);
    DSANLS_LAUNCH_CHECK();
    // b = R + mu Z into st.dout (rows x k) for the network input
    k_rhs_b<<<nblk(rows * k), 256, 0, s>>>(R, Z, scal, rows * k, st.dout);
    DSANLS_LAUNCH_CHECK();
    mlp_forward(st, st.gf1, st.mu1, st.off1, 1, st.dout, rows, false, flag, s);
    const int64_t blocks = std::min<int64_t>(ceil_div(rows, LF_THREADS / 32), 152 * 8);
    k_learned_finish<<<(unsigned)blocks, LF_THREADS, 0, s>>>(Z, R, st.y, st.beta, st.s, Gf, kp, scal, rows, k,
                                                            pg_iters, plain_iters, kept, flag);
    DSANLS_LAUNCH_CHECK();
}

// ---------------------------------------------------------------------------
// harvesting training triples: exact proximal minimiser by FISTA (Beck and
// Teboulle 2009), one warp per row as above
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(LF_THREADS)
    k_harvest(const float *__restrict__ Z, const float *__restrict__ R, const float *__restrict__ Gf, int kp,
              const double *__restrict__ scal, int64_t rows, int k, int iters, float *__restrict__ b_out,
              float *__restrict__ x_out) {
    __shared__ float gs[32][33];
    for (int e = threadIdx.x; e < 32 * 32; e += blockDim.x) {
        const int a = e / 32, c = e % 32;
        gs[a][c] = (a < k && c < k) ? Gf[a * kp + c] : 0.0f;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const bool on = lane < k;
    const float mu = (float)scal[1];
    const float step = (float)(1.0 / (scal[0] * 1.0001 + scal[1]));  // 1 / (lambda_max(G) + mu)
    const int64_t nwarps = (int64_t)gridDim.x * (LF_THREADS / 32);
    for (int64_t r = (int64_t)blockIdx.x * (LF_THREADS / 32) + (threadIdx.x >> 5); r < rows; r += nwarps) {
        const float u = on ? Z[r * k + lane] : 0.0f;
        const float bb = on ? __fmaf_rn(mu, u, R[r * k + lane]) : 0.0f;
        if (on) b_out[r * k + lane] = bb;
        float x = u, yv = u, tk = 1.0f;
        for (int it = 0; it < iters; ++it) {
            const float v = yv - step * (row_times_g(yv, mu * yv, gs, lane) - bb);
            const float nx = (on && v > 0.0f) ? v : 0.0f;
            const float tn = 0.5f * (1.0f + sqrtf(1.0f + 4.0f * tk * tk));
            const float w = (tk - 1.0f) / tn;
            yv = nx + w * (nx - x);
            x = nx;
            tk = tn;
        }
        if (on) x_out[r * k + lane] = x;
    }
}

void mlp_harvest(const float *Z, const float *R, const float *Gf, int kp, const double *scal, int64_t rows, int k,
                 int iters, float *b_out, float *x_out, cudaStream_t s) {
    const int64_t blocks = std::min<int64_t>(ceil_div(rows, LF_THREADS / 32), 152 * 8);
    k_harvest<<<(unsigned)blocks, LF_THREADS, 0, s>>>(Z, R, Gf, kp, scal, rows, k, iters, b_out, x_out);
    DSANLS_LAUNCH_CHECK();
}

}  // namespace dsanls
