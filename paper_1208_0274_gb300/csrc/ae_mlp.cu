// Search-work predictor: query features, a 66-128-128-2 perceptron with its
// forward and backward passes on the bf16 tensor cores, and Adam training.
// The C ABI is declared in include/ae_mlp.h.  Nothing here changes a search
// result; the engine only reads the predictions as buffer-size hints.

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <vector>

#include "ae_device.cuh"
#include "ae_internal.h"
#include "ae_kernels.h"
#include "ae_mlp.h"

namespace {

constexpr int NIN = AE_MLP_IN, NH = AE_MLP_HIDDEN, NOUT = AE_MLP_OUT;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NH * NIN, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH,
              OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NOUT * NH, NPARAM = OFF_B3 + NOUT;
static_assert(NPARAM == AE_MLP_PARAMS, "packed parameter count");

// norm buffer: x_mu[66] | x_isd[66] | y_mu[2] | y_sd[2]
constexpr int NORM_XMU = 0, NORM_XISD = NIN, NORM_YMU = 2 * NIN, NORM_YSD = 2 * NIN + NOUT,
              NORM_SIZE = 2 * NIN + 2 * NOUT;

// ------------------------------------------------------------------ tensor-core GEMM
//
// C(m, n) = sum_k A(m, k) B(k, n) with A(m, k) = A[m*sam + k*sak] and
// B(k, n) = B[k*sbk + n*sbn] (fp32 in memory, rounded to bf16 for the
// product, fp32 accumulate).  Epilogue per element: + bias[n]; Z = that value
// (pre-activation); zeroed where mask <= 0; relu; stored to C (ld ldc).  One
// warp owns a 16 x 16 tile (two m16n8k16 products per k step of 16), or 16 x 32 where
// there are many rows.
//
// Split K: the weight gradients are products with a small output (at most
// 128 x 128) and K = the batch rows, which a few warps would walk alone.  With
// `part` set, gemm() splits K into up to GEMM_KSPLIT_MAX chunks, each block
// stores its raw partial tile to part[s][M][N], and k_gemm_reduce sums the chunks
// in chunk order and applies the epilogue, so the result does not depend on
// scheduling.
//
// A training step of 64 rows is a chain of small products, each bound by the
// latency of its loads and its launch.  So a warp loads four k steps' operands
// together, its tile is small (more warps), and products that wait for the same
// input share a launch (two GemmArgs), 10 launches a step instead of 15 (13 at 128
// rows, whose weight gradients split their sums): 82 us a step with one k step in
// flight and 16 x 32 tiles, 59 us so.

struct GemmArgs {
    const float *A;
    int64_t sam, sak;
    const float *B;
    int64_t sbk, sbn;
    float *C;
    int64_t ldc;
    const float *bias;
    const float *mask;
    float *Z;
    int M, N, K, relu;
    float *part;        // split-K partials (GEMM_KSPLIT_MAX * M * N floats), or null
    int kchunk;         // K per chunk (a multiple of 16), chunks, blocks per chunk; set by plan()
    int nsplit, blocks;
};
struct GemmPair {
    GemmArgs a[2];
};

// NT: n8 sub-tiles per warp, KU: k steps whose operands are loaded together.  From
// GEMM_WIDE tiles of 16 x 16 on (8,192 rows by 128 columns) there are warps enough to
// hide the loads and the operands' traffic counts: a warp then takes 16 x 32, one k step
// at a time.  Forward of 16,384 / 262,144 rows: 0.081 / 0.75 ms, with the small tile
// 0.102 / 0.955 (16 x 32 with two k steps 0.097 / 0.78; 16 x 64 with one 0.084 / 0.72
// but gradients of 262,144 rows 4.65 ms against 4.44).
constexpr int64_t GEMM_WIDE = 4096;
constexpr int GEMM_WARPS = 4;
constexpr int GEMM_KSPLIT_MAX = 64;
constexpr int GEMM_TARGET_BLOCKS = 2 * 152;

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);   // .x (low half) = lo
    return *reinterpret_cast<uint32_t *>(&v);
}

__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <int GEMM_NT, int GEMM_KU>
__global__ void __launch_bounds__(GEMM_WARPS * 32) k_gemm(GemmPair pr) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int nb0 = pr.a[0].blocks * pr.a[0].nsplit;
    const bool second = (int)blockIdx.x >= nb0;
    const GemmArgs a = second ? pr.a[1] : pr.a[0];
    const int block = (int)blockIdx.x - (second ? nb0 : 0), chunk = block / a.blocks;
    const int64_t tiles_n = (a.N + 8 * GEMM_NT - 1) / (8 * GEMM_NT);
    const int64_t tiles_m = (a.M + 15) / 16;
    const int64_t tile = (int64_t)(block % a.blocks) * GEMM_WARPS + warp;
    if (tile >= tiles_m * tiles_n) return;
    const int m0 = (int)(tile / tiles_n) * 16, n0 = (int)(tile % tiles_n) * 8 * GEMM_NT;
    const int kbeg = chunk * a.kchunk, kend = min(a.K, kbeg + a.kchunk);
    float acc[GEMM_NT][4];
#pragma unroll
    for (int j = 0; j < GEMM_NT; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
    // A fragment (16 x 16, row major): rows g and g+8, columns 2t, 2t+1 and 2t+8, 2t+9;
    // B fragment (16 x 8, column major): rows 2t, 2t+1 and 2t+8, 2t+9 of column g.
    // An element outside the operands reads the first of its row or column instead and
    // counts as 0, so that the loads need no branches and all go out together.
    const float *pa[2], *pb[GEMM_NT];
    bool va[2], vb[GEMM_NT];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        va[i] = m0 + g + 8 * i < a.M;
        pa[i] = a.A + (va[i] ? (int64_t)(m0 + g + 8 * i) * a.sam : 0);
    }
#pragma unroll
    for (int j = 0; j < GEMM_NT; ++j) {
        vb[j] = n0 + 8 * j + g < a.N;
        pb[j] = a.B + (vb[j] ? (int64_t)(n0 + 8 * j + g) * a.sbn : 0);
    }
    for (int k0 = kbeg; k0 < kend; k0 += 16 * GEMM_KU) {
        float fa[GEMM_KU][2][4], fb[GEMM_KU][GEMM_NT][4];
#pragma unroll
        for (int s = 0; s < GEMM_KU; ++s) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int k = k0 + 16 * s + 2 * t + (i & 1) + (i >> 1) * 8;
                const bool vk = k < kend;
                const int64_t ka = vk ? (int64_t)k * a.sak : 0, kb = vk ? (int64_t)k * a.sbk : 0;
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    const float v = pa[x][ka];
                    fa[s][x][i] = va[x] && vk ? v : 0.f;
                }
#pragma unroll
                for (int j = 0; j < GEMM_NT; ++j) {
                    const float v = pb[j][kb];
                    fb[s][j][i] = vb[j] && vk ? v : 0.f;
                }
            }
        }
#pragma unroll
        for (int s = 0; s < GEMM_KU; ++s) {
            const uint32_t ra[4] = {pack_bf16x2(fa[s][0][0], fa[s][0][1]), pack_bf16x2(fa[s][1][0], fa[s][1][1]),
                                    pack_bf16x2(fa[s][0][2], fa[s][0][3]), pack_bf16x2(fa[s][1][2], fa[s][1][3])};
#pragma unroll
            for (int j = 0; j < GEMM_NT; ++j)
                mma_bf16_16816(acc[j], ra, pack_bf16x2(fb[s][j][0], fb[s][j][1]),
                               pack_bf16x2(fb[s][j][2], fb[s][j][3]));
        }
    }
#pragma unroll
    for (int j = 0; j < GEMM_NT; ++j) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            // accumulator layout: rows g (i < 2) and g+8 (i >= 2), columns 2t + (i & 1)
            const int row = m0 + g + (i >= 2 ? 8 : 0);
            const int col = n0 + 8 * j + 2 * t + (i & 1);
            if (row >= a.M || col >= a.N) continue;
            if (a.nsplit > 1) {
                a.part[((int64_t)chunk * a.M + row) * a.N + col] = acc[j][i];
                continue;
            }
            float v = acc[j][i] + (a.bias ? a.bias[col] : 0.f);
            const int64_t idx = (int64_t)row * a.ldc + col;
            if (a.Z) a.Z[idx] = v;
            if (a.mask && !(a.mask[idx] > 0.f)) v = 0.f;
            if (a.relu) v = fmaxf(v, 0.f);
            a.C[idx] = v;
        }
    }
}

int grid1(int64_t n, int threads) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((n + threads - 1) / threads, 4096));
}

// sum of the split-K partials in chunk order, then the epilogue of k_gemm
__global__ void k_gemm_reduce(GemmArgs a) {
    const int64_t total = (int64_t)a.M * a.N;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int row = (int)(e / a.N), col = (int)(e % a.N);
        float v = 0.f;
        for (int s = 0; s < a.nsplit; ++s) v += a.part[(int64_t)s * total + e];
        v += a.bias ? a.bias[col] : 0.f;
        const int64_t idx = (int64_t)row * a.ldc + col;
        if (a.Z) a.Z[idx] = v;
        if (a.mask && !(a.mask[idx] > 0.f)) v = 0.f;
        if (a.relu) v = fmaxf(v, 0.f);
        a.C[idx] = v;
    }
}

void plan(GemmArgs &a, int nt) {
    const int64_t tiles_m = (a.M + 15) / 16;
    // blocks of 16 x 128, the unit that the number of chunks is chosen by
    const int64_t blocks = (tiles_m * ((a.N + 31) / 32) + 3) / 4;
    const int ksteps = (a.K + 15) / 16;
    // chunks of at least 4 k steps, enough of them to fill the GPU
    int nsplit = 1;
    if (a.part && blocks < GEMM_TARGET_BLOCKS && ksteps >= 8)
        nsplit = (int)std::min<int64_t>({GEMM_KSPLIT_MAX, (GEMM_TARGET_BLOCKS + blocks - 1) / blocks, ksteps / 4});
    const int steps_per = (ksteps + nsplit - 1) / nsplit;
    a.kchunk = 16 * std::max(steps_per, 1);
    a.nsplit = std::max(1, (a.K + a.kchunk - 1) / a.kchunk);
    a.blocks = (int)((tiles_m * ((a.N + 8 * nt - 1) / (8 * nt)) + GEMM_WARPS - 1) / GEMM_WARPS);
}

// one product, or two that do not depend on each other
void gemm(GemmArgs a, cudaStream_t st, const GemmArgs *b = nullptr) {
    GemmPair pr{};
    pr.a[0] = a;
    if (b) pr.a[1] = *b;
    int64_t tiles = 0;   // of 16 x 16
    for (const GemmArgs &x : pr.a) tiles += (int64_t)((x.M + 15) / 16) * ((x.N + 15) / 16);
    const bool wide = tiles >= GEMM_WIDE;
    const int nt = wide ? 4 : 2;
    plan(pr.a[0], nt);
    if (b) plan(pr.a[1], nt);
    const int blocks = pr.a[0].blocks * pr.a[0].nsplit + pr.a[1].blocks * pr.a[1].nsplit;
    ++g_launches;
    if (wide) k_gemm<4, 1><<<blocks, GEMM_WARPS * 32, 0, st>>>(pr);
    else k_gemm<2, 4><<<blocks, GEMM_WARPS * 32, 0, st>>>(pr);
    for (const GemmArgs &x : pr.a)
        if (x.nsplit > 1) {
            ++g_launches;
            k_gemm_reduce<<<grid1((int64_t)x.M * x.N, 256), 256, 0, st>>>(x);
        }
}

// ------------------------------------------------------------------ elementwise kernels

__global__ void k_standardize(const float *x, const float *norm, float *out, int64_t rows) {
    const int64_t total = rows * NIN;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(i % NIN);
        out[i] = (x[i] - norm[NORM_XMU + c]) * norm[NORM_XISD + c];
    }
}

__global__ void k_denorm(const float *y, const float *norm, float *out, int64_t rows) {
    const int64_t total = rows * NOUT;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(i % NOUT);
        out[i] = y[i] * norm[NORM_YSD + c] + norm[NORM_YMU + c];
    }
}

// Residuals against the normalised targets, dL/dy = r / B, and L = sum r^2 / (2B)
// written to *loss (one block; fixed summation order).
__global__ void k_loss(const float *y, const float *t, const float *norm, float *dy, int rows, float *loss) {
    __shared__ float part[256];
    float s = 0.f;
    const float inv_b = 1.f / (float)rows;
    for (int i = threadIdx.x; i < rows * NOUT; i += blockDim.x) {
        const int c = i % NOUT;
        const float tn = (t[i] - norm[NORM_YMU + c]) / norm[NORM_YSD + c];
        const float r = y[i] - tn;
        dy[i] = r * inv_b;
        s += r * r;
    }
    part[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *loss = part[0] * 0.5f * inv_b;
}

// The bias gradients: sums over the rows of the columns of dy, d2 and d1; one
// warp per column.
constexpr int COLSUM_COLS = NOUT + 2 * NH;
__global__ void k_bias_grads(const float *dy, const float *d2, const float *d1, int rows, float *g) {
    const int lane = threadIdx.x & 31;
    int col = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (col >= COLSUM_COLS) return;
    const float *src = dy;
    int N = NOUT, off = OFF_B3;
    if (col >= NOUT + NH) {
        src = d1, N = NH, off = OFF_B1, col -= NOUT + NH;
    } else if (col >= NOUT) {
        src = d2, N = NH, off = OFF_B2, col -= NOUT;
    }
    float s = 0.f;
    for (int r = lane; r < rows; r += 32) s += src[(int64_t)r * N + col];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    if (lane == 0) g[off + col] = s;
}

// Adam (Kingma and Ba, 2015) with decoupled weight decay (Loshchilov and
// Hutter, 2019): p -= lr * (m_hat / (sqrt(v_hat) + eps) + wd * p).
__global__ void k_adam(float *p, const float *g, float *m, float *v, int n, float lr, float bc1, float bc2, float wd) {
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float pi = p[i];
        p[i] = pi - lr * ((mi / bc1) / (sqrtf(vi / bc2) + eps) + wd * pi);
    }
}

// The rows of one step, standardised, and their targets
__global__ void k_gather(const float *x, const float *t, const float *norm, const int32_t *perm, int rows, float *xs,
                         float *tb) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < rows * NIN; i += gridDim.x * blockDim.x) {
        const int r = i / NIN, c = i % NIN;
        xs[i] = (x[(int64_t)perm[r] * NIN + c] - norm[NORM_XMU + c]) * norm[NORM_XISD + c];
    }
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < rows * NOUT; i += gridDim.x * blockDim.x) {
        const int r = i / NOUT, c = i % NOUT;
        tb[i] = t[(int64_t)perm[r] * NOUT + c];
    }
}

// ------------------------------------------------------------------ features

// Window length of the interval feature: ceil(log4(n + 1)) + 4 letters, long
// enough that a window of an unrelated query is rarely found in the text.
int interval_window(int64_t n) {
    int k = 0;
    for (int64_t r = 1; r < n + 1; r *= 4) ++k;
    return std::min(k + 4, 32);
}

__device__ __forceinline__ int dna_code(uint8_t ch, int *bad) {
    switch (ch) {
        case 'A': return 0;
        case 'C': return 1;
        case 'G': return 2;
        case 'T': return 3;
        default: atomicExch(bad, 1); return 0;
    }
}

// A query's features: the 3-mer spectrum, log1p(m), and the mean over the
// query's windows of K letters of log1p(|SA interval of the window|).  The
// interval of a window w comes from K backward steps with w's letters in
// order, which give the rows of reverse(w) in the index of the reversed text,
// one row per occurrence of w in T (Section 2.3, Section 5 (3)).
//
// A window is a chain of about 15 dependent occurrence look-ups, so k_features
// takes FEAT_POS positions of a query per block (two per thread; more where that
// would be more than about FEAT_PARTS blocks) and k_features_sum adds the blocks'
// counts and sums in a fixed order (64 queries of 200 to 20,000 letters, 100 Mbp text:
// 2.2 ms with a block per query, 0.1 ms so).  Where every query is one part (ALONE),
// its block writes the features itself (20,000 queries of 150 letters 0.575 -> 0.514 ms).
constexpr int FEAT_THREADS = 128;
constexpr int FEAT_POS = 256;
constexpr int64_t FEAT_PARTS = 1 << 16;

struct FeatPart {
    int cnt[64];
    float sum;
};

// The features of a query of m letters from its 3-mer counts (thread w has word
// w's) and the sum over its windows
__device__ __forceinline__ void put_features(float *f, int64_t m, int K, int c, float sum) {
    const float inv = m >= 3 ? 1.f / (float)(m - 2) : 0.f;
    if (threadIdx.x < 64) f[threadIdx.x] = (float)c * inv;
    if (threadIdx.x == 0) {
        f[64] = log1pf((float)m);
        f[65] = m >= K ? sum / (float)(m - K + 1) : 0.f;
    }
}

template <bool ALONE>
__global__ void __launch_bounds__(FEAT_THREADS) k_features(IndexView ix, const uint8_t *seq, const int64_t *off,
                                                           const int64_t *first, int nq, int64_t pos, int K, FeatPart *part,
                                                           float *feat, int *bad) {
    __shared__ int cnt[64];
    __shared__ float acc_s[FEAT_THREADS];
    int lo_q = ALONE ? (int)blockIdx.x : 0, hi_q = ALONE ? lo_q : nq - 1;
    while (lo_q < hi_q) {   // the query of this block: the last one that starts at or before it
        const int mid = (lo_q + hi_q + 1) >> 1;
        if (first[mid] <= (int64_t)blockIdx.x) lo_q = mid; else hi_q = mid - 1;
    }
    for (int w = threadIdx.x; w < 64; w += blockDim.x) cnt[w] = 0;
    __syncthreads();
    const int64_t b = off[lo_q], m = off[lo_q + 1] - b;
    const int64_t p0 = ALONE ? 0 : ((int64_t)blockIdx.x - first[lo_q]) * pos, p1 = min(p0 + pos, m);
    for (int64_t p = p0 + threadIdx.x; p < p1; p += blockDim.x) {
        const int c0 = dna_code(seq[b + p], bad);
        if (p + 2 < m) atomicAdd(&cnt[16 * c0 + 4 * dna_code(seq[b + p + 1], bad) + dna_code(seq[b + p + 2], bad)], 1);
    }
    float acc = 0.f;
    for (int64_t p = p0 + threadIdx.x; p < p1 && p + K <= m; p += blockDim.x) {
        uint32_t lo = 0, hi = (uint32_t)ix.rows;
        for (int s = 0; s < K && lo < hi; ++s) {
            const int c = dna_code(seq[b + p + s], bad);
            lo = ix.C[c] + aedev::occ_dna(ix, c, lo);
            hi = ix.C[c] + aedev::occ_dna(ix, c, hi);
        }
        acc += log1pf(lo < hi ? (float)(hi - lo) : 0.f);
    }
    acc_s[threadIdx.x] = acc;
    __syncthreads();
    for (int w = FEAT_THREADS / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) acc_s[threadIdx.x] += acc_s[threadIdx.x + w];
        __syncthreads();
    }
    if (ALONE) {
        put_features(feat + (int64_t)lo_q * NIN, m, K, threadIdx.x < 64 ? cnt[threadIdx.x] : 0, acc_s[0]);
        return;
    }
    FeatPart &o = part[blockIdx.x];
    for (int w = threadIdx.x; w < 64; w += blockDim.x) o.cnt[w] = cnt[w];
    if (threadIdx.x == 0) o.sum = acc_s[0];
}

// one block per query
__global__ void __launch_bounds__(FEAT_THREADS) k_features_sum(const int64_t *off, const int64_t *first, int K,
                                                               const FeatPart *part, float *feat) {
    __shared__ float acc_s[FEAT_THREADS];
    const int q = blockIdx.x;
    const int64_t m = off[q + 1] - off[q], f0 = first[q], f1 = first[q + 1];
    int c = 0;
    if (threadIdx.x < 64)
        for (int64_t f = f0; f < f1; ++f) c += part[f].cnt[threadIdx.x];
    float acc = 0.f;
    for (int64_t f = f0 + threadIdx.x; f < f1; f += FEAT_THREADS) acc += part[f].sum;
    acc_s[threadIdx.x] = acc;
    __syncthreads();
    for (int w = FEAT_THREADS / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) acc_s[threadIdx.x] += acc_s[threadIdx.x + w];
        __syncthreads();
    }
    put_features(feat + (int64_t)q * NIN, m, K, c, acc_s[0]);
}

uint64_t splitmix64(uint64_t &s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Per-thread device scratch of ae_mlp_features (offsets, each query's first
// part, the parts, and the error flag), grown on demand and kept so that calls
// allocate nothing once warm.
struct FeatScratch {
    int64_t *off = nullptr;      // offsets, then the first parts
    FeatPart *part = nullptr;
    std::vector<int64_t> host;
    int *bad = nullptr;
    int *h_bad = nullptr;
    int32_t cap = 0;
    int64_t part_cap = 0;
    void release() {
        if (off) cudaFree(off);
        if (part) cudaFree(part);
        if (bad) cudaFree(bad);
        if (h_bad) cudaFreeHost(h_bad);
        off = nullptr, part = nullptr, bad = nullptr, h_bad = nullptr;
        cap = 0;
        part_cap = 0;
    }
    ~FeatScratch() { release(); }
};
thread_local FeatScratch g_feat_scratch;

struct mlp_error {
    ae_status st;
};

#define MC(x)                                                          \
    do {                                                               \
        if ((x) != cudaSuccess) throw mlp_error{AE_ECUDA};             \
    } while (0)

}  // namespace

struct ae_mlp {
    float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr, *norm = nullptr;
    int64_t step = 0;
    int32_t cap = 0;
    float *x = nullptr, *z1 = nullptr, *a1 = nullptr, *z2 = nullptr, *a2 = nullptr, *y = nullptr, *dy = nullptr,
          *d1 = nullptr, *d2 = nullptr, *tb = nullptr, *loss = nullptr;
    float *part = nullptr;          // split-K partials of the weight gradients
    int32_t *perm = nullptr;
    int32_t perm_cap = 0, loss_cap = 0;
    float h_norm[NORM_SIZE];

    void free_acts() {
        float **bufs[] = {&x, &z1, &a1, &z2, &a2, &y, &dy, &d1, &d2, &tb};
        for (float **b : bufs) {
            if (*b) cudaFree(*b);
            *b = nullptr;
        }
        cap = 0;
    }
    ~ae_mlp() {
        free_acts();
        for (float *b : {p, g, m, v, norm, loss, part})
            if (b) cudaFree(b);
        if (perm) cudaFree(perm);
    }
    void reserve(int32_t rows) {
        if (rows <= cap) return;
        free_acts();
        const int32_t c = std::max(rows, 256);
        const size_t in = sizeof(float) * (size_t)c * NIN, hid = sizeof(float) * (size_t)c * NH,
                     out = sizeof(float) * (size_t)c * NOUT;
        struct {
            float **b;
            size_t bytes;
        } plan[] = {{&x, in}, {&z1, hid}, {&a1, hid}, {&z2, hid}, {&a2, hid}, {&y, out},
                    {&dy, out}, {&d1, hid}, {&d2, hid}, {&tb, out}};
        for (auto &e : plan)
            if (cudaMalloc(e.b, e.bytes) != cudaSuccess) {
                cudaGetLastError();
                free_acts();
                throw mlp_error{AE_ENOMEM};
            }
        cap = c;
    }

    // forward of `rows` standardised inputs already in x
    void forward_std(int32_t rows, cudaStream_t st) {
        GemmArgs a{};
        a.A = x, a.sam = NIN, a.sak = 1, a.B = p + OFF_W1, a.sbk = 1, a.sbn = NIN, a.C = a1, a.ldc = NH;
        a.bias = p + OFF_B1, a.Z = z1, a.M = rows, a.N = NH, a.K = NIN, a.relu = 1;
        gemm(a, st);
        a = GemmArgs{};
        a.A = a1, a.sam = NH, a.sak = 1, a.B = p + OFF_W2, a.sbk = 1, a.sbn = NH, a.C = a2, a.ldc = NH;
        a.bias = p + OFF_B2, a.Z = z2, a.M = rows, a.N = NH, a.K = NH, a.relu = 1;
        gemm(a, st);
        a = GemmArgs{};
        a.A = a2, a.sam = NH, a.sak = 1, a.B = p + OFF_W3, a.sbk = 1, a.sbn = NH, a.C = y, a.ldc = NOUT;
        a.bias = p + OFF_B3, a.M = rows, a.N = NOUT, a.K = NH;
        gemm(a, st);
    }

    // loss and gradients (into g) of `rows` inputs in x with raw targets t
    void backward(int32_t rows, const float *t, float *loss_slot, cudaStream_t st) {
        forward_std(rows, st);
        ++g_launches;
        k_loss<<<1, 256, 0, st>>>(y, t, norm, dy, rows, loss_slot);
        GemmArgs a{}, b{};
        // dW3 = dy^T a2 and d2 = (dy W3) * [z2 > 0]
        a.A = dy, a.sam = 1, a.sak = NOUT, a.B = a2, a.sbk = NH, a.sbn = 1, a.C = g + OFF_W3, a.ldc = NH;
        a.M = NOUT, a.N = NH, a.K = rows;
        a.part = part;
        b.A = dy, b.sam = NOUT, b.sak = 1, b.B = p + OFF_W3, b.sbk = NH, b.sbn = 1, b.C = d2, b.ldc = NH;
        b.mask = z2, b.M = rows, b.N = NH, b.K = NOUT;
        gemm(a, st, &b);
        // dW2 = d2^T a1 and d1 = (d2 W2) * [z1 > 0]
        a = b = GemmArgs{};
        a.A = d2, a.sam = 1, a.sak = NH, a.B = a1, a.sbk = NH, a.sbn = 1, a.C = g + OFF_W2, a.ldc = NH;
        a.M = NH, a.N = NH, a.K = rows;
        a.part = part;
        b.A = d2, b.sam = NH, b.sak = 1, b.B = p + OFF_W2, b.sbk = NH, b.sbn = 1, b.C = d1, b.ldc = NH;
        b.mask = z1, b.M = rows, b.N = NH, b.K = NH;
        gemm(a, st, &b);
        // dW1 = d1^T x
        a = GemmArgs{};
        a.A = d1, a.sam = 1, a.sak = NH, a.B = x, a.sbk = NIN, a.sbn = 1, a.C = g + OFF_W1, a.ldc = NIN;
        a.M = NH, a.N = NIN, a.K = rows;
        a.part = part;
        gemm(a, st);
        ++g_launches;
        k_bias_grads<<<(COLSUM_COLS + 3) / 4, 128, 0, st>>>(dy, d2, d1, rows, g);
    }

    void standardize(const float *raw, int32_t rows, float *dst, cudaStream_t st) {
        ++g_launches;
        k_standardize<<<grid1((int64_t)rows * NIN, 256), 256, 0, st>>>(raw, norm, dst, rows);
    }

    void adam_step(float lr, float wd, cudaStream_t st) {
        ++step;
        const double bc1 = 1.0 - std::pow(0.9, (double)step), bc2 = 1.0 - std::pow(0.999, (double)step);
        ++g_launches;
        k_adam<<<grid1(NPARAM, 256), 256, 0, st>>>(p, g, m, v, NPARAM, lr, (float)bc1, (float)bc2, wd);
    }
};

extern "C" {

ae_status ae_mlp_create(uint64_t seed, ae_mlp **out) {
    if (!out) return AE_EINVAL;
    *out = nullptr;
    ae_mlp *mlp = new (std::nothrow) ae_mlp();
    if (!mlp) return AE_ENOMEM;
    try {
        for (float **b : {&mlp->p, &mlp->g, &mlp->m, &mlp->v})
            if (cudaMalloc(b, sizeof(float) * NPARAM) != cudaSuccess) throw mlp_error{AE_ENOMEM};
        if (cudaMalloc(&mlp->norm, sizeof(float) * NORM_SIZE) != cudaSuccess) throw mlp_error{AE_ENOMEM};
        if (cudaMalloc(&mlp->part, sizeof(float) * GEMM_KSPLIT_MAX * NH * NH) != cudaSuccess)
            throw mlp_error{AE_ENOMEM};
        std::vector<float> h(NPARAM, 0.f);
        uint64_t s = seed;
        auto fill = [&](int off, int rows, int cols) {
            const double bound = std::sqrt(6.0 / cols);
            for (int i = 0; i < rows * cols; ++i) {
                const double u = (double)(splitmix64(s) >> 11) * (1.0 / 9007199254740992.0);
                h[off + i] = (float)((2.0 * u - 1.0) * bound);
            }
        };
        fill(OFF_W1, NH, NIN);
        fill(OFF_W2, NH, NH);
        fill(OFF_W3, NOUT, NH);
        MC(cudaMemcpy(mlp->p, h.data(), sizeof(float) * NPARAM, cudaMemcpyHostToDevice));
        MC(cudaMemset(mlp->m, 0, sizeof(float) * NPARAM));
        MC(cudaMemset(mlp->v, 0, sizeof(float) * NPARAM));
        MC(cudaMemset(mlp->g, 0, sizeof(float) * NPARAM));
        for (int i = 0; i < NIN; ++i) {
            mlp->h_norm[NORM_XMU + i] = 0.f;
            mlp->h_norm[NORM_XISD + i] = 1.f;
        }
        for (int i = 0; i < NOUT; ++i) {
            mlp->h_norm[NORM_YMU + i] = 0.f;
            mlp->h_norm[NORM_YSD + i] = 1.f;
        }
        MC(cudaMemcpy(mlp->norm, mlp->h_norm, sizeof(float) * NORM_SIZE, cudaMemcpyHostToDevice));
    } catch (const mlp_error &e) {
        cudaGetLastError();
        delete mlp;
        return e.st;
    }
    *out = mlp;
    return AE_OK;
}

void ae_mlp_free(ae_mlp *mlp) { delete mlp; }

ae_status ae_mlp_set_params(ae_mlp *mlp, const float *params) {
    if (!mlp || !params) return AE_EINVAL;
    if (cudaMemcpy(mlp->p, params, sizeof(float) * NPARAM, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(mlp->m, 0, sizeof(float) * NPARAM) != cudaSuccess ||
        cudaMemset(mlp->v, 0, sizeof(float) * NPARAM) != cudaSuccess)
        return AE_ECUDA;
    mlp->step = 0;
    return AE_OK;
}

ae_status ae_mlp_get_params(const ae_mlp *mlp, float *params) {
    if (!mlp || !params) return AE_EINVAL;
    return cudaMemcpy(params, mlp->p, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost) == cudaSuccess ? AE_OK
                                                                                                       : AE_ECUDA;
}

ae_status ae_mlp_set_norm(ae_mlp *mlp, const float *x_mu, const float *x_sd, const float *y_mu, const float *y_sd) {
    if (!mlp || !x_mu || !x_sd || !y_mu || !y_sd) return AE_EINVAL;
    for (int i = 0; i < NIN; ++i)
        if (!(x_sd[i] > 0.f)) return AE_EINVAL;
    for (int i = 0; i < NOUT; ++i)
        if (!(y_sd[i] > 0.f)) return AE_EINVAL;
    for (int i = 0; i < NIN; ++i) {
        mlp->h_norm[NORM_XMU + i] = x_mu[i];
        mlp->h_norm[NORM_XISD + i] = 1.f / x_sd[i];
    }
    for (int i = 0; i < NOUT; ++i) {
        mlp->h_norm[NORM_YMU + i] = y_mu[i];
        mlp->h_norm[NORM_YSD + i] = y_sd[i];
    }
    return cudaMemcpy(mlp->norm, mlp->h_norm, sizeof(float) * NORM_SIZE, cudaMemcpyHostToDevice) == cudaSuccess
               ? AE_OK
               : AE_ECUDA;
}

ae_status ae_mlp_features(const ae_index *idx, const uint8_t *d_seq, const int64_t *offsets, int32_t nq,
                          float *d_feat, void *stream) {
    if (!idx || !offsets || nq < 0 || (nq > 0 && !d_feat)) return AE_EINVAL;
    if (nq == 0) return AE_OK;
    if (offsets[0] != 0) return AE_EINVAL;
    int64_t longest = 0;
    for (int q = 0; q < nq; ++q) {
        if (offsets[q + 1] < offsets[q]) return AE_EINVAL;
        longest = std::max(longest, offsets[q + 1] - offsets[q]);
    }
    if (offsets[nq] > 0 && !d_seq) return AE_EINVAL;
    const IndexView *ix = ae_index_view(idx);
    if (ix->alphabet != AE_DNA) return AE_EUNSUPPORTED;
    cudaStream_t st = (cudaStream_t)stream;
    FeatScratch &fs = g_feat_scratch;
    // parts of `pos` positions
    const int64_t pos = std::max<int64_t>(FEAT_POS, (offsets[nq] + FEAT_PARTS - 1) / FEAT_PARTS);
    const size_t words = (size_t)nq + 1;
    const bool alone = longest <= pos;   // every query is one part: nothing to add up
    int64_t nparts = nq;
    const int64_t *host = offsets;
    if (!alone) {
        try {
            fs.host.resize(2 * words);
        } catch (const std::bad_alloc &) {
            return AE_ENOMEM;
        }
        nparts = 0;
        for (int q = 0; q <= nq; ++q) {
            fs.host[q] = offsets[q];
            fs.host[words + q] = nparts;
            if (q < nq) nparts += (offsets[q + 1] - offsets[q] + pos - 1) / pos;
        }
        host = fs.host.data();
    }
    if (fs.cap < nq + 1 || (!alone && fs.part_cap < nparts)) {
        const int32_t c = std::max({nq + 1, fs.cap, 1024});
        const int64_t pc = std::max<int64_t>({alone ? 0 : nparts, fs.part_cap, 4096});
        fs.release();
        if (cudaMalloc(&fs.off, 2 * sizeof(int64_t) * (size_t)c) != cudaSuccess ||
            cudaMalloc(&fs.part, sizeof(FeatPart) * pc) != cudaSuccess ||
            cudaMalloc(&fs.bad, sizeof(int)) != cudaSuccess || cudaMallocHost(&fs.h_bad, sizeof(int)) != cudaSuccess) {
            cudaGetLastError();
            fs.release();
            return AE_ENOMEM;
        }
        fs.cap = c;
        fs.part_cap = pc;
    }
    if (cudaMemcpyAsync(fs.off, host, (alone ? 1 : 2) * sizeof(int64_t) * words, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemsetAsync(fs.bad, 0, sizeof(int), st) != cudaSuccess)
        return AE_ECUDA;
    const int K = interval_window(ix->n);
    const int64_t *first = fs.off + words;
    ++g_launches;
    if (alone) {
        k_features<true><<<(unsigned)nparts, FEAT_THREADS, 0, st>>>(*ix, d_seq, fs.off, first, nq, pos, K, fs.part, d_feat,
                                                                   fs.bad);
    } else {
        k_features<false><<<(unsigned)nparts, FEAT_THREADS, 0, st>>>(*ix, d_seq, fs.off, first, nq, pos, K, fs.part, d_feat,
                                                                    fs.bad);
        ++g_launches;
        k_features_sum<<<nq, FEAT_THREADS, 0, st>>>(fs.off, first, K, fs.part, d_feat);
    }
    if (cudaGetLastError() != cudaSuccess ||
        cudaMemcpyAsync(fs.h_bad, fs.bad, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return AE_ECUDA;
    return *fs.h_bad ? AE_EINVAL : AE_OK;
}

ae_status ae_mlp_forward(ae_mlp *mlp, const float *d_x, int32_t B, float *d_y, void *stream) {
    if (!mlp || B < 0 || (B > 0 && (!d_x || !d_y))) return AE_EINVAL;
    if (B == 0) return AE_OK;
    cudaStream_t st = (cudaStream_t)stream;
    try {
        mlp->reserve(B);
        mlp->standardize(d_x, B, mlp->x, st);
        mlp->forward_std(B, st);
        ++g_launches;
        k_denorm<<<grid1((int64_t)B * NOUT, 256), 256, 0, st>>>(mlp->y, mlp->norm, d_y, B);
        MC(cudaGetLastError());
        MC(cudaStreamSynchronize(st));
    } catch (const mlp_error &e) {
        cudaGetLastError();
        return e.st;
    }
    return AE_OK;
}

ae_status ae_mlp_loss_grad(ae_mlp *mlp, const float *d_x, const float *d_t, int32_t B, float *loss, float *grads,
                           void *stream) {
    if (!mlp || B < 1 || !d_x || !d_t || !loss) return AE_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    try {
        mlp->reserve(B);
        if (mlp->loss_cap < 1) {
            MC(cudaMalloc(&mlp->loss, sizeof(float) * 1024));
            mlp->loss_cap = 1024;
        }
        mlp->standardize(d_x, B, mlp->x, st);
        mlp->backward(B, d_t, mlp->loss, st);
        MC(cudaGetLastError());
        MC(cudaMemcpyAsync(loss, mlp->loss, sizeof(float), cudaMemcpyDeviceToHost, st));
        if (grads) MC(cudaMemcpyAsync(grads, mlp->g, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, st));
        MC(cudaStreamSynchronize(st));
    } catch (const mlp_error &e) {
        cudaGetLastError();
        return e.st;
    }
    return AE_OK;
}

ae_status ae_mlp_train(ae_mlp *mlp, const float *d_x, const float *d_t, int32_t n, int32_t epochs, int32_t batch,
                       float lr, float weight_decay, uint64_t seed, float *loss, void *stream) {
    if (!mlp || n < 1 || !d_x || !d_t || epochs < 0 || batch < 1 || !(lr > 0.f) || !(weight_decay >= 0.f))
        return AE_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    batch = std::min(batch, n);
    const int32_t steps = (n + batch - 1) / batch;
    try {
        mlp->reserve(batch);
        if (mlp->perm_cap < n) {
            if (mlp->perm) cudaFree(mlp->perm);
            mlp->perm = nullptr;
            mlp->perm_cap = 0;
            MC(cudaMalloc(&mlp->perm, sizeof(int32_t) * n));
            mlp->perm_cap = n;
        }
        if (mlp->loss_cap < steps) {
            if (mlp->loss) cudaFree(mlp->loss);
            mlp->loss = nullptr;
            mlp->loss_cap = 0;
            MC(cudaMalloc(&mlp->loss, sizeof(float) * std::max(steps, 1024)));
            mlp->loss_cap = std::max(steps, 1024);
        }
        std::vector<int32_t> perm(n);
        std::vector<float> losses(steps, 0.f);
        uint64_t s = seed;
        for (int32_t e = 0; e < epochs; ++e) {
            for (int32_t i = 0; i < n; ++i) perm[i] = i;
            for (int32_t i = n - 1; i > 0; --i) {          // Fisher-Yates
                const int32_t j = (int32_t)(splitmix64(s) % (uint64_t)(i + 1));
                std::swap(perm[i], perm[j]);
            }
            MC(cudaMemcpyAsync(mlp->perm, perm.data(), sizeof(int32_t) * n, cudaMemcpyHostToDevice, st));
            for (int32_t k = 0; k < steps; ++k) {
                const int32_t r0 = k * batch, rows = std::min(batch, n - r0);
                ++g_launches;
                k_gather<<<grid1((int64_t)rows * NIN, 256), 256, 0, st>>>(d_x, d_t, mlp->norm, mlp->perm + r0, rows,
                                                                          mlp->x, mlp->tb);
                mlp->backward(rows, mlp->tb, mlp->loss + k, st);
                mlp->adam_step(lr, weight_decay, st);
            }
            // the host permutation buffer is rewritten next epoch: wait for the upload
            MC(cudaStreamSynchronize(st));
        }
        MC(cudaGetLastError());
        if (loss && epochs > 0) {
            MC(cudaMemcpyAsync(losses.data(), mlp->loss, sizeof(float) * steps, cudaMemcpyDeviceToHost, st));
            MC(cudaStreamSynchronize(st));
            double acc = 0;
            for (float v : losses) acc += v;
            *loss = (float)(acc / steps);
        }
    } catch (const mlp_error &e) {
        cudaGetLastError();
        return e.st;
    } catch (const std::bad_alloc &) {
        return AE_ENOMEM;
    }
    return AE_OK;
}

}  // extern "C"
