// Kernels of the warm-start network: a fully connected GELU network in BF16 with FP32
// accumulation (forward, backward, Adam).  The matrix products run on the tensor cores
// through warp-level mma.sync (m16n8k16, BF16 inputs, FP32 accumulators); the layers are
// small (32..256 wide), so a 64 x 64 block tile staged through shared memory is enough.
#pragma once

#include <cuda_bf16.h>

namespace wsn {

// C = op(A) op(B), M x N x K in BF16; the epilogue decides what is written (see Epi).  Each
// operand is stored with one of its dimensions contiguous (the kernel's AK / BK: that is K)
// and ld elements between neighbours of the other.
struct Gemm {
    const __nv_bfloat16 *A, *B;
    int lda, ldb;
    int avec, bvec;           // 16-byte copies: the pointer is 16-byte aligned, ld a multiple of 8
    int M, N, K;
    const float *bias;        // per column (BIAS, BIAS_GELU)
    const float *scale;       // per column, BIAS only: out = (C + bias) * scale (NULL: 1)
    float *out;               // FP32 output (ldo = N): C, C + bias, or the pre-activation
    __nv_bfloat16 *act;       // BF16 output (ldo = N): GELU(C + bias), or C * GELU'(pre)
    const float *pre;         // pre-activation read by GELU_BWD (ldo = N)
};

enum Epi { EPI_STORE = 0, EPI_BIAS = 1, EPI_BIAS_GELU = 2, EPI_GELU_BWD = 3 };

__device__ __forceinline__ float gelu_f(float u) { return 0.5f * u * (1.0f + erff(u * 0.70710678118654752f)); }

__device__ __forceinline__ float gelu_grad_f(float u)
{
    return 0.5f * (1.0f + erff(u * 0.70710678118654752f)) + u * 0.39894228040143268f * expf(-0.5f * u * u);
}

__device__ __forceinline__ void mma_bf16(float *c, const unsigned *a, const unsigned *b)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

constexpr int TM = 64, TN = 64, TK = 32, STAGES = 3;
// one operand's tile in shared memory: 64 rows of 32 K values (rows padded to 40) or 32 K rows
// of 64 values (padded to 72); both pads put the eight 16-byte rows that an ldmatrix reads at
// once into different banks
constexpr int LDK = TK + 8, LDMN = TM + 8;
constexpr int TILE = TM * LDK > TK * LDMN ? TM * LDK : TK * LDMN;

__device__ __forceinline__ unsigned sm_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void ldsm4(unsigned *r, unsigned addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}

__device__ __forceinline__ void ldsm4t(unsigned *r, unsigned addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}

// Rows x0 .. x0 + 63 of the non-K dimension (limit X) by k0 .. k0 + 31 (limit kend) into one
// stage, zeros outside: 16-byte asynchronous copies along the contiguous dimension, or (no
// such alignment: a width of 7) element by element, neighbouring threads on neighbouring
// addresses.
template <bool KC>
__device__ __forceinline__ void load_tile(__nv_bfloat16 *dst, const __nv_bfloat16 *src, int ld, bool vec,
                                          int x0, int X, int k0, int kend)
{
    constexpr int INNER = KC ? TK : TM, OUTER = KC ? TM : TK, LDS = KC ? LDK : LDMN;
    const int i0 = KC ? k0 : x0, ilim = KC ? kend : X, o0 = KC ? x0 : k0, olim = KC ? X : kend;
    if (vec) {
        // (the contiguous dimension spans whole rows of ld = a multiple of 8: a chunk is in or out)
        for (int c = threadIdx.x; c < OUTER * (INNER / 8); c += 128) {
            const int o = c / (INNER / 8), i = (c % (INNER / 8)) * 8;
            const bool in = o0 + o < olim && i0 + i < ilim;
            const __nv_bfloat16 *p = in ? src + (long long)(o0 + o) * ld + i0 + i : src;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                         ::"r"(sm_addr(dst + o * LDS + i)), "l"(p), "r"(in ? 16 : 0) : "memory");
        }
    } else {
        for (int c = threadIdx.x; c < OUTER * INNER; c += 128) {
            const int o = c / INNER, i = c % INNER;
            const bool in = o0 + o < olim && i0 + i < ilim;
            dst[o * LDS + i] = in ? src[(long long)(o0 + o) * ld + i0 + i] : __float2bfloat16(0.0f);
        }
    }
}

// The K range [kb, ke) of one 64 x 64 tile of C (128 threads): 4 warps in a 2 x 2
// arrangement, each a 32 x 32 block as 2 x 4 tiles of m16n8, K ascending in steps of 16 (the
// order of the sums does not depend on the tile's operand layout).  Three stages of 32 K
// values in flight.  COLSUM: with csum given, threads 0 .. 63 also sum the columns of B
// in K order.
// These layers are latency-bound, not tensor-bound (a 4096-row layer is 0.5 GFLOP), so the
// pipeline depth and the coalesced copies matter, not the instruction.
template <bool AK, bool BK, bool COLSUM>
__device__ __forceinline__ void gemm_tile(const Gemm &g, int m0, int n0, int kb, int ke,
                                          float (*acc)[4][4], float *csum)
{
    __shared__ __align__(16) __nv_bfloat16 As[STAGES][TILE], Bs[STAGES][TILE];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
    const int steps = (ke - kb + TK - 1) / TK;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0f;
    auto fill = [&](int t) {
        if (t < steps) {
            load_tile<AK>(As[t % STAGES], g.A, g.lda, g.avec, m0, g.M, kb + t * TK, ke);
            load_tile<BK>(Bs[t % STAGES], g.B, g.ldb, g.bvec, n0, g.N, kb + t * TK, ke);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int t = 0; t < STAGES - 1; ++t) fill(t);
    // ldmatrix source of a lane: matrix lane / 8, row lane % 8
    const int q8 = lane >> 3, r8 = lane & 7;
    for (int t = 0; t < steps; ++t) {
        asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
        __syncthreads();                      // stage t landed; stage t - 1 is free again
        fill(t + STAGES - 1);
        const __nv_bfloat16 *as = As[t % STAGES], *bs = Bs[t % STAGES];
#pragma unroll
        for (int kk = 0; kk < TK; kk += 16) {
            unsigned a[2][4], b[2][4];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                // matrices (m, k), (m + 8, k), (m, k + 8), (m + 8, k + 8)
                const int m = wm + 16 * i;
                if (AK) ldsm4(a[i], sm_addr(as + (m + (q8 & 1) * 8 + r8) * LDK + kk + (q8 >> 1) * 8));
                else ldsm4t(a[i], sm_addr(as + (kk + (q8 >> 1) * 8 + r8) * LDMN + m + (q8 & 1) * 8));
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                // matrices (n, k), (n, k + 8), (n + 8, k), (n + 8, k + 8)
                const int n = wn + 16 * j;
                if (BK) ldsm4(b[j], sm_addr(bs + (n + (q8 >> 1) * 8 + r8) * LDK + kk + (q8 & 1) * 8));
                else ldsm4t(b[j], sm_addr(bs + (kk + (q8 & 1) * 8 + r8) * LDMN + n + (q8 >> 1) * 8));
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], a[i], &b[j >> 1][2 * (j & 1)]);
        }
        if (COLSUM && csum && threadIdx.x < TN) {
            float s = *csum;
            for (int k = 0; k < TK; ++k) s += __bfloat162float(bs[k * LDMN + threadIdx.x]);
            *csum = s;
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// accumulator (i, j, q) of a thread: row wm + 16 i + gq (+ 8 for q >= 2), column
// wn + 8 j + 2 tq + (q & 1)
template <int EPI>
__device__ __forceinline__ void gemm_store(const Gemm &g, int m0, int n0, float (*acc)[4][4])
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32, gq = lane >> 2, tq = lane & 3;
    // neighbouring columns in one store: even N (n is even) and an 8-byte aligned output
    const bool pair = !(g.N & 1) && !((size_t)(EPI == EPI_GELU_BWD ? (const void *)g.act : (const void *)g.out) & 7);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int m = m0 + wm + 16 * i + gq + 8 * h, n = n0 + wn + 8 * j + 2 * tq;
                if (m >= g.M || n >= g.N) continue;
                const long long o = (long long)m * g.N + n;
                const bool two = n + 1 < g.N;
                float c[2], u[2];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    c[q] = acc[i][j][2 * h + q];
                    if (q && !two) continue;
                    if (EPI == EPI_BIAS) c[q] = g.scale ? (c[q] + g.bias[n + q]) * g.scale[n + q] : c[q] + g.bias[n + q];
                    if (EPI == EPI_BIAS_GELU) { c[q] = c[q] + g.bias[n + q]; u[q] = gelu_f(c[q]); }
                    if (EPI == EPI_GELU_BWD) u[q] = c[q] * gelu_grad_f(g.pre[o + q]);
                }
                if (EPI != EPI_GELU_BWD) {
                    if (pair) *reinterpret_cast<float2 *>(g.out + o) = make_float2(c[0], c[1]);
                    else { g.out[o] = c[0]; if (two) g.out[o + 1] = c[1]; }
                }
                if (EPI == EPI_BIAS_GELU || EPI == EPI_GELU_BWD) {
                    if (pair) *reinterpret_cast<__nv_bfloat162 *>(g.act + o) = __floats2bfloat162_rn(u[0], u[1]);
                    else { g.act[o] = __float2bfloat16(u[0]); if (two) g.act[o + 1] = __float2bfloat16(u[1]); }
                }
            }
        }
    }
}

// A layer: A with K contiguous (activations or output gradients, a row per sample), B the
// weights (N contiguous forward, K contiguous backward).
template <int EPI, bool BK>
__global__ void __launch_bounds__(128) gemm_kernel(Gemm g)
{
    float acc[2][4][4];
    const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
    gemm_tile<true, BK, false>(g, m0, n0, 0, g.K, acc, nullptr);
    gemm_store<EPI>(g, m0, n0, acc);
}

// Weight and bias gradients of up to kGroup layers in one launch: dW = act^T g and the column
// sums of g.  K is the batch, so a layer has few tiles and long sums (256 x 256 weights: 16
// tiles of 4096 terms each); the batch is split over blockIdx.y (chunks of `chunk` rows), each
// split writes its own partial gradient and grad_reduce_kernel adds the splits in order
// (deterministic).  With one launch per layer, unsplit, element-wise strided loads and a
// separate column-sum kernel of 8 blocks, the gradients of a 4096-row minibatch took 1520 us; with
// this 131 us: 11 dependent launches of 12 us on average, each mostly ramp-up and tail (the products
// themselves are 3.5 GFLOP, a few microseconds of tensor time).
constexpr int kGroup = 8;
struct WgradGroup {
    Gemm g[kGroup];
    long long woff[kGroup], boff[kGroup];
    int tile0[kGroup + 1];    // first tile of each layer
    int layers, chunk;
    long long stride;         // floats between the splits' partial gradients
    float *part;
};

__global__ void __launch_bounds__(128) wgrad_kernel(const __grid_constant__ WgradGroup w)
{
    int l = 0;
    while (l + 1 < w.layers && (int)blockIdx.x >= w.tile0[l + 1]) ++l;
    Gemm g = w.g[l];
    const int tile = blockIdx.x - w.tile0[l], nt = (g.N + TN - 1) / TN;
    const int m0 = tile / nt * TM, n0 = tile % nt * TN;
    const int kb = blockIdx.y * w.chunk, ke = min(g.K, kb + w.chunk);
    float *part = w.part + blockIdx.y * w.stride;
    g.out = part + w.woff[l];
    float acc[2][4][4], csum = 0.0f;
    gemm_tile<false, false, true>(g, m0, n0, kb, ke, acc, m0 == 0 ? &csum : nullptr);
    gemm_store<EPI_STORE>(g, m0, n0, acc);
    if (m0 == 0 && threadIdx.x < TN && n0 + (int)threadIdx.x < g.N)
        part[w.boff[l] + n0 + threadIdx.x] = csum;
}

__global__ void grad_reduce_kernel(const float *part, long long stride, int splits, float *grad,
                                   long long n)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        float s = part[i];
        for (int k = 1; k < splits; ++k) s += part[k * stride + i];
        grad[i] = s;
    }
}

// x (FP32) -> BF16 ((x - mean) / std per column)
__global__ void normalize_kernel(const float *x, long long ldx, const float *mean,
                                 const float *inv_std, __nv_bfloat16 *xb, int B, int D)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)B * D;
         i += (long long)gridDim.x * blockDim.x) {
        const long long b = i / D;
        const int d = (int)(i - b * D);
        xb[i] = __float2bfloat16((x[b * ldx + d] - mean[d]) * inv_std[d]);
    }
}

// output gradient g = mask (y - t / scale) / B (BF16) and the loss sum of
// mask (y - t / scale)^2 / (2B)
__global__ void output_grad_kernel(const float *y, const float *t, const float *mask,
                                   const float *scale, __nv_bfloat16 *g, int B, int N,
                                   float *loss)
{
    float part = 0.0f;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)B * N;
         i += (long long)gridDim.x * blockDim.x) {
        const int n = (int)(i % N);
        const float r = y[i] - t[i] / scale[n];
        const float d = mask[i] * r;
        g[i] = __float2bfloat16(d / (float)B);
        part += d * r;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if ((threadIdx.x & 31) == 0 && loss) atomicAdd(loss, 0.5f * part / (float)B);
}

// Per-column statistics of a B x D FP32 matrix (leading dimension ld), one block of 256
// threads per column, FP64 partial sums reduced in a fixed tree order (deterministic).
// mode 1: mean and 1 / std (std < 1e-6 gives 1); mode 0: scale = root mean square (0 -> 1).
__global__ void column_stats_kernel(const float *x, long long ld, int B, int D, float *mean,
                                    float *second, int mode)
{
    __shared__ double s1[256], s2[256];
    const int d = blockIdx.x;
    if (d >= D) return;
    double a = 0.0, q = 0.0;
    for (int b = threadIdx.x; b < B; b += blockDim.x) {
        const double v = (double)x[(long long)b * ld + d];
        a += v;
        q += v * v;
    }
    s1[threadIdx.x] = a;
    s2[threadIdx.x] = q;
    __syncthreads();
    for (int w = blockDim.x / 2; w; w >>= 1) {
        if ((int)threadIdx.x < w) { s1[threadIdx.x] += s1[threadIdx.x + w]; s2[threadIdx.x] += s2[threadIdx.x + w]; }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double mu = s1[0] / B, ms = s2[0] / B;
        if (mode == 1) {
            const double var = ms - mu * mu;
            const double sd = var > 1e-12 ? sqrt(var) : 1.0;
            mean[d] = (float)mu;
            second[d] = (float)(1.0 / sd);
        } else {
            const double rms = sqrt(ms);
            second[d] = rms > 0.0 ? (float)rms : 1.0f;
        }
    }
}

// Adam (bias-corrected) on the FP32 master parameters; refreshes their BF16 copies
__global__ void adam_kernel(float *p, __nv_bfloat16 *pb, const float *grad, float *m, float *v,
                            long long n, float lr, float beta1, float beta2, float eps, float c1,
                            float c2)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const float gr = grad[i];
        const float mi = beta1 * m[i] + (1.0f - beta1) * gr;
        const float vi = beta2 * v[i] + (1.0f - beta2) * gr * gr;
        m[i] = mi;
        v[i] = vi;
        const float w = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        p[i] = w;
        if (pb) pb[i] = __float2bfloat16(w);
    }
}

__global__ void to_bf16_kernel(const float *x, __nv_bfloat16 *y, long long n)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        y[i] = __float2bfloat16(x[i]);
}

}  // namespace wsn
