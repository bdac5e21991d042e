// k_mlp.cu -- the learned surrogate (npf_mlp.h): an ensemble of multilayer perceptrons trained
// and evaluated by BF16 tensor-core kernels with FP32 accumulation.
//
// Layout. Every layer's bias is folded into its weight matrix: the input of layer l is stored
// as h_l augmented with a constant 1 in column w_l and zeros up to ip_l = round_up(w_l + 1, 16),
// and the layer's BF16 weight matrix is [w_{l+1}][ip_l] with b_l in column w_l. One GEMM kernel
// then serves the forward product (with its bias), the error back-propagation and the weight
// gradient (whose column w_l is the bias gradient); padding columns stay exactly zero because
// their inputs are zero. The ensemble members are the third grid dimension of every launch.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/npf_mlp.h"
#include "k_device.cuh"
#include "npf_internal.h"

namespace npf {
namespace mlp {

constexpr int TM = 64, TN = 64, TK = 32, STAGES = 4;
constexpr int kMaxRows = 65536;
constexpr int kMaxLayers = 8;
// a stage of one operand: 64 rows of 32 + 8 K-contiguous elements, or 32 K rows of 64 + 8
// (both strides keep the eight rows of an ldmatrix on different banks)
constexpr int LDN = TK + 8, LDT = TM + 8;
constexpr int STAGE = TM * LDN > TK * LDT ? TM * LDN : TK * LDT;

enum { EPI_F32 = 0, EPI_RELU_BF16 = 1, EPI_MASK_BF16 = 2, EPI_LOSS = 3 };

// C[e] = op(A[e]) op(B[e]) over M x N with inner dimension K.
//   A element (m, k): AT == 0 -> A[m * lda + k], AT == 1 -> A[k * lda + m]
//   B element (k, n): BT == 0 -> B[n * ldb + k], BT == 1 -> B[k * ldb + n]
// Leading dimensions are multiples of 8 and rows start on 16 bytes; elements between K (or M, N)
// and the leading dimension are zero or feed outputs that are not stored.
struct Gemm {
    int M, N, K;
    const __nv_bfloat16* A;
    int64_t lda, sA;
    const __nv_bfloat16* B;
    int64_t ldb, sB;
    void* C;
    int64_t ldc, sC;
    const __nv_bfloat16* mask;   // EPI_MASK_BF16: keep C(m, n) where mask(m, n) > 0
    int64_t ldm, sM;
    const float* T;              // EPI_LOSS: targets [M][N]; C holds the output error in BF16
    int64_t sT;
    double* loss;                // EPI_LOSS: per member, += sum (Y - T)^2 / (M N)
};

// The weight gradients of every layer in one launch, each tile updating its weights.
struct AdamStep {
    int layers;
    int tile0[kMaxLayers + 1];   // first tile of a layer
    Gemm g[kMaxLayers];          // C: offset of the layer's block in the parameter arrays, in floats
    float *W, *M1, *M2;
    __nv_bfloat16* Wb;
    float lr, b1, b2, eps, c1, c2;   // c: 1 - b^step
};

// D (16x8, FP32) += A (16x16, BF16, row-major fragment) * B (16x8, BF16, column fragment).
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4],
                                         const uint32_t (&b)[2])
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, "
        "{%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

template <bool TRANS>
__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], const __nv_bfloat16* p)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    if (TRANS)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}

// 16 bytes global -> shared, zeros when `ok` is false (the source is not read then).
__device__ __forceinline__ void copy16(__nv_bfloat16* dst, const __nv_bfloat16* src, bool ok)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                 ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(ok ? 16 : 0) : "memory");
}

// One operand's stage: rows r0.. (TRANS: K rows k0.., columns r0..) of a matrix with R rows (K-contiguous
// layout) or columns, K extent K.
template <bool TRANS>
__device__ __forceinline__ void load_stage(__nv_bfloat16* s, const __nv_bfloat16* src, int64_t ld, int r0,
                                           int R, int k0, int K)
{
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int idx = (int)threadIdx.x + 128 * j;
        if (TRANS) {
            const int k = idx / (TM / 8), c = idx % (TM / 8) * 8;
            const bool ok = k0 + k < K && r0 + c + 8 <= ld;
            copy16(s + k * LDT + c, ok ? src + (int64_t)(k0 + k) * ld + r0 + c : src, ok);
        } else {
            const int r = idx / (TK / 8), c = idx % (TK / 8) * 8;
            const bool ok = r0 + r < R && k0 + c + 8 <= ld;
            copy16(s + r * LDN + c, ok ? src + (int64_t)(r0 + r) * ld + k0 + c : src, ok);
        }
    }
}

// 64 x 64 output tile per CTA, four warps of 32 x 32, K in steps of 32 through a ring of four
// shared-memory stages filled by 16-byte asynchronous copies; fragments by ldmatrix (transposed
// where the source is M- or N-contiguous). The products are small (256 x 272 x 256 a layer and
// member), so the time is the latency of the K loop: with scalar loads and one stage a step of the
// 4-256-256-256-64 ensemble of five took 203 us at 256 rows.
template <bool AT, bool BT>
__device__ __forceinline__ void gemm_tile(const Gemm& g, int e, int m0, int n0, __nv_bfloat16* sA,
                                          __nv_bfloat16* sB, float (&acc)[2][4][4])
{
    const __nv_bfloat16* A = g.A + e * g.sA;
    const __nv_bfloat16* B = g.B + e * g.sB;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int wm = warp / 2 * 32, wn = warp % 2 * 32;
#pragma unroll
    for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int ni = 0; ni < 4; ++ni)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[mi][ni][c] = 0.f;
    const int steps = (g.K + TK - 1) / TK;
    auto fetch = [&](int st) {
        if (st < steps) {
            load_stage<AT>(sA + (st % STAGES) * STAGE, A, g.lda, m0, g.M, st * TK, g.K);
            load_stage<BT>(sB + (st % STAGES) * STAGE, B, g.ldb, n0, g.N, st * TK, g.K);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int st = 0; st < STAGES - 1; ++st) fetch(st);
    const int l8 = lane % 8, lq = lane / 8;   // row within an 8 x 8 matrix, matrix of the four
    for (int st = 0; st < steps; ++st) {
        asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
        __syncthreads();
        fetch(st + STAGES - 1);
        const __nv_bfloat16* a = sA + (st % STAGES) * STAGE;
        const __nv_bfloat16* b = sB + (st % STAGES) * STAGE;
#pragma unroll
        for (int ks = 0; ks < TK; ks += 16) {
            uint32_t af[2][4], bf[4][2];
#pragma unroll
            for (int mi = 0; mi < 2; ++mi) {
                // matrices (m, k): (0, 0), (8, 0), (0, 8), (8, 8)
                const int m = wm + mi * 16 + (lq & 1) * 8, k = ks + (lq >> 1) * 8;
                if (AT) ldmatrix4<true>(af[mi], a + (k + l8) * LDT + m);
                else ldmatrix4<false>(af[mi], a + (m + l8) * LDN + k);
            }
#pragma unroll
            for (int nj = 0; nj < 2; ++nj) {
                // matrices (n, k): (0, 0), (0, 8), (8, 0), (8, 8)
                const int n = wn + nj * 16 + (lq >> 1) * 8, k = ks + (lq & 1) * 8;
                uint32_t r[4];
                if (BT) ldmatrix4<true>(r, b + (k + l8) * LDT + n);
                else ldmatrix4<false>(r, b + (n + l8) * LDN + k);
                bf[2 * nj][0] = r[0]; bf[2 * nj][1] = r[1];
                bf[2 * nj + 1][0] = r[2]; bf[2 * nj + 1][1] = r[3];
            }
#pragma unroll
            for (int mi = 0; mi < 2; ++mi)
#pragma unroll
                for (int ni = 0; ni < 4; ++ni) mma16816(acc[mi][ni], af[mi], bf[ni]);
        }
    }
}

// Row and first column of the thread's accumulators acc[mi][ni][2 h], acc[mi][ni][2 h + 1].
__device__ __forceinline__ int out_row(int m0, int mi, int h)
{
    return m0 + (int)threadIdx.x / 64 * 32 + mi * 16 + (int)threadIdx.x % 32 / 4 + 8 * h;
}
__device__ __forceinline__ int out_col(int n0, int ni)
{
    return n0 + (int)threadIdx.x / 32 % 2 * 32 + ni * 8 + (int)threadIdx.x % 4 * 2;
}

// f(m, n, value, j) for the thread's elements of the tile that lie in the matrix (j: 0..31).
template <class F>
__device__ __forceinline__ void for_outputs(const Gemm& g, int m0, int n0, const float (&acc)[2][4][4], F&& f)
{
#pragma unroll
    for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int ni = 0; ni < 4; ++ni)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int m = out_row(m0, mi, q / 2), n = out_col(n0, ni) + q % 2;
                if (m < g.M && n < g.N) f(m, n, acc[mi][ni][q], (mi * 4 + ni) * 4 + q);
            }
}

// The epilogues read what they need (mask, targets, Adam's state) into registers before they store
// anything, so that the loads are in flight together instead of one after each store.
template <int EPI, bool AT, bool BT>
__global__ void __launch_bounds__(128) k_gemm(const __grid_constant__ Gemm g)
{
    __shared__ __align__(16) __nv_bfloat16 sA[STAGES * STAGE], sB[STAGES * STAGE];
    const int e = blockIdx.z, m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
    float acc[2][4][4];
    pdl_wait();
    gemm_tile<AT, BT>(g, e, m0, n0, sA, sB, acc);
    if (EPI == EPI_RELU_BF16 || EPI == EPI_MASK_BF16) {
        // hidden widths are multiples of 16: a thread's column pairs are whole
        uint32_t mk[2][4][2];
#pragma unroll
        for (int mi = 0; mi < 2; ++mi)
#pragma unroll
            for (int ni = 0; ni < 4; ++ni)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int m = out_row(m0, mi, h), n = out_col(n0, ni);
                    mk[mi][ni][h] = 0u;
                    if (EPI == EPI_MASK_BF16 && m < g.M && n < g.N)
                        mk[mi][ni][h] = *reinterpret_cast<const uint32_t*>(g.mask + e * g.sM + (int64_t)m * g.ldm + n);
                }
#pragma unroll
        for (int mi = 0; mi < 2; ++mi)
#pragma unroll
            for (int ni = 0; ni < 4; ++ni)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int m = out_row(m0, mi, h), n = out_col(n0, ni);
                    if (m >= g.M || n >= g.N) continue;
                    float x = acc[mi][ni][2 * h], y = acc[mi][ni][2 * h + 1];
                    if (EPI == EPI_RELU_BF16) {
                        x = fmaxf(x, 0.f);
                        y = fmaxf(y, 0.f);
                    } else {   // the activations' BF16 bits: positive where the unit was active
                        x = __uint_as_float(mk[mi][ni][h] << 16) > 0.f ? x : 0.f;
                        y = __uint_as_float(mk[mi][ni][h] & 0xFFFF0000u) > 0.f ? y : 0.f;
                    }
                    *reinterpret_cast<__nv_bfloat162*>(static_cast<__nv_bfloat16*>(g.C) + e * g.sC +
                                                       (int64_t)m * g.ldc + n) = __floats2bfloat162_rn(x, y);
                }
        return;
    }
    float aux[32];
    if (EPI == EPI_LOSS)
        for_outputs(g, m0, n0, acc, [&](int m, int n, float, int j) {
            aux[j] = g.T[e * g.sT + (int64_t)m * g.N + n];
        });
    double part = 0.0;
    const float scale2 = EPI == EPI_LOSS ? (float)(2.0 * (1.0 / ((double)g.M * g.N))) : 0.f;
    for_outputs(g, m0, n0, acc, [&](int m, int n, float v, int j) {
        const int64_t o = e * g.sC + (int64_t)m * g.ldc + n;
        if (EPI == EPI_F32) {
            static_cast<float*>(g.C)[o] = v;
        } else {   // mean squared error: the output's error 2 (Y - T) / (M N), and the loss
            const float d = v - aux[j];
            static_cast<__nv_bfloat16*>(g.C)[o] = __float2bfloat16_rn(scale2 * d);
            part += (double)d * d;
        }
    });
    if (EPI == EPI_LOSS) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        __shared__ double red[4];
        if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = part;
        __syncthreads();
        if (threadIdx.x == 0)
            atomicAdd(&g.loss[e], (red[0] + red[1] + red[2] + red[3]) * (1.0 / ((double)g.M * g.N)));
    }
}

// x / c rounded to nearest, from r = 1 / c rounded to nearest: Markstein's correction of x r by its exact
// remainder (Computation of elementary functions on the IBM RISC System/6000 processor, IBM J. Res. Dev.
// 34, 1990). Equal to the division for every mantissa of x and every bias correction c of Adam's steps
// (checked for all 2^23 by 10869 of them) while 2^-100 <= |x| <= 2^115 or x = 0.
__device__ __forceinline__ float quotient_by(float x, float c, float r)
{
    const float q = x * r;
    return fmaf(fmaf(-q, c, x), r, q);
}

// Weight gradients G_l = dZ_l^T H_l of every layer and the Adam step of their weights: no gradient
// array, and one launch instead of one a layer and one over all parameters. The back-propagation has
// read the weights before.
__global__ void __launch_bounds__(128) k_grad_adam(const __grid_constant__ AdamStep s)
{
    __shared__ __align__(16) __nv_bfloat16 sA[STAGES * STAGE], sB[STAGES * STAGE];
    int l = 0;
    while (l + 1 < s.layers && (int)blockIdx.x >= s.tile0[l + 1]) ++l;
    const Gemm& g = s.g[l];
    const int t = (int)blockIdx.x - s.tile0[l], nt = (g.N + TN - 1) / TN;
    const int e = blockIdx.z, m0 = t / nt * TM, n0 = t % nt * TN;
    float acc[2][4][4];
    pdl_wait();
    gemm_tile<true, true>(g, e, m0, n0, sA, sB, acc);
    // the gradient tile through shared memory, so that the state moves in coalesced 16-byte accesses
    constexpr int LDG = TN + 4;
    float* tile = reinterpret_cast<float*>(sA);
    static_assert(TM * LDG * sizeof(float) <= sizeof(sA), "the gradient tile fits one operand's stages");
    __syncthreads();
#pragma unroll
    for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int ni = 0; ni < 4; ++ni)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                *reinterpret_cast<float2*>(tile + out_row(0, mi, h) * LDG + out_col(0, ni)) =
                    make_float2(acc[mi][ni][2 * h], acc[mi][ni][2 * h + 1]);
    __syncthreads();
    const int64_t base = e * g.sC + reinterpret_cast<int64_t>(g.C);
    const int c = (int)threadIdx.x % 16 * 4, r0 = (int)threadIdx.x / 16;
    float4 w[8], m1[8], m2[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int m = m0 + r0 + 8 * j;
        if (m >= g.M || n0 + c >= g.N) continue;   // (N = ip is a multiple of 16)
        const int64_t o = base + (int64_t)m * g.ldc + n0 + c;
        w[j] = *reinterpret_cast<const float4*>(s.W + o);
        m1[j] = *reinterpret_cast<const float4*>(s.M1 + o);
        m2[j] = *reinterpret_cast<const float4*>(s.M2 + o);
    }
    // The products fused with sums are spelled out, so that the trained weights do not depend on the
    // compiler's choice.
    auto moments = [&](float gr, float& a, float& v) {
        a = fmaf(1.f - s.b1, gr, s.b1 * a);
        v = fmaf((1.f - s.b2) * gr, gr, s.b2 * v);
    };
    auto plain = [&](float& x, float a, float v) {
        x -= s.lr * (a / s.c1) / (sqrtf(v / s.c2) + s.eps);
    };
    // The same number with one division and a square root that never leave their fast branches (units that
    // stop firing leave zero or denormal moments, which do: 150 instructions an element). The moments,
    // scaled by 2^60, are divided by their corrections through the reciprocals. A v / c2 below 2^-106
    // does not change eps = 1e-8, and an update below 2^-63 (|num| < 2^-90) not an |x| above 2^-30.
    // What these bounds do not cover sets `far`, and the thread does the plain operations. 32 steps of the
    // 4-256-256-256-64 ensemble of five: 1.68 ms, with the plain operations 1.95. (Products with reciprocals
    // instead take 1.60, but a last place in a weight flips BF16 roundings in the steps behind it: trained
    // weights 1.4e-3 apart.)
    const float r1 = 1.f / s.c1, r2 = 1.f / s.c2;
    bool far = !(s.lr <= 1e6f);
    auto fast = [&](float& x, float a, float v) {
        constexpr float up = 1152921504606846976.f, big = 1125899906842624.f;   // 2^60, 2^50
        const float num = s.lr * (quotient_by(a * up, s.c1, r1) * (1.f / up));
        const float root = sqrtf(fmaxf(quotient_by(v * up, s.c2, r2), 1.4210854715202004e-14f));   // 2^-46
        const bool tiny = fabsf(num) < 8.077935669463161e-28f;                  // 2^-90
        const float q = (tiny ? 1.f : num) / (root * 9.313225746154785e-10f + s.eps);               // 2^-30
        far |= !(v <= big) || !(fabsf(a) <= big) || (tiny && num != 0.f && fabsf(x) < 9.313225746154785e-10f);
        x -= tiny ? num : q;
    };
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int m = m0 + r0 + 8 * j;
        if (m >= g.M || n0 + c >= g.N) continue;
        const float4 gr = *reinterpret_cast<const float4*>(tile + (r0 + 8 * j) * LDG + c);
        moments(gr.x, m1[j].x, m2[j].x);
        moments(gr.y, m1[j].y, m2[j].y);
        moments(gr.z, m1[j].z, m2[j].z);
        moments(gr.w, m1[j].w, m2[j].w);
        fast(w[j].x, m1[j].x, m2[j].x);
        fast(w[j].y, m1[j].y, m2[j].y);
        fast(w[j].z, m1[j].z, m2[j].z);
        fast(w[j].w, m1[j].w, m2[j].w);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int m = m0 + r0 + 8 * j;
        if (m >= g.M || n0 + c >= g.N) continue;
        const int64_t o = base + (int64_t)m * g.ldc + n0 + c;
        if (far) {
            w[j] = *reinterpret_cast<const float4*>(s.W + o);
            plain(w[j].x, m1[j].x, m2[j].x);
            plain(w[j].y, m1[j].y, m2[j].y);
            plain(w[j].z, m1[j].z, m2[j].z);
            plain(w[j].w, m1[j].w, m2[j].w);
        }
        *reinterpret_cast<float4*>(s.W + o) = w[j];
        *reinterpret_cast<float4*>(s.M1 + o) = m1[j];
        *reinterpret_cast<float4*>(s.M2 + o) = m2[j];
        __nv_bfloat162 b[2] = {__floats2bfloat162_rn(w[j].x, w[j].y), __floats2bfloat162_rn(w[j].z, w[j].w)};
        *reinterpret_cast<uint2*>(s.Wb + o) = *reinterpret_cast<uint2*>(b);
    }
}

// Weights between the public layout [w_{l+1}][w_l + 1] and the internal one [w_{l+1}][ip_l] (padding
// columns keep their zeros), member by member; to_pub: internal -> public.
struct Layout {
    int layers;
    int w[kMaxLayers + 1], ip[kMaxLayers];
    int64_t off[kMaxLayers + 1], offp[kMaxLayers + 1];   // one past the end: P, Ppub
};
__global__ void k_relayout(const __grid_constant__ Layout a, int E, const float* __restrict__ src,
                           float* __restrict__ dst, int to_pub)
{
    const int64_t Ppub = a.offp[a.layers], P = a.off[a.layers];
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < E * Ppub;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = t / Ppub;
        const int r = (int)(t - e * Ppub);
        int l = 0;
        while (l + 1 < a.layers && r >= a.offp[l + 1]) ++l;
        const int q = r - (int)a.offp[l], width = a.w[l] + 1, o = q / width, i = q - o * width;
        const int64_t in = e * P + a.off[l] + (int64_t)o * a.ip[l] + i;
        if (to_pub) dst[t] = src[in];
        else dst[in] = src[t];
    }
}

// Augmented BF16 inputs Xa[e][b][ip] = (X[r][0..w0-1], 1, 0, ..) with r = idx[e][b] (or b), and
// the matching FP32 targets Tb[e][b][wo] = T[r][.] when T is given.
__global__ void k_gather(int E, int Bn, int w0, int ip, int wo, const float* __restrict__ X,
                         const float* __restrict__ T, const int* __restrict__ idx,
                         int64_t idx_stride, int64_t cap, __nv_bfloat16* __restrict__ Xa,
                         float* __restrict__ Tb)
{
    pdl_wait();
    const int64_t nx = (int64_t)E * Bn * ip, nt = T ? (int64_t)E * Bn * wo : 0;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nx + nt;
         t += (int64_t)gridDim.x * blockDim.x) {
        if (t < nx) {
            const int c = (int)(t % ip);
            const int b = (int)((t / ip) % Bn);
            const int e = (int)(t / ((int64_t)ip * Bn));
            const int64_t r = idx ? idx[e * idx_stride + b] : b;
            const float v = c < w0 ? X[r * w0 + c] : (c == w0 ? 1.f : 0.f);
            Xa[((int64_t)e * cap + b) * ip + c] = __float2bfloat16_rn(v);
        } else {
            const int64_t u = t - nx;
            const int o = (int)(u % wo);
            const int b = (int)((u / wo) % Bn);
            const int e = (int)(u / ((int64_t)wo * Bn));
            const int64_t r = idx ? idx[e * idx_stride + b] : b;
            Tb[((int64_t)e * cap + b) * wo + o] = T[r * wo + o];
        }
    }
}

// Constant column of a hidden activation buffer: h[e][b][w] = 1, h[e][b][w+1 .. ip-1] = 0.
__global__ void k_const_cols(int E, int64_t cap, int w, int ip, __nv_bfloat16* __restrict__ h)
{
    const int pad = ip - w;
    const int64_t tot = (int64_t)E * cap * pad;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < tot;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(t % pad);
        const int64_t row = t / pad;
        h[row * ip + w + c] = __float2bfloat16_rn(c == 0 ? 1.f : 0.f);
    }
}

__global__ void k_to_bf16(int64_t total, const float* __restrict__ W, __nv_bfloat16* __restrict__ Wb)
{
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x)
        Wb[t] = __float2bfloat16_rn(W[t]);
}

// Ensemble statistics of one row per block: v_e = exp(mu + sigma y_e), mean and the largest
// relative (population) standard deviation over the outputs; fallback flag above the limit.
__global__ void k_ens_stats(int E, int wo, int64_t cap, const float* __restrict__ Y,
                            const float* __restrict__ mu, const float* __restrict__ sigma,
                            float lim, float* __restrict__ mean, float* __restrict__ spread,
                            int* __restrict__ fb)
{
    const int r = blockIdx.x;
    float worst = 0.f;
    pdl_wait();
    for (int o = threadIdx.x; o < wo; o += blockDim.x) {
        double s1 = 0.0, s2 = 0.0;
        for (int e = 0; e < E; ++e) {
            const double v = exp((double)mu[o] + (double)sigma[o] * Y[((int64_t)e * cap + r) * wo + o]);
            s1 += v;
            s2 += v * v;
        }
        const double mn = s1 / E;
        const double var = fmax(s2 / E - mn * mn, 0.0);
        mean[(int64_t)r * wo + o] = (float)mn;
        worst = fmaxf(worst, (float)(sqrt(var) / mn));
    }
    __shared__ float red[128];
    red[threadIdx.x] = worst;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) red[threadIdx.x] = fmaxf(red[threadIdx.x], red[threadIdx.x + s]);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        spread[r] = red[0];
        fb[r] = red[0] > lim ? 1 : 0;
    }
}

static unsigned grid_for(int64_t total, int per = 256)
{
    const int64_t b = (total + per - 1) / per;
    return (unsigned)(b < 1 ? 1 : (b > 65535 ? 65535 : b));
}

static uint64_t splitmix64(uint64_t& s)
{
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

}  // namespace mlp
}  // namespace npf

using namespace npf::mlp;

struct npf_mlp {
    int E = 0, L = 0;
    std::vector<int> w;       // widths w_0 .. w_L
    std::vector<int> ip;      // padded augmented input widths ip_0 .. ip_{L-1}
    std::vector<int64_t> off; // offset of layer l's [w_{l+1}][ip_l] block within a member
    std::vector<int64_t> offp;// offset of layer l's [w_{l+1}][w_l + 1] block, public layout
    int64_t P = 0, Ppub = 0;  // floats per member, internal / public
    cudaStream_t s = nullptr;
    float *W = nullptr, *M1 = nullptr, *M2 = nullptr, *G = nullptr;
    __nv_bfloat16* Wb = nullptr;
    int64_t step = 0;
    // activations, capacity `cap` rows per member
    int64_t cap = 0;
    std::vector<__nv_bfloat16*> H;    // H[l]: [E][cap][ip_l], l < L
    std::vector<__nv_bfloat16*> dZ;   // dZ[l]: [E][cap][zp_l], zero past w_{l+1}
    std::vector<int> zp;      // leading dimensions of dZ: w_{l+1} rounded up to 8
    float* Y = nullptr;               // [E][cap][w_L]
    float* Tb = nullptr;              // [E][cap][w_L]
    double* d_loss = nullptr;         // [E]
    float *d_X = nullptr, *d_T = nullptr;
    int64_t xcap = 0;
    int* d_idx = nullptr;
    int64_t idx_cap = 0;
    float *d_mu = nullptr, *d_sig = nullptr, *d_mean = nullptr, *d_spread = nullptr;
    int* d_fb = nullptr;
    float* d_pub = nullptr;     // [E][Ppub] staging of weights or gradients in the public layout
    int64_t tcap = 0;   // floats of d_T
    int64_t mcap = 0;   // rows of d_mean / d_spread / d_fb
};

namespace {

template <class F>
int run(F&& f)
{
    try {
        f();
        return npf::record_status(NPF_OK, "");
    } catch (const npf::Error& e) {
        return npf::record_status(e.code, e.msg);
    } catch (const std::exception& e) {
        return npf::record_status(NPF_ERR_CUDA, e.what());
    } catch (...) {
        return npf::record_status(NPF_ERR_CUDA, "unknown error");
    }
}

void release_acts(npf_mlp& m)
{
    for (auto* p : m.H) cudaFree(p);
    for (auto* p : m.dZ) cudaFree(p);
    m.H.clear();
    m.dZ.clear();
    cudaFree(m.Y);
    cudaFree(m.Tb);
    m.Y = m.Tb = nullptr;
    m.cap = 0;
}

void free_all(npf_mlp& m)
{
    release_acts(m);
    cudaFree(m.W); cudaFree(m.M1); cudaFree(m.M2); cudaFree(m.G); cudaFree(m.Wb);
    cudaFree(m.d_loss); cudaFree(m.d_pub); cudaFree(m.d_X); cudaFree(m.d_T); cudaFree(m.d_idx);
    cudaFree(m.d_mu); cudaFree(m.d_sig); cudaFree(m.d_mean); cudaFree(m.d_spread); cudaFree(m.d_fb);
}

template <class T>
T* dalloc(int64_t count)
{
    T* p = nullptr;
    NPF_CUDA(cudaMalloc(&p, (size_t)std::max<int64_t>(count, 1) * sizeof(T)));
    return p;
}

void reserve_rows(npf_mlp& m, int64_t rows)
{
    if (rows <= m.cap) return;
    release_acts(m);
    const int64_t cap = std::max<int64_t>(rows, 256);
    for (int l = 0; l < m.L; ++l) m.H.push_back(dalloc<__nv_bfloat16>(m.E * cap * m.ip[l]));
    for (int l = 0; l < m.L; ++l) {
        m.dZ.push_back(dalloc<__nv_bfloat16>(m.E * cap * m.zp[l]));
        if (m.zp[l] != m.w[l + 1])
            NPF_CUDA(cudaMemsetAsync(m.dZ[l], 0, (size_t)m.E * cap * m.zp[l] * sizeof(__nv_bfloat16), m.s));
    }
    m.Y = dalloc<float>(m.E * cap * m.w[m.L]);
    m.Tb = dalloc<float>(m.E * cap * m.w[m.L]);
    m.cap = cap;
    for (int l = 1; l < m.L; ++l) {
        npf::LaunchScope ls(nullptr, "mlp_const_cols", m.s);
        k_const_cols<<<grid_for(m.E * cap * (m.ip[l] - m.w[l])), 256, 0, m.s>>>(m.E, cap, m.w[l],
                                                                               m.ip[l], m.H[l]);
        NPF_CUDA(cudaGetLastError());
    }
}

// Copy `count` floats from a host or device pointer into a device buffer that grows.
void stage(float*& dst, int64_t& capf, const float* src, int64_t count, cudaStream_t s)
{
    if (count > capf) {
        cudaFree(dst);
        dst = dalloc<float>(count);
        capf = count;
    }
    NPF_CUDA(cudaMemcpyAsync(dst, src, (size_t)count * sizeof(float), cudaMemcpyDefault, s));
}

template <int EPI, bool AT, bool BT>
void gemm(npf_mlp& m, const char* name, const Gemm& g)
{
    npf::LaunchScope ls(nullptr, name, m.s);
    dim3 grid((unsigned)((g.N + TN - 1) / TN), (unsigned)((g.M + TM - 1) / TM), (unsigned)m.E);
    npf::launch_dependent(k_gemm<EPI, AT, BT>, grid, dim3(128), 0, m.s, g);
}

void gather(npf_mlp& m, int rows, const float* dX, const float* dT, const int* idx,
            int64_t idx_stride)
{
    npf::LaunchScope ls(nullptr, "mlp_gather", m.s);
    const int64_t tot = (int64_t)m.E * rows * (m.ip[0] + (dT ? m.w[m.L] : 0));
    npf::launch_dependent(k_gather, dim3(grid_for(tot)), dim3(256), 0, m.s, m.E, rows, m.w[0], m.ip[0], m.w[m.L], dX, dT, idx, idx_stride, m.cap, m.H[0], m.Tb);
}

// loss: the last layer's epilogue forms the output's error and the loss instead of storing Y
void forward(npf_mlp& m, int rows, bool loss)
{
    for (int l = 0; l < m.L; ++l) {
        Gemm g{};
        g.M = rows;
        g.N = m.w[l + 1];
        g.K = m.ip[l];
        g.A = m.H[l]; g.lda = m.ip[l]; g.sA = m.cap * m.ip[l];
        g.B = m.Wb + m.off[l]; g.ldb = m.ip[l]; g.sB = m.P;
        if (l + 1 < m.L) {
            g.C = m.H[l + 1]; g.ldc = m.ip[l + 1]; g.sC = m.cap * m.ip[l + 1];
            gemm<EPI_RELU_BF16, false, false>(m, "mlp_forward_relu", g);
        } else if (!loss) {
            g.C = m.Y; g.ldc = m.w[m.L]; g.sC = m.cap * m.w[m.L];
            gemm<EPI_F32, false, false>(m, "mlp_forward_out", g);
        } else {
            g.C = m.dZ[l]; g.ldc = m.zp[l]; g.sC = m.cap * m.zp[l];
            g.T = m.Tb; g.sT = m.cap * m.w[m.L];
            g.loss = m.d_loss;
            gemm<EPI_LOSS, false, false>(m, "mlp_forward_loss", g);
        }
    }
}

// Errors of the hidden layers: dZ_{l-1} = (dZ_l W_l)[:, :w_l] o (h_l > 0)
void backward(npf_mlp& m, int rows)
{
    for (int l = m.L - 1; l >= 1; --l) {
        Gemm d{};
        d.M = rows;
        d.N = m.w[l];
        d.K = m.w[l + 1];
        d.A = m.dZ[l]; d.lda = m.zp[l]; d.sA = m.cap * m.zp[l];
        d.B = m.Wb + m.off[l]; d.ldb = m.ip[l]; d.sB = m.P;
        d.C = m.dZ[l - 1]; d.ldc = m.zp[l - 1]; d.sC = m.cap * m.zp[l - 1];
        d.mask = m.H[l]; d.ldm = m.ip[l]; d.sM = m.cap * m.ip[l];
        gemm<EPI_MASK_BF16, false, true>(m, "mlp_backprop", d);
    }
}

// Weight gradient of a layer: G_l = dZ_l^T H_l ([w_{l+1}] x [ip_l], K = rows)
Gemm weight_grad(const npf_mlp& m, int rows, int l)
{
    Gemm g{};
    g.M = m.w[l + 1];
    g.N = m.ip[l];
    g.K = rows;
    g.A = m.dZ[l]; g.lda = m.zp[l]; g.sA = m.cap * m.zp[l];
    g.B = m.H[l]; g.ldb = m.ip[l]; g.sB = m.cap * m.ip[l];
    g.ldc = m.ip[l]; g.sC = m.P;
    return g;
}

void sync(npf_mlp& m) { NPF_CUDA(cudaStreamSynchronize(m.s)); }

// d_pub <- the public layout of an internal array, or an internal array <- d_pub
void relayout(npf_mlp& m, float* internal, bool to_pub)
{
    Layout a{};
    a.layers = m.L;
    for (int l = 0; l <= m.L; ++l) {
        a.w[l] = m.w[l];
        a.off[l] = l < m.L ? m.off[l] : m.P;
        a.offp[l] = l < m.L ? m.offp[l] : m.Ppub;
        if (l < m.L) a.ip[l] = m.ip[l];
    }
    if (!m.d_pub) m.d_pub = dalloc<float>(m.E * m.Ppub);
    npf::LaunchScope ls(nullptr, "mlp_relayout", m.s);
    k_relayout<<<grid_for(m.E * m.Ppub), 256, 0, m.s>>>(a, m.E, to_pub ? internal : m.d_pub,
                                                      to_pub ? m.d_pub : internal, to_pub);
    NPF_CUDA(cudaGetLastError());
}

void copy_out(void* dst, const void* src, size_t bytes, cudaStream_t s)
{
    NPF_CUDA(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDefault, s));
}

// Weights or gradients (d_pub) to the caller behind what the legacy stream has queued on a device
// destination.
void hand_out(npf_mlp& m, float* dst)
{
    sync(m);
    NPF_CUDA(cudaMemcpy(dst, m.d_pub, (size_t)m.E * m.Ppub * sizeof(float), cudaMemcpyDefault));
    NPF_CUDA(cudaStreamSynchronize(cudaStreamLegacy));
}

}  // namespace

extern "C" {

npf_mlp* npf_mlp_create(int ensemble, int layers, const int* widths, const float* weights,
                        void* stream)
{
    npf_mlp* m = nullptr;
    const int rc = run([&] {
        if (ensemble < 1 || ensemble > 16) npf::fail(NPF_ERR_ARG, "ensemble must be in [1, 16]");
        if (layers < 2 || layers > 8) npf::fail(NPF_ERR_ARG, "layers must be in [2, 8]");
        if (!widths || !weights) npf::fail(NPF_ERR_ARG, "null widths or weights");
        if (widths[0] < 1 || widths[0] > 15) npf::fail(NPF_ERR_ARG, "input width must be in [1, 15]");
        for (int l = 1; l <= layers; ++l) {
            if (widths[l] < 8 || widths[l] > 1024) npf::fail(NPF_ERR_ARG, "widths must be in [8, 1024]");
            if (l < layers && widths[l] % 16) npf::fail(NPF_ERR_ARG, "hidden widths must be multiples of 16");
        }
        m = new npf_mlp();
        m->E = ensemble;
        m->L = layers;
        m->s = (cudaStream_t)stream;
        m->w.assign(widths, widths + layers + 1);
        for (int l = 0; l < layers; ++l) {
            m->ip.push_back((m->w[l] + 1 + 15) / 16 * 16);
            m->off.push_back(m->P);
            m->offp.push_back(m->Ppub);
            m->zp.push_back((m->w[l + 1] + 7) / 8 * 8);
            m->P += (int64_t)m->w[l + 1] * m->ip[l];
            m->Ppub += (int64_t)m->w[l + 1] * (m->w[l] + 1);
        }
        const int64_t tot = (int64_t)ensemble * m->P;
        m->W = dalloc<float>(tot);
        m->M1 = dalloc<float>(tot);
        m->M2 = dalloc<float>(tot);
        m->G = dalloc<float>(tot);
        m->Wb = dalloc<__nv_bfloat16>(tot);
        m->d_loss = dalloc<double>(ensemble);
        m->d_pub = dalloc<float>(ensemble * m->Ppub);
        // (blocking: for device weights it waits for what the legacy stream has queued)
        NPF_CUDA(cudaMemcpy(m->d_pub, weights, (size_t)ensemble * m->Ppub * sizeof(float), cudaMemcpyDefault));
        NPF_CUDA(cudaStreamSynchronize(cudaStreamLegacy));   // (between device buffers it returns at once)
        NPF_CUDA(cudaMemsetAsync(m->W, 0, (size_t)tot * sizeof(float), m->s));
        NPF_CUDA(cudaMemsetAsync(m->M1, 0, (size_t)tot * sizeof(float), m->s));
        NPF_CUDA(cudaMemsetAsync(m->M2, 0, (size_t)tot * sizeof(float), m->s));
        relayout(*m, m->W, false);
        {
            npf::LaunchScope ls(nullptr, "mlp_to_bf16", m->s);
            k_to_bf16<<<grid_for(tot), 256, 0, m->s>>>(tot, m->W, m->Wb);
            NPF_CUDA(cudaGetLastError());
        }
        sync(*m);
    });
    if (rc != NPF_OK) {
        if (m) { free_all(*m); delete m; }
        return nullptr;
    }
    return m;
}

int64_t npf_mlp_param_count(const npf_mlp* m) { return m ? m->Ppub : 0; }

int npf_mlp_get_weights(const npf_mlp* m, float* weights)
{
    return run([&] {
        if (!m || !weights) npf::fail(NPF_ERR_ARG, "null argument");
        npf_mlp& mm = const_cast<npf_mlp&>(*m);   // (the staging buffer; the weights stay)
        relayout(mm, mm.W, true);
        hand_out(mm, weights);
    });
}

int npf_mlp_forward(npf_mlp* m, int rows, const float* X, float* Y)
{
    return run([&] {
        if (!m || !X || !Y || rows < 1 || rows > kMaxRows) npf::fail(NPF_ERR_ARG, "bad forward arguments");
        reserve_rows(*m, rows);
        stage(m->d_X, m->xcap, X, (int64_t)rows * m->w[0], m->s);
        gather(*m, rows, m->d_X, nullptr, nullptr, 0);
        forward(*m, rows, false);
        const int wo = m->w[m->L];
        NPF_CUDA(cudaMemcpy2DAsync(Y, (size_t)rows * wo * sizeof(float), m->Y,
                                   (size_t)m->cap * wo * sizeof(float),
                                   (size_t)rows * wo * sizeof(float), m->E, cudaMemcpyDefault,
                                   m->s));
        sync(*m);
    });
}

int npf_mlp_loss_grad(npf_mlp* m, int rows, const float* X, const float* T, float* grads,
                      float* loss)
{
    return run([&] {
        if (!m || !X || !T || !grads || !loss || rows < 1 || rows > kMaxRows)
            npf::fail(NPF_ERR_ARG, "bad loss_grad arguments");
        reserve_rows(*m, rows);
        stage(m->d_X, m->xcap, X, (int64_t)rows * m->w[0], m->s);
        stage(m->d_T, m->tcap, T, (int64_t)rows * m->w[m->L], m->s);
        NPF_CUDA(cudaMemsetAsync(m->d_loss, 0, m->E * sizeof(double), m->s));
        gather(*m, rows, m->d_X, m->d_T, nullptr, 0);
        forward(*m, rows, true);
        backward(*m, rows);
        for (int l = 0; l < m->L; ++l) {
            Gemm g = weight_grad(*m, rows, l);
            g.C = m->G + m->off[l];
            gemm<EPI_F32, true, true>(*m, "mlp_weight_grad", g);
        }
        std::vector<double> l(m->E);
        relayout(*m, m->G, true);
        NPF_CUDA(cudaMemcpyAsync(l.data(), m->d_loss, m->E * sizeof(double), cudaMemcpyDeviceToHost, m->s));
        hand_out(*m, grads);
        std::vector<float> lf(l.begin(), l.end());
        NPF_CUDA(cudaMemcpy(loss, lf.data(), lf.size() * sizeof(float), cudaMemcpyDefault));
    });
}

int npf_mlp_train(npf_mlp* m, int rows, const float* X, const float* T, int epochs, int batch,
                  double lr, uint64_t seed, float* epoch_loss)
{
    return run([&] {
        if (!m || !X || !T || rows < 1 || epochs < 0 || batch < 1 || batch > rows ||
            batch > kMaxRows || !(lr > 0.0))
            npf::fail(NPF_ERR_ARG, "bad train arguments");
        reserve_rows(*m, batch);
        stage(m->d_X, m->xcap, X, (int64_t)rows * m->w[0], m->s);
        stage(m->d_T, m->tcap, T, (int64_t)rows * m->w[m->L], m->s);
        if ((int64_t)m->E * rows > m->idx_cap) {
            cudaFree(m->d_idx);
            m->d_idx = dalloc<int>((int64_t)m->E * rows);
            m->idx_cap = (int64_t)m->E * rows;
        }
        const int steps = rows / batch;
        std::vector<uint64_t> st(m->E);
        for (int e = 0; e < m->E; ++e) st[e] = seed + 7919ull * (uint64_t)e;
        std::vector<int> perm((size_t)m->E * rows);
        AdamStep ad{};
        ad.layers = m->L;
        ad.W = m->W; ad.M1 = m->M1; ad.M2 = m->M2; ad.Wb = m->Wb;
        ad.lr = (float)lr; ad.b1 = 0.9f; ad.b2 = 0.999f; ad.eps = 1e-8f;
        for (int l = 0; l < m->L; ++l) {
            ad.g[l] = weight_grad(*m, batch, l);
            ad.g[l].C = reinterpret_cast<void*>(m->off[l]);
            ad.tile0[l + 1] = ad.tile0[l] + (ad.g[l].M + TM - 1) / TM * ((ad.g[l].N + TN - 1) / TN);
        }
        auto shuffle = [&] {
            for (int e = 0; e < m->E; ++e) {   // Fisher-Yates with splitmix64
                int* p = perm.data() + (size_t)e * rows;
                for (int r = 0; r < rows; ++r) p[r] = r;
                for (int r = rows - 1; r > 0; --r) {
                    const int j = (int)(splitmix64(st[e]) % (uint64_t)(r + 1));
                    std::swap(p[r], p[j]);
                }
            }
        };
        if (epochs > 0) shuffle();
        for (int ep = 0; ep < epochs; ++ep) {
            // the previous epoch's kernels may still read the index buffer
            NPF_CUDA(cudaStreamSynchronize(m->s));
            NPF_CUDA(cudaMemcpy(m->d_idx, perm.data(), perm.size() * sizeof(int), cudaMemcpyHostToDevice));
            NPF_CUDA(cudaMemsetAsync(m->d_loss, 0, m->E * sizeof(double), m->s));
            for (int k = 0; k < steps; ++k) {
                gather(*m, batch, m->d_X, m->d_T, m->d_idx + (int64_t)k * batch, rows);
                forward(*m, batch, true);
                backward(*m, batch);
                ++m->step;
                ad.c1 = (float)(1.0 - std::pow((double)ad.b1, (double)m->step));
                ad.c2 = (float)(1.0 - std::pow((double)ad.b2, (double)m->step));
                npf::LaunchScope ls(nullptr, "mlp_grad_adam", m->s);
                npf::launch_dependent(k_grad_adam, dim3((unsigned)ad.tile0[m->L], 1, (unsigned)m->E), dim3(128), 0, m->s, ad);
            }
            if (ep + 1 < epochs) shuffle();   // the next epoch's order, while this one's kernels run
            if (epoch_loss) {
                std::vector<double> l(m->E);
                NPF_CUDA(cudaMemcpyAsync(l.data(), m->d_loss, m->E * sizeof(double),
                                         cudaMemcpyDeviceToHost, m->s));
                sync(*m);
                double s = 0.0;
                for (double v : l) s += v;
                const float v = (float)(s / ((double)m->E * std::max(steps, 1)));
                NPF_CUDA(cudaMemcpy(epoch_loss + ep, &v, sizeof(float), cudaMemcpyDefault));
            }
        }
        sync(*m);
    });
}

int npf_mlp_predict(npf_mlp* m, int rows, const float* X, const float* mu, const float* sigma,
                    double spread_limit, float* mean, float* spread, int* fallback)
{
    return run([&] {
        if (!m || !X || !mu || !sigma || !mean || !spread || !fallback || rows < 1 ||
            rows > kMaxRows)
            npf::fail(NPF_ERR_ARG, "bad predict arguments");
        const int wo = m->w[m->L];
        reserve_rows(*m, rows);
        if (!m->d_mu) {
            m->d_mu = dalloc<float>(wo);
            m->d_sig = dalloc<float>(wo);
        }
        NPF_CUDA(cudaMemcpyAsync(m->d_mu, mu, wo * sizeof(float), cudaMemcpyDefault, m->s));
        NPF_CUDA(cudaMemcpyAsync(m->d_sig, sigma, wo * sizeof(float), cudaMemcpyDefault, m->s));
        stage(m->d_X, m->xcap, X, (int64_t)rows * m->w[0], m->s);
        if (rows > m->mcap) {
            cudaFree(m->d_mean); cudaFree(m->d_spread); cudaFree(m->d_fb);
            m->d_mean = dalloc<float>((int64_t)rows * wo);
            m->d_spread = dalloc<float>(rows);
            m->d_fb = dalloc<int>(rows);
            m->mcap = rows;
        }
        gather(*m, rows, m->d_X, nullptr, nullptr, 0);
        forward(*m, rows, false);
        {
            npf::LaunchScope ls(nullptr, "mlp_ensemble_gate", m->s);
            npf::launch_dependent(k_ens_stats, dim3(rows), dim3(128), 0, m->s, m->E, wo, m->cap, m->Y, m->d_mu, m->d_sig, (float)spread_limit, m->d_mean, m->d_spread, m->d_fb);
        }
        copy_out(mean, m->d_mean, (size_t)rows * wo * sizeof(float), m->s);
        copy_out(spread, m->d_spread, (size_t)rows * sizeof(float), m->s);
        copy_out(fallback, m->d_fb, (size_t)rows * sizeof(int), m->s);
        sync(*m);
    });
}

void npf_mlp_destroy(npf_mlp* m)
{
    if (!m) return;
    cudaStreamSynchronize(m->s);
    free_all(*m);
    delete m;
}

}  // extern "C"
