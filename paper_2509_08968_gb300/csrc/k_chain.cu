// k_chain.cu -- one order's term in native FP64 with the whole chain of one (upper index, last
// output index) in a block's shared memory (orders 2 to 4).
//
// The upper index is contracted first on the packed tensor (k_chain_upper: S^i_Q = sum_j psi_ij A^j_Q,
// Algorithm 2 step 4 moved ahead). A block (i, p_N) then forms, over sorted tuples only (every
// intermediate is symmetric in the a's and in the p's it still has, pairs and triples stored in
// colexicographic rank),
//     X1[a's] = sum_a S^i_{sort(a's, a)} phi_{a p_N}          (steps 2-3)
//     order 4: X[a1 <= a2] = sum_a X1[sort(a1, a2, a)] phi_{a p_3}, for its p_3 <= p_4
//     X2[p_2 <= p_3][a1] = sum_a X[sort(a1, a)] phi_{a p_2}
//     h[p_1 <= p_2] = sum_a X2[p_2][a] phi_{a p_1} / (prod of run lengths! D)     (steps 5-11)
// and its share of Psi_N[i][k] (steps 12-19, Eq. 7); the last block of an upper index adds the
// shares in a fixed order, so results are reproducible bit for bit.
//
// Bound by the FP64 pipe (2 fused multiply-adds per clock and SM): a complex multiply-add takes 2
// clocks an SM whatever feeds it, so the operands come straight from shared memory and L1 and the
// index arithmetic of the sorted gathers hides behind them. Against the dense FP64 chain
// (k_fp64.cu) it does a third of the operations at order 3: n = 60, orders 2 and 3, 28.4 -> 9.0 ms
// (8.4 at the rate of cuBLAS's DGEMM); n = 8, order 3, 184 -> 59 us. It is faster wherever it fits in shared
// memory: order 2, n = 252 (of 255) 101 -> 62 ms; order 3, n = 66 and 92 (of 93) 58 -> 14 and 213 -> 69
// ms; order 4, n = 36 (of 37) 154 -> 15 ms. Against the tensor-core chain (eight launches and more an order)
// it is two launches, which is what small systems wait for: n = 10, orders 2 and 3, 243 -> 62 us. One
// block per (i, p_N) keeps 26 n^2 bytes at order 3, so that two blocks share an SM up to n = 65.
#include <algorithm>

#include "k_device.cuh"
#include "npf_internal.h"

namespace npf {
namespace {

constexpr int THREADS = 256;

struct ChainArgs {
    int n, nm;              // states; modes in use (the first nm)
    int ilo;                // first upper index
    int chunks;             // order 4: blocks that share one (i, p_4), taking every chunks-th p_3
    int64_t P;              // packed tuples
    const double2* S;       // [rows][P], rows from ilo on
    const int64_t* cnt;     // tuple-count table of the packed order
    const double2* U;
    const double2* W;       // reduction weights W[p][k]
    const double2* lam;
    double eps;
    int divide;
    double2* part;          // [rows][nm * chunks][n]
    unsigned* count;        // finished blocks per row (zero on entry and on exit)
    double2* out;           // [n][n]
    int accumulate;         // add to out instead of overwriting its rows
};

__host__ __device__ constexpr int tri(int b) { return b * (b + 1) / 2; }
__host__ __device__ constexpr int tet(int c) { return c * (c + 1) * (c + 2) / 6; }
__device__ __forceinline__ int pair_rank(int x, int y) { return x <= y ? tri(y) + x : tri(x) + y; }

// S[i - ilo][q] = sum_j psi_ij A[j][q], four upper indices a thread; the first block zeroes the
// counters of the chain.
__global__ void __launch_bounds__(128)
    k_chain_upper(int n, int ilo, int rows, int64_t P, const double* __restrict__ A,
                  const double2* __restrict__ V, double2* __restrict__ S, unsigned* __restrict__ count)
{
    pdl_wait();
    if (blockIdx.x == 0 && blockIdx.y == 0)
        for (int r = threadIdx.x; r < rows; r += blockDim.x) count[r] = 0u;
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int r0 = blockIdx.y * 4;
    if (q >= P) return;
    double2 acc[4] = {};
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
        const double v = A[(int64_t)j * P + q];
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (r0 + c < rows) rfma(acc[c], v, V[(int64_t)(ilo + r0 + c) * n + j]);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
        if (r0 + c < rows) S[(int64_t)(r0 + c) * P + q] = acc[c];
}

// Lanes that share one item's sum, so that few items still fill the block.
__device__ __forceinline__ int lanes_for(int items)
{
    return items > THREADS / 2 ? 1 : items > THREADS / 4 ? 2 : items > THREADS / 8 ? 4 : 8;
}

// item(it, s) = sum over s's terms; done(it, sum) on one lane per item. Every thread of the block
// runs the same number of rounds (warp shuffles).
template <class Sum, class Done>
__device__ __forceinline__ void for_items(int items, Sum&& sum, Done&& done)
{
    const int g = lanes_for(items), sub = threadIdx.x & (g - 1);
    for (int base = 0; base < items; base += THREADS / g) {
        const int it = base + (int)threadIdx.x / g;
        double2 s = make_double2(0.0, 0.0);
        if (it < items) s = sum(it, sub, g);
        for (int o = g / 2; o > 0; o >>= 1) {
            s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
            s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
        }
        if (it < items && sub == 0) done(it, s);
    }
}

template <int N>
__global__ void __launch_bounds__(THREADS) k_chain(ChainArgs a)
{
    extern __shared__ double2 sm[];
    const int n = a.n, nm = a.nm;
    double2* X1 = sm;                                            // sorted (N-1)-tuples of a's
    double2* Xp = N == 4 ? X1 + tet(n) : X1;                     // sorted pairs, then h
    double2* X2 = N == 2 ? X1 + n : Xp + tri(n);                 // [p_2][a1] (order 2: h)
    double2* psi = N == 2 ? X2 + nm : X2 + nm * n;               // [n]
    int* cn = (int*)(psi + n);                                   // counts of r-tuples in [v, n), r <= N
    unsigned* tab = (unsigned*)(cn + (N + 1) * (n + 1));         // pairs, then triples: 8 bits an index
    const int tid = threadIdx.x;
    const int b = (int)(gridDim.x - 1 - blockIdx.x);             // the largest p_N, the longest blocks, first
    const int pN = b / a.chunks, chunk = b - pN * a.chunks;
    const int row = blockIdx.y, i = a.ilo + row;
    const double2* Si = a.S + (int64_t)row * a.P;

    for (int k = tid; k < n; k += THREADS) psi[k] = make_double2(0.0, 0.0);
    if (N >= 3)
        for (int y = tid; y < n; y += THREADS)
            for (int x = 0; x <= y; ++x) tab[tri(y) + x] = (unsigned)x | (unsigned)y << 8;
    __syncthreads();
    unsigned* tab3 = tab + tri(n);
    pdl_wait();   // (the tables above need no global memory)
    for (int t = tid; t < (N + 1) * (n + 1); t += THREADS) cn[t] = (int)a.cnt[t];
    __syncthreads();
    if (N == 4) {
        for (int z = 0; z < n; ++z)
            for (int t = tid; t < tri(z + 1); t += THREADS) tab3[tet(z) + t] = tab[t] | (unsigned)z << 16;
        __syncthreads();
    }
    const int* c1 = cn + (n + 1);
    const int* c2 = c1 + (n + 1);
    const int* c3 = N >= 3 ? c2 + (n + 1) : nullptr;
    const int* c4 = N >= 4 ? c3 + (n + 1) : nullptr;

    // the last lower index: S gathered in its packed (lexicographic) order
    for_items(N == 2 ? n : N == 3 ? tri(n) : tet(n),
        [&](int it, int sub, int g) {
            double2 s = make_double2(0.0, 0.0);
            int x = it, y = 0, z = 0;
            if (N >= 3) {
                const unsigned t = N == 3 ? tab[it] : tab3[it];
                x = (int)(t & 255u); y = (int)((t >> 8) & 255u); z = (int)((t >> 16) & 255u);
            }
#pragma unroll 4
            for (int e = sub; e < n; e += g) {
                int r;
                if (N == 2) {
                    const int lo = min(x, e), hi = max(x, e);
                    r = c2[0] - c2[lo] + c1[lo] - c1[hi];
                } else if (N == 3) {
                    const int lo = min(x, e), hi = max(y, e), mid = x + y + e - lo - hi;
                    r = c3[0] - c3[lo] + c2[lo] - c2[mid] + c1[mid] - c1[hi];
                } else {
                    const int lo = min(x, e), hi = max(z, e);
                    const int m = max(x, e), w = min(z, e);       // middle two of (x, e, y, z): sort (m or w, y)
                    const int p = e <= y ? m : y, q = e <= y ? y : w;
                    r = c4[0] - c4[lo] + c3[lo] - c3[p] + c2[p] - c2[q] + c1[q] - c1[hi];
                }
                cfma(s, Si[r], a.U[(int64_t)e * n + pN]);
            }
            return s;
        },
        [&](int it, double2 s) { X1[it] = s; });
    __syncthreads();

    // h of (p_1, .., p_N) from the contracted value: 1 / prod(run lengths)! and the clamped divide
    auto entry = [&](double2 v, int den, double2 sigma) {
        const double f = 1.0 / (double)den;
        v.x *= f;
        v.y *= f;
        if (a.divide) v = cdiv_smith(v, clamp_denominator(csub(sigma, a.lam[i]), a.eps));
        return v;
    };

    if (N == 2) {
        for_items(pN + 1,
            [&](int p1, int sub, int g) {
                double2 s = make_double2(0.0, 0.0);
                for (int e = sub; e < n; e += g) cfma(s, X1[e], a.U[(int64_t)e * n + p1]);
                return s;
            },
            [&](int p1, double2 s) {
                X2[p1] = entry(s, p1 == pN ? 2 : 1, cadd(a.lam[p1], a.lam[pN]));
            });
        __syncthreads();
        for_items(n,
            [&](int k, int sub, int g) {
                double2 s = make_double2(0.0, 0.0);
                for (int p1 = sub; p1 <= pN; p1 += g) cfma(s, X2[p1], a.W[(int64_t)p1 * n + k]);
                return s;
            },
            [&](int k, double2 s) { psi[k] = cmul(s, a.W[(int64_t)pN * n + k]); });
    } else {
        for (int p3 = N == 3 ? pN : chunk; p3 <= pN; p3 += N == 3 ? 1 : a.chunks) {
            if (N == 4) {
                for_items(tri(n),
                    [&](int it, int sub, int g) {
                        const int x = (int)(tab[it] & 255u), y = (int)(tab[it] >> 8);
                        double2 s = make_double2(0.0, 0.0);
#pragma unroll 4
                        for (int e = sub; e < n; e += g) {
                            const int lo = min(x, e), hi = max(y, e), mid = x + y + e - lo - hi;
                            cfma(s, X1[tet(hi) + tri(mid) + lo], a.U[(int64_t)e * n + p3]);
                        }
                        return s;
                    },
                    [&](int it, double2 s) { Xp[it] = s; });
                __syncthreads();
            }
            for_items((p3 + 1) * n,
                [&](int it, int sub, int g) {
                    const int q = it / n, a1 = it - q * n;
                    double2 s = make_double2(0.0, 0.0);
#pragma unroll 4
                    for (int e = sub; e < n; e += g) cfma(s, Xp[pair_rank(a1, e)], a.U[(int64_t)e * n + q]);
                    return s;
                },
                [&](int it, double2 s) { X2[it] = s; });
            __syncthreads();
            double2 base = a.lam[p3];
            if (N == 4) base = cadd(base, a.lam[pN]);
            for_items(tri(p3 + 1),
                [&](int it, int sub, int g) {
                    const int p1 = (int)(tab[it] & 255u), p2 = (int)(tab[it] >> 8);
                    double2 s = make_double2(0.0, 0.0);
#pragma unroll 4
                    for (int e = sub; e < n; e += g) cfma(s, X2[p2 * n + e], a.U[(int64_t)e * n + p1]);
                    return s;
                },
                [&](int it, double2 s) {
                    const int p1 = (int)(tab[it] & 255u), p2 = (int)(tab[it] >> 8);
                    int run = 1, den = 1;
                    if (p1 == p2) den *= ++run; else run = 1;
                    if (p2 == p3) den *= ++run; else run = 1;
                    if (N == 4 && p3 == pN) den *= ++run;
                    Xp[it] = entry(s, den, cadd(cadd(a.lam[p1], a.lam[p2]), base));
                });
            __syncthreads();
            for_items(n,
                [&](int k, int sub, int g) {
                    double2 s = make_double2(0.0, 0.0);
                    for (int p2 = sub; p2 <= p3; p2 += g) {
                        double2 t = make_double2(0.0, 0.0);
                        for (int p1 = 0; p1 <= p2; ++p1) cfma(t, Xp[tri(p2) + p1], a.W[(int64_t)p1 * n + k]);
                        cfma(s, t, a.W[(int64_t)p2 * n + k]);
                    }
                    return s;
                },
                [&](int k, double2 s) { cfma(psi[k], s, a.W[(int64_t)p3 * n + k]); });
            __syncthreads();
        }
        if (N == 4)   // (the lane that owns psi[k] in for_items differs: past the barrier above)
            for (int k = tid; k < n; k += THREADS) psi[k] = cmul(psi[k], a.W[(int64_t)pN * n + k]);
    }
    __syncthreads();

    // the block's share, and the sum of all shares by the upper index's last block
    double2* part = a.part + (int64_t)row * gridDim.x * n;
    for (int k = tid; k < n; k += THREADS) part[(int64_t)b * n + k] = psi[k];
    __threadfence();
    __shared__ int last;
    __syncthreads();
    if (tid == 0) last = atomicAdd(&a.count[row], 1u) == gridDim.x - 1 ? 1 : 0;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for_items(n,
        [&](int k, int sub, int g) {
            double2 s = make_double2(0.0, 0.0);
#pragma unroll 4
            for (int c = sub; c < (int)gridDim.x; c += g) s = cadd(s, __ldcg(&part[(int64_t)c * n + k]));
            return s;
        },
        [&](int k, double2 s) {
            double2* o = a.out + (int64_t)i * n + k;
            *o = a.accumulate ? csub(*o, s) : make_double2(-s.x, -s.y);
        });
    if (tid == 0) a.count[row] = 0u;
}

// Blocks per (i, p_4), which share its p_3: few blocks are too short a grid, many repeat the first two
// stages. One / two / four take 91 / 58 / 55 us at n = 8, 156 / 141 / 129 at 12, 305 / 255 / 203 at 14, 610 /
// 490 / 597 at 18, 921 / 826 / 942 at 20, 2102 / 2014 / 2283 at 24, 8725 / 9439 / 11850 at 32.
int chunks_for(int N, int n) { return N < 4 ? 1 : n <= 12 ? 4 : n <= 20 ? 2 : 1; }

size_t smem_bytes(int N, int n, int nm)
{
    const size_t c = N == 2 ? (size_t)n + nm + n
                            : (size_t)(N == 4 ? tet(n) : 0) + tri(n) + (size_t)nm * n + n;
    const size_t t = N == 2 ? 0 : (size_t)tri(n) + (N == 4 ? tet(n) : 0);
    return c * sizeof(double2) + ((size_t)(N + 1) * (n + 1) + t) * 4;
}

constexpr size_t kMaxSmem = 227 * 1024 - 64;

template <int N>
void launch(Plan& p, const ChainArgs& a, int rows)
{
    const size_t bytes = smem_bytes(N, a.n, a.nm);
    // (a constant: the attribute is the function's, and other threads launch it for other sizes)
    NPF_CUDA(cudaFuncSetAttribute(k_chain<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem));
    LaunchScope ls(&p.prof, "fp64_chain", p.stream);
    launch_dependent(k_chain<N>, dim3((unsigned)(a.nm * a.chunks), (unsigned)rows), dim3(THREADS), bytes, p.stream, a);
}

}  // namespace

// Scratch of the chain over `rows` upper indices.
static size_t chain_scratch(const Plan& p, int N, int rows)
{
    return (size_t)rows * p.packed_count[N] * sizeof(double2) +
           (size_t)rows * p.nm * chunks_for(N, p.n) * p.n * sizeof(double2) + (size_t)rows * sizeof(unsigned) + 512;
}

bool chain_fits(const Plan& p, int N, size_t budget)
{
    return N >= 2 && N <= 4 && p.n <= 255 && smem_bytes(N, p.n, p.nm) <= kMaxSmem &&
           chain_scratch(p, N, p.nm) <= budget;
}

void chain_term(Plan& p, int N, double2* d_out, const double2* W, bool accumulate)
{
    const int n = p.n;
    const int lo = std::max(0, p.row_lo), hi = p.row_hi < 0 ? p.nm : std::min(p.row_hi, p.nm);
    const int rows = hi - lo;
    if (!accumulate && rows < n) launch_zero(p, d_out, (int64_t)n * n);   // the other rows
    if (rows <= 0) return;
    Arena& ar = p.scratch();
    ar.reserve(chain_scratch(p, N, rows), p.stream);
    ChainArgs a{};
    a.n = n;
    a.nm = p.nm;
    a.ilo = lo;
    a.chunks = chunks_for(N, n);
    a.P = p.packed_count[N];
    double2* S = (double2*)ar.base;
    a.S = S;
    a.part = S + (size_t)rows * a.P;
    a.count = (unsigned*)(a.part + (size_t)rows * p.nm * a.chunks * n);
    a.cnt = p.d_cnt;
    a.U = p.d_U;
    a.W = W ? W : p.d_V;
    a.lam = p.d_lam;
    a.eps = p.eps;
    a.divide = p.divide;
    a.out = d_out;
    a.accumulate = accumulate;
    {
        LaunchScope ls(&p.prof, "fp64_chain_upper", p.stream);
        launch_dependent(k_chain_upper, dim3((unsigned)((a.P + 127) / 128), (unsigned)((rows + 3) / 4)), dim3(128), 0,
                         p.stream, n, lo, rows, a.P, p.d_tensor[N], p.d_V, S, a.count);
    }
    if (N == 2) launch<2>(p, a, rows);
    else if (N == 3) launch<3>(p, a, rows);
    else launch<4>(p, a, rows);
}

}  // namespace npf
