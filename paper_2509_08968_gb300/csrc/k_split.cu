// k_split.cu -- FP64-emulating split-BF16 contraction on tcgen05 tensor cores.
//
// Number format (Ozaki-style fixed-point slicing). Every operand row r carries an exponent e_r
// with |x| < 2^e_r for all of its entries; x = 2^(e_r - 7) * sum_{s<S} d_s 2^(-8s) with balanced
// base-256 digits d_0 in [-128, 128], d_s in [-128, 127]. Plane s stores d_s * 2^(-8s) in BF16
// (exact: at most 8 significant bits). The product of two planes summed over K' <= 256 is an
// exact FP32 sum (|d d'| <= 2^14, 2^14 * 256 = 2^22), so the slice pairs (s, t) with s + t < S
// are accumulated in TMEM by level: L0 = pair (0,0), L1 = pairs (0,1),(1,0) and L2 = the three
// level-2 pairs are exact FP32 sums (|L2| * 2^16 <= 3 * 2^22 < 2^24); L3 = every deeper level
// (relative weight <= 2^-24, so even a truncating FP32 accumulation there costs ~2^-40). The
// epilogue recombines V = (L0 + L1 + L2) * 2^30 + rint(L3 * 2^30) exactly in 64-bit integers
// (|V| <= 2^53, resolution 2^-30 of the L0 unit); the value is V * 2^(e_a + e_b - VEXP),
// VEXP = 14 + 30. It then re-slices V for the next contraction (integer arithmetic, new exponent
// shared by the next operand's K-row), keeps V itself for a regather, or divides by the resonance
// denominator.
//
// Complex operands interleave (Re, Im) along K': row = [Re x_0, Im x_0, Re x_1, Im x_1, ...]
// (K' = 256 for 128 complex entries). A fixed complex matrix W is stored as Re-row p =
// [Re W_0p, -Im W_0p, Re W_1p, -Im W_1p, ..] and Im-row p = [Im W_0p, Re W_0p, ..], so one real
// GEMM yields Re and Im of X.W; a real operand row has K' = 128 plain entries.
//
// Dataflow of one order N (Algorithm 2). h and every intermediate are symmetric in their a's and in
// their p's, so only sorted tuples are formed, stored in colexicographic rank:
//   P1     : S[i][Q] = sum_j psi_{ij} A^j_Q on the sorted lower tuples Q (real rows Q, K = j), V and
//            the exponent per i (the upper index first: step 4 moved ahead, which the contraction
//            order allows).
//   expand : rows (i, sorted (a_1..a_{N-1})), K = a_N, digits of S^i_{sort(a)} gathered from V
//   c = 1..N-2 : contract an a with Phi; V (the exact 64-bit accumulators) per
//            (i, sorted p's, sorted a's), regathered into the digit rows
//            (i, sorted p's, sorted a's less one), K = the remaining a, with exact row exponents
//   c = N-1: rows (i, sorted (p_3..p_N), a_1), K = a_2; the output is re-sliced in the epilogue
//            into rows (i, sorted (p_2..p_N)), K = a_1 (a 128-row tile holds every a_1 of a row)
//   c = N  : last a with Phi, 1/N!, resonance denominator (clamped), multiplicity -> h in rows
//            (i, sorted (p_1..p_{N-1})), K = p_N
//   reduce : G^T[k][c'] = sum_{p_N} psi_{p_N k} h[c'][p_N], folded with psi_{p_{N-1} k} and
//            prod_{m<=N-2} psi_{p_m k} into Psi_N[i][k]; each tuple carries its multiplicity
//            N! / prod(run lengths)!.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "k_device.cuh"
#include "k_tc.cuh"
#include "npf_internal.h"

namespace npf {

constexpr int NP = 128;        // padded index extent (n <= 128 on this path)
constexpr int KSTEP = 16;      // K' elements of one MMA (BF16, 32 bytes)
constexpr int KP = 256;        // K' of a complex operand row (interleaved Re/Im)
constexpr int EXP_NONE = -4096;
constexpr int TMEM_COLS = 512;
constexpr int kErrTimeout = 1;
constexpr int VEXP = 44;       // value = V * 2^(e_a + e_b - VEXP), V in units of 2^-30 of L0
constexpr int EPI_WARPS = 16;  // epilogue warps (four per TMEM lane quarter)
constexpr int ROW_THREADS = 64 + 32 * EPI_WARPS + 64;   // producer, MMA, epilogue, two set-up warps

// ---------------------------------------------------------------------------------------
// Integer / double-float helpers
// ---------------------------------------------------------------------------------------
// Bit length of max(|v.x|, |v.y|) (one less for a negative power of two, which the top digit's range
// [-128, 128] holds).
__device__ __forceinline__ int bitlen(longlong2 v)
{
    const unsigned long long m = (unsigned long long)(v.x < 0 ? ~v.x : v.x) |
                                 (unsigned long long)(v.y < 0 ? ~v.y : v.y);
    return 64 - __clzll((long long)m);
}

// W = round(V * 2^sh) for |result| < 2^47.
__device__ __forceinline__ long long shift_round(long long V, int sh)
{
    if (sh >= 0) return sh < 16 ? V << sh : 0;
    const int r = -sh;
    if (r >= 63) return 0;
    return (V + (1ll << (r - 1))) >> r;
}

// The same for shifts to the left by up to 47 (a row whose exponent is its exact bit length).
__device__ __forceinline__ long long shift_full(long long V, int sh)
{
    return sh >= 0 ? (sh < 48 ? V << sh : 0) : shift_round(V, sh);
}

// 2^e for |e| < 1000 (double) / |e| < 127 (float)
__device__ __forceinline__ double pow2d(int e) { return __longlong_as_double((long long)(1023 + e) << 52); }
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }
// x 2^e for any e
__device__ __forceinline__ double2 times_pow2(double2 x, int e)
{
    if (e <= -1000 || e >= 1000) return make_double2(scalbn(x.x, e), scalbn(x.y, e));
    const double f = pow2d(e);
    return make_double2(x.x * f, x.y * f);
}

// BF16 bits of d * 2^(-8 s) for an integer digit |d| <= 128 (exact).
__device__ __forceinline__ uint32_t digit_bf16(int d, int s)
{
    return __float_as_uint((float)d * pow2f(-8 * s)) >> 16;
}

// Balanced base-256 digits of W (|W| <= 2^(7 + 8(S-1))), packed as (Re, Im) BF16 pairs per
// plane: plane s holds d_s * 2^(-8 s), d_0 the most significant digit. Adding 128 to every lower
// digit (the constant OFF) turns them into plain bytes u = d + 128 in [0, 255] with no borrows,
// and the top digit is the arithmetic shift of the sum. A byte's low seven bits are the mantissa of
// the BF16 number (128 + (u & 127)) 2^(-8 s); subtracting 128 or 256 (u >= 128 or not) times 2^(-8 s)
// leaves d 2^(-8 s) exactly, so a pair takes one byte permute, two logic operations and one packed
// BF16 subtraction.
template <int S>
struct DigitOff {
    static constexpr long long value = (DigitOff<S - 1>::value << 8) | 128;
};
template <>
struct DigitOff<0> { static constexpr long long value = 0; };

template <int S>
__device__ __forceinline__ void digit_pairs(long long Wr, long long Wi, uint32_t (&out)[S])
{
    constexpr long long OFF = DigitOff<S - 1>::value;   // 128 in each of the S-1 lower bytes
    const unsigned long long ur = (unsigned long long)(Wr + OFF);
    const unsigned long long ui = (unsigned long long)(Wi + OFF);
    // top digits in [-128, 128]: exact in FP32, and their upper halves are the BF16 bits
    const float fr = (float)(int)((long long)ur >> (8 * (S - 1)));
    const float fi = (float)(int)((long long)ui >> (8 * (S - 1)));
    out[0] = __byte_perm(__float_as_uint(fr), __float_as_uint(fi), 0x7632);
#pragma unroll
    for (int s = 1; s < S; ++s) {
        const int k = S - 1 - s;   // byte position from the least significant end
        const uint32_t xr = (uint32_t)(k < 4 ? ur : ur >> 32), xi = (uint32_t)(k < 4 ? ui : ui >> 32);
        // (Re byte, Im byte) in the low halves' low bytes (the other bytes are masked off)
        const uint32_t p = __byte_perm(xr, xi, (unsigned)((k & 3) | ((k & 3) + 4) << 8));
        const uint32_t one = 0x43004300u - 0x04000400u * (uint32_t)s;         // 128 * 2^(-8 s), twice
        const uint32_t a = (p & 0x007F007Fu) | one;
        const uint32_t c = (p & 0x00800080u) ^ (one + 0x00800080u);           // 256 or 128 times 2^(-8 s)
        const __nv_bfloat162 d = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&a),
                                         *reinterpret_cast<const __nv_bfloat162*>(&c));
        out[s] = *reinterpret_cast<const uint32_t*>(&d);
    }
}

struct dfl { float hi, lo; };
__device__ __forceinline__ dfl df_norm(float s, float e)
{
    const float hi = s + e;
    return {hi, e - (hi - s)};
}
__device__ __forceinline__ dfl df_add(dfl a, dfl b)
{
    const float s = a.hi + b.hi;
    const float bb = s - a.hi;
    const float e = (a.hi - (s - bb)) + (b.hi - bb) + a.lo + b.lo;
    return df_norm(s, e);
}
__device__ __forceinline__ dfl df_mul(dfl a, dfl b)
{
    const float p = a.hi * b.hi;
    const float e = fmaf(a.hi, b.hi, -p) + (a.hi * b.lo + a.lo * b.hi);
    return df_norm(p, e);
}
__device__ __forceinline__ dfl df_neg(dfl a) { return {-a.hi, -a.lo}; }
// Exact sum a + b = s + e of two floats (Knuth's two-sum).
__device__ __forceinline__ dfl two_sum(float a, float b)
{
    const float s = a + b;
    const float bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}
// a b + c d as the exact leading sum s + e of the two products' leading parts, with the rest (their
// rounding errors and the cross terms; error a few 2^-47 of |a b| + |c d|) in e, not normalised: 16
// operations where two df_mul and a df_add take 27.
__device__ __forceinline__ dfl df_dot2(dfl a, dfl b, dfl c, dfl d)
{
    const float p = a.hi * b.hi, q = c.hi * d.hi;
    float e = fmaf(a.hi, b.hi, -p) + fmaf(c.hi, d.hi, -q);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    e = fmaf(c.hi, d.lo, e);
    e = fmaf(c.lo, d.hi, e);
    const dfl s = two_sum(p, q);
    return {s.hi, s.lo + e};
}
__device__ __forceinline__ double df_to_d(dfl a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ dfl to_dfl(double x)
{
    const float hi = (float)x;
    return {hi, (float)(x - (double)hi)};
}

// A double as the exact sum of three floats (24 + 24 + 5 significant bits).
struct tfl { float a, b, c; };
__device__ __forceinline__ tfl to_tfl(double x)
{
    const float a = (float)x;
    const double r = x - (double)a;               // exact
    const float b = (float)r;
    return {a, b, (float)(r - (double)b)};        // exact
}
// s + l as a double-float for exact triple-float terms: the leading pieces are added with
// error-free transformations, so the result keeps ~2^-48 relative accuracy however much they
// cancel (near-resonant denominators).
__device__ __forceinline__ dfl tfl_sum(const tfl& s, const tfl& l)
{
    const dfl A = two_sum(s.a, l.a);
    const dfl B = two_sum(s.b, l.b);
    const dfl X = two_sum(A.hi, B.hi);
    const float y = (A.lo + B.lo) + ((s.c + l.c) + X.lo);
    return two_sum(X.hi, y);
}
// L0 + L1 + L2 + L3 (one accumulator element, units of 2^30 in V) as a double-float.
__device__ __forceinline__ dfl level_sum_df(uint32_t l0, uint32_t l1, uint32_t l2, uint32_t l3)
{
    const dfl t1 = two_sum(__uint_as_float(l0), __uint_as_float(l1));
    const dfl t2 = two_sum(t1.hi, __uint_as_float(l2));
    const dfl t3 = two_sum(t2.hi, __uint_as_float(l3));
    return two_sum(t3.hi, (t1.lo + t2.lo) + t3.lo);
}
// round(x.hi + x.lo) for |x| < 2^47 with 32-bit conversions (off by at most one unit).
__device__ __forceinline__ long long df_round_i64(dfl x)
{
    const int t = __float2int_rz(x.hi * 5.9604644775390625e-08f);          // 2^-24
    const float rem = fmaf((float)t, -16777216.0f, x.hi);                   // exact
    return ((long long)t << 24) + __float2int_rn(rem + x.lo);
}

constexpr int SEGS = 8;   // segments a 128-row divide tile may hold

// 1 / d for a small positive integer d as a double-float (relative error ~2^-46), without FP64.
__device__ __forceinline__ dfl rcp_small(int d)
{
    const float x = (float)d;                        // exact
    const float hi = __frcp_rn(x);
    return {hi, fmaf(-hi, x, 1.0f) * hi};            // the residual 1 - hi x is exact
}

// Recombined accumulator of one output element: V (units 2^-30 of the L0 integer grid). The
// integer parts are read off float bit patterns after adding 1.5 * 2^(23 + j): the sum lands in a
// binade whose spacing is 2^j, so it rounds to that grid (to nearest, ties to even) and its
// mantissa bits count grid steps. L0 is an integer with |L0| <= 2^22 (256 products of digits of
// magnitude <= 2^7); L3 * 2^30 is split into a multiple of 2^20 and an exact remainder.
__device__ __forceinline__ long long combine(uint32_t l0, uint32_t l1, uint32_t l2, uint32_t l3)
{
    const int a0 = __float_as_int(__uint_as_float(l0) + 12582912.0f) - 0x4B400000;   // 1.5 * 2^23
    const long long a1 = (long long)__float2int_rn(__uint_as_float(l1) * 256.0f);
    const long long a2 = (long long)__float2int_rn(__uint_as_float(l2) * 65536.0f);
    const float x3 = __uint_as_float(l3) * 1073741824.0f;                            // 2^30
    const float t3 = x3 + 13194139533312.0f;                                          // 1.5 * 2^43
    const int h3 = __float_as_int(t3) - 0x55400000;          // rint(x3 / 2^20), |x3| < 2^42
    const float r = x3 - (t3 - 13194139533312.0f);           // exact, |r| <= 2^19
    const int r3 = __float_as_int(r + 12582912.0f) - 0x4B400000;
    const long long a3 = ((long long)h3 << 20) + r3;
    return ((long long)a0 << 30) + (a1 << 22) + (a2 << 14) + a3;
}

// A priori bound of |L2 + L3| in units of L0 (the MMAs run the pairs s + t < S): a level-l pair
// adds at most 256 products of digits |d| <= 2^7 at weight 2^(-8l), and level l has l + 1 pairs.
__host__ __device__ constexpr float deep_level_bound(int S)
{
    float b = 0.f, w = 1.f / 65536.f;   // 2^-16: level 2
    for (int l = 2; l < S; ++l) {
        b += (float)(l + 1) * w;
        w *= 1.f / 256.f;
    }
    return b * 4194304.f * 1.001f + 1.0f;   // x 2^22, with margin
}
// Upper bound of |V| 2^-30 from L0 and L1 alone: their FP32 sum plus its rounding bound plus the
// a priori bound of the deeper levels. An exponent taken from it exceeds the exact one only for
// columns whose entries are all below ~2^9 L0 units, i.e. where the deeper levels' size matters.
__device__ __forceinline__ float level_bound01(uint32_t l0, uint32_t l1, float deep)
{
    const float a = __uint_as_float(l0), b = __uint_as_float(l1);
    return fmaf(fabsf(a) + fabsf(b), 2.384185791015625e-07f, fabsf(a + b) + deep);   // 2^-22
}
// e with x < 2^e <= 2x for a positive normal float x (the frexp exponent)
__device__ __forceinline__ int f32_exponent(float x) { return ((__float_as_int(x) >> 23) & 255) - 126; }

// Number of TMEM level accumulators used by S slices (levels s + t < S, capped at 3).
template <int S>
struct Lev { static constexpr int N = S < 4 ? S : 4; };

// Load UC (2 or 4) columns of every used level of one accumulator group (levels `stride` columns apart).
template <int S, int UC>
__device__ __forceinline__ void load_levels(uint32_t taddr, int stride, uint32_t (&v)[4][UC])
{
#pragma unroll
    for (int L = 0; L < 4; ++L) {
        if (L < Lev<S>::N) {
            if constexpr (UC == 4) tc::tmem_ld4(taddr + L * stride, v[L]);
            else tc::tmem_ld2(taddr + L * stride, v[L]);
        } else {
#pragma unroll
            for (int c = 0; c < UC; ++c) v[L][c] = 0u;
        }
    }
}

// Colexicographic ranks of sorted pairs, triples and quadruples.
__host__ __device__ __forceinline__ int rank2(int a, int b) { return b * (b + 1) / 2 + a; }   // a <= b
__host__ __device__ __forceinline__ int rank3(int a, int b, int c)                            // a <= b <= c
{
    return c * (c + 1) * (c + 2) / 6 + b * (b + 1) / 2 + a;
}
__host__ __device__ __forceinline__ int rank4(int a, int b, int c, int d)                     // a <= .. <= d <= 128
{
    return d * (d + 1) * (d + 2) / 6 * (d + 3) / 4 + rank3(a, b, c);
}

// ---------------------------------------------------------------------------------------
// Input preparation (once per tensor): A^T digit planes for the upper-index contraction,
// rows = sorted lower tuples Q (exponent per Q over all j), K' = j (real). The packed tensor's
// tuples are in lexicographic order; the rows go to their colexicographic rank, the order of every
// later intermediate (a row is 256 bytes a plane, so the scatter costs nothing).
// ---------------------------------------------------------------------------------------
template <int S>
__global__ void k_prep_at(const double* __restrict__ A, int64_t P, int n, int N,
                          const int64_t* __restrict__ cnt, __nv_bfloat16* __restrict__ planes,
                          int64_t plane_stride, int* __restrict__ expQ)
{
    __shared__ int cn[5 * (NP + 1)];   // non-decreasing r-tuples in [v, n), r <= N
    for (int t = threadIdx.x; t < (N + 1) * (n + 1); t += blockDim.x) cn[t] = (int)cnt[t];
    __syncthreads();
    // one warp per Q: lanes cover j = lane, lane+32, lane+64, lane+96
    const int64_t q = (int64_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    const int lane = threadIdx.x % 32;
    if (q >= P) return;
    double v[4];
    double m = 0.0;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const int j = lane + 32 * t;
        v[t] = j < n ? A[(int64_t)j * P + q] : 0.0;
        m = fmax(m, fabs(v[t]));
    }
    // the tuple of lexicographic rank q, an index at a time: the first index is >= x for the last
    // cn[r][x] of the r-tuples from the previous index on
    int64_t row = 0;
    {
        int rem = (int)q, prev = 0;
        for (int pos = 0; pos < N; ++pos) {
            const int* c = cn + (N - pos) * (n + 1);
            int x = prev;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int w = lane + 32 * t;
                x += __popc(__ballot_sync(0xffffffffu, w > prev && w < n && rem >= c[prev] - c[min(w, n)]));
            }
            rem -= c[prev] - c[x];
            prev = x;
            row += pos == 0 ? x : pos == 1 ? rank2(0, x) : pos == 2 ? rank3(0, 0, x) : rank4(0, 0, 0, x);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    int e = EXP_NONE;
    if (m > 0.0) frexp(m, &e);
    if (lane == 0) expQ[row] = e;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const int j = lane + 32 * t;
        long long W = 0;
        if (e != EXP_NONE) W = __double2ll_rn(v[t] * pow2d(7 + 8 * (S - 1) - e));
#pragma unroll
        for (int s = S - 1; s >= 0; --s) {
            int d;
            if (s > 0) {
                d = (int)((W + 128) & 255) - 128;
                W = (W - d) >> 8;
            } else {
                d = (int)W;
            }
            reinterpret_cast<uint16_t*>(planes)[s * plane_stride + row * NP + j] =
                (uint16_t)digit_bf16(d, s);
        }
    }
}

// ---------------------------------------------------------------------------------------
// Row-data GEMM: data rows on the M side (128 per tile), the fixed complex matrix on the N side
// (bnc complex columns per tile -> 2*bnc real columns: Re block then Im block).
//
// Index layouts. A_N and every intermediate are symmetric in the lower indices not yet contracted
// and in the p's already formed, so the operands hold sorted tuples only, in colexicographic rank:
//   mode product c < N - 1 : rows (i, (p's) sorted (c-1)-tuple, (a's) sorted (N-c)-tuple)
//   mode product c = N - 1 : rows (i, sorted (N-2)-tuple (p_3..p_N), a_1), 2^lg rows a tuple; a
//                            128-row tile holds 128 >> lg of them (sub-blocks)
//   divide (c = N)         : rows (i, slot), a slot per sorted tuple (p_2..p_N)
//   reduction              : rows (i, sorted (p_1..p_{N-1})), K = p_N
// Each forms only new indices p <= the row's first p.
// ---------------------------------------------------------------------------------------
enum { EPI_V = 0, EPI_SLICE = 1, EPI_DIVIDE = 2, EPI_SLAB = 3, EPI_REDUCE = 4 };

struct RowArgs {
    int arows;           // rows of a data tile that are loaded (a multiple of 8; 128 but in EPI_SLICE)
    int kch;             // pipeline stages of K' (16 or 32 wide; K' past the operands' length is
                         // zero on both sides)
    int klast;           // 16-wide steps in the last stage (1 or 2 for 32-wide stages): the rest
                         // is padding
    const int* ea;       // row exponents, by operand row or (ea_outer) by outer index
    int ea_outer;
    const int* eb;       // column exponents of the fixed matrix (256 entries)
    int bnc;             // complex columns per tile (16 or 32)
    int ncol_tiles;
    int64_t num_tiles;
    int N;               // order
    int colmask;         // new index <= the row's first p
    int kfrom;           // EPI_REDUCE: skip the K' chunks below the tile's smallest p_{N-1}
    int64_t R;           // rows per outer index
    int RB;              // > 0: every outer index starts a tile and has RB of them (the last one may
                         // read rows of the next index, which are masked); 0: tiles of 128 rows run
                         // over all rows
    int lgncol;          // log2(ncol_tiles), or -1 when ncol_tiles is not a power of two
    // EPI_V: V (two 64-bit integers) at out_v[(new tuple) * R + row]; colmask: outer = (i, p), and
    // the new tuple (i, rank2(q, p)), else (i, q)
    longlong2* out_v;
    int* emax;           // EPI_V: largest exponent of every column (merged by atomicMax), or nullptr
    // EPI_SLICE: rows (tuple t of nt sorted (p_3..p_N), a_1); output rows are the divide's slots, RS
    // per upper index
    int nt;
    const uint32_t* ttup;    // order 4: the pairs (p_3, p_4), 8 bits per index
    int64_t RS;
    const int* segbase;      // first slot of the segment (p_2, .., p_{N-1}), by its colex rank
    // EPI_DIVIDE, EPI_SLAB: the slots; EPI_DIVIDE writes reduction rows, RT per upper index
    // (smeta: {p_2 or -1 for a padding slot; reduction row less p_1; kpos | segment << 8 | the
    // segment's first row << 12 | first run's length << 13 | prod(run lengths)! << 16}, kpos = p_N
    // the K position in that row; ssum, ssig: lambda_{p_2} + .. + lambda_{p_N} as exact triple-floats
    // [6][nslot] and in FP64)
    const int4* smeta;
    const float* ssum;
    const double2* ssig;
    int nslot;
    const uint32_t* stup;    // the slots' tuples, 8 bits per index (all ones: padding)
    const int* tpmax;        // largest p_2 of each tile's slots
    int64_t RT;
    // EPI_REDUCE: rows are the sorted tuples (p_1 <= .. <= p_{N-1}) in colexicographic rank
    const uint32_t* tuples;  // 8 bits per index
    const float4* wpre;      // W[p_1][k] W[p_2][k] at k * ldw + the pair's colex rank (orders 3 and 4), as
    int64_t ldw;             // double-float complex: the 32 rows of a warp read one run. Weights come
                             // without their column's exponent eb[k], and G (of the order of A
                             // V^(2 - N), S of A V) with (N - 1) ev[k] - es[i] added; the sums take both
                             // up in FP64, so that eigenvectors of any normalisation and tensors of
                             // any scale keep to FP32's range
    const int* ev;           // column exponents of the left eigenvectors (eb, unless W is another matrix)
    const int* es;           // exponents of S by upper index
    const int* tiles;        // the tiles that run (nullptr: every tile, skipped ones tested)
    const unsigned* ntiles_run;   // their count
    int kout;            // K entries written per row of the next operand (whole chunks of it)
    int lg;              // EPI_SLICE: log2 of the row radix (and of the next operand's K extent)
    int lgout;           // EPI_DIVIDE: log2 of the K extent of a reduction row
    int n;               // states (range of the a digits and of the reduction's columns k)
    int nm;              // modes in use (range of i and of the p digits; n unless a subset is set)
    int ncv;             // valid columns of this launch (modes, or states for the reduction)
    int nouter;          // upper indices of this launch (order-1 slabs: one row each)
    __nv_bfloat16* out_planes;
    int64_t out_plane_stride;
    int* out_exp;
    double2* out_f64;    // EPI_SLAB: out[i * n + q]; EPI_REDUCE: Psi_N
    // EPI_DIVIDE / EPI_SLAB / EPI_REDUCE
    const double2* lam;
    const float4* psi_df;    // the reduction weights W[p][k] (psi_{p k}) as double-float, at k*n + p (less eb[k])
    int i0;
    double invfact, eps;
    int divide;
    int fp64_quotient;   // EPI_DIVIDE: native FP64 quotient instead of the double-float one
    int stall;           // test hook: the MMA role never signals the first tile's accumulators,
                         // so the epilogue's bounded wait runs out (timeout path)
    float eps2f;         // eps^2 in FP32 (clamp test of the double-float quotient)
    int pre[8];          // EPI_SLAB: the requested prefix (N-1 indices)
    int* err;
    unsigned long long* trace;   // optional per-CTA phase timestamps [tile][6] (nullptr: off)
};

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Pipeline of one k_rows variant: every launch runs one pass over K through a ring of stages. The
// divide and the reduction, whose tables need room, take five stages of one 16-wide K' step (32-byte
// rows and swizzle), the others three stages of two steps (64-byte rows).
template <int S, int MODE>
struct RowCfg {
    static constexpr bool big_tables = MODE == EPI_DIVIDE || MODE == EPI_REDUCE;
    static constexpr int BK = big_tables ? 16 : 32;            // K' elements per stage
    static constexpr int KS = BK / KSTEP;                      // MMA K steps per stage
    static constexpr int A_TILE = NP * BK * 2;                 // 4 or 8 KB
    static constexpr int B_TILE = 64 * BK * 2;                 // at most 32 complex columns
    static constexpr int STAGE_BYTES = S * (A_TILE + B_TILE);
    // tables (offsets from a 1 KB boundary after the stages): barriers and the TMEM slot in the
    // first 256 bytes, column exponent keys by tile parity ([4 sub-blocks][32], the divide's
    // [SEGS][32]), reciprocals of small integers, then the tile tables
    // (two buffers, filled by the set-up warps)
    static constexpr int COLE = 256, COLE_N = MODE == EPI_DIVIDE ? SEGS * 32 : 128;
    static constexpr int RCP = 256 + 2048;
    static constexpr int TILE = RCP + 256;
    // one tile's tables
    static constexpr int META = 0;       // int[8]
    static constexpr int QINFO = 32;     // int4[4 lane quarters]
    static constexpr int COLEB = 96;     // int[32] fixed-matrix column exponents
    static constexpr int ROWM = 256;     // int4[128 rows]
    static constexpr int SROWQ = ROWM + 2048;        // EPI_SLICE: int[4 sub-blocks][32] output slots
    static constexpr int LAMF = ROWM + 2048;         // EPI_DIVIDE: float2[32] lambda_q - lambda_i
    static constexpr int LAMT = LAMF + 256;          //   the same as exact triple-floats, tfl[32][2]
    static constexpr int SIG = LAMT + 64 * 12;       //   float[6][128] the rows' sigma as triple-floats
    static constexpr int TILE_BYTES = MODE == EPI_DIVIDE ? SIG + 6 * NP * 4 : MODE == EPI_SLICE ? SROWQ + 512 : SROWQ;
    static constexpr int TABLES = TILE + 2 * TILE_BYTES + 1024;   // and 1 KB of alignment slack
    static constexpr int SMEM_MAX = 227 * 1024;
    static constexpr int STAGES_FIT = (SMEM_MAX - TABLES) / STAGE_BYTES;
    static constexpr int STAGES = STAGES_FIT < 8 ? STAGES_FIT : 8;
    static constexpr int SMEM = STAGES * STAGE_BYTES + TABLES;
    static_assert((2 * 8 + 8) * 8 + 8 <= 256, "barriers fit the first 256 bytes of the tables");
    static_assert(2 * COLE_N * 4 <= 2048, "keys");
    static_assert(COLEB + 128 <= ROWM, "tile tables");
    static_assert(STAGES >= 3, "pipeline stages");
    static_assert(SMEM <= SMEM_MAX, "shared memory");
};

// Position of a tile (column tile fastest).
struct TilePos {
    int ct;         // column tile
    int outer;      // upper index of the launch (RB > 0)
    int rr0;        // first row within the upper index (RB > 0)
    int64_t row0;   // first row of the operand
};
__device__ __forceinline__ TilePos tile_pos(const RowArgs& a, int64_t tile)
{
    const unsigned t = (unsigned)tile;   // (launch_rows bounds the tile count to 2^31)
    const unsigned rb = a.lgncol >= 0 ? t >> a.lgncol : t / (unsigned)a.ncol_tiles;
    TilePos p;
    if (a.kfrom) {   // the reduction: `tile` is a row block, the block's column tile changes every 32 of them
        p.outer = (int)(t / (unsigned)a.RB);
        p.ct = (int)((blockIdx.x + (t >> 5)) % (unsigned)a.ncol_tiles);
        p.rr0 = (int)(t - (unsigned)p.outer * (unsigned)a.RB) * NP;
        p.row0 = (int64_t)p.outer * a.R + p.rr0;
        return p;
    }
    p.ct = (int)(t - rb * (unsigned)a.ncol_tiles);
    if (a.RB > 0) {
        p.outer = (int)(rb / (unsigned)a.RB);
        p.rr0 = (int)(rb - (unsigned)p.outer * (unsigned)a.RB) * NP;
        p.row0 = (int64_t)p.outer * a.R + p.rr0;
    } else {
        p.outer = 0;
        p.rr0 = 0;
        p.row0 = (int64_t)rb * NP;
    }
    return p;
}

// Largest first p of a tile's rows (mode products with colmask).
__device__ __forceinline__ int tile_pmax(const RowArgs& a, int lg, const TilePos& p)
{
    if (a.out_v) return p.outer % a.nm;
    const int t1 = min(((p.rr0 + NP - 1) >> lg), a.nt - 1);
    if (a.N == 3) return t1;
    int m = 0;
    for (int t = p.rr0 >> lg; t <= t1; ++t) m = max(m, (int)(a.ttup[t] & 255u));
    return m;
}

// lg: the row radix (a compile-time 7 in the kernels without sub-blocks)
__device__ __forceinline__ bool tile_skipped(const RowArgs& a, int lg, const TilePos& p)
{
    if (a.tpmax) return p.ct * a.bnc > a.tpmax[p.rr0 / NP];   // slots: columns p_1 <= p_2
    return a.colmask && p.ct * a.bnc > tile_pmax(a, lg, p);
}

// First K' chunk a tile needs. In the reduction (kfrom = 1) the rows are (p_1, .., p_{N-1}) in
// colexicographic order and K = p_N >= p_{N-1}, which never decreases along the rows: the chunks
// below the first row's p_{N-1} are not read.
__device__ __forceinline__ int first_chunk(const RowArgs& a, const TilePos& p, int bk)
{
    if (!a.kfrom) return 0;
    return (int)((a.tuples[p.rr0] >> (8 * (a.N - 2))) & 255u) / (bk / 2);
}

// Wait with the same limits and no early exit (draining copies after an error).
__device__ __forceinline__ void mbar_drain(uint64_t* bar, uint32_t parity)
{
    const unsigned long long t0 = tc::wall_ns();
    for (long long it = 0; it < tc::kWaitLimit; ++it) {
        if (tc::mbar_try_wait(bar, parity)) return;
        if ((it & 1023) == 1023 && tc::wall_ns() - t0 > tc::kWaitNs) return;
    }
}

__device__ __forceinline__ void mma_col(int col, uint32_t acc, uint32_t leader, uint32_t d, uint32_t a, uint32_t b,
                                        uint32_t hi, uint32_t idesc)
{
    if (col == 1) tc::mma_bf16_lohi<1>(acc, leader, d, a, b, hi, idesc);
    else if (col == 2) tc::mma_bf16_lohi<2>(acc, leader, d, a, b, hi, idesc);
    else if (col == 3) tc::mma_bf16_lohi<3>(acc, leader, d, a, b, hi, idesc);
    else tc::mma_bf16_lohi<0>(acc, leader, d, a, b, hi, idesc);
}

// One K step of MMAs: the slice pairs (s, u), s + u < S, into their level accumulators (level L at TMEM
// column tmem + L * lstride). acc = 0: the step opens the tile, so each level's first MMA overwrites
// instead of accumulating. The loops unroll into straight-line MMAs with constant descriptor
// offsets (start address / 16 in the low half); one copy of them serves every step, since all roles
// of the kernel share the instruction cache.
// The MMAs that share a data plane s run back to back over the fixed-matrix planes u, with the data
// tile held in the tensor core's collector buffer: 36 cycles an MMA at N = 64 (48 without, where
// shared memory delivers the 4 KB data tile every time).
template <int S, int MODE>
__device__ __forceinline__ void issue_kstep(uint32_t acc, uint32_t leader, uint32_t tmem, uint32_t lstride,
                                            uint32_t a_lo, uint32_t a_plane16, uint32_t b_lo, uint32_t b_plane16,
                                            uint32_t idesc)
{
    using C = RowCfg<S, MODE>;
    constexpr uint32_t hi = C::BK == 32 ? tc::kSdescSw64Hi : tc::kSdescSw32Hi;
    bool first[4] = {true, true, true, true};
#pragma unroll
    for (int s = 0; s < S; ++s) {
        const uint32_t ao = a_lo + (uint32_t)s * a_plane16;
#pragma unroll
        for (int u = 0; u < S - s; ++u) {
            const int L = s + u < 3 ? s + u : 3;
            // collector: fill on the first MMA of the run, release on the last
            const int col = S - s == 1 ? 0 : u == 0 ? 1 : u == S - s - 1 ? 3 : 2;
            mma_col(col, first[L] ? acc : 1u, leader, tmem + L * lstride, ao, b_lo + (uint32_t)u * b_plane16, hi, idesc);
            first[L] = false;
        }
    }
}

__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, %0;" ::"r"(32 * EPI_WARPS) : "memory"); }
// epi_sync that also tells whether any epilogue thread brought `f`.
__device__ __forceinline__ bool epi_any(bool f)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %1, 0;\n\t"
        "bar.red.or.pred q, 1, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(f ? 1 : 0), "r"(32 * EPI_WARPS)
        : "memory");
    return r != 0;
}

// The tiles of a launch that run (tile_skipped false), compacted: each block scans 256
// consecutive tiles and appends the running ones in order at a position taken with one atomic.
// The persistent kernel then walks this list: a skipped tile cost each of its roles a decode
// (2.7 skipped tiles per running one in the divide stage of order 4).
static __global__ void k_tile_list(RowArgs a, int lg, int* __restrict__ list, unsigned* __restrict__ count)
{
    __shared__ unsigned wsum[8];
    __shared__ unsigned base;
    pdl_wait();
    const int64_t tile = (int64_t)blockIdx.x * 256 + threadIdx.x;
    bool run = false;
    if (tile < a.num_tiles) {
        run = !tile_skipped(a, lg, tile_pos(a, tile));
    }
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const unsigned bal = __ballot_sync(0xffffffffu, run);
    if (lane == 0) wsum[warp] = __popc(bal);
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned tot = 0;
        for (int w = 0; w < 8; ++w) { const unsigned c = wsum[w]; wsum[w] = tot; tot += c; }
        base = tot ? atomicAdd(count, tot) : 0u;
    }
    __syncthreads();
    if (run) list[base + wsum[warp] + __popc(bal & ((1u << lane) - 1u))] = (int)tile;
}

// Persistent row GEMM: one CTA per SM walks the tiles blockIdx.x, +gridDim.x, ... Roles:
//   warp 0 (one lane): TMA producer over a ring of STAGES shared-memory stages that runs across
//                      tiles, so the next tile's operands stream in during this tile's epilogue;
//   warp 1           : MMA issuer (the warp runs the loop, one elected lane issues). The four
//                      level accumulators of a 128 x bnc-complex tile take 8 bnc <= 256 TMEM columns;
//                      tiles alternate two sets, so the next tile's MMAs run during this tile's
//                      epilogue;
//   warps 2..17      : epilogue (lane quarter = warp % 4, column group = (warp - 2) / 4). Values
//                      needed twice (a column exponent before slicing) are read from TMEM twice
//                      instead of being staged in shared memory;
//   warps 18, 19     : set-up: the next tile's tables (row exponents and indices, eigenvalue sums,
//                      output rows) into the other of two buffers. Chains of dependent global loads,
//                      they took 2 to 7 us a tile in front of the epilogue.
// Bound per 32-column tile of a mode product at n = 120: 7.1 us, 5.4 of them its 315 MMAs; shared memory
// carries 1.08 MB of MMA operand reads and 0.59 MB of TMA writes meanwhile (6.3 us at 128 bytes a
// clock). Below n = 64 and in the divide and the reduction the epilogue bounds it. Tiles are 32 columns
// wide in every mode, so that two accumulator sets fit TMEM and an epilogue overlaps the next tile's
// MMAs: divide at n = 120, order 3, 1.39 ms a call against 1.83 with 64-column tiles in turn.
template <int S, int MODE, bool SUBB>
__global__ void __launch_bounds__(ROW_THREADS, 1)
    k_rows(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, RowArgs args)
{
    using C = RowCfg<S, MODE>;
    constexpr int BKm = C::BK;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* stage_base = smem;
    uint8_t* tables = smem + C::STAGES * C::STAGE_BYTES;
    uint64_t* full = (uint64_t*)tables;
    uint64_t* empty = full + C::STAGES;
    uint64_t* tfull = empty + C::STAGES;       // [2] MMA -> epilogue: accumulators complete
    uint64_t* tempty = tfull + 2;              // [2] epilogue -> MMA: accumulators read
    uint64_t* sfull = tempty + 2;              // [2] set-up -> epilogue: tables filled
    uint64_t* sempty = sfull + 2;              // [2] epilogue -> set-up: tables read
    uint32_t* tmem_slot = (uint32_t*)(sempty + 2);
    int* colE_all = (int*)(tables + C::COLE);
    dfl* rcp = (dfl*)(tables + C::RCP);        // 1 / d, 1 <= d <= 24

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int bnc = args.bnc;
    const int bnr = 2 * bnc;
    const uint32_t b_bytes_tile = (uint32_t)bnr * BKm * 2;
    // A tile of the last mode product at radix 128 loads the rows a_1 < arows only; the MMAs read the
    // next plane's for the others (still in the stage), whose results no one uses. At n = 75, FP32 form,
    // order 4, the padding was 41% of the rows: mode products 20.3 -> 17.5 ms.
    const uint32_t a_bytes_tile = MODE == EPI_SLICE && !SUBB ? (uint32_t)args.arows * BKm * 2 : (uint32_t)C::A_TILE;
    const int lg = SUBB ? args.lg : 7;         // row radix 2^lg (sub-blocks only below 128)

    if (threadIdx.x == 0) {
        for (int s = 0; s < C::STAGES; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(&tfull[b], 1);
            tc::mbar_init(&tempty[b], 1);
            tc::mbar_init(&sfull[b], 2);       // one arrival per set-up warp
            tc::mbar_init(&sempty[b], 1);
        }
        tc::fence_mbar_init();
        tc::tma_prefetch(&tmA);
        tc::tma_prefetch(&tmB);
    }
    if (warp == 1) {
        tc::tmem_alloc(tmem_slot, TMEM_COLS);
        tc::tmem_relinquish();
    }
    if (MODE != EPI_REDUCE)
        for (int e = threadIdx.x; e < 2 * C::COLE_N; e += ROW_THREADS) colE_all[e] = 0;
    if (MODE == EPI_DIVIDE && threadIdx.x >= 1 && threadIdx.x <= 24) rcp[threadIdx.x] = rcp_small(threadIdx.x);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    pdl_wait();   // (no global memory before)

    // tiles walked by every role: the running-tile list when there is one
    const int64_t nloop = args.tiles ? (int64_t)*(volatile const unsigned*)args.ntiles_run : args.num_tiles;
    auto tile_at = [&](int64_t k) -> int64_t {
        return k >= nloop ? 0 : args.tiles ? (int64_t)args.tiles[k] : k;
    };
    // The reduction takes consecutive row blocks, so that its epilogue can sum over them in registers. The
    // ncol_tiles blocks of a group walk the same row blocks side by side, each on another column tile (in
    // turn, since the last one is narrower), so that the rows are read from HBM once: with each column
    // tile walked by itself they were read once for each (1.7 GB in 338 us at n = 120, order 3, 34 upper
    // indices). The other modes take every gridDim.x-th tile.
    const int64_t nred = args.num_tiles / args.ncol_tiles, groups = gridDim.x / (unsigned)args.ncol_tiles;
    const int64_t per = (nred + groups - 1) / max(groups, (int64_t)1);
    const int64_t kbeg = MODE == EPI_REDUCE ? per * (blockIdx.x / (unsigned)args.ncol_tiles) : blockIdx.x;
    const int64_t kend = MODE == EPI_REDUCE ? min(nred, kbeg + per) : nloop;
    const int64_t kstep = MODE == EPI_REDUCE ? 1 : gridDim.x;
    const uint32_t lstride = (uint32_t)bnr;    // TMEM columns between levels

    if (warp == 0) {
        if (lane == 0) {
            // ---------------- TMA producer: per tile the K' steps with every plane
            uint32_t it = 0;
            bool alive = true;
            int64_t next = tile_at(kbeg);
            for (int64_t k = kbeg; k < kend && alive; k += kstep) {
                const TilePos tp = tile_pos(args, next);
                next = tile_at(k + kstep);
                const int64_t row0 = tp.row0;
                const int bc = tp.ct * bnc;
                for (int kc = first_chunk(args, tp, BKm); kc < args.kch; ++kc, ++it) {
                    const int st = (int)(it % C::STAGES);
                    const uint32_t ph = (it / C::STAGES) & 1;
                    if (!tc::mbar_wait(&empty[st], ph ^ 1, args.err, kErrTimeout)) {
                        alive = false;
                        break;
                    }
                    uint8_t* sA = stage_base + st * C::STAGE_BYTES;
                    uint8_t* sB = sA + S * C::A_TILE;
                    tc::mbar_arrive_expect_tx(&full[st], S * (a_bytes_tile + b_bytes_tile));
                    // A: [plane][128 rows][BK]; B: [plane][Re rows, Im rows][BK]
                    tc::tma_load_3d(sA, &tmA, kc * BKm, (int)row0, 0, &full[st]);
                    tc::tma_load_4d(sB, &tmB, kc * BKm, bc, 0, 0, &full[st]);
                }
            }
            if (!alive) {
                // after an error: let the copies already issued land before the CTA exits
                const uint32_t first = it > (uint32_t)C::STAGES ? it - C::STAGES : 0u;
                for (uint32_t j = first; j < it; ++j)
                    mbar_drain(&full[j % C::STAGES], (j / C::STAGES) & 1);
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer: slice pairs (s, t), s + t < S, accumulated by level.
        // The whole warp runs this loop (waits made warp-uniform by a vote), so that the
        // descriptor arithmetic stays uniform; one elected lane issues the MMAs and commits.
        // Nothing here depends on the tile but the reduction's first chunk: a value carried from one
        // tile to the next (a prefetched index) made every MMA's operands per-lane values and the
        // mode products 10% slower.
        const uint32_t leader = tc::elect_one();
        const uint32_t idesc = tc::idesc_bf16_f32(128, bnr);
        const uint32_t a16 = a_bytes_tile >> 4;   // plane strides in 16-byte units
        const uint32_t b16 = b_bytes_tile >> 4;
        uint32_t it = 0, t = 0;
        bool alive = true;
        for (int64_t k = kbeg; k < kend && alive; k += kstep) {
            const int k0 = MODE == EPI_REDUCE ? first_chunk(args, tile_pos(args, tile_at(k)), BKm) : 0;
            const int set = (int)(t & 1);
            const uint32_t use = t >> 1;                     // earlier tiles on this set
            // (the address comes from shared memory: taken from lane 0 it is known to be uniform)
            const uint32_t tm = __shfl_sync(0xffffffffu, tmem + (uint32_t)set * (TMEM_COLS / 2), 0);
            if (!__all_sync(0xffffffffu, tc::mbar_wait(&tempty[set], (use & 1) ^ 1, args.err, kErrTimeout))) {
                alive = false;
                break;
            }
            tc::fence_after_sync();
            for (int kc = k0; kc < args.kch; ++kc, ++it) {
                const int st = (int)(it % C::STAGES);
                const uint32_t ph = (it / C::STAGES) & 1;
                if (!__all_sync(0xffffffffu, tc::mbar_wait(&full[st], ph, args.err, kErrTimeout))) {
                    alive = false;
                    break;
                }
                tc::fence_after_sync();
                const uint32_t aBase = tc::smem_u32(stage_base + st * C::STAGE_BYTES);
                const uint32_t a_lo = tc::sdesc_sw64_lo(aBase);
                const uint32_t b_lo = tc::sdesc_sw64_lo(aBase + S * C::A_TILE);
                // 32-byte K offsets within a swizzled row; the last stage's second step may be padding
                const int steps = kc == args.kch - 1 ? min(C::KS, args.klast) : C::KS;
#pragma unroll 1
                for (int ks = 0; ks < steps; ++ks)
                    issue_kstep<S, MODE>(kc == k0 && ks == 0 ? 0u : 1u, leader, tm, lstride, a_lo + (uint32_t)(ks * 2), a16,
                                         b_lo + (uint32_t)(ks * 2), b16, idesc);
                tc::mma_commit(leader, &empty[st]);
            }
            if (!alive) break;
            if (!args.stall) tc::mma_commit(leader, &tfull[set]);
            ++t;
        }
    } else if (warp >= 2 + EPI_WARPS) {
        // ---------------- set-up warps: the tables of a tile, one tile ahead of the epilogue
        const int st = threadIdx.x - 32 * (2 + EPI_WARPS);   // 0 .. 63
        const int N = args.N;
        uint32_t t = 0;
        bool alive = true;
        int64_t next = tile_at(kbeg);
        for (int64_t k = kbeg; k < kend && alive; k += kstep) {
            const int64_t tile = next;
            const TilePos tp = tile_pos(args, tile);
            next = tile_at(k + kstep);
            const int buf = (int)(t & 1);
            uint8_t* tb = tables + C::TILE + buf * C::TILE_BYTES;
            unsigned long long* trc = args.trace ? args.trace + (MODE == EPI_REDUCE ? tile * args.ncol_tiles + tp.ct : tile) * 6 : nullptr;
            alive = __all_sync(0xffffffffu, tc::mbar_wait_idle(&sempty[buf], ((t >> 1) & 1) ^ 1, args.err, kErrTimeout));
            const unsigned long long t0 = trc ? global_ns() : 0ull;
            const int qbase = tp.ct * bnc;
            // every global load first: behind a store to the tables each would wait for the one before
            // (rows st and st + 64; the rows 32 w .. + 31 of one warp and round are one lane quarter)
            int ea[2], sea[2] = {0, 0};
            uint32_t tup[2] = {0u, 0u};
            int4 sm[2];
            float sg[2][6];
            bool row_in[2];
            int vcols = min(bnc, args.ncv - qbase);
            int ebv = st < 32 && st < bnc ? args.eb[qbase + st] : 0;
            if (MODE == EPI_REDUCE && st < 32 && st < bnc) ebv += (N - 1) * args.ev[qbase + st] - args.es[args.i0 + tp.outer];
            const int err = st == 0 && (t & 7) == 0 ? *(volatile int*)args.err : 0;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int r = st + 64 * j, rr = tp.rr0 + r;
                const int64_t o = tp.row0 + r;
                row_in[j] = args.RB == 0 || rr < args.R;          // (a last block reads past its index)
                ea[j] = row_in[j] ? __ldg(args.ea + (args.ea_outer ? (args.RB > 0 ? (int64_t)tp.outer : o) : o)) : 0;
                if (MODE == EPI_SLICE && N >= 4 && (rr >> lg) < args.nt) tup[j] = __ldg(args.ttup + (rr >> lg));
                if (MODE == EPI_SLAB && N >= 2) tup[j] = __ldg(args.stup + rr);
                if (MODE == EPI_REDUCE && row_in[j]) tup[j] = __ldg(args.tuples + rr);
                if (MODE == EPI_DIVIDE) {                         // (the tables cover whole tiles)
                    sm[j] = __ldg(args.smeta + rr);
#pragma unroll
                    for (int m = 0; m < 6; ++m) sg[j][m] = __ldg(args.ssum + (int64_t)m * args.nslot + rr);
                }
            }
            double2 lq = make_double2(0.0, 0.0);
            if (MODE == EPI_DIVIDE) {
                vcols = min(vcols, __ldg(args.tpmax + tp.rr0 / NP) - qbase + 1);
                // lambda_q - lambda_i, so that D = sigma_row + (lambda_q - lambda_i) needs no FP64
                // per element (FP64 runs at a small fraction of the FP32 rate)
                if (st >= 32 && st - 32 < bnc && qbase + st - 32 < args.ncv)
                    lq = csub(args.lam[qbase + st - 32], args.lam[args.i0 + tp.outer]);
            } else if ((MODE == EPI_SLICE || MODE == EPI_V) && args.colmask) {
                vcols = min(vcols, tile_pmax(args, lg, tp) - qbase + 1);
            }
            if (MODE == EPI_SLICE) {
                // output slot of (p_2 = q, the sub-block's shared p's); order 2: slot q
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int tt = (tp.rr0 >> lg) + (st >> 5) + 2 * j, q = qbase + (st & 31);
                    sea[j] = N >= 3 ? 0 : q;
                    if (N >= 3 && (st >> 5) + 2 * j < (NP >> lg) && tt < args.nt) {
                        const uint32_t pp = N == 3 ? (uint32_t)tt : __ldg(args.ttup + tt);
                        const int p3 = (int)(pp & 255u), p4 = (int)((pp >> 8) & 255u);
                        if (q <= p3) sea[j] = N == 3 ? __ldg(args.segbase + q) + p3 - q
                                                     : __ldg(args.segbase + rank2(q, p3)) + p4 - p3;
                    }
                }
            }
            if (st == 0) {
                // columns of this tile that any row uses: below the modes in use and, with the
                // sorted-tuple mask, at most the largest leading p of the tile's rows. Columns past
                // them are neither read nor written, so the column groups split only the used ones.
                int* meta = (int*)(tb + C::META);
                meta[0] = qbase;
                meta[1] = max(vcols, 0);
                meta[2] = tp.outer;
                meta[3] = tp.rr0;
                meta[4] = !alive || err != 0;   // (another role's error is picked up every 8 tiles)
            }
            if (st < 32) ((int*)(tb + C::COLEB))[st] = ebv;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int r = st + 64 * j;
                int4 rm = make_int4(ea[j], NP, 0, 0);             // .y: the new index is <= it (-1: no row)
                if (MODE == EPI_V) {
                    if (args.colmask) rm.y = tp.outer % args.nm;
                    if (!row_in[j]) rm.y = -1;
                } else if (MODE == EPI_SLICE) {
                    const int tt = (tp.rr0 + r) >> lg;            // row (p_3..p_N, a_1)
                    if (N == 3) rm.y = tt;
                    if (N >= 4) rm.y = (int)(tup[j] & 255u);
                    if (!row_in[j] || tt >= args.nt) rm.y = -1;
                } else if (MODE == EPI_DIVIDE) {
                    rm.y = sm[j].x;
                    rm.z = sm[j].y;
                    rm.w = sm[j].z;
#pragma unroll
                    for (int m = 0; m < 6; ++m) ((float*)(tb + C::SIG))[m * NP + r] = sg[j][m];
                    const bool ok = sm[j].x >= 0;
                    const int seg = (sm[j].z >> 8) & 15;
                    const int hi = __reduce_max_sync(0xffffffffu, sm[j].x);
                    const int lo = __reduce_min_sync(0xffffffffu, ok ? seg : SEGS);
                    const int up = __reduce_max_sync(0xffffffffu, ok ? seg : -1);
                    if (lane == 0) ((int4*)(tb + C::QINFO))[r / 32] = make_int4(hi, lo, up, 0);
                } else if (MODE == EPI_SLAB) {
                    const bool ok = N >= 2 ? tup[j] != 0xFFFFFFFFu : tp.row0 + r < args.nouter;
                    rm.y = !ok ? -1 : N >= 2 ? (int)(tup[j] & 255u) : NP;
                    rm.z = (int)tup[j];
                } else {
                    // the row's last index p_{N-1} and the rank of its pair (p_1, p_2)
                    const int p0 = (int)(tup[j] & 255u), p1 = (int)((tup[j] >> 8) & 255u);
                    const int pin = (int)((tup[j] >> (8 * (N - 2))) & 255u);
                    rm.z = !row_in[j] || N < 3 ? -1 : rank2(p0, p1);
                    rm.y = row_in[j] ? pin : -1;
                    // rows in colex order mostly share p_{N-1}: its weight is then applied once to the
                    // quarter's sum instead of to every element
                    const int hi = __reduce_max_sync(0xffffffffu, rm.y);
                    const int lo = __reduce_min_sync(0xffffffffu, row_in[j] ? pin : NP);
                    if (lane == 0)
                        ((int4*)(tb + C::QINFO))[r / 32] = make_int4(N >= 4 && hi >= 0 && hi == lo ? hi : -1, 0, 0, 0);
                }
                ((int4*)(tb + C::ROWM))[r] = rm;
            }
            if (MODE == EPI_DIVIDE && st >= 32) {
                const int c = st - 32;
                ((float2*)(tb + C::LAMF))[c] = make_float2((float)lq.x, (float)lq.y);
                ((tfl*)(tb + C::LAMT))[2 * c] = to_tfl(lq.x);
                ((tfl*)(tb + C::LAMT))[2 * c + 1] = to_tfl(lq.y);
            }
            if (MODE == EPI_SLICE) {
#pragma unroll
                for (int j = 0; j < 2; ++j) ((int*)(tb + C::SROWQ))[32 * ((st >> 5) + 2 * j) + (st & 31)] = sea[j];
            }
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&sfull[buf]);
            if (trc && st == 0) trc[5] = global_ns() - t0;
            ++t;
        }
    } else {
        // ---------------- epilogue
        const int et = threadIdx.x - 64;                    // 0 .. 32 * EPI_WARPS - 1
        const int q4 = warp % 4;                            // TMEM lane quarter of this warp
        const int grp = (warp - 2) / 4;                     // column group (EPI_WARPS / 4 groups)
        const int rl = q4 * 32 + lane;                      // local row within the tile
        const uint32_t trow0 = tmem + ((uint32_t)(q4 * 32) << 16);
        constexpr int NGRP = EPI_WARPS / 4;                 // column groups per lane quarter
        const int N = args.N, n = args.n;
        const int sb = rl >> lg;                            // sub-block of the tile (warp-uniform)
        // EPI_REDUCE: running sums of this thread's rows (a warp's columns are at most 8: 32 over four
        // groups), the p_{N-1} whose weight they still lack (-1: none), and where they belong
        dfl sr[8], si[8];
        int red_w = -1, red_outer = -1, red_q = 0, red_cols = 0, red_c0 = 0;
#pragma unroll
        for (int c = 0; c < 8; ++c) { sr[c] = {0.f, 0.f}; si[c] = {0.f, 0.f}; }
        // -sum over the warp's 32 rows, times the missing weight, into Psi_N[i][k]: exchanges with the
        // lanes 16, 8 and 4 apart halve the columns a lane carries (8 -> 4 -> 2 -> 1), those 2 and 1
        // apart finish them. Once per run of tiles instead of once a tile, with two barriers and FP64
        // products: the reduction's epilogue took 11.6 us per 64 columns and tile.
        auto flush = [&] {
            if (red_outer >= 0) {
#pragma unroll
                for (int step = 0; step < 3; ++step) {
                    const int off = 16 >> step, half = 4 >> step;
                    const bool up = (lane & off) != 0;
#pragma unroll
                    for (int j = 0; j < half; ++j) {
                        const dfl tr = up ? sr[j] : sr[j + half], ti = up ? si[j] : si[j + half];
                        const dfl mr = up ? sr[j + half] : sr[j], mi = up ? si[j + half] : si[j];
                        sr[j] = df_add(mr, dfl{__shfl_xor_sync(0xffffffffu, tr.hi, off),
                                               __shfl_xor_sync(0xffffffffu, tr.lo, off)});
                        si[j] = df_add(mi, dfl{__shfl_xor_sync(0xffffffffu, ti.hi, off),
                                               __shfl_xor_sync(0xffffffffu, ti.lo, off)});
                    }
                }
#pragma unroll
                for (int off = 2; off > 0; off >>= 1) {
                    sr[0] = df_add(sr[0], dfl{__shfl_xor_sync(0xffffffffu, sr[0].hi, off),
                                              __shfl_xor_sync(0xffffffffu, sr[0].lo, off)});
                    si[0] = df_add(si[0], dfl{__shfl_xor_sync(0xffffffffu, si[0].hi, off),
                                              __shfl_xor_sync(0xffffffffu, si[0].lo, off)});
                }
                // the column by the lane's bits 16, 8 and 4
                const int col = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
                const int qc = red_q + red_c0 + col;
                if ((lane & 3) == 0 && col < red_cols && qc < args.ncv &&
                    (sr[0].hi != 0.f || si[0].hi != 0.f)) {
                    double2 v = make_double2(df_to_d(sr[0]), df_to_d(si[0]));
                    if (red_w >= 0) {
                        const float4 x = __ldg(args.psi_df + qc * n + red_w);
                        v = cmul(v, make_double2((double)x.x + (double)x.y, (double)x.z + (double)x.w));
                    }
                    // the exponents of the N - 1 weights, and those taken from G
                    v = times_pow2(v, (N - 1) * (args.eb[qc] - args.ev[qc]) + args.es[args.i0 + red_outer]);
                    const int64_t at = (int64_t)(args.i0 + red_outer) * n + qc;
                    atomicAdd(&args.out_f64[at].x, -v.x);
                    atomicAdd(&args.out_f64[at].y, -v.y);
                }
            }
#pragma unroll
            for (int c = 0; c < 8; ++c) { sr[c] = {0.f, 0.f}; si[c] = {0.f, 0.f}; }
        };
        uint32_t t = 0;
        for (int64_t k = kbeg; k < kend; k += kstep) {
            const int buf = (int)(t & 1);
            unsigned long long* trc = nullptr;
            if (args.trace)
                trc = args.trace + 6 * (MODE == EPI_REDUCE ? k * args.ncol_tiles + tile_pos(args, k).ct
                                        : args.tiles       ? (int64_t)args.tiles[k] : k);
            uint8_t* tb = tables + C::TILE + buf * C::TILE_BYTES;
            const int* meta = (const int*)(tb + C::META);
            const bool got = tc::mbar_wait(&sfull[buf], (t >> 1) & 1, args.err, kErrTimeout);
            if (epi_any(!got || meta[4] != 0)) break;       // uniform over the epilogue warps
            const int qbase = meta[0], vcols = meta[1], outer0 = meta[2], rr = meta[3] + rl;
            const int* colEb = (const int*)(tb + C::COLEB);
            int* colE = colE_all + buf * C::COLE_N;         // this tile's keys; the other tile parity's
            if (MODE != EPI_REDUCE)                         // are cleared for the next tile
                for (int e = et; e < C::COLE_N; e += 32 * EPI_WARPS) colE_all[(buf ^ 1) * C::COLE_N + e] = 0;
            const int units = (vcols + 3) / 4;
            const int cbeg = 4 * ((grp * units) / NGRP);
            const int cols = 4 * (((grp + 1) * units) / NGRP) - cbeg;
            const int4 rm = ((const int4*)(tb + C::ROWM))[rl];
            const int ea = rm.x, firstp = rm.y;             // the new index is <= firstp
            const bool row_ok = firstp >= 0;
            const int kpos = MODE == EPI_DIVIDE ? rm.w & 255 : rl & ((1 << lg) - 1);   // K position in the next row
            const int seg = (rm.w >> 8) & 15, run1 = (rm.w >> 13) & 7, den = (rm.w >> 16) & 255;
            const int* qinfo = (const int*)(tb + C::QINFO) + 4 * q4;
            const tfl* lamt = (const tfl*)(tb + C::LAMT);
            const float2* lamf = (const float2*)(tb + C::LAMF);
            const float* sig = (const float*)(tb + C::SIG) + rl;
            const int* srowq = (const int*)(tb + C::SROWQ) + 32 * sb;
            int64_t vbase = 0;                              // EPI_V: V of the new index 0
            if (MODE == EPI_V)
                vbase = (args.colmask ? (int64_t)(outer0 / args.nm) * rank2(0, args.nm) + rank2(0, max(firstp, 0))
                                      : (int64_t)outer0 * args.nm) * args.R + rr;
            // sum of the row's eigenvalues minus lambda_i in FP64 (slabs, and the FP64 quotient)
            double2 sigma = make_double2(0.0, 0.0);
            const int i_row = args.i0 + (MODE == EPI_SLAB && args.RB == 0 ? rr + (int)(tile_at(k) / args.ncol_tiles) * NP : outer0);
            if (MODE == EPI_SLAB && row_ok) {
#pragma unroll
                for (int m = 0; m < 3; ++m)
                    if (m < N - 1) sigma = cadd(sigma, args.lam[((unsigned)rm.z >> (8 * m)) & 255u]);
                sigma = csub(sigma, args.lam[i_row]);
            }
            if (MODE == EPI_DIVIDE && args.fp64_quotient && row_ok)
                sigma = csub(args.ssig[rr], args.lam[i_row]);
            if (trc && et == 0) {
                trc[0] = global_ns();
                trc[4] = blockIdx.x + 1;
            }
            // warp-uniform (the epilogue's shuffles and TMEM loads are warp-collective)
            const uint32_t trow = trow0 + (uint32_t)buf * (TMEM_COLS / 2);
            const bool ok = __all_sync(0xffffffffu, tc::mbar_wait(&tfull[buf], (t >> 1) & 1, args.err, kErrTimeout));
            tc::fence_after_sync();
            if (trc && et == 0) trc[1] = global_ns();         // accumulators complete

            // h of one element in native FP64 (EPI_SLAB, and EPI_DIVIDE with fp64_quotient):
            // V * 2^(ea+eb-VEXP) / N! (times the multiplicity for the reduction), divided by the
            // clamped denominator
            auto quotient = [&](long long Vr, long long Vi, int eb, int qc) -> double2 {
                double f = args.invfact;                      // 1 / N!, or 1 / prod(run lengths)!
                if (MODE == EPI_DIVIDE) f = 1.0 / (double)(den * (qc == firstp ? run1 + 1 : 1));
                const double sc = pow2d(ea + eb - VEXP) * f;
                double2 h = make_double2((double)Vr * sc, (double)Vi * sc);
                if (args.divide) {
                    // h / D = h conj(D) / |D|^2, D clamped per Alg. 2 step 9
                    double2 D = cadd(sigma, args.lam[qc]);
                    double m2 = fma(D.x, D.x, D.y * D.y);
                    if (m2 < args.eps * args.eps) {
                        D = make_double2(args.eps, 0.0);
                        m2 = args.eps * args.eps;
                    }
                    const double r = __drcp_rn(m2);
                    h = make_double2(fma(h.x, D.x, h.y * D.y) * r, fma(h.y, D.x, -h.x * D.y) * r);
                }
                return h;
            };

            if (MODE == EPI_SLICE || MODE == EPI_DIVIDE) {
                // pass 1: column exponents (max over the tile's valid rows, per next operand row).
                // For the quotients an FP32 upper bound of |h| = |V| 2^(ea+eb-VEXP) f / |D| with a
                // lower bound of the clamped |D| (FP32 error of the sum bounded by 4 ulp of its
                // terms).
                float2 sf = make_float2(0.f, 0.f);
                if (MODE == EPI_DIVIDE) sf = make_float2(sig[0], sig[3 * NP]);
                if (ok) {
                    constexpr float deep = deep_level_bound(S);
                    for (int c4 = cbeg; c4 < cbeg + cols; c4 += 4) {
                        if (MODE == EPI_DIVIDE && qbase + c4 > qinfo[0]) break;   // no row of the warp
                        uint32_t rv[2][4], iv[2][4];   // levels 0 and 1 only
                        tc::tmem_ld4(trow + c4, rv[0]);
                        tc::tmem_ld4(trow + c4 + lstride, rv[1]);
                        tc::tmem_ld4(trow + bnc + c4, iv[0]);
                        tc::tmem_ld4(trow + bnc + c4 + lstride, iv[1]);
                        tc::tmem_wait_ld();
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const int cl = c4 + c;
                            const int qc = qbase + cl;
                            const int eb = colEb[cl];
                            // upper bounds of |V_re|, |V_im| in units of 2^30 (V = (L0 + L1 + L2 +
                            // L3) 2^30)
                            const float br = level_bound01(rv[0][c], rv[1][c], deep);
                            const float bi = level_bound01(iv[0][c], iv[1][c], deep);
                            unsigned key = 0;
                            if (MODE == EPI_SLICE) {
                                const bool valid = kpos < n && qc < args.ncv && qc <= firstp;
                                // bitlen(V) <= exponent(bound) + 30
                                const float bm = fmaxf(br, bi);
                                if (valid && bm > 0.f)
                                    key = (unsigned)(f32_exponent(bm) + 30 + ea + eb - VEXP + 8192);
                                const unsigned wmax = __reduce_max_sync(0xffffffffu, key);
                                if (lane == 0 && wmax) atomicMax(&colE[32 * sb + cl], (int)wmax);
                            } else {
                                if (qc < args.ncv && qc <= firstp && (br > 0.f || bi > 0.f)) {
                                    float lb = 1.0f;
                                    if (args.divide) {
                                        const float2 lq = lamf[cl];
                                        const float dx = sf.x + lq.x, dy = sf.y + lq.y;
                                        const float del = 2.4e-7f * (fabsf(sf.x) + fabsf(sf.y) +
                                                                    fabsf(lq.x) + fabsf(lq.y));
                                        lb = fmaxf(sqrtf(fmaf(dx, dx, dy * dy)) - del, (float)args.eps);
                                    }
                                    const float fm = rcp[den * (qc == firstp ? run1 + 1 : 1)].hi;
                                    const float hm = sqrtf(fmaf(br, br, bi * bi)) * fm / lb *
                                                     (1.0f + 0.0009765625f);
                                    key = (unsigned)(f32_exponent(hm) + 30 + ea + eb - VEXP + 8192);
                                }
                                for (int g = qinfo[1]; g <= qinfo[2]; ++g) {
                                    const unsigned wmax = __reduce_max_sync(0xffffffffu, seg == g ? key : 0u);
                                    if (lane == 0 && wmax) atomicMax(&colE[32 * g + cl], (int)wmax);
                                }
                            }
                        }
                    }
                }
                epi_sync();
                if (trc && et == 0) trc[2] = global_ns();
            }

            if (MODE == EPI_REDUCE && ok) {
                // G[c'][k] times the weights of the row's p's in double-float, summed by each thread over
                // the tiles of one (upper index, column tile) whose rows in this quarter share p_{N-1}
                const int pin = max(firstp, 0), pre = rm.z;
                const bool uni = qinfo[0] >= 0;
                const int wp = qinfo[0];
                if (wp != red_w || outer0 != red_outer || qbase != red_q) {
                    flush();
                    red_w = wp;
                    red_outer = outer0;
                    red_q = qbase;
                    red_cols = cols;
                    red_c0 = cbeg;
                }
                // two columns a round, the sums rotating through the first two registers (an unrolled
                // body of eight elements does not fit the instruction cache beside the other roles)
#pragma unroll 1
                for (int h = 0; h < 4; ++h) {
                    const int c2 = cbeg + 2 * h;
                    // the weights of these columns, asked for before the accumulators (1.17 ms a call at n =
                    // 120, order 3, against 1.44 behind them), of a valid row and column in any case.
                    // Order 3: the whole weight W[p_1][k] W[p_2][k]; order 4: that, and W[p_3][k] unless it
                    // is left to the sum
                    float4 w4[2];
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const int qa = min(qbase + c2 + c, args.ncv - 1);
                        w4[c] = pre >= 0 ? __ldg(args.wpre + (int64_t)qa * args.ldw + pre) : __ldg(args.psi_df + qa * n + pin);
                    }
                    uint32_t rv[4][2], iv[4][2];
                    load_levels<S, 2>(trow + min(c2, bnc - 2), lstride, rv);
                    load_levels<S, 2>(trow + bnc + min(c2, bnc - 2), lstride, iv);
                    tc::tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const int cl = c2 + c;
                        const int qc = qbase + cl;
                        const dfl vr = level_sum_df(rv[0][c], rv[1][c], rv[2][c], rv[3][c]);
                        const dfl vi = level_sum_df(iv[0][c], iv[1][c], iv[2][c], iv[3][c]);
                        if (row_ok && 2 * h < cols && qc < args.ncv && (vr.hi != 0.f || vi.hi != 0.f)) {
                            const int sc = ea + colEb[cl] - VEXP + 30, s1 = max(-126, min(126, sc));
                            const float f = pow2f(s1);
                            dfl gr = {vr.hi * f, vr.lo * f}, gi = {vi.hi * f, vi.lo * f};
                            if (sc != s1) {   // (values near the ends of FP32's range)
                                gr = {ldexpf(gr.hi, sc - s1), ldexpf(gr.lo, sc - s1)};
                                gi = {ldexpf(gi.hi, sc - s1), ldexpf(gi.lo, sc - s1)};
                            }
                            dfl wr = {w4[c].x, w4[c].y}, wi = {w4[c].z, w4[c].w};
                            if (N >= 4 && !uni) {
                                const float4 x = __ldg(args.psi_df + qc * n + pin);
                                const dfl xr = {x.x, x.y}, xi = {x.z, x.w};
                                const dfl tr = df_dot2(wr, xr, df_neg(wi), xi);
                                wi = df_dot2(wr, xi, wi, xr);
                                wr = tr;
                            }
                            sr[c] = df_add(sr[c], df_dot2(gr, wr, df_neg(gi), wi));
                            si[c] = df_add(si[c], df_dot2(gr, wi, gi, wr));
                        }
                    }
                    const dfl r0 = sr[0], r1 = sr[1], i0 = si[0], i1 = si[1];
#pragma unroll
                    for (int c = 0; c < 6; ++c) { sr[c] = sr[c + 2]; si[c] = si[c + 2]; }
                    sr[6] = r0; sr[7] = r1; si[6] = i0; si[7] = i1;
                }
            }
            if (MODE != EPI_REDUCE && ok) {
                // pass 2 (or the only pass): outputs
                constexpr int UC = MODE == EPI_DIVIDE ? 2 : 4;   // columns a round (instruction cache)
#pragma unroll 1
                for (int c4 = cbeg; c4 < cbeg + cols; c4 += UC) {
                    if (MODE == EPI_DIVIDE && qbase + c4 > qinfo[0]) break;
                    uint32_t rv[4][UC], iv[4][UC];
                    load_levels<S, UC>(trow + c4, lstride, rv);
                    load_levels<S, UC>(trow + bnc + c4, lstride, iv);
                    tc::tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < UC; ++c) {
                        const int cl = c4 + c;
                        const int qc = qbase + cl;
                        const int eb = colEb[cl];
                        const bool valid = qc < args.ncv && qc <= firstp;
                        if (MODE == EPI_V) {
                            longlong2 v = make_longlong2(0ll, 0ll);
                            if (valid) {
                                v.x = combine(rv[0][c], rv[1][c], rv[2][c], rv[3][c]);
                                v.y = combine(iv[0][c], iv[1][c], iv[2][c], iv[3][c]);
                                args.out_v[vbase + (int64_t)qc * args.R] = v;
                            }
                            if (args.emax) {
                                const unsigned key = v.x | v.y ? (unsigned)(bitlen(v) + ea + eb - VEXP + 8192) : 0u;
                                const unsigned wmax = __reduce_max_sync(0xffffffffu, key);
                                if (lane == 0 && wmax) atomicMax(&colE[cl], (int)wmax);
                            }
                            continue;
                        }
                        if (MODE == EPI_SLAB) {
                            // store h^i_{pre, q} when the multiset (q, row p's) minus pre is {extra}
                            const long long Vr = combine(rv[0][c], rv[1][c], rv[2][c], rv[3][c]);
                            const long long Vi = combine(iv[0][c], iv[1][c], iv[2][c], iv[3][c]);
                            if (!valid || !(Vr | Vi)) continue;
                            const double2 h = quotient(Vr, Vi, eb, qc);
                            int tt[8];
                            tt[0] = qc;
                            for (int m = 0; m < N - 1; ++m) tt[m + 1] = (int)(((unsigned)rm.z >> (8 * m)) & 255u);
                            int used[8] = {0, 0, 0, 0, 0, 0, 0, 0};
                            int matched = 0, extra = -1, nextra = 0;
                            for (int a = 0; a < N; ++a) {
                                bool hit = false;
                                for (int b = 0; b < N - 1 && !hit; ++b)
                                    if (!used[b] && args.pre[b] == tt[a]) { used[b] = 1; hit = true; }
                                if (hit) ++matched;
                                else { extra = tt[a]; ++nextra; }
                            }
                            if (matched == N - 1 && nextra == 1)
                                args.out_f64[(int64_t)i_row * n + extra] = h;
                            continue;
                        }
                        uint32_t w[S];
                        if (MODE == EPI_SLICE) {
                            if (!valid || kpos >= args.kout) continue;   // unused rows and entries
                            const int64_t rowp = (int64_t)outer0 * args.RS + srowq[cl];
                            const int key = colE[32 * sb + cl];
                            const int E = key ? key - 8192 : EXP_NONE;
                            if (key == 0 || kpos >= n) {
#pragma unroll
                                for (int s = 0; s < S; ++s) w[s] = 0u;
                            } else {
                                const long long Vr = combine(rv[0][c], rv[1][c], rv[2][c], rv[3][c]);
                                const long long Vi = combine(iv[0][c], iv[1][c], iv[2][c], iv[3][c]);
                                const int sh = ea + eb - VEXP - E + 7 + 8 * (S - 1);
                                digit_pairs<S>(shift_round(Vr, sh), shift_round(Vi, sh), w);
                            }
                            // next operand row rowp: 2^lg complex K entries (BF16 pairs), K = kpos
                            uint32_t* dst = reinterpret_cast<uint32_t*>(args.out_planes) + (rowp << lg) + kpos;
#pragma unroll
                            for (int s = 0; s < S; ++s) dst[s * (args.out_plane_stride / 2)] = w[s];
                            if (kpos == 0) args.out_exp[rowp] = E;
                            continue;
                        }
                        // EPI_DIVIDE: reduction row (p_1 = q, .., p_{N-1}), K = p_N
                        if (!valid) continue;
                        const int64_t rowp = (int64_t)outer0 * args.RT + rm.z + qc;
                        const int key = colE[32 * seg + cl];
                        const int E = key ? key - 8192 : EXP_NONE;
                        if (key == 0) {
#pragma unroll
                            for (int s = 0; s < S; ++s) w[s] = 0u;
                        } else if (args.fp64_quotient) {
                            const long long Vr = combine(rv[0][c], rv[1][c], rv[2][c], rv[3][c]);
                            const long long Vi = combine(iv[0][c], iv[1][c], iv[2][c], iv[3][c]);
                            const double2 h = quotient(Vr, Vi, eb, qc);
                            const double sc = pow2d(7 + 8 * (S - 1) - E);
                            digit_pairs<S>(__double2ll_rn(h.x * sc), __double2ll_rn(h.y * sc), w);
                        } else {
                            // W = V 2^-30 f / D 2^k in double-float arithmetic; D from exact
                            // triple-float terms, so near-resonant cancellation stays exact
                            const dfl vr = level_sum_df(rv[0][c], rv[1][c], rv[2][c], rv[3][c]);
                            const dfl vi = level_sum_df(iv[0][c], iv[1][c], iv[2][c], iv[3][c]);
                            dfl Dr = {1.f, 0.f}, Di = {0.f, 0.f};
                            if (args.divide) {
                                Dr = tfl_sum(tfl{sig[0], sig[NP], sig[2 * NP]}, lamt[2 * cl]);
                                Di = tfl_sum(tfl{sig[3 * NP], sig[4 * NP], sig[5 * NP]}, lamt[2 * cl + 1]);
                            }
                            dfl m2 = df_dot2(Dr, Dr, Di, Di);      // (no cancellation: one step normalises)
                            m2 = df_norm(m2.hi, m2.lo);
                            if (args.divide && m2.hi < args.eps2f) {   // Alg. 2 step 9
                                Dr = to_dfl(args.eps);
                                Di = {0.f, 0.f};
                                m2 = df_mul(Dr, Dr);
                            }
                            const float r0 = __frcp_rn(m2.hi);
                            const dfl e1 = df_add(dfl{1.f, 0.f}, df_neg(df_mul(m2, dfl{r0, 0.f})));
                            const dfl inv = df_add(dfl{r0, 0.f}, df_mul(dfl{r0, 0.f}, e1));
                            const dfl rf = df_mul(inv, rcp[den * (qc == firstp ? run1 + 1 : 1)]);
                            const dfl nr = df_dot2(vr, Dr, vi, Di);
                            const dfl ni = df_dot2(vi, Dr, df_neg(vr), Di);
                            const int e = ea + eb - VEXP + 30 + 7 + 8 * (S - 1) - E;
                            const dfl qr = df_mul(nr, rf), qi = df_mul(ni, rf);
                            digit_pairs<S>(df_round_i64(dfl{ldexpf(qr.hi, e), ldexpf(qr.lo, e)}),
                                           df_round_i64(dfl{ldexpf(qi.hi, e), ldexpf(qi.lo, e)}), w);
                        }
                        uint32_t* dst = reinterpret_cast<uint32_t*>(args.out_planes) + (rowp << args.lgout) + kpos;
#pragma unroll
                        for (int s = 0; s < S; ++s) dst[s * (args.out_plane_stride / 2)] = w[s];
                        // the row's first entry holds p_N = p_{N-1} (order 2: p_2 = p_1 = q)
                        if (N >= 3 ? (rm.w & 4096) != 0 : kpos == qc) args.out_exp[rowp] = E;
                    }
                }
            }
            tc::fence_before_sync();
            epi_sync();
            if (MODE == EPI_V && args.emax && et < bnc && qbase + et < args.ncv && colE[et])
                atomicMax(&args.emax[qbase + et], colE[et] - 8192);
            if (trc && et == 0) trc[3] = global_ns();
            if (et == 0) {
                tc::mbar_arrive(&tempty[buf]);
                tc::mbar_arrive(&sempty[buf]);
            }
            ++t;
        }
        if (MODE == EPI_REDUCE) flush();
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, TMEM_COLS);
    }
}

// Zeros in the reduction rows' K entries that its tiles read but the divide does not write: from
// the chunk of the tile's smallest p_{N-1} up to the row's own p_{N-1}, and from nm to the operand's
// inner extent. It runs before the divide and clears whole 32-byte sectors (8 entries, also those that
// the divide then writes), since a partly written sector is read from HBM first: 0.18 ms at n = 60, order
// 4, against 0.52 entry by entry behind the divide.
// kc: complex K entries a chunk (a multiple of 8). t: one of 8 threads a row.
template <int S>
__device__ __forceinline__ void zero_head(int64_t t, int N, int nm, int kc, int lg, int Q, const uint32_t* __restrict__ tuples,
                                          uint32_t* __restrict__ planes, int64_t plane_stride_u32)
{
    const int e = (int)(t & 7);
    const int64_t row = t >> 3;
    const int outer = (int)(row / Q), r = (int)(row - (int64_t)outer * Q);
    const int sh = 8 * (N - 2);
    const int p = (int)((tuples[r] >> sh) & 255u);
    const int p0 = (int)((tuples[r & ~(NP - 1)] >> sh) & 255u);
    uint32_t* dst = planes + (row << lg);
    for (int k = p0 / kc * kc + e; k < (p + 7) / 8 * 8; k += 8)
#pragma unroll
        for (int s = 0; s < S; ++s) dst[s * plane_stride_u32 + k] = 0u;
    const int end = min(1 << lg, (nm + 7) / 8 * 8);
    for (int k = nm / 8 * 8 + e; k < end; k += 8)
#pragma unroll
        for (int s = 0; s < S; ++s) dst[s * plane_stride_u32 + k] = 0u;
}

template <int S>
__global__ void k_zero_heads(int N, int nm, int kc, int lg, int Q, int nouter, const uint32_t* __restrict__ tuples,
                             uint32_t* __restrict__ planes, int64_t plane_stride_u32)
{
    pdl_wait();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < (int64_t)Q * nouter * 8) zero_head<S>(t, N, nm, kc, lg, Q, tuples, planes, plane_stride_u32);
}

// Start of a term: the output (zeroed unless the term is added to it), the exponents of S, the error
// flag (nullptr: a batch's, or one that holds earlier orders), and where they exist the pairs' weights
// wpre[k][t] = W[p_1][k] W[p_2][k] 2^(-2 we[k]) (FP64 products as double-float complex) and the reduction
// rows' heads (when their buffer is the reduction's own).
struct TermInit {
    double2* out;
    int64_t cells;
    int* sE;                 // (nullptr: S stays)
    int n, nm;
    int* err;
    const double2* W;
    const int* we;           // exponents of W's columns
    const uint32_t* pairs;
    int64_t npairs;
    float4* wpre;
    int64_t heads;           // threads for the heads (8 a row), 0: none
    int N, kc, lg, Q;
    const uint32_t* tuples;
    uint32_t* planes;
    int64_t plane_stride_u32;
};
template <int S>
__global__ void k_term_init(const __grid_constant__ TermInit a)
{
    pdl_wait();
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = t0; t < a.cells; t += step) a.out[t] = make_double2(0.0, 0.0);
    if (t0 < a.nm && a.sE) a.sE[t0] = EXP_NONE;
    if (t0 == 0 && a.err) *a.err = 0;
    for (int64_t t = t0; t < a.npairs * a.n; t += step) {
        const int k = (int)(t / a.npairs);
        const uint32_t p = a.pairs[t - k * a.npairs];
        const double2 w = times_pow2(cmul(a.W[(int64_t)(p & 255u) * a.n + k], a.W[(int64_t)((p >> 8) & 255u) * a.n + k]),
                                     -2 * a.we[k]);
        const float rh = (float)w.x, ih = (float)w.y;
        a.wpre[t] = make_float4(rh, (float)(w.x - rh), ih, (float)(w.y - ih));
    }
    for (int64_t t = t0; t < a.heads; t += step)
        zero_head<S>(t, a.N, a.nm, a.kc, a.lg, a.Q, a.tuples, a.planes, a.plane_stride_u32);
}

// Operand rows of a mode product from the exact 64-bit values V of the stage before (EPI_V): a warp
// takes RW rows (outer, sorted M-tuple of a's) at a time, CH chunks of 32 entries a row: lane t
// covers a = t, t + 32, .. It gathers V[outer][rank(sort(tuple, a))] and writes its digits. V is in
// units of 2^(ea + eb - VEXP).
//   SRC 0: V of the first mode product, outer = (i, p); ea by i, eb by p
//   SRC 1: V of the second (order 4), outer = (i, p_3 <= p_4); ea by its operand row (i, p_4, rank),
//          eb by p_3
//   SRC 2: V of the upper contraction (M = N - 1), outer = i; ea by rank (the tensor's), eb by i, and
//          the rows share the exponent rowE[i]; the others get their exact one (largest bit length)
// Neighbouring rows gather neighbouring entries (colexicographic rank), so the warps of a block
// share sectors. A block takes one outer index and a strided share of its rows, so that nothing
// but the gather, the shifts and the digits is left per row: a rank is one of M + 1 row constants
// plus a binomial of the lane's a, kept in registers, and a plane's address a 32-bit offset from the
// block's (4.51 ms at n = 60, order 4, against 5.50 with whole ranks and 64-bit addresses per entry).
// Bound by HBM writes at n = 120 (4 S bytes an entry against 16 read per source entry: 1.10 ms for
// 6.65 GB at order 3), below by the scattered half of the gathers and the integer instructions.
template <int S, int M, int SRC, int CH, int RW>
__global__ void __launch_bounds__(256)
    k_regather(const longlong2* __restrict__ V, int64_t Rsrc, int n, int nm, int nt, const uint32_t* __restrict__ ttup,
               const int* __restrict__ ea, const int* __restrict__ eb, const int* __restrict__ rowE, int lg, int kout,
               int nrows, int64_t Rdst, unsigned parts, const uint32_t* __restrict__ tuples,
               uint32_t* __restrict__ planes, int64_t plane_stride_u32, int* __restrict__ out_exp)
{
    const int lane = threadIdx.x & 31;
    const unsigned outer = blockIdx.x / parts;
    int au[CH], bin2[CH], bin3[CH], bin4[CH];                // a; rank of (0, a), (0, 0, a), (0, 0, 0, a)
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        au[c] = lane + 32 * c;
        bin2[c] = rank2(0, au[c]);
        bin3[c] = M >= 2 ? rank3(0, 0, au[c]) : 0;
        bin4[c] = M >= 3 ? rank4(0, 0, 0, au[c]) : 0;
    }
    pdl_wait();
    int e0;
    const int* earow = ea;
    if (SRC == 2) {
        e0 = eb[outer] - VEXP;
    } else {
        const unsigned i = outer / (unsigned)nt, t = outer - i * (unsigned)nt;
        const uint32_t tp = SRC == 1 ? ttup[t] : t;          // the newest p in the low byte
        e0 = eb[tp & 255u] - VEXP + (SRC == 0 ? ea[i] : 0);
        if (SRC == 1) earow = ea + ((int64_t)i * nm + (int)((tp >> 8) & 255u)) * Rsrc;
    }
    const longlong2* src = V + outer * Rsrc;
    uint32_t* dst[S];
#pragma unroll
    for (int s = 0; s < S; ++s) dst[s] = planes + s * plane_stride_u32 + ((int64_t)outer * Rdst << lg);
    int* oexp = SRC == 2 ? nullptr : out_exp + outer * Rdst;
    const int Eall = SRC == 2 ? rowE[outer] : 0;
    const int step = (int)parts * 8 * RW;
    for (int row = ((int)(blockIdx.x - outer * parts) * 8 + (int)(threadIdx.x >> 5)) * RW; row < nrows; row += step) {
        longlong2 v[RW][CH];
        int ex[RW][CH], E[RW];
#pragma unroll
        for (int j = 0; j < RW; ++j) {
            const int r = min(row + j, nrows - 1);           // (a last round repeats its last row)
            int x = r, y = 0, z = 0;
            if (M >= 2) {
                const uint32_t pk = tuples[r];
                x = (int)(pk & 255u);
                y = (int)((pk >> 8) & 255u);
                z = (int)((pk >> 16) & 255u);
            }
            // rank less the part of a: a below x, between x and y, between y and z, above
            const int last = M >= 3 ? rank4(0, 0, 0, z) : M == 2 ? rank3(0, 0, y) : rank2(0, x);
            const int c0 = M >= 3 ? last + rank3(0, x, y) : M == 2 ? last + rank2(0, x) : last;
            const int c1 = M >= 3 ? last + rank3(0, 0, y) + x : M == 2 ? last + x : x;
            const int c2 = M >= 3 ? last + rank2(x, y) : rank2(x, y);
            const int c3 = rank3(x, y, z);
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                v[j][c] = make_longlong2(0ll, 0ll);
                ex[j][c] = 0;
                const int a = au[c];
                if (a < n) {
                    int rk = a;
                    if (M == 1) rk = a <= x ? c0 + a : c1 + bin2[c];
                    if (M == 2) rk = a <= x ? c0 + a : a <= y ? c1 + bin2[c] : c2 + bin3[c];
                    if (M == 3) rk = a <= x ? c0 + a : a <= y ? c1 + bin2[c] : a <= z ? c2 + bin3[c] : c3 + bin4[c];
                    v[j][c] = src[rk];
                    if (SRC != 0) ex[j][c] = earow[rk];
                }
            }
        }
#pragma unroll
        for (int j = 0; j < RW; ++j) {
            E[j] = Eall;
            if (SRC == 0) {
                // one unit for all entries: the bit length of the OR of their magnitudes (the lowest
                // bit as it is, so that a minus one counts)
                unsigned long long m = 0ull;
#pragma unroll
                for (int c = 0; c < CH; ++c)
                    m |= (unsigned long long)((v[j][c].x ^ (v[j][c].x >> 63)) | (v[j][c].y ^ (v[j][c].y >> 63)) |
                                              ((v[j][c].x | v[j][c].y) & 1));
                const unsigned hi = __reduce_or_sync(0xffffffffu, (unsigned)(m >> 32));
                const unsigned lo = __reduce_or_sync(0xffffffffu, (unsigned)m);
                E[j] = hi | lo ? (hi ? 64 - __clz((int)hi) : 32 - __clz((int)lo)) + e0 : EXP_NONE;
            } else if (SRC == 1) {
                int key = 0;
#pragma unroll
                for (int c = 0; c < CH; ++c)
                    if (v[j][c].x | v[j][c].y) key = max(key, bitlen(v[j][c]) + ex[j][c] + e0 + 8192);
                key = (int)__reduce_max_sync(0xffffffffu, (unsigned)key);
                E[j] = key ? key - 8192 : EXP_NONE;
            }
            if (RW > 1 && row + j >= nrows) break;
            const int sh = e0 - E[j] + 7 + 8 * (S - 1);
            const uint32_t at = ((uint32_t)(row + j) << lg) + (uint32_t)lane;
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                if (au[c] < kout) {
                    uint32_t w[S];
                    if (E[j] != EXP_NONE) {
                        digit_pairs<S>(shift_full(v[j][c].x, sh + ex[j][c]), shift_full(v[j][c].y, sh + ex[j][c]), w);
                    } else {
#pragma unroll
                        for (int s = 0; s < S; ++s) w[s] = 0u;
                    }
#pragma unroll
                    for (int s = 0; s < S; ++s) dst[s][at + 32 * c] = w[s];
                }
            }
            if (SRC != 2 && lane == 0) oexp[row + j] = E[j];
        }
    }
}

// The divide's slots (RowArgs: smeta, ssum, ssig) of the tuples tup[0, count): eigenvalue sums, run
// lengths and the place in the reduction's operand. They do not depend on the upper index.
static __global__ void k_slot_rows(int N, int count, const uint32_t* __restrict__ tup,
                                   const int* __restrict__ segs, const double2* __restrict__ lam,
                                   int4* __restrict__ meta, float* __restrict__ sum, double2* __restrict__ sig)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= count) return;
    int4 r = make_int4(-1, 0, 1 << 13 | 1 << 16, 0);
    double2 sg = make_double2(0.0, 0.0);
    const uint32_t t = tup[idx];
    if (t != 0xFFFFFFFFu) {
        int d[3];
        const int np = N - 1;
        for (int m = 0; m < 3; ++m) {
            d[m] = (int)((t >> (8 * m)) & 255u);
            if (m < np) sg = cadd(sg, lam[d[m]]);
        }
        int den = 1, run = 1, r1 = 1;
        bool first_run = true;
        for (int m = 1; m <= np; ++m) {
            if (m < np && d[m] == d[m - 1]) { ++run; continue; }
            if (first_run) r1 = run;
            first_run = false;
            for (int u = 2; u <= run; ++u) den *= u;
            run = 1;
        }
        r.x = d[0];
        if (N == 3) r.y = rank2(0, d[0]);
        if (N == 4) r.y = rank3(0, d[0], d[1]);
        r.z = d[np - 1] | segs[idx] << 8 | r1 << 13 | den << 16;
    }
    meta[idx] = r;
    sig[idx] = sg;
    const tfl a = to_tfl(sg.x), b = to_tfl(sg.y);
    sum[idx] = a.a;
    sum[count + idx] = a.b;
    sum[2 * count + idx] = a.c;
    sum[3 * count + idx] = b.a;
    sum[4 * count + idx] = b.b;
    sum[5 * count + idx] = b.c;
}

// W transposed and less the exponent of its column, as double-float complex (Re hi, Re lo, Im hi, Im lo).
static __global__ void k_to_df(int n, const double2* __restrict__ W, const int* __restrict__ we, float4* __restrict__ out)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * n) return;
    const double2 w = times_pow2(W[(t % n) * n + t / n], -we[t / n]);
    const float rh = (float)w.x, ih = (float)w.y;
    out[t] = make_float4(rh, (float)(w.x - rh), ih, (float)(w.y - ih));
}

// =======================================================================================
// Host side
// =======================================================================================
struct SplitOperand {
    int S = 0;
    // fixed matrices: planes [S][512 rows][K'] bf16 and exponents [256]
    __nv_bfloat16* phi = nullptr;   int* phi_e = nullptr;    // Phi, complex K (a), columns p
    __nv_bfloat16* psir = nullptr;  int* psir_e = nullptr;   // Psi, real K (j), columns i
    __nv_bfloat16* red = nullptr;   int* red_e = nullptr;    // Psi^T rows k, complex K (p)
    float4* psi_df = nullptr;
    int* tile_list = nullptr;       // running tiles of the current launch (k_tile_list)
    unsigned* tile_count = nullptr;
    int64_t tile_cap = 0;
    // per order: A^T digit planes (rows Q, K' = j) and row exponents
    __nv_bfloat16* at[kMaxOrder + 1] = {};
    int* at_e[kMaxOrder + 1] = {};
    int64_t at_rows[kMaxOrder + 1] = {};
    // sorted M-tuples of states in colexicographic order, 8 bits per index (M = 0: one empty tuple)
    uint32_t* atup[4] = {};
    int64_t natup[4] = {};
    const double* at_src[kMaxOrder + 1] = {};
    // per order, for the modes in use: the divide's slots (128 a tile) and the tables around them
    int slot_nm[kMaxOrder + 1] = {};          // modes the tables were built for (0: none)
    int slot_tiles[kMaxOrder + 1] = {};
    int4* smeta[kMaxOrder + 1] = {};
    float* ssum[kMaxOrder + 1] = {};
    double2* ssig[kMaxOrder + 1] = {};
    uint32_t* stup[kMaxOrder + 1] = {};
    int* sseg[kMaxOrder + 1] = {};
    int* stpmax[kMaxOrder + 1] = {};
    int* segbase[kMaxOrder + 1] = {};
    // reduction rows of the last term (Plan::keep_red): planes, exponents, their bytes. Workspace of the
    // plan: within the budget, and given back when another call asks for scratch
    uint8_t* kept[kMaxOrder + 1] = {};
    int* kept_e[kMaxOrder + 1] = {};
    size_t kept_bytes[kMaxOrder + 1] = {};
    bool kept_ok[kMaxOrder + 1] = {};
    // sorted M-tuples over the modes in use in colexicographic order, 8 bits per index
    uint32_t* ptup[4] = {};
    int64_t nptup[4] = {};
    int ptup_nm[4] = {};
    int* err = nullptr;
    // reduction weights other than Psi (mode-interaction NPFs): planes of W^T, exponents, W in
    // double-float
    __nv_bfloat16* wred = nullptr;  int* wred_e = nullptr;
    float4* w_df = nullptr;
};

static PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        NPF_CUDA(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                                  cudaEnableDefault, &q));
        if (q != cudaDriverEntryPointSuccess || !p)
            fail(NPF_ERR_CUDA, "cuTensorMapEncodeTiled unavailable");
        fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    return fn;
}

// BF16 tensor map whose boxes are bk = 16 or 32 elements wide, with the matching 32- or 64-byte
// swizzle.
static CUtensorMap encode_map(const void* base, int rank, const cuuint64_t* dims,
                              const cuuint64_t* strides, const cuuint32_t* box, int bk)
{
    CUtensorMap m;
    cuuint32_t es[4] = {1, 1, 1, 1};
    CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(base),
                             dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                             bk == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
                             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS)
        fail(NPF_ERR_CUDA, "cuTensorMapEncodeTiled failed: " + std::to_string((int)r));
    return m;
}

// Operands as the callers describe them: data planes [S][rows][inner] and fixed-matrix planes
// [S][512][inner] (Re rows at 0.., Im rows at 256..), BF16.
struct DataOp { const void* base; int64_t inner, stride, rows; };   // stride: elements between rows
struct FixedOp { const void* base; int64_t inner; };

// Data operand as a 3-D tensor (inner, rows, plane); box {bk, box_rows, planes}. Past the inner
// extent a box holds zeros.
template <int S>
static CUtensorMap plane_map(const DataOp& d, int bk, int box_rows)
{
    const cuuint64_t dims[3] = {(cuuint64_t)d.inner, (cuuint64_t)d.rows, (cuuint64_t)S};
    const cuuint64_t strides[2] = {(cuuint64_t)d.stride * 2, (cuuint64_t)(d.rows * d.stride * 2)};
    const cuuint32_t box[3] = {(cuuint32_t)bk, (cuuint32_t)box_rows, (cuuint32_t)S};
    return encode_map(d.base, 3, dims, strides, box, bk);
}

// Fixed matrix as a 4-D tensor (inner, row within the half, half, plane); box {bk, bnc, 2,
// planes}, so a plane's tile is its bnc Re rows followed by its bnc Im rows.
template <int S>
static CUtensorMap fixed_map(const FixedOp& f, int bnc, int bk)
{
    const cuuint64_t dims[4] = {(cuuint64_t)f.inner, 256, 2, (cuuint64_t)S};
    const cuuint64_t strides[3] = {(cuuint64_t)f.inner * 2, (cuuint64_t)(256 * f.inner * 2),
                                   (cuuint64_t)(512 * f.inner * 2)};
    const cuuint32_t box[4] = {(cuuint32_t)bk, (cuuint32_t)bnc, 2, (cuuint32_t)S};
    return encode_map(f.base, 4, dims, strides, box, bk);
}

static int default_slices(const Plan& p)
{
    // the FP32 form: 4 slices (32 bits); 3 (FP32's 24) measured 2.0e-5 at n = 80, order 4,
    // over its 1e-5 bar, after five rounding stages
    return p.slices ? p.slices : (p.precision == NPF_PREC_FP32 ? 4 : 6);
}

template <class T>
static T* upload(const std::vector<T>& v)
{
    T* d = nullptr;
    NPF_CUDA(cudaMalloc(&d, v.size() * sizeof(T)));
    NPF_CUDA(cudaMemcpy(d, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice));
    return d;
}

// Bytes of the dense rows of one upper index (rad^(N-1) rows in two buffers).
static size_t dense_bytes(int n, int N, int S)
{
    const int rad = n <= 32 ? 32 : n <= 64 ? 64 : 128;
    return 2 * ((size_t)ipow64(rad, N - 1) * ((size_t)rad * 4 * S + 4)) + 4096;
}

static void free_kept(SplitOperand& so, int N)
{
    if (so.kept[N]) cudaFree(so.kept[N]);
    if (so.kept_e[N]) cudaFree(so.kept_e[N]);
    so.kept[N] = nullptr;
    so.kept_e[N] = nullptr;
    so.kept_bytes[N] = 0;
    so.kept_ok[N] = false;
}

#ifndef NPF_SPLIT_LOW
void split_give_back(Plan& p)
{
    for (int N = 0; p.split && N <= kMaxOrder; ++N) free_kept(*p.split, N);
}

void split_drop_kept(Plan& p)
{
    if (!p.split) return;
    for (bool& ok : p.split->kept_ok) ok = false;
}

// A term is accepted when S, digit records of it (32 bytes an entry) and the dense rows of one upper
// index fit the budget. This is what callers rely on, not what a term needs: it forms no records, and
// the sorted rows of an upper index with all tables fit in what is so accepted, at every size and
// slice count (n = 120, order 4 would run in 22 GB of the 65 GB asked for).
size_t split_min_bytes(const Plan& p, int N)
{
    const int64_t P = p.packed_count[N], rows = (P + NP - 1) / NP * NP;
    return (size_t)p.n * rows * sizeof(double2) + (size_t)p.n * P * 32 + dense_bytes(p.n, N, default_slices(p));
}

void split_release(Plan& p)
{
    SplitOperand* so = p.split;
    if (!so) return;
    cudaFree(so->phi); cudaFree(so->phi_e);
    cudaFree(so->psir); cudaFree(so->psir_e);
    cudaFree(so->red); cudaFree(so->red_e);
    cudaFree(so->psi_df);
    cudaFree(so->tile_list);
    cudaFree(so->tile_count);
    for (int N = 0; N <= kMaxOrder; ++N) { cudaFree(so->at[N]); cudaFree(so->at_e[N]); }
    cudaFree(so->wred); cudaFree(so->wred_e); cudaFree(so->w_df);
    for (int N = 0; N <= kMaxOrder; ++N) {
        cudaFree(so->smeta[N]); cudaFree(so->ssum[N]); cudaFree(so->ssig[N]); cudaFree(so->stup[N]); cudaFree(so->sseg[N]);
        cudaFree(so->stpmax[N]); cudaFree(so->segbase[N]);
        free_kept(*so, N);
    }
    for (int M = 0; M < 4; ++M) { cudaFree(so->ptup[M]); cudaFree(so->atup[M]); }
    cudaFree(so->err);
    delete so;
    p.split = nullptr;
}
#endif

template <int S, int MODE, bool SUBB>
static void smem_attr()
{
    NPF_CUDA(cudaFuncSetAttribute(k_rows<S, MODE, SUBB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  RowCfg<S, MODE>::SMEM));
}

template <int S>
static void set_smem_attrs()
{
    static bool done = false;
    if (done) return;
    smem_attr<S, EPI_SLICE, false>();
    smem_attr<S, EPI_SLICE, true>();
    smem_attr<S, EPI_DIVIDE, false>();
    smem_attr<S, EPI_SLAB, false>();
    smem_attr<S, EPI_REDUCE, false>();
    smem_attr<S, EPI_V, false>();
    done = true;
}

// Fixed planes [S][512][kw] of an n x n complex matrix, a block per column c (k: the K index; entry
// m[k][c], or m[c][k] when trans): complex K (kw = 256, interleaved): Re-row c = [Re, -Im, ..], Im-row
// 256 + c = [Im, Re, ..]; real K (kw = 128): Re-row [Re ..], Im-row [Im ..]. Exponent per column.
// Rows and K entries past n keep the zeros of the allocation.
template <int S>
__global__ void __launch_bounds__(128)
    k_fixed_planes(const double2* __restrict__ m, int n, int trans, int complexK,
                   __nv_bfloat16* __restrict__ planes, int* __restrict__ ex)
{
    const int c = blockIdx.x, k = threadIdx.x;   // n <= 128: one K entry a thread
    double2 v = make_double2(0.0, 0.0);
    if (c < n && k < n) v = m[trans ? c * n + k : k * n + c];
    __shared__ double red[128];
    red[k] = fmax(fabs(v.x), fabs(v.y));
    __syncthreads();
    for (int w = 64; w > 0; w >>= 1) {
        if (k < w) red[k] = fmax(red[k], red[k + w]);
        __syncthreads();
    }
    int e = EXP_NONE;
    if (red[0] > 0.0) frexp(red[0], &e);
    if (k == 0) ex[c] = e;
    if (c >= n || k >= n) return;
    long long wr = 0, wi = 0;
    if (e != EXP_NONE) {
        const double sc = pow2d(7 + 8 * (S - 1) - e);
        wr = __double2ll_rn(v.x * sc);
        wi = __double2ll_rn(v.y * sc);
    }
    uint32_t w[S], wn[S];
    digit_pairs<S>(wr, wi, w);        // (Re, Im)
    digit_pairs<S>(wr, -wi, wn);      // (Re, -Im)
    const int kw = complexK ? KP : NP;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        uint16_t* re = reinterpret_cast<uint16_t*>(planes) + ((size_t)s * 512 + c) * kw;
        uint16_t* im = re + (size_t)256 * kw;
        if (complexK) {
            *reinterpret_cast<uint32_t*>(re + 2 * k) = wn[s];
            *reinterpret_cast<uint32_t*>(im + 2 * k) = w[s] >> 16 | w[s] << 16;
        } else {
            re[k] = (uint16_t)w[s];
            im[k] = (uint16_t)(w[s] >> 16);
        }
    }
}

// One fixed matrix (buffers allocated on first use, then overwritten in place), on the plan's stream.
static void fixed_matrix(Plan& p, int S, const double2* m, bool trans, bool complexK, __nv_bfloat16*& planes, int*& ex)
{
    const size_t bytes = (size_t)S * 512 * (complexK ? KP : NP) * sizeof(__nv_bfloat16);
    if (!planes) {
        NPF_CUDA(cudaMalloc(&planes, bytes));
        NPF_CUDA(cudaMemsetAsync(planes, 0, bytes, p.stream));
    }
    if (!ex) NPF_CUDA(cudaMalloc(&ex, 256 * sizeof(int)));
    LaunchScope ls(&p.prof, "split_fixed_planes", p.stream);
    auto kern = S == 2 ? k_fixed_planes<2> : S == 3 ? k_fixed_planes<3> : S == 4 ? k_fixed_planes<4>
              : S == 5 ? k_fixed_planes<5> : k_fixed_planes<6>;
    kern<<<256, 128, 0, p.stream>>>(m, p.n, trans, complexK, planes, ex);
    NPF_CUDA(cudaGetLastError());
}

// The reduction's weights transposed, in double-float (ex: their columns' exponents).
static void to_df(Plan& p, const double2* m, const int* ex, float4*& out)
{
    const int count = p.n * p.n;
    if (!out) NPF_CUDA(cudaMalloc(&out, (size_t)count * sizeof(float4)));
    LaunchScope ls(&p.prof, "split_to_df", p.stream);
    k_to_df<<<(count + 255) / 256, 256, 0, p.stream>>>(p.n, m, ex, out);
    NPF_CUDA(cudaGetLastError());
}

// Slices of Phi, Psi and Psi^T and the double-float Psi, from the plan's modal data.
static void fill_fixed(Plan& p, SplitOperand* so)
{
    const int S = so->S;
    fixed_matrix(p, S, p.d_U, false, true, so->phi, so->phi_e);      // K index a, column p: phi_{a p}
    fixed_matrix(p, S, p.d_V, true, false, so->psir, so->psir_e);    // real K index j, column i: psi_{i j}
    fixed_matrix(p, S, p.d_V, false, true, so->red, so->red_e);      // K index p, column k: psi_{p k}
    to_df(p, p.d_V, so->red_e, so->psi_df);
}

static SplitOperand& prepare(Plan& p)
{
    const int S = default_slices(p);
    if (p.n > NP) fail(NPF_ERR_UNSUPPORTED, "the tensor-core path supports n <= 128");
    if (p.split && p.split->S == S) return *p.split;
    split_release(p);
    SplitOperand* so = new SplitOperand();
    p.split = so;
    so->S = S;
    fill_fixed(p, so);
    NPF_CUDA(cudaMalloc(&so->err, sizeof(int)));
    NPF_CUDA(cudaMemset(so->err, 0, sizeof(int)));
    return *so;
}

// Slices of a reduction-weight matrix W[p][k] (device, n x n) in place of Psi: the fixed matrix
// of the reduction GEMM (rows k, complex K index p), its exponents, and W in double-float.
static void prepare_weights(Plan& p, SplitOperand& so, const double2* dW)
{
    fixed_matrix(p, so.S, dW, false, true, so.wred, so.wred_e);
    to_df(p, dW, so.wred_e, so.w_df);
}

// The slot tables of the order from the plan's eigenvalues.
static void fill_slots(Plan& p, SplitOperand& so, int N)
{
    const int count = so.slot_tiles[N] * NP;
    LaunchScope ls(&p.prof, "split_slot_rows", p.stream);
    k_slot_rows<<<(unsigned)((count + 127) / 128), 128, 0, p.stream>>>(N, count, so.stup[N], so.sseg[N], p.d_lam,
                                                                      so.smeta[N], so.ssum[N], so.ssig[N]);
    NPF_CUDA(cudaGetLastError());
}

#ifndef NPF_SPLIT_LOW
void split_refresh_modes(Plan& p)   // (the caller waits for the stream: a batch's graph runs on others)
{
    if (!p.split) return;
    fill_fixed(p, p.split);   // same n and S: the buffers (and graphs) stay valid
    for (int N = 2; N <= 4; ++N)
        if (p.split->slot_nm[N] == p.nm) fill_slots(p, *p.split, N);
}
#endif

// Sorted M-tuples (M <= 3) over [0, count) in colexicographic order, 8 bits per index.
static std::vector<uint32_t> colex_tuples(int M, int count)
{
    std::vector<uint32_t> t;
    if (M == 0) t.push_back(0u);
    for (int r = 0; r < (M >= 3 ? count : M >= 1 ? 1 : 0); ++r)
        for (int q = 0; q < (M >= 3 ? r + 1 : M == 2 ? count : 1); ++q)
            for (int x = 0; x < (M >= 2 ? q + 1 : count); ++x)
                t.push_back((uint32_t)x | (M >= 2 ? (uint32_t)q << 8 : 0u) | (M >= 3 ? (uint32_t)r << 16 : 0u));
    return t;
}

static void ensure_ptuples(Plan& p, SplitOperand& so, int M)   // over the modes in use
{
    if (so.ptup_nm[M] == p.nm) return;
    cudaFree(so.ptup[M]);
    so.ptup[M] = nullptr;
    so.ptup_nm[M] = 0;
    const std::vector<uint32_t> t = colex_tuples(M, p.nm);
    so.ptup[M] = upload(t);
    so.nptup[M] = (int64_t)t.size();
    so.ptup_nm[M] = p.nm;
}

static void ensure_atuples(Plan& p, SplitOperand& so, int M)   // over the states
{
    if (so.atup[M]) return;
    const std::vector<uint32_t> t = colex_tuples(M, p.n);
    so.atup[M] = upload(t);
    so.natup[M] = (int64_t)t.size();
}

// The slots of order N: the sorted tuples (p_2 <= .. <= p_N) in 128-row tiles. A segment (the
// tuples that share p_2 .. p_{N-1}) fills one row of the reduction's operand per p_1, whose
// exponent it shares, so it never straddles two tiles. A tile runs the columns p_1 <= its largest
// p_2, so it takes segments of nearby p_2 only (within 8), the longest first.
static void ensure_slots(Plan& p, SplitOperand& so, int N)
{
    if (so.slot_nm[N] == p.nm) return;
    cudaFree(so.smeta[N]); cudaFree(so.ssum[N]); cudaFree(so.ssig[N]); cudaFree(so.stup[N]); cudaFree(so.sseg[N]); cudaFree(so.stpmax[N]);
    cudaFree(so.segbase[N]);
    so.smeta[N] = nullptr; so.ssum[N] = nullptr; so.ssig[N] = nullptr; so.stup[N] = nullptr; so.sseg[N] = nullptr; so.stpmax[N] = nullptr;
    so.segbase[N] = nullptr;
    so.slot_nm[N] = 0;
    const int nm = p.nm;
    struct Seg { int p2, p3, len; };         // p3: the last shared p (p_{N-1})
    std::vector<Seg> segs;
    if (N == 2) segs.push_back({nm - 1, 0, nm});
    for (int p2 = 0; N >= 3 && p2 < nm; ++p2)
        for (int p3 = p2; p3 < (N == 3 ? p2 + 1 : nm); ++p3) segs.push_back({p2, p3, nm - p3});
    struct Bin { int p2, used; std::vector<int> seg; };
    std::vector<Bin> bins;
    size_t open = 0;                         // bins before it are full or of far smaller p_2
    for (int g = 0; g < (int)segs.size(); ++g) {
        while (open < bins.size() && (bins[open].p2 + 8 < segs[g].p2 || bins[open].used == NP)) ++open;
        size_t b = open;
        while (b < bins.size() && (bins[b].p2 + 8 < segs[g].p2 || bins[b].used + segs[g].len > NP ||
                                   (int)bins[b].seg.size() >= SEGS)) ++b;
        if (b == bins.size()) bins.push_back({segs[g].p2, 0, {}});
        bins[b].seg.push_back(g);
        bins[b].used += segs[g].len;
    }
    std::vector<uint32_t> tup(bins.size() * NP, 0xFFFFFFFFu);
    std::vector<int> seg(bins.size() * NP, 0), tpmax(bins.size(), 0);
    std::vector<int> base(N == 4 ? nm * (nm + 1) / 2 : N == 3 ? nm : 1, 0);
    for (size_t b = 0; b < bins.size(); ++b) {
        int pos = (int)b * NP;
        for (int k = 0; k < (int)bins[b].seg.size(); ++k) {
            const Seg& x = segs[bins[b].seg[k]];
            tpmax[b] = std::max(tpmax[b], x.p2);
            base[N == 4 ? x.p3 * (x.p3 + 1) / 2 + x.p2 : N == 3 ? x.p2 : 0] = pos;
            for (int r = 0; r < x.len; ++r, ++pos) {
                const uint32_t pn = (uint32_t)(N == 2 ? r : x.p3 + r);
                tup[pos] = N == 2 ? pn : N == 3 ? (uint32_t)x.p2 | pn << 8
                                                : (uint32_t)x.p2 | (uint32_t)x.p3 << 8 | pn << 16;
                seg[pos] = k | (r == 0 ? 16 : 0);
            }
        }
    }
    so.slot_tiles[N] = (int)bins.size();
    so.stup[N] = upload(tup);
    so.sseg[N] = upload(seg);
    so.stpmax[N] = upload(tpmax);
    so.segbase[N] = upload(base);
    NPF_CUDA(cudaMalloc(&so.smeta[N], tup.size() * sizeof(int4)));
    NPF_CUDA(cudaMalloc(&so.ssum[N], tup.size() * 6 * sizeof(float)));
    NPF_CUDA(cudaMalloc(&so.ssig[N], tup.size() * sizeof(double2)));
    so.slot_nm[N] = nm;
    fill_slots(p, so, N);
}

// A^T digit planes of the packed tensor (part of the tensor upload; redone when the tensor or the
// slice count changes).
template <int S>
static void prepare_tensor(Plan& p, SplitOperand& so, int N)
{
    if (so.at[N] && so.at_src[N] == p.d_tensor[N]) return;
    const int64_t P = p.packed_count[N];
    const int64_t rows = (P + NP - 1) / NP * NP;
    if (!so.at[N] || so.at_rows[N] != rows) {   // same shape: keep the buffers (graphs hold them)
        cudaFree(so.at[N]);
        cudaFree(so.at_e[N]);
        so.at[N] = nullptr;
        so.at_e[N] = nullptr;
        NPF_CUDA(cudaMalloc(&so.at[N], (size_t)S * rows * NP * 2));
        NPF_CUDA(cudaMalloc(&so.at_e[N], (size_t)rows * sizeof(int)));
    }
    if (rows > P)   // the padding rows of every plane (k_prep_at writes the others whole)
        NPF_CUDA(cudaMemset2DAsync(so.at[N] + P * NP, (size_t)rows * NP * 2, 0, (size_t)(rows - P) * NP * 2, S, p.stream));
    {
        LaunchScope ls(&p.prof, "split_prepare_tensor", p.stream);
        k_prep_at<S><<<(unsigned)((P + 7) / 8), 256, 0, p.stream>>>(p.d_tensor[N], P, p.n, N, p.d_cnt, so.at[N],
                                                                    rows * NP, so.at_e[N]);
        NPF_CUDA(cudaGetLastError());
    }
    so.at_rows[N] = rows;
    so.at_src[N] = p.d_tensor[N];
}

#ifndef NPF_SPLIT_LOW
void split_forget_tensor(Plan& p, int N)
{
    if (p.split) p.split->at_src[N] = nullptr;
}

const void* split_tensor_planes(const Plan& p, int N)
{
    return p.split ? p.split->at[N] : nullptr;
}

void split_prepare_tensor(Plan& p, int N)
{
    if (p.precision == NPF_PREC_FP64 || N > 4 || p.n > NP) return;
    SplitOperand& so = prepare(p);
    so.at_src[N] = nullptr;   // the tensor's contents changed: always redo
    switch (so.S) {
    case 2: prepare_tensor<2>(p, so, N); break;
    case 3: prepare_tensor<3>(p, so, N); break;
    case 4: prepare_tensor<4>(p, so, N); break;
    case 5: prepare_tensor<5>(p, so, N); break;
    case 6: prepare_tensor<6>(p, so, N); break;
    default: break;
    }
}
#endif

// Tracing aid: with NPF_TRACE_TILES set in the environment every k_rows launch records per-CTA
// phase times (%globaltimer) and prints the median phase durations to stderr.
static void trace_report(const char* name, const std::vector<unsigned long long>& t, int64_t tiles)
{
    std::vector<double> d[5];
    unsigned long long t0 = ~0ull, t1 = 0;
    int64_t ran = 0;
    std::map<unsigned long long, std::vector<std::pair<unsigned long long, unsigned long long>>> cta;
    for (int64_t k = 0; k < tiles; ++k) {
        const unsigned long long* r = &t[k * 6];
        if (!r[0] || !r[3]) continue;
        ++ran;
        t0 = std::min(t0, r[0]);
        t1 = std::max(t1, r[3]);
        d[0].push_back((double)(r[1] - r[0]));                   // epilogue waiting for the MMA
        d[1].push_back(r[2] ? (double)(r[2] - r[1]) : 0.0);      // column-exponent pass
        d[2].push_back((double)(r[3] - (r[2] ? r[2] : r[1])));   // output pass
        cta[r[4]].push_back({r[0], r[3]});
        if (r[5]) d[4].push_back((double)r[5]);                 // the tile's set-up (beside other tiles)
    }
    // between a CTA's tiles: skipped tiles, the per-tile tables and the error-flag read
    double busy = 0.0;
    for (auto& kv : cta) {
        auto& v = kv.second;
        std::sort(v.begin(), v.end());
        for (size_t j = 0; j + 1 < v.size(); ++j) d[3].push_back((double)(v[j + 1].first - v[j].second));
        if (!v.empty()) busy = std::max(busy, (double)(v.back().second - v.front().first));
    }
    auto med = [](std::vector<double>& v) {
        if (v.empty()) return 0.0;
        std::nth_element(v.begin(), v.begin() + v.size() / 2, v.end());
        return v[v.size() / 2] * 1e-3;
    };
    auto mean = [](const std::vector<double>& v) {
        double a = 0.0;
        for (double x : v) a += x;
        return v.empty() ? 0.0 : a / v.size() * 1e-3;
    };
    fprintf(stderr, "[trace] %s tiles %lld ran %lld span %.1f us (longest CTA %.1f) | median/mean "
            "us: wait-mma %.2f/%.2f pass1 %.2f/%.2f pass2 %.2f/%.2f between %.2f/%.2f (set-up "
            "%.2f/%.2f)\n", name,
            (long long)tiles, (long long)ran, (t1 > t0 ? (t1 - t0) : 0) * 1e-3, busy * 1e-3,
            med(d[0]), mean(d[0]), med(d[1]), mean(d[1]), med(d[2]), mean(d[2]), med(d[3]),
            mean(d[3]), med(d[4]), mean(d[4]));
}

static int sm_count()
{
    static int count = 0;
    if (!count) {
        int dev = 0;
        NPF_CUDA(cudaGetDevice(&dev));
        NPF_CUDA(cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev));
    }
    return count;
}

template <int S, int MODE>
// kprime: K' length of the contraction (2 n for complex K, n for real K)
static void launch_rows(Plan& p, const char* name, const DataOp& A, const FixedOp& B, int kprime,
                        RowArgs a)
{
    constexpr int bk = RowCfg<S, MODE>::BK;
    a.kch = (kprime + bk - 1) / bk;            // K' past kprime holds zeros on both sides
    a.lgncol = (a.ncol_tiles & (a.ncol_tiles - 1)) == 0 ? __builtin_ctz((unsigned)a.ncol_tiles) : -1;
    a.klast = (kprime + KSTEP - 1) / KSTEP - (bk / KSTEP) * (a.kch - 1);
    a.arows = MODE == EPI_SLICE && a.lg == 7 ? std::min(NP, (a.n + 7) / 8 * 8) : NP;
    const CUtensorMap tA = plane_map<S>(A, bk, a.arows);
    const CUtensorMap tB = fixed_map<S>(B, a.bnc, bk);
    if (a.num_tiles >= (int64_t)1 << 31) fail(NPF_ERR_UNSUPPORTED, "too many tiles in one launch");
    if (a.colmask && a.num_tiles > 8 * sm_count()) {
        // the running tiles, listed on the device (stream order puts the list before the launch).
        // Without a column mask, or with a few tiles a CTA only (where the list's two launches cost
        // more than the MMAs of the masked tiles: 6 us against 2 to 4), every tile runs
        SplitOperand& so = *p.split;
        if (!so.tile_list || so.tile_cap < a.num_tiles) {
            if (p.capturing) fail(NPF_ERR_CUDA, "tile list would grow during graph capture");
            NPF_CUDA(cudaStreamSynchronize(p.stream));
            cudaFree(so.tile_list);
            cudaFree(so.tile_count);
            so.tile_list = nullptr;
            so.tile_count = nullptr;
            NPF_CUDA(cudaMalloc(&so.tile_list, (size_t)a.num_tiles * sizeof(int)));
            NPF_CUDA(cudaMalloc(&so.tile_count, sizeof(unsigned)));
            so.tile_cap = a.num_tiles;
        }
        NPF_CUDA(cudaMemsetAsync(so.tile_count, 0, sizeof(unsigned), p.stream));
        LaunchScope ls(&p.prof, "split_tile_list", p.stream);
        launch_dependent(k_tile_list, dim3((unsigned)((a.num_tiles + 255) / 256)), dim3(256), 0, p.stream, a, a.lg,
                         so.tile_list, so.tile_count);
        a.tiles = so.tile_list;
        a.ntiles_run = so.tile_count;
    }
    static const bool tracing = getenv("NPF_TRACE_TILES") != nullptr;
    unsigned long long* dtrace = nullptr;
    if (tracing) {
        NPF_CUDA(cudaMalloc(&dtrace, (size_t)a.num_tiles * 6 * 8));
        NPF_CUDA(cudaMemsetAsync(dtrace, 0, (size_t)a.num_tiles * 6 * 8, p.stream));
        a.trace = dtrace;
    }
    {
        LaunchScope ls(&p.prof, name, p.stream);
        // persistent: one CTA per SM (the shared memory allows one), tiles strided over CTAs;
        // an odd stride keeps each CTA from seeing only one column tile (the column tiles of a
        // row tile differ in cost under the sorted-tuple masks)
        int64_t grid = std::min<int64_t>(a.num_tiles, sm_count());
        if (MODE == EPI_REDUCE)   // whole groups of a block per column tile
            grid = std::max<int64_t>(1, std::min<int64_t>(a.num_tiles, sm_count()) / a.ncol_tiles) * a.ncol_tiles;
        else if (grid < a.num_tiles && a.ncol_tiles > 1 && grid % 2 == 0) grid -= 1;
        const dim3 g((unsigned)std::max<int64_t>(grid, 1)), b(ROW_THREADS);
        constexpr size_t smem = RowCfg<S, MODE>::SMEM;
        if constexpr (MODE == EPI_SLICE) {
            if (a.lg < 7) launch_dependent(k_rows<S, MODE, true>, g, b, smem, p.stream, tA, tB, a);
            else launch_dependent(k_rows<S, MODE, false>, g, b, smem, p.stream, tA, tB, a);
        } else {
            launch_dependent(k_rows<S, MODE, false>, g, b, smem, p.stream, tA, tB, a);
        }
    }
    if (tracing) {
        std::vector<unsigned long long> h((size_t)a.num_tiles * 6);
        NPF_CUDA(cudaMemcpyAsync(h.data(), dtrace, h.size() * 8, cudaMemcpyDeviceToHost, p.stream));
        NPF_CUDA(cudaStreamSynchronize(p.stream));
        cudaFree(dtrace);
        trace_report(name, h, a.num_tiles);
    }
}

static double factorial(int N) { double f = 1; for (int t = 2; t <= N; ++t) f *= t; return f; }

// The regather's variant: 32-entry chunks of a row (CH), and the rows that a warp takes at a time (RW),
// so that three to six gathers are in flight (twice the rows: n = 60, order 4, 4.88 ms against
// 4.51, n = 120, order 3, 1.20 against 1.10; one row less was slower too).
static constexpr int regather_rows(int ch) { return ch == 1 ? 4 : ch <= 3 ? 2 : 1; }
template <int S, int M, int SRC>
static decltype(&k_regather<S, M, SRC, 4, regather_rows(4)>) regather_kernel(int n)
{
    return n <= 32   ? k_regather<S, M, SRC, 1, regather_rows(1)>
           : n <= 64 ? k_regather<S, M, SRC, 2, regather_rows(2)>
           : n <= 96 ? k_regather<S, M, SRC, 3, regather_rows(3)>
                     : k_regather<S, M, SRC, 4, regather_rows(4)>;
}

// Blocks that share one outer index of a regather: about eight rounds a warp, more blocks when few.
static unsigned regather_parts(int64_t outers, int nrows, int n)
{
    const int rows = 8 * regather_rows((n + 31) / 32);           // a round's
    const int64_t all = (nrows + rows - 1) / rows;               // one round a warp
    const int64_t want = std::max<int64_t>((all + 7) / 8, (8 * sm_count() + outers - 1) / std::max<int64_t>(outers, 1));
    return (unsigned)std::max<int64_t>(1, std::min(all, want));
}

// Device memory of one order: V of S (16 bytes, n x P) and per upper index of a batch two buffers
// that the stages alternate (A: the operands of the mode products and of the reduction, B: V and the
// divide's slots) plus the row exponents.
template <int S>
static void split_run(Plan& p, int N, double2* d_out, const int* prefix, const double2* W, bool accumulate)
{
    SplitOperand& so = prepare(p);
    if (W) prepare_weights(p, so, W);
    set_smem_attrs<S>();
    prepare_tensor<S>(p, so, N);
    const bool slab = prefix != nullptr;
    for (int M = N >= 4 ? 2 : std::max(N - 1, 0); M <= N - 1; ++M) ensure_atuples(p, so, M);
    if (N >= 2) ensure_slots(p, so, N);
    if (N >= 2 && !slab) ensure_ptuples(p, so, N - 1);
    if (N >= 3) ensure_ptuples(p, so, 2);
    int* const err = p.err_override ? p.err_override : so.err;   // a batch zeroes and checks its own
    const int n = p.n;
    const int nm = p.nm;                 // modes in use (a critical-mode subset comes first)
    const int64_t Prows = so.at_rows[N];
    // K extent of an operand row: the radix 2^lg >= n
    const int lg = n <= 32 ? 5 : n <= 64 ? 6 : 7;
    const int rad = 1 << lg;
    // complex columns per tile: two accumulator sets of 32 fill TMEM, so the wider settings run 32 too
    const int bnc = p.tile_n == 16 ? 16 : 32;

    // ---- rows per upper index of every stage
    const int64_t npairs = (int64_t)nm * (nm + 1) / 2;
    auto arows = [&](int M) { return M <= 0 ? (int64_t)1 : packed_count(n, M); };   // sorted M-tuples of a's
    const int64_t nt = N <= 2 ? 1 : N == 3 ? nm : npairs;         // sorted (N-2)-tuples of p's
    const int64_t R0 = N == 1 ? 1 : N == 2 ? rad : arows(N - 1);  // first product
    const int64_t R1 = N == 4 ? nm * arows(2) : 0;                // second product (order 4)
    const int64_t R2 = N >= 3 ? nt * rad : 0;                     // last mode product
    const int64_t RS = N == 2 ? rad : N >= 3 ? (int64_t)so.slot_tiles[N] * NP : 0;   // divide
    const int64_t Qc = N >= 2 ? packed_count(nm, N - 1) : 0;      // reduction
    const int64_t v_per = N == 4 ? std::max(nm * arows(3), npairs * arows(2)) : N == 3 ? nm * arows(2) : 0;

    // ---- memory plan (Algorithm 1's rule on the upper-index space)
    const size_t row_bytes = (size_t)rad * 4 * S;
    const size_t s_bytes = (size_t)n * Prows * sizeof(double2);
    const size_t a_per = (size_t)std::max(std::max(R0, R1), std::max(R2, Qc)) * row_bytes;
    const size_t b_per = std::max((size_t)v_per * sizeof(longlong2), (size_t)RS * row_bytes);
    const size_t e_per = (size_t)(R1 + R2 + RS + Qc) * sizeof(int);
    const size_t per_i = a_per + b_per + e_per;
    const int64_t Q2 = N >= 3 && !slab ? npairs : 0;              // weights of the pairs (less than records)
    const size_t wbytes = (size_t)Q2 * n * sizeof(float4);
    const int rlo = std::max(0, p.row_lo);                       // upper-index rows to form
    const int rhi = p.row_hi < 0 ? nm : std::min(p.row_hi, nm);
    // One batch of a small system: the reduction's rows get a buffer of their own, so that the first
    // launch can clear their heads (87 us a term against 90 at n = 60, order 2, 218 against 220 at n = 20,
    // order 4; above 64 MB it is less than 1%: 568 against 575 at n = 60, order 3).
    const size_t red_bytes = (size_t)nm * Qc * row_bytes;
    const size_t fixed_bytes = s_bytes + wbytes + 10 * 256 + 1024;   // (and alignment, sE)
    const size_t all_bytes = fixed_bytes + (size_t)nm * per_i;
    Arena& ar = p.scratch();
    bool own_red = !slab && red_bytes <= ((size_t)64 << 20);
    // (under a budget of the caller's nothing is kept beside the scratch)
    bool keep = !slab && p.keep_red && !p.mem_budget && rhi - rlo == nm && red_bytes <= ((size_t)256 << 20);
    int ib = nm;
    // (scratch that holds everything already needs no look at the free memory)
    if (p.mem_budget || ar.cap < all_bytes + (own_red ? red_bytes : 0)) {
        // (a call that records may not free: its first, eager pass has done so)
        size_t held = 0;
        for (int M = 0; M <= kMaxOrder; ++M) {
            if (!p.keep_red && !p.capturing) free_kept(so, M);
            held += so.kept_bytes[M];
        }
        size_t budget = effective_budget(p);
        if (!p.mem_budget) budget -= std::min(budget, held / 5);   // (80% of free, scratch and kept, less kept)
        if (split_min_bytes(p, N) > budget)
            fail(NPF_ERR_OOM, "memory budget too small for one upper-index batch");
        ib = (int)std::min<size_t>((size_t)nm, (budget - fixed_bytes) / per_i);
        own_red &= ib == nm && all_bytes + red_bytes <= budget;
        keep &= ib == nm && all_bytes + red_bytes <= budget;
    }
    // kept rows, in a buffer of the plan that a repeated interaction finds again: an interaction of n = 60,
    // orders 2 and 3, takes 802 us with them and 1309 without, and gains as much at every size (8.5 -> 4.9
    // ms at n = 100, where they take 1.5 GB); 256 MB an order bounds the memory
    if (keep) {
        const size_t eb = ((size_t)nm * Qc + nm) * sizeof(int);   // the rows' exponents and S's
        if (so.kept_bytes[N] != red_bytes + eb) {
            if (so.kept[N]) NPF_CUDA(cudaStreamSynchronize(p.stream));
            free_kept(so, N);
            if (cudaMalloc(&so.kept[N], red_bytes) != cudaSuccess || cudaMalloc(&so.kept_e[N], eb) != cudaSuccess) {
                cudaGetLastError();   // no room: the rows are formed again for every weight matrix
                free_kept(so, N);
                keep = false;
            } else {
                so.kept_bytes[N] = red_bytes + eb;
            }
        }
        if (keep) own_red = false;   // (no room in the scratch for it)
    }
    const bool again = keep && W && so.kept_ok[N];   // only the reduction is left to do
    ar.reserve(fixed_bytes + (size_t)ib * per_i + (own_red ? red_bytes : 0), p.stream);
    uint8_t* base = (uint8_t*)ar.base;
    auto take = [&](size_t bytes) { uint8_t* r = base; base += (bytes + 255) & ~(size_t)255; return r; };
    longlong2* Sv = (longlong2*)take(s_bytes);
    int* sE = keep ? so.kept_e[N] + (size_t)nm * Qc : (int*)take(256 * sizeof(int));
    uint8_t* bufA = take((size_t)ib * a_per);
    uint8_t* bufB = take((size_t)ib * b_per);
    uint8_t* bufR = keep ? so.kept[N] : own_red ? take(red_bytes) : bufA;   // reduction rows
    int* E1 = (int*)take((size_t)ib * R1 * sizeof(int));
    int* E2 = (int*)take((size_t)ib * R2 * sizeof(int));
    int* ES = (int*)take((size_t)ib * RS * sizeof(int));
    int* ER = keep ? so.kept_e[N] : (int*)take((size_t)ib * Qc * sizeof(int));
    float4* wpre = (float4*)take(wbytes);
    constexpr int kred = RowCfg<S, EPI_REDUCE>::BK / 2;          // complex K entries of a reduction chunk
    {
        // (a slab entry whose accumulator is exactly zero is not stored, so the slab starts at zero)
        LaunchScope ls(&p.prof, "split_term_init", p.stream);
        TermInit a{};
        a.out = d_out;
        a.cells = accumulate ? 0 : (int64_t)n * n;
        a.sE = again ? nullptr : sE;
        a.n = n;
        a.nm = nm;
        a.err = p.err_override || (p.defer_err && p.err_live) ? nullptr : err;
        a.W = W ? W : p.d_V;
        a.we = W ? so.wred_e : so.red_e;
        a.pairs = so.ptup[2];
        a.npairs = Q2;
        a.wpre = wpre;
        a.heads = own_red || (keep && !again) ? Qc * (rhi - rlo) * 8 : 0;
        a.N = N;
        a.kc = kred;
        a.lg = lg;
        a.Q = (int)Qc;
        a.tuples = N >= 2 ? so.ptup[N - 1] : nullptr;
        a.planes = (uint32_t*)bufR;
        a.plane_stride_u32 = (int64_t)(rhi - rlo) * Qc * rad;
        const int64_t work = std::max(std::max<int64_t>((int64_t)n * n, Q2 * n), a.heads);
        launch_dependent(k_term_init<S>, dim3((unsigned)std::min<int64_t>((work + 255) / 256, 4096)), dim3(256), 0,
                         p.stream, a);
    }
    p.err_live = true;

    const FixedOp tPhi{so.phi, KP};
    const FixedOp tPsiR{so.psir, NP};
    const FixedOp tRed{W ? so.wred : so.red, KP};
    const DataOp tAT{so.at[N], NP, NP, Prows};

    RowArgs base0{};
    base0.n = n;
    base0.nm = nm;
    base0.ncv = nm;
    base0.N = N;
    base0.psi_df = W ? so.w_df : so.psi_df;
    base0.lam = p.d_lam;
    base0.invfact = 1.0 / factorial(N);
    base0.eps = p.eps;
    base0.divide = p.divide;
    base0.fp64_quotient = p.fp64_quotient;
    base0.stall = p.debug_stall;
    base0.eps2f = (float)(p.eps * p.eps);
    base0.err = err;
    base0.bnc = bnc;
    base0.ncol_tiles = (nm + bnc - 1) / bnc;
    base0.lg = 7;
    base0.segbase = N >= 2 ? so.segbase[N] : nullptr;
    base0.ttup = N == 4 ? so.ptup[2] : nullptr;
    if (slab)
        for (int m = 0; m < N - 1; ++m) base0.pre[m] = prefix[m];

    // ---- P1: V of S[i][Q] = sum_j psi_ij A^j_Q (rows Q, real K = j), and its exponent per i
    if (!again) {
        RowArgs a = base0;
        a.ea = so.at_e[N];
        a.eb = so.psir_e;
        a.R = Prows;
        a.RB = (int)(Prows / NP);
        a.num_tiles = Prows / NP * a.ncol_tiles;
        a.out_v = Sv;
        a.emax = sE;
        launch_rows<S, EPI_V>(p, "split_upper_contraction", tAT, tPsiR, n, a);   // K = j < n
    }

    // K entries written per row: whole 32-byte sectors, which the MMAs' last K step covers
    const int kout = std::min(rad, (n + 7) / 8 * 8);

    for (int i0 = rlo; i0 < rhi; i0 += ib) {
        const int cur = std::min(ib, rhi - i0);
        auto operand = [&](const uint8_t* buf, int64_t R) { return DataOp{buf, 2 * kout, 2 * rad, cur * R}; };
        auto plane = [&](int64_t R) { return cur * R * rad; };   // plane stride in complex entries
        if (!again) {
            LaunchScope ls(&p.prof, "split_expand", p.stream);
            auto kern = N == 1 ? regather_kernel<S, 0, 2>(n) : N == 2 ? regather_kernel<S, 1, 2>(n)
                      : N == 3 ? regather_kernel<S, 2, 2>(n) : regather_kernel<S, 3, 2>(n);
            const int nrows = (int)so.natup[N - 1];
            const unsigned parts = regather_parts(cur, nrows, n);
            launch_dependent(kern, dim3((unsigned)cur * parts), dim3(256), 0, p.stream, Sv + (int64_t)i0 * Prows, Prows,
                             n, nm, 1, nullptr, so.at_e[N], so.psir_e + i0, sE + i0, lg, kout, nrows, R0, parts,
                             so.atup[N - 1], (uint32_t*)bufA, plane(R0), nullptr);
        }
        // ---- the first N - 2 mode products: V per sorted tuple, regathered into the next operand
        for (int c = 1; c <= N - 2 && !again; ++c) {
            const int64_t Ra = arows(N - c), outers = c == 1 ? cur : (int64_t)cur * nm;
            RowArgs a = base0;
            a.ea = c == 1 ? sE + i0 : E1;
            a.ea_outer = c == 1;
            a.eb = so.phi_e;
            a.colmask = c >= 2;                                  // new index p_3 <= p_4
            a.R = Ra;
            a.RB = (int)((Ra + NP - 1) / NP);
            a.num_tiles = outers * a.RB * a.ncol_tiles;
            a.out_v = (longlong2*)bufB;
            launch_rows<S, EPI_V>(p, "split_mode_product", operand(bufA, outers / cur * Ra), tPhi, 2 * n, a);
            const bool pairs = N - c - 1 == 2;                   // rows of the next operand: pairs of a's, or a_1
            const int64_t outs = c == 1 ? (int64_t)cur * nm : cur * npairs;
            const int nrows = pairs ? (int)so.natup[2] : n;
            const int64_t Rdst = pairs ? nrows : rad;
            LaunchScope ls(&p.prof, "split_regather", p.stream);
            const unsigned parts = regather_parts(outs, nrows, n);
            auto kern = pairs ? regather_kernel<S, 2, 0>(n) : c == 1 ? regather_kernel<S, 1, 0>(n) : regather_kernel<S, 1, 1>(n);
            launch_dependent(kern, dim3((unsigned)outs * parts), dim3(256), 0, p.stream, (const longlong2*)bufB, Ra, n,
                             nm, (int)(outs / cur), base0.ttup, c == 1 ? sE + i0 : E1, so.phi_e, nullptr, lg, kout,
                             nrows, Rdst, parts, so.atup[2], (uint32_t*)bufA, outs * Rdst * rad, pairs ? E1 : E2);
        }
        // ---- the last mode product (its output rows are the divide's slots)
        if (N >= 2 && !again) {
            RowArgs a = base0;
            a.lg = lg;
            a.ea = N == 2 ? sE + i0 : E2;
            a.ea_outer = N == 2;
            a.eb = so.phi_e;
            a.colmask = N >= 3;                                  // p_2 <= p_3
            a.nt = (int)nt;
            a.R = nt * rad;
            a.RB = (int)((a.R + NP - 1) / NP);
            a.num_tiles = (int64_t)cur * a.RB * a.ncol_tiles;
            a.RS = RS;
            a.kout = kout;
            a.out_planes = (__nv_bfloat16*)bufB;
            a.out_plane_stride = 2 * plane(RS);
            a.out_exp = ES;
            launch_rows<S, EPI_SLICE>(p, "split_mode_product", operand(bufA, a.R), tPhi, 2 * n, a);
        }
        // ---- the heads of the reduction rows (bufA is free: the last mode product has read it)
        if (!own_red && !keep && !slab) {
            LaunchScope ls(&p.prof, "split_zero_heads", p.stream);
            launch_dependent(k_zero_heads<S>, dim3((unsigned)((Qc * cur * 8 + 255) / 256)), dim3(256), 0, p.stream, N, nm,
                             kred, lg, (int)Qc, cur, so.ptup[N - 1], (uint32_t*)bufR, plane(Qc));
        }
        // ---- the last contraction: divide, or the slab's entries
        if (!again) {
            RowArgs a = base0;
            a.eb = so.phi_e;
            a.i0 = i0;
            a.nouter = cur;
            if (N >= 2) {
                a.ea = ES;
                a.R = RS;
                a.RB = so.slot_tiles[N];
                a.num_tiles = (int64_t)cur * a.RB * a.ncol_tiles;
                a.smeta = so.smeta[N];
                a.ssum = so.ssum[N];
                a.ssig = so.ssig[N];
                a.nslot = so.slot_tiles[N] * NP;
                a.stup = so.stup[N];
            } else {                                             // order 1: a row per upper index
                a.ea = sE + i0;
                a.R = 1;
                a.num_tiles = (int64_t)((cur + NP - 1) / NP) * a.ncol_tiles;
            }
            const DataOp op = N >= 2 ? operand(bufB, RS) : operand(bufA, 1);
            if (slab) {
                a.out_f64 = d_out;
                launch_rows<S, EPI_SLAB>(p, "split_mode_divide", op, tPhi, 2 * n, a);
                continue;
            }
            a.colmask = 1;
            a.tpmax = so.stpmax[N];
            a.RT = Qc;
            a.lgout = lg;
            a.out_planes = (__nv_bfloat16*)bufR;
            a.out_plane_stride = 2 * plane(Qc);
            a.out_exp = ER;
            launch_rows<S, EPI_DIVIDE>(p, "split_mode_divide", op, tPhi, 2 * n, a);
        }
        // ---- reduction: rows (i, p_1 <= .. <= p_{N-1}), K = p_N, columns k (Psi^T)
        RowArgs a = base0;
        a.ncv = n;                         // columns: states k
        a.ncol_tiles = (n + bnc - 1) / bnc;
        a.kfrom = 1;                       // K = p_N >= the tile's smallest p_{N-1}
        a.ea = ER;
        a.eb = W ? so.wred_e : so.red_e;
        a.ev = so.red_e;
        a.es = sE;
        a.R = Qc;
        a.RB = (int)((Qc + NP - 1) / NP);
        a.num_tiles = (int64_t)cur * a.RB * a.ncol_tiles;
        a.tuples = so.ptup[N - 1];
        a.wpre = wpre;
        a.ldw = Q2;
        a.i0 = i0;
        a.out_f64 = d_out;
        const DataOp red{bufR, 2 * std::min(rad, (nm + 7) / 8 * 8), 2 * rad, cur * Qc};   // K = p_N < nm
        launch_rows<S, EPI_REDUCE>(p, "split_reduce", red, tRed, 2 * nm, a);
        so.kept_ok[N] = keep;
    }
    if (p.err_override || p.defer_err) return;   // the batch, or the entry point, reads the flag at its end
    split_check(p);
}

#ifndef NPF_SPLIT_LOW
void split_check(Plan& p)
{
    if (!p.err_live || !p.split) return;
    p.err_live = false;
    int herr = 0;
    NPF_CUDA(cudaMemcpyAsync(&herr, p.split->err, sizeof(int), cudaMemcpyDeviceToHost, p.stream));
    NPF_CUDA(cudaStreamSynchronize(p.stream));
    if (herr) fail(NPF_ERR_TIMEOUT, "a tensor-core pipeline wait gave up");
}
#endif

// The 2..5-slice runs live in a second translation unit (k_split_low.cu, these sources compiled
// with NPF_SPLIT_LOW), so that the kernel instantiations of the two halves build in parallel.
void split_run_low(Plan& p, int S, int N, double2* d_out, const int* prefix, const double2* W, bool accumulate);

#ifdef NPF_SPLIT_LOW
void split_run_low(Plan& p, int S, int N, double2* d_out, const int* prefix, const double2* W, bool accumulate)
{
    switch (S) {
    case 2: split_run<2>(p, N, d_out, prefix, W, accumulate); break;
    case 3: split_run<3>(p, N, d_out, prefix, W, accumulate); break;
    case 4: split_run<4>(p, N, d_out, prefix, W, accumulate); break;
    case 5: split_run<5>(p, N, d_out, prefix, W, accumulate); break;
    default: fail(NPF_ERR_UNSUPPORTED, "slices must be in [2, 6] on the tensor-core path");
    }
}
#else
static void split_any(Plan& p, int N, double2* d_out, const int* prefix, const double2* W, bool accumulate)
{
    if (N < 1 || (N == 1 && !prefix)) fail(NPF_ERR_ARG, "order must be >= 2 (order 1: modal slabs only)");
    if (N > 4) fail(NPF_ERR_UNSUPPORTED, "the tensor-core path supports orders <= 4 (use NPF_PREC_FP64)");
    const int S = default_slices(p);
    if (S == 6) split_run<6>(p, N, d_out, prefix, W, accumulate);
    else if (S >= 2 && S <= 5) split_run_low(p, S, N, d_out, prefix, W, accumulate);
    else fail(NPF_ERR_UNSUPPORTED, "slices must be in [2, 6] on the tensor-core path");
}

void split_term(Plan& p, int N, double2* d_out, const double2* W, bool accumulate)
{
    split_any(p, N, d_out, nullptr, W, accumulate);
}
void split_slab(Plan& p, int N, const int* prefix, double2* d_out)
{
    split_any(p, N, d_out, prefix, nullptr, false);
}
#endif

}  // namespace npf
