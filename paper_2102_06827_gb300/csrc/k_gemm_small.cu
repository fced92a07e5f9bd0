// Small FP32 contractions: one launch, no pre-pass, no scratch.
//
// A GEMM of a few million multiply-adds is over in a microsecond or two on the FP32 pipes, while the
// split form needs its chain of launches (abs-max, two splits, tcgen05 GEMM) whatever the size: 11 us
// at M = N = K = 192 (18 before those launches overlapped) against 5.5 here.  So
// steps below the line that small_gemm_us / the split model draw run here: operands are gathered
// through their own strides (the transposes of TTGT folded into the loads), products and sums are
// FP32, and every addition's rounding error is kept in a second sum (the error of an FMA into s is
// x*y + (s - t), one more FMA), so the result is as accurate as a sum in twice the precision: relative
// error 3e-8 against 1e-7 of the split form.
//
// The products are of the operands as they are, so those below FP32's range lose bits that the split
// form's scaling (or an alpha that lifts the result) would have kept: each at most 2^-150, K 2^-150
// in all, nothing beside a row's and a column's largest elements if their product reaches K 2^-123.  A tile
// with a sum too small to rule that out (a zero too) looks its rows' and columns' largest elements up, and
// where a pair's product lies below that line runs again with each of them scaled to about one.  At M = N = K =
// 192: 6.0 us, 8.8 with zeros in every tile, 14.6 where all products are below the line.
//
// Blocking: a 16 x 16 output tile per block of 256 threads, which also split K four ways (64
// threads with 2 x 2 outputs each per quarter): at M = N = K = 192 there are 144 tiles, about one for
// every SM, and 48 steps in a row.  What bounds it: latency (one gather of up to 256 K values per
// operand in flight at once, then the FMA chain); at the upper end of its range the four FP32
// operations per multiply-add and the 4-byte gathers (about 12 clocks per K value and tile).
#include <cuda_runtime.h>
#include <stdint.h>

#include "launch.h"
#include "params.h"
#include "split.cuh"
#include "split_schedule.h"

namespace comet {

namespace sg {
constexpr int T = 256, TM = 16, KC = 256;
// an operand's tile: [row][k] with rows two banks apart when its k values are contiguous in memory,
// else [k][row]; either way the copies fill consecutive banks and a thread reads pairs of values
constexpr int KP = KC + 2, TILE = TM * KP;
constexpr int SMEM = 2 * TILE * 4;
constexpr int NONE = 1 << 20;      // exponent of a row of zeros
}  // namespace sg

// One operand's TM x nk values into its tile: asynchronous 4-byte copies, threads along the
// operand's contiguous direction; zeros beyond its rows and at k = nk when nk is odd
template <bool KCONTIG>
__device__ __forceinline__ void gather(const float *__restrict__ base, const int64_t *row, const int64_t *koff, int rows,
                                       int nk, float *s, const DbgRange &rg, int *status) {
    using namespace sg;
    const uint32_t sb = (uint32_t)__cvta_generic_to_shared(s);
    const int t = threadIdx.x, nk2 = nk + (nk & 1);
    auto one = [&](int r, int k) {
        const int at = KCONTIG ? r * KP + k : k * TM + r;
        const float *src = base + row[r] + koff[k];
        if (r < rows && k < nk && dbg_ok(rg, src, 4, status))
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sb + (uint32_t)at * 4), "l"(src) : "memory");
        else
            s[at] = 0.0f;
    };
    if (KCONTIG) {   // a warp takes two rows, its lanes run along k
        for (int r = t >> 5; r < TM; r += T / 32)
#pragma unroll 4
            for (int k = t & 31; k < nk2; k += 32) one(r, k);
    } else {         // sixteen threads run along the rows
#pragma unroll 4
        for (int k = t / TM; k < nk2; k += T / TM) one(t % TM, k);
    }
}

// values (row r, r + 1) x (k, k + 1) of a tile
template <bool KCONTIG>
__device__ __forceinline__ void read22(const float *s, int r, int k, float (&v)[2][2]) {
    using namespace sg;
    const float2 x = *reinterpret_cast<const float2 *>(s + (KCONTIG ? r * KP + k : k * TM + r));
    const float2 y = *reinterpret_cast<const float2 *>(s + (KCONTIG ? (r + 1) * KP + k : (k + 1) * TM + r));
    v[0][0] = x.x; v[1][1] = y.y;
    v[0][1] = KCONTIG ? x.y : y.x;
    v[1][0] = KCONTIG ? y.x : x.y;
}

// Element offsets of a tile's rows and columns in the operands and in C, and of a chunk's K values
struct Offsets {
    int64_t a_row[sg::TM], b_col[sg::TM], c_row[sg::TM], c_col[sg::TM], a_k[sg::KC + 1], b_k[sg::KC + 1];
};

// K values k0 .. k0 + nk - 1 (returned) of both operands into their tiles
template <bool AK, bool BK>
__device__ __forceinline__ int load_chunk(const GemmParams &p, Offsets &o, float *sm, uint32_t k0, int rows, int cols) {
    using namespace sg;
    const int t = threadIdx.x, nk = (int)min((uint32_t)KC, p.K - k0);
    __syncthreads();   // the previous chunk has been read (and the row offsets are set)
    if (t < nk) {
        int64_t o0, o1;
        radix_offsets(p.k, k0 + t, o0, o1);
        o.a_k[t] = o0; o.b_k[t] = o1;
    } else if (t == nk) {
        o.a_k[t] = o.b_k[t] = 0;
    }
    __syncthreads();
    gather<AK>(reinterpret_cast<const float *>(p.A), o.a_row, o.a_k, rows, nk, sm, p.dbg_a, p.status);
    gather<BK>(reinterpret_cast<const float *>(p.B), o.b_col, o.b_k, cols, nk, sm + TILE, p.dbg_b, p.status);
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    return nk;
}

// Adds a chunk's products to this thread's 2 x 2 sums s and their errors c: every fourth pair of k
template <bool AK, bool BK>
__device__ __forceinline__ void multiply_chunk(const float *sm, int nk, float (&s)[2][2], float (&c)[2][2]) {
    using namespace sg;
    const int kq = threadIdx.x >> 6, q = threadIdx.x & 63, tm = (q & 7) * 2, tn = (q >> 3) * 2;
#pragma unroll 2
    for (int k = 2 * kq; k < nk; k += 8) {
        float a[2][2], b[2][2];
        read22<AK>(sm, tm, k, a);
        read22<BK>(sm + TILE, tn, k, b);
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const float n = fmaf(a[i][u], b[j][u], s[i][j]);
                    c[i][j] += fmaf(a[i][u], b[j][u], s[i][j] - n);
                    s[i][j] = n;
                }
    }
}

// The quarters' sums, [quarter][column][row], then output (t % 16, t / 16) per thread: sum and its error.
// *any: whether `flag` is set in some thread of the block.
__device__ __forceinline__ float2 add_quarters(float *sm, const float (&s)[2][2], const float (&c)[2][2], bool flag, bool *any) {
    using namespace sg;
    const int t = threadIdx.x, kq = t >> 6, q = t & 63, tm = (q & 7) * 2, tn = (q >> 3) * 2;
    __syncthreads();
    float2 *part = reinterpret_cast<float2 *>(sm);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) part[(kq * TM + tn + j) * TM + tm + i] = make_float2(s[i][j], c[i][j]);
    *any = __syncthreads_or(flag);
    float hi = 0.0f, lo = 0.0f;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const float2 v = part[(g * TM + (t >> 4)) * TM + (t & 15)];
        const float u = hi + v.x, z = u - hi;
        lo += ((hi - (u - z)) + (v.x - z)) + v.y;
        hi = u;
    }
    return make_float2(hi, lo);
}

// A tile with a sum so small that products may have lost bits below the range (see above): the sum and error
// of this thread's output again, as 2^-e_sum of the result, or v as it was.  The whole block calls it.
template <bool AK, bool BK>
__device__ __forceinline__ float2 sum_scaled(const GemmParams &p, Offsets &o, float *sm, int rows, int cols, float2 v, int *e_sum) {
    using namespace sg;
    const int t = threadIdx.x, r = t & 15, n = t >> 4;
    // the rows' and columns' largest finite magnitudes, eight threads each
    const int row = (t >> 3) & 15;
    auto own = [&](int k) -> float & {
        return t < 128 ? sm[AK ? row * KP + k : k * TM + row] : sm[TILE + (BK ? row * KP + k : k * TM + row)];
    };
    uint32_t largest = 0;
    for (uint32_t k0 = 0; k0 < p.K; k0 += KC) {
        const int nk = load_chunk<AK, BK>(p, o, sm, k0, rows, cols);
        for (int k = t & 7; k < nk; k += 8) {
            const uint32_t bits = __float_as_uint(own(k)) & 0x7FFFFFFFu;
            if (bits < 0x7F800000u) largest = max(largest, bits);
        }
    }
#pragma unroll
    for (int i = 4; i > 0; i >>= 1) largest = max(largest, __shfl_xor_sync(0xffffffffu, largest, i));
    int *top = reinterpret_cast<int *>(o.a_k);   // (six blocks fill an SM's shared memory: no array of its own)
    const int e_own = largest ? exponent_of(__uint_as_float(largest)) : NONE;
    if ((t & 7) == 0) top[t >> 3] = e_own;
    __syncthreads();
    const int ea = top[r], eb = top[TM + n];
    if (!__syncthreads_or(r < rows && n < cols && ea != NONE && eb != NONE && ea + eb < 32 - __clz(p.K) - 123)) return v;
    // again with every row and column scaled to about one (by normal powers of two)
    auto scale = [](int e) { return e == NONE ? 0 : min(max(e, -126), 126); };
    const float f = __uint_as_float((uint32_t)(127 - scale(e_own)) << 23);
    float s[2][2] = {}, c[2][2] = {};
    for (uint32_t k0 = 0; k0 < p.K; k0 += KC) {
        const int nk = load_chunk<AK, BK>(p, o, sm, k0, rows, cols);
        for (int k = t & 7; k < nk; k += 8) own(k) *= f;
        __syncthreads();
        multiply_chunk<AK, BK>(sm, nk, s, c);
    }
    *e_sum = scale(ea) + scale(eb);
    bool any;
    return add_quarters(sm, s, c, false, &any);
}

template <bool AK, bool BK>
__global__ void __launch_bounds__(sg::T) gemm_small_kernel(const __grid_constant__ GemmParams p) {
    using namespace sg;
    extern __shared__ __align__(16) float sm[];
    __shared__ Offsets o;
    const int t = threadIdx.x;
    const uint32_t m0 = blockIdx.x * TM, n0 = blockIdx.y * TM;
    const int rows = (int)min((uint32_t)TM, p.M - m0), cols = (int)min((uint32_t)TM, p.N - n0);
    if (t < TM) {
        int64_t o0 = 0, o1 = 0;
        if (t < rows) radix_offsets(p.ma, m0 + t, o0, o1);
        o.a_row[t] = o0; o.c_row[t] = o1;
    } else if (t < 2 * TM) {
        int64_t o0 = 0, o1 = 0;
        if (t - TM < cols) radix_offsets(p.nb, n0 + t - TM, o0, o1);
        o.b_col[t - TM] = o0; o.c_col[t - TM] = o1;
    }
    pdl_wait();
    float s[2][2] = {}, c[2][2] = {};
    for (uint32_t k0 = 0; k0 < p.K; k0 += KC) {
        const int nk = load_chunk<AK, BK>(p, o, sm, k0, rows, cols);
        multiply_chunk<AK, BK>(sm, nk, s, c);
    }
    // Whether a quarter's sum is as small as K products of less than K 2^-123.  (The vote is the barrier that the
    // quarters meet at anyway; behind a barrier of its own, and with sum_scaled not inlined, 64 registers: 12 to 15 %
    // more at the upper end of this kernel's sizes.)
    bool tiny = false;
    const int q = t & 63, tm = (q & 7) * 2, tn = (q >> 3) * 2;
    const float line = (float)p.K * (float)p.K * 0x1p-123f;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) tiny |= tm + i < rows && tn + j < cols && fabsf(s[i][j]) < line;
    tiny &= 2 * (t >> 6) < p.K;   // (a quarter without a K value says nothing)
    int e_sum = 0;   // v carries 2^-e_sum of the result
    float2 v = add_quarters(sm, s, c, tiny, &tiny);
    if (__builtin_expect(tiny, 0)) v = sum_scaled<AK, BK>(p, o, sm, rows, cols, v, &e_sum);
    const int r = t & 15, n = t >> 4;
    const bool in = r < rows && n < cols;
    pdl_launch();   // (before the quarters meet it costs 2 us on M = N = K = 192: the next grid's blocks crowd in)
    if (!in) return;
    double sum = (double)v.x + (double)v.y;
    float out = v.x + v.y;
    if (!(fabsf(out) < INFINITY)) {
        // an FP32 product or partial sum left the range (the result itself may not): again in FP64
        const float *A = reinterpret_cast<const float *>(p.A) + o.a_row[r], *B = reinterpret_cast<const float *>(p.B) + o.b_col[n];
        sum = 0.0;
        for (uint32_t k = 0; k < p.K; ++k) {
            int64_t oa, ob;
            radix_offsets(p.k, k, oa, ob);
            if (dbg_ok(p.dbg_a, A + oa, 4, p.status) && dbg_ok(p.dbg_b, B + ob, 4, p.status))
                sum = fma((double)A[oa], (double)B[ob], sum);
        }
        out = (float)sum;
    } else if (e_sum != 0) {
        sum = ldexp(sum, e_sum);
        out = (float)sum;
    }
    float *dst = reinterpret_cast<float *>(p.C) + o.c_row[r] + o.c_col[n];
    if (!dbg_ok(p.dbg_c, dst, 4, p.status)) return;
    if (p.alpha != 1.0 || p.beta != 0.0) {
        const double w = p.alpha * sum;
        out = (float)(p.beta != 0.0 ? w + p.beta * (double)*dst : w);
    }
    *dst = out;
}

cudaError_t launch_gemm_small(const GemmParams &p, bool a_kcontig, bool b_kcontig, cudaStream_t s) {
    using namespace sg;
    if (p.M == 0 || p.N == 0) return cudaSuccess;
    const dim3 grid((p.M + TM - 1) / TM, (p.N + TM - 1) / TM);
    if (!small_gemm_fits(p.N)) return cudaErrorInvalidConfiguration;   // the planner does not send such a step here
    if (a_kcontig && b_kcontig) launch_pdl(gemm_small_kernel<true, true>, grid, T, SMEM, s, p);
    else if (a_kcontig) launch_pdl(gemm_small_kernel<true, false>, grid, T, SMEM, s, p);
    else if (b_kcontig) launch_pdl(gemm_small_kernel<false, true>, grid, T, SMEM, s, p);
    else launch_pdl(gemm_small_kernel<false, false>, grid, T, SMEM, s, p);
    return cudaGetLastError();
}

}  // namespace comet
