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
// Blocking: a 16 x 16 output tile per block of 256 threads, which also split K four ways (64
// threads with 2 x 2 outputs each per quarter): at M = N = K = 192 there are 144 tiles, about one for
// every SM, and 48 steps in a row.  What bounds it: latency (one gather of up to 256 K values per
// operand in flight at once, then the FMA chain); at the upper end of its range the four FP32
// operations per multiply-add and the 4-byte gathers (about 12 clocks per K value and tile).
#include <cuda_runtime.h>
#include <stdint.h>

#include "launch.h"
#include "params.h"

namespace comet {

namespace sg {
constexpr int T = 256, TM = 16, KC = 256;
// an operand's tile: [row][k] with rows two banks apart when its k values are contiguous in memory,
// else [k][row]; either way the copies fill consecutive banks and a thread reads pairs of values
constexpr int KP = KC + 2, TILE = TM * KP;
constexpr int SMEM = 2 * TILE * 4;
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

template <bool AK, bool BK>
__global__ void __launch_bounds__(sg::T) gemm_small_kernel(const GemmParams p) {
    using namespace sg;
    extern __shared__ __align__(16) float sm[];
    float *As = sm, *Bs = sm + TILE;
    __shared__ int64_t a_row[TM], b_col[TM], c_row[TM], c_col[TM], a_k[KC + 1], b_k[KC + 1];
    const int t = threadIdx.x;
    const uint32_t m0 = blockIdx.x * TM, n0 = blockIdx.y * TM;
    const int rows = (int)min((uint32_t)TM, p.M - m0), cols = (int)min((uint32_t)TM, p.N - n0);
    if (t < TM) {
        int64_t o0 = 0, o1 = 0;
        if (t < rows) radix_offsets(p.ma, m0 + t, o0, o1);
        a_row[t] = o0; c_row[t] = o1;
    } else if (t < 2 * TM) {
        int64_t o0 = 0, o1 = 0;
        if (t - TM < cols) radix_offsets(p.nb, n0 + t - TM, o0, o1);
        b_col[t - TM] = o0; c_col[t - TM] = o1;
    }
    pdl_wait();
    const float *A = reinterpret_cast<const float *>(p.A), *B = reinterpret_cast<const float *>(p.B);
    const int kq = t >> 6, q = t & 63, tm = (q & 7) * 2, tn = (q >> 3) * 2;   // 2 x 2 outputs, every fourth pair of k
    float s[2][2] = {}, c[2][2] = {};
    for (uint32_t k0 = 0; k0 < p.K; k0 += KC) {
        const int nk = (int)min((uint32_t)KC, p.K - k0);
        __syncthreads();   // the previous chunk has been read (and the row offsets are set)
        if (t < nk) {
            int64_t o0, o1;
            radix_offsets(p.k, k0 + t, o0, o1);
            a_k[t] = o0; b_k[t] = o1;
        } else if (t == nk) {
            a_k[t] = b_k[t] = 0;
        }
        __syncthreads();
        gather<AK>(A, a_row, a_k, rows, nk, As, p.dbg_a, p.status);
        gather<BK>(B, b_col, b_k, cols, nk, Bs, p.dbg_b, p.status);
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        __syncthreads();
#pragma unroll 2
        for (int k = 2 * kq; k < nk; k += 8) {
            float a[2][2], b[2][2];
            read22<AK>(As, tm, k, a);
            read22<BK>(Bs, tn, k, b);
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
    // the quarters' sums, [quarter][column][row], then one output per thread
    __syncthreads();
    float2 *part = reinterpret_cast<float2 *>(sm);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) part[(kq * TM + tn + j) * TM + tm + i] = make_float2(s[i][j], c[i][j]);
    __syncthreads();
    pdl_launch();
    const int r = t & 15, n = t >> 4;
    if (r >= rows || n >= cols) return;
    float hi = 0.0f, lo = 0.0f;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const float2 v = part[(g * TM + n) * TM + r];
        const float u = hi + v.x, z = u - hi;
        lo += ((hi - (u - z)) + (v.x - z)) + v.y;
        hi = u;
    }
    double sum = (double)hi + (double)lo;
    float out = hi + lo;
    if (!(fabsf(out) < INFINITY)) {
        // an FP32 product or partial sum left the range (the result itself may not): again in FP64
        sum = 0.0;
        for (uint32_t k = 0; k < p.K; ++k) {
            int64_t oa, ob;
            radix_offsets(p.k, k, oa, ob);
            if (dbg_ok(p.dbg_a, A + a_row[r] + oa, 4, p.status) && dbg_ok(p.dbg_b, B + b_col[n] + ob, 4, p.status))
                sum = fma((double)A[a_row[r] + oa], (double)B[b_col[n] + ob], sum);
        }
        out = (float)sum;
    }
    float *dst = reinterpret_cast<float *>(p.C) + c_row[r] + c_col[n];
    if (!dbg_ok(p.dbg_c, dst, 4, p.status)) return;
    if (p.alpha != 1.0 || p.beta != 0.0) {
        const double v = p.alpha * sum;
        out = (float)(p.beta != 0.0 ? v + p.beta * (double)*dst : v);
    }
    *dst = out;
}

cudaError_t launch_gemm_small(const GemmParams &p, bool a_kcontig, bool b_kcontig, cudaStream_t s) {
    using namespace sg;
    if (p.M == 0 || p.N == 0) return cudaSuccess;
    const dim3 grid((p.M + TM - 1) / TM, (p.N + TM - 1) / TM);
    if (grid.y > 65535) return cudaErrorInvalidConfiguration;
    if (a_kcontig && b_kcontig) launch_pdl(gemm_small_kernel<true, true>, grid, T, SMEM, s, p);
    else if (a_kcontig) launch_pdl(gemm_small_kernel<true, false>, grid, T, SMEM, s, p);
    else if (b_kcontig) launch_pdl(gemm_small_kernel<false, true>, grid, T, SMEM, s, p);
    else launch_pdl(gemm_small_kernel<false, false>, grid, T, SMEM, s, p);
    return cudaGetLastError();
}

}  // namespace comet
