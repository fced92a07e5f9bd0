// Split contraction kernel on the tcgen05 tensor cores.
//
// The GEMM of the TTGT reformulation (Section 2, C_p[i,k] = A_p[i,j] * B_p[j,k]; Section 6
// "GEMM optimizations" for the blocking of C into tiles and of K into panels) with FP32 (or
// FP64) operands carried as two FP16 parts x * 2^(14-e) = h + l (written by the split pre-pass in
// [plane][row][K] order, K contiguous; see split2 in split.cuh).
//
// Numerics.  Three products are kept: hh, hl and lh (ll is at most 2^-22 of the operands'
// leading powers of two).  The tensor core's FP32 accumulation truncates, so a long K would
// pile up a one-sided error: K runs in chunks of 32 or 64 values, each summed in tensor memory from
// zero, its correction MMAs (2^-11 of the result) first and its two or four hh MMAs last, and the
// epilogue warps add the chunks into FP32 register sums of two levels (round to nearest).  At
// the end of a tile the sum is scaled by alpha * 2^(eA + eB - 28) and stored.
// Relative 2-norm error against FP64, K = 64 / 576 / 1633 / 12288, and what three fixed-point
// bfloat16 parts with six products gave (whose parts are relative to the largest element):
//   uniform in [-1, 1)   0.98 1.13 1.23 1.63e-7   (1.30 1.33 1.32 1.5e-7)
//   uniform in +-0.7     1.09 1.22 1.31 1.69e-7   (2.2e-7)
//   normal               1.05 1.19 1.29 1.68e-7   (18e-7)
// Chunks of 64 throughout: 1.26 .. 1.63e-7 (uniform); one level of sums: 2.8e-7 at K = 12288.
//
// GB300 form: one persistent pair of CTAs (cluster of two, 512 threads each) per two SMs, the
// pair's output tile 256 x bn (bn = 48 .. 192, chosen by split_schedule):
//   warp 0       TMA producer: one 3-D tensor load per operand and stage brings both planes of
//                the CTA's 128 rows of A and bn/2 rows of B, 64 K values, 128-byte swizzled; all
//                of a stage's loads, from both CTAs, complete on CTA 0's barrier
//   warp 1       allocates 512 tensor-memory columns (two accumulators); in CTA 0, lane 0 issues
//                tcgen05.mma.cta_group::2 (M=256, N=bn, K=16) and commits to both CTAs
//   warps 4..15  epilogue: each owns one tensor-memory lane quadrant and one third of the
//                columns; drains an accumulator after every chunk into register sums (64 columns
//                in two levels: 128 registers of a thread's 160) while the MMAs fill the other one,
//                and at the end of the tile stores through the output's strides (the output
//                permutation of TTGT folded in)
//   3-stage shared-memory ring (56 KB per stage and CTA at bn = 192).
// What bounds it: the power cap at large sizes.  M = N = K = 12288: 7.4-7.7 ms = 1.44-1.5 PFLOP/s of
// MMA at 1630-1690 MHz (six bf16 products: 10.7-10.9 ms); ncu at 5120^3, alone: tensor pipe 93 %.
// Why pairs: with one CTA per 128 x 256 tile a stage reads 144 KB of operands from shared memory
// and fills 96 KB per 1536 MMA cycles, 160 bytes per clock against the SM's 128; in a pair each
// CTA holds half of B (bn = 192: 84 + 56 KB per 1152 cycles, 121).  Tiles of 240 and 256 columns run
// 5 % faster at 12288^3 (7.0 ms) but leave no registers for the second level of sums.
// Every wait is bounded (%globaltimer); on expiry the CTA records COMET_ERR_TIMEOUT in the
// status word, drains its own copies in flight, frees its tensor memory and returns.
#include <cuda.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <stdint.h>

#include <algorithm>

#include "launch.h"
#include "params.h"
#include "sm100.cuh"
#include "split.cuh"
#include "split_schedule.h"

namespace comet {

namespace split {
constexpr int BM = 128;                         // rows per CTA
constexpr int BN = kSplitMaxBN;                 // columns per pair (largest)
constexpr int BK = kSplitBK, STAGES = 3;
constexpr int A_PLANE = BM * BK * 2;            // 16 KB
constexpr int B_PLANE = BN / 2 * BK * 2;        // 12 KB at bn = 192
constexpr int A_STAGE = 2 * A_PLANE;
constexpr int STAGE_BYTES = A_STAGE + 2 * B_PLANE;   // 56 KB
constexpr int EPI_WARPS = 12;                   // four lane quadrants x three column groups
constexpr int GN = BN / 3;                      // columns per group (largest)
constexpr int THREADS = 128 + 32 * EPI_WARPS;
constexpr uint32_t TMEM_COLS = 512;             // two accumulators of 256 columns
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /*align*/ + BN * 8 /*c_col*/ + 256;
constexpr int STRIP = 24;                       // columns per block of the reduce kernel
constexpr uint32_t SW128 = 2;                   // descriptor swizzle code: 128-byte swizzle
constexpr uint32_t SBO = 8 * BK * 2;            // 8 rows of 128 bytes
}  // namespace split

struct SplitArgs {
    uint32_t m_tiles, n_tiles;   // pair tiles
    uint32_t bn;                 // columns per pair tile
    uint32_t nch;                // K stages of 64
    uint32_t items;              // work items: m_tiles x n_tiles x ksplit
    uint32_t ksplit;             // K slices (1 = whole K per tile; > 1: FP32 partials to `partial`)
    uint32_t kslice_chunks;      // stages per slice
    uint32_t chunk_steps;        // K steps of 16 per accumulation chunk (4 or 2)
    uint32_t group;              // chunks per first-level sum
    float *partial;              // per slice, tile and CTA bn x 128 partial sums (scaled by
                                 // 2^(eA+eB)), [slice][tile][CTA][column][row], row fastest
    DbgRange dbg_p;              // debug builds: the partial sums' buffer
    int debug_flags;
    const void *scale_a;         // bits of max |A|, max |B| (input precision)
    const void *scale_b;
};

// work item's tile -> (m tile, n tile): bands of 8 m-tiles, n-major inside a band, for L2 reuse
__device__ __forceinline__ void split_tile_coords(uint32_t tile, uint32_t m_tiles, uint32_t n_tiles, uint32_t &mt,
                                                  uint32_t &nt) {
    const uint32_t G = 8;
    const uint32_t band = tile / (G * n_tiles);
    const uint32_t base = band * G;
    const uint32_t g = min(G, m_tiles - base);
    const uint32_t r = tile - band * G * n_tiles;
    mt = base + r % g;
    nt = r / g;
}

// The MMAs of one stage in chunks of STEPS K steps of 16 (32 bytes further in a swizzled row each),
// corrections first; `ch` counts the chunks.  False: the wait for an accumulator ran out.
template <int STEPS>
__device__ __forceinline__ bool mma_stage(uint32_t sa, uint32_t sb, uint32_t b_plane, uint32_t idesc, uint32_t tmem,
                                          uint32_t &ch, uint64_t *tfull, uint64_t *tempty, uint64_t tmo,
                                          volatile int *abort_flag) {
    using namespace split;
    using namespace sm100;
    const uint64_t ah = smem_desc(sa, 16, SBO, SW128), al = smem_desc(sa + A_PLANE, 16, SBO, SW128);
    const uint64_t bh = smem_desc(sb, 16, SBO, SW128), bl = smem_desc(sb + b_plane, 16, SBO, SW128);
#pragma unroll
    for (int k0 = 0; k0 < BK / 16; k0 += STEPS, ++ch) {
        // accumulator ch % 2: the epilogue warps of both CTAs have drained it
        const uint32_t buf = ch & 1, use = ch >> 1, acc = tmem + buf * 256;
        if (use > 0 && !mbar_wait(&tempty[buf], (use - 1) & 1, tmo, abort_flag)) return false;
        tc_fence_after();
#pragma unroll
        for (int k = k0; k < k0 + STEPS; ++k) {
            mma_f16_pair(acc, al + 2 * k, bh + 2 * k, idesc, k == k0 ? 0u : 1u);
            mma_f16_pair(acc, ah + 2 * k, bl + 2 * k, idesc, 1);
        }
#pragma unroll
        for (int k = k0; k < k0 + STEPS; ++k) mma_f16_pair(acc, ah + 2 * k, bh + 2 * k, idesc, 1);
        mma_commit_pair(&tfull[buf]);   // chunk complete: ready to drain in both CTAs
    }
    return true;
}

template <typename TOut, bool KSPLIT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(split::THREADS, 1)
    gemm_split_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                      const GemmParams p, const SplitArgs x) {
    using namespace split;
    using namespace sm100;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t *smem = smem_raw + (((raw + 1023) & ~1023u) - raw);
    uint8_t *stage_base = smem;
    int64_t *c_col = reinterpret_cast<int64_t *>(smem + STAGES * STAGE_BYTES);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + STAGES * STAGE_BYTES + BN * 8);
    uint64_t *full = bars, *empty = bars + STAGES, *tfull = bars + 2 * STAGES, *tempty = tfull + 2,
             *mma_done = tempty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(mma_done + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const uint32_t pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
    const uint64_t tmo = (uint64_t)p.timeout_ns;
    const uint32_t tiles = x.m_tiles * x.n_tiles;
    const uint32_t stage_bytes = (uint32_t)A_STAGE + x.bn * (BK * 2);   // one CTA's loads of a stage
    // work item t: K slice t / tiles of output tile t % tiles
    auto kslice = [&](uint32_t t, uint32_t &c0, uint32_t &c1) -> uint32_t {
        if constexpr (!KSPLIT) {
            c0 = 0;
            c1 = x.nch;
            return 0;
        } else {
            const uint32_t ks = t / tiles;
            c0 = ks * x.kslice_chunks;
            c1 = min(x.nch, c0 + x.kslice_chunks);
            return ks;
        }
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&tfull[b], 1); mbar_init(&tempty[b], 2 * EPI_WARPS); }
        mbar_init(mma_done, 1);
        *abort_flag = 0;
        fence_barrier_init();
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
    }
    if (warp == 1) tmem_alloc_pair(tmem_slot, TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    cluster_sync();   // both CTAs' barriers are set up before either CTA signals the other
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    pdl_wait();       // the pre-passes' planes and scales, and whoever read or wrote C before

    auto fail = [&]() {
        *abort_flag = 1;
        atomicExch(p.status, (int)COMET_ERR_TIMEOUT);
    };
    auto tile_coords = [&](uint32_t t, uint32_t &mt, uint32_t &nt) {
        if constexpr (KSPLIT) t %= tiles;
        split_tile_coords(t, x.m_tiles, x.n_tiles, mt, nt);
    };

    // registers: 512 threads launch at 128 each; 12 x 32 x 160 + 4 x 32 x 32 = 65536
    if (warp < 4) {
    regs_down<32>();
    if (warp == 0) {
        if (lane == 0) {
            // ---------------- TMA producer ----------------
            uint32_t it = 0;
            bool ok = true;
            bool injected = false;
            for (uint32_t t = pair; t < x.items && ok; t += n_pairs) {
                uint32_t mt, nt, c0, c1;
                tile_coords(t, mt, nt);
                kslice(t, c0, c1);
                for (uint32_t c = c0; c < c1; ++c, ++it) {
                    const uint32_t s = it % STAGES, round = it / STAGES;
                    if (round > 0 && !mbar_wait(&empty[s], (round - 1) & 1, tmo, abort_flag)) {
                        fail(); ok = false; break;
                    }
                    if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * stage_bytes);
                    if ((x.debug_flags & 1) && !injected && blockIdx.x == 0) {
                        injected = true;   // fault injection: this stage's loads are withheld
                        continue;
                    }
                    const uint32_t bar = map_to_rank(&full[s], 0);
                    uint8_t *sa = stage_base + s * STAGE_BYTES;
                    tma_load_3d_pair(&tmA, bar, sa, c * BK, mt * (2 * BM) + rank * BM, 0);
                    tma_load_3d_pair(&tmB, bar, sa + A_STAGE, c * BK, nt * x.bn + rank * (x.bn / 2), 0);
                }
            }
            // drain: wait for every load still in flight, of both CTAs (at most one per stage)
            if (rank == 0) {
                const uint32_t first = it > (uint32_t)STAGES ? it - STAGES : 0;
                for (uint32_t j = first; j < it; ++j) {
                    const uint32_t s = j % STAGES, round = j / STAGES;
                    mbar_wait(&full[s], round & 1, tmo, nullptr);
                }
            }
        }
    } else if (warp == 1) {
        if (rank == 0 && lane == 0) {
            // ---------------- MMA issuer ----------------
            const uint32_t idesc = idesc_f16_f32(2 * BM, x.bn);
            const uint32_t b_plane = x.bn / 2 * (BK * 2);
            uint32_t it = 0, ch = 0;   // stages and chunks so far
            bool ok = true;
            for (uint32_t t = pair; t < x.items && ok; t += n_pairs) {
                uint32_t c0, c1;
                kslice(t, c0, c1);
                for (uint32_t c = c0; c < c1; ++c, ++it) {
                    const uint32_t s = it % STAGES, round = it / STAGES;
                    if (!mbar_wait(&full[s], round & 1, tmo, abort_flag)) { fail(); ok = false; break; }
                    const uint32_t sa = smem_u32(stage_base + s * STAGE_BYTES), sb = sa + A_STAGE;
                    ok = x.chunk_steps == 4 ? mma_stage<4>(sa, sb, b_plane, idesc, tmem_base, ch, tfull, tempty, tmo, abort_flag)
                                            : mma_stage<2>(sa, sb, b_plane, idesc, tmem_base, ch, tfull, tempty, tmo, abort_flag);
                    if (!ok) { fail(); break; }
                    mma_commit_pair(&empty[s]);   // the stage is free in both CTAs once read
                }
            }
            // make sure no MMA is still writing tensor memory before it is freed
            mma_commit_pair(mma_done);
            mbar_wait(mma_done, 0, tmo, nullptr);
        }
    }
    } else {
        regs_up<160>();
        // ---------------- epilogue (warps 4..15) ----------------
        const int quad = warp & 3;                  // tensor-memory lanes 32*quad .. 32*quad+31
        const uint32_t gn = x.bn / 3, g0 = (uint32_t)((warp - 4) >> 2) * gn;   // columns g0 .. g0 + gn - 1
        const int et = threadIdx.x - 128;           // 0..383
        const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
        const int e_sum = half_exponent<TOut>(scale_exponent<TOut>(x.scale_a)) +
                          half_exponent<TOut>(scale_exponent<TOut>(x.scale_b));
        // 2^(eA+eB-28) in two factors: the sums carry 2^28 more than the result's scale
        constexpr float kShift = 1.0f / (float)(1 << (2 * kHalfShift));
        const uint32_t tempty0 = map_to_rank(tempty, 0);
        uint32_t ch = 0;     // chunks so far
        const uint32_t per_stage = BK / 16 / x.chunk_steps;
        bool dead = false;   // once set, the warp keeps pace with the barriers but does no work
        TOut *C = reinterpret_cast<TOut *>(p.C);
        for (uint32_t t = pair; t < x.items; t += n_pairs) {
            uint32_t mt, nt, c0, c1;
            tile_coords(t, mt, nt);
            const uint32_t ks = kslice(t, c0, c1);
            if constexpr (!KSPLIT) {
                // column offsets of this tile in C (all eight epilogue warps always meet here)
                named_bar_sync(1, 32 * EPI_WARPS);
                int64_t o0 = 0, o1 = 0;
                if ((uint32_t)et < x.bn && nt * x.bn + et < p.N) radix_offsets(p.nb, nt * x.bn + et, o0, o1);
                if (et < BN) c_col[et] = o1;
                named_bar_sync(1, 32 * EPI_WARPS);
            }
            // two levels of sums, two columns per register pair: T over x.group chunks, S over the groups
            uint64_t T[GN / 2], S[GN / 2];
#pragma unroll
            for (int j = 0; j < GN / 2; ++j) T[j] = S[j] = 0;
            const uint32_t n_ch = (c1 - c0) * per_stage;
            uint32_t left = x.group;
            for (uint32_t c = 0; c < n_ch; ++c, ++ch) {
                if (dead) continue;
                const uint32_t buf = ch & 1;
                bool ok = mbar_wait(&tfull[buf], (ch >> 1) & 1, tmo, abort_flag);
                ok = __all_sync(0xffffffffu, ok);   // warp-uniform before the .sync.aligned loads
                if (!ok) { if (lane == 0) fail(); dead = true; continue; }
                tc_fence_after();
                const uint32_t src = tmem_base + lane_base + buf * 256 + g0;
#pragma unroll
                for (int c16 = 0; c16 < GN / 16; ++c16) {
                    if ((uint32_t)c16 * 16 < gn) {
                        uint32_t r[16];
                        tmem_ld16(src + c16 * 16, r);
                        tmem_ld_wait();
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            uint64_t &t = T[c16 * 8 + q];
                            t = f32x2_add(t, f32x2_pack(r[2 * q], r[2 * q + 1]));
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(tempty0 + buf * 8);
                if (--left == 0 || c + 1 == n_ch) {
                    left = x.group;
#pragma unroll
                    for (int j = 0; j < GN / 2; ++j) {
                        S[j] = f32x2_add(S[j], T[j]);
                        T[j] = 0;
                    }
                }
            }
            if (dead) continue;
            auto result = [&](int j) {   // column j of the group, without the splits' 2^28
                const float2 v = f32x2_unpack(S[j / 2]);
                return (j & 1 ? v.y : v.x) * kShift;
            };
            const uint32_t ml = quad * 32 + lane, m = mt * (2 * BM) + rank * BM + ml;
            const uint32_t n0 = nt * x.bn + g0;
            const int n_here = (int)min(gn, p.N > n0 ? p.N - n0 : 0u);
            if constexpr (KSPLIT) {   // K slice partial: scaled sums to the tile's slot, row fastest (coalesced)
                if (m < p.M) {
                    const float sc = (float)ldexp(1.0, e_sum);
                    float *P = x.partial + ((((size_t)ks * tiles + t % tiles) * 2 + rank) * x.bn + g0) * BM + ml;
#pragma unroll
                    for (int j = 0; j < GN; ++j)
                        if (j < n_here && dbg_ok(x.dbg_p, P + (size_t)j * BM, 4, p.status))
                            P[(size_t)j * BM] = sc * result(j);
                }
            } else if (m < p.M) {
                int64_t r0 = 0, c_row = 0;
                radix_offsets(p.ma, m, r0, c_row);
                TOut *row = C + c_row;
                const int64_t *cc = c_col + g0;
                const double scale = ldexp(p.alpha, e_sum);
                if (p.beta == 0.0) {
                    const TOut sc = (TOut)scale;
#pragma unroll
                    for (int j = 0; j < GN; ++j)
                        if (j < n_here && dbg_ok(p.dbg_c, row + cc[j], (int)sizeof(TOut), p.status))
                            row[cc[j]] = sc * (TOut)result(j);
                } else {
#pragma unroll
                    for (int j = 0; j < GN; ++j)
                        if (j < n_here && dbg_ok(p.dbg_c, row + cc[j], (int)sizeof(TOut), p.status)) {
                            TOut *dst = row + cc[j];
                            *dst = (TOut)(scale * (double)result(j) + p.beta * (double)*dst);
                        }
                }
            }
        }
    }
    pdl_launch();
    tc_fence_before();
    __syncthreads();
    cluster_sync();   // neither CTA frees its tensor memory or leaves while the other may still use it
    tc_fence_after();
    if (warp == 1) tmem_dealloc_pair(tmem_base, TMEM_COLS);
}

// K-slice partials -> C: C[m, n] = alpha * sum_ks P[ks][tile][CTA][n][m] (+ beta C), through C's
// strides.  A block takes 32 columns of one CTA's 128 rows: a thread keeps one row (its offset
// is worked out once) and walks 16 columns, whose offsets the block tabulates, so reads and stores
// run along the rows.  The slices are added with an exact error term (two-sum) in FP32: FP64 adds
// run at 1/64 of that rate here (39 us of 163 on a 1633^3 contraction with two slices).
template <typename TOut>
__global__ void __launch_bounds__(256) split_reduce_kernel(const GemmParams p, const SplitArgs x) {
    using namespace split;
    __shared__ int64_t c_col[STRIP];
    const uint32_t strips = x.bn / STRIP;
    const uint32_t strip = blockIdx.x % strips, cta = blockIdx.x / strips, tile = cta >> 1, rank = cta & 1;
    uint32_t mt, nt;
    split_tile_coords(tile, x.m_tiles, x.n_tiles, mt, nt);
    const uint32_t ml = threadIdx.x & 127, m = mt * (2 * BM) + rank * BM + ml, n0 = nt * x.bn + strip * STRIP;
    if (threadIdx.x < STRIP && n0 + threadIdx.x < p.N) {
        int64_t o0, o1;
        radix_offsets(p.nb, n0 + threadIdx.x, o0, o1);
        c_col[threadIdx.x] = o1;
    }
    int64_t r0 = 0, c_row = 0;
    if (m < p.M) radix_offsets(p.ma, m, r0, c_row);
    pdl_wait();
    __syncthreads();
    if (m >= p.M) return;
    const size_t slice = (size_t)x.m_tiles * x.n_tiles * 2 * x.bn * BM;
    const float *P = x.partial + ((size_t)cta * x.bn + strip * STRIP) * BM + ml;
#pragma unroll 4
    for (uint32_t j = threadIdx.x >> 7; j < STRIP; j += 2) {
        if (n0 + j >= p.N) break;
        float s = 0.0f, lo = 0.0f;
        for (uint32_t k = 0; k < x.ksplit; ++k) {
            const float *q = P + k * slice + (size_t)j * BM;
            if (!dbg_ok(x.dbg_p, q, 4, p.status)) continue;
            const float v = *q, t = s + v, z = t - s;
            lo += (s - (t - z)) + (v - z);
            s = t;
        }
        TOut *c = reinterpret_cast<TOut *>(p.C) + c_row + c_col[j];
        if (!dbg_ok(p.dbg_c, c, (int)sizeof(TOut), p.status)) continue;
        if (!(fabsf(s) < INFINITY)) lo = 0.0f;   // the error term of an infinite sum is not a number
        if (sizeof(TOut) == 4 && p.alpha == 1.0 && p.beta == 0.0) {
            *c = (TOut)(s + lo);
        } else {
            const double r = p.alpha * ((double)s + (double)lo);
            *c = (TOut)(p.beta != 0.0 ? r + p.beta * (double)*c : r);
        }
    }
}

// ---- host side --------------------------------------------------------------------------------

static PFN_cuTensorMapEncodeTiled_v12000 get_encode() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        cudaDriverEntryPointQueryResult q;
        void *f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
    }
    return fn;
}

// 3-D map over [2 planes][rows][K] FP16 with rows of kpad elements; box = K 64 x rows box_rows x 2
static bool make_map(CUtensorMap *m, const void *base, uint64_t rows, uint64_t K, uint64_t kpad,
                     uint32_t box_rows) {
    auto enc = get_encode();
    if (!enc) return false;
    cuuint64_t dims[3] = {K, rows, 2};
    cuuint64_t strides[2] = {kpad * 2, rows * kpad * 2};
    cuuint32_t box[3] = {(cuuint32_t)split::BK, box_rows, 2};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void *>(base), dims, strides, box,
                     estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

static int sm_count() {
    static int n = 0;
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 1;
    }
    return n;
}

// the shared-memory attribute is set once per kernel instantiation
template <typename TOut, bool KSPLIT>
static void launch_split_kernel(const CUtensorMap &ta, const CUtensorMap &tb, const GemmParams &p,
                                const SplitArgs &x, int ctas, cudaStream_t s) {
    static const bool attr = [] {
        cudaFuncSetAttribute(gemm_split_kernel<TOut, KSPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             split::SMEM_BYTES);
        return true;
    }();
    (void)attr;
    launch_pdl(gemm_split_kernel<TOut, KSPLIT>, ctas, split::THREADS, split::SMEM_BYTES, s, ta, tb, p, x);
}

cudaError_t launch_gemm_split(const GemmParams &p, const void *parts_a, const void *parts_b,
                              int64_t kpad, const void *scale_a, const void *scale_b,
                              int out_bytes, int debug_flags, cudaStream_t s,
                              uint32_t want_ksplit, float *partial, int64_t partial_bytes) {
    using namespace split;
    if (p.M == 0 || p.N == 0) return cudaSuccess;
    const uint32_t pairs = (uint32_t)std::max(1, sm_count() / 2);
    const SplitSchedule sch = split_schedule(p.M, p.N, p.K, pairs, want_ksplit, partial ? partial_bytes : 0);
    CUtensorMap ta, tb;
    if (!make_map(&ta, parts_a, p.M, p.K, (uint64_t)kpad, BM)) return cudaErrorInvalidValue;
    if (!make_map(&tb, parts_b, p.N, p.K, (uint64_t)kpad, sch.bn / 2)) return cudaErrorInvalidValue;
    SplitArgs x;
    x.m_tiles = (p.M + kSplitBM - 1) / kSplitBM;
    x.n_tiles = (p.N + sch.bn - 1) / sch.bn;
    x.bn = sch.bn;
    x.nch = (p.K + BK - 1) / BK;
    x.ksplit = sch.ksplit;
    x.kslice_chunks = (x.nch + sch.ksplit - 1) / sch.ksplit;
    x.items = x.m_tiles * x.n_tiles * x.ksplit;
    split_chunks(x.kslice_chunks, &x.chunk_steps, &x.group);
    x.partial = partial;
    x.dbg_p = dbg_range(partial, split_partial_bytes(p.M, p.N, sch));
    x.debug_flags = debug_flags;
    x.scale_a = scale_a;
    x.scale_b = scale_b;
    const int ctas = 2 * (int)std::min(pairs, x.items);
    if (out_bytes == 8) {
        if (x.ksplit > 1) launch_split_kernel<double, true>(ta, tb, p, x, ctas, s);
        else launch_split_kernel<double, false>(ta, tb, p, x, ctas, s);
    } else {
        if (x.ksplit > 1) launch_split_kernel<float, true>(ta, tb, p, x, ctas, s);
        else launch_split_kernel<float, false>(ta, tb, p, x, ctas, s);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || x.ksplit == 1) return e;
    const uint32_t blocks = x.m_tiles * x.n_tiles * 2 * (x.bn / STRIP);
    if (out_bytes == 8) launch_pdl(split_reduce_kernel<double>, blocks, 256, 0, s, p, x);
    else launch_pdl(split_reduce_kernel<float>, blocks, 256, 0, s, p, x);
    return cudaGetLastError();
}

}  // namespace comet
