// Split contraction kernel on the tcgen05 tensor cores.
//
// The GEMM of the TTGT reformulation (Section 2, C_p[i,k] = A_p[i,j] * B_p[j,k]; Section 6
// "GEMM optimizations" for the blocking of C into tiles and of K into panels) with FP32 (or
// FP64) operands carried as two FP16 parts x * 2^(14-e) = h + l (written by the split pre-pass in
// [plane][row][K] order, K contiguous; see HalfScale in split.cuh).
//
// Numerics.  Three products are kept: hh, hl and lh (ll is at most 2^-22 of the operands'
// leading powers of two).  The tensor core's FP32 accumulation truncates, so a long K would
// pile up a one-sided error: K runs in chunks of 32 or 64 values, each summed in tensor memory from
// zero, its correction MMAs (2^-11 of the result) first and its two or four hh MMAs last, and the
// epilogue warps add the chunks into FP32 register sums of two levels (round to nearest).  At
// the end of a tile the sum is scaled by alpha * 2^(eA + eB - 28) and stored.
// Relative 2-norm error against FP64, measured (M = N = 1024, K = 64 / 576 / 1633 / 4800 / 12288), and in
// brackets that of three fixed-point bfloat16 parts with six products, whose parts are relative to the
// largest element and whose leading products sum exactly:
//   uniform in [-1, 1)   0.87 1.02 1.13 1.45 1.56e-7   (1.10 1.11 1.16 1.24 3.99e-7; 1.2 to 4.0 by the seed)
//   uniform in +-0.7     1.10 1.23 1.32 1.59 1.70e-7   (2.17 2.19 2.21 2.26 2.32e-7)
//   normal               1.06 1.19 1.29 1.57 1.68e-7   (18.3 18.4 18.4 18.4 18.4e-7)
//   uniform in [0, 1)    0.91 0.93 0.94 1.91 1.92e-7   (0.34 0.31 0.34 0.64 0.81e-7)
// So operands of one sign, whose chunks are all truncated the same way, lose by it.  Chunks of 32 beyond
// K = 4096 too (plan option kc): uniform 1.28 and 1.47e-7, one sign 1.02 and 1.09e-7, 15 to 30 % more time.
//
// GB300 form: one persistent pair of CTAs (cluster of two, 512 threads each) per two SMs, the
// pair's output tile 256 x bn (bn = 48 .. 192, chosen by split_schedule):
//   warp 0       TMA producer: one 3-D tensor load per operand and stage brings both planes of
//                the CTA's 128 rows of A and bn/2 rows of B, 64 K values, 128-byte swizzled; all
//                of a stage's loads, from both CTAs, complete on CTA 0's barrier
//   warp 1       allocates 512 tensor-memory columns (two to four accumulators, see NBUF); in CTA 0
//                the whole warp runs the loop and one elected lane issues tcgen05.mma.cta_group::2
//                (M=256, N=bn, K=16) and commits to both CTAs
//   warps 4..15  epilogue: each owns one tensor-memory lane quadrant and one third of the
//                columns; drains an accumulator after every chunk into register sums (64 columns
//                in two levels: 128 registers of a thread's 160) while the MMAs fill the other one,
//                and at the end of the tile stores through the output's strides (the output
//                permutation of TTGT folded in; through shared memory where its runs lie along N)
//   3-stage shared-memory ring (56 KB per stage and CTA at bn = 192).
// What bounds it: the power cap at large sizes.  M = N = K = 12288: 6.8 to 7.4 ms by the box = 1.5 to
// 1.6 PFLOP/s of MMA (six bf16 products: 10.7-10.9 ms); at middle sizes the hand-over of an accumulator per chunk (see NBUF).
// Why pairs: with one CTA per 128 x 256 tile a stage reads 144 KB of operands from shared memory
// and fills 96 KB per 1536 MMA cycles, 160 bytes per clock against the SM's 128; in a pair each
// CTA holds half of B (bn = 192: 84 + 56 KB per 1152 cycles, 121).  Tiles of 240 and 256 columns ran
// 5 % faster at 12288^3 (before the warp-wide issue) but leave no registers for the second level of sums.
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
constexpr int THREADS = 128 + 32 * EPI_WARPS;
constexpr uint32_t TMEM_COLS = 512;             // two accumulators of 256 columns, or eight of 64 (bn = 48)
constexpr int MAXBUF = 8;
constexpr int TURN = 32 * 17 * 4;               // one warp's 32 rows x 16 columns, turned (n_fast)
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /*align*/ + 2 * BN * 8 /*c_col*/ + 256 + EPI_WARPS * TURN;
constexpr int STRIP = 24;                       // columns per block of the reduce kernel
constexpr uint32_t SW128 = 2;                   // descriptor swizzle code: 128-byte swizzle
constexpr uint32_t SBO = 8 * BK * 2;            // 8 rows of 128 bytes
}  // namespace split

struct SplitArgs {
    uint32_t m_tiles, n_tiles;   // pair tiles
    FastDiv fd_band, fd_last;    // division by 8 x n_tiles and by the last band's m-tiles
    uint32_t bn;                 // columns per pair tile
    uint32_t nch;                // K stages of 64
    uint32_t items;              // work items: m_tiles x n_tiles x ksplit
    uint32_t ksplit;             // K slices (1 = whole K per tile; > 1: FP32 partials to `partial`)
    uint32_t kslice_chunks;      // stages per slice
    uint32_t chunk_steps;        // K steps of 16 per accumulation chunk (4 or 2)
    uint32_t group;              // chunks per first-level sum
    int n_fast;                  // C's stride-1 label is in the N group: a warp's stores run along columns
    float *partial;              // per slice, tile and CTA bn x 128 partial sums (of the scaled
                                 // operands), [slice][tile][CTA][column][row], row fastest
    DbgRange dbg_p;              // debug builds: the partial sums' buffer
    int debug_flags;
    const void *scale_a;         // bits of max |A|, max |B| (input precision)
    const void *scale_b;
};

// work item's tile -> (m tile, n tile): bands of 8 m-tiles, n-major inside a band, for L2 reuse
__device__ __forceinline__ void split_tile_coords(uint32_t tile, const SplitArgs &x, uint32_t &mt, uint32_t &nt) {
    const uint32_t G = 8;
    const uint32_t band = fd_div(tile, x.fd_band);
    const uint32_t base = band * G;
    const uint32_t r = tile - band * G * x.n_tiles;
    if (x.m_tiles - base >= G) {
        mt = base + r % G;
        nt = r / G;
    } else {
        nt = fd_div(r, x.fd_last);
        mt = base + r - nt * (x.m_tiles - base);
    }
}

// chunks of stages c0 .. c1 - 1: per_stage each, except that the end of K may leave the second half of its
// stage empty
__device__ __forceinline__ uint32_t split_chunk_count(uint32_t c0, uint32_t c1, uint32_t per_stage, uint32_t K) {
    const uint32_t n = (c1 - c0) * per_stage;
    return per_stage == 2 && c1 * split::BK >= K + split::BK / 2 ? n - 1 : n;
}

// The MMAs of one stage in chunks of STEPS K steps of 16 (32 bytes further in a swizzled row each),
// corrections first, as far as k_steps steps hold K values; `ch` counts the chunks.  False: the wait for
// an accumulator ran out.
template <int STEPS, uint32_t nbuf>
__device__ __forceinline__ bool mma_stage(int k_steps, uint32_t sa, uint32_t sb, uint32_t b_plane, uint32_t idesc, uint32_t tmem,
                                          uint32_t &ch, uint64_t *tfull, uint64_t *tempty, uint64_t tmo,
                                          volatile int *abort_flag) {
    using namespace split;
    using namespace sm100;
    const uint64_t ah = smem_desc(sa, 16, SBO, SW128), al = smem_desc(sa + A_PLANE, 16, SBO, SW128);
    const uint64_t bh = smem_desc(sb, 16, SBO, SW128), bl = smem_desc(sb + b_plane, 16, SBO, SW128);
#pragma unroll
    for (int k0 = 0; k0 < BK / 16; k0 += STEPS) {
        if (k0 >= k_steps) break;
        // accumulator ch % nbuf: the epilogue warps of both CTAs have drained it
        const uint32_t buf = ch % nbuf, use = ch / nbuf, acc = tmem + buf * (nbuf == 3 ? 160 : 512 / nbuf);
        if (use > 0 && !__all_sync(0xffffffffu, mbar_wait(&tempty[buf], (use - 1) & 1, tmo, abort_flag))) return false;
        tc_fence_after();
        if (elect_one()) {
#pragma unroll
            for (int k = k0; k < k0 + STEPS; ++k) {
                mma_f16_pair(acc, al + 2 * k, bh + 2 * k, idesc, k == k0 ? 0u : 1u);
                mma_f16_pair(acc, ah + 2 * k, bl + 2 * k, idesc, 1);
            }
#pragma unroll
            for (int k = k0; k < k0 + STEPS; ++k) mma_f16_pair(acc, ah + 2 * k, bh + 2 * k, idesc, 1);
            mma_commit_pair(&tfull[buf]);   // chunk complete: ready to drain in both CTAs
        }
        __syncwarp();
        ++ch;
    }
    return true;
}

template <typename TOut, bool KSPLIT, int NBUF>
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
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + STAGES * STAGE_BYTES + 2 * BN * 8);
    uint64_t *full = bars, *empty = bars + STAGES, *tfull = bars + 2 * STAGES, *tempty = tfull + MAXBUF,
             *mma_done = tempty + MAXBUF;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(mma_done + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    volatile uint32_t *issued = tmem_slot + 2;   // stages that CTA 0 and CTA 1 of the pair have loaded

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const uint32_t pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
    const uint64_t tmo = (uint64_t)p.timeout_ns;
    const uint32_t tiles = x.m_tiles * x.n_tiles;
    // Accumulators: as many as tensor memory holds of the tile's columns (2 of 256, 3 of 160, 4 of 128).  With
    // two, a chunk of 32 K values takes the round trip of a hand-over, about 1050 clocks, whatever
    // its width.
    // NBUF 8 (narrow tiles of few chunks): each group of four epilogue warps takes whole tiles in turn,
    // three at a time, and tensor memory holds eight accumulators.  With a third of 48 columns per warp
    // the fixed work per tile (offsets, waits, a barrier) was most of it: 995 K x 48, K = 48: 177 us,
    // 130 us so.  A tile has at most three chunks then: a group that has seen its last tile's chunks
    // waits for one at most seven further on, so the accumulator's phase before that one is over and the
    // parity it waits for is not the older phase's.
    constexpr bool solo = NBUF == 8;
    constexpr uint32_t nbuf = NBUF, buf_cols = NBUF == 3 ? 160 : 512 / NBUF;
    constexpr int GN = NBUF == 2 ? 64 : NBUF == 4 ? 32 : 48;   // a warp's columns, at most
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
        for (int b = 0; b < MAXBUF; ++b) { mbar_init(&tfull[b], 1); mbar_init(&tempty[b], 2 * (solo ? 4 : EPI_WARPS)); }
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
        split_tile_coords(t, x, mt, nt);
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
            // both CTAs learn of the other's count (compared behind the cluster barrier below)
            issued[rank] = it;
            store_cluster(map_to_rank(const_cast<uint32_t *>(issued) + rank, rank ^ 1), it);
            // drain: wait for the loads still in flight, of both CTAs (at most one per stage)
            if (rank == 0) {
                const uint32_t first = it > (uint32_t)STAGES ? it - STAGES : 0;
                for (uint32_t j = first; j < it; ++j) {
                    const uint32_t s = j % STAGES, round = j / STAGES;
                    mbar_wait(&full[s], round & 1, tmo, nullptr);
                }
            }
        }
    } else if (warp == 1) {
        if (rank == 0) {
            // ---------------- MMA issuer (the whole warp; one lane issues) ----------------
            const uint32_t idesc = idesc_f16_f32(2 * BM, x.bn);
            const uint32_t b_plane = x.bn / 2 * (BK * 2);
            uint32_t it = 0, ch = 0;   // stages and chunks so far
            bool ok = true;
            for (uint32_t t = pair; t < x.items && ok; t += n_pairs) {
                uint32_t c0, c1;
                kslice(t, c0, c1);
                for (uint32_t c = c0; c < c1; ++c, ++it) {
                    const uint32_t s = it % STAGES, round = it / STAGES;
                    ok = __all_sync(0xffffffffu, mbar_wait(&full[s], round & 1, tmo, abort_flag));
                    if (!ok) { if (lane == 0) fail(); break; }
                    const uint32_t sa = smem_u32(stage_base + s * STAGE_BYTES), sb = sa + A_STAGE;
                    const int k_steps = (int)(min(p.K - c * BK, (uint32_t)BK) + 15) / 16;
                    ok = x.chunk_steps == 4 ? mma_stage<4, nbuf>(k_steps, sa, sb, b_plane, idesc, tmem_base, ch, tfull, tempty, tmo, abort_flag)
                                            : mma_stage<2, nbuf>(k_steps, sa, sb, b_plane, idesc, tmem_base, ch, tfull, tempty, tmo, abort_flag);
                    if (!ok) { if (lane == 0) fail(); break; }
                    if (elect_one()) mma_commit_pair(&empty[s]);   // the stage is free in both CTAs once read
                    __syncwarp();
                }
            }
            // make sure no MMA is still writing tensor memory before it is freed
            if (elect_one()) mma_commit_pair(mma_done);
            __syncwarp();
            mbar_wait(mma_done, 0, tmo, nullptr);
        }
    }
    } else {
        regs_up<160>();
        // ---------------- epilogue (warps 4..15) ----------------
        const int quad = warp & 3;                  // tensor-memory lanes 32*quad .. 32*quad+31
        const uint32_t grp = (uint32_t)(warp - 4) >> 2;
        const uint32_t gn = solo ? x.bn : x.bn / 3, g0 = solo ? 0 : grp * gn;   // columns g0 .. g0 + gn - 1
        const int meet = solo ? 128 : 32 * EPI_WARPS;                          // threads that share a tile
        const int et = solo ? (int)(threadIdx.x & 127) : (int)threadIdx.x - 128;
        int64_t *cols = c_col + (solo ? grp * 128 : 0);                        // two tiles' column offsets
        const uint32_t cols_half = solo ? 64 : BN;
        const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
        const int e_sum = half_exponent<TOut>(scale_exponent<TOut>(x.scale_a)) +
                          half_exponent<TOut>(scale_exponent<TOut>(x.scale_b));
        // 2^(eA+eB-28) in two factors: the sums carry 2^28 more than the result's scale
        constexpr float kShift = 1.0f / (float)(1 << (2 * kHalfShift));
        const uint32_t tempty0 = map_to_rank(tempty, 0);
        const double scale = ldexp(p.alpha, e_sum);
        const TOut sc = (TOut)scale;
        const bool plain = p.beta == 0.0;
        float *turn = reinterpret_cast<float *>(smem + STAGES * STAGE_BYTES + 2 * BN * 8 + 256) + (warp - 4) * (TURN / 4);
        uint32_t ch = 0;     // chunks so far
        uint32_t cb = 0;     // this tile's half of c_col
        const uint32_t per_stage = BK / 16 / x.chunk_steps;
        bool dead = false;   // once set, the warp keeps pace with the barriers but does no work
        TOut *C = reinterpret_cast<TOut *>(p.C);
        uint32_t turn_of = 0;   // the group whose turn the item is (narrow tiles)
        for (uint32_t t = pair; t < x.items; t += n_pairs) {
            uint32_t mt, nt, c0, c1;
            const uint32_t ks = kslice(t, c0, c1);
            const uint32_t n_ch = split_chunk_count(c0, c1, per_stage, p.K);
            const bool mine = !solo || turn_of == grp;
            turn_of = turn_of == 2 ? 0 : turn_of + 1;
            if (!mine) {
                ch += n_ch;
                continue;
            }
            tile_coords(t, mt, nt);
            int64_t c_row = 0;
            if constexpr (!KSPLIT) {
                // offsets of this tile's columns in C, in the half that no warp still reads (all
                // epilogue warps meet here, so the half's last readers are two tiles back), and of
                // this thread's row
                cb ^= 1;
                int64_t o0 = 0, o1 = 0;
                if ((uint32_t)et < x.bn && nt * x.bn + et < p.N) radix_offsets(p.nb, nt * x.bn + et, o0, o1);
                if (et < (int)cols_half) cols[cb * cols_half + et] = o1;
                const uint32_t mr = mt * (2 * BM) + rank * BM + quad * 32 + lane;
                if (mr < p.M) radix_offsets(p.ma, mr, o0, c_row);
                named_bar_sync(solo ? 1 + (int)grp : 1, meet);   // ids 1..3
            }
            // two levels of sums, two columns per register pair: T over x.group chunks, S over the groups
            uint64_t T[GN / 2], S[GN / 2];
#pragma unroll
            for (int c16 = 0; c16 < GN / 16; ++c16)   // a narrow tile works on the columns that it has
                if ((uint32_t)c16 * 16 < gn) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) T[c16 * 8 + q] = S[c16 * 8 + q] = 0;
                }
            uint32_t left = x.group;
            for (uint32_t c = 0; c < n_ch; ++c, ++ch) {
                if (dead) continue;
                const uint32_t buf = ch % nbuf;
                bool ok = mbar_wait(&tfull[buf], (ch / nbuf) & 1, tmo, abort_flag);
                ok = __all_sync(0xffffffffu, ok);   // warp-uniform before the .sync.aligned loads
                if (!ok) { if (lane == 0) fail(); dead = true; continue; }
                tc_fence_after();
                const uint32_t src = tmem_base + lane_base + buf * buf_cols + g0;
                if constexpr (GN == 32) {   // both loads, then one wait: the registers allow it here
                    uint32_t r[32];
                    tmem_ld16(src, *reinterpret_cast<uint32_t(*)[16]>(&r[0]));
                    if (gn > 16) tmem_ld16(src + 16, *reinterpret_cast<uint32_t(*)[16]>(&r[16]));
                    tmem_ld_wait();
#pragma unroll
                    for (int q = 0; q < 16; ++q)
                        if (q < 8 || gn > 16) T[q] = f32x2_add(T[q], f32x2_pack(r[2 * q], r[2 * q + 1]));
                } else {
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
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(tempty0 + buf * 8);
                if (--left == 0 || c + 1 == n_ch) {
                    left = x.group;
#pragma unroll
                    for (int c16 = 0; c16 < GN / 16; ++c16)
                        if ((uint32_t)c16 * 16 < gn) {
#pragma unroll
                            for (int j = c16 * 8; j < c16 * 8 + 8; ++j) {
                                S[j] = f32x2_add(S[j], T[j]);
                                T[j] = 0;
                            }
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
            if constexpr (KSPLIT) {   // K slice partial: the sums to the tile's slot, row fastest (coalesced)
                if (m < p.M) {
                    float *P = x.partial + ((((size_t)ks * tiles + t % tiles) * 2 + rank) * x.bn + g0) * BM + ml;
#pragma unroll
                    for (int j = 0; j < GN; ++j)
                        if (j < n_here && dbg_ok(x.dbg_p, P + (size_t)j * BM, 4, p.status))
                            P[(size_t)j * BM] = result(j);
                }
            } else if (x.n_fast) {
                // through shared memory, 16 columns at a time, so that sixteen lanes store one row's
                // columns (64-byte runs): along the rows each store would touch 32 sectors
                                const int64_t *cc = cols + cb * cols_half + g0;
                const int m_here = (int)min(32u, p.M > m - lane ? p.M - (m - lane) : 0u);   // the warp's rows inside C
#pragma unroll
                for (int c16 = 0; c16 < GN / 16; ++c16) {
                    if (c16 * 16 < n_here) {   // uniform over the warp
                        __syncwarp();
#pragma unroll
                        for (int j = 0; j < 16; ++j) turn[lane * 17 + j] = result(c16 * 16 + j);
                        __syncwarp();
                        const int col = lane & 15;
                        const bool in_n = c16 * 16 + col < n_here;
                        TOut *at = C + cc[c16 * 16 + col];
                        // two loops: FP64 conversions on the += path must not be computed for the plain one
                        if (plain) {
#pragma unroll 4
                            for (int r = lane >> 4; r < 32; r += 2) {
                                TOut *dst = at + __shfl_sync(0xffffffffu, c_row, r);
                                if (r < m_here && in_n && dbg_ok(p.dbg_c, dst, (int)sizeof(TOut), p.status))
                                    *dst = sc * (TOut)turn[r * 17 + col];
                            }
                        } else {
#pragma unroll 1
                            for (int r = lane >> 4; r < 32; r += 2) {
                                TOut *dst = at + __shfl_sync(0xffffffffu, c_row, r);
                                if (r < m_here && in_n && dbg_ok(p.dbg_c, dst, (int)sizeof(TOut), p.status))
                                    *dst = (TOut)(scale * (double)turn[r * 17 + col] + p.beta * (double)*dst);
                            }
                        }
                    }
                }
            } else if (m < p.M) {
                TOut *row = C + c_row;
                const int64_t *cc = cols + cb * cols_half + g0;
                if (plain) {
#pragma unroll
                    for (int c16 = 0; c16 < GN / 16; ++c16)
                        if (c16 * 16 < n_here) {
#pragma unroll
                            for (int j = c16 * 16; j < c16 * 16 + 16; ++j)
                                if (j < n_here && dbg_ok(p.dbg_c, row + cc[j], (int)sizeof(TOut), p.status))
                                    row[cc[j]] = sc * (TOut)result(j);
                        }
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
    // the commits signal CTA 1's barriers too; it stays until the last of them has (one thread: the whole warp's
    // wait made the 192-column tiles 1 % slower)
    if (rank == 1 && threadIdx.x == 32) mbar_wait(mma_done, 0, tmo, nullptr);
    __syncwarp();
    cluster_sync();   // neither CTA frees its tensor memory or leaves while the other may still use it
    if (issued[1] > issued[0]) {
        // After a wait that ran out CTA 1 may have loaded a stage more than CTA 0: those loads complete
        // on CTA 0's barrier, which nobody has armed for them, and CTA 1 must not leave before they do.
        if (rank == 0 && threadIdx.x == 0)
            for (uint32_t j = issued[0]; j < issued[1]; ++j) {
                mbar_arrive_expect_tx(&full[j % STAGES], stage_bytes);
                mbar_wait(&full[j % STAGES], (j / STAGES) & 1, tmo, nullptr);
            }
        __syncwarp();
        __syncthreads();
        cluster_sync();
    }
    tc_fence_after();
    if (warp == 1) tmem_dealloc_pair(tmem_base, TMEM_COLS);
}

// K-slice partials -> C: C[m, n] = alpha 2^(eA+eB) sum_ks P[ks][tile][CTA][n][m] (+ beta C), through
// C's strides.  The operands' scale comes in here, with alpha, and not into the FP32 partials, whose range it
// may leave (FP64 operands, or an alpha that brings the result back).
// A block takes 24 columns of one CTA's 128 rows: a thread keeps one row (its offset
// is worked out once) and walks 12 columns, whose offsets the block tabulates, so reads and stores
// run along the rows.  The slices are added with an exact error term (two-sum) in FP32: FP64 adds
// run at 1/64 of that rate here (39 us of 163 on a 1633^3 contraction with two slices).
template <typename TOut>
__global__ void __launch_bounds__(256) split_reduce_kernel(const GemmParams p, const SplitArgs x) {
    using namespace split;
    __shared__ int64_t c_col[STRIP];
    __shared__ int s_exp;
    const uint32_t strips = x.bn / STRIP;
    const uint32_t strip = blockIdx.x % strips, cta = blockIdx.x / strips, tile = cta >> 1, rank = cta & 1;
    uint32_t mt, nt;
    split_tile_coords(tile, x, mt, nt);
    const uint32_t ml = threadIdx.x & 127, m = mt * (2 * BM) + rank * BM + ml, n0 = nt * x.bn + strip * STRIP;
    if (threadIdx.x < STRIP && n0 + threadIdx.x < p.N) {
        int64_t o0, o1;
        radix_offsets(p.nb, n0 + threadIdx.x, o0, o1);
        c_col[threadIdx.x] = o1;
    }
    int64_t r0 = 0, c_row = 0;
    if (m < p.M) radix_offsets(p.ma, m, r0, c_row);
    // (before the wait: the GEMM in front let this kernel begin after its own wait for the pre-passes, whose words
    // these are; looked up after it they cost another 0.3 us)
    if (threadIdx.x == 0)
        s_exp = half_exponent<TOut>(scale_exponent<TOut>(x.scale_a)) + half_exponent<TOut>(scale_exponent<TOut>(x.scale_b));
    pdl_wait();
    __syncthreads();
    if (m >= p.M) return;
    const int e_sum = s_exp;
    const size_t slice = (size_t)x.m_tiles * x.n_tiles * 2 * x.bn * BM;
    const float *P = x.partial + ((size_t)cta * x.bn + strip * STRIP) * BM + ml;
    // Four columns at a time, so that their loads are in flight together (those of columns beyond N too, whose
    // slots hold nothing and are not stored): one after the other, the few blocks of a small result wait for
    // memory (a whole 256 x 256 x 1024 contraction, eight slices: 22.0 us, now 15.9)
    constexpr int U = 4;
    static_assert(STRIP % (2 * U) == 0, "a thread's columns in whole groups");
    auto each = [&](auto &&store) {   // store(element of C, sum, its error)
        for (uint32_t j0 = threadIdx.x >> 7; j0 < STRIP; j0 += 2 * U) {
            float s[U] = {}, lo[U] = {};
#pragma unroll 4
            for (uint32_t k = 0; k < x.ksplit; ++k) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const float *q = P + k * slice + (size_t)(j0 + 2 * u) * BM;
                    if (!dbg_ok(x.dbg_p, q, 4, p.status)) continue;
                    const float v = *q, t = s[u] + v, z = t - s[u];
                    lo[u] += (s[u] - (t - z)) + (v - z);
                    s[u] = t;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (n0 + j0 + 2 * u >= p.N) break;
                TOut *c = reinterpret_cast<TOut *>(p.C) + c_row + c_col[j0 + 2 * u];
                // (the error term of an infinite sum is not a number)
                if (dbg_ok(p.dbg_c, c, (int)sizeof(TOut), p.status)) store(c, s[u], fabsf(s[u]) < INFINITY ? lo[u] : 0.0f);
            }
        }
    };
    if (sizeof(TOut) == 4 && p.alpha == 1.0 && p.beta == 0.0 && e_sum >= -126 && e_sum <= 127) {
        // plain FP32 results: one product with a normal power of two
        const float sc = __int_as_float((e_sum + 127) << 23);
        each([&](TOut *c, float s, float lo) { *c = (TOut)(sc * (s + lo)); });
    } else {
        const double scale = ldexp(p.alpha, e_sum);
        each([&](TOut *c, float s, float lo) {
            const double r = scale * ((double)s + (double)lo);
            *c = (TOut)(p.beta != 0.0 ? r + p.beta * (double)*c : r);
        });
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
template <typename TOut, bool KSPLIT, int NBUF>
static void launch_split_kernel(const CUtensorMap &ta, const CUtensorMap &tb, const GemmParams &p,
                                const SplitArgs &x, int ctas, cudaStream_t s) {
    static const bool attr = [] {
        cudaFuncSetAttribute(gemm_split_kernel<TOut, KSPLIT, NBUF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             split::SMEM_BYTES);
        return true;
    }();
    (void)attr;
    launch_pdl(gemm_split_kernel<TOut, KSPLIT, NBUF>, ctas, split::THREADS, split::SMEM_BYTES, s, ta, tb, p, x);
}

cudaError_t launch_gemm_split(const GemmParams &p, const void *parts_a, const void *parts_b,
                              int64_t kpad, const void *scale_a, const void *scale_b,
                              int64_t kc, int out_bytes, int debug_flags, cudaStream_t s,
                              uint32_t want_ksplit, float *partial, int64_t partial_bytes) {
    using namespace split;
    if (p.M == 0 || p.N == 0) return cudaSuccess;
    const uint32_t pairs = (uint32_t)std::max(1, sm_count() / 2);
    const SplitSchedule sch = split_schedule(p.M, p.N, p.K, pairs, want_ksplit, partial ? partial_bytes : 0, kc);
    CUtensorMap ta, tb;
    if (!make_map(&ta, parts_a, p.M, p.K, (uint64_t)kpad, BM)) return cudaErrorInvalidValue;
    if (!make_map(&tb, parts_b, p.N, p.K, (uint64_t)kpad, sch.bn / 2)) return cudaErrorInvalidValue;
    SplitArgs x;
    x.m_tiles = (p.M + kSplitBM - 1) / kSplitBM;
    x.n_tiles = (p.N + sch.bn - 1) / sch.bn;
    x.fd_band = make_fastdiv(8 * x.n_tiles);
    x.fd_last = make_fastdiv(x.m_tiles % 8 ? x.m_tiles % 8 : 8);
    x.bn = sch.bn;
    x.nch = (p.K + BK - 1) / BK;
    x.ksplit = sch.ksplit;
    x.kslice_chunks = (x.nch + sch.ksplit - 1) / sch.ksplit;
    x.items = x.m_tiles * x.n_tiles * x.ksplit;
    split_chunks(x.kslice_chunks, kc, &x.chunk_steps, &x.group);
    x.partial = partial;
    x.dbg_p = dbg_range(partial, split_partial_bytes(p.M, p.N, sch));
    // along columns where the N group's first label is C's stride-1 label (and the M group's is not)
    x.n_fast = p.nb.n > 0 && p.nb.s1[0] == 1 && p.nb.ext[0] > 1 && !(p.ma.n > 0 && p.ma.s1[0] == 1 && p.ma.ext[0] > 1);
    x.debug_flags = debug_flags;
    x.scale_a = scale_a;
    x.scale_b = scale_b;
    const int ctas = 2 * (int)std::min(pairs, x.items);
    const bool solo = x.bn == 48 && x.ksplit == 1 && split_chunks_of(x.nch, x.chunk_steps, p.K) <= 3;
    const int nbuf = solo ? 8 : x.bn <= 128 ? 4 : x.bn <= 160 ? 3 : 2;
#define CM_SPLIT(T, K, B) launch_split_kernel<T, K, B>(ta, tb, p, x, ctas, s)
#define CM_SPLIT_T(T)                                                                   \
    do {                                                                                \
        if (x.ksplit > 1) nbuf == 4 ? CM_SPLIT(T, true, 4) : nbuf == 3 ? CM_SPLIT(T, true, 3) : CM_SPLIT(T, true, 2); \
        else if (solo) CM_SPLIT(T, false, 8);                                           \
        else nbuf == 4 ? CM_SPLIT(T, false, 4) : nbuf == 3 ? CM_SPLIT(T, false, 3) : CM_SPLIT(T, false, 2); \
    } while (0)
    if (out_bytes == 8) CM_SPLIT_T(double);
    else CM_SPLIT_T(float);
#undef CM_SPLIT_T
#undef CM_SPLIT
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || x.ksplit == 1) return e;
    const uint32_t blocks = x.m_tiles * x.n_tiles * 2 * (x.bn / STRIP);
    if (out_bytes == 8) launch_pdl(split_reduce_kernel<double>, blocks, 256, 0, s, p, x);
    else launch_pdl(split_reduce_kernel<float>, blocks, 256, 0, s, p, x);
    return cudaGetLastError();
}

}  // namespace comet
