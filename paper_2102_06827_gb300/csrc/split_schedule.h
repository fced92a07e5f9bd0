// Tile width and K slicing of the split GEMM, chosen from the GEMM's sizes.  Shared by the
// planner (which sizes the partial sums' workspace) and the launcher.
#pragma once
#include <stdint.h>

#include <algorithm>

namespace comet {

constexpr int kSplitBM = 256;     // output rows per CTA pair
constexpr int kSplitBK = 64;      // K values per shared-memory stage
constexpr int kSplitMaxBN = 192;  // output columns per CTA pair: 48, 96, 144, 192

struct SplitSchedule {
    uint32_t bn = kSplitMaxBN;    // output columns per pair
    uint32_t ksplit = 1;          // K slices per output tile (FP32 partials when above 1)
    double us = 0;                // modelled time
};

// Accumulation of a K slice of `stages` stages: K steps of 16 values per chunk in tensor memory (which
// truncates: short chunks lose less, but each costs a drain) and chunks per first-level sum of
// the epilogue (about the square root of the chunks, so that neither level adds many terms).  kc: the
// caller's upper limit of a chunk's K values (0 = none); 32 is the least there is.
inline void split_chunks(uint32_t stages, int64_t kc, uint32_t *steps, uint32_t *group) {
    // 32 values up to K = 4096 (12 % more of the GEMM's time at 1633^3, error 1.43 -> 1.23e-7), 64 beyond
    // (8.6 against 7.7 ms at 12288^3, where the sums' own rounding is as large)
    *steps = stages <= 64 || (kc > 0 && kc < 64) ? 2 : 4;
    const uint32_t n = stages * (4 / *steps);
    uint32_t g = 1;
    while (g * g < n) ++g;
    *group = g;
}

// bytes of the FP32 partial sums of a schedule
inline int64_t split_partial_bytes(uint64_t M, uint64_t N, const SplitSchedule &s) {
    if (s.ksplit <= 1) return 0;
    const int64_t tiles = (int64_t)((M + kSplitBM - 1) / kSplitBM) * (int64_t)((N + s.bn - 1) / s.bn);
    return tiles * s.ksplit * kSplitBM * s.bn * 4;
}

// Chunks of a whole-K tile: the end of K may leave the second half of its stage empty.
inline uint32_t split_chunks_of(uint32_t stages, uint32_t steps, uint64_t K) {
    const uint32_t n = stages * (4 / steps);
    return steps == 2 && (uint64_t)stages * kSplitBK >= K + kSplitBK / 2 ? n - 1 : n;
}

// The schedule with the least modelled time over the tile widths and K slices whose partial
// sums fit `partial_limit` bytes.  want_ksplit: 0 = free, k = as near to k slices as K allows; kc as above.
// The model, in clocks at 1.9 GHz, from kernel times on 1633^3, 2700^3, 4864 x 960 x 4800, 200000 x 48 x
// (96, 160) and 200000 x 192 x 48 at every width: a stage of 64 K values takes 1300 / 1420 / 1860 / 2150
// (widths 48 / 96 / 144 / 192) in chunks of 32 and 1000 / 1130 / 1320 / 1480 in chunks of 64, a tile 2000 +
// 26 a column around its stages, or 4700 in all for a narrow tile of at most three chunks; 3000 once; K
// slices add a launch and their partial sums' traffic.
inline SplitSchedule split_schedule(uint64_t M, uint64_t N, uint64_t K, uint32_t pairs, uint32_t want_ksplit,
                                    int64_t partial_limit, int64_t kc = 0) {
    static const double stage32[4] = {1300, 1420, 1860, 2150}, stage64[4] = {1000, 1130, 1320, 1480};
    const uint64_t mt = (M + kSplitBM - 1) / kSplitBM;
    const uint32_t nch = (uint32_t)std::max<uint64_t>(1, (K + kSplitBK - 1) / kSplitBK);
    SplitSchedule best;
    bool have = false;
    uint32_t k_lo = want_ksplit ? std::min(want_ksplit, nch) : 1, k_hi = want_ksplit ? k_lo : std::min(16u, nch);
    for (; !have && k_lo > 0; k_hi = --k_lo) {   // once, or down to as many slices as their partial sums may take
        for (uint32_t w = 0; w < 4; ++w) {
            const uint32_t bn = 48 * (w + 1);
            const uint64_t tiles = mt * ((N + bn - 1) / bn);
            for (uint32_t k = k_lo; k <= k_hi; ++k) {
                SplitSchedule s;
                const uint32_t per = (nch + k - 1) / k;
                s.bn = bn;
                s.ksplit = (nch + per - 1) / per;   // every slice holds at least one stage
                const int64_t pb = split_partial_bytes(M, N, s);
                if (pb > partial_limit) continue;
                uint32_t steps, group;
                split_chunks(per, kc, &steps, &group);
                const double waves = (double)((tiles * s.ksplit + pairs - 1) / pairs);
                const bool narrow = w == 0 && s.ksplit == 1 && split_chunks_of(nch, steps, K) <= 3;
                const double tile = narrow ? 4700.0 : per * (steps == 2 ? stage32 : stage64)[w] + 2000.0 + 26.0 * bn;
                s.us = (3000.0 + waves * tile) / 1900.0;
                if (s.ksplit > 1) s.us += 3.0 + (double)pb / 2.0e6;   // written and read back, mostly in L2
                if (!have || s.us < best.us * (1 - 1e-9)) { best = s; have = true; }
            }
        }
    }
    return best;
}

// Modelled time of the same GEMM as one launch on the FP32 pipes (k_gemm_small.cu), at 1.9 GHz: tiles
// of 16 x 16 over 152 SMs, 900 clocks a tile and 22 per K value, or 42 where an operand's contiguous
// runs are short (its 4-byte gathers then take as many cache lines), and 3 us of launch.  Measured:
// 192^3 6.1 us, 300^3 14.4, 1000 x 1000 x 16 18.5; with runs of 8 and 10 values 6.9, 26.4, -.
inline double small_gemm_us(uint64_t M, uint64_t N, uint64_t K, bool long_runs) {
    const uint64_t tiles = ((M + 15) / 16) * ((N + 15) / 16);
    return 3.0 + (double)((tiles + 151) / 152) * (900.0 + (double)K * (long_runs ? 22.0 : 42.0)) / 1900.0;
}

// Whether its grid takes the size: N runs along y (the planner's own forms put the longer side on M)
inline bool small_gemm_fits(uint64_t N) { return (N + 15) / 16 <= 65535; }

// The emulated-FP64 GEMM: whole-K tiles of 128 x 80 in full waves over the SMs, the tiles left over in
// K slices of whole chunks (192 values) whose int64 partial sums a second kernel adds.
constexpr int kEmuBM = 128, kEmuBN = 80, kEmuChunk = 192;

struct EmuSchedule {
    uint32_t full = 0;      // tiles computed whole
    uint32_t tail = 0;      // tiles left over
    uint32_t slices = 1;    // K slices of each of them (1: whole as well)
};

inline int64_t emu_partial_bytes(const EmuSchedule &s) {
    return s.slices > 1 ? (int64_t)s.tail * s.slices * kEmuBM * kEmuBN * 8 : 0;
}

// The slices of the left-over tiles that end soonest, in units of a chunk's time (about 8 us): rounds
// over the SMs times chunks per slice plus 0.4 around each item, plus 0.5 for the second kernel.
// At 1728^3 (308 tiles, nine chunks) the four tiles after two rounds of 152 run in 36 slices on idle SMs
// instead of a third round.  Chunks keep their boundaries and the sums are integers, so slicing
// changes no bit of the result.
inline EmuSchedule emu_schedule(uint64_t M, uint64_t N, uint64_t K, uint32_t sms, int64_t partial_limit) {
    const uint32_t tiles = (uint32_t)(((M + kEmuBM - 1) / kEmuBM) * ((N + kEmuBN - 1) / kEmuBN));
    const uint32_t nch = (uint32_t)std::max<uint64_t>(1, (K + kEmuChunk - 1) / kEmuChunk);
    EmuSchedule s, best;
    s.full = tiles / sms * sms;
    s.tail = tiles - s.full;
    best.full = tiles;
    if (s.tail == 0) return best;
    double least = (double)nch + 0.4;
    for (uint32_t k = 2; k <= std::min(nch, 32u); ++k) {
        const uint32_t per = (nch + k - 1) / k;
        s.slices = (nch + per - 1) / per;
        if (emu_partial_bytes(s) > partial_limit) break;
        const double t = (double)((s.tail * s.slices + sms - 1) / sms) * (per + 0.4) + 0.5;
        if (t < least) { least = t; best = s; }
    }
    return best;
}

}  // namespace comet
