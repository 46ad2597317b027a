// How the pair kernels cut their sources into slices of partial sums (far.cu). Plain C++ (no
// CUDA): the host tests compile it on its own.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

namespace pb {

constexpr int TPB64 = 128;  // threads (= targets) per CTA of the one-direction FP64 kernel
constexpr int TS64 = 64;    // its sources per shared-memory tile

// Slices of nacc sums of `size` bytes a point that `cap` bytes hold (at least one); cap 0: any.
inline int capped_slices(double cap, int64_t np, int nacc, int size) {
    return cap > 0.0 ? (int)std::max(1.0, std::min(64.0, std::floor(cap / ((double)nacc * size * (double)np)))) : 64;
}

// split count of the scalar and one-direction FP64 kernels: fill the GPU in whole waves
inline int choose_splits(int64_t np, int tpc, int tile, int slots, int most = 32) {
    int64_t nb = (np + tpc - 1) / tpc;
    int64_t ntiles = (np + tile - 1) / tile;
    int best = 1;
    double best_cost = 1e300;
    for (int S = 1; S <= std::min(most, 32); ++S) {
        if (S > ntiles) break;
        int64_t ctas = nb * S;
        int64_t waves = (ctas + slots - 1) / slots;
        int64_t per = (ntiles + S - 1) / S;
        double cost = (double)waves * (double)per * (1.0 + 0.01 * S);
        if (cost < best_cost) { best_cost = cost; best = S; }
    }
    return best;
}

// Sources of a slice of the packed kernel's fast variant at most: their sums stay in FP32 until the
// slices are added in FP64, so longer slices cost accuracy (twice as long: 43,320 points, V/K rows 1.3
// instead of 1.1e-7 from the FP64 application). The length, in whole tiles of ts records, is that of
// whole waves of 1,024 targets a CTA, 4 (V/K rows) or 2 CTAs resident on an SM. The split-coordinate
// variant adds every tile's sums to wide ones: any length.
inline int64_t x2_longest(int64_t np, int mode, int ts, int num_sms) {
    const int S = choose_splits(np, 1024, ts, (mode == 0 ? 4 : 2) * num_sms);
    return ((np + S - 1) / S + ts - 1) / ts * ts;
}

// Split count of the packed kernel, tiles with room for ts records (whole threes are used), no more
// than `longest` sources to a slice (0: any): an SM's pair rate hardly depends on how many CTAs
// share it (one alone 5 % less, measured), so the time goes with the most CTAs that one SM gets times
// their tiles; more slices cost the reduction, 0.2 % each. (By whole waves of resident CTAs, with 1 % a
// slice, a part of the SMs had stood idle: 58,080 points, V/K + D/T rows 3,750 -> 3,510 us, split V/K
// rows 3,050 -> 2,810 us at the counts chosen here.)
constexpr int X2_MAX_SLICES = 36;  // 32 of the longest slices in tiles of fewer points than ts
inline int x2_splits(int64_t np, int tpc, int ts, int num_sms, int64_t longest = 0, int most = 64,
                     double* cost_out = nullptr) {
    const int tile = ts / 3 * 3;
    const int64_t nb = (np + tpc - 1) / tpc, ntiles = (np + tile - 1) / tile;
    const int64_t per_max = longest > 0 ? std::max<int64_t>(1, (longest + tile / 2) / tile) : ntiles;  // to the nearest tile
    int best = (int)std::min<int64_t>(std::min(most, X2_MAX_SLICES), ntiles);  // as short as they can be
    double best_cost = 1e300;
    for (int S = 1; S <= std::min(most, longest > 0 ? X2_MAX_SLICES : 32) && S <= ntiles; ++S) {
        const int64_t deep = (nb * S + num_sms - 1) / num_sms, per = (ntiles + S - 1) / S;
        if (per > per_max) continue;
        const double cost = (double)(deep * per) * (1.0 + 0.05 / (double)deep) * (1.0 + 0.002 * S);
        if (cost < best_cost) { best_cost = cost; best = S; }
    }
    if (cost_out) *cost_out = best_cost * tpc * tile;
    return best;
}

// Untuned launch shape of the fast variant: 0 (1,024 targets a CTA) or, below 16,384 points, 3 (512,
// one packed pair a thread), whose CTAs share out more evenly what bounded slices leave of a small
// surface. V/K + D/T rows, us, 1,024 | 512 targets: 3,000 points 75 | 63, 5,880: 117 | 100, 9,720: 171 | 150, 14,520:
// 280 | 261. V/K rows take a tenth longer a pair with 512 and do so only where the busiest SM has that
// much less to do: 5,880: 80 | 73, 9,720: 134 | 112, but 7,680: 94 | 98, 12,000: 155 | 162.
constexpr int X2_SMALL_CTAS = 3;
inline int x2_fast_shape(int64_t np, int mode, int num_sms, int most = 64) {
    if (np >= 16384) return 0;
    if (mode == 1) return X2_SMALL_CTAS;
    const int64_t longest = x2_longest(np, mode, 64, num_sms);
    double large, small;
    x2_splits(np, 1024, 64, num_sms, longest, most, &large);
    x2_splits(np, 512, 64, num_sms, longest, most, &small);
    return 1.1 * small < 0.97 * large ? X2_SMALL_CTAS : 0;
}

// split count after the tuned scale, within [1, tiles] and <= 32 (or the untuned one) and <= most
inline int scaled_splits(int S, double scale, int64_t np, int tile, int most = 64) {
    const int64_t ntiles = (np + tile - 1) / tile;
    int s2 = (int)(S * scale + 0.5);
    s2 = std::max(1, std::min({s2, std::max(S, 32), most}));
    return (int)std::min<int64_t>(s2, ntiles);
}

// ------------------------------------------------------------- FP64 kernels
// Shape of the both-directions kernel; nblock = 0: the one-direction kernel runs.
struct Sym64 {
    int warps, sub;        // W and SB
    int nblock, half;      // I blocks, and the largest distance
    int nsplit;
    int slices() const { return nsplit + half; }
};

// FP64 instructions of a pair of points, both directions, by row mode and kind (the kernels'
// KIND; V/K rows: 1 no Yukawa term, 0 otherwise)
inline double pair64_instr(int mode, int kind, bool both) {
    static const double one[2][3] = {{68.0, 36.0, 68.0}, {100.0, 48.0, 92.0}};
    static const double two[2][3] = {{41.0, 22.0, 41.0}, {65.0, 37.0, 61.0}};
    return (both ? two : one)[mode ? 1 : 0][kind];
}

// The launch of an FP64 application of np points.
struct Pair64Plan {
    Sym64 sym;      // nblock > 0: both directions at once
    int nsplit;     // one direction: slices
    int64_t chunk;  // and their sources
    double cost;    // FP64 instructions of the busiest SM, in units of a 32 x 32 tile's instruction
    int slices() const { return sym.nblock ? sym.slices() : nsplit; }
};

// The FP64 pipe, not the number of resident warps, sets an SM's rate, down to about six warps; the
// cost of a launch is that of the SM with the most work.
inline double few_warps(double resident) { return resident < 6.0 ? 6.0 / resident : 1.0; }

// One direction at a time, by whole waves of `slots` resident CTAs.
inline Pair64Plan pair64_one(int64_t np, int mode, int kind, int num_sms, int slots, double cap = 0.0) {
    Pair64Plan p = {{0, 0, 0, 0, 0}, 1, 0, 0.0};
    p.nsplit = choose_splits(np, TPB64, TS64, slots, capped_slices(cap, np, mode == 0 ? 2 : 10, 8));
    p.chunk = ((np + p.nsplit - 1) / p.nsplit + TS64 - 1) / TS64 * TS64;
    p.nsplit = (int)((np + p.chunk - 1) / p.chunk);
    const int64_t ctas = (np + TPB64 - 1) / TPB64 * p.nsplit, on_sm = (ctas + num_sms - 1) / num_sms;
    p.cost = (double)on_sm * (TPB64 / 32) * (double)(p.chunk / 32) * few_warps((double)ctas / num_sms * (TPB64 / 32)) *
             0.5 * pair64_instr(mode, kind, false) * (1.0 + 0.002 * p.nsplit);
    return p;
}

// Both directions at once: the shape whose busiest SM has the least work. The partial sums stay within 32 slices, or 64 while they are
// below 32 MB; a block has 1,024 points at most, so 63 blocks (64,512 points) are the most.
inline Pair64Plan pair64_both(int64_t np, int mode, int kind, int num_sms, double cap = 0.0) {
    static const int shapes[5][2] = {{2, 1}, {4, 1}, {8, 1}, {8, 2}, {8, 4}};
    const int nacc = mode == 0 ? 2 : 10, most = capped_slices(cap, np, nacc, 8);
    Pair64Plan best = {{0, 0, 0, 0, 0}, 0, 0, 1e300};
    for (const auto& sh : shapes) {
        Sym64 c;
        c.warps = sh[0];
        c.sub = sh[1];
        const int64_t pts = 32 * c.warps * c.sub, nb = (np + pts - 1) / pts;
        if (nb > 64) continue;
        c.nblock = (int)nb;
        c.half = c.nblock / 2;
        const int units = (c.half + 1) * c.warps * c.sub;
        for (c.nsplit = 1; c.nsplit <= units && c.slices() <= most; ++c.nsplit) {
            if (c.slices() > 32 && (double)c.slices() * nacc * np * 8.0 > 32e6) break;
            const int64_t ctas = nb * c.nsplit, per = (units + c.nsplit - 1) / c.nsplit;
            const int64_t on_sm = (ctas + num_sms - 1) / num_sms;
            const double resident = std::min<double>((double)ctas / num_sms, 16.0 / c.warps) * c.warps;
            const double cost = (double)on_sm * per * c.sub * c.warps * few_warps(resident) *
                                (1.0 + 0.002 * c.slices()) * pair64_instr(mode, kind, true);
            if (cost < best.cost) {
                best.cost = cost;
                best.sym = c;
            }
        }
    }
    return best;
}

// The cheaper of the two: both directions at once takes about 0.63 of the instructions, but its
// slices leave too few CTAs for the GPU's SMs as the blocks approach 63 (from 62,465 points on one
// block of rows an SM and 41 % of the FP64 pipe: 63,480 points, V/K + D/T rows 551 ms, one direction at a time
// 340; V/K rows 376 and 250).
// cap: bytes that the partial sums may take (0: any).
inline Pair64Plan pair64_plan(int64_t np, int mode, int kind, int num_sms, int slots, double cap = 0.0) {
    const Pair64Plan both = pair64_both(np, mode, kind, num_sms, cap);
    const Pair64Plan one = pair64_one(np, mode, kind, num_sms, slots, cap);
    return both.sym.nblock && both.cost <= one.cost ? both : one;
}

// ------------------------------------------------------- a request's partial sums
// Bytes of the direct applications' partial sums of a served request, any operator: as the rules
// above would have it, and the least that they are held to where a budget does not allow that (whole
// waves of the packed kernel's CTAs, in FP64).
inline double part_bytes(int64_t np, int num_sms, bool mixed) {
    double b = 0.0;
    for (int mode = 0; mode < 2; ++mode) {
        const double sum = (double)np * (mode == 0 ? 2 : 10);
        if (mixed) {
            b = std::max(b, 8.0 * sum * x2_splits(np, 512, 64, num_sms));
            b = std::max(b, 4.0 * sum * x2_splits(np, 1024, 64, num_sms, x2_longest(np, mode, 64, num_sms)));
        } else {
            for (int kind = 0; kind < (mode == 0 ? 2 : 3); ++kind)
                b = std::max(b, 8.0 * sum * pair64_plan(np, mode, kind, num_sms, 6 * num_sms).slices());
        }
    }
    return b;
}
inline double least_part_bytes(int64_t np, int num_sms) {
    return 80.0 * (double)np *
           std::max(choose_splits(np, 512, 64, 2 * num_sms), choose_splits(np, 1024, 64, 2 * num_sms));
}

}  // namespace pb
