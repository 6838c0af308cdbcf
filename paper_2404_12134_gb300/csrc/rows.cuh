// Rows per lane of a DTW launch that does not name them.
//
// Few rows make short steps and many bands: best while the warps are few, when
// the latency of a band's chain of steps sets the time.  Many rows spread a
// step's fixed work over more cells: best once the warps fill the schedulers.
// The choice is the smallest of this estimate over the row counts:
//   every warp resident   (N + lag x bands) steps of the longest pair, each as
//               long as the larger of a warp's own latency and what the warps of
//               its scheduler issue
//   more warps  all warp-steps over all schedulers at the issue time of a step,
//               and a third of one pair alone for the start and the last warps
// with the times of a step measured per channel count, row count and what is
// computed: alone on one pair of 16,000 x 16,000, at full issue on 200 cycles
// of 6,000 (cost alone: on their pairwise matrix of 20).  Another count than the
// fixed one (32 up to two channels, else 16) must be estimated 10 % faster, 14 %
// with more warps than are resident.
// Measured, rows 4 / 8 / 16 / 32, wavefront in us (cost + |pi|; d = 6: codes):
//   d = 1,   1 pair  of  1,100   102 /   121 /   168 /   265
//   d = 1,   4 pairs of 24,000  2802 /  2772 /  3938 /  6337
//   d = 1,  48 pairs of 24,000 15201 / 15682 / 11079 /  9550
//   d = 3,  16 pairs of 24,000  6865 /  6938 /  8100 /  9074
//   d = 6,  16 pairs of  3,000   350 /   540 /   753
//   d = 6, 150 pairs of  8,000  8005 /  6934 /  6055
#pragma once

#include <algorithm>
#include <cstdint>

#include "plan.cuh"

namespace wts {

enum RowForm : int { kRowPlen = 0, kRowCodes = 1, kRowCost = 2 };

// ns of a step of a warp alone, and per scheduler at full issue, by RowForm.
struct RowStep {
    short alone[3], full[3];
};
struct RowTable {
    int D;
    RowStep rows[4];     // 4, 8, 16, 32 rows per lane
};

constexpr int kRowCounts[4] = {4, 8, 16, 32};
constexpr int kRowLag[4] = {66, 96, 75, 45};     // steps between a band and the next
constexpr RowTable kRowTable[] = {
    {1, {{{62, 61, 54}, {38, 34, 23}}, {{79, 79, 68}, {68, 64, 37}},
         {{137, 129, 116}, {116, 128, 59}}, {{241, 246, 207}, {208, 224, 194}}}},
    {2, {{{68, 61, 54}, {44, 36, 29}}, {{83, 83, 70}, {71, 73, 48}},
         {{144, 142, 125}, {133, 130, 105}}, {{272, 269, 241}, {245, 257, 239}}}},
    {3, {{{67, 64, 58}, {45, 43, 35}}, {{87, 87, 75}, {82, 80, 62}},
         {{171, 158, 137}, {169, 164, 131}}, {{329, 294, 266}, {318, 314, 228}}}},
    {4, {{{69, 66, 62}, {50, 46, 42}}, {{92, 98, 80}, {89, 94, 78}},
         {{220, 198, 152}, {192, 190, 152}}, {}}},
    {6, {{{75, 72, 66}, {64, 63, 56}}, {{107, 108, 97}, {133, 116, 104}},
         {{203, 201, 199}, {250, 190, 199}}, {}}},
    {8, {{{83, 79, 73}, {80, 81, 74}}, {{139, 136, 121}, {160, 134, 126}},
         {{284, 238, 223}, {254, 240, 262}}, {}}},
    {9, {{{83, 82, 77}, {86, 90, 81}}, {{133, 133, 116}, {155, 146, 146}},
         {{326, 326, 245}, {269, 296, 272}}, {}}},
    {12, {{{97, 96, 88}, {99, 100, 102}}, {{172, 175, 157}, {202, 185, 161}},
         {{603, 584, 497}, {400, 395, 348}}, {}}},
    {16, {{{123, 123, 113}, {130, 133, 139}}, {{210, 216, 197}, {248, 225, 208}},
         {{928, 801, 846}, {697, 565, 580}}, {}}},
};
constexpr double kSchedulers = 4 * 152;

// The launch as the estimate sees it, per row count.
struct RowLoad {
    int64_t steps[4] = {};       // sum over pairs of bands x (N + 31)
    int64_t bands[4] = {};       // sum over pairs
    int64_t longest[4] = {};     // max over pairs of N + 31 + lag x bands

    void add(int64_t M, int64_t N)
    {
        for (int r = 0; r < 4; ++r) {
            const int64_t nb = cdiv(M, 32 * kRowCounts[r]);
            steps[r] += nb * (N + 31);
            bands[r] += nb;
            longest[r] = std::max(longest[r], N + 31 + kRowLag[r] * nb);
        }
    }

    // warps per scheduler resident at once (registers)
    static int resident(int R, int D)
    {
        return R == 4 ? (D <= 8 ? 3 : 2) : R == 8 ? (D <= 4 ? 4 : (D <= 8 ? 3 : 2)) : (R == 16 && D <= 4) ? 3 : 2;
    }

    double estimate(int r, int D, int form) const
    {
        const RowTable* t = kRowTable;
        while (t->D != D) ++t;
        const double alone = t->rows[r].alone[form], full = t->rows[r].full[form];
        const double w = (double)bands[r] / kSchedulers;
        if (w > resident(kRowCounts[r], D))
            return (double)steps[r] / kSchedulers * full + 0.3 * (double)longest[r] * alone;
        // (some schedulers hold one warp more than others)
        const double busy = w <= 1 ? 0 : 0.5 * (w + (double)(int64_t)(w + 0.999));
        return (double)longest[r] * std::max(alone, busy * full);
    }

    // fixed: the row count taken unless another is clearly faster.
    int rows(int D, int form, int fixed) const
    {
        int best = fixed;
        double best_t = 0.9 * estimate(fixed == 32 ? 3 : 2, D, form);
        for (int r = 0; r < 4; ++r) {
            if (kRowCounts[r] == fixed || (kRowCounts[r] == 32 && D > 3)) continue;
            double t = estimate(r, D, form);
            if ((double)bands[r] / kSchedulers > resident(kRowCounts[r], D)) t *= 1.05;
            if (t < best_t) { best = kRowCounts[r]; best_t = t; }
        }
        return best;
    }
};

}  // namespace wts
