// Backtrack, DBA averaging and barycenter initialisation kernels.
#pragma once

#include <algorithm>

#include "plan.cuh"
#include "wts_common.cuh"

namespace wts {

struct BTParams {
    const PairDesc* pairs;
    int P;
    int R;
    const uint32_t* dirs;
    int32_t* jlo;        // [P][M] indexed by PairDesc::out
    int32_t* jhi;
    int32_t* plen;       // [P] (may be null)
    int64_t M;           // row stride of jlo/jhi
    // codes available for bands [band_lo, band_hi) only (band b at dirs offset
    // b - band_lo): the walk covers their rows.  state[q] = the column at which
    // the path of pair q enters the row below them (-1: the walk failed),
    // written after one group of bands and read by the next one down
    // (null: all bands at once).
    int band_lo, band_hi;
    int32_t* state;
    int first;           // 1: start every walk at (M-1, N-1), else at state
    // Sub-DTW (Sec. 3.2): start at (M-1, bstar[out]) and stop when the walk
    // leaves row 0 (the free start), writing that column to astar[out]
    int subseq;
    const int32_t* bstar;
    int32_t* astar;
    // segmented walk (not Sub-DTW): the rows are cut into nseg segments of
    // seg_rows rows.  The first launch walks them all at once, each from a guessed
    // cell lead_rows above its top (a walk off the path joins it on the way down);
    // the second (join) takes a pair's segments from the top down and
    // walks those again that the path enters elsewhere.  seg[(q * nseg + k) * 4 + ..] =
    // {start column, exit column, unused, status (1 = the codes were invalid or a
    // wait gave up)}; the exit is the path's column in the row below the segment.
    int nseg, seg_rows, lead_rows, join;
    int32_t* seg;
    // the call's workspace header: a raised abort word (set with the status
    // when the DP left early) makes the walk do nothing (may be null)
    const WsHeader* hdr;
};

// Rows above a segment's top at which its walk starts, off the path: it joins the
// path after about as many rows as it starts columns away, and the line from the
// path's entry to the origin stays within a tenth of the rows or so (smooth
// six-channel cycles of 25,000: entered on the path after 256 / 512 / 1,024 / 2,048
// rows in 5 / 10 / 20 / 28 of 28 segments).  Stage in us, rows above 0 / 128 / 256 /
// 512 / 1,024: 16 of 1.1k, segments of 128: 142 / 82 / 74 / 105 / -; 24 of 8.2k, of 256:
// 660 / 554 / 501 / 251 / 174; 60 of 25k, of 1,280, rows above 1,536 / 2,048 / 2,560 /
// 3,072: 976 / 641 / 704 / 766.
constexpr int kBtResident = 152 * 12;     // walks resident at once (two per block of 33 KB)
inline int bt_lead_rows(int64_t M)
{
    return (int)std::min<int64_t>(4096, std::max<int64_t>(192, cdiv(M, 10 * 128) * 128));
}
// Rows per segment: as many segments as there are warps resident (200 pairs of
// 25,000 rows, segments of 2,048 / 2,560 / 3,200 / 4,096: 1.23 / 1.17 / 1.06 / 1.13 ms),
// but a quarter of the rows above at least (those are walked twice).  All rows where
// a segment and the rows above it are no shorter.
inline int bt_seg_rows(int64_t rows, int P, int lead)
{
    const int64_t nseg = std::max<int64_t>(1, kBtResident / P);
    const int64_t s = std::max(cdiv(cdiv(rows, nseg), 128) * 128, cdiv(lead, 4 * 128) * 128);
    return (int)(s + lead + 64 >= rows ? rows : s);
}

cudaError_t launch_backtrack(const BTParams& p, cudaStream_t st);
// After the two launches of a segmented walk: state, and once the first row is
// walked |pi| = sum_i (jhi(i) - jlo(i) + 1) per pair, or -1 if a segment failed
// or the segments do not join up.
cudaError_t launch_backtrack_seg_final(const BTParams& p, cudaStream_t st);

// B_out[i] = mean of the cycle samples aligned to row i over all cycles;
// counts[i] = number of aligned samples; cost_before = sum_k costs[k].
cudaError_t launch_dba_average(const float* data, const int64_t* offsets, int T, int d, int64_t M,
                               const int32_t* jlo, const int32_t* jhi, const float* costs,
                               float* B_out, int32_t* counts, double* cost_before, cudaStream_t st);

// score[k] = cost[k] / plen[k] (one FP32 division, Eq. 8); NaN where the walk failed.
cudaError_t launch_score_divide(const float* cost, const int32_t* plen, float* score, int T, cudaStream_t st);

cudaError_t launch_resample(const float* x, int64_t N, int d, float* out, int64_t M, cudaStream_t st);
cudaError_t launch_euclid_mean(const float* data, const int64_t* offsets, int T, int d, int64_t M,
                               float* out, cudaStream_t st);
cudaError_t launch_medoid(const float* C, int T, int32_t* index_out, double* sums_out, cudaStream_t st);

}  // namespace wts
