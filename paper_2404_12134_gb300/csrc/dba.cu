// Backtrack of the tie-rule path, DBA averaging, and initial barycenters.
#include "dba.cuh"
#include "walk_window.h"

namespace wts {

namespace {

constexpr int kBtWarps = 2;      // warps per backtrack CTA
constexpr long long kBtSpin = 1ll << 24;
constexpr int kBtBurst = 64;     // rows a second walk takes unchecked between looks for the first

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t phase)
{
    for (long long it = 0; it < kBtSpin; ++it) {
        uint32_t ok;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                     " selp.u32 %0, 1, 0, p;\n}" : "=r"(ok) : "r"(smem_u32(bar)), "r"(phase) : "memory");
        if (ok) return true;
    }
    return false;
}

// Walk the stored predecessor codes back from (M-1, N-1) to (0, 0).
// A cell (i, j) of band b sits in lane t = (i mod BR) / R at step s = j + t,
// as bit R-1-k, k = i mod R ("not diag") and bit 2R-1-k ("not up") of the
// lane's 2R code bits of that step.  For R >= 16 those are the W = R / 16 words at
// dirs[dir_off + b*(N+31)*32*W + (s*32 + t)*W + w]; for R = 8 and 4 the word
// dirs[dir_off + b*band_dir_words(N, R) + (s/S)*32 + t] holds the S = 32/(2R)
// steps S*(s/S) .. of the lane, 2R bits each: R = 8 the earlier step in the
// low half; R = 4 from the top bit down, step by step, row by row,
// "not diag" before "not up".  Along the walk s only decreases inside a
// band, so a window of kBtWords / 32 consecutive word rows (one contiguous
// block of global memory) is brought into shared memory by one bulk
// asynchronous copy (completion on an mbarrier, bounded wait) and the walk
// reads it; every lane walks the same path, and the lanes look ahead along
// runs of equal moves (one vote per run).
// Row i's range is [jlo(i), jhi(i)]: jhi when the walk enters the row, jlo
// when it leaves it (Definition "Alignment path": monotone, so each row's
// columns are contiguous).
// Bound by the walk's chain of dependent instructions (about 5 cycles each, one
// warp per walk): 45 of them per run in the unchecked loop; 16 paths of 1.1k in 9
// segments 70 us (one walk a path 235), 200 of 25k in 9 1.00 ms, 32 of 110k in 14
// checkpointed groups 7.3 ms (22.3), whatever the range arrays hold.
template <int R>
__global__ void __launch_bounds__(32 * kBtWarps) backtrack_kernel(BTParams p)
{
    using Win = WalkWindow<R>;
    constexpr int W = Win::W, SPW = Win::SPW, LOG_R = Win::LOG_R, kBtRows = Win::ROWS;
    __shared__ __align__(128) uint32_t win_all[kBtWarps][kBtWords];
    __shared__ __align__(8) uint64_t bars[kBtWarps];
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    // the call's DP left early (a non-finite sample, or a wait that gave up):
    // its codes and b* were never written, so there is nothing to walk
    if (p.hdr != nullptr && ld_volatile(&p.hdr->abort)) return;
    uint32_t* win = win_all[wid];
    uint64_t* bar = &bars[wid];
    if (lane == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    // the lane's look-ahead: u moves of its group's kind (0 diagonal, 1 up, 2 left)
    const int group = lane < 16 ? 0 : (lane < 24 ? 1 : 2);
    const int u = lane - (group == 0 ? 0 : (group == 1 ? 16 : 24));
    const bool g_i = group != 2, g_j = group != 1;
    const int u_i = g_i ? u : 0, u_j = g_j ? u : 0;
    uint32_t phase = 0;
    bool failed = false;
    const bool seg = p.nseg > 0;
    const int units = seg && !p.join ? p.P * p.nseg : p.P;
    for (int un = blockIdx.x * kBtWarps + wid; un < units && !failed; un += gridDim.x * kBtWarps) {
        const int q = seg && !p.join ? un / p.nseg : un;
        const PairDesc pd = p.pairs[q];
        const int N = pd.N;
        int32_t* jlo = p.jlo + (int64_t)pd.out * p.M;
        int32_t* jhi = p.jhi + (int64_t)pd.out * p.M;
        const int row_lo = p.band_lo * 32 * R, row_hi = min((int64_t)pd.M, (int64_t)p.band_hi * 32 * R);
        // the segments of this warp: one, or (join) all but the topmost from the top down
        int sk = 0, sk_end = 0, above = 0;
        if (seg && !p.join) {
            sk = sk_end = un - q * p.nseg;
            if (row_lo + sk * p.seg_rows >= row_hi) continue;
        } else if (seg) {
            sk = (row_hi - row_lo + p.seg_rows - 1) / p.seg_rows - 1;
            above = p.seg[4 * ((int64_t)q * p.nseg + sk) + 1];
            --sk;
        }
        for (; sk >= sk_end && !failed; --sk) {
            int i, j, len = 0;
            int i_lo = row_lo;
            int32_t* sg = seg ? p.seg + 4 * ((int64_t)q * p.nseg + sk) : nullptr;
            bool mergeable = false, merged = false;
            bool lead = false;               // above the segment: nothing is recorded
            int old_exit = -1;
            if (seg) {
                // segment sk: rows [row_lo + sk * seg_rows, top]; the topmost one holds the group's last row
                i_lo = row_lo + sk * p.seg_rows;
                const int top = min(row_hi, i_lo + p.seg_rows) - 1;
                if (!p.join) {
                    // the path enters the group's last row at `entry` and ends at (0, 0):
                    // from the line between them, lead_rows above the segment's top
                    const int entry = p.first ? N - 1 : p.state[q];
                    const int from = (int)min((int64_t)top + p.lead_rows, (int64_t)row_hi - 1);
                    i = from;
                    j = from == row_hi - 1 ? entry : (int)((int64_t)from * entry / (row_hi - 1));
                    lead = from > top;
                    if (entry < 0 || entry >= N) {       // the group above failed
                        if (lane == 0) { sg[0] = -1; sg[1] = -1; sg[3] = 1; }
                        continue;
                    }
                    if (lead) i_lo = top + 1;
                    if (lane == 0) {
                        sg[0] = lead ? -1 : j;
                        if (!lead) jhi[i] = j;
                    }
                } else {
                    if (above == sg[0]) {                // the walk recorded stands
                        above = sg[1];
                        continue;
                    }
                    if (above < 0 || above >= N) {       // the segment above failed
                        __syncwarp();
                        if (lane == 0) { sg[0] = above; sg[1] = -1; sg[3] = 1; }
                        above = -1;
                        continue;
                    }
                    // A second walk stops where it enters the first one of this
                    // segment, whose ranges the arrays hold: from a shared cell the
                    // walks are the same.  Row top of the first is [jlo(top), its start].
                    mergeable = sg[3] == 0;
                    old_exit = sg[1];
                    const bool at_top = mergeable && jlo[top] <= above && above <= sg[0];
                    __syncwarp();
                    if (lane == 0) { jhi[top] = above; sg[0] = above; }
                    if (at_top) {
                        above = old_exit;
                        continue;
                    }
                    i = top; j = above;
                }
            } else {
                i = pd.M - 1; j = p.subseq ? p.bstar[pd.out] : N - 1;
                if (j < 0 || j >= N) {                    // b* is not a column of this cycle: no walk
                    if (lane == 0) {
                        if (p.astar) p.astar[pd.out] = -1;
                        if (p.plen) p.plen[pd.out] = -1;
                    }
                    continue;
                }
                if (lane == 0) jhi[i] = j;
            }
            bool vote_next = false;                     // a second walk: after unchecked rows, a checked run
            int band = -1, wlo = 0, whi = -1;           // word rows in the window
            bool left_group = false;
            for (;;) {
                ++len;
                if (i == 0 && j == 0) break;
                const int b = i >> (LOG_R + 5);
                const int row = (j + ((i >> LOG_R) & 31)) / SPW;     // word row of step s = j + t
                if (b != band || row < wlo || row > whi) {
                    band = b;
                    whi = row;
                    wlo = max(0, row - kBtRows + 1);
                    const uint32_t* src = p.dirs + pd.dir_off + (int64_t)(b - p.band_lo) * band_dir_words(N, R) +
                                          (int64_t)wlo * 32 * W;
                    const uint32_t bytes = (uint32_t)(whi - wlo + 1) * 32 * W * 4;
                    __syncwarp();
                    if (lane == 0) {
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                                     :: "r"(smem_u32(bar)), "r"(bytes) : "memory");
                        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                     :: "r"(smem_u32(win)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
                    }
                    const bool ok = mbar_wait(bar, phase);
                    phase ^= 1u;
                    if (!ok) {
                        // the copy did not land in time: give up on this pair,
                        // wait (bounded) for the copy still in flight, stop
                        mbar_wait(bar, phase ^ 1u);
                        len = -1;
                        failed = true;
                        break;
                    }
                }
                // away from the window's and the rows' ends: the same runs without a check
                // (in a loop of its own: a warp walking alone is bound by the chain of
                // dependent instructions, about 5 cycles each)
                // (a second walk: kBtBurst rows at a time, then a run that looks for the first walk)
                int floor = max(b << (LOG_R + 5), i_lo + 1);
                if (mergeable) floor = max(floor, i - kBtBurst);
                const int first = wlo * SPW;             // the window's first step; jw: columns from there
                int jw = j - first;
                if (!vote_next && Win::inside(i, jw, first, floor)) {
                    vote_next = mergeable;
                    int taken = 0;
                    do {
                        const int iu = i - u_i, ju = jw - u_j;
                        const int tt = (iu >> LOG_R) & 31;
                        const int ss = ju + tt;
                        const uint32_t* wp = win + Win::word(ss, tt);
                        const int kk = iu & (R - 1);
                        // "not diag" and "not up" of the cell at fixed places of x
                        uint32_t x;
                        if (R == 32) x = ((wp[0] << kk) & 0x80000000u) | (((wp[W - 1] << kk) >> 1) & 0x40000000u);
                        else x = wp[0] << (R == 4 ? (ss % SPW) * 2 * R + 2 * kk : R == 8 ? kk + 16 - (ss & 1) * 16 : kk);
                        constexpr uint32_t ND = R == 16 ? 0x8000u : (R == 8 ? 0x800000u : 0x80000000u);
                        constexpr uint32_t NU = R == 16 || R == 8 ? 0x80000000u : 0x40000000u;
                        const uint32_t mask = group == 0 ? ND : (ND | NU);
                        const uint32_t want = group == 0 ? 0u : (group == 1 ? ND : (ND | NU));
                        const uint32_t votes = __ballot_sync(FULL, (x & mask) == want);
                        const int base = __ffs(votes & 0x01010001u) - 1;
                        const int run = __ffs(~((votes >> base) & (base == 0 ? 0xffffu : 0xffu))) - 1;
                        const int di = base != 24, dj = base != 16;
                        if (di && !lead && lane >= base && lane < base + run) {
                            jlo[iu] = first + ju;
                            jhi[iu - 1] = first + ju - dj;
                        }
                        i -= di ? run : 0;
                        jw -= dj ? run : 0;
                        taken += run;
                    } while (Win::inside(i, jw, first, floor));
                    j = first + jw;
                    len += taken - 1;
                    continue;
                }
                vote_next = false;
                // Runs: the lanes read ahead along all three kinds of move at once,
                // 16 cells on the diagonal, 8 up, 8 left (lane u of a group the cell
                // that u moves of its kind would reach); a lane agrees if its cell is
                // in the window and codes the group's move and, past the first, the
                // move is an ordinary one (not out of the grid, not out of the rows
                // loaded).  The first lane of one group agrees, which is the cell's
                // own move, and the lanes that agree after it are the run: the same
                // walk as one cell at a time, with one shared-memory read and one
                // vote per run (the read of the cell, then of its run, took two).
                const int iu = i - u_i, ju = j - u_j;
                const int tt = (iu >> LOG_R) & 31;
                const int ss = ju + tt;
                const bool here = iu >= (b << (LOG_R + 5)) && ju >= 0 && ss >= first;
                // cell (iu, ju) of the window: lane t = (iu mod BR) / R, row k = iu
                // mod R, step s = ju + t
                const uint32_t* wp = win + (here ? Win::word(ss - first, tt) : 0);
                const int kk = iu & (R - 1);
                uint32_t nd, nu;
                if (R == 4) {
                    const uint32_t w1 = wp[0] << ((ss % SPW) * 2 * R + 2 * kk);
                    nd = w1 >> 31;
                    nu = (w1 >> 30) & 1u;
                } else {
                    const uint32_t w0 = R < 16 ? wp[0] >> ((ss % SPW) * 2 * R) : wp[0];
                    nd = (w0 >> (R - 1 - kk)) & 1u;
                    nu = R <= 16 ? (w0 >> (2 * R - 1 - kk)) & 1u : (wp[W - 1] >> (R - 1 - kk)) & 1u;
                }
                // codes: diag (nd = 0) moves up-left, up (nd = 1, nu = 0) moves up,
                // left (nd = nu = 1) moves left
                const int kind = nd == 0u ? 0 : (nu == 0u ? 1 : 2);
                const bool agree = here && kind == group &&
                                   (u == 0 || ((!g_i || (iu > 0 && iu - 1 >= i_lo)) && (!g_j || ju > 0)));
                const uint32_t votes = __ballot_sync(FULL, agree);
                const int base = __ffs(votes & 0x01010001u) - 1;       // the group's first lane
                const int di = base != 24, dj = base != 16;
                // Sub-DTW: a move up from row 0 reaches the free start
                if (p.subseq && i == 0 && di) break;
                // a valid code matrix only moves left on row 0 and only up on
                // column 0; anything else is reported as |pi| = -1
                if ((i == 0 && di) || (j == 0 && dj)) { len = -1; break; }
                int run = __ffs(~((votes >> base) & (base == 0 ? 0xffffu : 0xffu))) - 1;
                // a re-walk: does the move of c_u enter a row at a cell of the
                // previous walk (read before this run's writes)?
                const bool mine = lane >= base && lane < base + run && di;
                uint32_t mv = 0u;
                if (mergeable) {                         // warp-uniform
                    bool mg = false;
                    if (mine && iu - 1 >= i_lo) {
                        const int je = ju - dj;
                        mg = jlo[iu - 1] <= je && je <= jhi[iu - 1];
                    }
                    mv = __ballot_sync(FULL, mg);
                    if (mv) run = __ffs(mv) - base;      // up to and including the first such move
                }
                if (mine && !lead && lane < base + run) {
                    jlo[iu] = ju;
                    jhi[iu - 1] = ju - dj;
                }
                i -= run * di;
                j -= run * dj;
                len += run - 1;
                if (mv) { merged = true; break; }
                if (i < i_lo) {
                    if (!lead) { left_group = true; break; }   // the rest lies in bands not loaded
                    // the segment's top row: from here on the walk is recorded
                    lead = false;
                    i_lo = row_lo + sk * p.seg_rows;
                    if (lane == 0) { jhi[i] = j; sg[0] = j; }
                }
            }
            if (seg) {
                // the path's column in the row below (merged: the rest is the first walk's)
                above = merged ? old_exit : (left_group ? j : -1);
                if (lane == 0 && !merged) {
                    sg[1] = above;
                    sg[3] = len < 0 ? 1 : 0;
                    if (!left_group && i == 0 && j == 0 && len > 0) jlo[0] = 0;
                }
                continue;
            }
            if (lane == 0) {
                if (p.subseq) {
                    if (len > 0) jlo[0] = j;
                    p.astar[pd.out] = len > 0 ? j : -1;
                } else if (i == 0 && j == 0 && len > 0) {
                    jlo[0] = 0;
                }
                if (p.plen) p.plen[pd.out] = len;
            }
        }
    }
}

// One warp per pair, after the two launches of a segmented walk: the segments
// must join up (each one's start = the exit of the one above) and none may
// have failed; then |pi| = sum_i (jhi(i) - jlo(i) + 1), the cells of a monotone
// path being row by row contiguous.
__global__ void __launch_bounds__(128) bt_seg_final_kernel(BTParams p)
{
    const int lane = threadIdx.x & 31;
    const int q = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (q >= p.P) return;
    if (p.hdr != nullptr && ld_volatile(&p.hdr->abort)) return;      // nothing was walked
    const PairDesc pd = p.pairs[q];
    const int rows = min((int64_t)pd.M, (int64_t)p.band_hi * 32 * p.R) - p.band_lo * 32 * p.R;
    const int nseg = (rows + p.seg_rows - 1) / p.seg_rows;
    bool bad = false;
    for (int k = lane; k < nseg; k += 32) {
        const int32_t* sg = p.seg + 4 * ((int64_t)q * p.nseg + k);
        if (sg[3] != 0) bad = true;
        if (k + 1 < nseg && sg[0] != sg[4 + 1]) bad = true;
    }
    bad = __any_sync(FULL, bad);
    if (p.state != nullptr && lane == 0) p.state[q] = bad ? -1 : p.seg[4 * (int64_t)q * p.nseg + 1];
    if (p.band_lo > 0) return;                       // rows below are still to be walked
    const int32_t* jlo = p.jlo + (int64_t)pd.out * p.M;
    const int32_t* jhi = p.jhi + (int64_t)pd.out * p.M;
    long long cells = 0;
    for (int i = lane; i < pd.M; i += 32) cells += (long long)(jhi[i] - jlo[i] + 1);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cells += __shfl_xor_sync(FULL, cells, o);
    if (lane == 0 && p.plen) p.plen[pd.out] = bad ? -1 : (int32_t)cells;
}

// One thread per (prototype row i, channel c); the sum of channel c of row i
// is taken in double, cycles in ascending order, samples in ascending order,
// then one division and one rounding to float (the thread of channel 0 also
// writes the count).  The ranges of the next kPre cycles are loaded ahead so
// that the dependent range -> sample loads of successive cycles overlap.
constexpr int kPre = 8;

__global__ void __launch_bounds__(256) dba_average_kernel(const float* __restrict__ data,
                                                          const int64_t* __restrict__ offsets, int T, int d,
                                                          int64_t M, const int32_t* __restrict__ jlo,
                                                          const int32_t* __restrict__ jhi,
                                                          const float* __restrict__ costs, float* __restrict__ B_out,
                                                          int32_t* __restrict__ counts, double* cost_before)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q < M * d) {
        const int64_t i = q / d;
        const int c = (int)(q - i * d);
        double acc = 0.0;
        int64_t cnt = 0;
        for (int k0 = 0; k0 < T; k0 += kPre) {
            int a[kPre], b[kPre];
            int64_t o[kPre];
#pragma unroll
            for (int u = 0; u < kPre; ++u) {
                const int k = k0 + u;
                if (k < T) {
                    o[u] = __ldg(offsets + k);
                    const int n = (int)(__ldg(offsets + k + 1) - o[u]);
                    // ranges come from the backtrack; clamping keeps every read
                    // inside the cycle even if a range were never written
                    a[u] = max(__ldg(jlo + (int64_t)k * M + i), 0);
                    b[u] = min(__ldg(jhi + (int64_t)k * M + i), n - 1);
                } else {
                    o[u] = 0; a[u] = 0; b[u] = -1;
                }
            }
            float first[kPre];
#pragma unroll
            for (int u = 0; u < kPre; ++u)
                first[u] = b[u] >= a[u] ? __ldg(data + (o[u] + a[u]) * d + c) : 0.f;
#pragma unroll
            for (int u = 0; u < kPre; ++u) {
                if (b[u] < a[u]) continue;
                acc = __dadd_rn(acc, (double)first[u]);
                for (int j = a[u] + 1; j <= b[u]; ++j)
                    acc = __dadd_rn(acc, (double)__ldg(data + (o[u] + j) * d + c));
                cnt += b[u] - a[u] + 1;
            }
        }
        B_out[q] = __double2float_rn(__ddiv_rn(acc, (double)(cnt > 0 ? cnt : 1)));
        if (counts && c == 0) counts[i] = (int32_t)cnt;
    }
    if (q == 0 && cost_before) {
        double s = 0.0;
        for (int k = 0; k < T; ++k) s = __dadd_rn(s, (double)costs[k]);
        *cost_before = s;
    }
}

__global__ void score_divide_kernel(const float* __restrict__ cost, const int32_t* __restrict__ plen,
                                    float* __restrict__ score, int T)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < T) {
        const int32_t c = plen[k];
        score[k] = c > 0 ? __fdiv_rn(cost[k], (float)c) : __int_as_float(0x7fc00000);
    }
}

// Linear resampling: p = m (N-1)/(M-1), i = floor(p), x_i + (p - i)(x_{i+1} - x_i),
// in double with every operation rounded separately, then rounded to float.
__device__ __forceinline__ float resample_at(const float* x, int64_t N, int d, int c, int64_t m, int64_t M)
{
    const double pos = M > 1 ? __ddiv_rn((double)(m * (N - 1)), (double)(M - 1)) : 0.0;
    int64_t i = (int64_t)floor(pos);
    if (i > N - 1) i = N - 1;
    const double f = __dsub_rn(pos, (double)i);
    const double xi = (double)x[i * d + c];
    double v = xi;
    if (i + 1 < N) v = __dadd_rn(xi, __dmul_rn(f, __dsub_rn((double)x[(i + 1) * d + c], xi)));
    return __double2float_rn(v);
}

__global__ void resample_kernel(const float* x, int64_t N, int d, float* out, int64_t M)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q < M * d) out[q] = resample_at(x, N, d, (int)(q % d), q / d, M);
}

__global__ void euclid_mean_kernel(const float* data, const int64_t* offsets, int T, int d, int64_t M, float* out)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= M * d) return;
    const int c = (int)(q % d);
    const int64_t m = q / d;
    double acc = 0.0;
    for (int k = 0; k < T; ++k) {
        const int64_t o = offsets[k];
        acc = __dadd_rn(acc, (double)resample_at(data + o * d, offsets[k + 1] - o, d, c, m, M));
    }
    out[q] = __double2float_rn(__ddiv_rn(acc, (double)T));
}

// Row sums of the symmetric pairwise cost matrix in double (ascending column),
// then the first index of the smallest sum.
__global__ void medoid_kernel(const float* C, int T, int32_t* index_out, double* sums)
{
    for (int a = threadIdx.x; a < T; a += blockDim.x) {
        double s = 0.0;
        for (int b = 0; b < T; ++b) s = __dadd_rn(s, (double)C[(int64_t)a * T + b]);
        sums[a] = s;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int best = 0;
        for (int a = 1; a < T; ++a)
            if (sums[a] < sums[best]) best = a;
        *index_out = best;
    }
}

}  // namespace

cudaError_t launch_backtrack(const BTParams& p, cudaStream_t st)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const bool by_segment = p.nseg > 0 && !p.join;
    const int units = by_segment ? p.P * p.nseg : p.P;
    const int need = (units + kBtWarps - 1) / kBtWarps;
    const int cap = (by_segment ? 8 : 4) * sms;
    const int grid = need < cap ? need : cap;
    if (p.R == 4) backtrack_kernel<4><<<grid, 32 * kBtWarps, 0, st>>>(p);
    else if (p.R == 8) backtrack_kernel<8><<<grid, 32 * kBtWarps, 0, st>>>(p);
    else if (p.R == 16) backtrack_kernel<16><<<grid, 32 * kBtWarps, 0, st>>>(p);
    else if (p.R == 32) backtrack_kernel<32><<<grid, 32 * kBtWarps, 0, st>>>(p);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t launch_backtrack_seg_final(const BTParams& p, cudaStream_t st)
{
    const int warps = 4;
    bt_seg_final_kernel<<<(p.P + warps - 1) / warps, 32 * warps, 0, st>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_dba_average(const float* data, const int64_t* offsets, int T, int d, int64_t M,
                               const int32_t* jlo, const int32_t* jhi, const float* costs,
                               float* B_out, int32_t* counts, double* cost_before, cudaStream_t st)
{
    const int64_t n = M * d;
    // few rows: blocks of one warp spread the FP64 adds over the SMs (1,093 rows
    // x 16 cycles: 19.3 -> 16.2 us)
    const int block = n <= 152 * 256 ? 32 : 256;
    const int grid = (int)((n + block - 1) / block);
    dba_average_kernel<<<grid, block, 0, st>>>(data, offsets, T, d, M, jlo, jhi, costs, B_out, counts, cost_before);
    return cudaGetLastError();
}

cudaError_t launch_score_divide(const float* cost, const int32_t* plen, float* score, int T, cudaStream_t st)
{
    score_divide_kernel<<<(T + 255) / 256, 256, 0, st>>>(cost, plen, score, T);
    return cudaGetLastError();
}

cudaError_t launch_resample(const float* x, int64_t N, int d, float* out, int64_t M, cudaStream_t st)
{
    const int64_t n = M * d;
    resample_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(x, N, d, out, M);
    return cudaGetLastError();
}

cudaError_t launch_euclid_mean(const float* data, const int64_t* offsets, int T, int d, int64_t M,
                               float* out, cudaStream_t st)
{
    const int64_t n = M * d;
    euclid_mean_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(data, offsets, T, d, M, out);
    return cudaGetLastError();
}

cudaError_t launch_medoid(const float* C, int T, int32_t* index_out, double* sums, cudaStream_t st)
{
    medoid_kernel<<<1, 256, 0, st>>>(C, T, index_out, sums);
    return cudaGetLastError();
}

}  // namespace wts
