// Kernel templates of the hard-min band wavefront for DTW (Eq. 1, computed by
// the recursion Eq. 5 with gamma = 0; the alignment path of Definition
// "Alignment path").  Each dtw_wavefront_*.cu file instantiates one set of
// them (rows per lane R, local cost, with or without a band), so that the
// sets compile in parallel; dtw_wavefront.cu dispatches between the sets.
//
//   r(0,0) = 0, r(i,0) = r(0,j) = +inf,
//   r(i,j) = delta(i,j) + min(r(i-1,j-1), r(i-1,j), r(i,j-1)),
//   delta(i,j) = sum_c (b_ic - y_jc)^2   (squared Euclidean local cost), or
//   its square root (COST = kCostL2: the l2 norm, Sec. 3.2's wording).
//
// Ties between predecessors resolve diag first, then up (i-1,j), then left
// (i,j-1).  With m = min(dg, up, lf): the predecessor is diag iff dg == m,
// else up iff up == m, else left.  The CPU oracle takes the same decision in
// the same float arithmetic (subtract, then one fused multiply-add per channel
// from 0, the IEEE square root for the l2 norm, then one add), so paths match
// bit for bit.
//
// One warp owns a band of 32*R rows of one pair; lane t holds R rows, their
// prototype samples (as row pairs, for the packed f32x2 arithmetic) and their
// last column of r in registers.  Lanes are skewed by one column (lane t is at
// column s - t in step s), so the value above a lane's first row comes from
// lane t-1 by __shfl_up_sync.  Cycle samples are staged per warp in a
// shared-memory ring as duplicated pairs {y, y}, refilled every 32
// steps from registers loaded ahead.  Lane 0 of band b > 0 reads the bottom row
// of band b-1 from a hand-off row in global memory (L2), 32 columns at a time,
// also one chunk ahead; each slot is NaN until its producer has written it
// (the row is pre-filled before the launch), so the consumer re-reads only the
// slots that are not there yet.
// Each warp takes (pair, band) items in order from a global cursor, so the
// producer of any item it waits for was started earlier: no deadlock, with or
// without co-residency.  Every wait is bounded (wait_progress).
//
// Predecessor codes (kModeDirs) are two bit-planes per lane and step: bit
// p*R + R-1-k of the lane's W = R/16 words is plane p of row k, plane 0 = "not
// diag", plane 1 = "not up" (meaningful only when plane 0 is set).  With R = 8
// a step has 16 bits and two consecutive steps share one word, the earlier in
// the lower bits.
#pragma once

#include <type_traits>

#include "dtw_wavefront.cuh"

namespace wts {

namespace {

typedef unsigned long long u64;

__device__ __forceinline__ u64 pack2(float lo, float hi)
{
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ void unpack2(u64 v, float& lo, float& hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

__device__ __forceinline__ u64 fsub2(u64 a, u64 b)
{
    u64 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ u64 fmul2(u64 a, u64 b)
{
    u64 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ u64 ffma2(u64 a, u64 b, u64 c)
{
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

__device__ __forceinline__ float min3f(float a, float b, float c)
{
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// all ones if a != b, else 0
__device__ __forceinline__ uint32_t ne_mask(float a, float b)
{
    uint32_t r;
    asm("set.ne.u32.f32 %0, %1, %2;" : "=r"(r) : "f"(a), "f"(b));
    return r;
}

// Columns of cycle samples staged per warp: four chunks of 32, each at its own
// place, chunk c (columns 32 c ..) at 32 (c mod 4), or 128 where that is 0.
// The chunk at 128 has a copy at 0, and the first columns of the one at 32 a
// copy at 160, so that every column that a chunk's steps read (31 behind to 3
// ahead) lies at a fixed distance from the chunk's own place: the steps' shared
// loads need no address arithmetic.
constexpr int kRing = 164;
__device__ __forceinline__ int ring_place(int s0) { return (s0 & 127) ? (s0 & 127) : 128; }
// From seven channels on, but for nine, and for one channel's count at 16 rows, a step
// computes its own addresses (StepBand) and the ring is the four chunks alone, without
// copies.
template <int D, int R, int MODE, int COST>
constexpr bool kPerStep = (D > 6 && D != 9) ||
                          (D == 1 && R == 16 && MODE == kModePlen && COST == kCostSqEuclid);
template <int D, int R, int MODE, int COST>
constexpr int kRingOf = kPerStep<D, R, MODE, COST> ? 128 : kRing;
constexpr int kSlot = 4;     // u64 words after a warp's ring: its band's columns and the band

// Up to this many channels a code bit is the sign of m - v (an FMA-pipe subtraction
// and a funnel shift), from there on a comparison to a mask (two ALU instructions and
// their share of an OR): with six channels the FMA pipe is the fuller one (60 pairs
// of 16k x 4 ch by sign 12.9 -> 10.2 ms; 200 of 25k x 6 ch 70.0 -> 83.5).
constexpr int kSignD = 4;

// Steps of the inner loop unrolled.  Four where a step is short (8 rows up to four
// channels), and for cost + |pi| up to four channels (uneven scoring, 1,000 cycles x 3
// ch: wavefront 143.5 -> 137.6 ms; under a band it costs, l2 100 x 6k x 3 ch 6.3 -> 7.1
// ms); two else: four of the long steps run the warps of a scheduler out of the
// instruction cache (batched DBA, 6 ch: 68.7 -> 74.1 ms; 8 rows, 6 ch, pairwise 24 of 6k
// 5.2 -> 5.6 ms).
template <int D, int R, int MODE, bool BANDED>
constexpr int kUnroll = (R == 8 && D <= 4) || (R == 16 && MODE == kModePlen && D <= 4 && !BANDED) ? 4 : 2;

// c[k] for a k known only at run time, by a binary tree of selects on the bits
// of k (R - 1 selects, no local memory)
template <int R>
__device__ __forceinline__ float pick_row(const float (&c)[R], int k)
{
    float v[R];
#pragma unroll
    for (int q = 0; q < R; ++q) v[q] = c[q];
#pragma unroll
    for (int w = R / 2; w >= 1; w /= 2) {
        const bool hi = (k & w) != 0;
#pragma unroll
        for (int q = 0; q < w; ++q) v[q] = hi ? v[q + w] : v[q];
    }
    return v[0];
}

// The results of one pair: r(M, N), and (kModePlen) |pi| and their quotient.
template <int MODE>
__device__ __forceinline__ void write_pair(const DPParams& p, const PairDesc& pd, float v, int c)
{
    if (p.cost_out) p.cost_out[pd.out] = v;
    if (MODE == kModePlen) {
        if (p.plen_out) p.plen_out[pd.out] = c;
        if (p.score_out) p.score_out[pd.out] = __fdiv_rn(v, (float)c);
    }
    if (p.cost_matrix) {
        int a = 0, rem = pd.out;
        while (rem >= p.T - 1 - a) { rem -= p.T - 1 - a; ++a; }
        const int bb = a + 1 + rem;
        p.cost_matrix[(int64_t)a * p.T + bb] = v;
        p.cost_matrix[(int64_t)bb * p.T + a] = v;
    }
}

template <int D, int R, int MODE, bool BANDED, int COST>
struct Band {
    static constexpr int BR = 32 * R;
    static constexpr int W = R / 16;        // code words per lane per step (0: part of a word)
    static constexpr int SPW = R >= 16 ? 1 : 32 / (2 * R);     // steps per code word
    static constexpr int Q = R / 2;         // row pairs

    u64 bp[Q][D];                           // prototype rows as pairs
    float col[R];                           // r at the lane's last column
    float dl[R];                            // local costs of the lane's next column
    int cnt[R];                             // path cells (kModePlen)
    float prev_up;                          // r(i0-1, j-1) for the first row
    int prev_upc;
    float topv;                             // lane l: r(band top - 1, s0 + l)
    int topc;
    uint32_t half;                          // R < 16: codes of the word's earlier steps
    // kModeSubDirs, matrix's last band: running minimum of r(M-1, j) over the
    // lane's columns (row kk of the lane), and its first column
    int kk;
    float best;
    int bestj;
    static constexpr bool CODES = MODE == kModeDirs || MODE == kModeSubDirs;
    static constexpr bool SIGNS = D <= kSignD;
    // hand-off slots: 4 bytes (r), or 8 bytes ({r, cells}) with |pi|
    static constexpr int SLOT = MODE == kModePlen ? 8 : 4;
    // the chunk's addresses (begin_chunk)
    const u64* yb;
    uint32_t* db;
    char* hb;
    int j0;
    bool puts;                              // this lane writes the band's hand-off row

    // Local costs of column jc for the lane's rows, pair q (two rows at once).
    __device__ __forceinline__ void cost_pair(const u64* yy, int q)
    {
        u64 t = fsub2(bp[q][0], yy[0]);
        u64 acc = fmul2(t, t);
#pragma unroll
        for (int c = 1; c < D; ++c) {
            t = fsub2(bp[q][c], yy[c]);
            acc = ffma2(t, t, acc);
        }
        unpack2(acc, dl[2 * q], dl[2 * q + 1]);
        if (COST == kCostL2) {                   // the norm itself: IEEE square root
            dl[2 * q] = __fsqrt_rn(dl[2 * q]);
            dl[2 * q + 1] = __fsqrt_rn(dl[2 * q + 1]);
        }
    }

    // samples of column j0 + o
    __device__ __forceinline__ void load_samples(int o, u64* yy)
    {
#pragma unroll
        for (int c = 0; c < D; ++c) yy[c] = yb[c * kRing + o];
    }

    // Addresses of the chunk of steps s0 .. s0 + 31.
    __device__ __forceinline__ void begin_chunk(const u64* ring, int s0, int lane, void* hcur, uint32_t* dout)
    {
        yb = ring + (ring_place(s0) - lane);
        j0 = s0 - lane;
        if (CODES) db = dout + ((int64_t)(s0 / SPW) * 32 + lane) * (W > 0 ? W : 1);
        if (puts) hb = static_cast<char*>(hcur) + (int64_t)j0 * SLOT;
    }

    // Step u of the chunk: the lane's column j = j0 + u (in range when FULLCHUNK).
    // dl holds the local costs of column j on entry and those of column j+1 on
    // exit: the next column's costs are computed between the links of this
    // column's min-plus chain, which is serial down the rows.
    template <bool FULLCHUNK, bool MASK = false, bool TRACK = false>
    __device__ __forceinline__ void step(const u64* slot, int u, int lane, int N, bool top)
    {
        const float INF = inf_f();
        const float above = __shfl_up_sync(FULL, col[R - 1], 1);
        const float tv = __shfl_sync(FULL, topv, u);
        // above the matrix: +inf (DTW), 0 for Sub-DTW (a path may start in any column)
        const float top_in = MODE == kModeSubDirs ? 0.f : INF;
        const float up_in = lane == 0 ? (top ? top_in : tv) : above;
        const float dg_in = prev_up;
        prev_up = up_in;
        int upc_in = 0, dgc_in = 0;
        if (MODE == kModePlen) {
            const int abovec = __shfl_up_sync(FULL, cnt[R - 1], 1);
            const int tc = __shfl_sync(FULL, topc, u);
            upc_in = lane == 0 ? tc : abovec;
            dgc_in = prev_upc;
            prev_upc = upc_in;
        }
        const int j = j0 + u;
        u64 yy[D];
        load_samples(u + 1, yy);
        uint32_t pl0 = 0u, pl1 = 0u;             // the step's code planes (in the low R bits)
        // partial chunks with a band read the band's columns (and the band)
        // from the warp's slot after the sample ring:
        // [jlo | jhi << 32, row0 | M << 32, bnd]
        bool valid = true;
        int klo = 0, khi = R - 1;
        if (!FULLCHUNK && !BANDED) valid = j >= 0 && j < N;
        if (!FULLCHUNK && BANDED) {
            const u64 cols = slot[0];
            valid = j >= (int)(uint32_t)cols && j <= (int)(cols >> 32);
            if (MASK) {
                // rows k in [klo, khi] lie in the band at column j
                const u64 im = slot[1];
                const int64_t bnd = (int64_t)slot[2];
                const int i0 = (int)(uint32_t)im + lane * R;
                const int64_t jm = (int64_t)j * (int64_t)(im >> 32);
                klo = (int)max((int64_t)-1, ceil_div64(jm - bnd, N) - i0);
                khi = (int)min((int64_t)R, floor_div64(jm + bnd, N) - i0);
            }
        }
        if (FULLCHUNK || valid) {
            float dg = dg_in, up = up_in;
            int cdg = dgc_in, cup = upc_in;
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const float lf = col[k];
                const float m = min3f(dg, up, lf);
                float r = __fadd_rn(dl[k], m);
                if (MASK && (k < klo || k > khi)) r = INF;     // outside the band
                if (CODES) {
                    if (SIGNS) {
                        // the sign of m - v (0 when equal, also at +inf: that NaN is positive)
                        pl0 = __funnelshift_l(__float_as_uint(__fsub_rn(m, dg)), pl0, 1);
                        pl1 = __funnelshift_l(__float_as_uint(__fsub_rn(m, up)), pl1, 1);
                    } else {
                        static_assert(R < 32 || SIGNS, "32 rows' codes are taken by sign");
                        pl0 |= ne_mask(dg, m) & (1u << (R - 1 - k));
                        pl0 |= ne_mask(up, m) & (1u << ((2 * R - 1 - k) & 31));
                    }
                } else if (MODE == kModePlen) {
                    const int cl = cnt[k];
                    const int cn = 1 + (dg == m ? cdg : (up == m ? cup : cl));
                    cdg = cl;
                    cup = cn;
                    cnt[k] = cn;
                }
                dg = lf;
                up = r;
                col[k] = r;
                if (k & 1) cost_pair(yy, k >> 1);      // rows k-1, k of column j+1
            }
            if (TRACK) {
                const float v = pick_row<R>(col, kk);
                const bool less = v < best;
                best = less ? v : best;
                bestj = less ? j : bestj;
            }
            if (puts) {
                if (MODE == kModePlen)
                    __stcg(reinterpret_cast<u64*>(hb) + u, pack2(col[R - 1], __int_as_float(cnt[R - 1])));
                else
                    __stcg(reinterpret_cast<float*>(hb) + u, col[R - 1]);
            }
        } else {
#pragma unroll
            for (int q = 0; q < Q; ++q) cost_pair(yy, q);
        }
        if (CODES) {
            if (W < 2 && SIGNS) pl0 = R == 16 ? __byte_perm(pl0, pl1, 0x5410) : (pl1 << R) | pl0;
            if (W == 0) {                    // (chunks start at multiples of 32)
                if ((u & 1) == 0)
                    half = pl0;
                else
                    __stcs(db + (u >> 1) * 32, __byte_perm(half, pl0, 0x5410));
            } else if (W == 1) {
                __stcs(db + u * 32, pl0);
            } else {
                __stcs(reinterpret_cast<uint2*>(db) + u * 32, make_uint2(pl0, pl1));
            }
        }
    }
};

// The step for wide samples (kPerStep): addresses from the step's number, code bits
// by comparison, a Sub-DTW band's last row tracked behind a branch.  A chunk's
// addresses, held beside 16 rows of 8 channels and more, and a second loop for the
// tracked band cost these instances more than they save; with sixteen channels the
// prototype rows spill, and a ring with copies takes the L1 that holds them (shared
// memory of two blocks 130 -> 170 KB of the SM's 256).  Wavefront, 300 pairs of 6k (100 at 16
// channels), 16 rows, per chunk / per step in ms: 8 channels codes 8.5 / 7.7, 16
// channels codes 10.9 / 7.0, cost + |pi| 16.5 / 9.0, l2 checkpointed 50 / 23.6, Sub-DTW
// l2 28 / 13.4, 12 channels 28 / 23.4.  At nine channels: codes 8.4 / 9.4.  One channel,
// cost + |pi|, 16 rows: 3.79 / 3.35, under a band of 0.4 3.46 / 3.34.
template <int D, int R, int MODE, bool BANDED, int COST>
struct StepBand : Band<D, R, MODE, BANDED, COST> {
    using B = Band<D, R, MODE, BANDED, COST>;
    using B::CODES; using B::W; using B::Q;
    using B::col; using B::dl; using B::cnt; using B::prev_up; using B::prev_upc; using B::topv; using B::topc;
    using B::half; using B::kk; using B::best; using B::bestj; using B::cost_pair;
    static constexpr int RING = kRingOf<D, R, MODE, COST>;
    bool track;

    __device__ __forceinline__ void load_column(const u64* ring, int jc, u64* yy)
    {
        const u64* yr = ring + (jc & (RING - 1));
#pragma unroll
        for (int c = 0; c < D; ++c) yy[c] = yr[c * RING];
    }

    // One step: the lane's column j = s - lane (in range when FULLCHUNK), the value
    // above its band's first row in lane u.
    template <bool FULLCHUNK, bool MASK = false>
    __device__ __forceinline__ void step_at(const u64* ring, int s, int u, int lane, int N, bool top, void* hcur,
                                            uint32_t* dout)
    {
        const float INF = inf_f();
        const float above = __shfl_up_sync(FULL, col[R - 1], 1);
        const float tv = __shfl_sync(FULL, topv, u);
        const float top_in = MODE == kModeSubDirs ? 0.f : INF;
        const float up_in = lane == 0 ? (top ? top_in : tv) : above;
        const float dg_in = prev_up;
        prev_up = up_in;
        int upc_in = 0, dgc_in = 0;
        if (MODE == kModePlen) {
            const int abovec = __shfl_up_sync(FULL, cnt[R - 1], 1);
            const int tc = __shfl_sync(FULL, topc, u);
            upc_in = lane == 0 ? tc : abovec;
            dgc_in = prev_upc;
            prev_upc = upc_in;
        }
        const int j = s - lane;
        u64 yy[D];
        load_column(ring, j + 1, yy);
        uint32_t word = 0u;
        const u64* slot = ring + D * RING;
        bool valid = true;
        int klo = 0, khi = R - 1;
        if (!FULLCHUNK && !BANDED) valid = j >= 0 && j < N;
        if (!FULLCHUNK && BANDED) {
            const u64 cols = slot[0];
            valid = j >= (int)(uint32_t)cols && j <= (int)(cols >> 32);
            if (MASK) {
                const u64 im = slot[1];
                const int64_t bnd = (int64_t)slot[2];
                const int i0 = (int)(uint32_t)im + lane * R;
                const int64_t jm = (int64_t)j * (int64_t)(im >> 32);
                klo = (int)max((int64_t)-1, ceil_div64(jm - bnd, N) - i0);
                khi = (int)min((int64_t)R, floor_div64(jm + bnd, N) - i0);
            }
        }
        if (FULLCHUNK || valid) {
            float dg = dg_in, up = up_in;
            int cdg = dgc_in, cup = upc_in;
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const float lf = col[k];
                const float m = min3f(dg, up, lf);
                float r = __fadd_rn(dl[k], m);
                if (MASK && (k < klo || k > khi)) r = INF;     // outside the band
                if (CODES) {
                    word |= ne_mask(dg, m) & (1u << (R - 1 - k));
                    word |= ne_mask(up, m) & (1u << (2 * R - 1 - k));
                } else if (MODE == kModePlen) {
                    const int cl = cnt[k];
                    const int cn = 1 + (dg == m ? cdg : (up == m ? cup : cl));
                    cdg = cl;
                    cup = cn;
                    cnt[k] = cn;
                }
                dg = lf;
                up = r;
                col[k] = r;
                if (k & 1) cost_pair(yy, k >> 1);      // rows k-1, k of column j+1
            }
            if (MODE == kModeSubDirs && track) {
                const float v = pick_row<R>(col, kk);
                if (v < best) { best = v; bestj = j; }
            }
            if (lane == 31 && hcur != nullptr) {
                if (MODE == kModePlen)
                    __stcg(reinterpret_cast<u64*>(hcur) + j, pack2(col[R - 1], __int_as_float(cnt[R - 1])));
                else
                    __stcg(reinterpret_cast<float*>(hcur) + j, col[R - 1]);
            }
        } else {
#pragma unroll
            for (int q = 0; q < Q; ++q) cost_pair(yy, q);
        }
        if (CODES) {
            if (W == 0) {
                if ((s & 1) == 0)
                    half = word;
                else
                    __stcs(dout + (int64_t)(s >> 1) * 32 + lane, __byte_perm(half, word, 0x5410));
            } else {
                __stcs(dout + (int64_t)s * 32 + lane, word);
            }
        }
    }
};

template <int D, int R, int MODE, bool BANDED, int COST>
__device__ __forceinline__ void run_band(const DPParams& p, const PairDesc& pd, int band, int lane, u64* ring)
{
    constexpr bool PER_STEP = kPerStep<D, R, MODE, COST>;
    using BandT =
        std::conditional_t<PER_STEP, StepBand<D, R, MODE, BANDED, COST>, Band<D, R, MODE, BANDED, COST>>;
    constexpr int BR = BandT::BR;
    constexpr int RING = kRingOf<D, R, MODE, COST>;
    constexpr int W = BandT::W;
    const int M = pd.M, N = pd.N, d = p.d;
    const int i0 = band * BR + lane * R;
    const bool top = band == 0;
    const bool last = band == pd.nbands - 1;
    const float INF = inf_f();

    BandT st;
#pragma unroll
    for (int q = 0; q < BandT::Q; ++q)
#pragma unroll
        for (int c = 0; c < D; ++c) {
            const int ia = i0 + 2 * q, ib = ia + 1;
            const float va = (ia < M && c < d) ? __ldg(pd.X + (int64_t)ia * d + c) : 0.f;
            const float vb = (ib < M && c < d) ? __ldg(pd.X + (int64_t)ib * d + c) : 0.f;
            st.bp[q][c] = pack2(va, vb);
        }
#pragma unroll
    for (int k = 0; k < R; ++k) { st.col[k] = INF; st.cnt[k] = 0; }
    // r(i0-1, j-1) at j = 0: r(0,0) = 0 (0 cells) for the matrix's first row, +inf otherwise
    st.prev_up = (top && lane == 0) ? 0.f : INF;
    st.prev_upc = 0;
    st.topv = INF;
    st.topc = 0;
    st.half = 0u;
    if constexpr (PER_STEP) st.track = MODE == kModeSubDirs && last;
    st.kk = M - 1 - i0;
    st.best = INF;
    st.bestj = 0;

    // Sakoe-Chiba band: row i keeps columns [lo(i), hi(i)] with
    // lo(i) = ceil((i N - bnd) / M), hi(i) = floor((i N + bnd) / M), both
    // nondecreasing in i.  The band's columns run from lo(first row) to
    // hi(last row); the row above is +inf outside [lo, hi] of that row; a lane
    // needs no masking where all its rows are in: [lo(last row), hi(first row)].
    const int64_t bnd = BANDED ? pd.band_bound : -1;
    int jlo_b = 0, jhi_b = N - 1, jtop_lo = 0, jtop_hi = N - 1, full_lo = 0, full_hi = N - 1;
    if (BANDED) {
        auto lo_of = [&](int64_t i) { return (int)max((int64_t)0, ceil_div64(i * N - bnd, M)); };
        auto hi_of = [&](int64_t i) { return (int)min((int64_t)N - 1, floor_div64(i * N + bnd, M)); };
        const int64_t r0 = (int64_t)band * BR, r1 = min(r0 + BR, (int64_t)M) - 1;
        jlo_b = lo_of(r0);
        jhi_b = hi_of(r1);
        if (!top) { jtop_lo = lo_of(r0 - 1); jtop_hi = hi_of(r0 - 1); }
        if (i0 < M) { full_lo = lo_of(min(i0 + R - 1, M - 1)); full_hi = hi_of(i0); }
    }
    u64* slot = ring + D * RING;
    if (BANDED) {
        __syncwarp();
        if (lane == 0) {
            slot[0] = (u64)(uint32_t)jlo_b | ((u64)(uint32_t)jhi_b << 32);
            slot[1] = (u64)(uint32_t)(band * BR) | ((u64)(uint32_t)M << 32);
            slot[2] = (u64)bnd;
        }
        __syncwarp();
    }
    // chunks of 32 steps from a multiple of 32, starting at or before column
    // jlo_b - 1: lane 0 takes its first diagonal, r(r0 - 1, jlo_b - 1), from
    // the row above at the step before its first column (that cell may be
    // inside the band)
    const int s_begin = max(0, (jlo_b - 1) & ~31);
    const int s_end = jhi_b + 32;           // one past the last step (column jhi_b in lane 31)

    constexpr int SLOT = BandT::SLOT;
    char* hb = static_cast<char*>(p.hbuf);
    const char* hprev = top ? nullptr : hb + (pd.hbuf_off + (int64_t)(band - 1) * N) * SLOT;
    // a recomputed band reads its stored top row and produces no hand-off row
    void* hcur = (last || p.recompute || p.skip_handoff) ? nullptr : hb + (pd.hbuf_off + (int64_t)band * N) * SLOT;
    uint32_t* dout = BandT::CODES ? p.dirs + pd.dir_off + (int64_t)(band - p.band_lo) * band_dir_words(N, R)
                                         : nullptr;

    st.puts = lane == 31 && hcur != nullptr;

    // Cycle samples go through the ring two chunks of 32 columns ahead of the
    // step that first reads them (a step also reads the next column), loaded
    // into registers one chunk before that; the bottom row of the band above
    // (NaN until its producer has written it) is read one chunk ahead.
    float ynext[D];
    u64 tnext = 0;
    auto load_y = [&](int jj) {
#pragma unroll
        for (int c = 0; c < D; ++c) ynext[c] = (jj < N && c < d) ? __ldg(pd.Y + (int64_t)jj * d + c) : 0.f;
    };
    auto put_y = [&](int jj) {
#pragma unroll
        for (int c = 0; c < D; ++c) {
            u64* row = ring + c * RING;
            const u64 v = pack2(ynext[c], ynext[c]);
            const int i = jj & 127;
            if (PER_STEP) {
                row[i] = v;
                continue;
            }
            row[i < 32 ? i + 128 : i] = v;
            if (i < 36) row[i < 32 ? i : i + 128] = v;
        }
    };
    auto load_t = [&](int jj) -> u64 {
        if (jj >= N) return 0;
        if (SLOT == 8) return __ldcv(reinterpret_cast<const u64*>(hprev) + jj);
        return (u64)__float_as_uint(__ldcv(reinterpret_cast<const float*>(hprev) + jj));
    };
    __syncwarp();
    load_y(s_begin + lane);
    put_y(s_begin + lane);
    load_y(s_begin + lane + 32);
    put_y(s_begin + lane + 32);
    load_y(s_begin + lane + 64);
    if (!top) tnext = load_t(s_begin + lane);
    __syncwarp();
    if constexpr (!PER_STEP) st.begin_chunk(ring, s_begin, lane, hcur, dout);
    {
        // local costs of the lane's first column (j = s_begin - lane)
        u64 yy[D];
        if constexpr (PER_STEP)
            st.load_column(ring, s_begin - lane, yy);
        else
            st.load_samples(0, yy);
#pragma unroll
        for (int q = 0; q < BandT::Q; ++q) st.cost_pair(yy, q);
    }

    for (int s0 = s_begin; s0 < s_end; s0 += 32) {
        if (s0 <= jhi_b) {
            const int jj = s0 + lane;
            if (s0 > s_begin) {
                __syncwarp();
                put_y(jj + 32);
                load_y(jj + 64);
                __syncwarp();
            }
            if (!top) {
                // only the row above's columns inside the band are written (and waited for)
                const bool need = jj >= jtop_lo && jj <= jtop_hi;
                u64 t = tnext;
                const bool ok = wait_filled(need && is_nan_bits((uint32_t)t),
                                            [&]() { t = load_t(jj); return is_nan_bits((uint32_t)t); }, p.hdr, 1,
                                            p.spin_limit);
                if (!ok) return;
                st.topv = need ? __uint_as_float((uint32_t)t) : INF;
                if (MODE == kModePlen) st.topc = (int)(t >> 32);
                tnext = load_t(jj + 32);
            }
        }
        if constexpr (!PER_STEP) st.begin_chunk(ring, s0, lane, hcur, dout);
        // every lane in the band's columns and inside the band all chunk long
        const bool full = BANDED ? (s0 - 31 >= jlo_b && s0 + 31 <= jhi_b &&
                                    __all_sync(FULL, s0 - lane >= full_lo && s0 + 31 - lane <= full_hi))
                                 : (s0 >= 31 && s0 + 32 <= N);
        if constexpr (PER_STEP) {
            if (full) {
#pragma unroll 2
                for (int u = 0; u < 32; ++u) st.template step_at<true>(ring, s0 + u, u, lane, N, top, hcur, dout);
            } else {
                const int n = min(32, s_end - s0);
                for (int u = 0; u < n; ++u)
                    st.template step_at<false, BANDED>(ring, s0 + u, u, lane, N, top, hcur, dout);
            }
        } else {
            auto chunk = [&](auto track) {
                constexpr bool TRACK = decltype(track)::value;
                if (full) {
#pragma unroll (kUnroll<D, R, MODE, BANDED>)
                    for (int u = 0; u < 32; ++u) st.template step<true, false, TRACK>(slot, u, lane, N, top);
                } else {
                    const int n = min(32, s_end - s0);
#pragma unroll 1
                    for (int u = 0; u < n; ++u) st.template step<false, BANDED, TRACK>(slot, u, lane, N, top);
                }
            };
            if (MODE == kModeSubDirs && last)
                chunk(std::true_type{});
            else
                chunk(std::false_type{});
        }
    }

    constexpr int SPW = BandT::SPW;
    if (BandT::CODES && W == 0 && (s_end % SPW) != 0)
        __stcs(dout + (int64_t)((s_end - 1) / SPW) * 32 + lane, st.half);

    if (MODE == kModeSubDirs) {
        if (last && lane == (M - 1 - band * BR) / R) {
            if (p.cost_out) p.cost_out[pd.out] = st.best;
            p.bstar_out[pd.out] = st.bestj;
        }
    } else if (last && !p.recompute) {
        const int ilast = M - 1 - band * BR;
        if (lane == ilast / R) {
            const int kk = ilast % R;
            float v = st.col[0];
            int c = st.cnt[0];
#pragma unroll
            for (int k = 1; k < R; ++k)
                if (k == kk) { v = st.col[k]; c = st.cnt[k]; }
            write_pair<MODE>(p, pd, v, c);
        }
    }
}

// Blocks of at most 4 warps.  R = 16: three resident blocks (12 warps, <= 170
// registers) where the prototype rows fit easily, two otherwise (the
// software-pipelined step keeps enough independent work per warp).  R = 8
// halves the prototype registers: four blocks (16 warps, <= 128 registers) up
// to 4 channels, three up to 8 (at 6 the four spilled).
template <int D, int R>
constexpr int min_blocks()
{
    return R == 8 ? (D <= 4 ? 4 : (D <= 8 ? 3 : 2)) : ((R == 16 && D <= 4) ? 3 : 2);
}

// The (place q in the work list's pair order, band) of an item.  EQUAL: every pair
// has the same bands.
template <bool EQUAL>
__device__ __forceinline__ void item_of(const DPParams& p, int item, int& q, int& band)
{
    if (p.group_pairs > 0) {
        // groups of G pairs (in the work list's order), band-major within
        // a group: a group's bands start in the order their producers
        // do, and its items about fill the resident warps once (G = P:
        // every pair's band b before any band b + 1, as under a band,
        // where a pair has few bands ready at a time).  A pair of fewer than
        // group_bands bands (pairwise: the rows are a cycle) leaves its last
        // items empty; recompute runs the range [band_lo, band_lo + band_cnt)
        // of each pair.  Band b - 1 of a pair is earlier in the list (no
        // deadlock).
        const int nb = p.recompute ? p.band_cnt : (EQUAL ? p.prefix[1] - p.prefix[0] : p.group_bands);
        const int G = p.group_pairs;
        const int g = item / (G * nb), q0 = g * G;
        const int Gg = min(G, p.P - q0);
        const int r = item - q0 * nb;
        q = q0 + r % Gg;
        band = (p.recompute ? p.band_lo : 0) + r / Gg;
    } else if (p.recompute) {
        q = item / p.band_cnt;
        band = p.band_lo + item % p.band_cnt;
    } else {
        q = find_slot(p.prefix, p.P, item);
        band = item - p.prefix[q];
    }
}

template <int D, int R, int MODE, bool BANDED, int COST>
__global__ void __launch_bounds__(128, min_blocks<D, R>()) dtw_wavefront_kernel(DPParams p)
{
    extern __shared__ u64 ring_all[];
    const int lane = threadIdx.x & 31;
    u64* ring = ring_all + (threadIdx.x >> 5) * (D * kRingOf<D, R, MODE, COST> + kSlot);
    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(&p.hdr->item_counter, 1);
        item = __shfl_sync(FULL, item, 0);
        if (item >= p.n_items) break;
        if (ld_volatile(&p.hdr->abort)) break;
        // (known to the compiler for wide samples: it changes the step's schedule, codes of
        // 100 x 6k x 16 ch, 8 rows, 5.8 -> 5.2 ms)
        constexpr bool EQUAL = kPerStep<D, R, MODE, COST> && MODE != kModeCost;
        int q, band;
        item_of<EQUAL>(p, item, q, band);
        const PairDesc pd = p.pairs[p.order[q]];
        if (EQUAL || band < pd.nbands) run_band<D, R, MODE, BANDED, COST>(p, pd, band, lane, ring);
    }
}

template <int D, int R, int MODE, int COST>
constexpr size_t ring_bytes(int block)
{
    return (size_t)(block / 32) * (D * kRingOf<D, R, MODE, COST> + kSlot) * sizeof(u64);
}

template <int D, int R, int MODE, bool BANDED, int COST>
cudaError_t launch_one(const DPParams& p, int grid, int block, cudaStream_t st)
{
    const size_t smem = ring_bytes<D, R, MODE, COST>(block);
    cudaFuncSetAttribute(dtw_wavefront_kernel<D, R, MODE, BANDED, COST>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)smem);
    dtw_wavefront_kernel<D, R, MODE, BANDED, COST><<<grid, block, smem, st>>>(p);
    return cudaGetLastError();
}

template <int D, int R, int MODE, bool BANDED, int COST>
int occ_one(int block)
{
    int n = 0;
    const size_t smem = ring_bytes<D, R, MODE, COST>(block);
    cudaFuncSetAttribute(dtw_wavefront_kernel<D, R, MODE, BANDED, COST>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, dtw_wavefront_kernel<D, R, MODE, BANDED, COST>, block, smem);
    return n;
}

// The three DTW modes for every instance; Sub-DTW (never banded) for R = 8 and 16.
template <int D, int R, bool BANDED, int COST>
cudaError_t launch_mode(int mode, const DPParams& p, int grid, int block, cudaStream_t st)
{
    switch (mode) {
        case kModeCost: return launch_one<D, R, kModeCost, BANDED, COST>(p, grid, block, st);
        case kModePlen: return launch_one<D, R, kModePlen, BANDED, COST>(p, grid, block, st);
        case kModeDirs: return launch_one<D, R, kModeDirs, BANDED, COST>(p, grid, block, st);
        case kModeSubDirs:
            if constexpr (!BANDED && R <= 16) return launch_one<D, R, kModeSubDirs, false, COST>(p, grid, block, st);
            break;
        default: break;
    }
    return cudaErrorInvalidValue;
}

template <int D, int R, bool BANDED, int COST>
int occ_mode(int mode, int block)
{
    switch (mode) {
        case kModeCost: return occ_one<D, R, kModeCost, BANDED, COST>(block);
        case kModePlen: return occ_one<D, R, kModePlen, BANDED, COST>(block);
        case kModeDirs: return occ_one<D, R, kModeDirs, BANDED, COST>(block);
        case kModeSubDirs:
            if constexpr (!BANDED && R <= 16) return occ_one<D, R, kModeSubDirs, false, COST>(block);
            break;
        default: break;
    }
    return 0;
}

// One set of instances: every padded channel count D (1, 2, 3 only for R = 32).
#define WTS_WF_SWITCH_D(FN, ...)                                              \
    switch (D) {                                                             \
        case 1: return FN<1, R, BANDED, COST>(__VA_ARGS__);                   \
        case 2: return FN<2, R, BANDED, COST>(__VA_ARGS__);                   \
        case 3: return FN<3, R, BANDED, COST>(__VA_ARGS__);                   \
        default: break;                                                      \
    }                                                                        \
    if constexpr (R < 32) {                                                  \
        switch (D) {                                                         \
            case 4: return FN<4, R, BANDED, COST>(__VA_ARGS__);               \
            case 6: return FN<6, R, BANDED, COST>(__VA_ARGS__);               \
            case 8: return FN<8, R, BANDED, COST>(__VA_ARGS__);               \
            case 9: return FN<9, R, BANDED, COST>(__VA_ARGS__);               \
            case 12: return FN<12, R, BANDED, COST>(__VA_ARGS__);             \
            case 16: return FN<16, R, BANDED, COST>(__VA_ARGS__);             \
            default: break;                                                  \
        }                                                                    \
    }

template <int R, bool BANDED, int COST>
cudaError_t launch_set(int mode, int D, const DPParams& p, int grid, int block, cudaStream_t st)
{
    WTS_WF_SWITCH_D(launch_mode, mode, p, grid, block, st)
    return cudaErrorInvalidValue;
}

template <int R, bool BANDED, int COST>
int occ_set(int mode, int D, int block)
{
    WTS_WF_SWITCH_D(occ_mode, mode, block)
    return 0;
}

#undef WTS_WF_SWITCH_D

}  // namespace

}  // namespace wts

// Defines the entry points wf_launch_TAG / wf_occ_TAG of one instance set.
#define WTS_WF_ENTRY(TAG, R, BANDED, COST)                                                        \
    namespace wts {                                                                               \
    cudaError_t wf_launch_##TAG(int mode, int D, const DPParams& p, int grid, int block, cudaStream_t st) \
    {                                                                                             \
        return launch_set<R, BANDED, COST>(mode, D, p, grid, block, st);                          \
    }                                                                                             \
    int wf_occ_##TAG(int mode, int D, int block) { return occ_set<R, BANDED, COST>(mode, D, block); } \
    }
