// Hard-min wavefront for launches with fewer bands than the GPU has schedulers
// (one long pair, a handful of short ones): there the latency of a step and the
// lag from band to band set the time, not the instruction rate.
//
// The recursion, the lane skew, the local cost and the work list are those of
// dtw_wavefront_impl.cuh (results are the same bit for bit).  What differs:
//  - four rows per lane, so a step is short and a pair has many bands;
//  - steps run in blocks of eight without a branch, at a band's two ends too
//    (lanes outside the matrix keep their state by selects), every address an
//    offset from the block's, the samples read a step ahead;
//  - the row above is taken eight columns at a time, so a band follows the one
//    above more closely;
//  - a code bit is the sign of m - v, shifted into the word (one subtraction on
//    the FMA pipe and one funnel shift, where a comparison to a mask and its OR
//    are three ALU instructions).
// Measured (one pair, cost + |pi|): a step of 128 rows 62 ns at one channel, 83 at
// nine, bands 66 steps apart; 1.1k x 1.1k x 1 ch 102 us against 121 with 8 rows per
// lane and 265 with 32; Sub-DTW windows of 16k x 32k x 9 ch 6.35 -> 3.5 ms.  Bound
// by dependent latencies: a step's 128 cycles (one channel, 2.07 GHz) hold the shuffle
// from the lane above and, one after the other down four rows, a minimum, an addition
// and the count's selects, with one warp on a scheduler to issue them.
#pragma once

#include "dtw_wavefront_impl.cuh"

namespace wts {

namespace {

// Shared memory by 32-bit addresses (a step's loads are then one instruction each).
__device__ __forceinline__ u64 lds64(uint32_t a)
{
    u64 v;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts64(uint32_t a, u64 v)
{
    asm volatile("st.shared.b64 [%0], %1;" :: "r"(a), "l"(v) : "memory");
}

template <int D, int R, int MODE, int COST>
struct Lean {
    static constexpr int Q = R / 2;
    static constexpr int SPW = 32 / (2 * R);            // steps per code word
    static constexpr bool CODES = MODE == kModeDirs || MODE == kModeSubDirs;
    static constexpr int SLOT = MODE == kModePlen ? 8 : 4;

    u64 bp[Q][D];
    float col[R], dl[R];
    int cnt[R];
    float prev_up;
    int prev_upc;
    float above;                     // r(i0-1, j) of the next step (lanes > 0), and its cells
    int abovec;
    u64 ynx[D];                      // samples of the lane's next column
    uint32_t half;                   // codes of the word so far
    int kk;                          // kModeSubDirs, last band: the lane's row M-1, its minimum and first column
    float best;
    int bestj;
    // the block's addresses
    uint32_t yb;
    uint32_t* db;
    char* hb;                        // the hand-off row
    bool puts;                       // this lane writes it
    int j0;
    int left;                        // steps from the block's first to the band's end
    float topv;                      // lane l: the value above at column (block's first) + l mod 8
    int topc;

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
        if (COST == kCostL2) {
            dl[2 * q] = __fsqrt_rn(dl[2 * q]);
            dl[2 * q + 1] = __fsqrt_rn(dl[2 * q + 1]);
        }
    }
    __device__ __forceinline__ void load_samples(int o, u64* yy)
    {
#pragma unroll
        for (int c = 0; c < D; ++c) yy[c] = lds64(yb + (c * kRing + o) * 8);
    }

    // Step v of the block.  FULLBLOCK: every lane's column is inside the matrix
    // in every step of the block; else a lane outside keeps its state.
    template <bool FULLBLOCK, bool TRACK>
    __device__ __forceinline__ void step(int v, int lane, int N)
    {
        const float tv = __shfl_sync(FULL, topv, v);
        const float up_in = lane == 0 ? tv : above;
        const float dg_in = prev_up;
        prev_up = up_in;
        int upc_in = 0, dgc_in = 0;
        if (MODE == kModePlen) {
            const int tc = __shfl_sync(FULL, topc, v);
            upc_in = lane == 0 ? tc : abovec;
            dgc_in = prev_upc;
            prev_upc = upc_in;
        }
        u64 yz[D];
        load_samples(v + 2, yz);
        const int j = j0 + v;
        const bool valid = FULLBLOCK || (j >= 0 && j < N);
        float dgs[R], ups[R], ms[R];
        {
            float dg = dg_in, up = up_in;
            int cdg = dgc_in, cup = upc_in;
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const float lf = col[k];
                const float m = fminf(fminf(dg, lf), up);   // (two minima: only the second on the chain)
                const float r = __fadd_rn(dl[k], m);
                if (CODES) { dgs[k] = dg; ups[k] = up; ms[k] = m; }
                if (MODE == kModePlen) {
                    const int cl = cnt[k];
                    const int cn = 1 + (dg == m ? cdg : (up == m ? cup : cl));
                    cdg = cl;
                    cup = cn;
                    cnt[k] = valid ? cn : cl;
                }
                dg = lf;
                up = r;
                col[k] = valid ? r : lf;
            }
        }
        // the row below the lane's last takes this step's value in the next step
        above = __shfl_up_sync(FULL, col[R - 1], 1);
        if (MODE == kModePlen) abovec = __shfl_up_sync(FULL, cnt[R - 1], 1);
        if (puts && valid) {
            if (MODE == kModePlen)
                __stcg(reinterpret_cast<u64*>(hb) + v, pack2(col[R - 1], __int_as_float(cnt[R - 1])));
            else
                __stcg(reinterpret_cast<float*>(hb) + v, col[R - 1]);
        }
        if (TRACK) {
            const float w = pick_row<R>(col, kk);
            const bool less = valid && w < best;
            best = less ? w : best;
            bestj = less ? j : bestj;
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) cost_pair(ynx, q);          // column j + 1
        if (CODES) {
            // "not diag" and "not up" of each row: the sign of m - dg and of
            // m - up (0 when equal, also at +inf: NaN is positive), shifted in
            const int sl = v & (SPW - 1);
#pragma unroll
            for (int k = 0; k < R; ++k) {
                half = __funnelshift_l(__float_as_uint(__fsub_rn(ms[k], dgs[k])), half, 1);
                half = __funnelshift_l(__float_as_uint(__fsub_rn(ms[k], ups[k])), half, 1);
            }
            // (rows of words past the last step do not exist)
            if (sl == SPW - 1 && (FULLBLOCK || v - (SPW - 1) < left)) __stcs(db + (v / SPW) * 32, half);
        }
#pragma unroll
        for (int c = 0; c < D; ++c) ynx[c] = yz[c];
    }
};

template <int D, int R, int MODE, int COST>
__device__ __forceinline__ void lean_band(const DPParams& p, const PairDesc& pd, int band, int lane, uint32_t ring)
{
    using C = Lean<D, R, MODE, COST>;
    constexpr int BR = 32 * R;
    constexpr int SLOT = C::SLOT;
    constexpr int SPW = C::SPW;
    const int M = pd.M, N = pd.N, d = p.d;
    const int i0 = band * BR + lane * R;
    const bool top = band == 0;
    const bool last = band == pd.nbands - 1;
    const float INF = inf_f();

    C st;
#pragma unroll
    for (int q = 0; q < C::Q; ++q)
#pragma unroll
        for (int c = 0; c < D; ++c) {
            const int ia = i0 + 2 * q, ib = ia + 1;
            const float va = (ia < M && c < d) ? __ldg(pd.X + (int64_t)ia * d + c) : 0.f;
            const float vb = (ib < M && c < d) ? __ldg(pd.X + (int64_t)ib * d + c) : 0.f;
            st.bp[q][c] = pack2(va, vb);
        }
#pragma unroll
    for (int k = 0; k < R; ++k) { st.col[k] = INF; st.cnt[k] = 0; }
    st.prev_up = (top && lane == 0) ? 0.f : INF;
    st.prev_upc = 0;
    st.above = INF;
    st.abovec = 0;
    st.half = 0u;
    st.kk = M - 1 - i0;
    st.best = INF;
    st.bestj = 0;
    // above the matrix: +inf (DTW), 0 for Sub-DTW (a path may start in any column)
    st.topv = MODE == kModeSubDirs ? 0.f : INF;
    st.topc = 0;

    char* hrows = static_cast<char*>(p.hbuf);
    const char* hprev = top ? nullptr : hrows + (pd.hbuf_off + (int64_t)(band - 1) * N) * SLOT;
    char* hcur = hrows + (pd.hbuf_off + (int64_t)band * N) * SLOT;
    st.puts = lane == 31 && !last && !p.skip_handoff;
    uint32_t* dout = C::CODES ? p.dirs + pd.dir_off + (int64_t)band * band_dir_words(N, R) + lane : nullptr;
    const int s_end = N + 31;

    float ynext[D];
    auto load_y = [&](int jj) {
#pragma unroll
        for (int c = 0; c < D; ++c) ynext[c] = (jj < N && c < d) ? __ldg(pd.Y + (int64_t)jj * d + c) : 0.f;
    };
    auto put_y = [&](int jj) {
        const int i = jj & 127;
#pragma unroll
        for (int c = 0; c < D; ++c) {
            const uint32_t row = ring + c * kRing * 8;
            const u64 v = pack2(ynext[c], ynext[c]);
            sts64(row + (i < 32 ? i + 128 : i) * 8, v);
            if (i < 36) sts64(row + (i < 32 ? i : i + 128) * 8, v);
        }
    };
    auto load_t = [&](int jj) -> u64 {
        if (jj >= N) return 0;
        if (SLOT == 8) return __ldcv(reinterpret_cast<const u64*>(hprev) + jj);
        return (u64)__float_as_uint(__ldcv(reinterpret_cast<const float*>(hprev) + jj));
    };
    load_y(lane);
    put_y(lane);
    load_y(lane + 32);
    put_y(lane + 32);
    load_y(lane + 64);
    u64 t0 = 0, t1 = 0;              // the row above in the next two blocks of columns
    if (!top) {
        t0 = load_t(lane & 7);
        t1 = load_t(8 + (lane & 7));
    }
    __syncwarp();
    st.yb = ring + (ring_place(0) - lane) * 8;
    {
        u64 yy[D];
        st.load_samples(0, yy);
#pragma unroll
        for (int q = 0; q < C::Q; ++q) st.cost_pair(yy, q);
        st.load_samples(1, st.ynx);
    }

    auto steps = [&](auto track, int s) {
        constexpr bool TRACK = decltype(track)::value;
        if (s >= 31 && s + 8 <= N) {
#pragma unroll
            for (int v = 0; v < 8; ++v) st.template step<true, TRACK>(v, lane, N);
        } else {
#pragma unroll
            for (int v = 0; v < 8; ++v) st.template step<false, TRACK>(v, lane, N);
        }
    };
    for (int s = 0; s < s_end; s += 8) {
        if ((s & 31) == 0 && s > 0 && s < N) {
            __syncwarp();
            put_y(s + lane + 32);
            load_y(s + lane + 64);
            __syncwarp();
        }
        if (!top && s < N) {
            // the row above is taken eight columns at a time, read sixteen steps ahead
            const int jj = s + (lane & 7);
            u64 t = t0;
            if (!wait_filled<32>(jj < N && is_nan_bits((uint32_t)t),
                                 [&]() { t = load_t(jj); return is_nan_bits((uint32_t)t); }, p.hdr, 1, p.spin_limit))
                return;
            st.topv = __uint_as_float((uint32_t)t);
            if (MODE == kModePlen) st.topc = (int)(t >> 32);
            t0 = t1;
            t1 = load_t(jj + 16);
        }
        st.yb = ring + (ring_place(s & ~31) + (s & 31) - lane) * 8;
        st.j0 = s - lane;
        st.left = s_end - s;
        if (C::CODES) st.db = dout + (int64_t)(s / SPW) * 32;
        st.hb = hcur + (int64_t)(s - 31) * SLOT;
        if (MODE == kModeSubDirs && last)
            steps(std::true_type{}, s);
        else
            steps(std::false_type{}, s);
    }

    if (MODE == kModeSubDirs) {
        if (last && lane == (M - 1 - band * BR) / R) {
            if (p.cost_out) p.cost_out[pd.out] = st.best;
            p.bstar_out[pd.out] = st.bestj;
        }
    } else if (last) {
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

template <int D, int R, int MODE, int COST>
__global__ void __launch_bounds__(128, D <= 8 ? 3 : 2) dtw_lean_kernel(DPParams p)
{
    extern __shared__ __align__(16) unsigned char lean_smem[];
    const int lane = threadIdx.x & 31;
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(lean_smem) + (threadIdx.x >> 5) * D * kRing * 8;
    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(&p.hdr->item_counter, 1);
        item = __shfl_sync(FULL, item, 0);
        if (item >= p.n_items) break;
        if (ld_volatile(&p.hdr->abort)) break;
        int q, band;
        item_of<false>(p, item, q, band);
        const PairDesc pd = p.pairs[p.order[q]];
        if (band < pd.nbands) lean_band<D, R, MODE, COST>(p, pd, band, lane, ring);
    }
}

template <int D, int R, int MODE, int COST>
cudaError_t lean_launch_one(const DPParams& p, int grid, int block, cudaStream_t st)
{
    const size_t smem = (size_t)(block / 32) * D * kRing * 8;
    cudaFuncSetAttribute(dtw_lean_kernel<D, R, MODE, COST>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    dtw_lean_kernel<D, R, MODE, COST><<<grid, block, smem, st>>>(p);
    return cudaGetLastError();
}

template <int D, int R, int MODE, int COST>
int lean_occ_one(int block)
{
    int n = 0;
    const size_t smem = (size_t)(block / 32) * D * kRing * 8;
    cudaFuncSetAttribute(dtw_lean_kernel<D, R, MODE, COST>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, dtw_lean_kernel<D, R, MODE, COST>, block, smem);
    return n;
}

// (the l2 norm: codes and cost only)
#define WTS_LEAN_SWITCH(FN, ...)                                                       \
    if (mode == kModeCost) return FN<D, R, kModeCost, COST>(__VA_ARGS__);               \
    if (mode == kModeDirs) return FN<D, R, kModeDirs, COST>(__VA_ARGS__);               \
    if constexpr (COST != kCostL2) {                                                   \
        if (mode == kModePlen) return FN<D, R, kModePlen, COST>(__VA_ARGS__);           \
        if (mode == kModeSubDirs) return FN<D, R, kModeSubDirs, COST>(__VA_ARGS__);     \
    }

template <int D, int R, int COST>
cudaError_t lean_launch_mode(int mode, const DPParams& p, int grid, int block, cudaStream_t st)
{
    WTS_LEAN_SWITCH(lean_launch_one, p, grid, block, st)
    return cudaErrorInvalidValue;
}

template <int D, int R, int COST>
int lean_occ_mode(int mode, int block)
{
    WTS_LEAN_SWITCH(lean_occ_one, block)
    return 0;
}

#undef WTS_LEAN_SWITCH

#define WTS_LEAN_SWITCH_D(FN, ...)                            \
    switch (D) {                                              \
        case 1: return FN<1, R, COST>(__VA_ARGS__);            \
        case 2: return FN<2, R, COST>(__VA_ARGS__);            \
        case 3: return FN<3, R, COST>(__VA_ARGS__);            \
        case 4: return FN<4, R, COST>(__VA_ARGS__);            \
        case 6: return FN<6, R, COST>(__VA_ARGS__);            \
        case 8: return FN<8, R, COST>(__VA_ARGS__);            \
        case 9: return FN<9, R, COST>(__VA_ARGS__);            \
        case 12: return FN<12, R, COST>(__VA_ARGS__);          \
        case 16: return FN<16, R, COST>(__VA_ARGS__);          \
        default: break;                                       \
    }

template <int R, int COST>
cudaError_t lean_launch_set(int mode, int D, const DPParams& p, int grid, int block, cudaStream_t st)
{
    WTS_LEAN_SWITCH_D(lean_launch_mode, mode, p, grid, block, st)
    return cudaErrorInvalidValue;
}

template <int R, int COST>
int lean_occ_set(int mode, int D, int block)
{
    WTS_LEAN_SWITCH_D(lean_occ_mode, mode, block)
    return 0;
}

#undef WTS_LEAN_SWITCH_D

}  // namespace

}  // namespace wts

// Defines the entry points wf_launch_TAG / wf_occ_TAG of one instance set.
#define WTS_LEAN_ENTRY(TAG, R, COST)                                                             \
    namespace wts {                                                                               \
    cudaError_t wf_launch_##TAG(int mode, int D, const DPParams& p, int grid, int block, cudaStream_t st) \
    {                                                                                             \
        return lean_launch_set<R, COST>(mode, D, p, grid, block, st);                            \
    }                                                                                             \
    int wf_occ_##TAG(int mode, int D, int block) { return lean_occ_set<R, COST>(mode, D, block); } \
    }
