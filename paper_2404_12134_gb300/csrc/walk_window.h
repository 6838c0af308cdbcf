// The window of direction words that a walk reads: where a cell's word lies in
// it and where the walk may go without a check.  Plain C++ for host and device.
#pragma once

#ifdef __CUDACC__
#define WTS_HD __host__ __device__ __forceinline__
#else
#define WTS_HD inline
#endif

namespace wts {

constexpr int kBtWords = 4096;   // 16 KB of direction words cached per warp

template <int R>
struct WalkWindow {
    static constexpr int W = R >= 16 ? R / 16 : 1;         // words per (word row, lane)
    static constexpr int SPW = R >= 16 ? 1 : 32 / (2 * R); // steps per word row
    static constexpr int LOG_R = R == 4 ? 2 : (R == 8 ? 3 : (R == 16 ? 4 : 5));
    static constexpr int ROWS = kBtWords / (32 * W);       // word rows of one band in the window

    // Word of lane t at step s, s counted from the window's first step (an
    // absolute step times the words of a word row leaves 32 bits in cycles that
    // are accepted).
    static WTS_HD int word(int s, int t) { return ((int)((unsigned)s / SPW) * 32 + t) * W; }

    // From row i, column first + j on (first: the window's first step), 16 moves on
    // the diagonal, 8 up or 8 left stay in the window, above row floor and right
    // of column 0.
    static WTS_HD bool inside(int i, int j, int first, int floor)
    {
        return i >= floor + 16 && j >= 17 - first && j + ((i >> LOG_R) & 31) >= 21;
    }
};

}  // namespace wts
