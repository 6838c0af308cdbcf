"""The backtrack's window arithmetic (csrc/walk_window.h), compiled for the host
with signed overflow trapped: over the whole range of accepted cycle lengths the
cells that the unchecked walk reads lie in the loaded window, at the word where
the checked walk finds them.  No GPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdint>
#include <cstdio>
#include <random>
#include "walk_window.h"

template <int R>
int check()
{
    using V = wts::WalkWindow<R>;
    std::mt19937_64 rng(R);
    const int N = 1 << 30, BR = 32 * R;
    int seen = 0;
    for (int trial = 0; trial < 400000; ++trial) {
        // the window: up to ROWS word rows that end with the cell's own
        const int band = (int)(rng() % 3);
        const int i = band * BR + (int)(rng() % BR);
        int span = 2 << (rng() % 30);
        if (span > N) span = N;
        const int j = N - 1 - (int)(rng() % span);
        const int t = (i >> V::LOG_R) & 31;
        const int whi = (j + t) / V::SPW;
        const int wlo = whi - V::ROWS + 1 > 0 ? whi - V::ROWS + 1 : 0;
        // a cell walked on to within it, and the first row that may be left
        const int jj = j - (int)(rng() % (V::ROWS * V::SPW));
        const int floor = band * BR + (int)(rng() % BR / 2);
        if (jj < 0 || (jj + t) / V::SPW < wlo) continue;
        if (!V::inside(i, jj - wlo * V::SPW, wlo * V::SPW, floor)) continue;
        ++seen;
        for (int lane = 0; lane < 32; ++lane) {
            const int kind = lane < 16 ? 0 : (lane < 24 ? 1 : 2);
            const int u = lane - (kind == 0 ? 0 : (kind == 1 ? 16 : 24));
            const int iu = i - (kind != 2 ? u : 0), ju = jj - (kind != 1 ? u : 0);
            if (iu - 1 < floor || iu / BR != band || ju < 1) return std::printf("R=%d cell (%d, %d)\n", R, iu, ju), 1;
            const int tt = (iu >> V::LOG_R) & 31;
            const int64_t row = (int64_t)(ju + tt) / V::SPW;
            if (row < wlo || row > whi) return std::printf("R=%d row %lld\n", R, (long long)row), 1;
            const int64_t want = ((row - wlo) * 32 + tt) * V::W;
            if (V::word(ju + tt - wlo * V::SPW, tt) != want || want + V::W > wts::kBtWords)
                return std::printf("R=%d word\n", R), 1;
        }
    }
    return seen > 1000 ? 0 : (std::printf("R=%d: %d cells\n", R, seen), 1);
}

int main() { return check<4>() | check<8>() | check<16>() | check<32>(); }
"""


def test_unchecked_walk_stays_in_the_window(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O1", "-std=c++17", "-fsanitize=signed-integer-overflow",
                    "-fsanitize-undefined-trap-on-error", "-I",
                    os.path.join(ROOT, "paper_2404_12134_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout)
