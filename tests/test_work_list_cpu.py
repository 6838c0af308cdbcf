"""The bound of a grouped work list (csrc/work_list.h), compiled for the host:
the item cursor, which every resident warp moves once past the list's end, stays
in 31 bits for every list that is accepted.  No GPU."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "work_list.h"

int main()
{
    // pairwise lists (T <= 4,096 cycles, bands of the longest) next to 2^31 items
    long near = 0;
    for (int64_t T = 2; T <= 4096; ++T) {
        const int64_t P = T * (T - 1) / 2, top = ((int64_t)1 << 31) / P;
        for (int64_t nb = top > 1 ? top - 1 : 1; nb <= top + 1; ++nb)
            for (int64_t warps : {1, 608, 1824, 2432, 9728}) {
                if (!wts::grouped_list_fits(P, nb, warps)) continue;
                near += P * nb > ((int64_t)1 << 31) - 20000;
                if (P * nb + warps > INT32_MAX)
                    return std::printf("%lld pairs x %lld\n", (long long)P, (long long)nb), 1;
            }
    }
    // ordinary lists are grouped
    if (!wts::grouped_list_fits(120, 196, 1824) || !wts::grouped_list_fits(499500, 782, 1824)) return 2;
    return near > 0 ? 0 : 3;
}
"""


def test_cursor_of_a_grouped_list(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_2404_12134_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout)
