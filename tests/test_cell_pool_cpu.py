"""The pool of the located search's long candidate lists, on the CPU: the cursor's own type
and test from the library's header hand out words to more bins than 2^32 words would
serve, and no two lists may share a word.
"""
import os
import subprocess
import tempfile

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#define __host__
#define __device__
#define __align__(n) alignas(n)
#include <cstdio>
#include "qt_internal.h"
int main()
{
    // 800 grids of 104 x 104 bins, every bin with all 1024 points: 8.9e9 words asked for
    qt::DevStatus st{};
    const uint32_t cap = 104u * 104u * 800u / 4u + 65536u;
    unsigned long long top = 0, lists = 0, shared = 0;
    for (long long bin = 0; bin < 104ll * 104 * 800; ++bin) {
        const uint32_t cnt = 1024;
        const unsigned long long off = st.cell_cursor;
        st.cell_cursor += cnt;
        if (!qt::pool_holds(off, cnt, cap)) continue;
        if (off < top) ++shared;
        top = off + cnt;
        ++lists;
    }
    std::printf("%llu %llu %llu\n", lists, shared, (unsigned long long)cap / 1024);
    return 0;
}
"""


def test_no_two_lists_share_a_word():
    with tempfile.TemporaryDirectory() as td:
        src, exe = os.path.join(td, "pool.cpp"), os.path.join(td, "pool")
        with open(src, "w") as f:
            f.write(SRC)
        subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1101_3228_gb300", "csrc"), src, "-o",
                        exe], check=True)
        lists, shared, most = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert shared == 0 and lists == most
