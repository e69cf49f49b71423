"""The count buffer of the radix sort is allocated once, for the largest sort a
context can hold, and used by sorts of every smaller size: radix_counts(N) has
to cover radix_geom(nt).counts() for all nt <= N, over every number of tiles
that int32 indices allow."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1809_08013_gb300", "csrc")
SRC = r"""
#include <stdio.h>
#include "radix_geom.cuh"
using namespace sph;
int main() {
    long long bad = 0, most = 0;
    auto at = [&](int64_t first, int64_t last) {  // the key counts first to last share one tiling
        const long long c = radix_geom(last).counts();
        if (c > most) most = c;
        // the smallest capacity that holds `first` keys holds all smaller sorts too
        if (radix_counts(first) < most && bad++ == 0)
            printf("capacity %lld: %lld counts a pass, %lld used\n", (long long)first,
                   (long long)radix_counts(first), most);
    };
    const int64_t small = (int64_t)kRadixThreads * kRadixItemsSmall;
    const int64_t large = (int64_t)kRadixThreads * kRadixItems;
    for (int64_t n = 1; n <= kRadixSmallN; n += small) at(n, n + small - 1);
    for (int64_t n = kRadixSmallN + 1; n < ((int64_t)1 << 20) * large;) {
        const int64_t last = (n + large - 1) / large * large;
        at(n, last);
        n = last + 1;
    }
    printf("%lld\n", bad);
    return bad != 0;
}
"""


def test_count_buffer_covers_every_smaller_sort(tmp_path):
    src, exe = tmp_path / "r.cpp", tmp_path / "r"
    src.write_text(SRC)
    subprocess.check_call(["g++", "-std=c++17", "-x", "c++", "-I", CSRC, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
