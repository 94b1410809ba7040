"""The host's count of the pairs that blocks and windows force, compiled from the library's source: against a
count row by row, and at a cost that does not grow with the number of blocks."""
import os
import subprocess

from conftest import ROOT

MAIN = r"""
#include <algorithm>
#include <cstdint>
%s
int64_t by_rows(int64_t N, int64_t block, int64_t W)
{
    int64_t total = 0;
    for (int64_t i = 0; i < N; ++i) {
        int64_t lo = std::max<int64_t>(0, i - std::max<int64_t>(W, 1) + 1);
        if (block > 0) lo = std::min(lo, i / block * block);
        total += i - lo + 1;
    }
    return total;
}
int main()
{
    for (int64_t N = 1; N <= 40; ++N)
        for (int64_t block = 0; block <= 45; ++block)
            for (int64_t W = 0; W <= 45; ++W)
                if (suffix_pairs_of(N, block, W) != by_rows(N, block, W)) return 1;
    if (suffix_pairs_of(5000, 700, 300) != by_rows(5000, 700, 300)) return 2;
    for (int k = 0; k < 50; ++k)
        if (suffix_pairs_of(2147483647, 1, 1 + (k & 1)) != 2147483647LL + (k & 1) * 2147483646LL) return 3;
    return 0;
}
"""


def test_forced_pairs_in_closed_form(tmp_path):
    src = open(os.path.join(ROOT, "paper_2607_21927_gb300", "csrc", "ris_api.cu")).read()
    code = src[src.index("int64_t range_sum("):src.index("// Design of a layer call: 0 register gather")]
    (tmp_path / "t.cpp").write_text(MAIN % code)
    subprocess.run(["g++", "-O2", "-std=c++17", "-o", tmp_path / "t", tmp_path / "t.cpp"], check=True)
    assert subprocess.run([tmp_path / "t"], timeout=20).returncode == 0
