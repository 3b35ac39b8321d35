"""The radix sort's block rule on the host, for several SM counts: the blocks a
sort takes never exceed what grid and look-back words are sized for, and a sort
that fits one wave of the device takes one."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_08551_gb300", "csrc")

MAIN = """
#include <cstdio>
#include "sort_plan.cuh"
using namespace gi;
int main() {
    const int waves[] = {1, 7, 108, 148, 152, 160, 304};
    for (int wave : waves) {
        const int64_t w = int64_t(wave) * kSortThreads;
        auto check = [&](int64_t K, int64_t capacity) {
            if (K < 1 || K > capacity || capacity >= (int64_t(1) << 30)) return;
            const int items = sort_items((int)K, wave);
            const int64_t blocks = (K + kSortThreads * items - 1) / (kSortThreads * items);
            if (items < 4 || items > kSortMaxItems) std::printf("items %d at K %lld\\n", items, (long long)K);
            if (blocks > sort_blocks(capacity, wave))
                std::printf("wave %d K %lld capacity %lld: %lld blocks > %lld\\n", wave, (long long)K, (long long)capacity,
                            (long long)blocks, (long long)sort_blocks(capacity, wave));
            if (K <= kSortMaxItems * w && blocks > wave) std::printf("wave %d K %lld: %lld blocks\\n", wave, (long long)K, (long long)blocks);
        };
        for (int64_t f = 1; f <= 200; ++f)
            for (int64_t d = -1; d <= 1; ++d)
                for (int64_t extra : {int64_t(0), int64_t(1), 3 * w, 40 * w}) check(f * w + d, f * w + d + extra);
        for (int64_t K = 1; K < (int64_t(1) << 30); K = K * 9 / 8 + 1) {
            check(K, K);
            check(K, (int64_t(1) << 30) - 1);
        }
    }
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no g++")
def test_blocks_fit_and_one_wave_suffices(tmp_path):
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = tmp_path / "main"
    subprocess.run(["g++", "-std=c++17", "-O1", "-x", "c++", "-I", CSRC, str(tmp_path / "main.cpp"), "-o", str(exe)],
                   check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout == ""
