"""asked_once (ppd_kernels.h), which keeps the device's answers that the attention's
plans need: an answer is kept, a query that failed is not (no GPU needed)."""
import os
import subprocess

from paper_2405_18628_gb300 import build

PROGRAM = r"""
#include "ppd_kernels.h"
#include <cstdio>
int main()
{
    std::atomic<int> slot{0};
    int calls = 0;
    const int answers[] = {-1, -1, 36, 7};
    for (int i = 0; i < 4; ++i) {
        const int n = ppd::asked_once(slot, [&] { return answers[calls++]; });
        std::printf("%d ", n);
    }
    std::atomic<int> none{0};   // an answer of 0 is an answer
    for (int i = 0; i < 2; ++i) (void)ppd::asked_once(none, [&] { ++calls; return 0; });
    std::printf("%d\n", calls);
}
"""


def test_a_failed_query_is_asked_again(tmp_path):
    src, exe = tmp_path / "asked.cu", tmp_path / "asked"
    src.write_text(PROGRAM)
    subprocess.run([build.nvcc(), "-std=c++17", "-I", build.CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert out == ["0", "0", "36", "36", "4"]   # two failures, one answer, one answer of 0
