"""The level-2 kernel's share of a row's columns (csrc/l2_columns.cuh), gone through
on the host for every padded sketch size and thread: each row group reads every pair
of neighbouring columns exactly once, and nothing past the row."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_05865_gb300", "csrc")

PROGRAM = """
#include "l2_columns.cuh"
#include <cstdio>
template <int SP> void go() {
    using C = msp::L2Columns<SP, 512>;
    for (int t = 0; t < 512; ++t)
        for (int k = 0; k < C::per_thread; ++k)
            if (C::active(t) && C::has(C::first(t), k))
                std::printf("%d %d %d\\n", SP, C::group(t), C::first(t) + 512 * k);
}
int main() {
    go<128>(); go<256>(); go<384>(); go<512>(); go<640>(); go<768>(); go<896>(); go<1024>(); go<1536>(); go<2048>();
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_every_pair_once_and_none_past_the_row(tmp_path):
    src, exe = tmp_path / "go.cpp", tmp_path / "go"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    seen = {}
    for line in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n"):
        if line:
            sp, group, pair = map(int, line.split())
            seen.setdefault(sp, {}).setdefault(group, []).append(pair)
    assert sorted(seen) == [128, 256, 384, 512, 640, 768, 896, 1024, 1536, 2048]
    for sp, groups in seen.items():
        assert sorted(groups) == list(range(max(1, 512 // (sp // 2))))
        for pairs in groups.values():
            assert sorted(pairs) == list(range(sp // 2)), sp
