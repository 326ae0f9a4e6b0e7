"""The wrap test of the push kernel's window words, compiled for the host with signed overflow trapped."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_wraps_are_found_without_signed_overflow(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    text = open(os.path.join(ROOT, "paper_1008_1685_gb300", "csrc", "k_push.cu")).read()
    body = re.search(r"__device__ __forceinline__ (int win_wrapped\(int old, int t\) \{.*?\n\})", text, re.S).group(1)
    edge = [0, 1, 2, 3, 2**30, 2**30 + 1, 2**31 - 2, 2**31 - 1]
    edge = sorted({s * v + d for v in edge for s in (1, -1) for d in (-1, 0, 1) if -(2**31) <= s * v + d < 2**31} | {-(2**31)})
    src = tmp_path / "w.cpp"
    src.write_text("#include <cstdio>\n#include <cstdlib>\n" + body + """
int main(int argc, char** argv) {
    for (int i = 1; i < argc; ++i)
        for (int j = 1; j < argc; ++j)
            std::printf("%d\\n", win_wrapped(static_cast<int>(std::atoll(argv[i])), static_cast<int>(std::atoll(argv[j]))) < 0);
}
""")
    exe = tmp_path / "w"
    subprocess.run([cxx, "-O2", "-std=c++17", "-fsanitize=signed-integer-overflow", "-fsanitize-undefined-trap-on-error", str(src),
                    "-o", str(exe)], check=True)
    out = subprocess.run([str(exe), *map(str, edge)], check=True, capture_output=True, text=True).stdout.split()
    assert [int(v) for v in out] == [int(not -(2**31) <= a + b < 2**31) for a in edge for b in edge]
