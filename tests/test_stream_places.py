"""Places of a block's rows in the factor streams are int32: row numbers reach every
block an int32 can number, byte offsets are refused where they would wrap.  A small C++ program compiled here includes
the library's own header and prints both sides of each bound."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "internal.h"
namespace gemslr {
void fail(gemslr_status st, const std::string &msg) { throw Error{st, msg}; }
}
int main() {
    const long long last = 2147483647ll;
    const long long asked[][2] = {{0, 16}, {last, 1}, {last + 1, 1}, {last / 8, 8}, {last / 8 + 1, 8},
                                  {last / 16, 16}, {last / 16 + 1, 16}, {last / 4 + 1, 4}};
    for (auto &a : asked) {
        try {
            std::printf("%d\n", (int)gemslr::vector_place(a[0], a[1]));
        } catch (const gemslr::Error &e) {
            std::printf("%s\n", e.st == GEMSLR_ERR_UNSUPPORTED ? "unsupported" : "other");
        }
    }
    return 0;
}
"""


def test_places_cover_int32_rows_and_never_wrap(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "places.cpp", tmp_path / "places"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2205_03224_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    last = 2**31 - 1
    assert out == ["0", str(last), "unsupported", str(last // 8 * 8), "unsupported", str(last // 16 * 16),
                   "unsupported", "unsupported"]
