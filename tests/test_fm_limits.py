"""The FM search's limits (csrc/fm_limits.h), compiled for the host."""
import os
import shutil
import subprocess

import pytest

from paper_1012_0006_gb300.build import CSRC


def _run(tmp_path, body):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include "fm_limits.h"\n#include <cstdio>\n#include <initializer_list>\nusing namespace fr;\n'
                   '#define REQUIRE(x) if (!(x)) { std::printf("line %d: %s\\n", __LINE__, #x); return 1; }\n'
                   "int main() {\n" + body + "\nreturn 0; }\n")
    subprocess.run([cxx, "-std=c++17", "-O1", "-fsanitize=undefined", "-fno-sanitize-recover", "-I", CSRC, str(src),
                    "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


def test_a_row_of_two_entries_is_no_longer_than_a_row(tmp_path):
    _run(tmp_path, """
    // rows of 0 to 1,023 arcs; every begin with every end
    const int big = INT_MAX - 65;
    const int row[][3] = {{0, 1023, 5000}, {1023, 1023, 5000}, {1023, 1024, 5000}, {3000, 4023, 5000}, {4977, 5000, 5000},
                          {0, 7, big}, {big - 1023, big, big}, {big - 1, big, big}, {1 << 30, (1 << 30) + 40, big}};
    for (auto &b : row)
        for (auto &e : row) {
            if (b[2] != e[2]) continue;
            const int end = fm_row_end(b[0], e[1], b[2]);
            REQUIRE(end <= b[2] && end <= e[1]);
            REQUIRE((long long)end - b[0] <= kFmMaxDeg);
            if (&b == &e) REQUIRE(end == e[1]);
        }
    """)


def test_entries_are_counted_in_32_bits(tmp_path):
    _run(tmp_path, """
    const long long most = INT_MAX;
    for (long long n : {1LL, 1000LL, 1LL << 20, most / 2, most}) {
        // the largest graph that fits: its last entry + 1, and 32 positions past it, are ints
        const long long nnz = most - 64 - n;
        if (nnz >= 0) {
            REQUIRE(fm_entries_fit(n, nnz));
            const int end = (int)(n + nnz);
            REQUIRE(end + 32 > end && end + 1 > 0);
        }
        REQUIRE(!fm_entries_fit(n, nnz + 1));
        REQUIRE(!fm_entries_fit(n, most));
    }
    REQUIRE(fm_entries_fit(1 << 30, (1 << 30) - 65));
    """)
