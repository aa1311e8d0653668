"""Index steps near the ends of the int32 range (compiled for the host; no matrix of that size is made)."""
from __future__ import annotations

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_02207_gb300", "csrc")

PROGRAM = r"""
#include <climits>
#include <cstdio>
#include <initializer_list>
#include "index_range.h"
using namespace ll;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
// every row has `per` entries; an index outside [0, n] is a fault
struct Even {
    long long n; int per; bool* bad;
    int operator[](int i) const { if (i < 0 || i > n) { *bad = true; return 0; } return (int)((long long)i * per); }
};
int main() {
    for (int end : {0, 1, 7, INT_MAX - 1, INT_MAX}) {
        for (int step : {1, 2, 12, 32, 64}) {
            CHECK(step_to(end, step, end) == end);
            for (int back = 0; back <= 3 * step && back <= end; ++back) {
                int k = end - back, trips = 0;
                for (; k < end; k = step_to(k, step, end)) ++trips;   // ends, and visits every batch
                CHECK(k == end && trips == (back + step - 1) / step);
                CHECK(step_to(end - back, step, end) >= end - back);
            }
        }
    }
    for (int n : {1, 2, 1000, (1 << 30) + 5, INT_MAX}) {
        for (int per : {0, 1}) {
            bool bad = false;
            const Even rp{n, per, &bad};
            const long long total = (long long)n * (per + 7);
            for (int w = 0; w <= 8; ++w) {
                const long long t = total / 8 * w + (w < total % 8 ? w : total % 8);
                const int i = rows_start(rp, n, 7, t);
                CHECK(i >= 0 && i <= n && (long long)i * (per + 7) >= t && (i == 0 || (long long)(i - 1) * (per + 7) < t));
            }
            CHECK(!bad);
        }
    }
    return 0;
}
"""


def test_index_steps_stay_in_range(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-fsanitize=signed-integer-overflow", "-fno-sanitize-recover=all", "-I", CSRC, str(src), "-o",
                    str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr

