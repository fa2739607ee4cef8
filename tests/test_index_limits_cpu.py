"""Index arithmetic of the solve kernels at the largest sizes a plan accepts, with the
kernels' own helpers compiled for the host."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1710_04985_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "cursor.h"
#include "sptrsv.h"
using namespace sptrsv;
typedef long long ll;

static int bad = 0;
static void check(bool ok, const char* what, ll a, ll b) {
    if (!ok) {
        std::printf("%s %lld %lld\n", what, a, b);
        bad = 1;
    }
}

// a lane of the last row (1 to 40 entries, the last stored one at the limit) while the
// warp goes through the chunks of a row of `longest` entries
static void cursor(int lanes, int slots, int len, int longest) {
    const int end = SPTRSV_MAX_SIZE, step = lanes * slots;
    for (int sl = 0; sl < lanes; ++sl) {
        int q = end - len + sl;
        for (ll at = 0; at < longest; at += step) {
            const ll furthest = (ll)q + step + lanes * (slots - 1);  // of the chunk ahead
            check(furthest <= end + (ll)kCursorAhead && furthest <= 2147483647ll, "entry index",
                  furthest, lanes);
            // inside the row the cursor is where the chunk number says
            const ll want = (ll)end - len + sl + at;
            check(want >= end ? q >= end : q == want, "cursor", q, want);
            q = advance(q, step, end);
        }
    }
}

// the windows of the last rows of a system of n rows: all of them, each once
static void windows(int rows, int n) {
    int base = n - n % rows - 3 * rows, seen = 0, count = 0;
    if (base < 0) base = 0;
    const int from = base;
    for (; base < n; base = next_window(base, rows, n)) {
        check(count == 0 || (base - from) % rows == 0, "window", base, n);
        seen += n - base < rows ? n - base : rows;
        if (++count > 5) break;
    }
    check(base == n && seen == n - from, "windows", base, seen);
}

int main() {
    for (int rows : {12288, 24576})
        for (int less : {0, 1, 255, 12287, 12288, 12289, 24576}) {
            windows(rows, SPTRSV_MAX_SIZE - less);
            windows(rows, less + 1);
        }
    for (int lanes = 1; lanes <= 32; lanes *= 2)
        for (int len = 1; len <= 40; ++len) cursor(lanes, lanes >= 16 ? 2 : 4, len, 5000);
    return bad;
}
"""


@pytest.fixture(scope="module")
def answer(tmp_path_factory):
    cc = shutil.which("g++")
    if cc is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("limits")
    (d / "p.cpp").write_text(PROGRAM)
    r = subprocess.run([cc, "-std=c++17", "-Wall", "-Werror", "-fsanitize=signed-integer-overflow",
                        "-fno-sanitize-recover=all", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                        str(d / "p.cpp"), "-o", str(d / "p")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return subprocess.run([str(d / "p")], capture_output=True, text=True)


def test_helpers_stay_inside_int(answer):
    assert answer.returncode == 0, answer.stdout + answer.stderr


def test_windows_are_stepped_by_the_helper():
    text = open(os.path.join(CSRC, "solve_cluster.cu")).read()
    assert not re.search(r"base \+=|base \+ H", text)


def test_chunks_of_a_warp_are_stepped_by_the_helper():
    """In the kernels whose lanes go through chunks as long as the longest row."""
    for name in ("solve_self.cu", "solve_cluster.cu"):
        text = open(os.path.join(CSRC, name)).read()
        free = text[text.index("self_solve_k1(const" if name == "solve_self.cu" else
                               "cluster_solve_k1(const"):]
        steps = [ln.strip() for ln in free.splitlines() if re.search(r"q0 \+= W \* E", ln)]
        # the one that is left belongs to rows that each have more of their own
        assert steps == ([] if name == "solve_self.cu" else ["q0 += W * E;"]), (name, steps)
