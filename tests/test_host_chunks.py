"""The host side of dirotq_linear_host (csrc/host_chunks.h), compiled as plain C++ and run against a recorder in the place of the device:
every row is in exactly one chunk, the number of chunks fits the event tables, each chunk is copied in, computed and copied out in
that order, and a call that fails at any step is still joined, last, exactly once."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "host_chunks.h"
#include <stdio.h>
#include <stdlib.h>
#include <vector>
using namespace dirotq;

#define CHECK(c) do { if (!(c)) { printf("line %d: %s (M = %d)\n", __LINE__, #c, M); exit(1); } } while (0)

struct Recorder {  // fails at step `fail` (counted from 0 over fork, copies and computations); -1: never
    int fail, step = 0, joined = 0, m = 0;
    bool join_ok = true, after_join = false;
    std::vector<int> log;
    bool did(int what) {
        if (joined) after_join = true;
        log.push_back(what);
        return step++ != fail;
    }
    bool fork() { return did(0); }
    bool copy_in(int c, int m0, int rows) { if (m0 != m) exit(2); m += rows; (void)c; return did(1); }
    bool compute(int, int, int) { return did(2); }
    bool copy_out(int, int, int) { return did(3); }
    bool join(bool) { ++joined; return join_ok; }
};

int main() {
    const size_t widths[] = {16, 64, 512, 1152, 3072, 9216, 12288, 65536};
    std::vector<long> sizes;
    for (long M = kMinPipelinedRows; M < 6000; ++M) sizes.push_back(M);
    for (long M = 6000; M < 2000000000l; M = M * 17 / 16 + 1) sizes.push_back(M);
    sizes.push_back(2147483647l);
    for (long big : sizes)
        for (size_t K : widths)
            for (size_t N : widths) {
                const int M = (int)big;
                int rows[kMaxHostChunks + 8];
                for (int& r : rows) r = -7;
                const int n = plan_host_chunks(M, 2 * K, 2 * N, rows);
                CHECK(n >= 1 && n <= kMaxHostChunks && rows[kMaxHostChunks] == -7);
                long sum = 0;
                for (int c = 0; c < n; ++c) { CHECK(rows[c] >= 1 && (rows[c] >= 128 || n == 1 || c == n - 1)); sum += rows[c]; }
                CHECK(sum == M);
            }
    const int M = 5000;
    int rows[kMaxHostChunks];
    const int n = plan_host_chunks(M, 6144, 6144, rows), steps = 1 + 3 * n;
    CHECK(n > 3);
    for (int fail = -1; fail < steps; ++fail) {
        Recorder r{fail};
        const bool ok = run_host_chunks(rows, n, r);
        CHECK(ok == (fail < 0) && r.joined == 1 && !r.after_join);
        CHECK((int)r.log.size() == (fail < 0 ? steps : fail + 1));  // nothing is enqueued after a failure
        for (int i = 1; i < (int)r.log.size(); ++i) CHECK(r.log[i] == 1 + (i - 1) % 3);
    }
    Recorder bad{-1};
    bad.join_ok = false;
    CHECK(!run_host_chunks(rows, n, bad));
    return 0;
}
"""


def test_chunks_and_their_order(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-fsanitize=undefined", "-fno-sanitize-recover",
                           "-I", os.path.join(ROOT, "paper_2605_16732_b200", "csrc"), str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
