"""The choice among the grouped INT4 second kernels' plans (csrc/w4a4_plan.h), compiled as plain C++: what each value of dirotq_set_gemm_tile means
for these kernels, and over calls of all sizes a plan that exists, that groups of the call's size have, and that leaves no row block of a tile idle."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "w4a4_plan.h"
#include <stdio.h>
#include <stdlib.h>
using namespace dirotq;

#define CHECK(c) do { if (!(c)) { printf("line %d: %s (M = %d, N = %d, K_lp = %d, G = %d: %d)\n", __LINE__, #c, M, N, K, G, plan); exit(1); } } while (0)

int main() {
    int M = 0, N = 0, K = 0, G = 0, plan = 0;
    // a value that names no plan of these kernels leaves them choosing for themselves
    CHECK(w4a4_forced_plan(0) == 0 && w4a4_forced_plan(512) == 0);
    for (const int p : {32, 64, 66, 128, 130, 192, 256, 258}) CHECK(w4a4_forced_plan(p) == p);
    for (const int p : {-1, 1, 34, 96, 132, 194, 260, 384, 514, 1024}) CHECK(w4a4_forced_plan(p) == -1);
    long chosen[1024] = {};
    for (M = 1; M <= 70000; M = M < 300 ? M + 1 : M * 9 / 8 + 1)
        for (N = 16; N <= 24576; N += N < 512 ? 16 : 400)
            for (K = 128; K <= 15360; K = K * 3 / 2 / 64 * 64)
                for (G = 64; G <= 128; G += 64) {
                    plan = choose_w4a4_plan(M, N, K, G, 148);
                    CHECK(w4a4_plan_exists(plan) && plan != 66);  // (66 adds in another order)
                    CHECK(plan != 32 || G == 64);
                    CHECK(M > 128 || N > 12288 || (plan != 130 && plan != 258));  // the second 128 rows would be idle
                    ++chosen[plan];
                }
    for (const int p : {32, 64, 128, 130, 192, 256, 258}) { plan = p; CHECK(chosen[p] > 0); }
    plan = choose_w4a4_plan(M = 2147483647, N = 24576, K = 3072, G = 64, 148);
    CHECK(w4a4_plan_exists(plan));
    return 0;
}
"""


def test_rule(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-fsanitize=undefined", "-fno-sanitize-recover",
                           "-I", os.path.join(ROOT, "paper_2605_16732_b200", "csrc"), str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
