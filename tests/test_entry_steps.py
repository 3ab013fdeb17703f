"""Walks of the mode passes over the last items of the largest tensors (2^31 - 1 entries), on
the host: the functions the kernels step with, in the kernels' loops, under the compiler's
check for signed overflow.  Every entry is met once and none past the end."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1410_5209_gb300", "csrc")

SRC = r"""
#include <stdio.h>
#include <stdlib.h>
#include <vector>
#include "entry_steps.h"
using namespace tfs;
static int64_t lo, hi;
static std::vector<int> met;
static void meet(int j) {
    if (j < lo || j >= hi) { printf("entry %d outside %lld..%lld\n", j, (long long)lo, (long long)hi); exit(1); }
    ++met[(size_t)(j - lo)];
}
static void all_met(const char *walk) {
    for (int &m : met) {
        if (m != 1) { printf("%s: an entry of %lld..%lld met %d times\n", walk, (long long)lo, (long long)hi, m); exit(1); }
        m = 0;
    }
}
int main() {
    for (int64_t end : {(int64_t)2147483647, (int64_t)2147483647 - 33, (int64_t)1000})
        for (int len = 0; len < 300; ++len) {
            lo = end - len, hi = end;
            met.assign((size_t)len, 0);
            const tf_item item = {lo, len, 0, 0, 0};
            // a lane per entry, steps of 32 (mode_pass.cuh, tma_pass.cuh)
            for (Step s = first_step(item, 0);; s = step_on(s)) {
                for (int lane = 0; lane < 32; ++lane)
                    if (has_entry(s.j0, lane, s.jend)) meet(s.j0 + lane);
                if (s.flags & 4) break;
            }
            all_met("steps of 32");
            // four entries a lane, steps of 128 (k_pass_one)
            int j0 = (int)item.begin;
            const int e = (int)(item.begin + item.len);
            while (j0 < e) {
                for (int lane = 0; lane < 32; ++lane)
                    for (int u = 0; u < 4; ++u)
                        if (has_entry(j0, u * 32 + lane, e)) meet(j0 + (u * 32 + lane));
                if (last_step(j0, 128, e)) break;
                j0 += 128;
            }
            all_met("steps of 128");
            // the next step's entries loaded ahead (k_pass_mma)
            for (int step : {8, 16}) {
                int j = (int)item.begin, jend = (int)(item.begin + item.len);
                auto load = [&](int at) {
                    for (int k = 0; k < step; ++k)
                        if (has_entry(at, k, jend)) meet(at + k);
                };
                load(j);
                for (;;) {
                    const bool last = last_step(j, step, jend);
                    const int next = last ? jend : j + step;
                    load(next);
                    if (last) break;
                    j = next;
                }
                all_met("steps loaded ahead");
            }
        }
    printf("ok\n");
}
"""


def test_walks_end_with_the_item(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ missing")
    src, exe = tmp_path / "walk.cpp", tmp_path / "walk"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=signed-integer-overflow",
                    "-fno-sanitize-recover", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
