"""Host check of the rule that ends the solvers' device loop (csrc/plq_loop.h, compiled
here by the host compiler): a loop whose right-hand sides never stop ends after maxit
iterations, and one whose right-hand sides stop by then is never cut short."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "plq_loop.h"
int main() {
    const int caps[] = {-1, 0, 1, 2, 3, 4, 5, 17, 20000};
    for (int maxit : caps) {
        // no right-hand side ever stops
        unsigned done = 0;
        while (!plq::loop_over(++done, maxit, false))
            if (done > 100000u) { std::printf("FAIL endless at maxit %d\n", maxit); return 1; }
        if (done != (unsigned)(maxit < 1 ? 1 : maxit)) { std::printf("FAIL %d ends after %u\n", maxit, done); return 1; }
        // a right-hand side with `before` iterations from earlier loops stops at maxit
        for (int before = 0; before < maxit && before < 40; ++before) {
            int iter = before;
            done = 0;
            bool over = false;
            while (!over) {
                const bool stopped = ++iter >= maxit;
                over = plq::loop_over(++done, maxit, stopped);
                if (over != stopped) { std::printf("FAIL cut at %d of %d\n", iter, maxit); return 1; }
            }
        }
    }
    if (!plq::loop_over(0x80000000u, 0x7fffffff, false) || plq::loop_over(0x7ffffffeu, 0x7fffffff, false)) return 2;
    std::printf("ok\n");
    return 0;
}
"""


def test_device_loop_ends_after_maxit_iterations(tmp_path):
    src = tmp_path / "loop_check.cpp"
    exe = tmp_path / "loop_check"
    src.write_text(PROGRAM)
    inc = os.path.join(ROOT, "paper_1405_0700_gb300", "csrc")
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-I" + inc, str(src), "-o", str(exe)], capture_output=True,
                       text=True)
    if r.returncode != 0:
        pytest.fail(r.stderr)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and out.stdout.startswith("ok"), out.stdout + out.stderr
