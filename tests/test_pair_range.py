"""Which numbers the FP64 collision in FP32 pairs (csrc/pair.cuh) may be given,
compiled for the host: a density that sets a Knudsen number is taken only where
its pair is that density to 2^-47, and refused where it is not finite, not
positive or out of the pairs' range."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include <cmath>
#include <initializer_list>
#include "pair.cuh"
using namespace clb::pr;
int main() {
    for (double v : {0x1p-12, 0x1.8p-12, 0.388, 1.0, 2.47, 0x1.fffffffffffffp29, 0x1.fffffffffffffp-1}) {
        const P p = split(v);
        if (!in_range(v)) return printf("refused %a\n", v), 1;
        if (fabs((double)p.h + (double)p.l - v) > 0x1p-47 * v) return printf("split %a\n", v), 1;
    }
    for (double v : {(double)NAN, -(double)NAN, (double)INFINITY, -(double)INFINITY, 0.0, -0.0, -1.0, -1e-3, 1e40, -1e40,
                     1e300, 1e-300, 5e-324, 0x1.fffffffffffffp-13, 0x1p31})
        if (in_range(v)) return printf("took %g\n", v), 1;
    return 0;
}
"""


def compile_and_run(source, tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(source)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_1603_01955_gb300", "csrc"), str(src), "-o", str(exe), "-lm"], check=True)
    return subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)


def test_densities_taken(tmp_path):
    r = compile_and_run(SOURCE, tmp_path)
    assert r.returncode == 0, r.stdout
