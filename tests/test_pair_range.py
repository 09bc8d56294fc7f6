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


CONSTANTS = r"""
#include <cstdio>
#include <cmath>
#include <initializer_list>
#include "pair.cuh"
using namespace clb::pr;
// The increments with launch constants from every Knudsen number whose constants
// fit, against long double: the rates' error, 2^-40 at the most, times the
// deviations, plus that of the pairs.
int main() {
    int taken = 0;
    for (double e = -320; e < 308; e += 0.25) {
        const double kn = pow(10.0, e), ny = 8, A = sqrt(6 / M_PI) * ny * kn, B = 2 * kn, A316 = 3 / (16 * A), CA = M_PI * 0.55 / 4 * A;
        bool fit = true;
        for (double v : {A, B, A316, CA}) fit = fit && fits(v);
        if (e >= -12 && e <= 10 && !fit) return printf("refused %g\n", kn), 1;
        if (!fit) continue;
        ++taken;
        const Const c{pair_of(1.1 / 12), pair_of(0.3), {}, {}, pair_of(A), pair_of(B), pair_of(A316), pair_of(CA), {}, {}, true};
        double f[9];
        float R;
        P d[9], o[9];
        for (int i = 0; i < 9; ++i) f[i] = (i == 0 ? 4. / 9 : i < 5 ? 1. / 9 : 1. / 36) * (1 + 1e-3 * ((7 * i) % 5 - 2));
        if (!deviations(f, R, d)) return printf("state\n"), 1;
        collide<false>(R, d, c, nullptr, o);
        // g5 = s_v/4 (rho ux uy - kxy) is the part of o[5] + o[7] - o[6] - o[8] (Eq. 6)
        long double rho = 0, jx = 0, jy = 0, kxy = 0;
        const int ex[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, ey[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
        for (int i = 0; i < 9; ++i) rho += f[i], jx += ex[i] * (long double)f[i], jy += ey[i] * (long double)f[i], kxy += ex[i] * ey[i] * (long double)f[i];
        const long double q = rho + B, sv = q / (q / 2 + A), g5 = sv / 4 * (jx * jy / rho - kxy);
        const long double got = ((long double)o[5].h + o[5].l + o[7].h + o[7].l - o[6].h - o[6].l - o[8].h - o[8].l) / 4;
        if (!(fabsl(got - g5) <= 1e-3L * 0x1p-40L)) return printf("kn %g: %Lg against %Lg\n", kn, got, g5), 1;
    }
    return taken < 80;
}
"""


def test_constants_taken(tmp_path):
    r = compile_and_run(CONSTANTS, tmp_path)
    assert r.returncode == 0, r.stdout
