"""The FP64 collision in FP32 pairs (csrc/pair.cuh), compiled for the host with
the same arithmetic: its error against long double, next to that of the plain
FP64 collision, over the flows it is taken for (both drives; velocities to 0.04;
non-equilibrium parts to 1 %; densities 0.9 to 2.6; Kn 0.02 to 2; heights 5 to
300), its refusal of everything else, and the bit-level conversions.

Bounds, derived: the populations' rms error must not exceed the plain
collision's, which it replaces; density and momentum, which the plain collision
keeps to its own rounding, to 1.5 times its rms; the conversions are the sum
rounded to FP64 (join), or rounded at 2^-47 (split: 24 bits and the other 29 rounded to 24)."""
import os
import platform
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include <cmath>
#include <random>
#include "pair.cuh"
using namespace clb::pr;
typedef long double Q;
template <class L> struct K { L s3_12, s8_4, sv4, sq4, A, B, A316, CA, fx; };
static double mad_(double a, double b, double c) { return fma(a, b, c); }
static Q mad_(Q a, Q b, Q c) { return a * b + c; }
// Eq. 4 and 6-10, products fused as the plain FP64 collision of the library has them
template <class L> void collide_ref(L* d, const K<L>& c, bool force) {
    const L two3 = L(2) / 3, ninth = L(1) / 9;
    const L a57 = d[5] + d[7], a68 = d[6] + d[8], p57 = d[5] - d[7], p86 = d[8] - d[6];
    const L nkxy = a68 - a57, kxxyy = a57 + a68, kxxy = p57 - p86, kxyy = p57 + p86;
    const L s13 = d[1] + d[3], s24 = d[2] + d[4], kxx = s13 + kxxyy, kyy = s24 + kxxyy;
    const L rho = ((d[0] + s13) + s24) + kxxyy, jx = (d[1] - d[3]) + kxyy, jy = (d[2] - d[4]) + kxxy;
    L sv4 = c.sv4, sq4 = c.sq4;
    const L fx = force ? c.fx : L(0);
    if (!force) {
        const L q = rho + c.B;
        sv4 = q / 4 / mad_(q, L(0.5), c.A);
        sq4 = q / 4 / mad_(q, mad_(c.A316, q, L(0.5)), c.CA);
    }
    const L ux = jx / rho + fx / 2, uy = jy / rho, ux2 = ux * ux, uy2 = uy * uy, uxy = ux * uy, nr = -rho;
    const L t5u = mad_(rho, uxy, nkxy);
    L t3 = mad_(rho, mad_(ux, ux, uy2), two3 * rho) - (kxx + kyy), t4 = mad_(rho, mad_(-uy, uy, ux2), kyy - kxx), t5 = t5u;
    L t6 = mad_(2 * ux, t5u, mad_(-uy, kxx, kxxy)), t7 = mad_(2 * uy, t5u, mad_(-ux, kyy, kxyy));
    L t8 = mad_(2 * uy, kxxy, mad_(2 * ux, kxyy, mad_(uxy, mad_(L(3), t5u, nkxy), ninth * rho))) -
           mad_(ux2, kyy, mad_(uy2, kxx, kxxyy));
    if (force) {
        t3 = mad_(nr, fx * ux, t3), t4 = mad_(nr, fx * ux, t4), t5 = mad_(nr / 2, fx * uy, t5);
        t6 = mad_(nr, fx * uxy, t6), t7 = mad_(nr / 2, fx * uy2, t7), t8 = mad_(nr, fx * ux * uy2, t8);
    }
    const L g3 = c.s3_12 * t3, g4 = sv4 * t4, g5 = sv4 * t5;
    const L hp = mad_(L(1.5), g3, g4 / 2), hm = mad_(L(1.5), g3, -g4 / 2);
    const L g6 = mad_(sq4, t6, mad_(-uy, hp, -2 * ux * g5)), g7 = mad_(sq4, t7, mad_(-ux, hm, -2 * uy * g5));
    const L g8 = mad_(c.s8_4, t8, mad_(-2 * ux, g7, mad_(-2 * uy, g6, mad_(-4 * uxy, g5, mad_(-ux2, hm, mad_(-uy2, hp, -2 * g3))))));
    const L ca = g4 - g3, s34 = g3 + g4, e5 = 2 * g3 + g8 + g5, e6 = 2 * g3 + g8 - g5, gp = g6 + g7, gm = g6 - g7;
    d[0] = mad_(L(-4), g3 - g8, d[0]);
    d[1] += mad_(L(2), g7 - g8, ca), d[3] += mad_(L(-2), g7 + g8, ca);
    d[2] -= mad_(L(-2), g6 - g8, s34), d[4] -= mad_(L(2), g6 + g8, s34);
    d[5] += e5 - gp, d[7] += e5 + gp, d[6] += e6 - gm, d[8] += e6 + gm;
    if (force) {
        const L F = rho * fx, m1 = F, m3 = 2 * F * ux, m5 = F * uy, m6 = 2 * F * uxy, m7 = F * uy2, m8 = 2 * F * ux * uy2;
        d[0] += m8 - m3;
        d[1] += (m3 - m8 + m1 - m7) / 2, d[3] += (m3 - m8 - m1 + m7) / 2;
        d[2] -= (m8 + m6) / 2, d[4] += (m6 - m8) / 2;
        d[5] += (m5 + m6 + m7 + m8) / 4, d[6] += (m6 - m5 + m8 - m7) / 4;
        d[7] += (m8 - m7 - m6 + m5) / 4, d[8] += (m7 + m8 - m5 - m6) / 4;
    }
}
int main() {
    std::mt19937_64 g(7);
    auto U = [&](double a, double b) { return a + (b - a) * (g() >> 11) * 0x1p-53; };
    for (int i = 0; i < 300000; ++i) {
        const double v = ldexp(U(1, 2), (int)U(-70, 0)) * (g() & 1 ? 1 : -1);
        const P s = split(v);
        if (fabs((double)s.h + (double)s.l - v) > 0x1p-47 * fabs(v)) return printf("split %a\n", v), 1;
        const float h = ldexpf((float)U(1, 2), (int)U(-50, 0)) * (g() & 1 ? 1 : -1);
        const float edge = ldexpf(g() & 1 ? 1.0f : -1.0f, (int)U(-50, 0));
        for (float top : {h, edge}) {
            const P n = norm({top, top * (float)U(-0x1p-25, 0x1p-25)});
            if (join(n) != (double)n.h + (double)n.l) return printf("join %a %a\n", n.h, n.l), 1;
        }
    }
    if (!(fabs(join({0, 0})) < 1e-37) || !(fabsf(split(0.0).h) < 2e-22f)) return printf("zero\n"), 1;
    const double EX[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, EY[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
    const double sets[][2] = {{1e-6, 1e-8}, {1e-3, 1e-4}, {1e-2, 1e-3}, {2e-2, 5e-3}, {4e-2, 1e-2}};
    for (int force = 0; force < 2; ++force)
        for (auto& s : sets) {
            double e[2] = {}, r[2] = {}, j[2] = {};
            long n = 0, refused = 0;
            for (int k = 0; k < 40000; ++k) {
                const double rho = U(0.9, 2.6), ux = s[0] * U(-1, 1), uy = 0.3 * s[0] * U(-1, 1);
                const double kn = exp(U(log(0.02), log(2.0))), ny = exp(U(log(5.0), log(300.0)));
                const double A = sqrt(6 / M_PI) * ny * kn, B = 2 * kn, tau = A / (1 + B), fx = exp(U(log(1e-7), log(1e-4)));
                const double sv = 1 / (0.5 + tau), sq = 1 / (0.5 + (3 + 4 * M_PI * tau * tau * 0.55) / (16 * tau));
                double f[9], p[9], h[9];
                Q q[9];
                for (int i = 0; i < 9; ++i) {
                    const double w = i == 0 ? 4. / 9 : i < 5 ? 1. / 9 : 1. / 36, eu = EX[i] * ux + EY[i] * uy;
                    f[i] = w * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * (ux * ux + uy * uy)) * (1 + s[1] * U(-1, 1));
                    p[i] = f[i], q[i] = f[i];
                }
                const K<double> c{1.1 / 12, 0.3, sv / 4, sq / 4, A, B, 3 / (16 * A), M_PI * 0.55 / 4 * A, fx};
                const K<Q> cq{c.s3_12, c.s8_4, c.sv4, c.sq4, c.A, c.B, c.A316, c.CA, c.fx};
                const Const pc{pair_of(c.s3_12), pair_of(c.s8_4), pair_of(c.sv4), pair_of(c.sq4), pair_of(A), pair_of(B),
                               pair_of(c.A316), pair_of(c.CA), pair_of(fx), pair_of(fx / 2)};
                collide_ref<double>(p, c, force);
                collide_ref<Q>(q, cq, force);
                float R;
                P d[9], o[9];
                if (!deviations(f, R, d)) {
                    ++refused;
                    continue;
                }
                if (force) collide<true>(R, d, pc, nullptr, o);
                else collide<false>(R, d, pc, nullptr, o);
                ++n;
                Q sr[2] = {}, sj[2] = {};
                for (int i = 0; i < 9; ++i) {
                    h[i] = f[i] + join(norm(o[i]));
                    const Q err[2] = {p[i] - q[i], h[i] - q[i]};
                    for (int m = 0; m < 2; ++m) e[m] += (double)(err[m] * err[m]), sr[m] += err[m], sj[m] += EX[i] * err[m];
                }
                for (int m = 0; m < 2; ++m) r[m] += (double)(sr[m] * sr[m]), j[m] += (double)(sj[m] * sj[m]);
            }
            printf("%d u %g ne %g plain %.3g pair %.3g rho %.3g %.3g jx %.3g %.3g refused %ld of 40000\n", force, s[0], s[1],
                   sqrt(e[0] / n / 9), sqrt(e[1] / n / 9), sqrt(r[0] / n), sqrt(r[1] / n), sqrt(j[0] / n), sqrt(j[1] / n), refused);
            if (e[1] > e[0] || r[1] > 2.25 * r[0] || j[1] > 2.25 * j[0] || refused > 0) return 1;
        }
    // refused: not near equilibrium, not finite, not positive, out of range
    const double rest[9] = {4. / 9, 1. / 9, 1. / 9, 1. / 9, 1. / 9, 1. / 36, 1. / 36, 1. / 36, 1. / 36};
    const double odd[] = {NAN, INFINITY, -INFINITY, 1e300, -1e300, 1e40, 0.6, -0.4444, 1e12};
    for (double v : odd)
        for (int i = 0; i < 9; ++i) {
            double f[9];
            float R;
            P d[9];
            for (int k = 0; k < 9; ++k) f[k] = rest[k];
            f[i] = v;
            if (deviations(f, R, d)) return printf("took %g in %d\n", v, i), 1;
        }
    for (double sc : {1e-5, 2e9, 1e-300, 1e300, -1.0, 0.0}) {
        double f[9];
        float R;
        P d[9];
        for (int k = 0; k < 9; ++k) f[k] = sc * rest[k];
        if (deviations(f, R, d)) return printf("took density %g\n", sc), 1;
    }
    return 0;
}
"""


def test_pair_collision_error_on_the_host(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE)
    fma = ["-mfma"] if platform.machine() == "x86_64" else []
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", *fma, "-I",
                    os.path.join(ROOT, "paper_1603_01955_gb300", "csrc"), str(src), "-o", str(exe), "-lm"], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
