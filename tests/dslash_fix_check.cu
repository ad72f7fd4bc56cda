// Host-side check of the fixed-point hop (dslash_fix.cuh) against 80-bit sums: one row of the colour
// multiply for random unit rows and half spinors over the exponent range, with zero components, with
// every component at the bound, with components far below the largest, and the conversions to and from FP64 and double-float.  Prints "ok" or
// the first failure.
#include <cmath>
#include <cstdio>
#include <random>

#include "dslash_fix.cuh"

using namespace ov;

static int fail(const char* what, double a, double b)
{
    std::printf("%s: %.17g %.17g\n", what, a, b);
    return 1;
}

static double fix_to_link(Fix a) { return std::ldexp((double)a.h, -30) + std::ldexp((double)a.l, -62); }

int main()
{
    std::mt19937_64 g(1);
    std::normal_distribution<double> n;
    double bias = 0;  // mean relative error of the conversion to pairs
    for (int t = 0; t < 200000; ++t) {
        double u[6], nn = 0, h[12], mx = 0;
        for (double& x : u) {
            x = t % 4 == 0 ? (g() % 2 ? 1.0 : -1.0) : n(g);  // every entry equal: the largest product sums
            nn += x * x;
        }
        for (double& x : u) x /= std::sqrt(nn);
        const double sc = std::ldexp(1.0, (int)(g() % 1600) - 800);
        for (double& x : h) x = (t % 4 < 2 ? (g() % 2 ? 1.0 : -1.0) * (2.0 - 4e-16) : n(g)) * sc * (t % 3 == 0 && g() % 5 == 0 ? 0.0 : 1.0);
        for (double x : h) mx = std::fmax(mx, std::fabs(x));
        if (mx == 0) continue;
        const uint32_t em = fix_range(h);
        if (em == FIX_BAD) return fail("refused", mx, 0);
        FixProd re{}, im{};
        long double rr = 0, ri = 0;
        for (int j = 0; j < 3; ++j) {
            const Fix ur = link_to_fix(u[2 * j]), ui = link_to_fix(u[2 * j + 1]);
            const Fix a = to_fix(h[2 * j], em), b = to_fix(h[2 * j + 1], em);
            if (std::fabs(fix_to_link(ur) - u[2 * j]) > 1.2e-16 * std::fabs(u[2 * j]) + 2.2e-19) return fail("link", fix_to_link(ur), u[2 * j]);
            fix_mac(re, ur, a);
            fix_mac(re, ui, fix_neg(b));
            fix_mac(im, ur, b);
            fix_mac(im, ui, a);
            rr += (long double)u[2 * j] * h[2 * j] - (long double)u[2 * j + 1] * h[2 * j + 1];
            ri += (long double)u[2 * j] * h[2 * j + 1] + (long double)u[2 * j + 1] * h[2 * j];
        }
        // 2^-55 of the largest component: half an FP64 rounding of one product of that size
        const int e = (int)(em >> 20);
        for (int k = 0; k < 2; ++k) {
            const long long v = fix_sum(k ? im : re);
            const long double ex = ldexpl((long double)v, e - 1080), ref = k ? ri : rr;
            if (fabsl(ex - ref) > ldexpl(mx, -55)) return fail("row", (double)ex, (double)ref);
            if (fabsl(fix_to_f64(v, e) - ex) > ldexpl(fabsl(ex), -53)) return fail("to f64", fix_to_f64(v, e), (double)ex);
            const uint32_t sh = (uint32_t)(g() % 100);
            if (fix_sar(v, sh) != (v >> (sh < 63 ? sh : 63))) return fail("shift", (double)v, sh);
            // double-float result: 47 significand bits, low word at most half a unit of the high one
            float a, b;
            const int ed = 80 + (int)(g() % 160);
            fixd_from_fix(v, ed, a, b);
            const long double tv = ldexpl((long double)v, ed - 184);
            if (fabsl((long double)a + b - tv) > ldexpl(fabsl(tv), -47) || std::fabs(b) > std::ldexp(std::fabs(a), -24))
                return fail("to df", a, (double)tv);
            if (v) bias += (double)(((long double)a + b - tv) / tv) / 400000.0;
        }
        // links that mix no colours, components down to 2^-60 of the largest: what is not formed again keeps the
        // field's precision relative to the complex component itself
        if (t % 2) {
            double hw[12];
            float fh[12], fl[12];
            for (int i = 0; i < 12; ++i) {
                hw[i] = i == 11 ? sc : std::ldexp(n(g), -(int)(g() % 60)) * sc;
                fh[i] = (float)(hw[i] / sc);
                fl[i] = (float)(hw[i] / sc - fh[i]);
            }
            const uint32_t ew = fix_range(hw), efw = fixd_range(fh, fl);
            if (ew == FIX_BAD || efw == FIX_BAD) return fail("wide refused", 0, 0);
            const double ph = 0.7 + 1e-5 * t, cr = std::cos(ph), sr = std::sin(ph);
            const Fix ur = link_to_fix(cr), ui = link_to_fix(sr);
            for (int j = 0; j < 6; ++j)
                for (int df = 0; df < 2; ++df) {
                    const long double xr = df ? (long double)fh[2 * j] + fl[2 * j] : hw[2 * j];
                    const long double xi = df ? (long double)fh[2 * j + 1] + fl[2 * j + 1] : hw[2 * j + 1];
                    const Fix a = df ? fixd_to_fix(fh[2 * j], fl[2 * j], efw) : to_fix(hw[2 * j], ew);
                    const Fix b = df ? fixd_to_fix(fh[2 * j + 1], fl[2 * j + 1], efw) : to_fix(hw[2 * j + 1], ew);
                    FixProd pr{}, pi{};
                    fix_mac(pr, ur, a);
                    fix_mac(pr, ui, fix_neg(b));
                    fix_mac(pi, ur, b);
                    fix_mac(pi, ui, a);
                    const long long vr = fix_sum(pr), vi = fix_sum(pi);
                    if (fix_small(vr, vi, df ? FIXD_KEEP : FIX_KEEP)) continue;
                    const int ex = df ? (int)(efw >> 23) - 184 : (int)(ew >> 20) - 1080;
                    const long double er = ldexpl((long double)vr, ex) - ((long double)cr * xr - (long double)sr * xi);
                    const long double ei = ldexpl((long double)vi, ex) - ((long double)cr * xi + (long double)sr * xr);
                    const long double mag = hypotl(xr, xi), err = hypotl(er, ei);
                    // per part: two conversions of one unit of 2^-60, dropped terms 2 x 2^-60 and half a unit of
                    // 2^-58 (all below one unit of 2^-58) of a scale that is below 2^KEEP of the component
                    if (err > ldexpl(mag, df ? FIXD_KEEP - 57 : FIX_KEEP - 57)) return fail("component", (double)(err / mag), df);
                }
        }
        // exact zeros stay zero, whatever the link, forward and backward
        if (t % 8 == 0) {
            const double hz[12] = {0, 0, h[2], h[3], 0, 0, 0, 0, 0, 0, 0, 0};
            const uint32_t ez = fix_range(hz);
            if (ez != FIX_BAD && ez != 0) {
                Fix f[6];
                for (int i = 0; i < 6; ++i) f[i] = to_fix(hz[i], ez);
                for (int m = 0; m >= -1; --m) {
                    FixProd zr{}, zi{};
                    const double uz[6] = {u[0], u[1], 0, 0, u[4], -u[5]};  // no coupling to the filled colour
                    for (int j = 0; j < 3; ++j) {
                        const Fix ur = link_to_fix(uz[2 * j]), ui = fix_sign(link_to_fix(uz[2 * j + 1]), m);
                        fix_mac(zr, ur, f[2 * j]);
                        fix_mac(zr, ui, fix_neg(f[2 * j + 1]));
                        fix_mac(zi, ur, f[2 * j + 1]);
                        fix_mac(zi, ui, f[2 * j]);
                    }
                    if (fix_sum(zr) != 0 || fix_sum(zi) != 0) return fail("zero product", (double)fix_sum(zr), (double)fix_sum(zi));
                }
            }
        }
        // negation and the link's conjugate are exact
        for (int i = 0; i < 12; ++i) {
            const Fix x = to_fix(h[i], em), y = fix_neg(x);
            const long long vx = (long long)x.h * 4294967296ll + x.l, vy = (long long)y.h * 4294967296ll + y.l;
            if (vx + vy != (x.l == -2147483647 - 1 ? -1 : 0)) return fail("negation", (double)vx, (double)vy);
        }
        for (int j = 0; j < 6; ++j) {
            const Fix x = link_to_fix(u[j]), y = fix_sign(x, -1);
            if (x.h != -y.h || x.l != -y.l || x.l == -2147483647 - 1) return fail("conjugate", u[j], 0);
        }
        // double-float input
        float hh[12], hl[12], m = 0;
        for (int i = 0; i < 12; ++i) {
            const double x = std::ldexp(h[i] / sc, (int)(t % 101) - 40);
            hh[i] = (float)x;
            hl[i] = (float)(x - hh[i]);
            m = std::fmax(m, std::fabs(hh[i]));
        }
        const uint32_t ed = fixd_range(hh, hl);
        if (ed == FIX_BAD) return fail("df refused", m, 0);
        for (int i = 0; i < 12; ++i) {
            const Fix f = fixd_to_fix(hh[i], hl[i], ed);
            const long double val = ldexpl((long double)(f.h * 4294967296.0L + f.l), (int)(ed >> 23) - 186);
            // two cut words, one unit each: 2^-59 of twice the largest component at most
            if (fabsl(val - ((long double)hh[i] + hl[i])) > ldexpl(m, -58)) return fail("from df", hh[i], (double)val);
        }
    }
    // rounding to nearest: 2^-49 in the root mean square, 2^-58 in the mean of 400 000 (cut: -2^-48.5)
    if (std::fabs(bias) > std::ldexp(1.0, -54)) return fail("bias", bias, 0);
    // sums of every size at every exponent of the double-float hops, down to the smallest
    for (int e = (int)(FIXD_ELO >> 23); e < (int)(FIXD_EHI >> 23); ++e)
        for (int k = 0; k < 62; ++k)
            for (long long v : {1ll << k, -(1ll << k), (1ll << k) + (1ll << k) / 3, -(1ll << k) - (1ll << k) / 5}) {
                float a, b;
                fixd_from_fix(v, e, a, b);
                const long double tv = ldexpl((long double)v, e - 184);
                if (!(fabsl((long double)a + b - tv) <= ldexpl(fabsl(tv), -47) + ldexpl(1.0L, -126)))
                    return fail("small to df", a, (double)tv);
            }
    double z[12] = {};
    if (fix_range(z) != 0) return fail("zero", 0, 0);
    z[3] = 5e-324;
    if (fix_range(z) != FIX_BAD) return fail("subnormal", 0, 0);
    z[3] = INFINITY;
    if (fix_range(z) != FIX_BAD) return fail("inf", 0, 0);
    z[3] = NAN;
    if (fix_range(z) != FIX_BAD) return fail("nan", 0, 0);
    if (fix_to_f64(0, 1000) != 0.0 || fix_to_f64(-1, 1080) != -1.0) return fail("to f64 ends", 0, 0);
    std::printf("ok\n");
    return 0;
}
