"""The double-float step's sums without intermediate normalisation (teuk_step_common.cuh: p_tfma,
Lin<DF>), compiled for the host from the kernels' own header and held to bounds derived by hand.

With u = 2^-24, w the size of an operand (the sum of the moduli of the normalised pairs that it is a
sum or difference of: two, or four for a difference of two sums), t = |a| w the size of a term, M
the sum of the sizes of all terms of a chain and n its links:
  an operand's low part is at most 3 u w, its error 8 u^2 w;
  a product's low part at most 5 u t, its error (its operand's included) 20 u^2 t;
  a link adds u |S| + 5 u t to the low part l of the running sum S and errs by
  u (5 u t + l) + u (u |S| + 5 u t + l); the chain starts with an operand.
So l <= (n + 8) u M and the error <= (38 + n + 2 n (n + 8)) u^2 M, whatever cancels."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r'''
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <cuda_runtime.h>
// the device intrinsics that the header uses, on the host
#undef __forceinline__
#define __forceinline__ inline
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
static inline double __fma_rn(double a, double b, double c) { return fma(a, b, c); }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline float2 __fadd2_rn(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
static inline float2 __fmul2_rn(float2 a, float2 b) { return make_float2(a.x * b.x, a.y * b.y); }
static inline float2 __ffma2_rn(float2 a, float2 b, float2 c) { return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y)); }
static inline float rsqrtf(float x) { return 1.0f / sqrtf(x); }
template <class T> static inline T __ldg(const T* p) { return *p; }
static inline int __float_as_int(float v) { int i; memcpy(&i, &v, 4); return i; }
static inline float __int_as_float(int i) { float v; memcpy(&v, &i, 4); return v; }
static inline int __double2hiint(double v) { int64_t i; memcpy(&i, &v, 8); return (int)(i >> 32); }
static inline int __double2loint(double v) { int64_t i; memcpy(&i, &v, 8); return (int)i; }
static inline double __hiloint2double(int h, int l) { int64_t i = ((int64_t)h << 32) | (uint32_t)l; double v; memcpy(&v, &i, 8); return v; }
#include "teuk_step_common.cuh"
using namespace teuk;
#ifdef __aarch64__
typedef long double quad;
#else
typedef __float128 quad;
#endif
static quad q(DF v) { return (quad)v.hi + (quad)v.lo; }
static quad mag(quad v) { return v < 0 ? -v : v; }
static uint64_t state = 88172645463325252ull;
static double rnd() {   // xorshift64, uniform in (-1, 1)
    state ^= state << 13; state ^= state >> 7; state ^= state << 17;
    return (double)(int64_t)(state >> 11) / 4503599627370496.0 - 1.0;
}
static DF number(int spread) { return DF(ldexp(rnd(), (int)(rnd() * spread))); }
static const double u = ldexp(1.0, -24);
static double worst_l = 0, worst_e = 0, worst_m = 0, worst_z = 0;
static int zeros = 0;
static void note(quad got_err, double l, quad M, double n) {
    const double m = (double)M;
    if (m == 0) return;
    worst_l = fmax(worst_l, fabs(l) / ((n + 8) * u * m));
    worst_e = fmax(worst_e, (double)mag(got_err) / ((38 + n + 2 * n * (n + 8)) * u * u * m));
}
int main(int argc, char** argv) {
    InstDev d;
    const Lin<DF> A(d);
    const long count = atol(argv[1]);
    for (long k = 0; k < count; ++k) {
        const int spread = (int)(k % 7);
        auto cx = [&] { Cx<DF> c; c.re = number(spread); c.im = number(spread); return c; };
        // this row's two columns, the rows above and below (p, m), the source term
        Cx<DF> F0 = cx(), F1 = cx(), P0 = cx(), P1 = cx(), Fp0 = cx(), Fp1 = cx(), Fm0 = cx(), Fm1 = cx(), src = cx();
        if (k & 1) {   // neighbours that agree in their first bits: differences cancel
            auto near = [&](Cx<DF> c) {
                Cx<DF> r;
                r.re = DF(c.re.to_double() * (1 + ldexp(rnd(), -20)));
                r.im = DF(c.im.to_double() * (1 + ldexp(rnd(), -30)));
                return r;
            };
            F1 = near(F0), Fp0 = near(F0), Fp1 = near(F0), Fm0 = near(F0), Fm1 = near(F0);
            P1 = near(P0);
        }
        const Cx<DF> s = A.add(F0, F1), s_p = A.add(Fp0, Fp1), s_m = A.add(Fm0, Fm1);
        DF cf[kNCoef];
        for (int i = 0; i < kNCoef; ++i) cf[i] = number(spread);
        const DF hdt = number(2);
        // the predictor's sums in exact arithmetic, component by component, and their sizes
        struct Q { quad re, im; };
        auto Z = [](Cx<DF> c) { return Q{q(c.re), q(c.im)}; };
        auto add = [](Q a, Q b) { return Q{a.re + b.re, a.im + b.im}; };
        auto sub = [](Q a, Q b) { return Q{a.re - b.re, a.im - b.im}; };
        auto ab = [](Q a) { return Q{mag(a.re), mag(a.im)}; };
        auto sc = [](quad c, Q a) { return Q{c * a.re, c * a.im}; };
        auto cm = [](quad cr, quad ci, Q a) { return Q{cr * a.re - ci * a.im, cr * a.im + ci * a.re}; };
        auto cmm = [](quad cr, quad ci, Q a) { return Q{mag(cr) * a.re + mag(ci) * a.im, mag(cr) * a.im + mag(ci) * a.re}; };
        const Q f0 = Z(F0), f1 = Z(F1), p0 = Z(P0), p1 = Z(P1), sq = add(f0, f1);
        const Q sp = add(Z(Fp0), Z(Fp1)), sm = add(Z(Fm0), Z(Fm1));
        const Q sP = add(p0, p1), wP = add(ab(p0), ab(p1)), dP = sub(p1, p0), dF = sub(f1, f0), wF = add(ab(f0), ab(f1));
        const Q ws = wF, up = sub(sp, sq), wup = add(ws, add(ab(Z(Fp0)), ab(Z(Fp1))));
        const Q dn = sub(sq, sm), wdn = add(ws, add(ab(Z(Fm0)), ab(Z(Fm1))));
        const quad G = q(cf[C_G]);
        auto base = [&] {
            Q a = add(sP, sc(G, dP));
            a = add(a, cm(q(cf[C_E1R]), q(cf[C_E1I]), sP));
            a = add(a, cm(q(cf[C_E2R]), q(cf[C_E2I]), dF));
            a = add(a, cm(q(cf[C_E3R]), q(cf[C_E3I]), sq));
            a = add(a, sc(q(cf[C_EP]), up));
            return sub(a, sc(q(cf[C_EM]), dn));
        };
        // every second pair: a source that cancels the whole sum to its last bits
        if ((k >> 1) & 1) {
            const Q b = base();
            src.re = DF((double)-b.re);
            src.im = DF((double)-b.im);
        }
        const Q ex = add(base(), Z(src));
        Q M = add(wP, sc(mag(G), wP));
        M = add(M, cmm(q(cf[C_E1R]), q(cf[C_E1I]), wP));
        M = add(M, cmm(q(cf[C_E2R]), q(cf[C_E2I]), wF));
        M = add(M, cmm(q(cf[C_E3R]), q(cf[C_E3I]), ws));
        M = add(M, sc(mag(q(cf[C_EP])), wup));
        M = add(M, sc(mag(q(cf[C_EM])), wdn));
        M = add(M, ab(Z(src)));
        const HalfX<DF> h = predict_x<DF, true>(A, F0, P0, F1, P1, s, s_p, s_m, cf, hdt, src);
        note(q(h.P.re) - ex.re, h.P.re.lo, M.re, 10);
        note(q(h.P.im) - ex.im, h.P.im.lo, M.im, 10);
        const Q hF = sub(add(sq, sc(q(hdt), sP)), sc(G, dF)), MF = add(ws, add(sc(mag(q(hdt)), wP), sc(mag(G), wF)));
        note(q(h.F.re) - hF.re, h.F.re.lo, MF.re, 2);
        note(q(h.F.im) - hF.im, h.F.im.lo, MF.im, 2);
        // a cancelled pair (also with everything in its low part) times a coefficient, and added
        // to the state: errors against the sizes before the cancellation
        Cx<DF> D = A.sub(F1, F0);
        if (k % 3 == 0) D.re = DF(0.f, D.re.lo), D.im = DF(0.f, D.im.lo), ++zeros;
        const Cx<DF> pr = A.mul(cf[0], D);
        const quad e = mag(q(pr.re) - G * q(D.re));
        const double size = (double)(mag(G) * wF.re);
        if (size > 0) worst_m = fmax(worst_m, (double)e / (20 * u * u * size));
        const Cx<DF> v = A.update(F0, D);
        const double sv = (double)(mag(q(F0.re)) + wF.re);
        if (sv > 0) {
            worst_z = fmax(worst_z, (double)mag(q(v.re) - (q(F0.re) + q(D.re))) / (20 * u * u * sv));
            if (fabsf(v.re.lo) > ldexp(fabsf(v.re.hi), -23)) worst_z = 9;   // what is stored is normalised
        }
    }
    printf("%.17g %.17g %.17g %.17g %d\n", worst_l, worst_e, worst_m, worst_z, zeros);
    return 0;
}
'''


def test_low_parts_and_errors_of_chains_stay_within_their_bounds(tmp_path):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    src, exe = tmp_path / "chains.cpp", tmp_path / "chains"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-w", "-I", os.path.join(cuda, "include"),
                           "-I", os.path.join(ROOT, "paper_1001_3631_gb300", "csrc"), str(src), "-o", str(exe)])
    low, err, mul, upd, zeros = map(float, subprocess.check_output([str(exe), "400000"], text=True).split())
    assert zeros > 1000
    assert 0 < low <= 1 and 0 < err <= 1 and mul <= 1 and upd <= 1, (low, err, mul, upd)
