"""The fixed-point EGARCH recursion of the FP64 path (csrc/egarch_fx.cuh),
compiled with the host compiler and compared with the recursion as written in
long double (64-bit significand or more), beside the same in double (CPU only).

The requirement is that fixed point loses nothing against FP64: over the
particles of a case its root-mean-square error is at most that of the same
recursion in double, or one rounding (2^-52) of the magnitudes that are summed,
sum_t |log h_t| + |l_t + log h_t|, where both are that small.  A state is held
to 2^-52 of the largest |v|, |eps| that the series can amplify it from (100
here)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_1304_4334_gb300", "csrc", "egarch_fx.cuh")
TABLE = os.path.join(ROOT, "paper_1304_4334_gb300", "csrc", "exp2_table.h")

SRC = r"""
#include <cstdio>
#include <random>
#include <vector>
#include "HEADER"
#define __device__
#include "TABLE"
using namespace smc;
typedef long double R;
struct Par { double mu, lsy, al[4], be[4], ga[4], p[4], m[4], s[4]; };
template <class R, int K, int I> R plain(const Par& q, const std::vector<double>& y, R* st, R* mag) {
    R v[K] = {}, eps = 0, acc = 0, c = sqrtl(2 / M_PIl);
    *mag = 0;
    for (size_t t = 0; t < y.size(); ++t) {
        if (t) for (int k = 0; k < K; ++k) v[k] = q.al[k] * v[k] + q.be[k] * (std::fabs(eps) - c) + q.ga[k] * eps;
        R lh = q.lsy;
        for (int k = 0; k < K; ++k) lh += v[k] / 2;
        eps = ((R)y[t] - q.mu) * std::exp(-lh);
        R s = 0, mx = -1e30, x[I];
        for (int i = 0; i < I; ++i) {
            R z = (eps - q.m[i]) / q.s[i];
            x[i] = std::log((R)q.p[i]) - std::log((R)q.s[i]) - z * z / 2;
            mx = x[i] > mx ? x[i] : mx;
        }
        for (int i = 0; i < I; ++i) s += std::exp(x[i] - mx);
        const R l = mx + std::log(s);
        acc += l - lh;
        *mag += std::fabs(l) + std::fabs(lh);
    }
    for (int k = 0; k < K; ++k) st[k] = v[k];
    st[K] = eps;
    return acc - (R)y.size() * std::log(2 * (R)M_PIl) / 2;
}
template <int K, int I> void test(int T, int P, double outlier) {
    std::mt19937_64 g(100 * K + 10 * I + T);
    std::normal_distribution<double> N;
    std::uniform_real_distribution<double> U(0, 1);
    std::vector<double> y(T);
    for (auto& x : y) x = 0.0003 + 0.01 * N(g) * (U(g) < 0.05 ? outlier : 1.0);
    double e2 = 0, d2 = 0, m2 = 0, state = 0;
    int bad = 0;
    for (int p = 0; p < P; ++p) {
        Par q;
        q.mu = 0.0003 + 1e-5 * N(g);
        q.lsy = log(0.01) + 0.05 * N(g);
        for (int k = 0; k < K; ++k) {
            q.al[k] = tanh(1.8 + 0.05 * N(g));
            q.be[k] = exp(log(0.1) + 0.05 * N(g));
            q.ga[k] = 0.05 * N(g);
        }
        double ps = 0, pm = 0, v = 0;
        for (int i = 0; i < I; ++i) {
            ps += q.p[i] = 1 + tanh(0.05 * N(g) - 0.3 * i);
            q.m[i] = 0.05 * N(g);
            q.s[i] = exp(0.4 * i + 0.05 * N(g));
        }
        for (int i = 0; i < I; ++i) { q.p[i] /= ps; pm += q.p[i] * q.m[i]; }
        for (int i = 0; i < I; ++i) { q.m[i] -= pm; v += q.p[i] * (q.m[i] * q.m[i] + q.s[i] * q.s[i]); }
        for (int i = 0; i < I; ++i) { q.m[i] /= sqrt(v); q.s[i] /= sqrt(v); }
        if (I == 1) q.p[0] = q.s[0] = 1, q.m[0] = 0;
        R sq[K + 1], mag;
        double sd[K + 1], magd;
        const R lq = plain<R, K, I>(q, y, sq, &mag);
        const R ed = plain<double, K, I>(q, y, sd, &magd) - lq;
        EgarchFx<K, I> f;
        f.setup(q.mu, q.lsy, q.al, q.be, q.ga, q.p, q.m, q.s, 0, 1.0 / log(2.0));
        for (int t = 0; t < T; ++t) {
            if (t == 0) f.template chain<true>(y[0], g_exp2_neg256);
            else f.template chain<false>(y[t], g_exp2_neg256);
            f.mix(f.E, f.neg, g_exp2_neg256);
            if ((t & 7) == 7) f.flush();
        }
        f.flush();
        double st[K + 1];
        f.state_out(st, log(2.0));
        bad += f.bad != 0;
        const R e = f.finish(T, log(2.0), log(2 * M_PI)) - lq;
        e2 += (double)(e * e);
        d2 += (double)(ed * ed);
        m2 += (double)(mag * mag);
        for (int k = 0; k <= K; ++k) state = fmax(state, (double)fabsl(st[k] - sq[k]));
    }
    printf("%d %d %d %.17g %.17g %.17g %.17g %d\n", K, I, T, sqrt(e2 / P), sqrt(d2 / P), sqrt(m2 / P), state, bad);
}
int main() {
    std::mt19937_64 g(1);
    double w = 0;
    for (int i = 0; i < 100000; ++i) {
        const uint64_t X = i < 4096 ? (uint64_t)i << 43 : g() & ((1ull << 55) - 1);
        const R e = exp2l(-(R)X * 0x1p-55L);
        w = fmax(w, (double)fabsl((R)fx_exp2neg(X, g_exp2_neg256) * 0x1p-63L / e - 1));
    }
    printf("exp2neg %.17g\n", w);
    double u = 0;
    for (int i = 0; i < 100000; ++i) {
        const double x = (i & 1 ? -1 : 1) * 127.9 * (double)(g() >> 11) * 0x1p-53;
        u = fmax(u, (double)fabsl(fx_exp_neg(x, g_exp2_neg256) / expl(-(R)x) - 1));
    }
    const double ends[] = {0.0, -0.0, 1e-300, 700.0, 745.0, -709.0, 1023.0, -1023.0, 1e300, -1e300, INFINITY, -INFINITY};
    bool same = std::isnan(fx_exp_neg(NAN, g_exp2_neg256));
    for (double x : ends) same = same && fx_exp_neg(x, g_exp2_neg256) == exp(-x);
    printf("exp %.17g %d\n", u, (int)same);
    for (int T : {1, 37, 500, 3000}) {
        test<1, 1>(T, T > 1000 ? 10 : 100, 1);
        test<2, 2>(T, T > 1000 ? 10 : 100, 1);
        test<3, 4>(T, T > 1000 ? 10 : 100, 1);
        test<4, 3>(T, T > 1000 ? 10 : 100, 1);
    }
    test<2, 2>(500, 50, 20);
    test<1, 1>(500, 50, 20);
}
"""


def test_fixed_point_recursion_against_long_double(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "fx.cpp"
    src.write_text(SRC.replace("HEADER", HEADER).replace("TABLE", TABLE))
    exe = tmp_path / "fx"
    subprocess.run([gxx, "-O1", "-std=gnu++17", "-o", str(exe), str(src)], check=True)
    lines = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")
    name, w = lines[0].split()
    assert name == "exp2neg" and float(w) < 2.0 ** -58
    name, u, same = lines[1].split()
    # rounding of the result (2^-53) and of x log2(e) (2^-55 units of the exponent)
    assert name == "exp" and float(u) < 2.0 ** -52 and same == "1"
    rows = [x.split() for x in lines[2:] if x]
    assert len(rows) == 18
    for K, I, T, fx, dbl, mag, state, bad in rows:
        assert bad == "0", (K, I, T)
        assert float(fx) <= max(float(dbl), float(mag) * 2.0 ** -52), (K, I, T, fx, dbl, mag)
        assert float(state) <= 100 * 2.0 ** -52, (K, I, T, state)


SETUP = r"""
#include <cstdio>
#include "HEADER"
#define __device__
#include "TABLE"
using namespace smc;
// every parameter in turn NaN, inf, -inf: setup() must send the particle to FP64
template <int K, int I> int test() {
    int wrong = 0;
    const double bad[] = {NAN, INFINITY, -INFINITY};
    for (int j = -1; j < 2 + 3 * K + (I > 1 ? 3 * I : 0); ++j)
        for (double x : bad) {
            double v[2 + 3 * K + 3 * I] = {0.0003, -4.6};
            for (int k = 0; k < K; ++k) v[2 + k] = 0.9, v[2 + K + k] = 0.1, v[2 + 2 * K + k] = -0.05;
            for (int i = 0; i < I; ++i) v[2 + 3 * K + i] = 1.0 / I, v[2 + 3 * K + I + i] = 0.0, v[2 + 3 * K + 2 * I + i] = 1.0;
            if (j >= 0) v[j] = x;
            EgarchFx<K, I> f;
            f.setup(v[0], v[1], v + 2, v + 2 + K, v + 2 + 2 * K, v + 2 + 3 * K, v + 2 + 3 * K + I,
                    v + 2 + 3 * K + 2 * I, 0, 1.0 / log(2.0));
            if ((f.bad != 0u) != (j >= 0)) ++wrong, printf("K=%d I=%d parameter %d value %g: bad %u\n", K, I, j, x, f.bad);
        }
    return wrong;
}
int main() { return test<1, 1>() + test<2, 2>() + test<3, 4>() + test<4, 3>() ? 1 : 0; }
"""


def test_setup_refuses_every_parameter_that_is_not_finite(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "setup.cpp"
    src.write_text(SETUP.replace("HEADER", HEADER).replace("TABLE", TABLE))
    exe = tmp_path / "setup"
    subprocess.run([gxx, "-O1", "-std=gnu++17", "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


WEIGHTS = r"""
#include <cstdio>
#include <random>
#include "HEADER"
#define __device__
#include "TABLE"
using namespace smc;
typedef long double R;
// largest |r / exact - 1| / ((1 + |d|) 2^-50) over components, d its log2 distance from the largest
template <int I> double test(double spread) {
    std::mt19937_64 g(I);
    std::normal_distribution<double> N;
    const double z1[1] = {0.9}, z2[1] = {0.1}, z3[1] = {0.0};
    double worst = 0;
    for (int rep = 0; rep < 20000; ++rep) {
        double p[I], m[I], s[I], r[I];
        for (int i = 0; i < I; ++i) p[i] = exp(spread * N(g)), m[i] = 0.5 * N(g), s[i] = exp(0.5 * N(g));
        EgarchFx<1, I> f;
        f.setup(0, -4.6, z1, z2, z3, p, m, s, 0, 1.0 / log(2.0));
        const double e = 2 * N(g);
        if (f.bad || !f.weights(e * 0x1p53, r, g_exp2_neg256)) continue;
        R x[I], mx = -1e30L, sum = 0;
        for (int i = 0; i < I; ++i) {
            const R z = ((R)e - m[i]) / s[i];
            x[i] = std::log((R)p[i]) - std::log((R)s[i]) - z * z / 2;
            mx = x[i] > mx ? x[i] : mx;
        }
        for (int i = 0; i < I; ++i) sum += std::exp(x[i] - mx);
        for (int i = 0; i < I; ++i) {
            const R d = (mx - x[i]) / std::log((R)2);
            if (d > 120) continue;
            worst = fmax(worst, (double)(fabsl(r[i] / (std::exp(x[i] - mx) / sum) - 1) / ((1 + d) * 0x1p-50L)));
        }
    }
    return worst;
}
int main() { printf("%g %g %g %g\n", test<2>(1), test<2>(12), test<3>(12), test<4>(12)); }
"""


def test_component_weights_against_long_double(tmp_path):
    """Every weight relative to itself: d_i is a quadratic in FP64 whose terms are
    up to a few times its own size (setup's rounding, two FMAs: 2^-50 of 1 + |d_i|,
    in log2 units, covers them), whatever the weight's size."""
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "weights.cpp"
    src.write_text(WEIGHTS.replace("HEADER", HEADER).replace("TABLE", TABLE))
    exe = tmp_path / "weights"
    subprocess.run([gxx, "-O1", "-std=gnu++17", "-o", str(exe), str(src)], check=True)
    worst = [float(v) for v in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()]
    assert max(worst) < 8.0, worst


EXP = r"""
#include <cstdio>
#include <random>
#include "HEADER"
#define __device__
#include "TABLE"
using namespace smc;
int main() {
    std::mt19937_64 g(2);
    double u = 0;
    for (int i = 0; i < 1000000; ++i) {
        const double x = (i & 1 ? -1 : 1) * (128.0 + 572.0 * (double)(g() >> 11) * 0x1p-53);
        u = fmax(u, (double)fabsl(fx_exp_neg(x, g_exp2_neg256) / expl(-(long double)x) - 1));
    }
    for (double x : {128.0, 255.999999999999, 256.0, 511.999999999999, 512.0, 699.999999999999})
        for (double s : {-1.0, 1.0})
            u = fmax(u, (double)fabsl(fx_exp_neg(s * x, g_exp2_neg256) / expl(-(long double)(s * x)) - 1));
    printf("%.17g\n", u);
}
"""


def test_exponential_from_128_to_700(tmp_path):
    """Rounding of the result (2^-53), of log2(e) (2^-64 of up to 1010: 2^-54) and
    of the product (2^-55), the last two times ln 2: below 2^-52."""
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "exp.cpp"
    src.write_text(EXP.replace("HEADER", HEADER).replace("TABLE", TABLE))
    exe = tmp_path / "exp"
    subprocess.run([gxx, "-O1", "-std=gnu++17", "-o", str(exe), str(src)], check=True)
    u = float(subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout)
    assert u < 2.0 ** -52, u


BLOCK = "#include <algorithm>\n" + SRC[:SRC.index("template <int K, int I> void test(")] + r"""
// Blocks of any length with the state taken out and up again in between; beta of
// any size (the coefficients' three scales, cs = 0, 2, 4).
template <int K, int I> void test(int T, double beta, int cs) {
    std::mt19937_64 g(1000 * K + 10 * I + cs);
    std::normal_distribution<double> N;
    std::vector<double> fx, dbl, mags;
    int used = 0, wrong = 0;
    for (int p = 0; p < 4000; ++p) {
        std::vector<double> y(T);
        for (auto& x : y) x = 0.0003 + 0.01 * N(g);
        Par q;
        q.mu = 0.0003;
        q.lsy = log(0.01);
        for (int k = 0; k < K; ++k) q.al[k] = 0.3 + 0.1 * N(g), q.be[k] = beta * exp(0.05 * N(g)), q.ga[k] = 0.05 * N(g);
        double v = 0;
        for (int i = 0; i < I; ++i) q.p[i] = 1.0 / I, q.m[i] = 0, q.s[i] = exp(0.3 * i), v += q.p[i] * q.s[i] * q.s[i];
        for (int i = 0; i < I; ++i) q.s[i] /= sqrt(v);
        EgarchFx<K, I> f;
        f.setup(q.mu, q.lsy, q.al, q.be, q.ga, q.p, q.m, q.s, 0, 1.0 / log(2.0));
        wrong += f.cs != cs;
        for (int t = 0, n = 1; t < T; t += n, n = 1 + (5 * n) % 33) {
            n = n < T - t ? n : T - t;
            f.block(&y[t], n, t == 0, g_exp2_neg256);
            double st[K + 1];
            f.state_out(st, log(2.0));
            if (!f.bad && !f.enter(st, st[K])) f.bad = 1;
        }
        if (f.bad) continue;                 // (left the ranges: not this test's)
        R sq[K + 1], mag;
        double sd[K + 1], magd;
        const R lq = plain<R, K, I>(q, y, sq, &mag);
        const R ed = plain<double, K, I>(q, y, sd, &magd) - lq, e = f.finish(T, log(2.0), log(2 * M_PI)) - lq;
        fx.push_back((double)fabsl(e)), dbl.push_back((double)fabsl(ed)), mags.push_back((double)mag), ++used;
    }
    for (auto* x : {&fx, &dbl, &mags}) std::sort(x->begin(), x->end());
    for (double at : {0.5, 0.9}) {
        const int n = (int)(at * used);
        printf("%d %d %d %.17g %.17g %.17g %d %d\n", K, I, cs, fx[n], dbl[n], mags[n], used, wrong);
    }
}
int main() {
    test<1, 1>(90, 0.1, 0);
    test<2, 3>(90, 0.5, 0);
    test<1, 2>(90, 1.8, 2);
    test<2, 2>(60, 1.7, 2);
    test<1, 1>(12, 7.0, 4);
    test<1, 3>(12, 7.0, 4);
}
"""


def test_blocks_and_large_coefficients_against_long_double(tmp_path):
    """As the first test, through block() and enter(): at the median particle and at
    the 90% one (a recursion with beta = 7 amplifies any rounding, so that one
    particle can make up a mean square) no larger an error than the recursion in
    double, or 2^-52 of the magnitudes summed."""
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "block.cpp"
    src.write_text(BLOCK.replace("HEADER", HEADER).replace("TABLE", TABLE))
    exe = tmp_path / "block"
    subprocess.run([gxx, "-O1", "-std=gnu++17", "-o", str(exe), str(src)], check=True)
    rows = [x.split() for x in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n") if x]
    assert len(rows) == 12
    for K, I, cs, fx, dbl, mag, used, wrong in rows:
        assert int(used) >= 500 and wrong == "0", (K, I, cs, used, wrong)
        assert float(fx) <= max(float(dbl), float(mag) * 2.0 ** -52), (K, I, cs, fx, dbl, mag)
