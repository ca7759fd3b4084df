"""The other fixed-point forms (csrc/tdse_fix.cuh) compiled for the host, in fixed point, in double and in 113 bits:
NUMEROV_SPLIT and FULL_CN by composed short segments.  As for the 32-wide FULL_CN sweep (test_fixed_point_sweep), the
fixed-point state has to be no further from the 113-bit one than the double state is.  And the reciprocal's bound."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2507_04115_gb300", "csrc")

PROGRAM = r"""
#include "tdse_fix.cuh"
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>
using namespace tdse;
using std::vector;
typedef __float128 quad;
typedef std::complex<double> cd;
struct Q {
    quad r, i;
};
static Q operator*(Q a, Q b) { return {a.r * b.r - a.i * b.i, a.r * b.i + a.i * b.r}; }
static Q operator-(Q a, Q b) { return {a.r - b.r, a.i - b.i}; }
static Q inverse(Q a)
{
    const quad n = a.r * a.r + a.i * a.i;
    return {a.r / n, -a.i / n};
}
static Q expi(quad x)   // e^{ix}, |x| < 100: the series at x / 2^10, squared ten times
{
    const quad t = x / 1024;
    Q s{1, 0}, p{1, 0};
    for (int k = 1; k < 28; ++k) {
        p = p * Q{0, t / k};
        s = {s.r + p.r, s.i + p.i};
    }
    for (int k = 0; k < 10; ++k) s = s * s;
    return s;
}

struct Grid {
    int N, nt;
    double dx, dt;
    vector<double> x, V, m, E;
    vector<cd> p0;
    Grid(int N, double dx, double dt, int nt) : N(N), nt(nt), dx(dx), dt(dt), x(N), V(N), m(N, 1.0), E(nt + 1), p0(N)
    {
        double n2 = 0;
        for (int j = 0; j < N; ++j) {
            x[j] = (j - .5 * (N - 1)) * dx;
            V[j] = -1 / std::sqrt(x[j] * x[j] + 1.19 * 1.19);
            const double ax = std::fabs(x[j]) - (0.5 * N * dx - 20);
            if (ax > 0) m[j] = std::pow(std::cos(.5 * M_PI * ax / 20), .125);
            p0[j] = std::exp(-std::sqrt(x[j] * x[j] + 1)) + 0.1 * std::exp(-(x[j] - 20) * (x[j] - 20) / 60.) * std::exp(cd(0, 1.2 * x[j]));
            n2 += std::norm(p0[j]);
        }
        for (auto& z : p0) z /= std::sqrt(n2 * dx);
    }
    void field(double top)
    {
        for (int n = 0; n <= nt; ++n) E[n] = top * std::cos(.057 * n * dt + 0.3);
    }
};

// the state of a slice in integers, rescaled every 16 steps as the kernels do
struct Slice {
    vector<int64_t> r, i;
    vector<cd> p;
    int sigma = 0, top;
    Slice(const vector<cd>& p0, int top) : r(p0.size()), i(p0.size()), p(p0), top(top) { load(); }
    void load()
    {
        double t = 0;
        for (auto& z : p) t += std::norm(z);
        int e2;
        std::frexp(t, &e2);
        sigma = top - ((e2 - 1 + 2) >> 1);
        auto fix = [&](double v) {
            uint64_t b;
            std::memcpy(&b, &v, 8);
            return double_to_fix(b, sigma);
        };
        for (size_t j = 0; j < p.size(); ++j) {
            r[j] = fix(p[j].real());
            i[j] = fix(p[j].imag());
        }
    }
    void store()
    {
        auto dbl = [&](int64_t v) {
            const uint64_t b = fix_to_double(v, sigma);
            double w;
            std::memcpy(&w, &b, 8);
            return w;
        };
        for (size_t j = 0; j < p.size(); ++j) p[j] = {dbl(r[j]), dbl(i[j])};
    }
};

static int compare(const char* what, const Grid& g, const vector<Q>& P, const vector<cd>& d, const vector<cd>& f, double most)
{
    quad nd = 0, nf = 0, nq = 0;
    auto sq = [](Q z) { return z.r * z.r + z.i * z.i; };
    for (int j = 0; j < g.N; ++j) {
        nq += sq(P[j]);
        nd += sq(P[j] - Q{d[j].real(), d[j].imag()});
        nf += sq(P[j] - Q{f[j].real(), f[j].imag()});
    }
    const double ed = std::sqrt((double)(nd / nq)), ef = std::sqrt((double)(nf / nq));
    std::printf("%s N %d dx %g dt %g steps %d: double %.3g fixed %.3g largest 2^%.2f\n", what, g.N, g.dx, g.dt, g.nt, ed, ef, std::log2(most));
    return ef <= ed && most < 0x1p62 ? 0 : 12;
}

// NUMEROV_SPLIT: segments of m points (the phase starts anew in each)
static int numerov(int N, double dx, double dt, int nt, int m)
{
    Grid g(N, dx, dt, nt);
    g.field(0.06);
    const auto &V = g.V, &E = g.E;
    const double h = 0.5 * dt, inv2 = 1.0 / (dx * dx), x0 = -.5 * (N - 1) * dx;
    vector<cd> W(N), L(N), C(N), d(N), p = g.p0;
    vector<Q> qW(N), qL(N), qC(N), D(N), P(N);
    const quad i2 = 1 / ((quad)dx * dx), hq = (quad)dt / 2, tw = (quad)1 / 12;
    for (int j = 0; j < N; ++j) {
        const cd lo = j ? cd(1. / 12, h * (-.5 * inv2 + V[j - 1] / 12)) : cd(0, 0), di = cd(10. / 12, h * (inv2 + 10. / 12 * V[j])),
                 up = j < N - 1 ? cd(1. / 12, h * (-.5 * inv2 + V[j + 1] / 12)) : cd(0, 0);
        const cd w = 1.0 / (di - lo * (j ? C[j - 1] : cd(0, 0)));
        W[j] = w / 12.0;
        L[j] = lo * w;
        C[j] = up * w;
        const Q ql = j ? Q{tw, hq * (-i2 / 2 + V[j - 1] * tw)} : Q{0, 0}, qd{10 * tw, hq * (i2 + 10 * tw * V[j])},
                qu = j < N - 1 ? Q{tw, hq * (-i2 / 2 + V[j + 1] * tw)} : Q{0, 0};
        const Q qw = inverse(qd - ql * (j ? qC[j - 1] : Q{0, 0}));
        qW[j] = qw * Q{tw, 0};
        qL[j] = ql * qw;
        qC[j] = qu * qw;
        P[j] = {p[j].real(), p[j].imag()};
    }
    for (int n = 0; n < nt; ++n) {
        Q v{0, 0}, y{0, 0};
        for (int j = 0; j < N; ++j) {
            const Q l = j ? P[j - 1] : Q{0, 0}, r = j < N - 1 ? P[j + 1] : Q{0, 0};
            v = D[j] = qW[j] * Q{l.r + 10 * P[j].r + r.r, l.i + 10 * P[j].i + r.i} - qL[j] * v;
        }
        Q ph = expi(-(quad)dt * E[n] * ((N - 1) * (quad).5 * dx));
        const Q turn = expi((quad)dt * E[n] * dx);
        for (int j = N - 1; j >= 0; --j) {
            y = D[j] - qC[j] * y;
            P[j] = Q{2 * y.r - P[j].r, 2 * y.i - P[j].i} * ph * Q{g.m[j], 0};
            ph = ph * turn;
        }
    }
    for (int n = 0; n < nt; ++n) {   // the FP64 sweep: fused, the phase from sincos every 64 points of a segment
        double dr = 0, di = 0, yr = 0, yi = 0, phr = 1, phi = 0;
        for (int j = 0; j < N; ++j) {
            const cd l = j ? p[j - 1] : cd(0, 0), r = j < N - 1 ? p[j + 1] : cd(0, 0);
            const double rr = std::fma(10.0, p[j].real(), l.real() + r.real()), ri = std::fma(10.0, p[j].imag(), l.imag() + r.imag());
            const double wr = W[j].real(), wi = W[j].imag(), lr = L[j].real(), li = L[j].imag();
            const double nr = std::fma(wr, rr, std::fma(-wi, ri, std::fma(-lr, dr, li * di)));
            di = std::fma(wr, ri, std::fma(wi, rr, std::fma(-lr, di, -li * dr)));
            dr = nr;
            d[j] = cd(dr, di);
        }
        const double wr = std::cos(dt * E[n] * dx), wi = std::sin(dt * E[n] * dx);
        for (int j = N - 1; j >= 0; --j) {
            const double cr = C[j].real(), ci = C[j].imag(), nr = std::fma(-cr, yr, std::fma(ci, yi, d[j].real()));
            yi = std::fma(-cr, yi, std::fma(-ci, yr, d[j].imag()));
            yr = nr;
            if ((std::min(N, (j / m + 1) * m) - 1 - j) % 64 == 0) {
                phr = std::cos(-dt * E[n] * (x0 + j * dx));
                phi = std::sin(-dt * E[n] * (x0 + j * dx));
            }
            const double tr = std::fma(2., yr, -p[j].real()), ti = std::fma(2., yi, -p[j].imag());
            p[j] = cd(std::fma(tr, phr, -ti * phi) * g.m[j], std::fma(tr, phi, ti * phr) * g.m[j]);
            const double q = std::fma(phr, wr, -phi * wi);
            phi = std::fma(phr, wi, phi * wr);
            phr = q;
        }
    }
    struct Row {
        Digits wr, wi, lr, li, cr, ci, m;
    };
    vector<Row> T(N);
    auto dig = [](double v, int k) { return digits(std::llrint(std::ldexp(v, k))); };
    for (int j = 0; j < N; ++j)
        T[j] = Row{dig(W[j].real(), 65), dig(W[j].imag(), 65), dig(-L[j].real(), 64), dig(-L[j].imag(), 64), dig(-C[j].real(), 64),
                   dig(-C[j].imag(), 64), dig(g.m[j], 61)};
    Slice s(g.p0, 59);
    vector<int64_t> er(N), ei(N);
    const double th = dt * 0.15915494309189535, tl = std::fma(dt, 0.15915494309189535, -th) + dt * -9.839338337591243e-18;
    auto turns = [&](double xx, double e) {
        const double a = e * th, al = std::fma(e, th, -a) + e * tl, b = a * xx, bl = std::fma(a, xx, -b) + al * xx;
        return 2 * (uint64_t)std::llrint((b - std::rint(b)) * 9223372036854775808.0) + (uint64_t)std::llrint(bl * 18446744073709551616.0);
    };
    double most = 0;
    for (int n = 0; n < nt; ++n) {
        if (n % 16 == 0) {
            if (n) s.store();
            s.load();
        }
        int64_t dr = 0, di = 0, yr = 0, yi = 0, phr = 0, phi = 0, qr, qi;
        for (int j = 0; j < N; ++j) {
            const int64_t vr = (j ? s.r[j - 1] : 0) + 10 * s.r[j] + (j < N - 1 ? s.r[j + 1] : 0), vi = (j ? s.i[j - 1] : 0) + 10 * s.i[j] + (j < N - 1 ? s.i[j + 1] : 0);
            const Digits rr = digits(vr), ri = digits(vi), a = digits(dr), b = digits(di);
            const Row& t = T[j];
            dr = er[j] = mul2_fix(t.lr, a, negative(t.li), b, mul2_fix(t.wr, rr, negative(t.wi), ri));
            di = ei[j] = mul2_fix(t.lr, b, t.li, a, mul2_fix(t.wr, ri, t.wi, rr));
            for (int64_t v : {vr, vi, dr, di}) most = std::max(most, (double)std::abs(v));
        }
        fix_cos_sin(turns(dx, E[n]), qr, qi);
        const Digits tr = digits(qr), ti = digits(qi), nti = negative(ti);
        for (int j = N - 1; j >= 0; --j) {
            const Row& t = T[j];
            const Digits a = digits(yr), b = digits(yi);
            yr = mul2_fix(t.cr, a, negative(t.ci), b, er[j]);
            yi = mul2_fix(t.cr, b, t.ci, a, ei[j]);
            if (j == N - 1 || (j + 1) % m == 0) fix_cos_sin(turns(-(x0 + j * dx), E[n]), phr, phi);
            const Digits zr = digits(yr - s.r[j]), zi = digits(yi - s.i[j]), fr = digits(phr), fi = digits(phi), nfi = negative(fi);
            int64_t xr = mul2_fix62(zr, fr, zi, nfi), xi = mul2_fix62(zr, fi, zi, fr);
            phr = mul2_fix62(fr, tr, fi, nti);
            phi = mul2_fix62(fr, ti, fi, tr);
            if (g.m[j] != 1.0) {
                xr = mul_fix<3>(t.m, digits(xr));
                xi = mul_fix<3>(t.m, digits(xi));
            }
            s.r[j] = xr;
            s.i[j] = xi;
        }
    }
    s.store();
    return compare("numerov", g, P, p, s.p, most);
}

// FULL_CN by composed short segments of m points, halo K
static int short_segments(int N, double dx, double dt, int nt, int m, int K)
{
    Grid g(N, dx, dt, nt);
    const double beta = dt / (4 * dx * dx), h = 0.5 * dt, ib = 1 / beta, d2 = 2 * dx * dx;
    const FixClass F = fix_class(N, dx, dt, 2 + d2 / 1.19, d2 * .5 * (N - 1) * dx, 0.5);
    if (!F.ok) return 10;
    g.field(std::min(.06, .5 * F.E_lim));
    const auto& E = g.E;
    vector<Q> P(N), G(N), D(N);
    vector<cd> p = g.p0, gg(N), dd(N);
    for (int j = 0; j < N; ++j) P[j] = {p[j].real(), p[j].imag()};
    const quad qb = (quad)dt / (4 * (quad)dx * dx), i2 = 1 / ((quad)dx * dx);
    for (int n = 0; n < nt; ++n) {
        const quad eb = ((quad)E[n] + E[n + 1]) / 2;
        Q c{0, 0}, v{0, 0}, y{0, 0};
        for (int j = 0; j < N; ++j) {   // gamma = i conj(q) / |q|^2, D = -i gamma (psi + i D)
            const quad qr = 1 / qb + c.i, qi = (quad)h * (i2 + g.V[j] + (j - (quad).5 * (N - 1)) * dx * eb) / qb - c.r, w = 1 / (qr * qr + qi * qi);
            c = G[j] = {qi * w, qr * w};
            v = D[j] = Q{0, -1} * c * Q{P[j].r - v.i, P[j].i + v.r};
        }
        for (int j = N - 1; j >= 0; --j) {
            const Q t = G[j] * y;
            y = {t.r + D[j].r, t.i + D[j].i};
            P[j] = {(2 / qb * y.r - P[j].r) * g.m[j], (2 / qb * y.i - P[j].i) * g.m[j]};
        }
    }
    for (int n = 0; n < nt; ++n) {
        const double eb = .5 * (E[n] + E[n + 1]);
        double c = 0, s = 0, u = 0, v = 0, yr = 0, yi = 0;
        for (int j = 0; j < N; ++j) {
            const double qr = ib + s, qi = std::fma(h * g.x[j] / beta, eb, h * (1 / (dx * dx) + g.V[j]) / beta) - c, w = 1 / std::fma(qr, qr, qi * qi);
            c = qi * w;
            s = qr * w;
            const double ur = p[j].real() - v, ui = p[j].imag() + u;
            u = std::fma(c, ui, s * ur);
            v = std::fma(s, ui, -c * ur);
            gg[j] = {c, s};
            dd[j] = {u, v};
        }
        for (int j = N - 1; j >= 0; --j) {
            const double a = gg[j].real(), b = gg[j].imag(), t = std::fma(a, yr, std::fma(-b, yi, dd[j].real()));
            yi = std::fma(a, yi, std::fma(b, yr, dd[j].imag()));
            yr = t;
            p[j] = cd(std::fma(2 * ib, yr, -p[j].real()) * g.m[j], std::fma(2 * ib, yi, -p[j].imag()) * g.m[j]);
        }
    }
    const int n_seg = (N + m - 1) / m, Kg = (K + 1) / 2, Kr = std::min(m, K), T = (K + m - 1) / m, M = n_seg * m;
    vector<FixPoint> tab(N);
    vector<Digits> mask(N), ga(M), gb(M);
    vector<int64_t> Dr(M), Di(M);
    for (int j = 0; j < N; ++j) {
        tab[j] = fix_point(F, j, N, dx, g.V[j]);
        const FixObs o = fix_obs(F, 0.0, g.m[j]);
        mask[j] = Digits{o.m_h, o.m_l};
    }
    struct Edge {
        int64_t dr, di, yr, yi;
        Digits hr, hi;
    };
    vector<Edge> e(n_seg);
    Slice s(g.p0, F.top);
    auto pr = [&](int j) { return j < N ? s.r[j] : 0; };
    auto pi = [&](int j) { return j < N ? s.i[j] : 0; };
    double most = 0;
    for (int n = 0; n < nt; ++n) {
        if (n % 16 == 0) {
            if (n) s.store();
            s.load();
        }
        const Digits Eb = digits(std::llrint(.5 * (E[n] + E[n + 1]) * F.e_scale));
        auto row = [&](int j) { return diag_row(tab[std::min(std::max(j, 0), N - 1)], Eb); };
        for (int q = 0; q < n_seg; ++q) {
            int64_t gr = 0, gi = 0, dr = 0, di = 0;
            for (int j = q * m - Kg; j < q * m; ++j) {
                gamma_row(F.inv_b, row(j), gr, gi);
                if (j < 0) gr = gi = 0;
            }
            for (int r = 0; r < m; ++r) {
                const int j = q * m + r;
                gamma_row(F.inv_b, row(j), gr, gi);
                if (j >= N) gr = gi = 0;
                const Digits a = ga[j] = digits(gr << 6), b = gb[j] = digits(gi << 6);
                mul_minus_i(a, b, digits(pr(j) - di), digits(pi(j) + dr), dr, di);
                Dr[j] = dr;
                Di[j] = di;
                if (r == 0) {
                    e[q].hr = a;
                    e[q].hi = b;
                } else {
                    const int64_t x = mul2_fix(a, e[q].hr, negative(b), e[q].hi), y = mul2_fix(a, e[q].hi, b, e[q].hr);
                    e[q].hr = digits(x);
                    e[q].hi = digits(y);
                }
                if (T == 1) e[q].hr = e[q].hi = Digits{0, 0};
            }
            e[q].dr = dr;
            e[q].di = di;
        }
        auto compose = [&](int from, int step, int64_t Edge::*vr, int64_t Edge::*vi, int64_t& yr, int64_t& yi) {
            yr = yi = 0;
            for (int k = T; k >= 1; --k) {
                const int q = from + k * step;
                if (q < 0 || q >= n_seg) continue;
                const Digits a = digits(yr), b = digits(yi);
                const int64_t x = mul2_fix(e[q].hr, a, negative(e[q].hi), b, e[q].*vr), y = mul2_fix(e[q].hr, b, e[q].hi, a, e[q].*vi);
                yr = x;
                yi = y;
            }
        };
        auto back = [&](int j, int64_t& yr, int64_t& yi) {
            const Digits u = digits(yr), v = digits(yi);
            yr = mul2_fix(ga[j], u, negative(gb[j]), v, Dr[j]);
            yi = mul2_fix(ga[j], v, gb[j], u, Di[j]);
        };
        vector<Edge> first = e;
        for (int q = 0; q < n_seg; ++q) {
            int64_t dr, di, yr = 0, yi = 0;
            compose(q, -1, &Edge::dr, &Edge::di, dr, di);
            for (int r = 0; r < Kr; ++r) {
                const int j = q * m + r;
                mul_minus_i(ga[j], gb[j], digits(pr(j) - di), digits(pi(j) + dr), dr, di);
                Dr[j] = dr;
                Di[j] = di;
                most = std::max(most, (double)std::max(std::abs(dr), std::abs(di)));
            }
            for (int r = Kr - 1; r >= 0; --r) back(q * m + r, yr, yi);
            first[q].yr = yr;
            first[q].yi = yi;
        }
        e = first;
        for (int q = 0; q < n_seg; ++q) {
            int64_t yr, yi;
            compose(q, 1, &Edge::yr, &Edge::yi, yr, yi);
            for (int r = m - 1; r >= 0; --r) {
                const int j = q * m + r;
                back(j, yr, yi);
                if (j >= N) continue;
                int64_t xr = update_fix(F.ci, F.cf, digits(yr), s.r[j]), xi = update_fix(F.ci, F.cf, digits(yi), s.i[j]);
                if (g.m[j] != 1.0) {
                    xr = mul_fix<3>(mask[j], digits(xr));
                    xi = mul_fix<3>(mask[j], digits(xi));
                }
                s.r[j] = xr;
                s.i[j] = xi;
                most = std::max(most, (double)std::max(std::abs(xr), std::abs(xi)));
            }
        }
    }
    s.store();
    return compare("short", g, P, p, s.p, most);
}

// reciprocal: within 2^-53 over its range, 2^-55 for |Q|^2 < 128 (n < 2^59)
static int reciprocal()
{
    uint64_t state = 1;
    for (int k = 0; k < 2000000; ++k) {
        state = state * 6364136223846793005ull + 1442695040888963407ull;
        const int b = 55 + k % 6;
        const int64_t n = (int64_t(1) << b) + (int64_t)((state >> 3) & ((uint64_t(1) << b) - 1));
        const quad ex = (quad)std::ldexp(1.0, 116) / n;
        if (std::fabs((double)((recip_fix(n) - ex) / ex)) > std::ldexp(1.0, n < (int64_t(1) << 59) ? -55 : -53)) return 1;
    }
    return 0;
}

int main(int argc, char** argv)
{
    if (argc == 1) return reciprocal();
    const int N = std::atoi(argv[2]), nt = std::atoi(argv[5]), m = std::atoi(argv[6]);
    const double dx = std::atof(argv[3]), dt = std::atof(argv[4]);
    return argv[1][0] == 'n' ? numerov(N, dx, dt, nt, m) : short_segments(N, dx, dt, nt, m, std::atoi(argv[7]));
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not found")
    d = tmp_path_factory.mktemp("forms")
    (d / "forms.cpp").write_text(PROGRAM)
    r = subprocess.run(["g++", "-O2", "-std=gnu++17", "-I", CSRC, str(d / "forms.cpp"), "-o", str(d / "forms")],
                       capture_output=True, text=True)
    if "__float128" in r.stderr:
        pytest.skip("no 113-bit type on this machine")
    assert r.returncode == 0, r.stderr[-2000:]
    return str(d / "forms")


def test_reciprocal_bound(program):
    assert subprocess.run([program]).returncode == 0


# the workloads' grids and segments, odd sizes, one segment, the largest N
@pytest.mark.parametrize("N,dx,dt,steps,m", [(4096, 0.15, 0.02, 160, 256), (2000, 0.2, 0.05, 160, 63), (1537, 0.2, 0.05, 300, 200),
                                             (8192, 0.2, 0.02, 40, 512), (64, 0.2, 0.05, 100, 64), (401, 0.2, 0.05, 300, 401),
                                             (257, 0.12, 0.02, 300, 33), (32768, 0.2, 0.02, 8, 2048)])
def test_numerov_state_is_no_further_off_than_double(program, N, dx, dt, steps, m):
    r = subprocess.run([program, "n"] + [str(v) for v in (N, dx, dt, steps, m)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


# halos as planned (beta^K < 1e-18); segments of one row, shorter than the halo, as long, several times as long
@pytest.mark.parametrize("N,dx,dt,steps,m,K", [(2000, 0.2, 0.05, 160, 11, 36), (2048, 0.15, 0.02, 160, 64, 28), (401, 0.2, 0.05, 300, 36, 36),
                                               (300, 0.2, 0.05, 200, 1, 36), (1000, 0.2, 0.02, 160, 80, 20), (257, 0.2, 0.05, 300, 5, 36)])
def test_short_segments_are_no_further_off_than_double(program, N, dx, dt, steps, m, K):
    r = subprocess.run([program, "s"] + [str(v) for v in (N, dx, dt, steps, m, K)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
