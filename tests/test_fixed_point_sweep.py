"""The fixed-point arithmetic of the FULL_CN sweep (csrc/tdse_fix.cuh), compiled for the host: the same
steps in fixed point, in double and in 113 bits, on the grids' ranges.  The fixed-point state has to be
no further from the 113-bit one than the double state is, and its conversions and reciprocal within
their stated errors."""
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
#include <random>
#include <vector>
using namespace tdse;
using std::vector;
typedef __float128 quad;

static int conversions()
{
    std::mt19937_64 g(1);
    for (int i = 0; i < 300000; ++i) {
        // reciprocal: within 2^-53 over its range
        const int b = 55 + (int)(g() % 6);
        const int64_t n = (int64_t(1) << b) + (int64_t)(g() & ((uint64_t(1) << b) - 1));
        const quad ex = (quad)std::ldexp(1.0, 116) / n;
        if (std::fabs((double)((recip_fix(n) - ex) / ex)) > std::ldexp(1.0, -53)) return 1;
        // digits and back; the product of two numbers to one unit
        const int64_t v = (int64_t)g() >> 2, u = (int64_t)g() >> 2;
        if (undigits(digits(v)) != v) return 2;
        const quad p = (quad)v * u / (quad)std::ldexp(1.0, 64);
        if (std::fabs((double)(mul_fix<0>(digits(v), digits(u)) - p)) > 1.0) return 3;
        // doubles: to fixed point within half a unit, back within half an ulp
        const int sigma = 40 + (int)(g() % 30);
        const double d = std::ldexp((double)v, -(int)(g() % 90)) * std::ldexp(1.0, -sigma - 1);
        uint64_t bits;
        std::memcpy(&bits, &d, 8);
        const int64_t f = double_to_fix(bits, sigma);
        if (std::fabs((double)((quad)f - (quad)d * (quad)std::ldexp(1.0, sigma))) > 0.5) return 4;
        bits = fix_to_double(v, sigma);
        double w;
        std::memcpy(&w, &bits, 8);
        if (w != std::ldexp((double)v, -sigma) && std::fabs(w - std::ldexp((double)v, -sigma)) > std::fabs(w) * std::ldexp(1.0, -52)) return 5;
    }
    for (double d : {0.0, -0.0, 5e-324, -1e-310, 1e-300}) {
        uint64_t bits;
        std::memcpy(&bits, &d, 8);
        if (double_to_fix(bits, 61) != 0) return 6;
    }
    return fix_to_double(0, 61) == 0 ? 0 : 7;
}

// one batch instance: nt steps of FULL_CN on N points, three ways
static int sweep(int N, double dx, double dt, int nt)
{
    const double beta = dt / (4 * dx * dx), a = 1.19, h = 0.5 * dt;
    vector<double> x(N), V(N), m(N, 1.0), S0(N), X(N);
    double s0m = 0, xm = 0;
    for (int j = 0; j < N; ++j) {
        x[j] = (j - .5 * (N - 1)) * dx;
        V[j] = -1 / std::sqrt(x[j] * x[j] + a * a);
        S0[j] = h * (1 / (dx * dx) + V[j]) / beta;
        X[j] = h * x[j] / beta;
        s0m = std::max(s0m, std::fabs(S0[j]));
        xm = std::max(xm, std::fabs(X[j]));
        const double ax = std::fabs(x[j]) - (0.5 * N * dx - 20);
        if (ax > 0) m[j] = std::pow(std::cos(.5 * M_PI * ax / 20), .125);
    }
    const FixClass C = fix_class(N, dx, dt, s0m, xm, 0.5);
    if (!C.ok) return 10;
    vector<double> E(nt + 1);
    for (int n = 0; n <= nt; ++n) E[n] = std::min(.06, .5 * C.E_lim) * std::cos(.057 * n * dt);
    vector<std::complex<double>> p0(N);
    double n2 = 0;
    for (int j = 0; j < N; ++j) {
        p0[j] = std::exp(-std::sqrt(x[j] * x[j] + 1)) + 0.1 * std::exp(-(x[j] - 20) * (x[j] - 20) / 60.) * std::exp(std::complex<double>(0, 1.2 * x[j]));
        n2 += std::norm(p0[j]);
    }
    for (auto& z : p0) z /= std::sqrt(n2 * dx);

    vector<quad> Pr(N), Pi(N), Gr(N), Gi(N), Dr(N), Di(N);
    vector<double> pr(N), pi(N), gr(N), gi(N), dr(N), di(N);
    for (int j = 0; j < N; ++j) {
        Pr[j] = pr[j] = p0[j].real();
        Pi[j] = pi[j] = p0[j].imag();
    }
    const quad qb = (quad)dt / (4 * (quad)dx * dx);
    for (int n = 0; n < nt; ++n) {
        const quad Eb = ((quad)E[n] + E[n + 1]) / 2;
        quad c = 0, s = 0, u = 0, v = 0;
        for (int j = 0; j < N; ++j) {
            const quad Qr = 1 / qb + s, Qi = (quad)h * (1 / ((quad)dx * dx) + V[j] + (j - (quad).5 * (N - 1)) * dx * Eb) / qb - c;
            const quad inv = 1 / (Qr * Qr + Qi * Qi), ur = Pr[j] - v, ui = Pi[j] + u;
            c = Qi * inv;
            s = Qr * inv;
            u = c * ui + s * ur;
            v = s * ui - c * ur;
            Gr[j] = c; Gi[j] = s; Dr[j] = u; Di[j] = v;
        }
        quad yr = 0, yi = 0;
        for (int j = N - 1; j >= 0; --j) {
            const quad t = Gr[j] * yr - Gi[j] * yi + Dr[j];
            yi = Gr[j] * yi + Gi[j] * yr + Di[j];
            yr = t;
            Pr[j] = (2 / qb * yr - Pr[j]) * m[j];
            Pi[j] = (2 / qb * yi - Pi[j]) * m[j];
        }
    }
    const double ib = 1 / beta;
    for (int n = 0; n < nt; ++n) {
        const double Eb = .5 * (E[n] + E[n + 1]);
        double c = 0, s = 0, u = 0, v = 0;
        for (int j = 0; j < N; ++j) {
            const double Qr = ib + s, Qi = std::fma(X[j], Eb, S0[j]) - c, inv = 1 / std::fma(Qr, Qr, Qi * Qi);
            c = Qi * inv;
            s = Qr * inv;
            const double ur = pr[j] - v, ui = pi[j] + u;
            u = std::fma(c, ui, s * ur);
            v = std::fma(s, ui, -c * ur);
            gr[j] = c; gi[j] = s; dr[j] = u; di[j] = v;
        }
        double yr = 0, yi = 0;
        for (int j = N - 1; j >= 0; --j) {
            const double t = std::fma(gr[j], yr, std::fma(-gi[j], yi, dr[j]));
            yi = std::fma(gr[j], yi, std::fma(gi[j], yr, di[j]));
            yr = t;
            pr[j] = std::fma(2 * ib, yr, -pr[j]) * m[j];
            pi[j] = std::fma(2 * ib, yi, -pi[j]) * m[j];
        }
    }
    // fixed point: directions alternate, (gamma, u) stored, psi recovered exactly
    int sigma = 0;
    vector<int64_t> fr(N), fi(N);
    vector<Digits> kr(N), ki(N), ur(N), ui(N);
    vector<FixPoint> T(N);
    vector<FixObs> O(N);
    for (int j = 0; j < N; ++j) {
        T[j] = fix_point(C, j, N, dx, V[j]);
        O[j] = fix_obs(C, 0.0, m[j]);
    }
    auto to_fix = [&](double v) {
        uint64_t b;
        std::memcpy(&b, &v, 8);
        return double_to_fix(b, sigma);
    };
    auto to_double = [&](int64_t v) {
        const uint64_t b = fix_to_double(v, sigma);
        double w;
        std::memcpy(&w, &b, 8);
        return w;
    };
    // as a scheduling slice starts: the state in double, scaled by its norm
    auto load = [&]() {
        double t = 0;
        for (auto& z : p0) t += std::norm(z);
        int e2;
        std::frexp(t, &e2);
        sigma = C.top - ((e2 - 1 + 2) >> 1);
        for (int j = 0; j < N; ++j) {
            fr[j] = to_fix(p0[j].real());
            fi[j] = to_fix(p0[j].imag());
        }
    };
    auto store = [&]() {
        for (int j = 0; j < N; ++j) p0[j] = {to_double(fr[j]), to_double(fi[j])};
    };
    int64_t most = 0;
    for (int n = 0; n < nt; ++n) {
        if (n % 16 == 0) {
            if (n > 0) store();
            load();
        }
        const int d = n % 2 ? -1 : 1;
        const Digits Ed = digits(std::llrint(.5 * (E[n] + E[n + 1]) * C.e_scale));
        int64_t c = 0, s = 0, u = 0, v = 0;
        for (int t = 0; t < N; ++t) {
            const int j = d > 0 ? t : N - 1 - t;
            gamma_row(C.inv_b, diag_row(T[j], Ed), c, s);
            kr[j] = digits(c << 6);
            ki[j] = digits(s << 6);
            ur[j] = digits(fr[j] - v);
            ui[j] = digits(fi[j] + u);
            mul_minus_i(kr[j], ki[j], ur[j], ui[j], u, v);
            most = std::max(most, std::max(std::abs(undigits(ur[j])), std::abs(u)));
        }
        int64_t yr = 0, yi = 0;
        for (int t = N - 1; t >= 0; --t) {
            const int j = d > 0 ? t : N - 1 - t, k = j - d;
            int64_t ar, ai, br = 0, bi = 0;
            mul_minus_i(kr[j], ki[j], ur[j], ui[j], ar, ai);
            if (t > 0) mul_minus_i(kr[k], ki[k], ur[k], ui[k], br, bi);
            const Digits y = digits(yr), z = digits(yi);
            yr = mul2_fix(kr[j], y, negative(ki[j]), z, ar);
            yi = mul2_fix(kr[j], z, ki[j], y, ai);
            const int64_t qr = undigits(ur[j]) + bi, qi = undigits(ui[j]) - br;
            if (qr != fr[j] || qi != fi[j]) return 11;
            int64_t nr = update_fix(C.ci, C.cf, digits(yr), qr), ni = update_fix(C.ci, C.cf, digits(yi), qi);
            if (m[j] != 1.0) {
                const Digits mm{O[j].m_h, O[j].m_l};
                nr = mul_fix<3>(mm, digits(nr));
                ni = mul_fix<3>(mm, digits(ni));
            }
            fr[j] = nr;
            fi[j] = ni;
        }
    }
    store();
    quad nd = 0, nf = 0, nq = 0;
    for (int j = 0; j < N; ++j) {
        const quad f = p0[j].real(), g = p0[j].imag();
        nq += Pr[j] * Pr[j] + Pi[j] * Pi[j];
        nd += (Pr[j] - pr[j]) * (Pr[j] - pr[j]) + (Pi[j] - pi[j]) * (Pi[j] - pi[j]);
        nf += (Pr[j] - f) * (Pr[j] - f) + (Pi[j] - g) * (Pi[j] - g);
    }
    const double ed = std::sqrt((double)(nd / nq)), ef = std::sqrt((double)(nf / nq));
    std::printf("N %d dx %g dt %g steps %d: double %.3g fixed %.3g largest 2^%.2f\n", N, dx, dt, nt, ed, ef, std::log2((double)most));
    return ef <= ed && most < (int64_t(1) << 61) ? 0 : 12;
}

int main(int argc, char** argv)
{
    if (argc == 1) return conversions();
    return sweep(std::atoi(argv[1]), std::atof(argv[2]), std::atof(argv[3]), std::atoi(argv[4]));
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not found")
    d = tmp_path_factory.mktemp("fix")
    (d / "fix.cpp").write_text(PROGRAM)
    r = subprocess.run(["g++", "-O2", "-std=gnu++17", "-I", CSRC, str(d / "fix.cpp"), "-o", str(d / "fix")],
                       capture_output=True, text=True)
    if "__float128" in r.stderr:
        pytest.skip("no 113-bit type on this machine")
    assert r.returncode == 0, r.stderr[-2000:]
    return str(d / "fix")


def test_conversions_products_and_reciprocal(program):
    assert subprocess.run([program]).returncode == 0


# the grids of the workloads, odd sizes, both ends of beta's range, the largest N
@pytest.mark.parametrize("N,dx,dt,steps", [(4096, 0.15, 0.02, 160), (2000, 0.2, 0.05, 160), (8192, 0.2, 0.02, 40),
                                           (8192, 0.15, 0.02, 20), (1537, 0.2, 0.05, 300), (257, 0.12, 0.02, 300),
                                           (501, 0.26, 0.02, 200), (32768, 0.2, 0.02, 8), (64, 0.2, 0.05, 100)])
def test_fixed_point_state_is_no_further_off_than_double(program, N, dx, dt, steps):
    r = subprocess.run([program, str(N), str(dx), str(dt), str(steps)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
