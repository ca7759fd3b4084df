// NUMEROV_SPLIT sweep in 64-bit fixed point (FP64 batches): one scheduling slice of a group, 32-wide or
// lane-split (lane geometry of GroupDesc), with the arithmetic of tdse_fix.cuh on the integer pipe.
//
// The step of tdse_numerov.cu: d_j = W_j r_j - L_j d_{j-1} with r = psi_{j-1} + 10 psi_j + psi_{j+1} forward,
// y_j = d_j - C_j y_{j+1} backward, psi' = m e^{-i dt E x} (2 y - psi).  Scales:
//   psi    2^sigma, 2-norm in [2^58, 2^59): |r| <= sqrt(102) ||psi|| < 2^62.4
//   W/12   2^65, L, C 2^64 (|L|, |C| <= 0.35), so d and y come at 2^(sigma+1): 2 y is y's integer
//   phase  2^62, turned from point to point by a fixed-point product (2^-62 a turn) from one sincos a step
//          at the segment's last point
// The factors are the FP64 path's, rounded to 2^-65; all else carries 59 bits of the state's norm.
//   During the slice the group's wavefunctions hold integers in place of the doubles; they are converted
// when the slice begins and ends.  A warp's forward sweep starts K rows before its segment (reading the
// neighbours' psi), its back substitution K rows after it (reading the neighbours' d, which the barrier
// between the sweeps has completed): no row of the scratch is computed twice.
//
// What bounds it: about 250 instructions a row on the integer pipes (five complex products of 30, observables
// 45), against 28 FP64 instructions of 64 cycles each; 80 B of traffic a point and step.
#pragma once

#include "tdse_sched.cuh"

namespace tdse {

struct FixZ {
    int64_t r, i;
};
__device__ __forceinline__ FixZ load_fix(const double2* p)
{
    const int4 v = __ldcg(reinterpret_cast<const int4*>(p));
    return FixZ{(int64_t)(((uint64_t)(uint32_t)v.y << 32) | (uint32_t)v.x), (int64_t)(((uint64_t)(uint32_t)v.w << 32) | (uint32_t)v.z)};
}
__device__ __forceinline__ void store_fix(double2* p, int64_t r, int64_t i)
{
    __stcg(reinterpret_cast<int4*>(p), make_int4((int)(uint32_t)(uint64_t)r, (int)(uint32_t)((uint64_t)r >> 32),
                                                 (int)(uint32_t)(uint64_t)i, (int)(uint32_t)((uint64_t)i >> 32)));
}

// Returns false, having changed nothing, when a live instance's field is not finite (or beyond any use) or its
// norm out of range: the caller then takes the FP64 sweep.
__device__ __forceinline__ bool fix_numerov_slice(const GroupDesc& G, const ClassDesc& C, const double* __restrict__ tab,
                                                  double2* ps, int64_t nt, int64_t row, int64_t slot, int64_t n0, int64_t n1,
                                                  bool initial, double dt, const double* __restrict__ E,
                                                  double* __restrict__ d_out, double* __restrict__ a_out, int64_t sample_base,
                                                  int4* buf, double* red, int* status, int jm_lo, int jm_hi)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, P = blockDim.x >> 5;
    const int I = G.I, i = lane & (I - 1), q = lane / I;
    const int N = G.N, K = G.K, m = G.m;
    const bool on = w < G.P;
    const int s = (w * (kLanes / I) + q) * m;
    const int s_own = on ? min(N, s) : N, e_own = on ? min(N, s + m) : N;
    const bool live = nt > n0;
    const double dx = C.dx, x0 = -0.5 * (N - 1) * dx;
    const int4* __restrict__ tW = reinterpret_cast<const int4*>(tab + tab_fnw(C));   // (W/12, -L, -C) as digits per point
    const int4* __restrict__ tO = reinterpret_cast<const int4*>(tab + tab_fob(C));
    auto at = [&](int j) { return ps + (int64_t)j * I + i; };

    bool ok = true;
    if (live)   // the phase dt E x below 10^6 rad, where its reduction keeps 2^-60
        for (int64_t n = n0; n <= min(n1, nt); ++n) ok = ok && fabs(E[row + n - sample_base] * (dt * x0)) < 1e6;
    float sq = 0.0f;
    if (live)
        for (int j = s_own; j < e_own; ++j) {
            const double2 p = ld_cg(at(j));
            const float a = d2f(p.x), b = d2f(p.y);
            sq = fmaf(a, a, fmaf(b, b, sq));
        }
    for (int off = I; off < kLanes; off <<= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
    float* redf = reinterpret_cast<float*>(red);
    redf[w * kLanes + lane] = sq;
    __syncthreads();
    float tot = 0.0f;
    for (int k = 0; k < P; ++k) tot += redf[k * kLanes + lane];
    __syncthreads();
    ok = ok && (!live || (tot > 1e-30f && tot < 1e30f));
    if (!__all_sync(0xffffffffu, ok)) return false;
    const int e2 = live ? (int)((__float_as_uint(tot) >> 23) & 0xffu) - 127 : 0;
    const int sigma = 59 - ((e2 + 2) >> 1);

    auto lane_sum = [&](ObsSums o) {
        for (int off = I; off < kLanes; off <<= 1) {
            o.n += __shfl_xor_sync(0xffffffffu, o.n, off);
            o.x += __shfl_xor_sync(0xffffffffu, o.x, off);
            o.v += __shfl_xor_sync(0xffffffffu, o.v, off);
        }
        return o;
    };
    if (initial) {
        const double2* __restrict__ tab_xv2 = reinterpret_cast<const double2*>(tab + tab_xv(C));
        ObsSums o{0.0, 0.0, 0.0};
        for (int j = s_own; j < e_own; ++j) {
            const double2 p = ld_cg(at(j));
            const double rho = fma(p.x, p.x, p.y * p.y);
            const double2 xv = __ldg(tab_xv2 + j);
            o.n += rho;
            o.x = fma(xv.x, rho, o.x);
            o.v = fma(xv.y, rho, o.v);
        }
        const ObsSums t = reduce_obs(lane_sum(o), red, P);
        if (w == 0 && q == 0 && nt >= 0) {
            const double E0 = E[row - sample_base];
            d_out[row - sample_base] = t.x * dx;
            a_out[row - sample_base] = fma(E0, t.n, t.v) * dx;
        }
    }
    // to integers, in place (own points of live instances)
    if (live)
        for (int j = s_own; j < e_own; ++j) {
            const double2 p = ld_cg(at(j));
            store_fix(at(j), double_to_fix((uint64_t)__double_as_longlong(p.x), sigma),
                      double_to_fix((uint64_t)__double_as_longlong(p.y), sigma));
        }
    __syncthreads();

    const double unit = __hiloint2double((1023 + 56 - 2 * sigma) << 20, 0);   // rho_int = |psi|^2 2^(2 sigma - 56)
    int4* own = buf + (int64_t)w * m * kLanes + lane;   // d of row r at own + r * 32
    auto load_psi = [&](int j) { return live && (unsigned)j < (unsigned)N ? load_fix(at(j)) : FixZ{0, 0}; };

    // x dt E in turns, modulo one, at 2^64: dt / (2 pi) and the products as pairs of doubles
    const double turn_h = dt * 0.15915494309189535, turn_l = fma(dt, 0.15915494309189535, -turn_h) + dt * -9.839338337591243e-18;
    auto turns = [&](double x, double e) {
        const double a = e * turn_h, al = fma(e, turn_h, -a) + e * turn_l;
        const double b = a * x, bl = fma(a, x, -b) + al * x;
        return 2 * (uint64_t)__double2ll_rn((b - rint(b)) * 9223372036854775808.0) + (uint64_t)__double2ll_rn(bl * 18446744073709551616.0);
    };

    for (int64_t n = n0; n < n1; ++n) {
        const bool active = n < nt;
        double En = 0.0, En1 = 0.0;
        if (active) {
            En = E[row + n - sample_base];
            En1 = E[row + n + 1 - sample_base];
        }
        // ---- forward, ascending, from K rows before the segment
        if (on) {
            int64_t dr = 0, di = 0;
            FixZ pm = load_psi(s - K - 1), pc = load_psi(s - K), pn = load_psi(s - K + 1), x1 = load_psi(s - K + 2);
            const int4* __restrict__ t0 = tW + 3 * (int64_t)min(max(s - K, 0), N - 1);
            const int4* __restrict__ t1 = tW + 3 * (int64_t)min(max(s - K + 1, 0), N - 1);
            int4 twn = __ldg(t0), tln = __ldg(t0 + 1);   // factors two rows ahead: the table (196 KB at
            int4 tw2 = __ldg(t1), tl2 = __ldg(t1 + 1);   // N = 4096) is read from L2 as much as from L1
            for (int r = -K; r < m; ++r) {
                const int j = s + r;
                const FixZ x2 = r + 2 < m ? load_psi(j + 3) : FixZ{0, 0};
                const bool in = (unsigned)j < (unsigned)N;
                const int4 tw = twn, tl = tln;
                const int4* __restrict__ t = tW + 3 * (int64_t)min(max(j + 2, 0), N - 1);
                twn = tw2;
                tln = tl2;
                tw2 = __ldg(t);
                tl2 = __ldg(t + 1);
                const Digits wr{tw.x, tw.y}, wi{tw.z, tw.w}, lr{tl.x, tl.y}, li{tl.z, tl.w};
                const Digits rr = digits(pm.r + 10 * pc.r + pn.r), ri = digits(pm.i + 10 * pc.i + pn.i);
                const Digits er = digits(dr), ei = digits(di);
                const int64_t nr = mul2_fix(lr, er, negative(li), ei, mul2_fix(wr, rr, negative(wi), ri));
                const int64_t ni = mul2_fix(lr, ei, li, er, mul2_fix(wr, ri, wi, rr));
                dr = in ? nr : 0;
                di = in ? ni : 0;
                if (r >= 0) {
                    const Digits a = digits(dr), b = digits(di);
                    __stcg(own + (int64_t)r * kLanes, make_int4(a.h, a.l, b.h, b.l));
                }
                pm = pc;
                pc = pn;
                pn = x1;
                x1 = x2;
            }
        }
        __syncthreads();   // every d is complete; every read of psi^n by a neighbour precedes its update

        // ---- backward, descending, from K rows after the segment
        ObsSums o{0.0, 0.0, 0.0};
        if (on) {
            int64_t yr = 0, yi = 0;
            const bool whole = K > 0;
            int r = m - 1 + (whole ? K : 0);
            int dq = r / m, lr_ = r - dq * m;
            auto load_d = [&](int j) {   // d at the current (segment, row); steps down one row
                int4 v = make_int4(0, 0, 0, 0);
                if ((unsigned)j < (unsigned)N) {
                    const int col = w * kLanes + lane + dq * I;
                    v = __ldcg(buf + ((int64_t)(col >> 5) * m + lr_) * kLanes + (col & 31));
                }
                if (--lr_ < 0) {
                    lr_ = m - 1;
                    --dq;
                }
                return v;
            };
            auto back = [&](const int4& d, const int4& c) {
                const Digits cr{c.x, c.y}, ci{c.z, c.w}, er = digits(yr), ei = digits(yi);
                const int64_t a = undigits(Digits{d.x, d.y}), b = undigits(Digits{d.z, d.w});
                yr = mul2_fix(cr, er, negative(ci), ei, a);
                yi = mul2_fix(cr, ei, ci, er, b);
            };
            auto coef = [&](int j) { return __ldg(tW + 3 * (int64_t)min(max(j, 0), N - 1) + 2); };
            int j = s + r;
            int4 d0 = load_d(j), d1 = load_d(j - 1), d2 = load_d(j - 2);
            int4 c0 = coef(j), c1 = coef(j - 1);
            for (; r >= m; --r, --j) {   // d of rows at or beyond the far wall is zero: y stays zero there
                const int4 d = d0, c = c0;
                d0 = d1;
                d1 = d2;
                d2 = r > 2 ? load_d(j - 3) : make_int4(0, 0, 0, 0);
                c0 = c1;
                c1 = coef(j - 2);
                back(d, c);
            }
            // phase e^{-i dt E x_j} at the segment's last point, and its turn to the next lower one
            int64_t phr, phi, qr_, qi_;
            fix_cos_sin(turns(-(x0 + j * dx), En), phr, phi);
            fix_cos_sin(turns(dx, En), qr_, qi_);
            const Digits tr = digits(qr_), ti = digits(qi_), nti = negative(ti);
            int64_t sn = 0, sxh = 0, sxl = 0, svh = 0, svm = 0;
            FixZ p0 = load_psi(j), p1 = load_psi(j - 1);
            int4 o0 = __ldg(tO + min(max(j, 0), N - 1)), o1 = __ldg(tO + min(max(j - 1, 0), N - 1));
            for (; r >= 0; --r, --j) {
                const int4 d = d0, c = c0, ob = o0;
                const FixZ p = p0;
                d0 = d1;
                d1 = d2;
                d2 = r > 2 ? load_d(j - 3) : make_int4(0, 0, 0, 0);
                c0 = c1;
                c1 = coef(j - 2);
                p0 = p1;
                p1 = r > 1 ? load_psi(j - 2) : FixZ{0, 0};
                o0 = o1;
                o1 = __ldg(tO + min(max(j - 2, 0), N - 1));
                back(d, c);
                const Digits zr = digits(yr - p.r), zi = digits(yi - p.i);   // 2 y - psi
                const Digits fr = digits(phr), fi = digits(phi), nfi = negative(fi);
                int64_t xr = mul2_fix62(zr, fr, zi, nfi), xi = mul2_fix62(zr, fi, zi, fr);
                phr = mul2_fix62(fr, tr, fi, nti);
                phi = mul2_fix62(fr, ti, fi, tr);
                if (j < jm_lo || j > jm_hi) {
                    const Digits mm{ob.w, ob.z};
                    xr = mul_fix<3>(mm, digits(xr));
                    xi = mul_fix<3>(mm, digits(xi));
                }
                const bool in = (unsigned)j < (unsigned)N;
                if (!in) xr = xi = 0;
                if (active && in) store_fix(at(j), xr, xi);
                const Digits a = digits(xr), b = digits(xi);
                const uint64_t ll = (uint64_t)mad(a.l, a.l, mad(b.l, b.l, 0)) >> 33;
                const int64_t rho = combine<8, 23>(mad(a.h, a.h, mad(b.h, b.h, 0)),
                                                   mad(a.h, a.l, mad(b.h, b.l, (int64_t)ll + (int64_t(1) << 22))));
                const Digits rd = digits(rho);
                const int wj = 2 * j - N + 1;
                sn += rho;
                sxh = mad(rd.h, wj, sxh);
                sxl = mad(rd.l, wj, sxl);
                svh = mad(rd.h, ob.y, svh) + (mad(rd.l, ob.y, int64_t(1) << 31) >> 32);
                svm = mad(rd.h, ob.x, svm);
            }
            const double two32 = 4294967296.0;
            o.n = (double)sn * unit;
            o.x = fma((double)sxh, two32, (double)sxl) * (0.5 * dx * unit);
            o.v = fma((double)svh, two32, (double)svm) * (two32 * C.fix.v_scale * unit);
        }
        const ObsSums t = reduce_obs(lane_sum(o), red, P);   // its barrier orders this step's writes
        if (w == 0 && q == 0 && active) {
            const int64_t kk = row + n + 1 - sample_base;
            d_out[kk] = t.x * dx;
            a_out[kk] = fma(En1, t.n, t.v) * dx;
            if (!(t.n * dx <= 1.0 + 1e-6)) status[slot] = 1;
        }
    }
    // back to doubles
    if (live)
        for (int j = s_own; j < e_own; ++j) {
            const FixZ p = load_fix(at(j));
            __stcg(at(j), make_double2(__longlong_as_double((long long)fix_to_double(p.r, sigma)),
                                       __longlong_as_double((long long)fix_to_double(p.i, sigma))));
        }
    __syncthreads();
    return true;
}

}  // namespace tdse
