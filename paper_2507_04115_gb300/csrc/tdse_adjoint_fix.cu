// The adjoint of FULL_CN (see tdse_adjoint.cu for the method and its formulas) with both of its sweeps in
// 64-bit fixed point on the integer pipe: the recomputation of a checkpoint interval and the backward
// sweeps each solve with A_n by short_solve (tdse_cn_fix.cuh), which serves segments of any length.
//
//   * psi of an interval: converted from its checkpoint at 2^sp; the pre-mask states of every step go to
//     the CTA's tape as integers; sum |psi^n|^2 and sum x^2 |psi^n|^2 of every sample to a small per-CTA array.
//   * the backward sweep carries kappa = conj(lambda): rhs = M kappa^{n+1}, A_n y = rhs, kappa^n = 2 y - rhs +
//     conj(g^n), g^n = w_j psi^n_j with w_j = 2 dx (gd_n x_j + ga_n (dV_j + E_n)), the next rhs = M kappa^n.  Its
//     scale 2^sk follows its norm: the solve does not increase the 2-norm, so ||M kappa^{n+1}|| + ||g^n|| bounds
//     the step, the first measured by the step before, ||g^n|| <= 2 dx (|gd| ||x psi|| + |ga| (max |dV| + |E|)
//     ||psi||) from the two sums above; rhs is shifted with its exponent.  (One scale per interval, from the sum
//     of all its bounds, is some four bits coarser.)  Between intervals rhs is kept as doubles.
//   * w_j at 2^(61-e) (|w_j| < 2^e): x_j = (2j - N + 1) dx/2 times a constant with up to 12 extra bits, dV_j times a
//     constant, a constant.
// A group with a field, a state or a gradient outside the fixed-point range is left to k_adjoint_full_cn, which is
// launched behind this kernel for the groups marked in `left`.
//
// What bounds it: the integer pipes, as in fix_short_slice; the FP64 kernel takes 27 FP64 instructions a row forward and
// 30 backward, of 64 cycles each.  Measured, 1024 x 2048 points, 96 steps, an interval of 32, the recording given:
// 44.4 ms with the FP64 kernel, 14.7 here.  Error of the gradient against 113 bits, dx 0.2, dt 0.05, N = 601 and 2000:
// 1.5 and 1.0e-15 there, 1.1 and 0.8e-15 here; dx 0.15, dt 0.02, N = 1001: 1.0e-15 and 0.2e-15.
#include "tdse_cn_fix.cuh"

namespace tdse {

namespace {

__device__ __forceinline__ double pow2(int k) { return __hiloint2double((1023 + k) << 20, 0); }

// (w p) 2^-(32 + t) rounded, 1 <= t <= 95, all four partial products: `round` is half a unit of the result, in
// the words below 2^64 (t <= 32, lo) or above (hi).
struct Shift {
    int t;
    int64_t round_lo, round_hi;
};
__device__ __forceinline__ Shift shift_of(int sh)
{
    const int t = sh - 32;
    return Shift{t, t <= 32 ? int64_t(1) << (t - 1) : 0, t <= 32 ? 0 : int64_t(1) << (t - 33)};
}
__device__ __forceinline__ int64_t mul_shift(Digits w, Digits p, const Shift& S)
{
    const int64_t low = mad(w.l, p.l, 0) >> 32;
    const int64_t mid = mad(w.h, p.l, mad(w.l, p.h, S.round_lo + low));
    const int64_t hi = fold(mad(w.h, p.h, S.round_hi), mid);   // the product 2^-64; the low word of mid below it
    const uint32_t a = (uint32_t)(uint64_t)mid, b = (uint32_t)(uint64_t)hi, c = (uint32_t)((uint64_t)hi >> 32);
    const int64_t fine = (int64_t)(((uint64_t)__funnelshift_r(b, c, S.t) << 32) | __funnelshift_r(a, b, S.t));
    return S.t < 32 ? fine : hi >> (S.t - 32);
}

struct FixWeights {
    Digits cx, cv;
    int64_t ce;
    int e;
};

}  // namespace

__global__ void __launch_bounds__(512, 1)
k_adjoint_fix(const GroupDesc* __restrict__ groups, int64_t n_groups, const ClassDesc* __restrict__ cls,
              const double* __restrict__ tab, const int64_t* __restrict__ slot_row, const int64_t* __restrict__ slot_nt,
              const double2* __restrict__ psi0_all, double2* __restrict__ lam_all, double2* __restrict__ ckpt_all,
              const int64_t* __restrict__ ckpt_off, double2* __restrict__ sums_all, double2* __restrict__ tape_all,
              int4* __restrict__ scratch_all, int64_t scratch_per_cta, int n_max, int kc, const double* __restrict__ E,
              const double* __restrict__ gd, const double* __restrict__ ga, double* __restrict__ gE, int mask_on,
              int* __restrict__ busy, int* __restrict__ progress, int* __restrict__ left, int have_ckpt)
{
    extern __shared__ double red[];   // [P][3][32], then the edges
    __shared__ int s_g, s_bad;
    __shared__ double s_bound[kLanes], s_norm[kLanes];   // of an instance's kappa
    __shared__ FixWeights s_w[kLanes];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, P = blockDim.x >> 5;
    FixEdge* const edge = reinterpret_cast<FixEdge*>(red + P * 3 * kLanes);
    int4* const buf = scratch_all + (int64_t)blockIdx.x * scratch_per_cta;
    int4* const tape = reinterpret_cast<int4*>(tape_all) + (int64_t)blockIdx.x * kc * n_max * kLanes;
    double2* const sums = sums_all + (int64_t)blockIdx.x * n_max * kLanes;   // sample na + k of instance i at k * 32 + i
    const int64_t whole = int64_t(1) << 40;

    for (;;) {
        if (w == 0) {
            int k = 0;
            const int g = pick_group(groups, n_groups, busy, progress, 0, whole, (int)(whole >> 10), &k);
            if (lane == 0) {
                s_g = g;
                s_bad = 0;
            }
        }
        __syncthreads();
        const int gi = s_g;
        __threadfence();
        __syncthreads();
        if (gi < 0) break;

        const GroupDesc G = groups[gi];
        const ClassDesc C = cls[G.cls];
        const FixClass& F = C.fix;
        const int N = G.N, I = G.I, m = G.m, K = G.K;
        const int i = lane & (I - 1), q = lane / I, L = kLanes / I;
        const bool on = w < G.P;
        const int sg = w * L + q, n_seg = G.P * L, s = sg * m;
        const int s_own = on ? min(N, s) : N, e_own = on ? min(N, s + m) : N;
        const int64_t slot = G.slot0 + i, nt = slot_nt[slot], row = slot_row[slot], nt_max = G.nt_max;
        const int64_t state = (int64_t)N * I;
        const int xb = min(12, 31 - __clz(max(N - 1, 1)));   // extra bits of the x weight: its integer stays below 2^62
        const double dx = C.dx, x_max = 0.5 * (N - 1) * dx, dv_max = pow2(F.kv);
        const int4* __restrict__ tO = reinterpret_cast<const int4*>(tab + tab_fob(C));
        const int jm_lo = mask_on ? C.jm_lo : 0, jm_hi = mask_on ? C.jm_hi : N - 1;
        double2* __restrict__ lam = lam_all + G.psi_off;
        double2* __restrict__ ck = ckpt_all + ckpt_off[gi];
        const int64_t n_int = (nt_max + kc - 1) / kc;
        const bool real = nt >= 0;
        int4* const own = buf + (int64_t)w * m * (3 * kLanes) + lane;
        const ShortGeom geo{N, K, m, I, s, sg, n_seg, w * kLanes + lane, on, own, edge, reinterpret_cast<const int4*>(tab + tab_fxp(C)),
                            F.inv_b};
        const int32_t ci = F.ci;
        const Digits cf = F.cf;
        auto at = [&](int j) { return (int64_t)j * I + i; };

        // every field of the group in range?
        bool ok = F.ok && K > 0;
        if (real)
            for (int64_t n = w * L + q; n <= nt; n += P * L) {
                gE[row + n] = 0.0;
                ok = ok && fabs(E[row + n]) <= F.E_lim;
            }
        if (!ok) s_bad = 1;
        __syncthreads();
        bool bad = s_bad != 0;

        // sum of |p|^2 over the grid points of an instance, on every lane of it
        auto norm2 = [&](const double2* __restrict__ p, bool use) {
            double t = 0.0;
            if (use)
                for (int j = s_own; j < e_own; ++j) {
                    const double2 v = ld_cg(p + at(j));
                    t = fma(v.x, v.x, fma(v.y, v.y, t));
                }
            for (int off = I; off < kLanes; off <<= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
            red[w * kLanes + lane] = t;
            __syncthreads();
            double r = 0.0;
            for (int k = 0; k < P; ++k) r += red[k * kLanes + lane];
            __syncthreads();
            return r;
        };
        // binary exponent such that v < 2^result (v > 0 finite)
        auto above = [](double v) { return ((__double2hiint(v) >> 20) & 0x7ff) - 1022; };
        // one forward step on the rows' right-hand sides; the pre-mask state goes to tape_n (or nowhere)
        auto forward = [&](int64_t n, int4* tape_n, double2* ck_out, int sigma, double& n_sum, double& x2_sum) {
            const bool active = n < nt;
            const Digits Eb = digits(active ? __double2ll_rn(0.5 * (E[row + n] + E[row + n + 1]) * F.e_scale) : 0);
            int64_t yr, yi;
            short_solve(geo, Eb, yr, yi);
            int64_t sn = 0;
            float x2 = 0.0f;
            if (on) {
                int4* o = own + (int64_t)(m - 1) * (3 * kLanes);
                int4 gn = o[0], pn = o[kLanes], dn = o[2 * kLanes];
                for (int r = m - 1; r >= 0; --r) {
                    const int j = s + r;
                    const int4 g = gn, p = pn, d = dn;
                    if (r > 0) {
                        gn = o[-3 * kLanes];
                        pn = o[-2 * kLanes];
                        dn = o[-kLanes];
                    }
                    back_row(g, d, yr, yi);
                    int64_t xr = update_fix(ci, cf, digits(yr), lo64(p)), xi = update_fix(ci, cf, digits(yi), hi64(p));
                    if (!active || j >= N) {   // finished instances keep their state
                        xr = lo64(p);
                        xi = hi64(p);
                    }
                    if (tape_n && j < N) {
                        int4 v;
                        put64(&v, xr, xi);
                        __stcg(tape_n + at(j), v);
                    }
                    if (active && (j < jm_lo || j > jm_hi)) {
                        const int4 ob = __ldg(tO + min(j, N - 1));
                        const Digits mm{ob.w, ob.z};
                        xr = mul_fix<3>(mm, digits(xr));
                        xi = mul_fix<3>(mm, digits(xi));
                    }
                    put64(o + kLanes, xr, xi);
                    if (ck_out && j < N)
                        ck_out[at(j)] = make_double2(__longlong_as_double((long long)fix_to_double(xr, sigma)),
                                                     __longlong_as_double((long long)fix_to_double(xi, sigma)));
                    const Digits a = digits(xr), b = digits(xi);
                    const uint64_t ll = (uint64_t)mad(a.l, a.l, mad(b.l, b.l, 0)) >> 33;
                    const int64_t rho = combine<4, 27>(mad(a.h, a.h, mad(b.h, b.h, 0)),
                                                       mad(a.h, a.l, mad(b.h, b.l, (int64_t)ll + (int64_t(1) << 26))));
                    sn += rho;
                    const float xf = (float)(2 * j - N + 1);
                    x2 = fmaf(xf * xf, (float)((int32_t)((uint64_t)rho >> 32) + 1), x2);   // from above
                    o -= 3 * kLanes;
                }
            }
            // rho = |psi|^2 2^(2 sigma - 60)
            const double unit = __hiloint2double((1023 + 60 - 2 * sigma) << 20, 0);
            ObsSums o{(double)sn * unit, (double)x2 * (unit * 4294967296.0 * 0.25 * dx * dx), 0.0};
            const ObsSums t = reduce_obs(fix_lane_sum(o, I), red, P);
            n_sum = t.n;     // warp 0
            x2_sum = t.x;
        };
        // the state at p (doubles) into the rows, at the scale of its norm; returns the scale
        auto load_state = [&](const double2* __restrict__ p, bool use, double n2, int top) {
            const int sigma = use ? top - ((above(n2) + 1) >> 1) : 0;   // n2 < 2^a: norm < 2^ceil(a/2)
            if (on)
                for (int r = 0; r < m; ++r) {
                    const int j = s + r;
                    const double2 v = use && j < N ? ld_cg(p + at(j)) : make_double2(0.0, 0.0);
                    put64(own + r * (3 * kLanes) + kLanes, double_to_fix((uint64_t)__double_as_longlong(v.x), sigma),
                          double_to_fix((uint64_t)__double_as_longlong(v.y), sigma));
                }
            return sigma;
        };
        auto in_range = [](double n2) { return n2 > 1e-60 && n2 < 1e60; };

        // forward pass writing the checkpoints, unless a checkpointed propagation has
        if (!have_ckpt && !bad) {
            for (int64_t c = 0; c < n_int && !bad; ++c) {
                const double2* src = c == 0 ? psi0_all + G.psi_off : ck + c * state;
                const double n2 = norm2(src, real);
                if (__any_sync(0xffffffffu, real && !in_range(n2))) bad = true;   // the same on every warp
                if (bad) break;
                const int sigma = load_state(src, real, n2, F.top);
                if (c == 0 && on)
                    for (int j = s_own; j < e_own; ++j) ck[at(j)] = ld_cg(src + at(j));
                const int64_t nb = min(nt_max, (c + 1) * kc);
                for (int64_t n = c * kc; n < nb; ++n) {
                    double u, v;
                    forward(n, nullptr, n + 1 == nb && nb < nt_max ? ck + (c + 1) * state : nullptr, sigma, u, v);
                }
                __syncthreads();
            }
        }
        bool first = true;   // lambda is zero until the first interval has been swept
        for (int64_t c = n_int - 1; c >= 0 && !bad; --c) {
            const int64_t na = c * kc, nb = min(nt_max, na + kc);
            const double2* __restrict__ cks = ck + c * state;
            const bool use = real && nt > na;   // instances with a step in this interval
            const double n2 = norm2(cks, use);
            if (__any_sync(0xffffffffu, use && !in_range(n2))) {
                bad = true;
                break;
            }
            // ---- recompute the interval onto the tape
            const int sp = load_state(cks, use, n2, F.top);
            {   // sums of sample na
                double x2 = 0.0;
                if (use)
                    for (int j = s_own; j < e_own; ++j) {
                        const double2 v = ld_cg(cks + at(j));
                        const double x = (j - 0.5 * (N - 1)) * dx;
                        x2 = fma(x * x, fma(v.x, v.x, v.y * v.y), x2);
                    }
                const ObsSums t = reduce_obs(fix_lane_sum(ObsSums{0.0, x2, 0.0}, I), red, P);
                if (w == 0 && q == 0) sums[i] = make_double2(n2, t.x);
                __syncthreads();
            }
            for (int64_t n = na; n < nb; ++n) {
                double a, b;
                forward(n, tape + (n - na) * (int64_t)n_max * kLanes, nullptr, sp, a, b);
                if (w == 0 && q == 0) sums[(n + 1 - na) * kLanes + i] = make_double2(a, b);
            }
            __syncthreads();
            // ---- kappa of the interval before: its norm, and bounds of ||g^n|| in place of the second sums
            const double k2 = first ? 0.0 : norm2(lam, use);
            for (int64_t n = na + w; n <= nb; n += P)
                if (q == 0 && use && n <= nt) {
                    double2* u = sums + (n - na) * kLanes + i;
                    u->y = 2.002 * dx * (fabs(gd[row + n]) * sqrt(u->y) + fabs(ga[row + n]) * (dv_max + fabs(E[row + n])) * sqrt(u->x));
                }
            __syncthreads();
            if (w == 0) {
                double B = 0.0;   // bounds every kappa of the interval
                const double k0 = use ? sqrt(k2) * 1.001 : 0.0;
                if (use) {
                    B = k0;
                    for (int64_t n = na; n <= min(nb, nt); ++n) B += sums[(n - na) * kLanes + i].y;
                }
                if (lane < I) {
                    s_bound[i] = B;
                    s_norm[i] = k0;
                }
            }
            __syncthreads();
            const double B = use ? s_bound[i] : 0.0;
            const bool any = B > 1e-30;   // else every gradient of the instance in the interval is zero
            if (__any_sync(0xffffffffu, use && (!(B < 1e30) || (B > 0.0 && !any)))) {
                bad = true;
                break;
            }
            const int sk_max = any ? F.top - above(B) + 40 : 0;
            auto scale_for = [&](double bound) { return bound > 0.0 ? min(sk_max, F.top - above(bound)) : sk_max; };
            int sk = any ? scale_for(s_norm[i]) : 0;
            if (on)
                for (int r = 0; r < m; ++r) {
                    const int j = s + r;
                    const double2 v = use && any && !first && j < N ? ld_cg(lam + at(j)) : make_double2(0.0, 0.0);
                    put64(own + r * (3 * kLanes) + kLanes, double_to_fix((uint64_t)__double_as_longlong(v.x), sk),
                          double_to_fix((uint64_t)__double_as_longlong(v.y), sk));
                }
            // weights of a sample as integers: w_j = (2j - N + 1) cx + dV_j cv + ce, at 2^(61 - e)
            auto weights = [&](int64_t n, bool on_lane) {
                FixWeights W{};
                if (!on_lane) return W;
                const double cx = 2.0 * dx * gd[row + n], cv = 2.0 * dx * ga[row + n], ce = cv * E[row + n];
                const double top = fabs(cx) * x_max + fabs(cv) * dv_max + fabs(ce);
                if (!(top > 1e-60)) return W;   // zero (or far below the bound's scale)
                const int e = above(top);
                W.cx = digits(__double2ll_rn(cx * (0.5 * dx) * pow2(61 + xb - e)));
                W.cv = digits(__double2ll_rn(cv * pow2(61 + F.kv - e)));
                W.ce = __double2ll_rn(ce * pow2(61 - e));
                W.e = e;
                return W;
            };
            auto product_shift = [&](const FixWeights& W) { return shift_of(max(33, min(127, 61 - W.e + sp - sk))); };
            auto weight = [&](const FixWeights& W, int j, const int4& ob) {
                const int wj = 2 * j - N + 1;
                const int64_t x = (int64_t)((uint64_t)mad(wj, W.cx.h, 0) << (32 - xb)) + (mad(wj, W.cx.l, (int64_t(1) << xb) >> 1) >> xb);
                return digits(x + mul_fix<3>(Digits{ob.y, ob.x}, W.cv) + W.ce);
            };
            // every sample's shift in range?  (before anything of the interval is added to gE)
            for (int64_t n = na + w; n <= nb; n += P)
                if (use && any && n <= nt) {
                    const FixWeights W = weights(n, true);
                    const double g = sums[(n - na) * kLanes + i].y;   // sk <= top - above(g)
                    if (g > 0.0 && 61 - W.e + sp - F.top + above(g) <= 32) s_bad = 1;
                }
            __syncthreads();
            if (s_bad) {
                bad = true;
                break;
            }
            auto rescale = [&](int by) {   // the right-hand side by 2^by, rounded
                if (on)
                    for (int r = 0; r < m; ++r) {
                        int4* p = own + r * (3 * kLanes) + kLanes;
                        const int4 v = *p;
                        int64_t a = lo64(v), b = hi64(v);
                        if (by >= 0) {
                            a = (int64_t)((uint64_t)a << by);
                            b = (int64_t)((uint64_t)b << by);
                        } else {
                            const int k = min(-by, 63);
                            a = (a + (int64_t(1) << (k - 1))) >> k;
                            b = (b + (int64_t(1) << (k - 1))) >> k;
                        }
                        put64(p, a, b);
                    }
            };
            // ---- backward
            for (int64_t n = nb - 1; n >= na; --n) {
                const bool active = use && n < nt, term = use && n + 1 == nt;
                const int4* __restrict__ t1 = tape + (n - na) * (int64_t)n_max * kLanes;                      // psi~^{n+1}
                const int4* __restrict__ t0 = n > na ? tape + (n - na - 1) * (int64_t)n_max * kLanes : nullptr;   // psi~^n
                // scale of this step: ||M kappa^{n+1}|| (or ||g^{n+1}||) + ||g^n|| bounds kappa^n and all between
                int by = 0;
                if (any) {
                    double bound = s_norm[i];
                    if (term) bound += sums[(n + 1 - na) * kLanes + i].y;
                    if (active) bound += sums[(n - na) * kLanes + i].y;
                    by = min(scale_for(bound) - sk, 40);
                }
                if (__any_sync(0xffffffffu, by != 0)) rescale(by);
                sk += by;
                // this step's weights, by one warp for all (short_solve's barriers lie between)
                if (w == (int)((n - na) % P)) {
                    const FixWeights W = weights(n, active && any);
                    if (q == 0) s_w[i] = W;
                }
                if (__any_sync(0xffffffffu, term)) {   // lambda^{Nt} = g^{Nt}
                    const FixWeights W = weights(n + 1, term && any);
                    const Shift S = product_shift(W);
                    if (on && term && any)
                        for (int r = 0; r < m; ++r) {
                            const int j = s + r;
                            if (j >= N) break;
                            const int4 v = __ldcg(t1 + at(j)), ob = __ldg(tO + j);
                            const Digits wt = weight(W, j, ob), mm{ob.w, ob.z};
                            int64_t pr = lo64(v), pi = hi64(v);
                            const bool masked = j < jm_lo || j > jm_hi;
                            if (masked) {
                                pr = mul_fix<3>(mm, digits(pr));
                                pi = mul_fix<3>(mm, digits(pi));
                            }
                            int64_t kr = mul_shift(wt, digits(pr), S), ki = -mul_shift(wt, digits(pi), S);
                            if (masked) {
                                kr = mul_fix<3>(mm, digits(kr));
                                ki = mul_fix<3>(mm, digits(ki));
                            }
                            put64(own + r * (3 * kLanes) + kLanes, kr, ki);
                        }
                }
                const Digits Eb = digits(active ? __double2ll_rn(0.5 * (E[row + n] + E[row + n + 1]) * F.e_scale) : 0);
                int64_t yr, yi;
                short_solve(geo, Eb, yr, yi);
                const FixWeights W = s_w[i];
                const Shift S = product_shift(W);
                int64_t sxh = 0, sxm = 0, sxl = 0;
                float sq = 0.0f;
                if (on) {
                    int4* o = own + (int64_t)(m - 1) * (3 * kLanes);
                    auto tape_at = [&](const int4* t, int j) { return j < N ? __ldcg(t + at(j)) : make_int4(0, 0, 0, 0); };
                    auto psi_at = [&](int j) {   // psi~^n, or psi^n at the interval's start
                        if (t0) return tape_at(t0, j);
                        int4 v = make_int4(0, 0, 0, 0);
                        if (use && j < N) {
                            const double2 z = ld_cg(cks + at(j));
                            put64(&v, double_to_fix((uint64_t)__double_as_longlong(z.x), sp),
                                  double_to_fix((uint64_t)__double_as_longlong(z.y), sp));
                        }
                        return v;
                    };
                    int4 gn = o[0], pn = o[kLanes], dn = o[2 * kLanes];
                    int4 an = psi_at(s + m - 1), bn = tape_at(t1, s + m - 1), on4 = __ldg(tO + min(s + m - 1, N - 1));
                    for (int r = m - 1; r >= 0; --r) {
                        const int j = s + r;
                        const int4 g = gn, p = pn, d = dn, a4 = an, b4 = bn, ob = on4;
                        if (r > 0) {
                            gn = o[-3 * kLanes];
                            pn = o[-2 * kLanes];
                            dn = o[-kLanes];
                            an = psi_at(j - 1);
                            bn = tape_at(t1, j - 1);
                            on4 = __ldg(tO + min(j - 1, N - 1));
                        }
                        back_row(g, d, yr, yi);
                        const bool masked = j < jm_lo || j > jm_hi;
                        const Digits mm{ob.w, ob.z};
                        int64_t pr = lo64(a4), pi = hi64(a4);   // psi^n
                        if (masked && t0) {
                            pr = mul_fix<3>(mm, digits(pr));
                            pi = mul_fix<3>(mm, digits(pi));
                        }
                        const Digits wt = weight(W, j, ob), er = digits(yr), ei = digits(yi);
                        int64_t kr = update_fix(ci, cf, er, lo64(p)) + mul_shift(wt, digits(pr), S);
                        int64_t ki = update_fix(ci, cf, ei, hi64(p)) - mul_shift(wt, digits(pi), S);
                        if (masked) {
                            kr = mul_fix<3>(mm, digits(kr));
                            ki = mul_fix<3>(mm, digits(ki));
                        }
                        if (!active || j >= N) kr = ki = 0;
                        put64(o + kLanes, kr, ki);
                        const float fr = (float)(int32_t)((uint64_t)kr >> 32), fi = (float)(int32_t)((uint64_t)ki >> 32);
                        sq = fmaf(fr, fr, fmaf(fi, fi, sq));
                        // x Im(conj(mu) (psi^n + psi~^{n+1})) = x (Yr si + Yi sr) / beta: all four partial products, as the
                        // rows far out, of no weight in psi, count with their x
                        const Digits sr = digits(pr + lo64(b4)), si = digits(pi + hi64(b4));
                        const bool in = j < N;
                        const int64_t mid = mad(er.h, si.l, mad(er.l, si.h, mad(ei.h, sr.l, mad(ei.l, sr.h, 0))));
                        const Digits vh = digits(in ? mad(er.h, si.h, mad(ei.h, sr.h, 0)) : 0);
                        const Digits vm = digits(in ? fold(fold(mid, mad(er.l, si.l, 0)), mad(ei.l, sr.l, 0)) : 0);
                        const int wj = 2 * j - N + 1;
                        sxh = mad(vh.h, wj, sxh);
                        sxm = mad(vh.l, wj, mad(vm.h, wj, sxm));
                        sxl = mad(vm.l, wj, sxl);
                        o -= 3 * kLanes;
                    }
                }
                ObsSums o{fma((double)sxh, 4294967296.0, fma((double)sxl, 1.0 / 4294967296.0, (double)sxm)), (double)sq, 0.0};
                const ObsSums t = reduce_obs(fix_lane_sum(o, I), red, P);
                if (w == 0 && q == 0)   // ||M kappa^n||: each component's high word is off by less than 1
                    s_norm[i] = active ? (double)(sqrtf((float)t.x) * 1.001f + 256.0f) * pow2(32 - sk) : 0.0;
                __syncthreads();
                if (w == 0 && q == 0 && active) {
                    // h / beta = 2 dx^2; the sum is at 2^(sk + sp - 64), x in half grid steps
                    const double gbar = any ? 2.0 * dx * dx * (0.5 * dx) * t.n * pow2(64 - sk - sp) : 0.0;
                    if (term) gE[row + nt] += ga[row + nt] * dx * sums[(nt - na) * kLanes + i].x;
                    gE[row + n] += 0.5 * gbar + ga[row + n] * dx * sums[(n - na) * kLanes + i].x;
                    gE[row + n + 1] += 0.5 * gbar;
                }
            }
            // rhs of the next interval, in double
            if (on)
                for (int r = 0; r < m; ++r) {
                    const int j = s + r;
                    if (j >= N) break;
                    const int4 p = own[r * (3 * kLanes) + kLanes];
                    lam[at(j)] = use && any ? make_double2(__longlong_as_double((long long)fix_to_double(lo64(p), sk)),
                                                           __longlong_as_double((long long)fix_to_double(hi64(p), sk)))
                                            : make_double2(0.0, 0.0);
                }
            first = false;
            __syncthreads();
        }
        // an instance without steps: only the direct term of a_0
        if (!bad) {
            const double2* p0 = have_ckpt ? ck : psi0_all + G.psi_off;
            const double t = norm2(p0, nt == 0);
            if (w == 0 && q == 0 && nt == 0) gE[row] = ga[row] * dx * t;
            __syncthreads();
        }

        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) {
            left[gi] = bad ? 0 : 1;   // progress of the FP64 kernel behind: 1 = nothing to do
            __threadfence();
            *(volatile int*)(progress + gi) = 1;
            __threadfence();
            atomicExch(busy + gi, 0);
        }
    }
}

cudaError_t launch_adjoint_fix(const GroupDesc* d_groups, int64_t n_groups, int P, int ctas, const ClassDesc* d_cls,
                               const double* d_tab, const int64_t* d_slot_row, const int64_t* d_slot_nt, const void* d_psi0,
                               void* d_lam, void* d_ckpt, const int64_t* d_ckpt_off, void* d_work, void* d_tape, void* d_scratch,
                               int64_t scratch_per_cta, int n_max, int kc, const double* E, const double* gd, const double* ga,
                               double* gE, int mask_on, int* d_busy, int* d_progress, int* d_left, cudaStream_t st, int have_ckpt)
{
    if (n_groups == 0 || ctas == 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(d_busy, 0, sizeof(int) * n_groups, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(d_progress, 0, sizeof(int) * n_groups, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(d_left, 0, sizeof(int) * n_groups, st);
    if (e != cudaSuccess) return e;
    const size_t smem = (size_t)P * kLanes * (3 * sizeof(double) + kEdgeBytes);
    k_adjoint_fix<<<(unsigned)ctas, P * kLanes, smem, st>>>(
        d_groups, n_groups, d_cls, d_tab, d_slot_row, d_slot_nt, static_cast<const double2*>(d_psi0),
        static_cast<double2*>(d_lam), static_cast<double2*>(d_ckpt), d_ckpt_off, static_cast<double2*>(d_work),
        static_cast<double2*>(d_tape), static_cast<int4*>(d_scratch), scratch_per_cta, n_max, kc, E, gd, ga, gE, mask_on, d_busy,
        d_progress, d_left, have_ckpt);
    return cudaGetLastError();
}

}  // namespace tdse
