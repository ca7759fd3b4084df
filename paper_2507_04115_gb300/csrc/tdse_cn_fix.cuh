// FULL_CN sweep in 64-bit fixed point (FP64 batches): one scheduling slice of a group.
//
// The same segmented Thomas sweeps as tdse_full_cn.cu (halo K, lane geometry of GroupDesc), with the
// arithmetic of tdse_fix.cuh on the integer pipe, and two consecutive steps fused into one pass:
//   * step n is eliminated in one direction (first slice step: ascending j) and back-substituted in the
//     other; the pass that back-substitutes it, travelling in direction dir, has psi^{n+1}_j in hand and
//     eliminates step n+1 in the same direction at once.  Directions alternate from pass to pass.
//   * only (gamma_j, u_j), u = psi + i D_prev, is stored: D_j = -i gamma_j u_j is formed again when it is
//     read, and psi_j = u_j - i D_{j+dir} is exact in integers.  A pass therefore reads 32 bytes per
//     point and writes 32 (the two-sweep form with psi, gamma and D moves 112), in place.
//   * own rows m .. : row r of segment sigma sits at [column / 32][r][gamma | u][column % 32] of the
//     CTA's scratch, column = sigma I + i, so that a lead-in row is a coalesced read of a neighbour's
//     rows whatever the group's width.
// A pass: (a) 2K lead-in rows before the segment in travel order -- K rows of back substitution alone,
// then K rows that also restart the elimination --, a barrier, (b) the m own rows, in place.  All reads
// of other segments' rows happen in (a), so (b) may overwrite.  The state is read from and written to
// the double2 wavefunctions once per slice (and at an instance's last step).
//
// What bounds it: the integer pipes and the latency of their in-order chains -- about 350 instructions a
// row (pivot 65, D twice 60, Y 30, update 30, observables 40, the rest addressing, 64-bit adds and moves),
// the multiply-add pipe 69 % busy with 16 warps an SM; HBM traffic (72 B per point and step) needs half
// the time.  Measured, 8192 x 4096 points, 160 steps: 274 ms with the FP64 sweep (27 FP64 instructions a row,
// 64 cycles each), 99.8 ms with this one; one atom, 512 steps: 54.4 ms and 18.6 ms.  The observable sums on
// the otherwise idle FP64 pipe (5 instructions a row) made it slower, 104 ms: a warp waits out each one.
// More registers a thread (168, 220) made it slower too, 111 and 133 ms at the warps that then fit.
#pragma once

#include <type_traits>

#include "tdse_sched.cuh"

namespace tdse {

struct FixSlot {
    Digits gr, gi, ur, ui;
};

__device__ __forceinline__ FixSlot load_slot(const int4* __restrict__ p)
{
    const int4 g = __ldcg(p), u = __ldcg(p + kLanes);
    return FixSlot{Digits{g.x, g.y}, Digits{g.z, g.w}, Digits{u.x, u.y}, Digits{u.z, u.w}};
}

// Is the group's shape one that fix_slice takes?  (m >= 4: a pass reads its own rows three ahead.)
__device__ __forceinline__ bool fix_shape(const GroupDesc& G, const ClassDesc& C) { return C.fix.ok && G.m >= 4; }

__device__ __forceinline__ ObsSums fix_lane_sum(ObsSums o, int I)
{
    for (int off = I; off < kLanes; off <<= 1) {
        o.n += __shfl_xor_sync(0xffffffffu, o.n, off);
        o.x += __shfl_xor_sync(0xffffffffu, o.x, off);
        o.v += __shfl_xor_sync(0xffffffffu, o.v, off);
    }
    return o;
}

// Range of the slice's fields, norm and scale of the state: false when an instance is outside the
// fixed-point range (the same answer on every warp).
__device__ __forceinline__ bool fix_range(const GroupDesc& G, const FixClass& F, const double2* __restrict__ ps,
                                          const double* __restrict__ E, int64_t row, int64_t nt, int64_t n0, int64_t n1,
                                          int64_t sample_base, int s_own, int e_own, double* red, int& sigma)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, P = blockDim.x >> 5;
    const int I = G.I, i = lane & (I - 1);
    const bool live = nt > n0;
    bool ok = true;
    if (live)
        for (int64_t n = n0; n <= min(n1, nt); ++n) ok = ok && fabs(E[row + n - sample_base]) <= F.E_lim;
    float sq = 0.0f;
    if (live)
        for (int j = s_own; j < e_own; ++j) {
            const double2 p = ld_cg(ps + (int64_t)j * I + i);
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
    // ||psi||^2 = f 2^e, f in [1, 2): 2^sigma puts the norm in [2^(top-1), 2^top)
    const int e2 = live ? (int)((__float_as_uint(tot) >> 23) & 0xffu) - 127 : 0;
    sigma = F.top - ((e2 + 2) >> 1);
    return __all_sync(0xffffffffu, ok);
}

// Observables (and checkpoint 0) of the initial state.
template <bool kCkpt>
__device__ __forceinline__ void fix_initial(const GroupDesc& G, const ClassDesc& C, const double* __restrict__ tab,
                                            const double2* __restrict__ ps, int64_t nt, int64_t row, int s_own, int e_own,
                                            const double* __restrict__ E, double* __restrict__ d_out,
                                            double* __restrict__ a_out, int64_t sample_base, double* red, double2* __restrict__ ck)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, P = blockDim.x >> 5;
    const int I = G.I, i = lane & (I - 1);
    const double dx = C.dx;
    const double2* __restrict__ tab_xv2 = reinterpret_cast<const double2*>(tab + tab_xv(C));
    ObsSums o{0.0, 0.0, 0.0};
    for (int j = s_own; j < e_own; ++j) {
        const double2 p = ld_cg(ps + (int64_t)j * I + i);
        if constexpr (kCkpt) ck[(int64_t)j * I + i] = p;
        const double rho = fma(p.x, p.x, p.y * p.y);
        const double2 xv = __ldg(tab_xv2 + j);
        o.n += rho;
        o.x = fma(xv.x, rho, o.x);
        o.v = fma(xv.y, rho, o.v);
    }
    const ObsSums t = reduce_obs(fix_lane_sum(o, I), red, P);
    if (w == 0 && lane < I && nt >= 0) {
        const double E0 = E[row - sample_base];
        d_out[row - sample_base] = t.x * dx;
        a_out[row - sample_base] = fma(E0, t.n, t.v) * dx;
    }
    __syncthreads();
}

// rho = |psi|^2 2^-60 in integers and its sums: over the points, times x in half grid steps (wj = 2 j - N + 1),
// times dV (ob.x, ob.y: its digits); the last two as high and low parts.
__device__ __forceinline__ void fix_observe(int64_t xr, int64_t xi, int wj, const int4& ob, int64_t& sn, int64_t& sxh,
                                            int64_t& sxl, int64_t& svh, int64_t& svm)
{
    const Digits a = digits(xr), b = digits(xi);
    const uint64_t ll = (uint64_t)mad(a.l, a.l, mad(b.l, b.l, 0)) >> 33;
    const int64_t rho = combine<4, 27>(mad(a.h, a.h, mad(b.h, b.h, 0)),
                                       mad(a.h, a.l, mad(b.h, b.l, (int64_t)ll + (int64_t(1) << 26))));
    const Digits rd = digits(rho);
    sn += rho;
    sxh = mad(rd.h, wj, sxh);
    sxl = mad(rd.l, wj, sxl);
    svh = mad(rd.h, ob.y, svh) + (mad(rd.l, ob.y, int64_t(1) << 31) >> 32);
    svm = mad(rd.h, ob.x, svm);
}

// Returns false, having changed nothing, when an instance's field or norm is outside the fixed-point
// range of this slice (or not finite): the caller then takes the FP64 sweep.
template <bool kCkpt>
__device__ __forceinline__ bool fix_slice(const GroupDesc& G, const ClassDesc& C, const double* __restrict__ tab,
                                          double2* __restrict__ ps, int64_t nt, int64_t row, int64_t slot, int64_t n0,
                                          int64_t n1, bool initial, const double* __restrict__ E,
                                          double* __restrict__ d_out, double* __restrict__ a_out, int64_t sample_base,
                                          int4* __restrict__ buf, double* red, int* status, double2* __restrict__ ck,
                                          int kc, int jm_lo, int jm_hi)
{
    const FixClass& F = C.fix;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, P = blockDim.x >> 5;
    const int I = G.I, i = lane & (I - 1), q = lane / I;
    const int N = G.N, K = G.K, m = G.m;
    const bool on = w < G.P;   // warps beyond the group's segments only meet the barriers
    const int s = (w * (kLanes / I) + q) * m;
    const int s_own = on ? min(N, s) : N, e_own = on ? min(N, s + m) : N;
    const bool live = nt > n0;
    const double dx = C.dx;
    const int4* __restrict__ tT = reinterpret_cast<const int4*>(tab + tab_fxp(C));
    const int4* __restrict__ tO = reinterpret_cast<const int4*>(tab + tab_fob(C));

    auto field = [&](int64_t n) { return n <= nt ? E[row + n - sample_base] : 0.0; };   // live lanes, n >= n0
    int sigma;
    if (!fix_range(G, F, ps, E, row, nt, n0, n1, sample_base, s_own, e_own, red, sigma)) return false;
    if (initial) fix_initial<kCkpt>(G, C, tab, ps, nt, row, s_own, e_own, E, d_out, a_out, sample_base, red, ck);

    // scales of the observable sums: rho_int = |psi|^2 2^(2 sigma - 60)
    const double unit = __hiloint2double((1023 + 60 - 2 * sigma) << 20, 0);   // |sigma| <= 112
    const int64_t inv_b = F.inv_b;
    const int32_t ci = F.ci;
    const Digits cf = F.cf;
    int4* __restrict__ own = buf + ((int64_t)w * m * 2) * kLanes + lane;   // row r at own + r * 64
    auto fix_field = [&](int64_t n) {   // field of the elimination of step n
        return digits(live && n < nt ? __double2ll_rn(0.5 * (field(n) + field(n + 1)) * F.e_scale) : 0);
    };

    // state of the elimination: gamma (2^58) and D of the previous row
    int64_t gr = 0, gi = 0, dr = 0, di = 0;
    // one row of the elimination: psi -> slot (gamma at 2^64, u) and D
    auto eliminate = [&](const int4& t, const Digits& Eb, bool in, int64_t pr, int64_t pi) {
        gamma_row(inv_b, diag_row(FixPoint{t.x, t.y, t.z, t.w}, Eb), gr, gi);
        gr = in ? gr : 0;   // rows outside the grid: the exact wall
        gi = in ? gi : 0;
        const FixSlot v{digits(gr << 6), digits(gi << 6), digits(pr - di), digits(pi + dr)};
        mul_minus_i(v.gr, v.gi, v.ur, v.ui, dr, di);
        return v;
    };
    auto store_slot = [&](int4* p, const FixSlot& v) {
        __stcg(p, make_int4(v.gr.h, v.gr.l, v.gi.h, v.gi.l));
        __stcg(p + kLanes, make_int4(v.ur.h, v.ur.l, v.ui.h, v.ui.l));
    };

    // ---- prologue: elimination of step n0, ascending
    if (on) {
        const Digits Eb = fix_field(n0);
        auto load_psi = [&](int j) {
            return live && (unsigned)j < (unsigned)N ? ld_cg(ps + (int64_t)j * I + i) : make_double2(0.0, 0.0);
        };
        double2 pa = load_psi(s - K), pb = load_psi(s - K + 1);
        for (int r = -K; r < m; ++r) {
            const int j = s + r;
            const double2 p = pa;
            pa = pb;
            pb = r + 2 < m ? load_psi(j + 2) : make_double2(0.0, 0.0);
            const bool in = (unsigned)j < (unsigned)N;
            const int64_t pr = double_to_fix((uint64_t)__double_as_longlong(p.x), sigma);
            const int64_t pi = double_to_fix((uint64_t)__double_as_longlong(p.y), sigma);
            const FixSlot v = eliminate(__ldg(tT + min(max(j, 0), N - 1)), Eb, in, pr, pi);
            if (r >= 0 && in) store_slot(own + (int64_t)r * (2 * kLanes), v);
        }
    }
    __syncthreads();

    // ---- passes: back substitution of step n, elimination of step n + 1
    for (int64_t n = n0; n < n1; ++n) {
        const int dir = ((n - n0) & 1) ? 1 : -1;
        const bool last = n + 1 == n1;
        const bool active = n < nt;
        const double En1 = active ? field(n + 1) : 0.0;
        ObsSums o{0.0, 0.0, 0.0};
        // states leave as doubles at the slice's end, at an instance's last step, at checkpoints
        const bool put = active && (last || n + 1 == nt);
        bool put_ck = false;
        if constexpr (kCkpt) put_ck = (n + 1) % kc == 0 && n + 1 < G.nt_max;
        const bool any_put = __any_sync(0xffffffffu, put) || put_ck;
        int64_t Yr = 0, Yi = 0, Dr = 0, Di = 0, Er = 0, Ei = 0;   // D at the current row, at the row past the segment
        FixSlot cur{}, x1{}, x2{};
        const Digits Eb = last ? Digits{0, 0} : fix_field(n + 1);
        const int j0 = dir < 0 ? s + m - 1 : s;   // grid point of row r: j0 + dir r
        auto row_back = [&](const FixSlot& nx, int64_t& nDr, int64_t& nDi) {   // Y of the current row, D of the next
            mul_minus_i(nx.gr, nx.gi, nx.ur, nx.ui, nDr, nDi);
            const Digits yr = digits(Yr), yi = digits(Yi);
            Yr = mul2_fix(cur.gr, yr, negative(cur.gi), yi, Dr);
            Yi = mul2_fix(cur.gr, yi, cur.gi, yr, Di);
        };
        auto row_psi = [&](int j, int64_t nDr, int64_t nDi, int64_t& xr, int64_t& xi) {
            xr = update_fix(ci, cf, digits(Yr), undigits(cur.ur) + nDi);
            xi = update_fix(ci, cf, digits(Yi), undigits(cur.ui) - nDr);
            if (j < jm_lo || j > jm_hi) {
                const int4 ob = __ldg(tO + min(max(j, 0), N - 1));
                const Digits mm{ob.w, ob.z};
                xr = mul_fix<3>(mm, digits(xr));
                xi = mul_fix<3>(mm, digits(xi));
            }
        };
        gr = gi = dr = di = 0;
        if (on) {
            // (a) lead-in rows r = -2K .. -1 (only the back substitution's K before the last elimination)
            int r = last ? -K : -2 * K;
            // position of the slot to load next: row lr of the segment dq segments on
            int off = dir < 0 ? m - 1 - r : r;
            int dq = off >= 0 ? off / m : -((m - 1 - off) / m);
            int lr = off - dq * m;
            int lj = j0 + dir * r;
            auto load_next = [&]() {
                FixSlot v{};
                if ((unsigned)lj < (unsigned)N) {
                    const int col = w * kLanes + lane + dq * I;
                    v = load_slot(buf + ((int64_t)(col >> 5) * m + lr) * (2 * kLanes) + (col & 31));
                }
                lj += dir;
                lr += dir;
                if (lr == m) { lr = 0; ++dq; }
                if (lr < 0) { lr = m - 1; --dq; }
                return v;
            };
            cur = load_next();
            mul_minus_i(cur.gr, cur.gi, cur.ur, cur.ui, Dr, Di);
            x1 = load_next();
            x2 = load_next();
            int4 tn = __ldg(tT + min(max(j0 - dir * K, 0), N - 1));   // table rows one ahead, from row -K
            for (; r < 0; ++r) {
                const FixSlot nx = x1;
                x1 = x2;
                x2 = load_next();
                int64_t nDr, nDi;
                row_back(nx, nDr, nDi);
                if (r >= -K && !last) {
                    const int j = j0 + dir * r;
                    const int4 t = tn;
                    tn = __ldg(tT + min(max(j + dir, 0), N - 1));
                    int64_t xr, xi;
                    row_psi(j, nDr, nDi, xr, xi);
                    eliminate(t, Eb, (unsigned)j < (unsigned)N, xr, xi);
                }
                cur = nx;
                Dr = nDr;
                Di = nDi;
            }
            // the row past the segment's end in travel order: its owner overwrites it in (b)
            const int je = j0 + dir * m;
            if ((unsigned)je < (unsigned)N) {
                const int col = w * kLanes + lane + dir * I;
                const FixSlot v = load_slot(buf + ((int64_t)(col >> 5) * m + (dir < 0 ? m - 1 : 0)) * (2 * kLanes) + (col & 31));
                mul_minus_i(v.gr, v.gi, v.ur, v.ui, Er, Ei);
            }
        }
        __syncthreads();
        if (on) {
            // (b) own rows
            int64_t sn = 0, sxh = 0, sxl = 0, svh = 0, svm = 0;
            int4* __restrict__ pw = own + (int64_t)(dir < 0 ? m - 1 : 0) * (2 * kLanes);
            const int step = dir * 2 * kLanes;
            const int4* __restrict__ pl = pw + 3 * step;
            int j = j0;
            int jc = min(max(j, 0), N - 1);
            int4 tn = __ldg(tT + jc), on4 = __ldg(tO + jc);
            for (int r = 0; r < m; ++r) {
                const FixSlot nx = x1;
                x1 = x2;
                x2 = FixSlot{};
                if (r + 3 < m && (unsigned)(j + 3 * dir) < (unsigned)N) x2 = load_slot(pl);
                pl += step;
                const int4 t = tn, ob = on4;
                jc = min(max(j + dir, 0), N - 1);
                tn = __ldg(tT + jc);
                on4 = __ldg(tO + jc);
                int64_t nDr, nDi, xr, xi;
                row_back(nx, nDr, nDi);
                if (r + 1 == m) {
                    nDr = Er;
                    nDi = Ei;
                }
                row_psi(j, nDr, nDi, xr, xi);
                const bool in = (unsigned)j < (unsigned)N;
                if (!in) xr = xi = 0;
                fix_observe(xr, xi, 2 * j - N + 1, ob, sn, sxh, sxl, svh, svm);
                if (any_put && in) {
                    const double2 v = make_double2(__longlong_as_double((long long)fix_to_double(xr, sigma)),
                                                   __longlong_as_double((long long)fix_to_double(xi, sigma)));
                    if (put) ps[(int64_t)j * I + i] = v;
                    if constexpr (kCkpt)
                        if (put_ck) ck[((n + 1) / kc) * ((int64_t)N * I) + (int64_t)j * I + i] = v;
                }
                if (!last) {
                    const FixSlot v = eliminate(t, Eb, in, xr, xi);
                    if (in) store_slot(pw, v);
                }
                pw += step;
                j += dir;
                cur = nx;
                Dr = nDr;
                Di = nDi;
            }
            const double two32 = 4294967296.0;
            o.n = (double)sn * unit;
            o.x = fma((double)sxh, two32, (double)sxl) * (0.5 * dx * unit);
            o.v = fma((double)svh, two32, (double)svm) * (two32 * F.v_scale * unit);
        }
        const ObsSums t = reduce_obs(fix_lane_sum(o, I), red, P);   // its barrier orders this pass's writes
        if (w == 0 && q == 0 && active) {
            const int64_t kk = row + n + 1 - sample_base;
            d_out[kk] = t.x * dx;
            a_out[kk] = fma(En1, t.n, t.v) * dx;
            if (!(t.n * dx <= 1.0 + 1e-6)) status[slot] = 1;
        }
    }
    return true;
}

// The same step for short segments (lane-split groups, m <= 4 K), where fix_slice's lead-in of 2K rows
// would cost several times the m own rows.  D and Y are affine in the value that enters a segment,
//     D_r = D^0_r + H_r D_in,  Y_r = Y^0_r + (prod_{k>=r} gamma_k) Y_in,  H_r = prod_{k<=r} gamma_k,
// so each segment runs from zero, publishes its outgoing D^0, Y^0 and its product H in shared memory, and
// composes what enters from the T = ceil(K / m) segments before (after) it; farther ones are below beta^K.
// Only gamma, whose recurrence is not linear, has a lead-in, and as its error falls by gamma^2 a row, K/2
// rows of it.  Then the first min(m, K) rows of D are run again from D_in, and all of Y from Y_in.
// psi (integers, converted once per slice), gamma and D of the own rows stay in the CTA's scratch, 1.5 KB a
// row and warp, which small batches find in L1.
// Measured, one atom (N = 2000, K = 36, 512 steps): 18.6 ms with fix_slice (4 warps), 8.3 here (6 warps); the uneven
// scan 19.5 ms and 15.0.
struct FixEdge {   // per column of the CTA
    int64_t dr, di;
    Digits hr, hi;
    int64_t yr, yi;
};

static_assert(sizeof(FixEdge) == kEdgeBytes, "shared memory of the launch");

__device__ __forceinline__ bool fix_short(const GroupDesc& G) { return G.I != kLanes && G.K > 0 && G.m <= 4 * G.K; }

// Geometry of a lane's segment in the short-segment form, and the own rows' scratch: row r holds gamma (digits),
// the right-hand side and D (64-bit pairs) at own + r * 96 + (0, 32, 64).
struct ShortGeom {
    int N, K, m, I, s, sg, n_seg, col;
    bool on;
    int4* own;
    FixEdge* edge;
    const int4* tT;
    int64_t inv_b;
};
__device__ __forceinline__ void put64(int4* p, int64_t a, int64_t b)
{
    *p = make_int4((int)(uint32_t)(uint64_t)a, (int)(uint32_t)((uint64_t)a >> 32), (int)(uint32_t)(uint64_t)b,
                   (int)(uint32_t)((uint64_t)b >> 32));
}
__device__ __forceinline__ int64_t lo64(const int4& v) { return (int64_t)(((uint64_t)(uint32_t)v.y << 32) | (uint32_t)v.x); }
__device__ __forceinline__ int64_t hi64(const int4& v) { return (int64_t)(((uint64_t)(uint32_t)v.w << 32) | (uint32_t)v.z); }
__device__ __forceinline__ void gam(const int4& v, Digits& r, Digits& i)
{
    r = Digits{v.x, v.y};
    i = Digits{v.z, v.w};
}
// (yr, yi) <- D + gamma Y at a row
__device__ __forceinline__ void back_row(const int4& g, const int4& d, int64_t& yr, int64_t& yi)
{
    Digits a, b;
    gam(g, a, b);
    const Digits u = digits(yr), v = digits(yi);
    yr = mul2_fix(a, u, negative(b), v, lo64(d));
    yi = mul2_fix(a, v, b, u, hi64(d));
}

// The elimination of A y = rhs over the whole group, leaving gamma and D of every own row in the scratch and
// the Y that enters this segment from the next ones in (yr, yi).  Two barriers inside; the caller's own
// rows may be overwritten right after, the edges only after another barrier.
__device__ __forceinline__ void short_solve(const ShortGeom& G, Digits Eb, int64_t& y_in_r, int64_t& y_in_i)
{
    const int N = G.N, K = G.K, m = G.m, I = G.I, s = G.s, sg = G.sg, n_seg = G.n_seg, col = G.col;
    const int Kg = (K + 1) / 2, Kr = min(m, K), T = (K + m - 1) / m;
    const bool on = G.on;
    int4* const own = G.own;
    FixEdge* const edge = G.edge;
    const int64_t inv_b = G.inv_b;
    auto table = [&](int j) { return __ldg(G.tT + min(max(j, 0), N - 1)); };
    // gamma (lead-in and own rows) and D from zero, ascending
    if (on) {
        int64_t gr = 0, gi = 0, dr = 0, di = 0;
        int4 tn = table(s - Kg);
        for (int r = -Kg; r < 0; ++r) {
            const int4 t = tn;
            tn = table(s + r + 1);
            gamma_row(inv_b, diag_row(FixPoint{t.x, t.y, t.z, t.w}, Eb), gr, gi);
            if (s + r < 0) gr = gi = 0;   // (a segment's lead-in never lies beyond the far wall unless it does itself)
        }
        Digits hr{0, 0}, hi{0, 0};
        int4 pn = own[kLanes];
        int4* o = own;
        for (int r = 0; r < m; ++r) {
            const int4 t = tn, p = pn;
            tn = table(s + r + 1);
            if (r + 1 < m) pn = o[4 * kLanes];
            gamma_row(inv_b, diag_row(FixPoint{t.x, t.y, t.z, t.w}, Eb), gr, gi);
            if (s + r >= N) gr = gi = 0;
            const Digits a = digits(gr << 6), b = digits(gi << 6);
            mul_minus_i(a, b, digits(lo64(p) - di), digits(hi64(p) + dr), dr, di);
            o[0] = make_int4(a.h, a.l, b.h, b.l);
            if (r >= Kr) put64(o + 2 * kLanes, dr, di);
            if (T > 1) {   // H: product of the segment's gamma
                if (r == 0) {
                    hr = a;
                    hi = b;
                } else {
                    const int64_t x = mul2_fix(a, hr, negative(b), hi), y = mul2_fix(a, hi, b, hr);
                    hr = digits(x);
                    hi = digits(y);
                }
            }
            o += 3 * kLanes;
        }
        edge[col].dr = dr;
        edge[col].di = di;
        edge[col].hr = hr;
        edge[col].hi = hi;
    }
    __syncthreads();
    // D entering the segment, D of its first Kr rows again, Y of those rows from zero
    if (on) {
        int64_t dr = 0, di = 0;
        for (int k = min(T, sg); k >= 1; --k) {
            const FixEdge& e = edge[col - k * I];
            const Digits a = digits(dr), b = digits(di);
            const int64_t x = mul2_fix(e.hr, a, negative(e.hi), b, e.dr), y = mul2_fix(e.hr, b, e.hi, a, e.di);
            dr = x;
            di = y;
        }
        int4* o = own;
        int4 gn = o[0], pn = o[kLanes];
        for (int r = 0; r < Kr; ++r) {
            const int4 g = gn, p = pn;
            if (r + 1 < Kr) {
                gn = o[3 * kLanes];
                pn = o[4 * kLanes];
            }
            Digits a, b;
            gam(g, a, b);
            mul_minus_i(a, b, digits(lo64(p) - di), digits(hi64(p) + dr), dr, di);
            put64(o + 2 * kLanes, dr, di);
            o += 3 * kLanes;
        }
        int64_t yr = 0, yi = 0;
        o -= 3 * kLanes;
        gn = o[0];
        pn = o[2 * kLanes];
        for (int r = Kr - 1; r >= 0; --r) {
            const int4 g = gn, d = pn;
            if (r > 0) {
                gn = o[-3 * kLanes];
                pn = o[-kLanes];
            }
            Digits a, b;
            gam(g, a, b);
            const Digits u = digits(yr), v = digits(yi);
            yr = mul2_fix(a, u, negative(b), v, lo64(d));
            yi = mul2_fix(a, v, b, u, hi64(d));
            o -= 3 * kLanes;
        }
        edge[col].yr = yr;
        edge[col].yi = yi;
    }
    __syncthreads();
    y_in_r = y_in_i = 0;
    if (on) {
        int64_t yr = 0, yi = 0;
        for (int k = min(T, n_seg - 1 - sg); k >= 1; --k) {
            const FixEdge& e = edge[col + k * I];
            const Digits a = digits(yr), b = digits(yi);
            const int64_t x = mul2_fix(e.hr, a, negative(e.hi), b, e.yr), y = mul2_fix(e.hr, b, e.hi, a, e.yi);
            yr = x;
            yi = y;
        }
        y_in_r = yr;
        y_in_i = yi;
    }
}

template <bool kCkpt>
__device__ __forceinline__ bool fix_short_slice(const GroupDesc& G, const ClassDesc& C, const double* __restrict__ tab,
                                                double2* __restrict__ ps, int64_t nt, int64_t row, int64_t slot, int64_t n0,
                                                int64_t n1, bool initial, const double* __restrict__ E,
                                                double* __restrict__ d_out, double* __restrict__ a_out, int64_t sample_base,
                                                int4* __restrict__ buf, double* red, FixEdge* edge, int* status,
                                                double2* __restrict__ ck, int kc, int jm_lo, int jm_hi)
{
    const FixClass& F = C.fix;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, P = blockDim.x >> 5;
    const int I = G.I, i = lane & (I - 1), q = lane / I;
    const int N = G.N, K = G.K, m = G.m;
    const bool on = w < G.P;
    const int sg = w * (kLanes / I) + q, n_seg = G.P * (kLanes / I);   // this lane's segment
    const int s = sg * m, col = w * kLanes + lane;
    const int s_own = on ? min(N, s) : N, e_own = on ? min(N, s + m) : N;
    const bool live = nt > n0;
    const double dx = C.dx;
    const int4* __restrict__ tO = reinterpret_cast<const int4*>(tab + tab_fob(C));
    auto field = [&](int64_t n) { return n <= nt ? E[row + n - sample_base] : 0.0; };
    int sigma;
    if (!fix_range(G, F, ps, E, row, nt, n0, n1, sample_base, s_own, e_own, red, sigma)) return false;
    if (initial) fix_initial<kCkpt>(G, C, tab, ps, nt, row, s_own, e_own, E, d_out, a_out, sample_base, red, ck);

    const double unit = __hiloint2double((1023 + 60 - 2 * sigma) << 20, 0);   // |sigma| <= 112
    const int32_t ci = F.ci;
    const Digits cf = F.cf;
    int4* __restrict__ own = buf + (int64_t)w * m * (3 * kLanes) + lane;   // row r: gamma, psi, D at own + r * 96 + (0, 32, 64)
    const ShortGeom geo{N, K, m, I, s, sg, n_seg, col, on, own, edge, reinterpret_cast<const int4*>(tab + tab_fxp(C)), F.inv_b};
    if (on)
        for (int r = 0; r < m; ++r) {
            const int j = s + r;
            const double2 p = live && j < N ? ld_cg(ps + (int64_t)j * I + i) : make_double2(0.0, 0.0);
            put64(own + r * (3 * kLanes) + kLanes, double_to_fix((uint64_t)__double_as_longlong(p.x), sigma),
                  double_to_fix((uint64_t)__double_as_longlong(p.y), sigma));
        }

    for (int64_t n = n0; n < n1; ++n) {
        const bool active = n < nt, last = n + 1 == n1;
        const double En1 = active ? field(n + 1) : 0.0;
        const bool put = active && (last || n + 1 == nt);
        bool put_ck = false;
        if constexpr (kCkpt) put_ck = (n + 1) % kc == 0 && n + 1 < G.nt_max;
        const bool any_put = __any_sync(0xffffffffu, put) || put_ck;
        const Digits Eb = digits(live && n < nt ? __double2ll_rn(0.5 * (field(n) + field(n + 1)) * F.e_scale) : 0);

        int64_t yr, yi;
        short_solve(geo, Eb, yr, yi);
        // the whole segment, descending: psi^{n+1} and the observables
        ObsSums ob_sum{0.0, 0.0, 0.0};
        if (on) {
            int64_t sn = 0, sxh = 0, sxl = 0, svh = 0, svm = 0;
            int4* o = own + (int64_t)(m - 1) * (3 * kLanes);
            int4 gn = o[0], pn = o[kLanes], dn = o[2 * kLanes];
            int4 obn = __ldg(tO + min(s + m - 1, N - 1));
            for (int r = m - 1; r >= 0; --r) {
                const int j = s + r;
                const int4 g = gn, p = pn, d = dn, ob = obn;
                if (r > 0) {
                    gn = o[-3 * kLanes];
                    pn = o[-2 * kLanes];
                    dn = o[-kLanes];
                    obn = __ldg(tO + min(j - 1, N - 1));
                }
                back_row(g, d, yr, yi);
                int64_t xr = update_fix(ci, cf, digits(yr), lo64(p)), xi = update_fix(ci, cf, digits(yi), hi64(p));
                if (j < jm_lo || j > jm_hi) {
                    const Digits mm{ob.w, ob.z};
                    xr = mul_fix<3>(mm, digits(xr));
                    xi = mul_fix<3>(mm, digits(xi));
                }
                if (j >= N) xr = xi = 0;
                put64(o + kLanes, xr, xi);
                fix_observe(xr, xi, 2 * j - N + 1, ob, sn, sxh, sxl, svh, svm);
                if (any_put && j < N) {
                    const double2 z = make_double2(__longlong_as_double((long long)fix_to_double(xr, sigma)),
                                                   __longlong_as_double((long long)fix_to_double(xi, sigma)));
                    if (put) ps[(int64_t)j * I + i] = z;
                    if constexpr (kCkpt)
                        if (put_ck) ck[((n + 1) / kc) * ((int64_t)N * I) + (int64_t)j * I + i] = z;
                }
                o -= 3 * kLanes;
            }
            const double two32 = 4294967296.0;
            ob_sum.n = (double)sn * unit;
            ob_sum.x = fma((double)sxh, two32, (double)sxl) * (0.5 * dx * unit);
            ob_sum.v = fma((double)svh, two32, (double)svm) * (two32 * F.v_scale * unit);
        }
        const ObsSums t = reduce_obs(fix_lane_sum(ob_sum, I), red, P);
        if (w == 0 && q == 0 && active) {
            const int64_t kk = row + n + 1 - sample_base;
            d_out[kk] = t.x * dx;
            a_out[kk] = fma(En1, t.n, t.v) * dx;
            if (!(t.n * dx <= 1.0 + 1e-6)) status[slot] = 1;
        }
    }
    return true;
}

}  // namespace tdse
