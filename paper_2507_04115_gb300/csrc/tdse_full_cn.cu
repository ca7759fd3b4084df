// FULL_CN real-time propagation kernel of libtdse (sm_103a), FP64 and MIXED precision.
//
// Numerical scheme (one step t_n -> t_{n+1}, h = dt/2, Ebar = (E_n + E_{n+1})/2):
//   A = 1 + i h H(Ebar) = tridiag(-i beta, 1 + i s_j, -i beta),  beta = dt/(4 dx^2),
//   s_j = h (1/dx^2 + V_j + x_j Ebar);  psi^{n+1} = m (A^{-1}(1 - i h H) psi^n) = m (2 A^{-1} psi^n - psi^n)
// because (1 - i h H) = 2 - A.  So each step is one tridiagonal solve A y = psi^n (Thomas: forward
// elimination, back substitution) and a pointwise update -- no right-hand-side product.
//
// Parallel layout (lane-batched segmented Thomas):
//   * a group = 32 instances of one grid class, one per lane, so every warp instruction works on
//     32 independent systems (the FP64 pipe costs the same per warp instruction whatever the
//     number of active lanes, so full warps matter);
//   * a CTA of P warps owns one group at a time; warp w owns the grid segment [w m, (w+1) m);
//   * a segment's sweep starts K points before the segment and closes K points after it.  A is
//     strictly diagonally dominant with Re(pivot) >= 1, so both the forward coefficients and the
//     back substitution forget their starting values by a factor <= beta per point; K is chosen so
//     that beta^K < 1e-18, below double rounding.  The outermost segments use the exact walls.
//   * scheduling: a persistent grid of CTAs picks groups dynamically, one time slice (a few tens
//     of steps) at a time, always the free group with the most remaining slices.  A group is
//     claimed with an atomic compare-and-swap and released after its slice; a CTA that finds no
//     free unfinished group exits.  No CTA ever waits on another, so there is nothing to time out.
//     Dynamic slices balance the load when the number of groups is not a multiple of the SM count
//     (8192 instances = 256 groups on 152 SMs) and when groups have different lengths.
// HBM layouts: psi [group][j][lane] (16 B per point, a warp reads 512 contiguous bytes), scratch per
// CTA [warp][row][gamma | D][lane].
//
// FP64 slices whose class, fields and states are within the fixed-point range run on the integer pipe
// (tdse_cn_fix.cuh: 2.7 times the rate on the volume batch, 6.5 on one atom); the FP64 sweeps here serve the others
// and MIXED.
#include "tdse_cn_fix.cuh"

namespace tdse {

// One scheduling slice of a lane-split group (G.I = 32/L instances, each over L lanes of every
// warp; see GroupDesc).  Lane l of warp w holds instance i = l % I and sweeps segment
// sigma = w L + l / I, i.e. sweep rows r = 0 .. m + 2K - 1 at points j = sigma m - K + r: every
// lane of a warp runs the same trip counts whatever its segment.  Rows before the first wall
// restart the forward coefficients at zero (the exact boundary condition of the Thomas sweep),
// rows at or beyond the far wall restart the back substitution at zero; the own segment is rows
// K .. K + m - 1.  Observables are summed over the L lanes of an instance by shuffles, then over the
// warps.  No bulk copies on this path (it serves small batches and the widened groups of uneven
// batches, where the FP64 elimination is the bound in both precisions).  The observable sums stay
// off the FP64 pipe as on the 32-wide path: float pairs (FP64) or floats (MIXED) over blocks of
// kObsBlock own rows, each block widened to double by integer operations; tab_obs is the class's
// float4 table, (x_hi, x_lo, dV_hi, dV_lo) for FP64 and (x, dV, m, -) for MIXED.
template <bool kMixed, bool kCkpt>
__device__ __forceinline__ void split_slice(const GroupDesc& G, const Fma64& F, typename Prec<kMixed>::C* __restrict__ ps,
                                            const double2* __restrict__ tab_ab2, const double2* __restrict__ tab_xv2,
                                            const double* __restrict__ tab_m, double inv_beta,
                                            typename Prec<kMixed>::R two_over_beta, double dx, int jm_lo, int jm_hi,
                                            int64_t nt, int64_t row, int64_t slot, int64_t n0, int64_t n1,
                                            bool initial, const double* __restrict__ E, double* __restrict__ d_out,
                                            double* __restrict__ a_out, int64_t sample_base,
                                            typename Prec<kMixed>::C* __restrict__ sc, double* red, int* status,
                                            double2* __restrict__ ck, int kc, const float4* __restrict__ tab_obs)
{
    using R = typename Prec<kMixed>::R;
    using Cx = typename Prec<kMixed>::C;
    const int lane = threadIdx.x & 31;
    const int w = threadIdx.x >> 5;
    const int P = blockDim.x >> 5;
    const int I = G.I, L = kLanes / G.I;
    const int i = lane & (I - 1), q = lane / I;
    const int N = G.N, K = G.K, m = G.m;
    const int sigma = w * L + q;
    const int nrows = w < G.P ? m + 2 * K : 0;   // warp-uniform
    const int base = sigma * m - K;
    const int s_own = min(N, sigma * m), e_own = min(N, sigma * m + m);
    auto lane_sum = [&](ObsSums o) {
        for (int off = I; off < kLanes; off <<= 1) {
            o.n += __shfl_xor_sync(0xffffffffu, o.n, off);
            o.x += __shfl_xor_sync(0xffffffffu, o.x, off);
            o.v += __shfl_xor_sync(0xffffffffu, o.v, off);
        }
        return o;
    };

    if (initial) {
        ObsSums o{0.0, 0.0, 0.0};
        if (w < G.P)
            for (int j = s_own; j < e_own; ++j) {
                const Cx p = ld_cg(ps + (int64_t)j * I + i);
                const double rho = fma((double)p.x, (double)p.x, (double)p.y * (double)p.y);
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
        if constexpr (kCkpt)   // checkpoint 0: the initial state (each lane copies its own points)
            if (w < G.P)
                for (int j = s_own; j < e_own; ++j) ck[(int64_t)j * I + i] = ld_cg(ps + (int64_t)j * I + i);
        __syncthreads();
    }

    for (int64_t n = n0; n < n1; ++n) {
        const bool active = n < nt;
        double En = 0.0, En1 = 0.0;
        if (active) {
            En = E[row + n - sample_base];
            En1 = E[row + n + 1 - sample_base];
        }
        const double Eb = 0.5 * (En + En1);

        // forward elimination (scaled variables as in the 32-wide path)
        {
            auto load_row = [&](int rr) -> Cx {
                const int j = base + rr;
                return (rr < nrows && (unsigned)j < (unsigned)N) ? ld_cg(ps + (int64_t)j * I + i) : mk(R(0), R(0));
            };
            double cr = 0.0, ci = 0.0;
            R Dr = 0, Di = 0;
            Cx pa = load_row(0), pb = load_row(1);
            Cx* r = sc;
            for (int rr = 0; rr < nrows; ++rr) {
                const Cx p = pa;
                pa = pb;
                pb = load_row(rr + 2);
                const int j = base + rr;
                const bool in = (unsigned)j < (unsigned)N;
                const double2 t = __ldg(tab_ab2 + min(max(j, 0), N - 1));
                const double Qr = F.add(ci, inv_beta);
                const double Qi = F.sub(fma(t.y, Eb, t.x), cr);
                const double q2 = fma(Qr, Qr, F.mul(Qi, Qi));
                const double inv = kMixed ? rcp_pos_2nd(q2) : rcp_pos(q2);
                cr = in ? F.mul(Qi, inv) : 0.0;
                ci = in ? F.mul(Qr, inv) : 0.0;
                R gr, gi;
                if constexpr (kMixed) {
                    gr = d2f(cr);
                    gi = d2f(ci);
                } else {
                    gr = cr;
                    gi = ci;
                }
                const R ur = F.sub(p.x, Di);
                const R ui = F.add(p.y, Dr);
                Dr = in ? fma(gr, ui, F.mul(gi, ur)) : R(0);
                Di = in ? fma(gi, ui, F.mul(-gr, ur)) : R(0);
                r[lane] = mk(gr, gi);
                r[kLanes + lane] = mk(Dr, Di);
                r += 2 * kLanes;
            }
        }
        __syncthreads();   // every read of psi^n precedes any write of psi^{n+1}

        // back substitution over rows nrows-1 .. K; own segment rows K .. K+m-1
        ObsSums o{0.0, 0.0, 0.0};
        {
            R Yr = 0, Yi = 0;
            float snh = 0.f, snl = 0.f, sxh = 0.f, sxl = 0.f, svh = 0.f, svl = 0.f;
            int blk = 0;
            auto fold = [&]() {
                o.n = F.add(f2d_int(snh), o.n);
                o.x = F.add(f2d_int(sxh), o.x);
                o.v = F.add(f2d_int(svh), o.v);
                if constexpr (!kMixed) {
                    o.n = F.add(f2d_int(snl), o.n);
                    o.x = F.add(f2d_int(sxl), o.x);
                    o.v = F.add(f2d_int(svl), o.v);
                }
                snh = snl = sxh = sxl = svh = svl = 0.f;
                blk = 0;
            };
            const Cx* r = sc + (int64_t)(nrows - 1) * (2 * kLanes);
#pragma unroll 2
            for (int rr = nrows - 1; rr >= K; --rr) {
                const int j = base + rr;
                const Cx g2 = r[lane];
                const Cx d2 = r[kLanes + lane];
                r -= 2 * kLanes;
                const R nr = fma(g2.x, Yr, fma(-g2.y, Yi, d2.x));
                const R ni = fma(g2.x, Yi, fma(g2.y, Yr, d2.y));
                Yr = j < N ? nr : R(0);   // Dirichlet restart at the far wall
                Yi = j < N ? ni : R(0);
                if (rr < K + m && j < N) {
                    Cx* pw = ps + (int64_t)j * I + i;
                    const Cx old = ld_cg(pw);
                    R xr = fma(two_over_beta, Yr, -old.x);
                    R xi = fma(two_over_beta, Yi, -old.y);
                    if (j < jm_lo || j > jm_hi) {
                        const R mm = (R)__ldg(tab_m + j);
                        xr = F.mul(xr, mm);
                        xi = F.mul(xi, mm);
                    }
                    if (active) *pw = mk(xr, xi);
                    const float4 tf = __ldg(tab_obs + j);
                    if constexpr (kMixed) {
                        const float rho = fmaf(xr, xr, xi * xi);
                        snh += rho;
                        sxh = fmaf(tf.x, rho, sxh);
                        svh = fmaf(tf.y, rho, svh);
                    } else {
                        float rh, rl;
                        sq_mod_ff(xr, xi, rh, rl);
                        ff_acc(snh, snl, rh, rl);
                        ff_fma_acc(sxh, sxl, tf.x, tf.y, rh, rl);
                        ff_fma_acc(svh, svl, tf.z, tf.w, rh, rl);
                    }
                    if (++blk == kObsBlock) fold();
                }
            }
            fold();
        }
        const ObsSums t = reduce_obs(lane_sum(o), red, P);   // its barrier orders this step's writes
        if (w == 0 && q == 0 && active) {
            const int64_t kk = row + n + 1 - sample_base;
            d_out[kk] = t.x * dx;
            a_out[kk] = fma(En1, t.n, t.v) * dx;
            if (!(t.n * dx <= (kMixed ? 1.0 + 1e-3 : 1.0 + 1e-6))) status[slot] = 1;
        }
        if constexpr (kCkpt)   // checkpoint (n + 1)/kc of the adjoint's recomputation
            if ((n + 1) % kc == 0 && n + 1 < G.nt_max && w < G.P) {
                double2* dst = ck + ((n + 1) / kc) * ((int64_t)N * I);
                for (int j = s_own; j < e_own; ++j) dst[(int64_t)j * I + i] = ld_cg(ps + (int64_t)j * I + i);
            }
    }
}

// One forward row of the elimination in float (the MIXED path's halo rows): gamma = (cr, ci),
// D = (Dr, Di), t = (S0_j, Xh_j)/beta rounded to float, p = psi_j.
__device__ __forceinline__ void fwd_row_f32(float2 t, float2 p, float Eb, float inv_beta, float& cr, float& ci,
                                            float& Dr, float& Di)
{
    float inv;
    const float Qr = ci + inv_beta;
    const float Qi = fmaf(t.y, Eb, t.x) - cr;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(fmaf(Qr, Qr, Qi * Qi)));
    cr = Qi * inv;
    ci = Qr * inv;
    const float ur = p.x - Di, ui = p.y + Dr;
    const float nDr = fmaf(cr, ui, ci * ur);
    Di = fmaf(ci, ui, -cr * ur);
    Dr = nDr;
}

// kFix: classes with the fixed-point form may be among the groups.  Batches without one run the kernel that holds their
// sweeps alone: beside the fixed-point forms the compiler's schedule of these is 2.5 to 5 % slower, and the forms' shared
// memory takes from L1 (64 x 8192 points at 32 lanes, dt / (4 dx^2) = 0.5, 64 steps: 14.64 ms and 14.06; 8192 x 4096
// points, 32 steps: 71.2 and 69.5).
template <bool kMixed, bool kCkpt, bool kFix>
__global__ void __launch_bounds__(512, 1)
k_propagate_full_cn(const GroupDesc* __restrict__ groups, int64_t n_groups, const ClassDesc* __restrict__ cls,
                    const double* __restrict__ tab, const int64_t* __restrict__ slot_row,
                    const int64_t* __restrict__ slot_nt, void* __restrict__ psi_raw, void* __restrict__ scratch_raw,
                    int rows, const double* __restrict__ E, double* __restrict__ d_out, double* __restrict__ a_out,
                    int64_t sample_base, int64_t step_begin, int64_t step_end, int slice, int mask_on,
                    int* __restrict__ busy, int* __restrict__ progress, int* __restrict__ status, int ring_slots, uint32_t wait_polls,
                    double2* __restrict__ ckpt, const int64_t* __restrict__ ckpt_off, int kc)
{
    using R = typename Prec<kMixed>::R;
    using Cx = typename Prec<kMixed>::C;
    extern __shared__ double red[];   // [P][3][32]
    __shared__ int s_g, s_k;
    const int lane = threadIdx.x & 31;
    const int w = threadIdx.x >> 5;
    const int P = blockDim.x >> 5;
    Cx* __restrict__ psi_all = static_cast<Cx*>(psi_raw);
    // MIXED: per-warp ring of bulk-copy slots after the reduction area (see the back substitution)
    const int kRing = ring_slots;   // bulk-copy slots per warp (MIXED)
    uint64_t* bars = reinterpret_cast<uint64_t*>(red + P * 3 * kLanes) + w * kRing;
    unsigned char* ring = reinterpret_cast<unsigned char*>(reinterpret_cast<uint64_t*>(red + P * 3 * kLanes) + P * kRing) +
                          (size_t)w * kRing * kSlotBytes;
    uint32_t rc = 0;            // ring slots consumed by this warp so far (slot and phase of the next)
    bool timed_out = false;
    if constexpr (kMixed) {
        if (lane == 0)
            for (int k = 0; k < kRing; ++k) mbar_init(bars + k, 1);
        fence_mbar_init();
        __syncthreads();
    }

    for (;;) {
        if (w == 0) {
            int k = 0;
            const int g = pick_group(groups, n_groups, busy, progress, step_begin, step_end, slice, &k);
            if (lane == 0) {
                s_g = g;
                s_k = k;
            }
        }
        __syncthreads();
        const int g = s_g;
        const int kslice = s_k;
        __threadfence();   // order this CTA's reads of the group's psi after the claim
        __syncthreads();   // s_g / s_k are rewritten only after every warp has read them
        if (g < 0) break;

        const GroupDesc G = groups[g];
        const ClassDesc C = cls[G.cls];
        const Fma64 F{C.one, C.nzero};
        const int N = G.N, K = G.K;
        const int64_t slot = G.slot0 + (lane & (G.I - 1));   // this lane's instance
        const int64_t nt = slot_nt[slot];   // -1 for padding lanes
        const int64_t row = slot_row[slot];
        const double beta = C.beta;
        const double inv_beta = 1.0 / beta;
        const R two_over_beta = (R)(2.0 / beta);
        const double dx = C.dx;
        Cx* __restrict__ ps = psi_all + G.psi_off;
        const double2* __restrict__ tab_ab2 = reinterpret_cast<const double2*>(tab + tab_ab(C));
        const double2* __restrict__ tab_xv2 = reinterpret_cast<const double2*>(tab + tab_xv(C));
        const double* __restrict__ tab_m = tab + tab_mk(C);
        const float4* __restrict__ tab_f4 = reinterpret_cast<const float4*>(tab + tab_fx(C));
        const int jm_lo = mask_on ? C.jm_lo : 0;
        const int jm_hi = mask_on ? C.jm_hi : N - 1;
        const int64_t n_end = min(step_end, G.nt_max);
        const int64_t n0 = step_begin + (int64_t)kslice * slice;
        const int64_t n1 = min(n_end, n0 + slice);

        bool done = false;
        if constexpr (kFix)
            if (C.fix.ok && fix_short(G))
                done = fix_short_slice<kCkpt>(G, C, tab, ps, nt, row, slot, n0, n1, kslice == 0 && step_begin == 0, E, d_out,
                                              a_out, sample_base,
                                              reinterpret_cast<int4*>(scratch_raw) + (int64_t)blockIdx.x * P * rows * (2 * kLanes),
                                              red, reinterpret_cast<FixEdge*>(red + P * 3 * kLanes), status,
                                              kCkpt ? ckpt + ckpt_off[g] : nullptr, kc, jm_lo, jm_hi);
            else if (fix_shape(G, C))
                done = fix_slice<kCkpt>(G, C, tab, ps, nt, row, slot, n0, n1, kslice == 0 && step_begin == 0, E, d_out, a_out,
                                        sample_base, reinterpret_cast<int4*>(scratch_raw) + (int64_t)blockIdx.x * P * rows * (2 * kLanes),
                                        red, status, kCkpt ? ckpt + ckpt_off[g] : nullptr, kc, jm_lo, jm_hi);
        if (!done) {   // (all that the FP64 sweeps need inside: held across the fixed-point forms it slows them by 1 to 7 %)
        Cx* __restrict__ sc = static_cast<Cx*>(scratch_raw) + ((int64_t)blockIdx.x * P + w) * rows * (2 * kLanes);
        GroupDesc H = G;
        if constexpr (kFix) {   // the FP64 sweeps' own split, packed into the CTA's scratch
            H.P = G.P64;
            H.m = G.m64;
            sc = static_cast<Cx*>(scratch_raw) + ((int64_t)blockIdx.x * P * rows + (int64_t)w * (H.m + 2 * K)) * (2 * kLanes);
        }
        // warps beyond the group's segment count own an empty segment
        const int Pg = H.P, m = H.m;
        const int s = w < Pg ? min(N, w * m) : N;
        const int e = w < Pg ? min(N, s + m) : N;
        const int lo = w < Pg ? max(0, s - K) : N;
        const int hi = w < Pg ? min(N, e + K) : N;
        if (G.I != kLanes) {
            split_slice<kMixed, kCkpt>(H, F, ps, tab_ab2, tab_xv2, tab_m, inv_beta, two_over_beta, dx, jm_lo, jm_hi,
                                       nt, row, slot, n0, n1, kslice == 0 && step_begin == 0, E, d_out, a_out,
                                       sample_base, sc, red, status, kCkpt ? ckpt + ckpt_off[g] : nullptr, kc,
                                       reinterpret_cast<const float4*>(tab + (kMixed ? tab_fx(C) : tab_xff(C))));
        } else {
        if (kslice == 0 && step_begin == 0) {
            // observables of the initial state
            ObsSums o{0.0, 0.0, 0.0};
            for (int j = s; j < e; ++j) {
                const Cx p = ld_cg(ps + (int64_t)j * kLanes + lane);
                const double rho = fma((double)p.x, (double)p.x, (double)p.y * (double)p.y);
                const double2 xv = __ldg(tab_xv2 + j);
                o.n += rho;
                o.x = fma(xv.x, rho, o.x);
                o.v = fma(xv.y, rho, o.v);
            }
            const ObsSums t = reduce_obs(o, red, P);
            if (w == 0 && nt >= 0) {
                const double E0 = E[row - sample_base];
                d_out[row - sample_base] = t.x * dx;
                a_out[row - sample_base] = fma(E0, t.n, t.v) * dx;
            }
            if constexpr (kCkpt && !kMixed) {   // checkpoint 0: the initial state (own rows)
                double2* dst = ckpt + ckpt_off[g];
                for (int j = s; j < e; ++j) dst[(int64_t)j * kLanes + lane] = ld_cg(ps + (int64_t)j * kLanes + lane);
            }
            __syncthreads();
        }

        for (int64_t n = n0; n < n1; ++n) {
            const bool active = n < nt;
            double En = 0.0, En1 = 0.0;
            if (active) {
                En = E[row + n - sample_base];
                En1 = E[row + n + 1 - sample_base];
            }
            const double Eb = 0.5 * (En + En1);

            // Forward elimination over [lo, hi) in scaled variables: Q = q/beta with
            // q_j = 1 + i s_j + beta^2 g_{j-1} the Thomas pivot, gamma = i beta g = i conj(Q)/|Q|^2,
            // D = beta d = -i gamma u with u = psi + i D_{j-1}.  Tables hold s_j/beta split as
            // (S0_j, Xh_j)/beta; Re Q = 1/beta + Im gamma_{j-1}, Im Q = s_j/beta - Re gamma_{j-1}.
            // FP64: every row in double.  MIXED: the own segment keeps the recurrence for Q and gamma
            // in double (its stability over 1e5 steps needs it); the halo rows only converge the
            // truncated recurrences to this path's float accuracy (the halo is kMixedHaloTol long),
            // so they run in float, and the top halo's rows are not stored (the back substitution
            // stops at s).
            if constexpr (kMixed) {
                float crf = 0.0f, cif = 0.0f;
                R Dr = 0, Di = 0;
                const float inv_beta_f = d2f(inv_beta);
                const float Ebf = d2f(Eb);
                const float2* __restrict__ taf = reinterpret_cast<const float2*>(tab + tab_af(C));
                {
                    const Cx* pj = ps + (int64_t)lo * kLanes + lane;
                    Cx pa = lo < s ? ld_cg(pj) : mk(R(0), R(0));
                    Cx pb = lo + 1 < s ? ld_cg(pj + kLanes) : mk(R(0), R(0));
                    const Cx* pnext = pj + 2 * kLanes;
                    for (int j = lo; j < s; ++j) {
                        const Cx p = pa;
                        pa = pb;
                        if (j + 2 < s) pb = ld_cg(pnext);
                        pnext += kLanes;
                        fwd_row_f32(__ldg(taf + j), p, Ebf, inv_beta_f, crf, cif, Dr, Di);
                    }
                }
                double cr = crf, ci = cif;
                Cx* r = sc + (int64_t)(s - lo) * (2 * kLanes);
                {
                    // pointers advance by increments: no 64-bit index arithmetic inside the loop
                    const Cx* pj = ps + (int64_t)s * kLanes + lane;
                    Cx pa = s < e ? ld_cg(pj) : mk(R(0), R(0));
                    Cx pb = s + 1 < e ? ld_cg(pj + kLanes) : mk(R(0), R(0));
                    const Cx* pnext = pj + 2 * kLanes;
                    const double2* tp = tab_ab2 + s;
#pragma unroll 2
                    for (int j = s; j < e; ++j) {
                        const Cx p = pa;
                        pa = pb;
                        if (j + 2 < e) pb = ld_cg(pnext);
                        pnext += kLanes;
                        const double2 t = __ldg(tp);
                        ++tp;
                        const double Qr = F.add(ci, inv_beta);
                        const double Qi = F.sub(fma(t.y, Eb, t.x), cr);
                        // gamma is rounded to float right after, so a 2^-40 reciprocal suffices (the
                        // recurrence damps an error by beta^2 per point; it stays ~1e-12)
                        const double inv = rcp_pos_2nd(fma(Qr, Qr, F.mul(Qi, Qi)));
                        cr = F.mul(Qi, inv);
                        ci = F.mul(Qr, inv);
                        const R gr = d2f(cr);
                        const R gi = d2f(ci);
                        const R ur = F.sub(p.x, Di);
                        const R ui = F.add(p.y, Dr);
                        Dr = fma(gr, ui, F.mul(gi, ur));
                        Di = fma(gi, ui, F.mul(-gr, ur));
                        r[lane] = mk(gr, gi);
                        r[kLanes + lane] = mk(Dr, Di);
                        r += 2 * kLanes;
                    }
                }
                if (e < hi) {
                    crf = d2f(cr);
                    cif = d2f(ci);
                    const Cx* pj = ps + (int64_t)e * kLanes + lane;
                    Cx pa = ld_cg(pj);
                    Cx pb = e + 1 < hi ? ld_cg(pj + kLanes) : mk(R(0), R(0));
                    const Cx* pnext = pj + 2 * kLanes;
                    for (int j = e; j < hi; ++j) {
                        const Cx p = pa;
                        pa = pb;
                        if (j + 2 < hi) pb = ld_cg(pnext);
                        pnext += kLanes;
                        fwd_row_f32(__ldg(taf + j), p, Ebf, inv_beta_f, crf, cif, Dr, Di);
                        r[lane] = mk(crf, cif);
                        r[kLanes + lane] = mk(Dr, Di);
                        r += 2 * kLanes;
                    }
                }
            } else {
                double cr = 0.0, ci = 0.0;
                R Dr = 0, Di = 0;
                // pointers advance by increments: no 64-bit index arithmetic inside the loop
                const Cx* pj = ps + (int64_t)lo * kLanes + lane;
                Cx pa = lo < hi ? ld_cg(pj) : mk(R(0), R(0));
                Cx pb = lo + 1 < hi ? ld_cg(pj + kLanes) : mk(R(0), R(0));
                const Cx* pnext = pj + 2 * kLanes;
                const double2* tp = tab_ab2 + lo;
                Cx* r = sc;
#pragma unroll 2
                for (int j = lo; j < hi; ++j) {
                    const Cx p = pa;
                    pa = pb;
                    if (j + 2 < hi) pb = ld_cg(pnext);
                    pnext += kLanes;
                    const double2 t = __ldg(tp);
                    ++tp;
                    const double Qr = F.add(ci, inv_beta);
                    const double Qi = F.sub(fma(t.y, Eb, t.x), cr);
                    const double inv = rcp_pos(fma(Qr, Qr, F.mul(Qi, Qi)));
                    cr = F.mul(Qi, inv);
                    ci = F.mul(Qr, inv);
                    const R ur = F.sub(p.x, Di);
                    const R ui = F.add(p.y, Dr);
                    Dr = fma(cr, ui, F.mul(ci, ur));
                    Di = fma(ci, ui, F.mul(-cr, ur));
                    r[lane] = mk(cr, ci);
                    r[kLanes + lane] = mk(Dr, Di);
                    r += 2 * kLanes;
                }
            }
            if constexpr (kMixed) fence_proxy_async();   // scratch and psi stores precede the bulk reads
            __syncthreads();   // every read of psi^n (own segment and halos) precedes any write of psi^{n+1}

            // Back substitution Y_j = D_j + gamma_j Y_{j+1} (Y = beta y), seeded with 0 at hi (exact at
            // the wall), then psi^{n+1}_j = m_j (2 Y_j / beta - psi^n_j) on the own segment.
            R Yr = 0, Yi = 0;
            ObsSums o{0.0, 0.0, 0.0};
            if constexpr (kMixed) {
                // Rows hi-1 .. s stream through a per-warp ring of shared-memory slots filled by bulk
                // asynchronous copies: a slot holds kSlotRows consecutive rows (their float2 gamma|D
                // scratch rows, 512 bytes each, then their float2 psi rows, 256 bytes each), brought in
                // by two copies completed on the slot's mbarrier, kRing slots ahead of the arithmetic:
                // the float back substitution is too short per row to hide HBM latency by itself.
                // After a wait that gives up (a failed copy) the ring is drained with bounded waits and
                // not used again: the instances are flagged and nothing can hang.
                const int nrows = hi - s;
                const int nblk = (nrows + kSlotRows - 1) / kSlotRows;
                auto issue = [&](int b) {
                    const int j_top = hi - 1 - b * kSlotRows;
                    const int cnt = min(kSlotRows, nrows - b * kSlotRows);
                    const int j_bot = j_top - cnt + 1;
                    const uint32_t k = (rc + b) % kRing;
                    unsigned char* dst = ring + k * kSlotBytes;
                    mbar_arrive_expect_tx(bars + k, (uint32_t)cnt * 768u);
                    bulk_g2s(dst, sc + (int64_t)(j_bot - lo) * (2 * kLanes), (uint32_t)cnt * 512u, bars + k);
                    bulk_g2s(dst + kSlotRows * 512, ps + (int64_t)j_bot * kLanes, (uint32_t)cnt * 256u, bars + k);
                };
                int issued = 0;
                if (!timed_out) {
                    if (lane == 0)
                        for (int b = 0; b < min(kRing, nblk); ++b) issue(b);
                    issued = min(kRing, nblk);
                }
                __syncwarp();
                R fn = 0, fx = 0, fv = 0;
                int blk = 0;
                for (int b = 0; b < nblk && !timed_out; ++b) {
                    const uint32_t k = (rc + b) % kRing;
                    const bool ok = __all_sync(0xffffffffu, mbar_wait(bars + k, ((rc + b) / kRing) & 1u, wait_polls));
                    if (!ok) {
                        // drain every copy still in flight (this slot's included) with the full
                        // bound before leaving the ring unused for the rest of the launch
                        timed_out = true;
                        for (int b2 = b; b2 < issued; ++b2)
                            mbar_wait(bars + (rc + b2) % kRing, ((rc + b2) / kRing) & 1u, kDrainPolls);
                        break;
                    }
                    const unsigned char* slotp = ring + k * kSlotBytes;
                    const int j_top = hi - 1 - b * kSlotRows;
                    const int cnt = min(kSlotRows, nrows - b * kSlotRows);
                    const int j_bot = j_top - cnt + 1;
                    for (int j = j_top; j >= j_bot; --j) {
                        const int rr = j - j_bot;
                        const float2* srow = reinterpret_cast<const float2*>(slotp + rr * 512);
                        const float2 g2 = srow[lane], d2 = srow[kLanes + lane];
                        const float2 old = reinterpret_cast<const float2*>(slotp + kSlotRows * 512 + rr * 256)[lane];
                        const R nr = fma(g2.x, Yr, fma(-g2.y, Yi, d2.x));
                        Yi = fma(g2.x, Yi, fma(g2.y, Yr, d2.y));
                        Yr = nr;
                        if (j < e) {
                            const float4 fxv = __ldg(tab_f4 + j);   // (x, dV/dx, m) in float
                            R xr = fma(two_over_beta, Yr, -old.x);
                            R xi = fma(two_over_beta, Yi, -old.y);
                            if (j < jm_lo || j > jm_hi) {
                                xr *= fxv.z;
                                xi *= fxv.z;
                            }
                            if (active) ps[(int64_t)j * kLanes + lane] = mk(xr, xi);
                            const R rho = fma(xr, xr, xi * xi);
                            fn += rho;
                            fx = fma(fxv.x, rho, fx);
                            fv = fma(fxv.y, rho, fv);
                            if (++blk == kObsBlock) {
                                o.n = F.add(f2d_int(fn), o.n);
                                o.x = F.add(f2d_int(fx), o.x);
                                o.v = F.add(f2d_int(fv), o.v);
                                fn = fx = fv = 0;
                                blk = 0;
                            }
                        }
                    }
                    __syncwarp();
                    if (b + kRing < nblk) {
                        if (lane == 0) {
                            fence_proxy_async();
                            issue(b + kRing);
                        }
                        issued = b + kRing + 1;
                    }
                }
                o.n = F.add(f2d_int(fn), o.n);
                o.x = F.add(f2d_int(fx), o.x);
                o.v = F.add(f2d_int(fv), o.v);
                rc += (uint32_t)max(nblk, 0);
            } else {
                const Cx* r = sc + (int64_t)(hi - 1 - lo) * (2 * kLanes);
                for (int j = hi - 1; j >= e; --j) {
                    const Cx g2 = r[lane];
                    const Cx d2 = r[kLanes + lane];
                    r -= 2 * kLanes;
                    const R nr = fma(g2.x, Yr, fma(-g2.y, Yi, d2.x));
                    Yi = fma(g2.x, Yi, fma(g2.y, Yr, d2.y));
                    Yr = nr;
                }
                // own segment, with the scratch row and the old psi prefetched two points ahead;
                // pointers step down by decrements
                Cx ga = mk(R(0), R(0)), da = ga, gb = ga, db = ga, pa = ga, pb = ga;
                Cx* pw = ps + (int64_t)(e - 1) * kLanes + lane;       // psi_j (store)
                const Cx* pl = pw - 2 * kLanes;                        // psi_{j-2} (prefetch)
                const double* tm = tab_m + (e - 1);
                const float4* txf = reinterpret_cast<const float4*>(tab + tab_xff(C)) + (e - 1);
                // observable sums: rho = |psi|^2 as a float pair (sq_mod_ff), summed as float pairs
                // over blocks of kObsBlock points on the FP32 pipe (with x and dV/dx as float pairs),
                // each block's pair widened to double (integer operations) and added in double: no
                // FP64 instruction per point, 2 per block and sum
                float snh = 0.f, snl = 0.f, sxh = 0.f, sxl = 0.f, svh = 0.f, svl = 0.f;
                int blk = 0;
                if (e - 1 >= s) {
                    ga = r[lane];
                    da = r[kLanes + lane];
                    pa = ld_cg(pw);
                }
                if (e - 2 >= s) {
                    gb = r[-2 * kLanes + lane];
                    db = r[-kLanes + lane];
                    pb = ld_cg(pw - kLanes);
                }
#pragma unroll 2
                for (int j = e - 1; j >= s; --j) {
                    const Cx g2 = ga, d2 = da, old = pa;
                    ga = gb;
                    da = db;
                    pa = pb;
                    if (j - 2 >= s) {
                        gb = r[-4 * kLanes + lane];
                        db = r[-3 * kLanes + lane];
                        pb = ld_cg(pl);
                    }
                    pl -= kLanes;
                    r -= 2 * kLanes;
                    const R nr = fma(g2.x, Yr, fma(-g2.y, Yi, d2.x));
                    Yi = fma(g2.x, Yi, fma(g2.y, Yr, d2.y));
                    Yr = nr;
                    R xr = fma(two_over_beta, Yr, -old.x);
                    R xi = fma(two_over_beta, Yi, -old.y);
                    if (j < jm_lo || j > jm_hi) {
                        const R mm = __ldg(tm);
                        xr = F.mul(xr, mm);
                        xi = F.mul(xi, mm);
                    }
                    --tm;
                    if (active) *pw = mk(xr, xi);
                    pw -= kLanes;
                    float rh, rl;   // rho = |psi|^2 as a float pair, off the FP64 pipe
                    sq_mod_ff(xr, xi, rh, rl);
                    const float4 xf = __ldg(txf);
                    --txf;
                    ff_acc(snh, snl, rh, rl);
                    ff_fma_acc(sxh, sxl, xf.x, xf.y, rh, rl);
                    ff_fma_acc(svh, svl, xf.z, xf.w, rh, rl);
                    if (++blk == kObsBlock) {
                        o.n = F.add(f2d_int(snh), F.add(f2d_int(snl), o.n));
                        o.x = F.add(f2d_int(sxh), F.add(f2d_int(sxl), o.x));
                        o.v = F.add(f2d_int(svh), F.add(f2d_int(svl), o.v));
                        snh = snl = sxh = sxl = svh = svl = 0.f;
                        blk = 0;
                    }
                }
                o.n = F.add(f2d_int(snh), F.add(f2d_int(snl), o.n));
                o.x = F.add(f2d_int(sxh), F.add(f2d_int(sxl), o.x));
                o.v = F.add(f2d_int(svh), F.add(f2d_int(svl), o.v));
            }
            const ObsSums t = reduce_obs(o, red, P);   // its barrier also orders this step's psi writes
            if (w == 0 && active) {
                const int64_t kk = row + n + 1 - sample_base;
                d_out[kk] = t.x * dx;
                a_out[kk] = fma(En1, t.n, t.v) * dx;
                // the norm never grows in exact arithmetic (unitary step, mask <= 1); the allowance
                // covers rounding: 1e-6 in FP64, 1e-3 in MIXED where float psi random-walks ~1e-5
                if (!(t.n * dx <= (kMixed ? 1.0 + 1e-3 : 1.0 + 1e-6))) status[slot] = 1;
            }
            if constexpr (kCkpt && !kMixed)   // checkpoint (n + 1)/kc of the adjoint's recomputation
                if ((n + 1) % kc == 0 && n + 1 < G.nt_max) {
                    double2* dst = ckpt + ckpt_off[g] + ((n + 1) / kc) * ((int64_t)N * kLanes);
                    for (int j = s; j < e; ++j) dst[(int64_t)j * kLanes + lane] = ld_cg(ps + (int64_t)j * kLanes + lane);
                }
        }
        }   // 32-wide group
        }

        if (timed_out) status[slot] = 2;   // a bulk copy did not complete in time

        // release the group: its psi writes become visible before the next owner's claim
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            *(volatile int*)(progress + g) = kslice + 1;
            __threadfence();
            atomicExch(busy + g, 0);
        }
    }
}

cudaError_t launch_propagate_full_cn(int mixed, int fix, const GroupDesc* d_groups, int64_t n_groups, int P, int ctas,
                                     const ClassDesc* d_cls, const double* d_tab, const int64_t* d_slot_row,
                                     const int64_t* d_slot_nt, void* d_psi, void* d_scratch, int rows,
                                     const double* E, double* d_out, double* a_out, int64_t sample_base,
                                     int64_t step_begin, int64_t step_end, int slice, int mask_on, int* d_busy,
                                     int* d_progress, int* d_status, int ring, uint32_t wait_polls, cudaStream_t st,
                                     void* d_ckpt, const int64_t* d_ckpt_off, int kc)
{
    if (n_groups == 0 || ctas == 0) return cudaSuccess;
    if (d_ckpt && (mixed || kc < 1)) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(d_busy, 0, sizeof(int) * n_groups, st);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(d_progress, 0, sizeof(int) * n_groups, st);
    if (e != cudaSuccess) return e;
    if (mixed && (ring < kMinRing || ring > kMaxRing)) return cudaErrorInvalidValue;
    const size_t smem = full_cn_smem_bytes(mixed, P, ring, fix);
    if (mixed) {
        static std::atomic<bool> attr_set[kMaxAttrDevices];
        int dev = 0;
        if (attr_needed(attr_set, &dev)) {
            e = cudaFuncSetAttribute(k_propagate_full_cn<true, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)full_cn_smem_max_bytes());
            if (e != cudaSuccess) return e;
            attr_done(attr_set, dev);
        }
        k_propagate_full_cn<true, false, false><<<(unsigned)ctas, P * kLanes, smem, st>>>(
            d_groups, n_groups, d_cls, d_tab, d_slot_row, d_slot_nt, d_psi, d_scratch, rows, E, d_out, a_out,
            sample_base, step_begin, step_end, slice, mask_on, d_busy, d_progress, d_status, ring, wait_polls,
            nullptr, nullptr, 0);
    } else {
        auto kernel = d_ckpt ? (fix ? k_propagate_full_cn<false, true, true> : k_propagate_full_cn<false, true, false>)
                             : (fix ? k_propagate_full_cn<false, false, true> : k_propagate_full_cn<false, false, false>);
        kernel<<<(unsigned)ctas, P * kLanes, smem, st>>>(
            d_groups, n_groups, d_cls, d_tab, d_slot_row, d_slot_nt, d_psi, d_scratch, rows, E, d_out, a_out,
            sample_base, step_begin, step_end, slice, mask_on, d_busy, d_progress, d_status, ring, wait_polls,
            static_cast<double2*>(d_ckpt), d_ckpt_off, kc);
    }
    return cudaGetLastError();
}

int propagate_ring_slots(int P, int per_sm) { return full_cn_ring_slots(P, per_sm); }

int propagate_max_ctas_per_sm(int mixed, int fix, int P)
{
    int n = 0;
    const size_t smem = full_cn_smem_bytes(mixed, P, kMinRing, fix);   // the shallowest ring
    if (mixed &&
        cudaFuncSetAttribute(k_propagate_full_cn<true, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)full_cn_smem_max_bytes()) != cudaSuccess) {
        cudaGetLastError();   // do not leave the failure for the next launch check
        return 1;
    }
    auto kernel = mixed ? k_propagate_full_cn<true, false, false>
                        : (fix ? k_propagate_full_cn<false, false, true> : k_propagate_full_cn<false, false, false>);
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, P * kLanes, smem);
    if (e != cudaSuccess) return 1;
    return n > 0 ? n : 1;
}

}  // namespace tdse
