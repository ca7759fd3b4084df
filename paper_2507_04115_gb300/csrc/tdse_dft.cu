// Fourier sums of long rows at a band of low frequencies (sm_103a):
//     S_r(w) = sum_n a_r,n exp(i w n dt),  n = 0 .. L_r - 1,
// for the dipole spectrum (frequencies given) and the power spectrum (DFT bins k of every row,
// w dt = -2 pi k / L_r).
//
// The direct sum costs 6 FP64 instructions per (sample, frequency) term: 2 to accumulate and 4 to turn the
// twiddle.  The frequencies of a spectrum, however, lie far below the sampling rate (harmonic 60 at
// dt = 0.02 turns by 0.07 rad a sample), so over a block of B samples exp(i w n dt) is smooth in n and
// the block's samples enter through a few Chebyshev moments only (Jacobi-Anger expansion):
//     n = c_b + (B/2) x,  x in (-1, 1):  e^{i w n dt} = e^{i w c_b dt} sum_q eps_q i^q J_q(phi) T_q(x),
//     phi = w dt B / 2,  eps_0 = 1, else 2,
//     S(w) = sum_b e^{i w c_b dt} sum_q eps_q i^q J_q(phi) M_{b,q},  M_{b,q} = sum_m a_{bB+m} T_q(x_m).
// k_moments forms the P moments of every block once (P/2 + 1 FP64 instructions per sample: T_q is even or
// odd about the block's centre, so samples are paired), k_band sums over blocks at P + 6 per (block,
// frequency).  The series is cut where 2 (phi/2)^P / P! < 1e-17, below double rounding.  J_q comes from
// Miller's backward recurrence, normalised by J_0 + 2 sum J_2k = 1; T_q(x_m) from the three-term
// recurrence in pairs of doubles; the block phases from products in pairs of doubles (or, for the bins,
// from k (2 c_b) mod 2 L in integers), re-seeded every 16 blocks.
//
// B and P come from dft_plan (tdse_rules.h), which minimises the instruction count L (P/2 + 1) + n_w (L / B)(P + 6)
// over them.  Measured, 512 rows of 55160 samples, 400 bins: 170 ms by the direct sum, 4.1 ms here (B = 512,
// P = 40); both kernels are bound by the FP64 pipe.  The direct sum stays where the band is too wide for
// blocks or has too few frequencies, for short rows (dft_plan), on a capturing stream, and without room for the moments.
#include "tdse_internal.h"

#include <algorithm>
#include <cmath>
#include <vector>

namespace tdse {

namespace {

constexpr int kBandThreads = 128;
constexpr int kBandTile = 16;   // blocks whose moments are staged in shared memory, and re-seed distance
constexpr double kPi = 3.14159265358979323846;

// hi + lo = a b exactly
__device__ __forceinline__ void two_prod(double a, double b, double& hi, double& lo)
{
    hi = a * b;
    lo = fma(a, b, -hi);
}

// T_q(x_m), q < P, x_m = (2 m + 1 - B) / B for m < B / 2 (the first half of a block; the second follows by
// parity), layout [m][q].  x is exact; the recurrence runs in pairs of doubles.
__global__ void k_cheb_table(int B, int P, double* __restrict__ T)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= B / 2) return;
    const double x = (2.0 * m + 1.0 - B) / B, x2 = 2.0 * x;
    double ah = 1.0, al = 0.0, bh = x, bl = 0.0;   // T_{q-1}, T_q
    T[(int64_t)m * P] = 1.0;
    for (int q = 1; q < P; ++q) {
        T[(int64_t)m * P + q] = bh + bl;
        double ph, pl;
        two_prod(x2, bh, ph, pl);
        pl = fma(x2, bl, pl);
        const double s = ph - ah;                     // two-sum of ph and -ah
        const double v = s - ph;
        const double e = (ph - (s - v)) + (-ah - v) + (pl - al);
        ah = bh;
        al = bl;
        bh = s + e;
        bl = e - (bh - s);
    }
}

// Moments of every block.  A warp holds 32 blocks (one per lane) and one parity of q: the pair of samples m
// and B - 1 - m enters the even moments by its sum and the odd ones by its difference.
template <int P>
__global__ void __launch_bounds__(128)
k_moments(const double* __restrict__ a, const int64_t* __restrict__ offs, const int64_t* __restrict__ boff, int64_t row0,
          int64_t n_rows, int B, const double* __restrict__ T, double* __restrict__ mom)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int odd = (int)(warp & 1);
    const int64_t first = boff[row0], total = boff[row0 + n_rows] - first;
    const int64_t g = (warp >> 1) * 32 + lane;
    if ((warp >> 1) * 32 >= total) return;
    const bool live = g < total;
    // row of the block
    int64_t lo = row0, hi = row0 + n_rows;   // boff[lo] <= first + g < boff[hi]
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (boff[mid] <= first + (live ? g : 0)) lo = mid;
        else hi = mid;
    }
    const int64_t base = offs[lo] + (first + (live ? g : 0) - boff[lo]) * B;
    const int64_t left = live ? offs[lo + 1] - base : 0;   // samples of the row from the block's start
    double acc[P / 2];
#pragma unroll
    for (int q = 0; q < P / 2; ++q) acc[q] = 0.0;
    const double sign = odd ? -1.0 : 1.0;
    auto sample = [&](int m) { return m < left ? a[base + m] : 0.0; };
    double u = sample(0), v = sample(B - 1);
    for (int m = 0; m < B / 2; ++m) {
        const double w = fma(v, sign, u);
        if (m + 1 < B / 2) {
            u = sample(m + 1);
            v = sample(B - 2 - m);
        }
        const double2* __restrict__ t = reinterpret_cast<const double2*>(T + (int64_t)m * P);
#pragma unroll
        for (int q = 0; q < P / 2; ++q) {
            const double2 tq = __ldg(t + q);
            acc[q] = fma(w, odd ? tq.y : tq.x, acc[q]);
        }
    }
    if (live) {
        double* o = mom + g * P + odd;
#pragma unroll
        for (int q = 0; q < P / 2; ++q) o[2 * q] = acc[q];
    }
}

// W_q = eps_q J_q(phi) (-1)^(q/2) (q even) or (-1)^((q-1)/2) (q odd), q < P
template <int P>
__device__ __forceinline__ void bessel_weights(double phi, double* W)
{
    const double x = fabs(phi);
    if (x < 0.125) {   // the recurrence would overflow: leading terms of the series
        const double h = 0.5 * x, h2 = -h * h;
        double lead = 1.0;
#pragma unroll
        for (int q = 0; q < P; ++q) {
            double s = 1.0, t = 1.0;
            for (int k = 1; k <= 6; ++k) {
                t *= h2 / (k * (double)(q + k));
                s += t;
            }
            W[q] = lead * s;
            lead *= h / (q + 1);
        }
    } else {
        const double r = 2.0 / x;
        double up = 0.0, cur = 1e-290, sum = 0.0;   // J_{q+1}, J_q, from q = P + 23
#pragma unroll 1
        for (int q = P + 23; q >= P; --q) {
            if ((q & 1) == 0) sum += 2.0 * cur;
            const double dn = fma(q * r, cur, -up);
            up = cur;
            cur = dn;
            if (fabs(cur) > 1e200) {
                cur *= 1e-250;
                up *= 1e-250;
                sum *= 1e-250;
            }
        }
#pragma unroll
        for (int q = P - 1; q >= 0; --q) {
            W[q] = cur;
            if ((q & 1) == 0) sum += (q == 0 ? 1.0 : 2.0) * cur;
            const double dn = fma(q * r, cur, -up);
            up = cur;
            cur = dn;
        }
        const double inv = 1.0 / sum;
#pragma unroll
        for (int q = 0; q < P; ++q) W[q] *= inv;
    }
#pragma unroll
    for (int q = 0; q < P; ++q) {
        const bool neg = ((q >> 1) & 1) != 0;
        const double e = q == 0 ? 1.0 : 2.0;
        W[q] *= neg ? -e : e;
        if ((q & 1) && phi < 0.0) W[q] = -W[q];
    }
}

// Sum over the blocks of R rows for one frequency per thread.  kBins: frequency k_begin + w of each row's
// DFT, the power spectrum out; else omega[w], weighted complex sums out.
template <int P, int R, bool kBins>
__global__ void __launch_bounds__(kBandThreads)
k_band(const double* __restrict__ mom, const int64_t* __restrict__ offs, const int64_t* __restrict__ boff, int64_t row0,
       int64_t n_rows, int B, double dt, const double* __restrict__ omega, int64_t k_begin, int64_t n_w,
       const double* __restrict__ weight, double* __restrict__ out)
{
    __shared__ double tile[kBandTile][R][P];
    const int64_t w = (int64_t)blockIdx.x * kBandThreads + threadIdx.x;
    const bool live = w < n_w;
    for (int64_t rt = blockIdx.y; rt * R < n_rows; rt += gridDim.y) {
        const int64_t r0 = row0 + rt * R;
        const int nr = (int)min((int64_t)R, row0 + n_rows - r0);
        int64_t nb = 0;
        for (int i = 0; i < nr; ++i) nb = max(nb, boff[r0 + i + 1] - boff[r0 + i]);
        const int64_t L = offs[r0 + 1] - offs[r0];   // kBins: all rows of the tile have this length
        const int64_t k = kBins ? (live ? k_begin + w : 0) : 0;
        const double om = kBins ? 0.0 : (live ? omega[w] : 0.0);
        double oh = 0.0, ol = 0.0, phi;
        if constexpr (kBins) {
            phi = L > 0 ? -kPi * ((double)k * (double)B) / (double)L : 0.0;
        } else {
            two_prod(om, dt, oh, ol);
            phi = oh * (0.5 * B);
        }
        double W[P];
        bessel_weights<P>(phi, W);
        // phase of sample position c2 / 2
        auto phase = [&](int64_t c2, double& s, double& c) {
            if constexpr (kBins) {
                const int64_t m = L > 0 ? (int64_t)(((unsigned long long)k * (unsigned long long)c2) % (unsigned long long)(2 * L)) : 0;
                sincospi(L > 0 ? -(double)m / (double)L : 0.0, &s, &c);
            } else {
                double th, tl, s0, c0;
                two_prod(oh, 0.5 * (double)c2, th, tl);
                tl = fma(ol, 0.5 * (double)c2, tl);
                sincos(th, &s0, &c0);
                s = fma(tl, c0, s0);
                c = fma(-tl, s0, c0);
            }
        };
        double wr, wi;   // from one block's centre to the next
        phase(2 * (int64_t)B, wi, wr);
        double ar[R], ai[R];
#pragma unroll
        for (int i = 0; i < R; ++i) ar[i] = ai[i] = 0.0;
        for (int64_t b0 = 0; b0 < nb; b0 += kBandTile) {
            __syncthreads();
            for (int e = threadIdx.x; e < kBandTile * R * P; e += kBandThreads) {
                const int q = e % P, i = (e / P) % R, t = e / (P * R);
                const int64_t b = b0 + t;
                double v = 0.0;
                if (i < nr && b < boff[r0 + i + 1] - boff[r0 + i]) v = mom[(boff[r0 + i] - boff[row0] + b) * P + q];
                tile[t][i][q] = v;
            }
            __syncthreads();
            double zr, zi;
            phase(2 * b0 * B + B - 1, zi, zr);
            const int cnt = (int)min((int64_t)kBandTile, nb - b0);
            for (int t = 0; t < cnt; ++t) {
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    double e = 0.0, o = 0.0;
#pragma unroll
                    for (int q = 0; q < P; q += 2) {
                        const double2 m2 = *reinterpret_cast<const double2*>(&tile[t][i][q]);
                        e = fma(W[q], m2.x, e);
                        o = fma(W[q + 1], m2.y, o);
                    }
                    ar[i] = fma(zr, e, fma(-zi, o, ar[i]));
                    ai[i] = fma(zr, o, fma(zi, e, ai[i]));
                }
                const double n2 = fma(zr, wr, -zi * wi);
                zi = fma(zr, wi, zi * wr);
                zr = n2;
            }
        }
        if (live)
            for (int i = 0; i < nr; ++i) {
                if constexpr (kBins) {
                    out[(r0 + i) * n_w + w] = (ar[i] * ar[i] + ai[i] * ai[i]) * dt * dt;
                } else {
                    const double wt = (weight ? weight[r0 + i] : 1.0) * dt * (1.0 / sqrt(2.0 * kPi));
                    reinterpret_cast<double2*>(out)[(r0 + i) * n_w + w] = make_double2(wt * ar[i], wt * ai[i]);
                }
            }
    }
}

template <int P>
cudaError_t run_band(const double* a, const int64_t* d_offs, const int64_t* d_boff, const std::vector<int64_t>& boff,
                     int64_t row0, int64_t n_rows, int B, double dt, const double* d_omega, int64_t k_begin, int64_t n_w,
                     const double* weight, bool bins, bool same_length, const double* d_T, double* d_mom, double* out,
                     cudaStream_t st)
{
    const int64_t blocks = boff[row0 + n_rows] - boff[row0];
    const int64_t warps = 2 * ((blocks + 31) / 32);
    if (warps > 0) k_moments<P><<<(unsigned)((warps + 3) / 4), 128, 0, st>>>(a, d_offs, d_boff, row0, n_rows, B, d_T, d_mom);
    const bool tile4 = n_rows >= 4 && (!bins || same_length);
    const int64_t tiles = tile4 ? (n_rows + 3) / 4 : n_rows;
    const dim3 grid((unsigned)((n_w + kBandThreads - 1) / kBandThreads), (unsigned)std::min<int64_t>(tiles, 65535));
    if (bins && tile4)
        k_band<P, 4, true><<<grid, kBandThreads, 0, st>>>(d_mom, d_offs, d_boff, row0, n_rows, B, dt, nullptr, k_begin, n_w, nullptr, out);
    else if (bins)
        k_band<P, 1, true><<<grid, kBandThreads, 0, st>>>(d_mom, d_offs, d_boff, row0, n_rows, B, dt, nullptr, k_begin, n_w, nullptr, out);
    else if (tile4)
        k_band<P, 4, false><<<grid, kBandThreads, 0, st>>>(d_mom, d_offs, d_boff, row0, n_rows, B, dt, d_omega, 0, n_w, weight, out);
    else
        k_band<P, 1, false><<<grid, kBandThreads, 0, st>>>(d_mom, d_offs, d_boff, row0, n_rows, B, dt, d_omega, 0, n_w, weight, out);
    return cudaGetLastError();
}

}  // namespace

bool band_dft_allowed(cudaStream_t st)
{
    cudaStreamCaptureStatus c = cudaStreamCaptureStatusActive;
    return cudaStreamIsCapturing(st, &c) == cudaSuccess && c == cudaStreamCaptureStatusNone;
}

cudaError_t launch_band_dft(const double* a, const int64_t* offs, int64_t n_rows, double dt, const double* omega_host,
                            int64_t k_begin, int64_t n_w, int B, int P, const double* weight, double* out, cudaStream_t st)
{
    const bool bins = omega_host == nullptr;
    bool same = true;
    std::vector<int64_t> boff((size_t)n_rows + 1);
    boff[0] = 0;
    for (int64_t r = 0; r < n_rows; ++r) {
        const int64_t L = offs[r + 1] - offs[r];
        same = same && L == offs[1] - offs[0];
        boff[r + 1] = boff[r] + (L + B - 1) / B;
    }
    // rows are taken in chunks whose moments stay below 256 MB
    const int64_t max_blocks = std::max<int64_t>((int64_t(256) << 20) / (8 * P), 1);
    int64_t most = 0;
    std::vector<int64_t> cuts{0};
    while (cuts.back() < n_rows) {
        const int64_t r0 = cuts.back();
        int64_t r1 = r0 + 1;
        while (r1 < n_rows && boff[r1 + 1] - boff[r0] <= max_blocks) ++r1;
        most = std::max(most, boff[r1] - boff[r0]);
        cuts.push_back(r1);
    }
    const size_t n_off = (size_t)n_rows + 1;
    const size_t doubles = 2 * n_off + (bins ? 0 : (size_t)n_w) + (size_t)(B / 2) * P + 2 + (size_t)most * P;
    double* buf = nullptr;
    cudaError_t e = cudaMallocAsync(reinterpret_cast<void**>(&buf), sizeof(double) * doubles, st);
    if (e != cudaSuccess) return e;
    int64_t* d_offs = reinterpret_cast<int64_t*>(buf);
    int64_t* d_boff = d_offs + n_off;
    double* d_T = buf + ((2 * n_off + 1) & ~size_t(1));   // 16-byte aligned for the double2 loads
    double* d_om = d_T + (size_t)(B / 2) * P;
    double* d_mom = d_om + (bins ? 0 : (size_t)n_w);
    // (a copy from pageable host memory has consumed the host buffer when cudaMemcpyAsync returns)
    if (e == cudaSuccess) e = cudaMemcpyAsync(d_offs, offs, sizeof(int64_t) * n_off, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(d_boff, boff.data(), sizeof(int64_t) * n_off, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && !bins) e = cudaMemcpyAsync(d_om, omega_host, sizeof(double) * n_w, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) {
        k_cheb_table<<<(B / 2 + 63) / 64, 64, 0, st>>>(B, P, d_T);
        e = cudaGetLastError();
    }
    for (size_t c = 0; e == cudaSuccess && c + 1 < cuts.size(); ++c) {
        const int64_t r0 = cuts[c], nr = cuts[c + 1] - cuts[c];
        auto run = P == 16 ? run_band<16> : (P == 24 ? run_band<24> : (P == 32 ? run_band<32> : run_band<40>));
        e = run(a, d_offs, d_boff, boff, r0, nr, B, dt, d_om, k_begin, n_w, weight, bins, same, d_T, d_mom, out, st);
    }
    const cudaError_t f = cudaFreeAsync(buf, st);
    return e != cudaSuccess ? e : f;
}

}  // namespace tdse
