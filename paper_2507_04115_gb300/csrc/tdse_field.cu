// Field ingestion (Sec. 4.2): coarsely sampled driving fields are moved to the time origin and
// interpolated to the propagation step by zero-padding their DFT.  For a row of M samples
// E_c[m] = E(t_min + m dt_c) the interpolant at t (measured from the first sample) is
//     E(t) = (1/M) sum_{k=-floor(M/2)}^{floor(M/2)} w_k Ehat_k exp(2 pi i k t / T),  T = M dt_c,
// w_k = 1/2 for |k| = M/2 when M is even, else 1.  The samples are real, so Ehat_{-k} = conj(Ehat_k)
// and E(t) = sum_{k=0}^{K} Re(c_k exp(2 pi i k t / T)), K = floor(M/2), with c_0 = Ehat_0 / M,
// c_k = 2 Ehat_k / M for 0 < k < M/2 and c_{M/2} = Ehat_{M/2} / M (even M).
//
// The sum over k is the same trigonometric polynomial at every output, so it is evaluated once on an
// oversampled uniform grid of G = 2^g >= 4 K nodes by a fast Fourier transform, and at the outputs by
// local interpolation with a Kaiser-Bessel window (the gridding method of non-uniform FFTs):
//     sum_l phi(x - l) e^{2 pi i k l / G} = e^{2 pi i k x / G} phihat(2 pi k / G) + aliases,
//     phi(z) = I0(b sqrt(1 - (2 z / w)^2)), |z| <= w / 2,
//     phihat(xi) = w sinh(sqrt(b^2 - (w xi / 2)^2)) / sqrt(b^2 - (w xi / 2)^2),
// the coefficients divided by phihat beforehand.  With w = 16 nodes and b = pi w (1 - K / G) the aliases
// are below e^-b ~ 1e-16 of a coefficient at the least oversampling, 2, and smaller above it.
//
//   k_field_tables  twiddles and, per output, its first node and w weights (shared by all rows)
//   k_field_coeffs  c_k: the samples m and M - m are paired (their sum meets the cosine, their
//                   difference the sine): M FP64 multiply-adds per coefficient, twiddles from a table
//   k_field_grid    one CTA per row: the G node values by a complex FFT of length G / 2 in shared memory
//   k_field_interp  16 multiply-adds per output
//   k_field_direct  the sum over k itself, for few coefficients and rows (resample_field_plan)
// Work per row: O(M^2 / 2 + G log G + 16 n_fine) FP64 instructions instead of O(3 M^2 + 3 M n_fine) for the
// direct sums with turning twiddles.  Measured, 256 rows of 2400 samples to 55160: 217 ms by the direct
// sums, 2.9 ms here: coefficients 1.8, tables 0.4, interpolation 0.4, grid 0.15.
#include "tdse_device.cuh"
#include "tdse_internal.h"

namespace tdse {

namespace {

constexpr int kWin = 16;            // nodes under the window
static_assert(kWin * sizeof(double) + sizeof(int) == kFieldOutputBytes, "tables per output");
constexpr int kInterpRows = 8;      // rows per thread of the interpolation
constexpr int kGridThreads = 512;
constexpr double kPi = 3.14159265358979323846;

// I0(x), |x| <= 16 pi, by its power series (all terms positive), r[k] = 1 / k^2: a division per term would be
// most of the work
constexpr int kI0Terms = 100;
__device__ double bessel_i0(double x, const double* r)
{
    const double h = 0.25 * x * x;
    double t = 1.0, s = 1.0;
    for (int k = 1; k < kI0Terms; ++k) {
        t *= h * r[k];
        s += t;
        if (__double2hiint(t) + (60 << 20) < __double2hiint(s)) break;   // below 2^-60 of the sum
    }
    return s;
}

// n dt_f / T as a pair of doubles
__device__ __forceinline__ void periods(int64_t n, double dt_f, double T, double& q, double& ql)
{
    const double t = (double)n * dt_f, tl = fma((double)n, dt_f, -t);
    q = t / T;
    ql = (fma(-q, T, t) + tl) / T;
}

// The tables of outputs n_first .. n_first + n_cnt - 1.
__global__ void k_field_tables(int M, int G, double b, double dt_f, double T, int64_t n_first, int64_t n_cnt,
                               double2* __restrict__ tw_m, double2* __restrict__ tw_g, int* __restrict__ node,
                               double* __restrict__ wgt)
{
    __shared__ double inv_k2[kI0Terms];
    for (int k = threadIdx.x; k < kI0Terms; k += blockDim.x) inv_k2[k] = k > 0 ? 1.0 / ((double)k * k) : 0.0;
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < M) {   // e^{2 pi i j / M}
        double s, c;
        sincospi(2.0 * (double)i / (double)M, &s, &c);
        tw_m[i] = make_double2(c, s);
    }
    if (i < G / 2) {   // e^{2 pi i j / G}
        double s, c;
        sincospi(2.0 * (double)i / (double)G, &s, &c);
        tw_g[i] = make_double2(c, s);
    }
    if (i < n_cnt * kWin) {
        const int64_t n = i / kWin;
        const int j = (int)(i % kWin);
        // x = G frac(n dt_f / T) as a node number and a remainder
        double q, ql;
        periods(n_first + n, dt_f, T, q, ql);
        const double xh = (q - floor(q)) * G, l = floor(xh);
        const double z = (xh - l) + ql * G;            // offset from node l, in [0, 1] to rounding
        const double y = (z + (kWin / 2 - 1) - j) * (2.0 / kWin);
        const double r = 1.0 - y * y;
        wgt[j * n_cnt + n] = r > 0.0 ? bessel_i0(b * sqrt(r), inv_k2) : 0.0;   // phi up to the factor in k_field_grid
        if (j == 0) node[n] = ((int)l - (kWin / 2 - 1) + G) & (G - 1);
    }
}

// c_k / phihat_k of every row, k = 0 .. K (one thread per k; the row's sums and differences in shared memory); kDirect: c_k,
// with twiddles of the block's own (one launch less for small calls)
template <bool kDirect>
__global__ void __launch_bounds__(128)
k_field_coeffs(const double* __restrict__ coarse, int M, int G, double b, const double2* __restrict__ tw, double2* __restrict__ coef)
{
    extern __shared__ double row[];
    const int64_t r = blockIdx.y;
    const int K = M / 2, H = (M - 1) / 2;   // pairs m = 1 .. H
    double* dif = row + H + 1;
    const double* x = coarse + r * M;
    for (int m = threadIdx.x + 1; m <= H; m += blockDim.x) {
        row[m] = x[m] + x[M - m];
        dif[m] = x[m] - x[M - m];
    }
    double2* own = reinterpret_cast<double2*>(row + 2 * (H + 1));
    if constexpr (kDirect)
        for (int m = threadIdx.x; m < M; m += blockDim.x) {
            double s, c;
            sincospi(2.0 * (double)m / (double)M, &s, &c);
            own[m] = make_double2(c, s);
        }
    auto twiddle = [&](int i) { return kDirect ? own[i] : __ldg(tw + i); };
    __syncthreads();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k > K) return;
    // Ehat_k = sum_m E_c[m] exp(-2 pi i k m / M)
    double sr = x[0], si = 0.0;
    if (M % 2 == 0) sr += (k & 1) ? -x[M / 2] : x[M / 2];
    int idx = 0;
    double2 z = make_double2(0.0, 0.0);
    if (H > 0) {
        idx = k % M;
        z = twiddle(idx);
    }
    for (int m = 1; m <= H; ++m) {
        const double2 c = z;
        idx += k;
        if (idx >= M) idx -= M;
        z = twiddle(idx);
        sr = fma(row[m], c.x, sr);
        si = fma(-dif[m], c.y, si);
    }
    double f = (k == 0 || 2 * k == M ? 1.0 : 2.0) / M;
    if (!kDirect) {   // Kaiser-Bessel window's transform at xi = 2 pi k / G
        const double xi = 2.0 * kPi * k / G, u = 0.5 * kWin * xi, v = sqrt(b * b - u * u);
        f = f * v / (kWin * sinh(v));
    }
    coef[r * (K + 1) + k] = make_double2(f * sr, f * si);
}

// Node values g_l = sum_k Re(c_k e^{2 pi i k l / G}), l < G: real data from a half spectrum X_k = c_k / 2
// (X_0 = c_0) by one complex transform of length N = G / 2, z_n = g_2n + i g_2n+1,
//     Z_k = (X_k + conj(X_{N-k})) + i e^{2 pi i k / G} (X_k - conj(X_{N-k})),
// decimation in time, in place.
__global__ void __launch_bounds__(kGridThreads)
k_field_grid(const double2* __restrict__ coef, int K, int G, int log_n, const double2* __restrict__ tw, double* __restrict__ grid)
{
    extern __shared__ double2 z[];
    const int64_t r = blockIdx.x;
    const int N = G / 2;
    const double2* c = coef + r * (K + 1);
    for (int k = threadIdx.x; k < N; k += blockDim.x) {
        const int kc = N - k;   // K < N / 2 * 2: both indexes are inside [0, N]
        double2 X = make_double2(0.0, 0.0), Y = X;
        if (k <= K) X = c[k];
        if (kc <= K) Y = c[kc];
        const double fx = k == 0 ? 1.0 : 0.5, fy = 0.5;
        X.x *= fx;
        X.y = k == 0 ? 0.0 : X.y * fx;   // c_0 is real, and so is the Nyquist coefficient of an even M
        Y.x *= fy;
        Y.y *= -fy;
        const double2 e = __ldg(tw + k);
        const double ar = X.x + Y.x, ai = X.y + Y.y, br = X.x - Y.x, bi = X.y - Y.y;
        // + i e (b)
        const double pr = e.x * br - e.y * bi, pi = e.x * bi + e.y * br;
        z[(int)(__brev((unsigned)k) >> (32 - log_n))] = make_double2(ar - pi, ai + pr);
    }
    for (int s = 1; s <= log_n; ++s) {
        __syncthreads();
        const int half = 1 << (s - 1);
        for (int t = threadIdx.x; t < N / 2; t += blockDim.x) {
            const int j = t & (half - 1), i0 = ((t >> (s - 1)) << s) + j, i1 = i0 + half;
            const double2 w = __ldg(tw + ((int64_t)j << (log_n + 1 - s)));   // e^{2 pi i j / 2^s}
            const double2 a = z[i0], b = z[i1];
            const double tr = fma(b.x, w.x, -b.y * w.y), ti = fma(b.x, w.y, b.y * w.x);
            z[i0] = make_double2(a.x + tr, a.y + ti);
            z[i1] = make_double2(a.x - tr, a.y - ti);
        }
    }
    __syncthreads();
    double2* g = reinterpret_cast<double2*>(grid + r * G);
    for (int n = threadIdx.x; n < N; n += blockDim.x) g[n] = z[n];
}

// The direct sum, an output per thread: Horner's rule in z = e^{2 pi i t / T} over blocks of 64 coefficients, each
// block times z to its first index (from a sincospi of its own: an error of z counts at most 63 times).
__global__ void __launch_bounds__(256)
k_field_direct(const double2* __restrict__ coef, int K, double dt_f, double T, int64_t n_fine, int64_t out_stride,
               double* __restrict__ out)
{
    extern __shared__ double2 c[];
    const int64_t r = blockIdx.y;
    for (int k = threadIdx.x; k <= K; k += blockDim.x) c[k] = coef[r * (K + 1) + k];
    __syncthreads();
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= n_fine) return;
    double q, ul;
    periods(n, dt_f, T, q, ul);
    const double uh = q - floor(q);
    auto power = [&](int k) {   // z^k
        const double ph = k * uh, pl = (fma((double)k, uh, -ph) + k * ul) * (2.0 * kPi);
        double s, co;
        sincospi(2.0 * (ph - floor(ph)), &s, &co);
        return make_double2(fma(-pl, s, co), fma(pl, co, s));
    };
    const double2 z = power(1);
    double sum = 0.0;
    for (int k0 = 0; k0 <= K; k0 += 64) {
        int k = min(k0 + 63, K);
        double hr = c[k].x, hi = c[k].y;
        for (--k; k >= k0; --k) {
            const double t = fma(hr, z.x, fma(-hi, z.y, c[k].x));
            hi = fma(hr, z.y, fma(hi, z.x, c[k].y));
            hr = t;
        }
        const double2 p = power(k0);
        sum = fma(hr, p.x, fma(-hi, p.y, sum));
    }
    out[r * out_stride + n] = sum;
}

// Outputs n_first .. n_first + n_cnt - 1 of the rows (out at output n_first).
__global__ void __launch_bounds__(256)
k_field_interp(const double* __restrict__ grid, int64_t n_rows, int G, int64_t n_cnt, int64_t out_stride,
               const int* __restrict__ node, const double* __restrict__ wgt, double* __restrict__ out)
{
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= n_cnt) return;
    double w[kWin];
#pragma unroll
    for (int j = 0; j < kWin; ++j) w[j] = wgt[j * n_cnt + n];
    const int l0 = node[n];
    const int64_t r0 = (int64_t)blockIdx.y * kInterpRows, r1 = min(n_rows, r0 + kInterpRows);
    for (int64_t r = r0; r < r1; ++r) {
        const double* g = grid + r * G;
        double s = 0.0, t = 0.0;
#pragma unroll
        for (int j = 0; j < kWin; j += 2) {
            s = fma(w[j], g[(l0 + j) & (G - 1)], s);
            t = fma(w[j + 1], g[(l0 + j + 1) & (G - 1)], t);
        }
        out[r * out_stride + n] = s + t;
    }
}

}  // namespace

cudaError_t launch_resample_field(const double* coarse, int64_t n_rows, int M, double dt_c, double dt_f,
                                  int64_t n_fine, int64_t out_stride, double* out, const FieldPlan& plan, void* work,
                                  cudaStream_t st)
{
    if (n_rows == 0 || n_fine == 0) return cudaSuccess;
    const int K = M / 2, G = plan.direct ? 0 : field_nodes(M);
    static std::atomic<bool> attr_set[kMaxAttrDevices];   // rows up to 8192 samples: 64 and 128 KB of shared memory
    int dev = 0;
    if (attr_needed(attr_set, &dev)) {
        cudaError_t e = cudaFuncSetAttribute(k_field_coeffs<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 8192 * 8);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_field_grid, cudaFuncAttributeMaxDynamicSharedMemorySize, 8192 * 16);
        if (e != cudaSuccess) return e;
        attr_done(attr_set, dev);
    }
    double2* tw_m = static_cast<double2*>(work);
    double2* tw_g = tw_m + (plan.direct ? 0 : M);
    double2* coef = tw_g + G / 2;
    double* grid = reinterpret_cast<double*>(coef + plan.rows * (K + 1));
    double* wgt = grid + plan.rows * G;
    int* node = reinterpret_cast<int*>(wgt + kWin * plan.outputs);
    const double T = M * dt_c, b = plan.direct ? 0.0 : kPi * kWin * (1.0 - (double)K / G);
    int log_n = 0;
    while ((1 << log_n) < G / 2) ++log_n;
    auto tables = [&](int64_t n0, int64_t cnt) {
        const int64_t items = std::max<int64_t>({(int64_t)M, (int64_t)G / 2, cnt * kWin});
        k_field_tables<<<(unsigned)((items + 255) / 256), 256, 0, st>>>(M, G, b, dt_f, T, n0, cnt, tw_m, tw_g, node, wgt);
    };
    const bool one = plan.outputs >= n_fine;   // every output's window fits: built once for all rows
    if (!plan.direct) tables(0, one ? n_fine : 0);
    cudaError_t e = cudaGetLastError();
    for (int64_t r0 = 0; e == cudaSuccess && r0 < n_rows; r0 += plan.rows) {
        const int64_t nr = std::min(plan.rows, n_rows - r0);
        const dim3 cgrid((unsigned)((K + 128) / 128), (unsigned)nr);
        const size_t csmem = sizeof(double) * 2 * ((M - 1) / 2 + 1);
        if (plan.direct) {
            k_field_coeffs<true><<<cgrid, 128, csmem + sizeof(double2) * M, st>>>(coarse + r0 * M, M, G, b, nullptr, coef);
            k_field_direct<<<dim3((unsigned)((n_fine + 255) / 256), (unsigned)nr), 256, sizeof(double2) * (K + 1), st>>>(
                coef, K, dt_f, T, n_fine, out_stride, out + r0 * out_stride);
            e = cudaGetLastError();
            continue;
        }
        k_field_coeffs<false><<<cgrid, 128, csmem, st>>>(coarse + r0 * M, M, G, b, tw_m, coef);
        k_field_grid<<<(unsigned)nr, kGridThreads, sizeof(double2) * (G / 2), st>>>(coef, K, G, log_n, tw_g, grid);
        for (int64_t n0 = 0; n0 < n_fine; n0 += plan.outputs) {
            const int64_t cnt = std::min(plan.outputs, n_fine - n0);
            if (!one) tables(n0, cnt);
            k_field_interp<<<dim3((unsigned)((cnt + 255) / 256), (unsigned)((nr + kInterpRows - 1) / kInterpRows)), 256, 0, st>>>(
                grid, nr, G, cnt, out_stride, node, wgt, out + r0 * out_stride + n0);
        }
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace tdse
