// Host rules of the batch-free entry points: passes and routes by the sizes of a call.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdint>

namespace tdse {

// ---- field ingestion (tdse_field.cu)

// Nodes of the oversampled grid: at least 4 per highest harmonic, and room for the window.
inline int field_nodes(int M)
{
    int G = 64;
    while (G < 4 * (M / 2)) G *= 2;
    return G;
}

// Bytes of the tables of an output (16 weights and a node).
constexpr int64_t kFieldOutputBytes = 132;

// Is the sum over k the quicker way?  In us: it takes rows x (3 M + 84) FP64 instructions per output (4 per coefficient and
// the phases) behind a chain of M / 2 coefficients; the grid takes 4700 per output for the window's weights, whatever the
// rows, 16 more per row, and the chains of its passes.  Measured, whole calls, direct and by the grid: 1 row of 100
// samples to 400000 outputs 416 and 2880 us, 8 of 100 to 55160 462 and 605, 16 of 100 683 and 620, 4 of 300 to 12000
// 327 and 342, 1 of 600 to 1000 329 and 286, 1 of 1200 to 400000 2256 and 3067, 2 of them 4023 and 3083.
inline bool field_direct(int64_t n_rows, int M, int64_t n_fine)
{
    const double r = (double)n_rows, n = (double)n_fine;
    const double direct = 0.17 * M + 1.4e-6 * n * r * (3.0 * M + 84.0);
    const double grid = 25.0 + 0.085 * M + 1.4e-6 * n * (4700.0 + 16.0 * r);
    return M <= 2000 && direct < grid;   // (M: samples and twiddles fit 48 KB of shared memory)
}

// Rows and outputs of a pass: the rows' coefficients and grids take at most `room` bytes, the outputs' tables a quarter
// of it (or those of one row, of one output).  bytes: the scratch of such a pass.
struct FieldPlan {
    bool direct;   // the sum over k itself: no grid, no tables per output
    int64_t rows, outputs;
    size_t bytes;
};
inline FieldPlan resample_field_plan(int64_t n_rows, int M, int64_t n_fine, size_t room)
{
    FieldPlan p;
    p.direct = field_direct(n_rows, M, n_fine);
    const int G = p.direct ? 0 : field_nodes(M);
    const int64_t per_row = 16 * (int64_t)(M / 2 + 1) + 8 * (int64_t)G;
    p.rows = std::max<int64_t>(1, std::min<int64_t>({n_rows, (int64_t)room / per_row, 65535}));
    p.outputs = p.direct ? 0 : std::max<int64_t>(1, std::min<int64_t>(n_fine, (int64_t)(room / 4) / kFieldOutputBytes));
    p.bytes = (p.direct ? 0 : 16 * ((size_t)M + G / 2)) + (size_t)p.rows * per_row + (size_t)p.outputs * kFieldOutputBytes;
    return p;
}

// ---- far field (tdse_hankel.cu)

// Nodes of the J0 table for arguments up to x_max, 0 where CUDA's j0 is the quicker way.  In us: the table takes
// 75 + 0.49 x to fill (a serial recurrence of x terms at its last node), and saves up to 2.5 a source point and thread
// (j0 takes 1 us at x = 3, 4 from x = 100 on; the table 0.75), as often as an SM has CTAs; beyond its end nothing (the
// share of smaller arguments taken as that of a product of three even factors k, rho, rho').  1.2: the estimate's
// error.  Measured, whole calls, j0 and table: 4 x 4 source points, 40 frequencies, 64 radii at x = 4000 294 and
// 2320 us; 8 x 8 at x = 100 470 and 441; 16 x 16 at x = 20, 500, 1500 846 and 533, 1277 and 884, 1261 and 1397;
// 32 x 32, 340, 256 at x = 30 8070 and 3660.
constexpr int kJ0MaxNodes = 16384;   // 1.5 MB of coefficients, arguments up to 4096
inline int j0_table_nodes(double x_max, int64_t n_rho, int64_t n_z, int64_t n_omega, int64_t n_obs, int sm_count)
{
    if (!std::isfinite(x_max)) return 0;
    const double end = 0.25 * kJ0MaxNodes, x = std::min(x_max, end);
    const double ctas = (double)n_omega * (double)((n_obs + 127) / 128);
    const double t = x / std::max(x_max, 1e-300), l = x_max > end ? std::log(t) : 0.0;
    const double inside = x_max > end ? t * (1.0 - l + 0.5 * l * l) : 1.0;
    const double saved = (double)n_rho * (double)n_z * std::max(1.0, ctas / std::max(1, sm_count)) * 2.5 * x / (x + 40.0) * inside;
    return saved > 1.2 * (75.0 + 0.49 * x) ? (int)std::min(4.0 * x_max + 3.0, (double)kJ0MaxNodes) : 0;
}

// ---- spectra (tdse_dft.cu)

// Block length and number of moments for n_rows rows of `samples` samples at n_w frequencies that turn by at most
// `turn` rad a sample; false where the direct sum is the better one: where blocks do not halve its instructions, and
// for short rows, whose chain of samples is shorter than the moments' kernels.  In us: the direct sum takes 0.235 a
// sample, or 1.3e-5 a sample and thread once these fill the pipe; the moments 130 + 2.2 P for their tables and weights,
// a warp's chain over half a block, and a CTA's over the blocks of its 4 rows (k_band), as often as an SM has CTAs.
// Measured, whole calls, direct and by moments: 64 rows of 512, 60 bins 325 and 547 us; 16 of 1000, 60 446 and 564; 4 of
// 2000, 120 677 and 737 (60: 676 and 593); 16 of 4000, 400 1154 and 1289 (120: 1151 and 762; 64 rows: 2023 and 1282).
inline bool dft_plan(int64_t samples, double turn, int64_t n_w, int64_t n_rows, int sm_count, int* B_out, int* P_out)
{
    *B_out = *P_out = 0;
    if (n_w < 32 || samples < 256 || !(turn < 0.8)) return false;
    double best = 0.5 * 6.0 * (double)n_w;   // the direct sum per sample; the blocks have to halve it
    int best_B = 0, best_P = 0;
    for (int B = 32; B <= 1024; B *= 2)
        for (int P = 16; P <= 40; P += 8) {
            const double phi = 0.5 * turn * B;
            if (phi > 0.0 && P * std::log(0.5 * phi) - std::lgamma(P + 1.0) + std::log(2.0) > std::log(1e-17)) continue;
            const double cost = 0.5 * P + 1.0 + (double)n_w * (P + 6.0) / B;
            if (cost < best) {
                best = cost;
                best_B = B;
                best_P = P;
            }
            break;
        }
    if (best_B == 0) return false;
    const double L = (double)samples, rows = (double)n_rows, B = best_B, P = best_P, sms = std::max(1, sm_count);
    const double tiles = (double)((n_w + 127) / 128), R = n_rows >= 4 ? 4.0 : 1.0, blocks = std::ceil(L / B);
    const double direct = L * std::max(0.235, 1.3e-5 * rows * tiles * 128.0);
    const double moments = 130.0 + 2.2 * P + 0.0083 * B * P * std::max(1.0, rows * blocks / 16.0 / (4.0 * sms)) +
                           0.0333 * blocks * R * (P + 6.0) * std::max(1.0, tiles * std::ceil(rows / R) / sms);
    if (moments >= direct) return false;
    *B_out = best_B;
    *P_out = best_P;
    return true;
}

}  // namespace tdse
