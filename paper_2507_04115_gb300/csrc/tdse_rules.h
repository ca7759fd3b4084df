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

// Rows and outputs of a pass: the rows' coefficients and grids take at most `room` bytes, the outputs' tables a quarter
// of it (or those of one row, of one output).  bytes: the scratch of such a pass.
struct FieldPlan {
    int64_t rows, outputs;
    size_t bytes;
};
inline FieldPlan resample_field_plan(int64_t n_rows, int M, int64_t n_fine, size_t room)
{
    const int G = field_nodes(M);
    const int64_t per_row = 16 * (int64_t)(M / 2 + 1) + 8 * (int64_t)G;
    FieldPlan p;
    p.rows = std::max<int64_t>(1, std::min<int64_t>({n_rows, (int64_t)room / per_row, 65535}));
    p.outputs = std::max<int64_t>(1, std::min<int64_t>(n_fine, (int64_t)(room / 4) / kFieldOutputBytes));
    p.bytes = 16 * ((size_t)M + G / 2) + (size_t)p.rows * per_row + (size_t)p.outputs * kFieldOutputBytes;
    return p;
}

}  // namespace tdse
