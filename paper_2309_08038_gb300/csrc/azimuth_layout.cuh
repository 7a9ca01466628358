// Shared memory of the run-time-plan row kernels (azimuth_rows.cu, azimuth_mig_fft.cu).
#pragma once

#include "row_fft.cuh"

namespace rosar {
namespace rowfft {

// Shared-memory layout of a row: x [padded], then (stage_h) the H row [padded], then the twiddle table.
struct Layout {
    int full_tab;
    int stage_h;
    size_t bytes;
};

constexpr size_t AF_SMEM_CAP = 200 * 1024;

inline Layout layout_for(int N, bool with_h) {
    Layout l{};
    const size_t row = sizeof(float2) * (size_t)padded_len(N);
    const size_t two = sizeof(float2) * (size_t)(64 + coarse_len(N));
    l.stage_h = with_h && (2 * row + two <= AF_SMEM_CAP);
    l.full_tab = 0;      // two-level table: ~N/64 + 64 sincospif per CTA instead of N
    l.bytes = row * (l.stage_h ? 2 : 1) + two;
    return l;
}

}  // namespace rowfft
}  // namespace rosar
