// What the row kernels (azimuth_rows.cu, azimuth_mig_fft.cu) and the readers of their spectra (azimuth_fft.cu) share:
// the row lengths with compile-time plans, and the shared memory of the run-time plans.
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

// A row length with a compile-time plan, taken where the run-time planner picks exactly these radices (H, made by the
// run-time plan, is in their order).
template <int N, int... R>
struct FixedRadices {
    static bool is(int n_az, const RowPlan &pl) {
        constexpr int rad[] = {R...};
        if (n_az != N || pl.pad_shift != 31 || pl.npass != (int)sizeof...(R)) return false;
        for (int i = 0; i < pl.npass; ++i)
            if (pl.rad[i] != rad[i]) return false;
        return true;
    }
    static constexpr int last = last_radix<R...>();
};

using Row360 = FixedRadices<360, 8, 3, 15>;
using Row1800 = FixedRadices<1800, 8, 15, 15>;
using Row3600 = FixedRadices<3600, 16, 15, 15>;
using Row7200 = FixedRadices<7200, 8, 4, 15, 15>;
using Row14400 = FixedRadices<14400, 8, 8, 15, 15>;

template <typename... P>
inline int last_radix_of(int n_az, const RowPlan &pl) {
    int r = 0;
    ((r = P::is(n_az, pl) ? P::last : r), ...);
    return r;
}

// Order in which the row filter stores a row's spectrum: radix-major for the last radix returned (element i = q*(N/rk) + b
// holds digit-reversed position b*rk + q) by the compile-time plans, digit-reversed (0) by the run-time plan.  The filter
// takes a compile-time plan where this is not 0, and the readers of its spectra ask here.
inline int stored_radix(int n_az, const RowPlan &pl) {
    return last_radix_of<Row360, Row1800, Row3600, Row7200, Row14400>(n_az, pl);
}

}  // namespace rowfft
}  // namespace rosar
