// Scans of a batch as the kernels read them, and groups of scans that one launch covers: the range compression of all
// scans of one length L, the azimuth rows of all scans of one n_az (batch.cu, range_compress.cu, azimuth_rows.cu).
#pragma once

#include "rosar_internal.cuh"
#include "row_fft.cuh"

namespace rosar {

struct ScanDev {
    const float2 *raw;
    const float *win;
    const float2 *w;
    const int32_t *o;
    float2 *S;
    float2 *out;
    const float2 *H;          // frequency-domain plan [L][n_az], or null: gather tiles
    int o_row_stride, n_az, L, K;
    int range_tiles, az_tiles_per_row, P, vec_store;
    int fixed;                // compile-time plan of the row FFT (1: 1800, 2: 3600, 3: 7200 pulses), 0: run-time plan
    rowfft::RowPlan plan;
};

// CTA b of a launch is tile (or row) b - first[i] of scan order[i], the last i with first[i] <= b.
struct ScanGroup {
    const ScanDev *scans;
    const int *order, *first;
    int n;

    // run by whole warps
    __device__ __forceinline__ const ScanDev &find(int b, int &local) const {
        int c = 0;
        for (int i = threadIdx.x & 31; i < n; i += 32) c += __ldg(first + i) <= b;
        const int i = __reduce_add_sync(0xffffffffu, c) - 1;
        local = b - __ldg(first + i);
        return scans[__ldg(order + i)];
    }
};

// Launches over a group (total = CTAs: tiles of range_group_pulses(L) pulses of every scan, or rows).  With `prepare`
// they only set the kernels' shared-memory limits, which a capture does not take.
int range_group_pulses(int L);
rosar_status launch_range_group(int L, const ScanGroup &g, int total, cudaStream_t s, bool prepare);
rosar_status launch_azimuth_group(int n_az, const ScanGroup &g, int total, cudaStream_t s, bool prepare);

}  // namespace rosar
