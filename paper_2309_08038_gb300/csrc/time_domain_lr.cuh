// Sizes and layout of the low-rank form of the time-domain paths (time_domain_lr.cu): the plan, the workspace, the
// transform lengths.
#pragma once

#include "rosar_internal.cuh"

namespace rosar {
namespace lr {

constexpr int MAX_PLANES = 32;
constexpr int MAX_LF = 2048;

// Planes of the interpolation of exp(-j t a), |t| <= 1, at Chebyshev nodes: its error is about
// 4 J_P(a) <= 4 (a/2)^P / P!, here at most 3e-6, reached at the ends of the samples only, where |t| = 1: under a
// window or not the image is within 1e-6 of the sums.
__host__ __device__ inline int planes_for(float a) {
    float term = 4.f;
    for (int P = 1; P <= MAX_PLANES; ++P) {
        term *= 0.5f * a / (float)P;
        if (P >= 2 && (float)P > 0.5f * a && term <= 3e-6f) return P;
    }
    return MAX_PLANES + 1;
}

// The residual bin positions eta = (rho/dR) Lf/L - l(r) of taps whose half angle has a sine of at most s_max lie in
// mid +- half: rho - r dR is at least 0 and at most its value 2 r0 s_max in row 0, and l(r) rounds r Lf/L.
struct Interval {
    float mid, half;
    int planes;
};
__host__ __device__ inline Interval residuals(float r0_over_dR, float s_max, int L, int Lf) {
    const float frac = Lf == L ? 0.f : 0.5f, stretch = (float)Lf / (float)L;
    const float lo = -frac - 1e-3f, hi = frac + 2.f * r0_over_dR * s_max * stretch + 1e-3f;
    Interval v;
    v.mid = 0.5f * (lo + hi);
    v.half = 0.5f * (hi - lo);
    v.planes = planes_for(3.14159265f * v.half / stretch);
    return v;
}

// Shape of one call; valid = 0 where the form does not apply.
struct Shape {
    int valid;
    int bpa;         // taps of back-projection, else of SAS
    int n_az, L, n_rng, K;
    int Lf;          // range transform length, a power of two >= L
    int N;           // azimuth transform length
    int pitch;       // row pitch of the spectra, a multiple of 16
    int fixed;       // compile-time plan of length N, else the run-time plan of n_az
    int off, len;    // element i < len of an azimuth row is pulse (i + off) mod n_az, the rest zero
    // byte offsets in the plan
    size_t w_at, offs_at, taps_at, h_at;
    // byte offsets in the workspace of a planned call
    size_t x_at, t_at, flags_at, ws_bytes;
    int flag_bytes;
    int cap;         // planes the plan has room for (set by the plan call)
    size_t h_plane;  // bytes of one plane of H
};

// First bytes of a plan: what it was made for.  The kernels of an image call compare it with the call's own shape, on
// which every address they form in the plan depends (a BPA plan's rows are padded otherwise than a SAS plan's): a plan
// of another kind or size, or something else, is not read any further and gives an image of NaN.
struct alignas(16) Header {
    int kind;        // kPlanTag + bpa
    int n_az, L, n_rng, K;
    int planes;
    float half;      // of the interval of eta
    int unused;
};
constexpr int kPlanTag = 0x6c725000;

Shape shape_of(bool bpa, int n_az, int L, int n_rng, int K);
// Planes a plan must have room for: one more than the host counts, whose float operations may round otherwise than
// the device's; offsets in device memory may reach half a turn.
int planes_bound(const TdParams &p, bool bpa, int K, int Lf);

}  // namespace lr
}  // namespace rosar
