// Geometry of one (row, aperture offset) of back-projection with nominal pulse positions, shared by the direct
// kernel (bpa.cu) and the frequency-domain one (bpa_fft.cu) (arXiv 2309.08038, Eqs. (2), (3), (8), (40)).
#pragma once

#include "rosar_internal.cuh"

namespace rosar {

// Offset d of row r, s = sin(pi*d/n_az): R_n - rho (no cancellation), bin x = r + (R_n - rho)/dR and
// alpha = max(0, cos(theta')), 1 where R_n = 0.
__device__ __forceinline__ void nominal_tap(float s, float R, float r0, float rho, float rf, float inv_dR, float &x,
                                            float &delta, float &alpha) {
    const float s2 = s * s;
    const float num = 4.f * R * r0 * s2;                // R_n^2 - rho^2
    const float Rn2 = fmaf(rho, rho, num);
    if (Rn2 > 0.f) {
        const float inv = rsqrtf(Rn2);
        const float Rn = Rn2 * inv;
        delta = __fdividef(num, Rn + rho);
        alpha = fmaxf(0.f, fmaf(-2.f * R, s2, rho) * inv);
    } else {
        delta = 0.f;
        alpha = 1.f;
    }
    x = fmaf(delta, inv_dR, rf);
}

// alpha * exp(-j*2*pi*(2*f_mid/c)*delta)
__device__ __forceinline__ float2 nominal_weight(float two_f_over_c, float delta, float alpha) {
    float ps, pc;
    sincospif(2.f * two_f_over_c * delta, &ps, &pc);
    return make_float2(alpha * pc, -alpha * ps);
}

// exp(-j*2*k_mid*rho) of the row, reduced in FP64
__device__ __forceinline__ float2 row_phase(const BpaParams &p, double rho) {
    double q = p.two_f_over_c_d * rho;
    q -= floor(q);
    double s, c;
    sincospi(2.0 * q, &s, &c);
    return make_float2((float)c, (float)-s);
}

// S at bin l, zero outside [0, L).  OVERLAPS: the kernel is launched to overlap the one that writes S, which is then not
// read by the non-coherent path (rows of the smallest images, read sample by sample: 5.8 us by that path, 6.2 without).
template <bool OVERLAPS = false>
__device__ __forceinline__ float2 read_bin(const float2 *__restrict__ S, int l, int L, size_t col, int n_az) {
    if (!(l >= 0 && l < L)) return make_float2(0.f, 0.f);
    return OVERLAPS ? __ldca(S + (size_t)l * n_az + col) : __ldg(S + (size_t)l * n_az + col);
}

// Sample at bin x of pulse (n mod n_az): from the staged rows [wlo, wtop) of its column (row pitch `pitch`) where they
// hold its bins, else through L2.
template <bool LINEAR>
__device__ __forceinline__ float2 sample_anywhere(const float2 *__restrict__ S, const float2 *col, int pitch, int wlo,
                                                  int wtop, float x, int L, int n_az, int n) {
    if (LINEAR) {
        const float fl = floorf(x);
        const int l0 = (int)fl;
        float2 s0, s1;
        if (l0 >= wlo && l0 + 1 < wtop) {
            s0 = col[(l0 - wlo) * pitch];
            s1 = col[(l0 + 1 - wlo) * pitch];
        } else {
            const int m = pmod(n, n_az);
            s0 = read_bin(S, l0, L, m, n_az);
            s1 = read_bin(S, l0 + 1, L, m, n_az);
        }
        return caxpy(x - fl, csub(s1, s0), s0);
    }
    const int l0 = (int)floorf(x + 0.5f);
    return (l0 >= wlo && l0 < wtop) ? col[(l0 - wlo) * pitch] : read_bin(S, l0, L, pmod(n, n_az), n_az);
}

}  // namespace rosar
