// K3: range-compressed back-projection, the FFT+BPA comparison path
// (arXiv 2309.08038, Sec. III-D after Eq. (43) with w_BP; Eq. (14); Eqs. (2), (3), (8), (37), (40)).
//
//   out[r][theta] = sum_d alpha_n * exp(-j*2*k_mid*R_n) * S(R_n/dR, n),  n = (theta + d) mod n_az
//
// Pixel (r, theta) is at R = r0 + r*dR, angle 2*pi*theta/n_az; pulse n at radius
// r0 + dr[n] and angle 2*pi*n/n_az + dphi[n].  With rho = R - r0 (the pixel's slant
// range seen from the facing pulse, exactly r bins) the kernel evaluates
//   R_n^2 - rho^2 = dr*(r_n + r0 - 2R) + 4*R*r_n*sin^2(dphi_n/2)            (no cancellation)
//   delta = R_n - rho = (R_n^2 - rho^2)/(R_n + rho),   bin x = r + delta/dR,
//   cos(theta') = ((rho - dr) - 2*R*sin^2(dphi_n/2))/R_n,   alpha = max(0, cos(theta')),
//   exp(-j*2*k_mid*R_n) = exp(-j*2*k_mid*rho) * exp(-j*2*pi*(2*f_mid/c)*delta),
// so every float32 quantity is small and well conditioned; the per-row factor
// exp(-j*2*k_mid*rho) is computed once per CTA in FP64.  sin(dphi_n/2) is
// sin(pi*d/n_az)*cos(eps/2) + cos(pi*d/n_az)*sin(eps/2) from a per-d table and a
// per-pulse table, both staged in shared memory.
//
// With no pulse errors supplied (nominal geometry) every per-pulse quantity
// depends on (r, d) only; that kernel variant tabulates (x, alpha*phase) per d
// and the pixel loop is two gathers, an interpolation and a complex MAC.  It serves
// the calls too small or too long for the frequency-domain form (bpa_fft.cu).
//
// With supplied errors the fine phase exp(-j*2*pi*(2*f_mid/c)*delta) of every (pixel, pulse) is taken as
// sin/cos of the phase in turns first reduced exactly by whole turns to [-1/2, 1/2] (delta spans tens of cycles)
// and then evaluated by the hardware sine and cosine (about 1e-6 absolute error there), instead of the accurate
// sincospif's software range reduction and polynomials: the per-sample work is issue-bound FP32 and SFU.
// The interpolation mode is a template parameter.
//
// Grid: (azimuth tiles of 256 pixels, rows).  Once S is staged in shared memory the nominal kernel is bound by
// shared-memory bandwidth (two 8-byte window reads per sample) and the supplied-error kernel by FP32 + SFU issue.

#include <type_traits>

#include "bpa_geometry.cuh"

namespace rosar {
namespace {

constexpr int BPA_THREADS = 256;
constexpr int BPA_WR = 6;     // range rows of the staged S window
// aperture offsets staged per chunk: 512 with nominal geometry; 256 with supplied errors, whose per-pulse table
// makes a CTA's shared memory the occupancy limit (256: 6 CTAs per SM instead of 3)
template <bool NOMINAL> constexpr int bpa_dc() { return NOMINAL ? 512 : 256; }
template <bool NOMINAL> constexpr int bpa_wc() { return BPA_THREADS + bpa_dc<NOMINAL>(); }   // window columns (pulses)
template <bool NOMINAL> constexpr int bpa_smem() { return BPA_WR * bpa_wc<NOMINAL>() * 8; }

// Per chunk of offsets the bins a pixel of row r reads lie in a few rows near r (x = r + (R_n - rho)/dR, within a
// couple of bins over a +-30 degree aperture): a window of rows around the chunk's range of x and the pulses
// th0 + dc .. th0 + dc + BPA_WC are staged in shared memory once.  The range of x is the nominal one widened by
// the largest distance a supplied pulse position lies from its nominal one: R_n is a distance from the pixel, so it
// moves by at most |pos_n - pos_n,nominal| <= |dr_n| + 2*r0*|sin(eps_n/2)| (triangle inequality).  When that range,
// with a bin of margin below and two above, fits the window (always with nominal geometry; with supplied errors
// unless some pulse lies more than a bin or so off), every sample's bins are in it, rows outside [0, L) are staged
// as zeros, and the pixel loop reads the window with no check.  Otherwise the window is the nominal one and each
// sample whose bins fall outside it reads S through L2.
// max that keeps a NaN (fmaxf drops it): a NaN error bound must reach the window test and fail it
__device__ __forceinline__ float nanmax(float a, float b) { return (a > b || a != a) ? a : b; }

// exp(-j*2*pi*q) for |q| up to 2^22 turns: q reduced by whole turns (q - rint(q), exact) to [-1/2, 1/2], then
// the hardware sine and cosine of 2*pi times the remainder.
__device__ __forceinline__ float2 expmj2pi_turns(float q) {
    const float r = q - rintf(q);
    float sn, cs;
    __sincosf(6.28318530717959f * r, &sn, &cs);
    return make_float2(cs, -sn);
}

template <bool NOMINAL, bool LINEAR>
__global__ void __launch_bounds__(BPA_THREADS)
bpa_kernel(const float2 *__restrict__ S, BpaParams p, const float *__restrict__ dphi, const float *__restrict__ dr,
           int L, int n_az, int M_ap, float2 *__restrict__ out) {
    constexpr int BPA_DC = bpa_dc<NOMINAL>(), BPA_WC = bpa_wc<NOMINAL>();
    extern __shared__ float2 wsm[];                           // [BPA_WR][BPA_WC]
    __shared__ float4 dtab[BPA_DC];                           // NOMINAL: (x, a.re, a.im, -); else (sin, cos, x_nominal, -)
    // per pulse, with this CTA's row folded in: (cos(eps/2), sin(eps/2), dr*(r_n + r0 - 2R), 4*R*r_n), and
    // rho - dr (the numerator of cos(theta') before its sin^2 term)
    __shared__ float4 ptab[NOMINAL ? 1 : BPA_THREADS + BPA_DC];
    __shared__ float pal[NOMINAL ? 1 : BPA_THREADS + BPA_DC];
    __shared__ float2 rowph;
    __shared__ float red_lo[BPA_THREADS / 32], red_hi[BPA_THREADS / 32], red_e[BPA_THREADS / 32];

    const int r = blockIdx.y;
    const int th0 = blockIdx.x * BPA_THREADS;
    const int th = th0 + threadIdx.x;
    const float rf = (float)r;
    const double rho_d = r * p.dR;
    const float rho = (float)rho_d;
    const float R = (float)(p.r0 + rho_d);
    const float r0 = (float)p.r0;
    if (threadIdx.x == 0) rowph = row_phase(p, rho_d);

    float2 acc = make_float2(0.f, 0.f);
    const int d_beg = -(M_ap / 2), d_end = M_ap - M_ap / 2;
    // chunks of equal size (at most BPA_DC offsets): M = 600 with BPA_DC = 256 gives 3 chunks of 200
    const int n_chunks = (M_ap + BPA_DC - 1) / BPA_DC;
    const int step = (M_ap + n_chunks - 1) / n_chunks;
    for (int dc = d_beg; dc < d_end; dc += step) {
        const int nd = min(step, d_end - dc);
        __syncthreads();
        float xlo = 1e30f, xhi = -1e30f;
        for (int i = threadIdx.x; i < nd; i += BPA_THREADS) {
            float s, c;
            sincospif((float)(dc + i) / (float)n_az, &s, &c);   // sin/cos(pi*d/n_az)
            float x, delta, alpha;
            nominal_tap(s, R, r0, rho, rf, p.inv_dR, x, delta, alpha);
            xlo = fminf(xlo, x);
            xhi = fmaxf(xhi, x);
            if (NOMINAL) {
                const float2 a = nominal_weight(p.two_f_over_c, delta, alpha);
                dtab[i] = make_float4(x, a.x, a.y, 0.f);
            } else {
                dtab[i] = make_float4(s, c, x, 0.f);
            }
        }
        float emax = 0.f;   // largest pulse position error of the chunk, in bins
        if (!NOMINAL) {
            for (int i = threadIdx.x; i < BPA_THREADS + nd; i += BPA_THREADS) {
                const int n = pmod(th0 + dc + i, n_az);
                const float e = dphi ? __ldg(dphi + n) : 0.f;
                float se, ce;
                sincosf(0.5f * e, &se, &ce);
                const float drn = dr ? __ldg(dr + n) : 0.f;
                const float rn = r0 + drn;
                ptab[i] = make_float4(ce, se, drn * (rn + r0 - 2.f * R), 4.f * R * rn);
                pal[i] = rho - drn;
                emax = nanmax(emax, fmaf(2.f * r0, fabsf(se), fabsf(drn)) * p.inv_dR);
            }
        }
        // the chunk's x range and error bound over the CTA
#pragma unroll
        for (int sft = 16; sft > 0; sft >>= 1) {
            xlo = fminf(xlo, __shfl_xor_sync(0xffffffffu, xlo, sft));
            xhi = fmaxf(xhi, __shfl_xor_sync(0xffffffffu, xhi, sft));
            if (!NOMINAL) emax = nanmax(emax, __shfl_xor_sync(0xffffffffu, emax, sft));
        }
        if ((threadIdx.x & 31) == 0) {
            red_lo[threadIdx.x >> 5] = xlo;
            red_hi[threadIdx.x >> 5] = xhi;
            red_e[threadIdx.x >> 5] = emax;
        }
        __syncthreads();
        xlo = red_lo[0];
        xhi = red_hi[0];
        emax = red_e[0];
        for (int i = 1; i < BPA_THREADS / 32; ++i) {
            xlo = fminf(xlo, red_lo[i]);
            xhi = fmaxf(xhi, red_hi[i]);
            if (!NOMINAL) emax = nanmax(emax, red_e[i]);
        }
        // covered: every sample's x lies in [xlo - emax, xhi + emax] (up to rounding, far below the margins), so
        // its bins floor(x) and floor(x) + 1 lie in rows [floor(xlo - emax) - 1, floor(xhi + emax) + 2]
        const float flo = floorf(xlo - emax), fhi = floorf(xhi + emax);
        const bool covered = fhi - flo <= (float)(BPA_WR - 4) && flo > -1e6f && fhi < 1e6f;   // false for NaN
        int wlo, nrow;
        if (covered) {
            wlo = (int)flo - 1;
            nrow = (int)(fhi - flo) + 4;
        } else {
            wlo = max(0, (int)floorf(xlo) - 1);
            nrow = min(BPA_WR, min(L - 1, (int)floorf(xhi) + 2) - wlo + 1);
        }
        const int wtop = wlo + nrow;                                  // rows [wlo, wtop) staged
        const int ncol = BPA_THREADS + nd;
        for (int e = threadIdx.x; e < nrow * ncol; e += BPA_THREADS) {
            const int rr = e / ncol, cc = e - rr * ncol;
            const int n = pmod(th0 + dc + cc, n_az);
            const int l = wlo + rr;
            wsm[rr * BPA_WC + cc] = (l >= 0 && l < L) ? __ldg(S + (size_t)l * n_az + n) : make_float2(0.f, 0.f);
        }
        __syncthreads();
        if (th >= n_az) continue;
        // bin x and weight alpha * exp(-j*2*pi*(2 f/c)*delta) of offset dc + i for this thread's pixel
        auto sample = [&](int i, auto checked, float &x, float2 &a) {
            const float4 t = dtab[i];
            if (NOMINAL) {
                x = t.x;
                a = make_float2(t.y, t.z);
            } else {
                const float4 pp = ptab[threadIdx.x + i];
                const float sh = fmaf(t.x, pp.x, t.y * pp.y);            // sin((pi*d/n_az) + eps/2)
                const float s2 = sh * sh;
                const float num = fmaf(pp.w, s2, pp.z);                  // R_n^2 - rho^2
                const float along = pal[threadIdx.x + i];                // R - r_n
                // off the window a pulse may pass close to the pixel, where rho^2 + num would cancel
                const float Rn2 = decltype(checked)::value ? fmaf(pp.w, s2, along * along) : fmaf(rho, rho, num);
                // branch-free: R_n = 0 (the facing pulse of row 0, or a supplied position on the pixel) gives
                // delta = num / rho = -rho exactly, or 0 when rho = 0 too, and alpha = 1 by the select
                const float inv = rsqrtf(fmaxf(Rn2, 1e-30f));
                const float Rn = Rn2 * inv;
                const float delta = __fdividef(num, fmaxf(Rn + rho, 1e-30f));
                // alpha = max(0, cos(theta')), cos(theta') <= 1: one saturating multiply
                const float a0 = __saturatef(fmaf(-2.f * R, s2, along) * inv);
                const float alpha = Rn2 > 0.f ? a0 : 1.f;
                x = fmaf(delta, p.inv_dR, rf);
                a = cscale(expmj2pi_turns(p.two_f_over_c * delta), alpha);
            }
        };
        if (covered) {
            // in-window by construction; the unsigned clamp keeps even a NaN x's read inside the staged rows
            const float2 *colp = wsm + threadIdx.x;
#pragma unroll 4
            for (int i = 0; i < nd; ++i) {
                float x;
                float2 a;
                sample(i, std::false_type{}, x, a);
                float2 sv;
                if (LINEAR) {
                    const float fl = floorf(x);
                    const unsigned rel = min((unsigned)(int)fl - (unsigned)wlo, (unsigned)(nrow - 2));
                    const float2 s0 = colp[rel * BPA_WC + i], s1 = colp[(rel + 1) * BPA_WC + i];
                    sv = caxpy(x - fl, csub(s1, s0), s0);
                } else {
                    const unsigned rel = min((unsigned)(int)floorf(x + 0.5f) - (unsigned)wlo, (unsigned)(nrow - 1));
                    sv = colp[rel * BPA_WC + i];
                }
                cmac(acc, a, sv);
            }
        } else {
#pragma unroll 4
            for (int i = 0; i < nd; ++i) {
                float x;
                float2 a;
                sample(i, std::true_type{}, x, a);
                const int col = threadIdx.x + i;
                float2 sv;
                if (LINEAR) {
                    const float fl = floorf(x);
                    const int l0 = (int)fl;
                    const float f = x - fl;
                    float2 s0, s1;
                    if (l0 >= wlo && l0 + 1 < wtop) {
                        s0 = wsm[(l0 - wlo) * BPA_WC + col];
                        s1 = wsm[(l0 + 1 - wlo) * BPA_WC + col];
                    } else {                  // off the staged window: pulse (th + d) mod n_az through L2
                        const int n = pmod(th + dc + i, n_az);
                        s0 = read_bin(S, l0, L, n, n_az);
                        s1 = read_bin(S, l0 + 1, L, n, n_az);
                    }
                    sv = caxpy(f, csub(s1, s0), s0);
                } else {
                    const int l0 = (int)floorf(x + 0.5f);
                    sv = (l0 >= wlo && l0 < wtop) ? wsm[(l0 - wlo) * BPA_WC + col]
                                                  : read_bin(S, l0, L, pmod(th + dc + i, n_az), n_az);
                }
                cmac(acc, a, sv);
            }
        }
    }
    if (th < n_az) out[(size_t)r * n_az + th] = cmul(rowph, acc);
}

// --------------------------------------------------------------------- supplied errors, two rows a thread --
// For grids that fill the SMs with half the threads.  Two rows (r, r + 1) a thread: the angle between pixel and pulse is
// the same in both, so the sine of its half (sh), 4 r_n sh^2 - 2 dr_n (u) and cos of the angle are taken once, and what
// depends on the row,
//   R_n^2 - rho^2 = R u + dr_n (r_n + r0),   rho - dr_n - 2 R sh^2 = R (1 - 2 sh^2) - r_n,
// through delta, the bin and the phase, runs as packed FP32x2 instructions over the two.  The whole part of the
// bin and of the phase in turns come from an addition that rounds to an integer in the low mantissa bits (no
// conversions, which share the SFU's slot with rsqrt, reciprocal, sine and cosine).  70 instructions for the two
// samples where a loop over one row took 56 for each: 3600 x 256, M = 600: 972 -> 722 us.  Bound by issue (71 %) and
// the FMA pipe (64 %, a packed instruction taking it twice).
//
// The window of S covers both rows: the nominal range of x over the chunk's offsets in row r, up to row r + 1's,
// widened by the largest distance a supplied pulse position lies from its nominal one: R_n is a distance from the
// pixel, so it moves by at most |pos_n - pos_n,nominal| <= |dr_n| + 2*r0*|sin(eps_n/2)| (triangle inequality).  When it
// fits, and the rows lie farther out than any pulse (R_n > 0), the loop needs no check; otherwise (row 0, pulses a
// bin and more off) each sample is taken on its own.
//
// Linear interpolation stages S as cells: a bin and its difference to the next, so that a sample is one 16-byte load.
constexpr int ERR_WR = 7;                     // rows of the staged window (one fewer cells)
constexpr int ERR_DC = 256;                   // aperture offsets per chunk
// shared memory of a chunk of `step` offsets: the window, per-pulse (16 + 4 bytes) and per-offset (8 bytes) tables
__host__ __device__ constexpr int err_window(int step) { return (ERR_WR - 1) * (BPA_THREADS + step) * 16; }
__host__ __device__ constexpr int err_smem(int step) {
    return err_window(step) + (BPA_THREADS + step) * 20 + step * 8 + 16;
}
inline int err_step(int M_ap) {               // equal chunks: M = 600 gives 3 of 200
    const int n = (M_ap + ERR_DC - 1) / ERR_DC;
    return (M_ap + n - 1) / n;
}
constexpr float kRound = 12582912.f;          // 1.5 * 2^23: x + kRound holds rint(x) in its low bits, |x| < 2^22

// The hardware approximations without the scaling that keeps subnormal arguments (none occur: R_n is over 1e-5 m).
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float sin_approx(float x) {
    float y;
    asm("sin.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float cos_approx(float x) {
    float y;
    asm("cos.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <bool LINEAR>
__global__ void __launch_bounds__(BPA_THREADS)
bpa_errors2_kernel(const float2 *__restrict__ S, BpaParams p, const float *__restrict__ dphi,
                  const float *__restrict__ dr, int L, int n_rng, int n_az, int M_ap, int step, float2 *__restrict__ out) {
    extern __shared__ __align__(16) float4 esm[];
    const int wc = BPA_THREADS + step;                        // window pitch: the pulses of a chunk
    float4 *cells = esm;                                      // [ERR_WR - 1][wc] (S, next bin's S - S), or
    float2 *wsm = reinterpret_cast<float2 *>(esm);            // [ERR_WR][wc] S itself
    float4 *ptab = esm + (ERR_WR - 1) * wc;                   // per pulse: cos(eps/2), sin(eps/2), r_n, -2 dr_n
    float2 *dtab = reinterpret_cast<float2 *>(ptab + wc);     // sin, cos(pi*d/n_az)
    float *pv = reinterpret_cast<float *>(dtab + step);       // dr_n (r_n + r0)
    __shared__ float2 rowph[2];
    __shared__ float red_lo[BPA_THREADS / 32], red_hi[BPA_THREADS / 32], red_e[BPA_THREADS / 32],
        red_d[BPA_THREADS / 32];

    const int r = 2 * blockIdx.y;
    const int th0 = blockIdx.x * BPA_THREADS;
    const int th = th0 + threadIdx.x;
    const double rho_d = r * p.dR, rho1_d = (r + 1) * p.dR;
    const float2 rho = make_float2((float)rho_d, (float)rho1_d);
    const float2 rho2 = make_float2((float)(rho_d * rho_d), (float)(rho1_d * rho1_d));
    const float2 R = make_float2((float)(p.r0 + rho_d), (float)(p.r0 + rho1_d));
    const float r0 = (float)p.r0;
    if (threadIdx.x < 2) rowph[threadIdx.x] = row_phase(p, threadIdx.x == 0 ? rho_d : rho1_d);

    float2 acc0 = make_float2(0.f, 0.f), acc1 = make_float2(0.f, 0.f);
    const int d_beg = -(M_ap / 2), d_end = M_ap - M_ap / 2;
    for (int dc = d_beg; dc < d_end; dc += step) {
        const int nd = min(step, d_end - dc);
        __syncthreads();
        float xlo = 1e30f, xhi = -1e30f;
        for (int i = threadIdx.x; i < nd; i += BPA_THREADS) {
            float s, c, x, delta, alpha;
            sincospif((float)(dc + i) / (float)n_az, &s, &c);   // sin/cos(pi*d/n_az)
            nominal_tap(s, R.x, r0, rho.x, (float)r, p.inv_dR, x, delta, alpha);
            xlo = fminf(xlo, x);
            nominal_tap(s, R.y, r0, rho.y, (float)(r + 1), p.inv_dR, x, delta, alpha);
            xhi = fmaxf(xhi, x);
            nominal_tap(s, R.x, r0, rho.x, (float)r, p.inv_dR, x, delta, alpha);
            xhi = fmaxf(xhi, x);
            dtab[i] = make_float2(s, c);
        }
        float emax = 0.f, dmax = 0.f;   // largest pulse position error of the chunk in bins, largest |dr|
        for (int i = threadIdx.x; i < BPA_THREADS + nd; i += BPA_THREADS) {
            const int n = pmod(th0 + dc + i, n_az);
            const float e = dphi ? __ldg(dphi + n) : 0.f;
            float se, ce;
            sincosf(0.5f * e, &se, &ce);
            const float drn = dr ? __ldg(dr + n) : 0.f;
            const float rn = r0 + drn;
            ptab[i] = make_float4(ce, se, rn, -2.f * drn);
            pv[i] = drn * (rn + r0);
            emax = nanmax(emax, fmaf(2.f * r0, fabsf(se), fabsf(drn)) * p.inv_dR);
            dmax = nanmax(dmax, fabsf(drn));
        }
        // the chunk's x range and error bounds over the CTA
#pragma unroll
        for (int sft = 16; sft > 0; sft >>= 1) {
            xlo = fminf(xlo, __shfl_xor_sync(0xffffffffu, xlo, sft));
            xhi = fmaxf(xhi, __shfl_xor_sync(0xffffffffu, xhi, sft));
            emax = nanmax(emax, __shfl_xor_sync(0xffffffffu, emax, sft));
            dmax = nanmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, sft));
        }
        if ((threadIdx.x & 31) == 0) {
            red_lo[threadIdx.x >> 5] = xlo;
            red_hi[threadIdx.x >> 5] = xhi;
            red_e[threadIdx.x >> 5] = emax;
            red_d[threadIdx.x >> 5] = dmax;
        }
        __syncthreads();
        xlo = red_lo[0];
        xhi = red_hi[0];
        emax = red_e[0];
        dmax = red_d[0];
        for (int i = 1; i < BPA_THREADS / 32; ++i) {
            xlo = fminf(xlo, red_lo[i]);
            xhi = fmaxf(xhi, red_hi[i]);
            emax = nanmax(emax, red_e[i]);
            dmax = nanmax(dmax, red_d[i]);
        }
        // covered: every sample's x lies in [xlo - emax, xhi + emax] (up to rounding, far below the margins), so its
        // bins floor(x) and floor(x) + 1 lie in rows [floor(xlo - emax) - 1, floor(xhi + emax) + 2]; and R_n > 0
        const float flo = floorf(xlo - emax), fhi = floorf(xhi + emax);
        const bool covered = fhi - flo <= (float)(ERR_WR - 4) && flo > -1e6f && fhi < 1e6f &&   // false for NaN
                             rho.x > 1.001f * dmax + 1e-4f * R.x;
        int wlo, nrow;
        if (covered) {
            wlo = (int)flo - 1;
            nrow = (int)(fhi - flo) + 4;
        } else {
            wlo = max(0, (int)floorf(xlo) - 1);
            nrow = min(ERR_WR, min(L - 1, (int)floorf(xhi) + 2) - wlo + 1);
        }
        const int wtop = wlo + nrow;                                  // rows [wlo, wtop) staged
        const int ncol = BPA_THREADS + nd;
        const bool as_cells = LINEAR && covered;
        for (int e = threadIdx.x; e < (as_cells ? nrow - 1 : nrow) * ncol; e += BPA_THREADS) {
            const int rr = e / ncol, cc = e - rr * ncol;
            const int n = pmod(th0 + dc + cc, n_az);
            const int l = wlo + rr;
            const float2 a = read_bin(S, l, L, n, n_az);
            if (as_cells) {
                const float2 dif = csub(read_bin(S, l + 1, L, n, n_az), a);
                cells[rr * wc + cc] = make_float4(a.x, a.y, dif.x, dif.y);
            } else {
                wsm[rr * wc + cc] = a;
            }
        }
        __syncthreads();
        if (th >= n_az) continue;
        if (covered) {
            const float2 *colp = wsm + threadIdx.x;
            const float4 *cellp = cells + threadIdx.x;
            const float2 k2 = make_float2(p.two_f_over_c, p.two_f_over_c), inv2 = make_float2(p.inv_dR, p.inv_dR);
            const float2 one_m = make_float2(-1.f, -1.f), rnd = make_float2(kRound, kRound), rnd_m = make_float2(-kRound, -kRound);
            const float2 turn = make_float2(6.28318530717959f, 6.28318530717959f);
            const unsigned top = (unsigned)(nrow - (LINEAR ? 2 : 1));
            const unsigned base0 = (unsigned)(r - wlo) - (unsigned)__float_as_int(kRound), base1 = base0 + 1u;
            const float2 rf = make_float2((float)r, (float)(r + 1));
#pragma unroll 2
            for (int i = 0; i < nd; ++i) {
                const float2 t = dtab[i];
                const float4 pp = ptab[threadIdx.x + i];
                const float v = pv[threadIdx.x + i];
                const float sh = fmaf(t.x, pp.x, t.y * pp.y);            // sin((pi*d/n_az) + eps/2)
                const float s2 = sh * sh;
                const float u = fmaf(4.f * pp.z, s2, pp.w), c2 = fmaf(-2.f, s2, 1.f);
                const float2 num = __ffma2_rn(R, make_float2(u, u), make_float2(v, v));       // R_n^2 - rho^2
                const float2 Rn2 = __fadd2_rn(rho2, num);
                const float2 inv = make_float2(rsqrt_approx(Rn2.x), rsqrt_approx(Rn2.y));
                const float2 sum = __ffma2_rn(Rn2, inv, rho);                                 // R_n + rho
                const float2 delta = __fmul2_rn(num, make_float2(rcp_approx(sum.x), rcp_approx(sum.y)));
                // alpha = max(0, cos(theta')), cos(theta') <= 1: one saturating multiply
                const float2 an = __ffma2_rn(R, make_float2(c2, c2), make_float2(-pp.z, -pp.z));
                const float al0 = __saturatef(an.x * inv.x), al1 = __saturatef(an.y * inv.y);
                // phase in turns less its whole turns, rounded once
                const float2 whole = __fadd2_rn(__ffma2_rn(delta, k2, rnd), rnd_m);
                const float2 frac = __ffma2_rn(delta, k2, __fmul2_rn(whole, one_m));
                const float2 ang = __fmul2_rn(frac, turn);
                const float sn0 = sin_approx(ang.x), cs0 = cos_approx(ang.x), sn1 = sin_approx(ang.y), cs1 = cos_approx(ang.y);
                float2 sv0, sv1;
                if (LINEAR) {
                    // the cell is the integer nearest to the bin offset from the row less 1/2 (at an integer offset the
                    // even one of two cells that meet there)
                    const float2 xm = __ffma2_rn(delta, inv2, make_float2(-0.5f, -0.5f));
                    const float2 mi = __fadd2_rn(xm, rnd);
                    const float2 f = __fadd2_rn(__ffma2_rn(__fadd2_rn(mi, rnd_m), one_m, xm), make_float2(0.5f, 0.5f));
                    // in-window by construction; the unsigned clamp keeps even a NaN's read inside the staged rows
                    const float4 q0 = cellp[min((unsigned)__float_as_int(mi.x) + base0, top) * wc + i];
                    const float4 q1 = cellp[min((unsigned)__float_as_int(mi.y) + base1, top) * wc + i];
                    sv0 = caxpy(f.x, make_float2(q0.z, q0.w), make_float2(q0.x, q0.y));
                    sv1 = caxpy(f.y, make_float2(q1.z, q1.w), make_float2(q1.x, q1.y));
                } else {
                    const float2 x = __ffma2_rn(delta, inv2, rf);
                    sv0 = colp[min((unsigned)(int)floorf(x.x + 0.5f) - (unsigned)wlo, top) * wc + i];
                    sv1 = colp[min((unsigned)(int)floorf(x.y + 0.5f) - (unsigned)wlo, top) * wc + i];
                }
                cmac(acc0, make_float2(al0 * cs0, -al0 * sn0), sv0);
                cmac(acc1, make_float2(al1 * cs1, -al1 * sn1), sv1);
            }
        } else {
            for (int i = 0; i < nd; ++i) {
                const float2 t = dtab[i];
                const float4 pp = ptab[threadIdx.x + i];
                const float sh = fmaf(t.x, pp.x, t.y * pp.y), s2 = sh * sh, drn = -0.5f * pp.w;
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const float Rb = b ? R.y : R.x, rhob = b ? rho.y : rho.x;
                    const float num = fmaf(4.f * Rb * pp.z, s2, drn * (pp.z + r0 - 2.f * Rb));
                    // not rho^2 + num: a pulse that passes close to the pixel would cancel them
                    const float along = rhob - drn;                       // R - r_n
                    const float Rn2 = fmaf(4.f * Rb * pp.z, s2, along * along);
                    // branch-free: R_n = 0 (the facing pulse of row 0, or a supplied position on the pixel) gives
                    // delta = num / rho = -rho exactly, or 0 when rho = 0 too, and alpha = 1 by the select
                    const float inv = rsqrtf(fmaxf(Rn2, 1e-30f));
                    const float Rn = Rn2 * inv;
                    const float delta = __fdividef(num, fmaxf(Rn + rhob, 1e-30f));
                    const float a0 = __saturatef(fmaf(-2.f * Rb, s2, along) * inv);
                    const float alpha = Rn2 > 0.f ? a0 : 1.f;
                    const float x = fmaf(delta, p.inv_dR, (float)(r + b));
                    const float2 sv = sample_anywhere<LINEAR>(S, wsm + threadIdx.x + i, wc, wlo, wtop, x, L, n_az,
                                                              th + dc + i);
                    cmac(b ? acc1 : acc0, cscale(expmj2pi_turns(p.two_f_over_c * delta), alpha), sv);
                }
            }
        }
    }
    if (th < n_az) {
        out[(size_t)r * n_az + th] = cmul(rowph[0], acc0);
        if (r + 1 < n_rng) out[(size_t)(r + 1) * n_az + th] = cmul(rowph[1], acc1);
    }
}

// Whether the two-row kernel's window holds the bins of most chunks of offsets, in the middle row and with pulses a tenth
// of a bin off: a chunk that it does not hold is summed sample by sample, at about half the rate of the one-row kernel,
// whose window is a bin wider.  Three chunks in four are enough.  Half a ring, where the outer chunks span three bins:
// 1800 x 256, M = 900 (two of four held): 970 us against the one-row kernel's 890; 2500 x 256, M = 1250 (three of five)
// 1514 and 1499; 1031 x 256, M = 340 (none) 348 and 271; 3600 x 100, M = 1800 (all) 909 and 1184; 1800 x 256, M = 594
// (all) 401 and 518.
bool pairs_window_holds(const BpaParams &p, int n_rng, int n_az, int M_ap) {
    const int step = err_step(M_ap), chunks = (M_ap + step - 1) / step;
    if (chunks > 256) return true;                            // of a degree each
    const double rho = 0.5 * n_rng * p.dR, R = p.r0 + rho;
    auto bin = [&](int d) {                                   // of offset d from the row
        const double s = sin(3.14159265358979323846 * d / n_az);
        return (sqrt(rho * rho + 4.0 * R * p.r0 * s * s) - rho) / p.dR;
    };
    int held = 0;
    for (int i = 0; i < chunks; ++i) {
        const int d0 = -(M_ap / 2) + i * step, d1 = min(d0 + step, M_ap - M_ap / 2) - 1;
        const double a = bin(d0), b = bin(d1), lo = d0 < 0 && d1 > 0 ? 0.0 : fmin(a, b);
        held += floor(fmax(a, b) + 0.1) + 1.0 - floor(lo - 0.1) <= (double)(ERR_WR - 4);
    }
    return 4 * held >= 3 * chunks;
}

}  // namespace

rosar_status launch_bpa(const float2 *S, const BpaParams &p, const float *dphi, const float *dr, int L, int n_rng,
                        int n_az, int M_ap, int interp, float2 *out, cudaStream_t s) {
    if (n_rng > 65535) return set_error(ROSAR_ERR_UNSUPPORTED, "bpa: n_rng=%d exceeds 65535", n_rng);
    const bool nominal = dphi == nullptr && dr == nullptr;
    if (nominal && bpa_fft_applies(p, n_rng, n_az, M_ap))
        return launch_bpa_fft(S, p, L, n_rng, n_az, M_ap, interp, out, s);
    // Two rows a thread from a full residency of those CTAs on (4 an SM): 2000 x 256, M = 330 (1024 CTAs): 311 -> 226
    // us; 1500 x 256, M = 250 (768): 181 -> 147; 1000 x 256, M = 160 (512): 80.6 and 81.7.  Fewer leave warps out and
    // make row 0, whose samples are taken one by one, the last to end: 512 x 128, M = 79: 18 against 32 us.
    const int tiles = (n_az + BPA_THREADS - 1) / BPA_THREADS, pairs = (n_rng + 1) / 2;
    if (!nominal && (long long)tiles * pairs >= 608 && pairs_window_holds(p, n_rng, n_az, M_ap)) {
        static int done2[2][kMaxDevices] = {};
        const int step = err_step(M_ap), smem = err_smem(step);
        const auto kernel = interp ? bpa_errors2_kernel<true> : bpa_errors2_kernel<false>;
        rosar_status st = ensure_smem((const void *)kernel, smem, done2[interp ? 1 : 0], "bpa");
        if (st != ROSAR_OK) return st;
        kernel<<<dim3(tiles, pairs), BPA_THREADS, smem, s>>>(S, p, dphi, dr, L, n_rng, n_az, M_ap, step, out);
        return check_launch("bpa");
    }
    dim3 grid((n_az + BPA_THREADS - 1) / BPA_THREADS, n_rng);
    static int done[4][kMaxDevices] = {};
    const int v = (nominal ? 0 : 2) + (interp ? 1 : 0);
    static const void *const ks[4] = {(const void *)bpa_kernel<true, false>, (const void *)bpa_kernel<true, true>,
                                      (const void *)bpa_kernel<false, false>, (const void *)bpa_kernel<false, true>};
    const int smem = nominal ? bpa_smem<true>() : bpa_smem<false>();
    rosar_status st = ensure_smem(ks[v], smem, done[v], "bpa");
    if (st != ROSAR_OK) return st;
    switch (v) {
        case 0: bpa_kernel<true, false><<<grid, BPA_THREADS, smem, s>>>(S, p, dphi, dr, L, n_az, M_ap, out); break;
        case 1: bpa_kernel<true, true><<<grid, BPA_THREADS, smem, s>>>(S, p, dphi, dr, L, n_az, M_ap, out); break;
        case 2: bpa_kernel<false, false><<<grid, BPA_THREADS, smem, s>>>(S, p, dphi, dr, L, n_az, M_ap, out); break;
        default: bpa_kernel<false, true><<<grid, BPA_THREADS, smem, s>>>(S, p, dphi, dr, L, n_az, M_ap, out); break;
    }
    return check_launch("bpa");
}

}  // namespace rosar
