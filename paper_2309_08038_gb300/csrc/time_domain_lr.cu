// Time-domain BPA and SAS (arXiv 2309.08038, Eq. (14); Algorithm 2 with W_SA) by transforms.
//
//   out[r][theta] = sum_k c[r][k] sum_m win[m] exp(-j 2 pi y[r][k] (m - m_ref)/Lf) raw[(theta + o_k) mod n_az][m]
//
// with y = (rho/dR) Lf/L the tap's slant range in bins of a range transform of length Lf >= L.  As a product over
// (tap, sample) this is the dense contraction of time_domain.cu: K L multiply-adds a pixel.  But y is close to the
// row: y = l(r) + eta, l(r) = round(r Lf/L), eta within a bin or two, so exp(-j 2 pi eta u), |u| <= 1/2, is smooth
// in eta and interpolated to float32 accuracy from its values at P Chebyshev nodes eta_q (P = 13 at eta in [0, 2.1]):
//
//   out[r] = sum_q sum_k c'[r][k] ell_q(eta[r][k]) S_q[r][. + o_k],
//   S_q[r][n] = sum_m (win[m] exp(-j 2 pi eta_q (m - mid)/Lf)) exp(-j 2 pi l(r) m/Lf) raw[n][m],
//
// P range transforms under P modulated windows, each followed by a circular azimuth filter.  The azimuth transform
// acts on n, the range transform on m: they commute, and the azimuth transform is taken once, of the raw samples.
//
//   plan      lr_taps_kernel     nodes, windows and the taps (c' 1/N, eta, position), FP64 geometry
//             lr_plan_*          H_q[r] = transform of the taps times ell_q
//   per scan  lr_turn_kernel     raw [n_az][L] -> [L][n_az]
//             lr_forward_*       azimuth transform of every sample's row
//             lr_combine_kernel  per azimuth frequency: P range transforms of one register-resident column, each
//                                times H_q, summed
//             lr_inverse_*       inverse azimuth transform of every row of the image
//
// P range transforms, one forward and one inverse azimuth transform a scan; the plan's planes H are the largest
// array read (P 8 bytes a pixel).  The azimuth length N is n_az where that has a plan (circular filter), else a
// plan length with room for the pulses the aperture wraps to.
//
// 3600 x 256, M = 600: planned 48 us (3130 on the tensor cores), plan and image 105 (3867); SAS with K = 64: 48 (437)
// and 95 (630).  Of the 48: turn 4, forward 6, combine 26, inverse 8, the rest hand-overs.  The relative L2 error is
// 8e-7 where the bf16-split contraction has 1.5e-5.
//
// A transform would spread a sample that is not finite, or so large that its rounding is, over the image.  The direct
// sums keep it to the pixels that read the pulse, and so does this: lr_turn_kernel zeroes such samples and marks their
// pulse, and lr_inverse_* adds their terms to the pixels whose aperture holds it (NaN where one is not finite).  Smaller
// samples go through the transforms: each leaves float32 rounding of its own size in every pixel.

#include <math.h>
#include <stddef.h>

#include "row_fft.cuh"
#include "time_domain_lr.cuh"

namespace rosar {
namespace {

using namespace rowfft;
using lr::Header;
using lr::MAX_PLANES;
using lr::Shape;

// ------------------------------------------------------------------------------------------- plan --

constexpr int TAPS_THREADS = 256;
constexpr int TAPS_ROWS = 8, TAPS_COLS = 64;   // per CTA: an offset's sine serves the CTA's rows

__device__ __forceinline__ int canonical(int o, int n) {
    const int c = pmod(o, n);
    return c > n / 2 ? c - n : c;
}

// exp(+j*2*pi*q) of a phase in cycles, reduced by whole turns in FP64
__device__ __forceinline__ float2 turns(double q) {
    q -= rint(q);
    float s, c;
    sincospif(2.f * (float)q, &s, &c);
    return make_float2(c, s);
}

// Planes of the plan, or 0 where it was not made for a call of this shape; after the grid-dependency wait, and not by the
// non-coherent path (the kernel may overlap the one that writes the plan).
__device__ __forceinline__ int plan_planes(const uint8_t *plan, const Shape &sh) {
    const int4 a = __ldcg(reinterpret_cast<const int4 *>(plan)), b = __ldcg(reinterpret_cast<const int4 *>(plan) + 1);
    static_assert(offsetof(Header, K) == 16 && offsetof(Header, planes) == 20 && sizeof(Header) == 32, "two vectors");
    const bool same = a.x == lr::kPlanTag + sh.bpa && a.y == sh.n_az && a.z == sh.L && a.w == sh.n_rng && b.x == sh.K;
    return same && b.y >= 0 && b.y <= MAX_PLANES ? b.y : 0;
}

__device__ __forceinline__ float cheb_node(int q, int P) { return cospif((float)(2 * q + 1) / (float)(2 * P)); }

// Taps of TAPS_ROWS rows x TAPS_COLS offsets: (c'.re, c'.im, t, position), c' with the row's phase
// exp(j 2 pi l mid/Lf), the reference sample's phase and 1/N, t = (eta - eta_mid)/eta_half.  The CTAs also share the
// windows, CTA (0, 0) writes the header and the CTAs of the first rows the canonical offsets.  FP64 as the direct
// forms (the two-way phase reaches 1e5 rad), at a rate of two operations a cycle and SM what bounds it: 14 a tap,
// the square root refined from the float one, what depends on the row or the offset alone taken once per CTA.
template <bool BPA>
__global__ void __launch_bounds__(TAPS_THREADS)
lr_taps_kernel(const float *__restrict__ win, const float2 *__restrict__ w, const int32_t *__restrict__ o, TdParams p,
               Shape sh, uint8_t *__restrict__ plan) {
    __shared__ int s_max;
    __shared__ lr::Interval s_iv;
    __shared__ double s2[TAPS_COLS];
    __shared__ int off_c[TAPS_COLS];
    __shared__ double row_rd[TAPS_ROWS], row_rd2[TAPS_ROWS], row_2R[TAPS_ROWS], row_c4[TAPS_ROWS], row_q[TAPS_ROWS], row_t[TAPS_ROWS];
    griddep_launch_dependents();
    const int K = sh.K, n_az = sh.n_az, L = sh.L, Lf = sh.Lf, tid = threadIdx.x;
    const int r_lo = blockIdx.x * TAPS_ROWS, rows = min(TAPS_ROWS, sh.n_rng - r_lo);
    const int k0 = blockIdx.y * TAPS_COLS, nk = min(TAPS_COLS, K - k0);
    int far = BPA ? K / 2 : 0;
    if (!BPA)
        for (int k = tid; k < K; k += TAPS_THREADS) far = max(far, abs(canonical(__ldg(o + k), n_az)));
    far = __reduce_max_sync(0xffffffffu, far);
    if (tid == 0) s_max = 0;
    __syncthreads();
    if ((tid & 31) == 0) atomicMax(&s_max, far);
    __syncthreads();
    // the sine of half the angle grows up to half a turn, the farthest
    if (tid == 0) s_iv = lr::residuals((float)(p.r0 / p.dR), sinpif((float)s_max / (float)n_az), L, Lf);
    int32_t *offs = reinterpret_cast<int32_t *>(plan + sh.offs_at);
    if (tid >= 32 && tid < 32 + nk) {
        const int i = tid - 32, c = BPA ? k0 + i - K / 2 : canonical(__ldg(o + k0 + i), n_az);
        const double s = sinpi((double)c / (double)n_az);
        s2[i] = s * s;
        off_c[i] = c;
        if (blockIdx.x == 0) offs[k0 + i] = c;
    }
    __syncthreads();
    const lr::Interval iv = s_iv;
    const int P = min(iv.planes, sh.cap), cta = blockIdx.y * gridDim.x + blockIdx.x;
    if (tid < rows) {
        const int r = r_lo + tid, l = (int)((2LL * r * Lf + L) / (2LL * L));
        const double rd = r * p.dR;
        row_rd[tid] = rd;
        row_rd2[tid] = rd * rd;
        row_2R[tid] = 2.0 * (p.r0 + rd);
        row_c4[tid] = 4.0 * (p.r0 + rd) * p.r0;
        row_q[tid] = (double)(((long long)l * (L - 1)) % (2LL * Lf)) / (2.0 * Lf);
        row_t[tid] = ((double)l + iv.mid) / iv.half;
    }
    if (cta == 0 && tid == 32) *reinterpret_cast<Header *>(plan) = Header{lr::kPlanTag + sh.bpa, n_az, L, sh.n_rng, K, P, iv.half, 0};
    float2 *W = reinterpret_cast<float2 *>(plan + sh.w_at);
    const double inv_lf = 1.0 / Lf;               // exact: a power of two
    for (int i = cta * TAPS_THREADS + tid; i < P * Lf; i += gridDim.x * gridDim.y * TAPS_THREADS) {
        const int q = i / Lf, m = i - q * Lf;
        float2 v = make_float2(0.f, 0.f);
        if (m < L) {
            const double eta = (double)iv.mid + (double)iv.half * cheb_node(q, P);
            v = turns(-eta * inv_lf * ((double)(2 * m - (L - 1)) * 0.5));
            if (win) v = cscale(v, __ldg(win + m));
        }
        W[i] = v;
    }
    __syncthreads();
    float4 *taps = reinterpret_cast<float4 *>(plan + sh.taps_at);
    // cycles a metre of slant range: the reference sample's (eta (mid - m_ref)/Lf) and BPA's two-way phase
    const double per_m = -0.5 * p.phi_scale * (0.5 * (L - 1) - (double)p.m_ref) - (BPA ? p.two_f_over_c : 0.0);
    const double t_per_m = 0.5 * p.phi_scale * Lf / iv.half;
    const float inv_n = 1.f / (float)sh.N;
    for (int i = tid; i < rows * nk; i += TAPS_THREADS) {
        const int rr = i / nk, k = i - rr * nk, r = r_lo + rr;
        const double sk = s2[k], rho2 = fma(row_c4[rr], sk, row_rd2[rr]);
        double rho = 0.0;
        const float rho2f = (float)rho2;
        float y = 0.f;
        if (rho2f > 0.f) {                        // float root, one FP64 Newton step (1e-14)
            y = rsqrtf(rho2f);
            rho = rho2 * (double)y;
            rho = fma((double)(0.5f * y), fma(-rho, rho, rho2), rho);
        }
        float2 c = turns(fma(per_m, rho, row_q[rr]));
        if (BPA) {                                // alpha = (r dR - 2 R s^2)/rho
            const float num = (float)fma(-row_2R[rr], sk, row_rd[rr]);
            c = cscale(c, rho2f > 0.f ? fmaxf(0.f, num * y) : 1.f);
        } else {
            c = cmul(__ldg(w + (size_t)r * K + k0 + k), c);
        }
        c = cscale(c, inv_n);
        const int e = off_c[k] - sh.off;
        taps[(size_t)r * K + k0 + k] = make_float4(c.x, c.y, (float)fma(t_per_m, rho, -row_t[rr]),
                                                   __int_as_float(e <= 0 ? -e : sh.N - e));
    }
}

// H_q of row r = blockIdx.x for q = blockIdx.y, + gridDim.y, ...: the taps times ell_q into x, then FWD (transform of
// x and store, run by the whole CTA).
template <typename FWD>
__device__ __forceinline__ void lr_plan_row(const Shape &sh, uint8_t *plan, float2 *x, int x_len, int pad_shift, FWD fwd) {
    __shared__ float node[MAX_PLANES];
    griddep_wait();                           // the taps are complete
    const int P = plan_planes(plan, sh);
    if (threadIdx.x < P) node[threadIdx.x] = cheb_node(threadIdx.x, P);
    const float4 *taps = reinterpret_cast<const float4 *>(plan + sh.taps_at) + (size_t)blockIdx.x * sh.K;
    for (int q = blockIdx.y; q < P; q += gridDim.y) {
        __syncthreads();
        for (int n = threadIdx.x; n < x_len; n += blockDim.x) x[n] = make_float2(0.f, 0.f);
        const float tq = node[q];
        float den = 1.f;
        for (int i = 0; i < P; ++i)
            if (i != q) den *= tq - node[i];
        const float inv = 1.f / den;
        __syncthreads();
        for (int k = threadIdx.x; k < sh.K; k += blockDim.x) {
            const float4 t = __ldcg(taps + k);
            float ell = inv;
            for (int i = 0; i < P; ++i)
                if (i != q) ell *= t.z - node[i];
            const int at = rpad(__float_as_int(t.w), pad_shift);
            atomicAdd(&x[at].x, t.x * ell);   // offsets may repeat
            atomicAdd(&x[at].y, t.y * ell);
        }
        __syncthreads();
        fwd(reinterpret_cast<float2 *>(plan + sh.h_at + q * sh.h_plane) + (size_t)blockIdx.x * sh.pitch);
    }
}

// The spectra of the compile-time plans are stored radix-major for their last radix RK: element i RK-th of block b at
// i (N/RK) + b, so that a warp's accesses are consecutive.  The run-time plan stores digit-reversed order.

// Last DIF pass (blocks of RK, twiddles 1) to global memory.
template <int N, int RK, int T>
__device__ __forceinline__ void store_last(const float2 *x, float2 *__restrict__ dst) {
    constexpr int NB = N / RK;
#pragma unroll 1
    for (int b = threadIdx.x; b < NB; b += T) {
        float2 v[RK];
#pragma unroll
        for (int i = 0; i < RK; ++i) v[i] = x[b * RK + i];
        small_dft<RK>(v);
#pragma unroll
        for (int i = 0; i < RK; ++i) dst[i * NB + b] = v[i];
    }
}

template <int T, int N, int R1, int... Rs>
__global__ void __launch_bounds__(T)
lr_plan_fixed_kernel(Shape sh, uint8_t *__restrict__ plan) {
    extern __shared__ float2 sm[];
    griddep_launch_dependents();
    const float2 *tc, *tf;
    build_twiddles(N, false, sm + N, &tc, &tf);
    lr_plan_row(sh, plan, sm, N, 31, [&](float2 *dst) {
        dif_pass_c<N, N, R1, false, T>(sm, tc, tf);
        dif_middle<N, N / R1, T, WholeCta, Rs...>(sm, tc, tf);
        store_last<N, last_radix<R1, Rs...>(), T>(sm, dst);
    });
}

template <int T>
__global__ void __launch_bounds__(T)
lr_plan_runtime_kernel(Shape sh, RowPlan pl, uint8_t *__restrict__ plan) {
    extern __shared__ float2 sm[];
    griddep_launch_dependents();
    const float2 *tc, *tf;
    build_twiddles(sh.N, false, sm + padded_len(sh.N), &tc, &tf);
    lr_plan_row(sh, plan, sm, padded_len(sh.N), pl.pad_shift, [&](float2 *dst) {
        row_dif(sm, sh.N, pl, tc, tf);
        for (int n = threadIdx.x; n < sh.N; n += T) dst[n] = sm[rpad(n, pl.pad_shift)];
    });
}

// ---------------------------------------------------------------------------------------- per scan --

// Samples up to this pass the transforms: sums of 16384 pulses, 2048 samples and the taps stay far inside float32.
constexpr float kSpreadLimit = 1e20f;
__device__ __forceinline__ bool passes(float2 v) { return fabsf(v.x) + fabsf(v.y) < kSpreadLimit; }   // false for NaN

constexpr int TURN_PULSES = 16, TURN_SAMPLES = 64, TURN_THREADS = 256;

// raw [n_az][L] -> turned [L][t_pitch], a tile of 16 pulses x 64 samples per CTA: rows of 64 samples in, runs of 16
// pulses out.  A value that may not pass is stored as zero and marks its pulse, flags [sample tiles][n_az].
__global__ void __launch_bounds__(TURN_THREADS)
lr_turn_kernel(const float2 *__restrict__ raw, Shape sh, int t_pitch, float2 *__restrict__ turned,
               uint8_t *__restrict__ flags) {
    __shared__ float2 tile[TURN_SAMPLES][TURN_PULSES + 1];
    __shared__ int bad[TURN_PULSES];
    constexpr int IT = TURN_PULSES * TURN_SAMPLES / TURN_THREADS;
    griddep_launch_dependents();
    const int n0 = blockIdx.x * TURN_PULSES, m0 = blockIdx.y * TURN_SAMPLES;
    if (threadIdx.x < TURN_PULSES) bad[threadIdx.x] = 0;
    __syncthreads();
    griddep_wait();                           // the kernel before may write raw, or still read the workspace
    float2 v[IT];
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        const int e = threadIdx.x + i * TURN_THREADS, p = e / TURN_SAMPLES, m = e % TURN_SAMPLES;
        v[i] = make_float2(0.f, 0.f);
        if (n0 + p < sh.n_az && m0 + m < sh.L) v[i] = __ldcs(raw + (size_t)(n0 + p) * sh.L + m0 + m);
    }
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        const int e = threadIdx.x + i * TURN_THREADS, p = e / TURN_SAMPLES, m = e % TURN_SAMPLES;
        if (!passes(v[i])) {
            bad[p] = 1;
            v[i] = make_float2(0.f, 0.f);
        }
        tile[m][p] = v[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        const int e = threadIdx.x + i * TURN_THREADS, p = e % TURN_PULSES, m = e / TURN_PULSES;
        if (n0 + p < sh.n_az && m0 + m < sh.L) turned[(size_t)(m0 + m) * t_pitch + n0 + p] = tile[m][p];
    }
    if (threadIdx.x < TURN_PULSES && n0 + threadIdx.x < sh.n_az)
        flags[(size_t)blockIdx.y * sh.n_az + n0 + threadIdx.x] = (uint8_t)bad[threadIdx.x];
    const int used = sh.n_az * (int)gridDim.y;
    if (blockIdx.x == 0 && blockIdx.y == 0 && used + (int)threadIdx.x < sh.flag_bytes) flags[used + threadIdx.x] = 0;
}

// Pulse of element e of an azimuth row, or -1 where the row is zero.
__device__ __forceinline__ int pulse_at(int e, const Shape &sh) {
    const int n = e + sh.off;
    return e < sh.len ? (n < 0 ? n + sh.n_az : n >= sh.n_az ? n - sh.n_az : n) : -1;
}

template <int T, int N, int R1, int... Rs>
__global__ void __launch_bounds__(T)
lr_forward_fixed_kernel(const float2 *__restrict__ turned, int t_pitch, Shape sh, float2 *__restrict__ X) {
    extern __shared__ float2 sm[];
    constexpr int s1 = N / R1;
    griddep_launch_dependents();
    const float2 *tc, *tf;
    build_twiddles(N, false, sm + N, &tc, &tf);
    __syncthreads();
    griddep_wait();
    const float2 *row = turned + (size_t)blockIdx.x * t_pitch;
#pragma unroll 1
    for (int j = threadIdx.x; j < s1; j += T) {
        float2 v[R1];
#pragma unroll
        for (int i = 0; i < R1; ++i) {
            const int n = pulse_at(j + i * s1, sh);
            v[i] = n >= 0 ? __ldcg(row + n) : make_float2(0.f, 0.f);
        }
        small_dft<R1>(v);
        sm[j] = v[0];
        float2 wq[R1];
        twiddle_powers<R1>(twiddle(j, tc, tf), wq);
#pragma unroll
        for (int i = 1; i < R1; ++i) sm[j + i * s1] = cmul(v[i], wq[i]);
    }
    __syncthreads();
    dif_middle<N, s1, T, WholeCta, Rs...>(sm, tc, tf);
    store_last<N, last_radix<R1, Rs...>(), T>(sm, X + (size_t)blockIdx.x * sh.pitch);
}

template <int T>
__global__ void __launch_bounds__(T)
lr_forward_runtime_kernel(const float2 *__restrict__ turned, int t_pitch, Shape sh, RowPlan pl, float2 *__restrict__ X) {
    extern __shared__ float2 sm[];
    griddep_launch_dependents();
    const float2 *tc, *tf;
    build_twiddles(sh.N, false, sm + padded_len(sh.N), &tc, &tf);
    griddep_wait();
    const float2 *row = turned + (size_t)blockIdx.x * t_pitch;
    for (int n = threadIdx.x; n < sh.N; n += T) sm[rpad(n, pl.pad_shift)] = __ldcg(row + n);
    __syncthreads();
    row_dif(sm, sh.N, pl, tc, tf);
    for (int n = threadIdx.x; n < sh.N; n += T) X[(size_t)blockIdx.x * sh.pitch + n] = sm[rpad(n, pl.pad_shift)];
}

// Range transforms of F azimuth frequencies, LF/16 threads and 16 samples a thread each (as fft_tile.cuh, but the
// frequencies lie fastest across lanes: the spectra's rows are read and written in runs of F).  The column stays in
// registers over the planes; per plane it is multiplied by the plane's window, transformed (radix-16 Stockham passes
// through shared memory, buffers alternating so that one barrier an exchange is enough) and accumulated times H_q,
// whose tile arrives by cp.async during the plane before.  Three CTAs of 128 threads an SM (168 registers).  Bound by
// issue (600 instructions a plane and thread, 50 % issue at 12 warps an SM) next to the read of H (96 MB of DRAM in
// 26 us at 3600 x 256 and 12 planes: 55 % of the copy bandwidth).
template <int LF>
struct Col {
    static constexpr int RM = 16, T = LF / RM, LG = fft::ilog2(LF);
    static constexpr int NF = LG / 4, RR = LF >> (4 * NF);
    static constexpr int F = LF <= 512 ? 2048 / LF : LF <= 1024 ? 4 : 2;
    static constexpr int THREADS = T * F;
    static constexpr int EX = (LF + LF / 16) * F;              // one exchange buffer
    static constexpr int HT = LF * F;                          // one plane's H tile
    static constexpr size_t SMEM = sizeof(float2) * (size_t)(2 * EX + 2 * HT + LF) + sizeof(int) * LF;
};

template <int LF, int R, int NS>
__device__ __forceinline__ void col_load(float2 (&v)[16], int t, const float2 *ex) {
    using C = Col<LF>;
#pragma unroll
    for (int b = 0; b < 16 / R; ++b)
#pragma unroll
        for (int r = 0; r < R; ++r) v[b * R + r] = ex[fft::pad16(t + b * C::T + r * (LF / R)) * C::F];
}

// twiddles and the radix-R butterflies; output r of butterfly b is left at v[b*R + brev(r)]
template <int LF, int R, int NS>
__device__ __forceinline__ void col_dft(float2 (&v)[16], int t, const float2 *tw) {
    using C = Col<LF>;
#pragma unroll
    for (int b = 0; b < 16 / R; ++b) {
        if (NS > 1) {
            const int k = ((t + b * C::T) & (NS - 1)) * (LF / (NS * R));
#pragma unroll
            for (int r = 1; r < R; ++r) v[b * R + r] = cmul(v[b * R + r], tw[r * k]);
        }
        fft::dft_dif<R>(v + b * R);
    }
}

template <int LF, int R, int NS>
__device__ __forceinline__ void col_store(const float2 (&v)[16], int t, float2 *ex) {
    using C = Col<LF>;
#pragma unroll
    for (int b = 0; b < 16 / R; ++b) {
        const int j = t + b * C::T, k = j & (NS - 1), base = (j - k) * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) ex[fft::pad16(base + r * NS) * C::F] = v[b * R + fft::brev(r, fft::ilog2(R))];
    }
}

__device__ __forceinline__ void cp_async16(void *dst_smem, const void *src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst_smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}

template <int LF>
__global__ void __launch_bounds__(Col<LF>::THREADS, (Col<LF>::THREADS <= 128 ? 3 : 1))
lr_combine_kernel(const float2 *__restrict__ X, const uint8_t *__restrict__ plan, Shape sh, float2 *__restrict__ Y) {
    using C = Col<LF>;
    constexpr int F = C::F, NF = C::NF, RR = C::RR;
    constexpr int RL = RR > 1 ? RR : 16, NSL = LF / RL;         // the last pass: bin l = j + r*NSL
    extern __shared__ __align__(16) float2 csm[];
    float2 *ex0 = csm, *hs = csm + 2 * C::EX, *tw = hs + 2 * C::HT;
    int *row_of = reinterpret_cast<int *>(tw + LF);
    griddep_launch_dependents();
    const int f = threadIdx.x % F, t = threadIdx.x / F, f0 = blockIdx.x * F;
    for (int i = threadIdx.x; i < LF; i += C::THREADS) {
        float s, c;
        sincospif(2.f * (float)i / (float)LF, &s, &c);
        tw[i] = make_float2(c, -s);
        // the row whose bin round(r LF/L) is i, or -1: r = ceil((2 i - 1) L / (2 LF))
        const long long a = (2LL * i - 1) * sh.L;
        const int r = a <= 0 ? 0 : (int)((a + 2LL * LF - 1) / (2LL * LF));
        row_of[i] = r < sh.n_rng && (int)((2LL * r * LF + sh.L) / (2LL * sh.L)) == i ? r : -1;
    }
    for (int i = threadIdx.x; i < 2 * C::HT; i += C::THREADS) hs[i] = make_float2(0.f, 0.f);
    __syncthreads();
    griddep_wait();
    const int P = plan_planes(plan, sh);
    const float2 *W = reinterpret_cast<const float2 *>(plan + sh.w_at);
    // H_q's tile: 16 bytes (two frequencies) a copy, 8 a thread; bins without a row stay zero
    int at[8];
    static_assert(C::HT / 2 == 8 * C::THREADS, "eight copies a thread");
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int e = threadIdx.x + i * C::THREADS, c = f0 + 2 * (e % (F / 2)), r = row_of[e / (F / 2)];
        at[i] = r >= 0 && c < sh.pitch ? r * sh.pitch + c : -1;
    }
    auto stage = [&](int q) {
        const float2 *H = reinterpret_cast<const float2 *>(plan + sh.h_at + q * sh.h_plane);
        float2 *dst = hs + (q & 1) * C::HT + 2 * threadIdx.x;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (at[i] >= 0) cp_async16(dst + 2 * i * C::THREADS, H + at[i]);
        cp_async_commit();
    };
    if (P > 0) stage(0);
    float2 x[16], acc[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int m = t + r * C::T;
        x[r] = m < sh.L && f0 + f < sh.pitch ? __ldcg(X + (size_t)m * sh.pitch + f0 + f) : make_float2(0.f, 0.f);
        acc[r] = make_float2(0.f, 0.f);
    }
    int nx = 0;                               // exchanges so far: buffer nx & 1
    for (int q = 0; q < P; ++q) {
        float2 v[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) v[r] = cmul(x[r], __ldca(W + q * LF + t + r * C::T));
        col_dft<LF, 16, 1>(v, t, tw);
        auto exchange = [&](auto R_, auto NS_, auto RN_, bool first) {
            constexpr int R = decltype(R_)::value, NS = decltype(NS_)::value, RN = decltype(RN_)::value;
            float2 *ex = ex0 + (nx++ & 1) * C::EX + f;
            col_store<LF, R, NS>(v, t, ex);
            if (first) cp_async_wait<0>();
            __syncthreads();
            if (first && q + 1 < P) stage(q + 1);   // every thread has read the tile it overwrites
            col_load<LF, RN, NS * R>(v, t, ex);
            col_dft<LF, RN, NS * R>(v, t, tw);
        };
        using I16 = std::integral_constant<int, 16>;
        if constexpr (NF == 1 && RR == 1) {   // LF = 16: no exchange
            cp_async_wait<0>();
            __syncthreads();
            if (q + 1 < P) stage(q + 1);
        }
        if constexpr (NF >= 2) exchange(I16{}, std::integral_constant<int, 1>{}, I16{}, true);
        if constexpr (NF >= 3) exchange(I16{}, I16{}, I16{}, false);
        if constexpr (RR > 1)
            exchange(I16{}, std::integral_constant<int, LF / RR / 16>{}, std::integral_constant<int, RR>{}, NF == 1);
        const float2 *h = hs + (q & 1) * C::HT + f;
#pragma unroll
        for (int b = 0; b < 16 / RL; ++b)
#pragma unroll
            for (int r = 0; r < RL; ++r)
                cmac(acc[b * RL + r], v[b * RL + fft::brev(r, fft::ilog2(RL))], h[(t + b * C::T + r * NSL) * F]);
    }
    if (f0 + f < sh.pitch) {
#pragma unroll
        for (int b = 0; b < 16 / RL; ++b)
#pragma unroll
            for (int r = 0; r < RL; ++r) {
                const int row = row_of[t + b * C::T + r * NSL];
                if (row >= 0) Y[(size_t)row * sh.pitch + f0 + f] = acc[b * RL + r];
            }
    }
}

__device__ __forceinline__ void fill_nan(float2 *__restrict__ out_row, int n) {
    const float nan = __int_as_float(0x7fc00000);
    for (int i = threadIdx.x; i < n; i += blockDim.x) out_row[i] = make_float2(nan, nan);
}

// Whether any pulse is marked, and the terms of the marked pulses' zeroed samples for the pixels of row r whose aperture
// holds one: the tap's phasor is the first node's window turned by the tap's distance from that node.  (The kernel
// overlaps the one before it, so nothing that this call wrote is read by the non-coherent path.)
__device__ __forceinline__ bool any_marked(const uint8_t *__restrict__ flags, const Shape &sh) {
    int any = 0;
    const int *words = reinterpret_cast<const int *>(flags);
    for (int n = threadIdx.x; n < sh.flag_bytes / 4; n += blockDim.x) any |= __ldcg(words + n);
    return __syncthreads_or(any) != 0;
}
__device__ __noinline__ void add_marked(const float2 *__restrict__ raw, const uint8_t *__restrict__ flags,
                                        const uint8_t *__restrict__ plan, const Shape &sh, int r,
                                        float2 *__restrict__ out_row) {
    const float half = __ldcg(reinterpret_cast<const float *>(plan + offsetof(Header, half)));
    const float node = cheb_node(0, plan_planes(plan, sh)), inv_lf = 1.f / (float)sh.Lf, mid = 0.5f * (float)(sh.L - 1);
    const float2 *W = reinterpret_cast<const float2 *>(plan + sh.w_at);
    const int32_t *offs = reinterpret_cast<const int32_t *>(plan + sh.offs_at);
    const float4 *taps = reinterpret_cast<const float4 *>(plan + sh.taps_at) + (size_t)r * sh.K;
    const int l = (int)((2LL * r * sh.Lf + sh.L) / (2LL * sh.L));
    __syncthreads();                          // after the row's own stores
    for (int th = threadIdx.x; th < sh.n_az; th += blockDim.x) {
        float2 add = make_float2(0.f, 0.f);
        bool hit = false, finite = true;
        for (int k = 0; k < sh.K; ++k) {
            const int n = pmod(th + __ldcg(offs + k), sh.n_az);
            for (int m0 = 0; m0 < sh.L; m0 += TURN_SAMPLES) {
                if (!__ldcg(flags + (size_t)(m0 / TURN_SAMPLES) * sh.n_az + n)) continue;
                hit = true;
                const float4 t = __ldcg(taps + k);
                const float per_m = half * (t.z - node) * inv_lf;
                float2 sum = make_float2(0.f, 0.f);
                for (int m = m0; m < min(m0 + TURN_SAMPLES, sh.L); ++m) {
                    const float2 v = __ldcg(raw + (size_t)n * sh.L + m);
                    if (passes(v)) continue;
                    finite = finite && isfinite(v.x) && isfinite(v.y);
                    float s, c;
                    sincospif(2.f * fmaf(per_m, (float)m - mid, (float)((l * m) & (sh.Lf - 1)) * inv_lf), &s, &c);
                    cmac(sum, cmul(__ldcg(W + m), make_float2(c, -s)), v);
                }
                cmac(add, make_float2(t.x * (float)sh.N, t.y * (float)sh.N), sum);
            }
        }
        if (hit) {
            const float nan = __int_as_float(0x7fc00000);
            out_row[th] = finite ? cadd(out_row[th], add) : make_float2(nan, nan);
        }
    }
}

template <int T, int N, int R1, int... Rs>
__global__ void __launch_bounds__(T)
lr_inverse_fixed_kernel(const float2 *__restrict__ Y, Shape sh, const uint8_t *__restrict__ plan,
                        const uint8_t *__restrict__ flags, const float2 *__restrict__ raw, float2 *__restrict__ out) {
    extern __shared__ float2 sm[];
    constexpr int s1 = N / R1, RK = last_radix<R1, Rs...>(), NB = N / RK;
    const float2 *tc, *tf;
    build_twiddles(N, false, sm + N, &tc, &tf);
    griddep_wait();
    const float2 *row = Y + (size_t)blockIdx.x * sh.pitch;
    float2 *out_row = out + (size_t)blockIdx.x * sh.n_az;
    if (plan_planes(plan, sh) == 0) return fill_nan(out_row, sh.n_az);
    const bool marked = any_marked(flags, sh);
#pragma unroll 1
    for (int b = threadIdx.x; b < NB; b += T) {
        float2 v[RK];
#pragma unroll
        for (int i = 0; i < RK; ++i) {
            v[i] = __ldcg(row + i * NB + b);
            v[i].y = -v[i].y;
        }
        small_dft<RK>(v);
#pragma unroll
        for (int i = 0; i < RK; ++i) sm[b * RK + i] = v[i];
    }
    __syncthreads();
    dit_middle<N, s1, T, WholeCta, Rs...>(sm, tc, tf);
#pragma unroll 1
    for (int j = threadIdx.x; j < s1; j += T) {
        float2 v[R1], wq[R1];
        twiddle_powers<R1>(twiddle(j, tc, tf), wq);
        v[0] = sm[j];
#pragma unroll
        for (int i = 1; i < R1; ++i) v[i] = cmul(sm[j + i * s1], wq[i]);
        small_dft<R1>(v);
#pragma unroll
        for (int i = 0; i < R1; ++i)
            if (j + i * s1 < sh.n_az) out_row[j + i * s1] = make_float2(v[i].x, -v[i].y);
    }
    if (marked) add_marked(raw, flags, plan, sh, blockIdx.x, out_row);
}

template <int T>
__global__ void __launch_bounds__(T)
lr_inverse_runtime_kernel(const float2 *__restrict__ Y, Shape sh, RowPlan pl, const uint8_t *__restrict__ plan,
                          const uint8_t *__restrict__ flags, const float2 *__restrict__ raw, float2 *__restrict__ out) {
    extern __shared__ float2 sm[];
    const float2 *tc, *tf;
    build_twiddles(sh.N, false, sm + padded_len(sh.N), &tc, &tf);
    griddep_wait();
    const float2 *row = Y + (size_t)blockIdx.x * sh.pitch;
    float2 *out_row = out + (size_t)blockIdx.x * sh.n_az;
    if (plan_planes(plan, sh) == 0) return fill_nan(out_row, sh.n_az);
    const bool marked = any_marked(flags, sh);
    for (int n = threadIdx.x; n < sh.N; n += T) {
        const float2 v = __ldcg(row + n);
        sm[rpad(n, pl.pad_shift)] = make_float2(v.x, -v.y);
    }
    __syncthreads();
    row_dit(sm, sh.N, pl, tc, tf);
    for (int n = threadIdx.x; n < sh.n_az; n += T) {
        const float2 v = sm[rpad(n, pl.pad_shift)];
        out_row[n] = make_float2(v.x, -v.y);
    }
    if (marked) add_marked(raw, flags, plan, sh, blockIdx.x, out_row);
}

// -------------------------------------------------------------------------------------------- host --

struct FixedRow {
    int N, threads;
    const void *plan, *forward, *inverse;
    int *done[3];
};

template <int T, int N, int... R>
FixedRow fixed_row() {
    static int done[3][kMaxDevices] = {};
    return FixedRow{N, T, (const void *)lr_plan_fixed_kernel<T, N, R...>,
                    (const void *)lr_forward_fixed_kernel<T, N, R...>,
                    (const void *)lr_inverse_fixed_kernel<T, N, R...>, {done[0], done[1], done[2]}};
}

const FixedRow *fixed_rows(int *n) {
    static const FixedRow rows[] = {
        fixed_row<64, 360, 8, 3, 15>(),      fixed_row<128, 720, 4, 12, 15>(),    fixed_row<128, 960, 8, 8, 15>(),
        fixed_row<128, 1440, 8, 12, 15>(),   fixed_row<128, 1800, 8, 15, 15>(),   fixed_row<256, 2400, 16, 10, 15>(),
        fixed_row<256, 3600, 16, 15, 15>(),  fixed_row<256, 4800, 8, 4, 10, 15>(), fixed_row<256, 5760, 8, 4, 12, 15>(),
        fixed_row<256, 7200, 8, 4, 15, 15>(), fixed_row<512, 9600, 8, 8, 10, 15>(), fixed_row<512, 14400, 8, 8, 15, 15>(),
    };
    *n = (int)(sizeof(rows) / sizeof(rows[0]));
    return rows;
}

const FixedRow *find_fixed(int N) {
    int n;
    const FixedRow *rows = fixed_rows(&n);
    for (int i = 0; i < n; ++i)
        if (rows[i].N == N) return rows + i;
    return nullptr;
}

size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

// Launch with programmatic overlap of the kernel before, which every kernel here waits for before its first access.
template <typename... P, typename... A>
rosar_status go(const char *what, void (*fn)(P...), dim3 grid, int threads, size_t smem, bool overlap, cudaStream_t s,
                A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = overlap ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, fn, static_cast<P>(args)...);
    if (e != cudaSuccess) return set_error(ROSAR_ERR_CUDA, "%s: launch failed: %s", what, cudaGetErrorString(e));
    return check_launch(what);
}

template <int LF>
rosar_status launch_combine(const char *what, const float2 *X, const uint8_t *plan, const Shape &sh, float2 *Y,
                            cudaStream_t s) {
    static int done[kMaxDevices] = {};
    rosar_status st = ensure_smem((const void *)lr_combine_kernel<LF>, Col<LF>::SMEM, done, what);
    if (st != ROSAR_OK) return st;
    static_assert(Col<LF>::SMEM <= 227 * 1024, "the column tile exceeds shared memory");
    return go(what, lr_combine_kernel<LF>, dim3((sh.N + Col<LF>::F - 1) / Col<LF>::F), Col<LF>::THREADS, Col<LF>::SMEM,
              true, s, X, plan, sh, Y);
}

int runtime_threads(int N) { return N <= 4096 ? 256 : 512; }
size_t row_bytes(int N, bool fixed) {
    return sizeof(float2) * (size_t)((fixed ? N : padded_len(N)) + 64 + coarse_len(N));
}

}  // namespace

namespace lr {

Shape shape_of(bool bpa, int n_az, int L, int n_rng, int K) {
    Shape sh = {};
    sh.bpa = bpa ? 1 : 0;
    sh.n_az = n_az;
    sh.L = L;
    sh.n_rng = n_rng;
    sh.K = K;
    if (L > MAX_LF || L < 16 || n_rng > L || n_az < 2 || n_az > AF_MAX_N || K < 1 || (bpa && K > n_az)) return sh;
    sh.Lf = 16;
    while (sh.Lf < L) sh.Lf *= 2;
    // n_az itself where it has a compile-time plan; a longer compile-time plan with room for the wrapped pulses (all
    // of the ring for offsets in device memory); the run-time plan of n_az where that room would cost more
    const int room = bpa ? n_az + K - 1 : 2 * n_az;
    RowPlan pl;
    const bool smooth = make_plan(n_az, &pl);
    if (find_fixed(n_az)) {
        sh.N = n_az;
        sh.fixed = 1;
    } else {
        int n;
        const FixedRow *rows = fixed_rows(&n);
        for (int i = n - 1; i >= 0; --i)
            if (rows[i].N >= room) sh.N = rows[i].N;
        sh.fixed = sh.N != 0;
        if (smooth && (!sh.N || sh.N > n_az + n_az / 2)) {
            sh.N = n_az;
            sh.fixed = 0;
        }
    }
    if (!sh.N) return sh;
    const bool circular = sh.N == n_az;
    sh.off = circular ? 0 : bpa ? -(K / 2) : -(n_az / 2);
    sh.len = circular ? n_az : room;
    sh.pitch = (sh.N + 15) & ~15;
    sh.h_plane = sizeof(float2) * (size_t)n_rng * sh.pitch;
    sh.w_at = 256;
    sh.offs_at = sh.w_at + align256(sizeof(float2) * (size_t)MAX_PLANES * sh.Lf);
    sh.taps_at = sh.offs_at + align256(sizeof(int32_t) * (size_t)K);
    sh.h_at = sh.taps_at + align256(sizeof(float4) * (size_t)n_rng * K);
    // the turned cube is dead once its transform is taken: it shares its place with the image's spectra
    const size_t t_bytes = sizeof(float2) * (size_t)L * ((n_az + 15) & ~15), y_bytes = sh.h_plane;
    sh.t_at = 0;
    sh.x_at = align256(t_bytes > y_bytes ? t_bytes : y_bytes);
    sh.flags_at = sh.x_at + align256(sizeof(float2) * (size_t)L * sh.pitch);
    sh.flag_bytes = (n_az * ((L + TURN_SAMPLES - 1) / TURN_SAMPLES) + 3) & ~3;    // read in words: the pad is written too
    sh.ws_bytes = sh.flags_at + align256((size_t)sh.flag_bytes);
    sh.valid = 1;
    return sh;
}

int planes_bound(const TdParams &p, bool bpa, int K, int Lf) {
    const double half_turns = bpa ? (double)(K / 2) / p.n_az : 0.5;
    const double s = sin(3.14159265358979323846 * (half_turns < 0.5 ? half_turns : 0.5));
    return residuals((float)(p.r0 / p.dR), (float)s, p.L, Lf).planes + 1;
}

}  // namespace lr

// Where the transforms are taken: the form exists for the sizes, its planes stay few, and the direct sums are long
// enough to pay for the six short kernels: from 4e7 multiply-adds, a little below the smallest sizes measured on both
// sides (369 x 64, M = 43, 6.5e7: 42 us with its plan against 79; 376 x 80, M = 50, 1.2e8, planned: 31 against 38).
bool time_domain_lr_applies(const TdParams &p, bool bpa, int K, size_t *plan_bytes, size_t *ws_bytes) {
    const Shape sh = lr::shape_of(bpa, p.n_az, p.L, p.n_rng, K);
    if (!sh.valid) return false;
    const int P = lr::planes_bound(p, bpa, K, sh.Lf);
    if (P > MAX_PLANES) return false;
    if ((double)p.n_az * p.n_rng * K * p.L < 4e7) return false;
    *plan_bytes = sh.h_at + (size_t)P * sh.h_plane;
    if (*plan_bytes == time_domain_plan_bytes(p.n_rng, p.L, K)) *plan_bytes += 256;   // the size tells the two plans apart
    *ws_bytes = sh.ws_bytes;
    return true;
}

// Whether SAS by transforms is the faster form, planned and with the plan built in the call, also where the offsets reach
// half a turn (the planes that its plan has room for): times in us of both forms as sums of their parts, fitted to 705
// sizes (97 to 14400 pulses, 16 to 2048 samples, 1 to 2048 rows, 2 to 256 taps, offsets over a sixth and the whole of the
// ring) to 20 to 30 %.  With the transforms asked to be 1.3 times as fast, 5 of them are slower with wide offsets (0.74 at
// the least) and none with narrow ones, where all of them by transforms were 128: 4501 x 208, K = 2: 214 us against 45;
// 14400 x 64, K = 2: 74 and 19; 3600 x 1024, 16 rows, K = 2: 152 and 147.  3600 x 256, K = 64 has 92 against 640.
bool time_domain_lr_pays(const TdParams &p, int K) {
    const Shape sh = lr::shape_of(false, p.n_az, p.L, p.n_rng, K);
    if (!sh.valid) return false;
    const double P = lr::planes_bound(p, false, K, sh.Lf), N = sh.N, L = p.L, q = p.n_rng, n = p.n_az;
    const double image = 9.0 + 0.66 * P + 1e-6 * (9.7 * n * L + 8.0 * L * N + 6.2 * q * N + 1.5 * P * N * sh.Lf);
    const double plan = 21.0 + 1e-6 * (2.9 * P * q * N + 14.5 * P * q * K + 340.0 * N);
    const double tiles = ceil(n / 128.0) * ceil(q / 64.0), sums = tiles * K * L;     // of the tensor cores
    const double direct = 40.0 + 2.53e-4 * sums + 3.9e-3 * L * K;
    const double direct_planned = 22.0 + 1.77e-4 * sums + 3.1e-3 * L * K + 0.034 * tiles;
    return direct > 1.3 * (image + plan) && direct_planned > 1.3 * image;
}

size_t time_domain_lr_workspace(bool bpa, int n_az, int L, int n_rng, int K) {
    const Shape sh = lr::shape_of(bpa, n_az, L, n_rng, K);
    return sh.valid ? sh.ws_bytes : 0;
}

size_t time_domain_lr_plan_least(bool bpa, int n_az, int L, int n_rng, int K) {
    const Shape sh = lr::shape_of(bpa, n_az, L, n_rng, K);
    return sh.valid ? sh.h_at + 2 * sh.h_plane : 0;      // two planes at least (planes_for)
}

rosar_status launch_time_domain_lr_plan(const float *win, const float2 *w, const int32_t *o, const TdParams &p, int K,
                                        bool bpa, void *plan, cudaStream_t s) {
    const char *what = bpa ? "bpa_time_plan" : "sas_time_plan";
    Shape sh = lr::shape_of(bpa, p.n_az, p.L, p.n_rng, K);
    sh.cap = lr::planes_bound(p, bpa, K, sh.Lf);
    uint8_t *pb = static_cast<uint8_t *>(plan);
    const dim3 tg((p.n_rng + TAPS_ROWS - 1) / TAPS_ROWS, (K + TAPS_COLS - 1) / TAPS_COLS);
    rosar_status st = bpa ? go(what, lr_taps_kernel<true>, tg, TAPS_THREADS, 0, false, s, win, w, o, p, sh, pb)
                          : go(what, lr_taps_kernel<false>, tg, TAPS_THREADS, 0, false, s, win, w, o, p, sh, pb);
    if (st != ROSAR_OK) return st;
    // planes of a row over several CTAs: a few CTAs an SM in all
    const int split = p.n_rng >= 1024 ? 1 : p.n_rng >= 256 ? 4 : 8;
    const dim3 grid(p.n_rng, split);
    const size_t smem = row_bytes(sh.N, sh.fixed != 0);
    if (sh.fixed) {
        const FixedRow *f = find_fixed(sh.N);
        st = ensure_smem(f->plan, smem, f->done[0], what);
        if (st != ROSAR_OK) return st;
        return go(what, reinterpret_cast<void (*)(Shape, uint8_t *)>(const_cast<void *>(f->plan)), grid, f->threads, smem,
                  true, s, sh, pb);
    }
    static int done[2][kMaxDevices] = {};
    RowPlan pl;
    make_plan(sh.N, &pl);
    const int T = runtime_threads(sh.N);
    auto fn = T == 256 ? lr_plan_runtime_kernel<256> : lr_plan_runtime_kernel<512>;
    st = ensure_smem((const void *)fn, smem, done[T == 512], what);
    if (st != ROSAR_OK) return st;
    return go(what, fn, grid, T, smem, true, s, sh, pl, pb);
}

rosar_status launch_time_domain_lr(const float2 *raw, int n_az, int L, int n_rng, int K, bool bpa, const void *plan,
                                   void *workspace, float2 *out, cudaStream_t s) {
    const char *what = bpa ? "bpa_time" : "sas_time";
    const Shape sh = lr::shape_of(bpa, n_az, L, n_rng, K);
    const uint8_t *pb = static_cast<const uint8_t *>(plan);
    uint8_t *ws = static_cast<uint8_t *>(workspace);
    float2 *turned = reinterpret_cast<float2 *>(ws + sh.t_at), *Y = turned;
    float2 *X = reinterpret_cast<float2 *>(ws + sh.x_at);
    uint8_t *flags = ws + sh.flags_at;
    const int t_pitch = (n_az + 15) & ~15;
    rosar_status st = go(what, lr_turn_kernel, dim3((n_az + TURN_PULSES - 1) / TURN_PULSES, (L + TURN_SAMPLES - 1) / TURN_SAMPLES), TURN_THREADS, 0,
                         true, s,
                         raw, sh, t_pitch, turned, flags);
    if (st != ROSAR_OK) return st;
    const size_t smem = row_bytes(sh.N, sh.fixed != 0);
    const FixedRow *f = sh.fixed ? find_fixed(sh.N) : nullptr;
    static int done[4][kMaxDevices] = {};
    RowPlan pl = {};
    const int T = f ? f->threads : runtime_threads(sh.N);
    if (f) {
        st = ensure_smem(f->forward, smem, f->done[1], what);
        if (st == ROSAR_OK)
            st = go(what, reinterpret_cast<void (*)(const float2 *, int, Shape, float2 *)>(const_cast<void *>(f->forward)),
                    dim3(L), T, smem, true, s, turned, t_pitch, sh, X);
    } else {
        make_plan(sh.N, &pl);
        auto fn = T == 256 ? lr_forward_runtime_kernel<256> : lr_forward_runtime_kernel<512>;
        st = ensure_smem((const void *)fn, smem, done[T == 512], what);
        if (st == ROSAR_OK) st = go(what, fn, dim3(L), T, smem, true, s, turned, t_pitch, sh, pl, X);
    }
    if (st != ROSAR_OK) return st;
    switch (sh.Lf) {
        case 16: st = launch_combine<16>(what, X, pb, sh, Y, s); break;
        case 32: st = launch_combine<32>(what, X, pb, sh, Y, s); break;
        case 64: st = launch_combine<64>(what, X, pb, sh, Y, s); break;
        case 128: st = launch_combine<128>(what, X, pb, sh, Y, s); break;
        case 256: st = launch_combine<256>(what, X, pb, sh, Y, s); break;
        case 512: st = launch_combine<512>(what, X, pb, sh, Y, s); break;
        case 1024: st = launch_combine<1024>(what, X, pb, sh, Y, s); break;
        default: st = launch_combine<2048>(what, X, pb, sh, Y, s); break;
    }
    if (st != ROSAR_OK) return st;
    if (f) {
        st = ensure_smem(f->inverse, smem, f->done[2], what);
        if (st != ROSAR_OK) return st;
        return go(what,
                  reinterpret_cast<void (*)(const float2 *, Shape, const uint8_t *, const uint8_t *, const float2 *, float2 *)>(
                      const_cast<void *>(f->inverse)),
                  dim3(n_rng), T, smem, true, s, Y, sh, pb, flags, raw, out);
    }
    auto fn = T == 256 ? lr_inverse_runtime_kernel<256> : lr_inverse_runtime_kernel<512>;
    st = ensure_smem((const void *)fn, smem, done[2 + (T == 512)], what);
    if (st != ROSAR_OK) return st;
    return go(what, fn, dim3(n_rng), T, smem, true, s, Y, sh, pl, pb, flags, raw, out);
}

}  // namespace rosar
