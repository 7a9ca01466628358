// K3f: back-projection of the range-compressed data with nominal pulse positions, row by row in the
// azimuth-frequency domain (arXiv 2309.08038, Sec. III-D after Eq. (43) with w_BP; Eq. (14)).
//
// Without position errors the bin x and the weight a of an aperture offset d depend on (r, d) only, so row r is a
// sum of circular filters, one per range row r + q that its taps read:
//
//   out[r][.] = e^{-j 2 k_mid rho} * sum_q g_{r,q} (*) S[r + q][.],
//   g_{r,q}[-d] = a_d * ((1 - f_d) [floor(x_d) = r + q] + f_d [floor(x_d) + 1 = r + q])     (linear interpolation)
//               = a_d * [floor(x_d + 1/2) = r + q]                                          (nearest bin)
//
// R_n >= rho puts every x_d at r or above, and over a 60 degree aperture within a bin of it for all but the first
// rows: two or three planes q.  One CTA per row; per plane its two groups of T threads transform the S row (group
// A) and the taps (group B, straight from the geometry) at the same time, A accumulates the product, and the whole
// CTA runs one inverse transform: 2 planes + 1 transforms of length N instead of M multiply-adds a pixel, and no
// scratch memory (shared: the two rows and the accumulated spectrum).  Same bins and weights as bpa_kernel; the
// sums differ by float32 rounding.
//
// N is n_az itself where it has a compile-time plan (the filter is circular), else the smallest plan with
// N >= n_az + M - 1: the S row is extended by the pulses its aperture wraps to and the first n_az outputs are kept.
//
// Bound: the transforms' issue slots and barriers (a row's chain of planes + 1 transforms), not memory.  3600 x 256,
// M = 600: 24.5 us where the direct kernel takes 400; 1800 x 512, M = 300: 22.6 (216); 7200 x 256, M = 1200: 45
// (1488).
//
// A transform spreads an infinity or a NaN of one pulse over the row, so group A looks at every value it loads and
// a row with a value that is not finite (or above 1e30, where the sums could overflow) is summed directly instead.

#include <math.h>

#include "bpa_geometry.cuh"
#include "row_fft.cuh"

namespace rosar {
namespace {

using namespace rowfft;

constexpr float kSpreadLimit = 1e30f;

// Row r summed offset by offset, for rows that hold values a transform would spread; tab: `cap` entries.
__device__ __noinline__ void bpa_row_direct(const float2 *__restrict__ S, const BpaParams &p, int r, int L, int n_az,
                                            int M_ap, bool linear, float2 rowph, float4 *tab, int cap,
                                            float2 *__restrict__ out) {
    const double rho_d = r * p.dR;
    const float rho = (float)rho_d, R = (float)(p.r0 + rho_d), r0 = (float)p.r0;
    const int d_beg = -(M_ap / 2);
    for (int t0 = 0; t0 < n_az; t0 += blockDim.x) {
        const int th = t0 + threadIdx.x;
        float2 acc = make_float2(0.f, 0.f);
        for (int i0 = 0; i0 < M_ap; i0 += cap) {
            const int nd = min(cap, M_ap - i0);
            __syncthreads();
            for (int i = threadIdx.x; i < nd; i += blockDim.x) {
                float s, c, x, delta, alpha;
                sincospif((float)(d_beg + i0 + i) / (float)n_az, &s, &c);
                nominal_tap(s, R, r0, rho, (float)r, p.inv_dR, x, delta, alpha);
                const float2 a = nominal_weight(p.two_f_over_c, delta, alpha);
                tab[i] = make_float4(x, a.x, a.y, 0.f);
            }
            __syncthreads();
            if (th >= n_az) continue;
            for (int i = 0; i < nd; ++i) {
                const float4 t = tab[i];
                const int n = pmod(th + d_beg + i0 + i, n_az);
                float2 sv;
                if (linear) {
                    const float fl = floorf(t.x);
                    const float2 s0 = read_bin<true>(S, (int)fl, L, n, n_az), s1 = read_bin<true>(S, (int)fl + 1, L, n, n_az);
                    sv = caxpy(t.x - fl, csub(s1, s0), s0);
                } else {
                    sv = read_bin<true>(S, (int)floorf(t.x + 0.5f), L, n, n_az);
                }
                cmac(acc, make_float2(t.y, t.z), sv);
            }
        }
        if (th < n_az) out[(size_t)r * n_az + th] = cmul(rowph, acc);
    }
}

// Shared memory: the S row, the taps, the accumulated spectrum, the twiddle table.
template <int N>
constexpr size_t bpa_rows_smem() { return sizeof(float2) * (size_t)(3 * N + 64 + coarse_len(N)); }

// off, len: element i < len of the row is pulse (i + off) mod n_az, the rest zero; the output of offset d from the
// element at off + i lands on element i of the result.
template <int T, int MINB, int N, int R1, int... Rs>
__global__ void __launch_bounds__(2 * T, MINB)
bpa_rows_kernel(const float2 *__restrict__ S, BpaParams p, int L, int n_az, int M_ap, int linear, int off, int len,
                float2 *__restrict__ out) {
    static_assert(pad_shift_for(N) == 31, "compile-time plans are for rows with an odd factor");
    constexpr int RK = last_radix<R1, Rs...>(), NB = N / RK, s1 = N / R1;
    using G = ThreadGroup<T>;
    extern __shared__ float2 sm[];
    float2 *x = sm, *g = sm + N, *y = sm + 2 * N, *tw = sm + 3 * N;
    __shared__ float2 rowph;
    __shared__ int s_top;
    const int r = blockIdx.x;
    const bool grp_a = threadIdx.x < T;
    const double rho_d = r * p.dR;
    const float rho = (float)rho_d, R = (float)(p.r0 + rho_d), r0 = (float)p.r0;
    const int d_beg = -(M_ap / 2), d_end = M_ap - M_ap / 2;
    const float2 *tc, *tf;
    build_twiddles(N, false, tw, &tc, &tf);
    if (threadIdx.x == 0) {
        rowph = row_phase(p, rho_d);
        s_top = 0;
    }
    __syncthreads();

    for (int q = 0;; ++q) {
        int bad = 0;
        if (grp_a) {
            if (q == 0) griddep_wait();              // S is complete
            const float2 *row = S + (size_t)(r + q) * n_az;
#pragma unroll 1
            for (int j = G::tid(); j < s1; j += T) {  // first pass (block N) on the extended row
                float2 v[R1];
#pragma unroll
                for (int i = 0; i < R1; ++i) {
                    const int e = j + i * s1;
                    int n = e + off;
                    n += n < 0 ? n_az : n >= n_az ? -n_az : 0;
                    v[i] = e < len ? __ldcg(row + n) : make_float2(0.f, 0.f);
                }
#pragma unroll
                for (int i = 0; i < R1; ++i) bad |= !(fabsf(v[i].x) + fabsf(v[i].y) < kSpreadLimit);
                small_dft<R1>(v);
                x[j] = v[0];
                float2 wq[R1];
                twiddle_powers<R1>(twiddle(j, tc, tf), wq);
#pragma unroll
                for (int i = 1; i < R1; ++i) x[j + i * s1] = cmul(v[i], wq[i]);
            }
            G::sync();
            dif_middle<N, s1, T, G, Rs...>(x, tc, tf);
        } else {
            for (int n = G::tid(); n < N; n += T) g[n] = make_float2(0.f, 0.f);
            G::sync();
            int top = 0;
            for (int d = d_beg + G::tid(); d < d_end; d += T) {
                float s, c, xb, delta, alpha;
                sincospif((float)d / (float)n_az, &s, &c);
                nominal_tap(s, R, r0, rho, (float)r, p.inv_dR, xb, delta, alpha);
                // plane of the lower (or nearest) bin; the fraction is taken of the offset from row r alone, which
                // the row number's magnitude would round off
                const float xr = delta * p.inv_dR, lf = linear ? floorf(xr) : floorf(xb + 0.5f) - (float)r;
                const int dq = (int)lf;
                top = max(top, dq + linear);
                const float wt = linear ? (dq == q ? 1.f - (xr - lf) : dq + 1 == q ? xr - lf : 0.f)
                                        : (dq == q ? 1.f : 0.f);
                if (wt != 0.f) {
                    const int e = d - off;            // >= 0 for an extended row, any sign for a circular one
                    g[e <= 0 ? -e : N - e] = cscale(nominal_weight(p.two_f_over_c, delta, alpha), wt * (1.f / (float)N));
                }
            }
            if (q == 0) {
                top = __reduce_max_sync(0xffffffffu, top);
                if ((threadIdx.x & 31) == 0) atomicMax(&s_top, top);
            }
            G::sync();
            dif_pass_c<N, N, R1, false, T, G>(g, tc, tf);
            dif_middle<N, s1, T, G, Rs...>(g, tc, tf);
#pragma unroll 1
            for (int b = G::tid(); b < NB; b += T) {  // last pass: blocks of RK, twiddles 1
                float2 v[RK];
#pragma unroll
                for (int i = 0; i < RK; ++i) v[i] = g[b * RK + i];
                small_dft<RK>(v);
#pragma unroll
                for (int i = 0; i < RK; ++i) g[b * RK + i] = v[i];
            }
            if (q == 0) griddep_wait();
        }
        if (__syncthreads_or(bad)) {
            bpa_row_direct(S, p, r, L, n_az, M_ap, linear != 0, rowph, reinterpret_cast<float4 *>(sm), N / 2, out);
            return;
        }
        const bool last = q >= min(s_top, L - 1 - r);
        if (grp_a) {
#pragma unroll 1
            for (int b = G::tid(); b < NB; b += T) {  // last pass of the S row, times the taps, onto the planes before
                float2 v[RK];
#pragma unroll
                for (int i = 0; i < RK; ++i) v[i] = x[b * RK + i];
                small_dft<RK>(v);
#pragma unroll
                for (int i = 0; i < RK; ++i) {
                    const float2 pr = cmul(g[b * RK + i], v[i]);
                    v[i] = q == 0 ? pr : cadd(y[b * RK + i], pr);
                }
                if (!last) {
#pragma unroll
                    for (int i = 0; i < RK; ++i) y[b * RK + i] = v[i];
                } else {                              // first pass of the inverse on the same block
#pragma unroll
                    for (int i = 0; i < RK; ++i) v[i].y = -v[i].y;
                    small_dft<RK>(v);
#pragma unroll
                    for (int i = 0; i < RK; ++i) x[b * RK + i] = v[i];
                }
            }
        }
        __syncthreads();
        if (last) break;
    }
    dit_middle<N, s1, 2 * T, WholeCta, Rs...>(x, tc, tf);
#pragma unroll 1
    for (int j = threadIdx.x; j < s1; j += 2 * T) {
        float2 v[R1], wq[R1];
        twiddle_powers<R1>(twiddle(j, tc, tf), wq);
        v[0] = x[j];
#pragma unroll
        for (int i = 1; i < R1; ++i) v[i] = cmul(x[j + i * s1], wq[i]);
        small_dft<R1>(v);
#pragma unroll
        for (int i = 0; i < R1; ++i) {
            const int e = j + i * s1;
            if (e < n_az) out[(size_t)r * n_az + e] = cmul(rowph, make_float2(v[i].x, -v[i].y));
        }
    }
}

using RowsFn = void (*)(const float2 *, BpaParams, int, int, int, int, int, int, float2 *);

struct RowsPlan {
    int N, threads;
    RowsFn fn;
    size_t smem;
    int *smem_done;
};

template <int T, int MINB, int N, int... R>
RowsPlan rows_plan() {
    static int done[kMaxDevices] = {};
    return RowsPlan{N, 2 * T, bpa_rows_kernel<T, MINB, N, R...>, bpa_rows_smem<N>(), done};
}

// Ascending lengths, at most 1.67 times apart; three passes each but for the longest.  Threads per group: the
// butterflies of a pass in one or two rounds.  Long rows hold one CTA of 2 x 256 threads an SM (128 registers) or
// two of 2 x 128; with at most two rows an SM the first is faster (3600 pulses, M = 600: 256 rows 24.5 against
// 26.4 us), with more the second (512 rows 36.8 against 42 us).
constexpr int kFewRows = 304;      // two per SM

const RowsPlan *find_rows(int n_rng, int n_az, int M_ap, bool *circular) {
    static const RowsPlan plans[] = {
        rows_plan<128, 2, 360, 8, 3, 15>(),      rows_plan<128, 2, 480, 8, 4, 15>(),
        rows_plan<128, 2, 600, 8, 5, 15>(),      rows_plan<128, 2, 720, 4, 12, 15>(),
        rows_plan<128, 2, 960, 8, 8, 15>(),      rows_plan<128, 2, 1200, 8, 10, 15>(),
        rows_plan<128, 2, 1440, 8, 12, 15>(),    rows_plan<128, 3, 1800, 8, 15, 15>(),
        rows_plan<256, 1, 2400, 16, 10, 15>(),   rows_plan<256, 1, 2880, 16, 12, 15>(),
        rows_plan<256, 1, 3600, 16, 15, 15>(),   rows_plan<256, 1, 4800, 8, 4, 10, 15>(),
        rows_plan<256, 1, 5760, 8, 4, 12, 15>(), rows_plan<256, 1, 7200, 8, 4, 15, 15>(),
    };
    static const RowsPlan many[] = {
        rows_plan<128, 2, 2400, 16, 10, 15>(), rows_plan<128, 2, 2880, 16, 12, 15>(),
        rows_plan<128, 2, 3600, 16, 15, 15>(),
    };
    int N = 0;
    for (const RowsPlan &p : plans)
        if (p.N == n_az) N = n_az;
    *circular = N != 0;
    for (const RowsPlan &p : plans)
        if (N == 0 && p.N >= n_az + M_ap - 1) N = p.N;
    if (n_rng > kFewRows)
        for (const RowsPlan &p : many)
            if (p.N == N) return &p;
    for (const RowsPlan &p : plans)
        if (p.N == N) return &p;
    return nullptr;
}

}  // namespace

// Where the transforms cost less than the direct sum.  A plane costs two transforms of the row, about 18 of the
// direct kernel's multiply-adds a pixel, and most rows have far fewer planes than row 0, whose count bounds them
// (R_n - rho <= 2 r0 sin(pi d/n_az) falls with rho): M >= 8 planes (whole ring of 97 pulses, 10 planes, 32 rows:
// 17.7 against 19.2 us direct; 3600 x 256, M = 24: 17.7 against 47.7).  Below about 2e6 pixel-pulses the direct
// kernel's one short wave is faster than a row's chain of transforms (360 x 64, M = 60: 8.6 against 9.3 us;
// 480 x 64, M = 80: 9.5 against 9.3; 800 x 64, M = 130: 14.0 against 9.9), and so is it for a few rows of few pulses
// (1800 x 32, M = 36: 8.6 against 9.2; 2500 x 32, M = 50: 11.0 against 11.5; 3600 x 32, M = 72: 15.0 against 12.2).
bool bpa_fft_applies(const BpaParams &p, int n_rng, int n_az, int M_ap) {
    bool circular;
    if (!find_rows(n_rng, n_az, M_ap, &circular)) return false;
    const double half = 3.14159265358979323846 * (double)(M_ap / 2) / (double)n_az;
    const double planes = 2.0 * p.r0 * sin(half) / p.dR + 2.0;
    return M_ap >= 8.0 * planes && (double)n_rng * n_az * M_ap >= 2e6 && (M_ap >= 64 || n_rng >= 40);
}

rosar_status launch_bpa_fft(const float2 *S, const BpaParams &p, int L, int n_rng, int n_az, int M_ap, int interp,
                            float2 *out, cudaStream_t s) {
    bool circular;
    const RowsPlan *pl = find_rows(n_rng, n_az, M_ap, &circular);
    rosar_status st = ensure_smem((const void *)pl->fn, pl->smem, pl->smem_done, "bpa");
    if (st != ROSAR_OK) return st;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_rng);
    cfg.blockDim = dim3(pl->threads);
    cfg.dynamicSmemBytes = pl->smem;
    cfg.stream = s;
    // the taps need nothing of the kernel before, which writes S: they start while it ends
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, pl->fn, S, p, L, n_az, M_ap, interp, circular ? 0 : -(M_ap / 2),
                                             circular ? n_az : n_az + M_ap - 1, out);
    if (e != cudaSuccess) return set_error(ROSAR_ERR_CUDA, "bpa: launch failed: %s", cudaGetErrorString(e));
    return check_launch("bpa");
}

}  // namespace rosar
