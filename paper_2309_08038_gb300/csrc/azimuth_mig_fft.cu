// K2mf: the range-migration-aware azimuth filter (arXiv 2309.08038, Sec. III-D: the
// per-pulse peak bin l*_n of Eq. (40) inside Eq. (43)) evaluated exactly in the
// azimuth-frequency domain.  Tap k of output row r reads range row r + dl[r][k];
// grouping the taps of row r by their row offset d,
//
//   out[r][.] = sum_d sum_{k: dl[r][k] = d} w[r][k] * S[r+d][(. + o_k) mod N]
//             = sum_d g_{r,d} (*) S[r+d][.],        g_{r,d}[(-o_k) mod N] += w[r][k]
//             = IFFT( sum_d FFT(S[r+d][.]) . FFT(g_{r,d})/N ),
//
// so one forward transform per S row (shared by every output row that reads it) and one
// inverse per output row replace the K-tap gather: the cost of the fixed-row FFT filter
// plus one product per plane d.  Rows r+d outside [0, n_bins) contribute nothing (they
// read zero, as in the gather form).
//
//   plan     H_d[r] = FFT(g_{r,d})/N for d = d_lo .. d_lo+n_d-1 (azimuth_plan_kernel with a
//            row-offset filter, azimuth_fft.cu), digit-reversed order as every plan here;
//   kernel 1 X[b] = DIF(S[b]) for every row b of S (the forward transform, same order);
//   kernel 2 Y_r = sum_d X[r+d] . H_d[r] in increasing d, then conj, DIT, conj (the
//            inverse, natural order), written to out[r].
// Every transform's outer pass runs on global memory where it can; the products are formed over consecutive elements
// (the plans' planes and the spectra are both in digit-reversed order), eight elements a thread and plane in flight.
// Each kernel is launched to overlap the one before it, and the second asks for its planes of H ahead of the wait,
// since they come from DRAM.  Bound by latency where the grid is short (256 rows of 3600 pulses are under two CTAs an
// SM), by the planes of H and the spectra (8 bytes each a plane and pixel) where it is long.  Against products formed
// per butterfly (strided reads of H and X), staged rows with run-time plans and no overlap of the first kernel: 3600
// pulses, three planes, 256 rows 20.4 -> 13.0 us, 512 rows 34.8 -> 20.4; 7200 x 256 43.8 -> 28.3; run-time plans 2048
// x 1024 81 -> 36, 12000 x 128 46.5 -> 32.2, 480 x 256 10.6 -> 9.7.

#include "azimuth_layout.cuh"

namespace rosar {
namespace {

using namespace rowfft;

// ---- the two halves around the transforms

template <int T>
__device__ __forceinline__ void store_row(const float2 *x, float2 *__restrict__ X, int N, int pad_shift) {
    for (int n = threadIdx.x; n < N; n += T) X[n] = x[rpad(n, pad_shift)];
}

// x = conj(sum_d H_d[r] . X[r + d]) over the planes whose rows exist, in increasing d; ends without a barrier.
struct Planes {
    const float2 *X, *H;
    int n_bins, n_rng, d_lo, n_d;
};

__device__ __forceinline__ void prefetch_planes(const Planes &p, int r, int N, int T) {
    for (int i = 0; i < p.n_d; ++i) {
        const char *h = reinterpret_cast<const char *>(p.H + ((size_t)i * p.n_rng + r) * N);
        for (int b = 128 * threadIdx.x; b < 8 * N; b += 128 * T) asm volatile("prefetch.global.L2 [%0];" ::"l"(h + b));
    }
}

__device__ __forceinline__ void sum_planes(const Planes &p, int r, int N, int T, int pad_shift, float2 *x) {
    constexpr int E = 8;
    const int i_lo = max(0, -(r + p.d_lo)), i_hi = min(p.n_d, p.n_bins - r - p.d_lo);
    for (int n0 = threadIdx.x; n0 < N; n0 += E * T) {
        float2 acc[E];
#pragma unroll
        for (int e = 0; e < E; ++e) acc[e] = make_float2(0.f, 0.f);
        for (int i = i_lo; i < i_hi; ++i) {
            const float2 *Xr = p.X + (size_t)(r + p.d_lo + i) * N, *Hr = p.H + ((size_t)i * p.n_rng + r) * N;
            float2 h[E], v[E];
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int n = n0 + e * T;
                h[e] = n < N ? __ldg(Hr + n) : make_float2(0.f, 0.f);
                v[e] = n < N ? __ldcg(Xr + n) : make_float2(0.f, 0.f);
            }
#pragma unroll
            for (int e = 0; e < E; ++e) acc[e] = i == i_lo ? cmul(h[e], v[e]) : cadd(acc[e], cmul(h[e], v[e]));
        }
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (n0 + e * T < N) x[rpad(n0 + e * T, pad_shift)] = make_float2(acc[e].x, -acc[e].y);
    }
}

// ---- compile-time plans

// The pass on blocks of RK (twiddles 1) in place.
template <int N, int RK, int T>
__device__ __forceinline__ void inner_pass(float2 *x) {
#pragma unroll 1
    for (int b = threadIdx.x; b < N / RK; b += T) {
        float2 v[RK];
#pragma unroll
        for (int q = 0; q < RK; ++q) v[q] = x[b * RK + q];
        small_dft<RK>(v);
#pragma unroll
        for (int q = 0; q < RK; ++q) x[b * RK + q] = v[q];
    }
    __syncthreads();
}

template <int T, int MINB, int N, int R1, int... Rs>
__global__ void __launch_bounds__(T, MINB)
azimuth_spectrum_fixed_kernel(const float2 *__restrict__ S, float2 *__restrict__ X) {
    extern __shared__ float2 sm[];
    griddep_launch_dependents();
    const size_t row = (size_t)blockIdx.x * N;
    const float2 *tc, *tf;
    build_twiddles(N, false, sm + N, &tc, &tf);
    __syncthreads();
    griddep_wait();                                  // S is complete, X no longer read
    dif_first_global<N, R1, T, false>(S + row, sm, tc, tf);
    dif_middle<N, N / R1, T, WholeCta, Rs...>(sm, tc, tf);
    inner_pass<N, last_radix<R1, Rs...>(), T>(sm);
    store_row<T>(sm, X + row, N, 31);
}

template <int T, int MINB, int N, int R1, int... Rs>
__global__ void __launch_bounds__(T, MINB)
azimuth_mig_combine_fixed_kernel(Planes p, float2 *__restrict__ out) {
    extern __shared__ float2 sm[];
    const int r = blockIdx.x;
    prefetch_planes(p, r, N, T);
    const float2 *tc, *tf;
    build_twiddles(N, false, sm + N, &tc, &tf);
    griddep_wait();                                  // X is complete
    sum_planes(p, r, N, T, 31, sm);
    __syncthreads();
    inner_pass<N, last_radix<R1, Rs...>(), T>(sm);
    dit_middle<N, N / R1, T, WholeCta, Rs...>(sm, tc, tf);
    dit_last_global<N, R1, T>(sm, out + (size_t)r * N, tc, tf);
}

// ---- run-time plans (blockDim.x threads); a plan of one pass (n_az <= 16) has no outer pass to keep on global memory

template <bool PAD>
__device__ __forceinline__ void runtime_spectrum(const float2 *src, float2 *x, int N, const RowPlan &pl,
                                                 const float2 *tc, const float2 *tf) {
    int M = N;
    if (pl.npass > 1) {
#define ROSAR_FIRST(R) rt_first<R, PAD>(src, x, N, tc, tf, nullptr)
        ROSAR_FOR_RADIX(pl.rad[0], ROSAR_FIRST)
#undef ROSAR_FIRST
        M /= pl.rad[0];
    } else {
        for (int n = threadIdx.x; n < N; n += blockDim.x) x[cpad<PAD>(n)] = __ldcg(src + n);
    }
    __syncthreads();
    for (int p = pl.npass > 1; p < pl.npass; ++p) {
        stage<true, PAD>(pl.rad[p], x, N, M, tc, tf);
        M /= pl.rad[p];
    }
}

template <bool PAD>
__device__ __forceinline__ void runtime_inverse(float2 *x, float2 *dst, int N, const RowPlan &pl, const float2 *tc,
                                                const float2 *tf) {
    int M = 1;
    for (int p = pl.npass - 1; p >= (pl.npass > 1); --p) {
        M *= pl.rad[p];
        stage<false, PAD>(pl.rad[p], x, N, M, tc, tf);
    }
    if (pl.npass > 1) {
#define ROSAR_LAST(R) rt_last<R, PAD>(x, dst, N, tc, tf)
        ROSAR_FOR_RADIX(pl.rad[0], ROSAR_LAST)
#undef ROSAR_LAST
    } else {
        for (int n = threadIdx.x; n < N; n += blockDim.x) {
            const float2 y = x[cpad<PAD>(n)];
            dst[n] = make_float2(y.x, -y.y);
        }
    }
}

template <int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB)
azimuth_spectrum_kernel(const float2 *__restrict__ S, int N, RowPlan pl, float2 *__restrict__ X) {
    extern __shared__ float2 sm[];
    griddep_launch_dependents();
    const size_t row = (size_t)blockIdx.x * N;
    const float2 *tc, *tf;
    build_twiddles(N, false, sm + padded_len(N), &tc, &tf);
    __syncthreads();
    griddep_wait();
    if (pl.pad_shift == 4) runtime_spectrum<true>(S + row, sm, N, pl, tc, tf);
    else runtime_spectrum<false>(S + row, sm, N, pl, tc, tf);      // both end with a barrier
    for (int n = threadIdx.x; n < N; n += blockDim.x) X[row + n] = sm[rpad(n, pl.pad_shift)];
}

template <int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB)
azimuth_mig_combine_kernel(Planes p, int N, RowPlan pl, float2 *__restrict__ out) {
    extern __shared__ float2 sm[];
    const int r = blockIdx.x;
    prefetch_planes(p, r, N, blockDim.x);
    const float2 *tc, *tf;
    build_twiddles(N, false, sm + padded_len(N), &tc, &tf);
    griddep_wait();
    sum_planes(p, r, N, blockDim.x, pl.pad_shift, sm);
    __syncthreads();
    if (pl.pad_shift == 4) runtime_inverse<true>(sm, out + (size_t)r * N, N, pl, tc, tf);
    else runtime_inverse<false>(sm, out + (size_t)r * N, N, pl, tc, tf);
}

// ---- launches

size_t row_smem(int N) { return sizeof(float2) * (size_t)(padded_len(N) + 64 + coarse_len(N)); }

struct MigCall {
    const float2 *S;
    Planes p;
    float2 *X, *out;
    int N;
    cudaStream_t s;
};

template <typename KA, typename KB, typename... A>
rosar_status launch_pair(const MigCall &c, KA spectrum, KB combine, int T, int (*done)[kMaxDevices], A... plan) {
    const char *what = "sparse_azimuth_migrating_fft";
    const size_t sm = row_smem(c.N);
    rosar_status st = ensure_smem((const void *)spectrum, sm, done[0], what);
    if (st == ROSAR_OK) st = ensure_smem((const void *)combine, sm, done[1], what);
    if (st != ROSAR_OK) return st;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c.p.n_bins);
    cfg.blockDim = dim3(T);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = c.s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, spectrum, c.S, plan..., c.X);
    cfg.gridDim = dim3(c.p.n_rng);
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, combine, c.p, plan..., c.out);
    if (e != cudaSuccess) return set_error(ROSAR_ERR_CUDA, "%s: launch failed: %s", what, cudaGetErrorString(e));
    return check_launch(what);
}

template <int T, int MINB, int N, int... R>
rosar_status launch_fixed(const MigCall &c) {
    static int done[2][kMaxDevices] = {};
    return launch_pair(c, azimuth_spectrum_fixed_kernel<T, MINB, N, R...>, azimuth_mig_combine_fixed_kernel<T, MINB, N, R...>,
                       T, done);
}

template <int MAXT, int MINB>
rosar_status launch_runtime(const MigCall &c, const RowPlan &pl, int T) {
    static int done[2][kMaxDevices] = {};
    return launch_pair(c, azimuth_spectrum_kernel<MAXT, MINB>, azimuth_mig_combine_kernel<MAXT, MINB>, T, done, c.N, pl);
}

constexpr int kFewRows = 304;      // as the row filter: up to two rows an SM a row's own latency counts

}  // namespace

rosar_status launch_sparse_azimuth_migrating_fft(const float2 *S, int n_bins, const float2 *H, int d_lo, int n_d,
                                                 int n_rng, int n_az, float2 *X, float2 *out, cudaStream_t s) {
    RowPlan pl;
    if (!make_plan(n_az, &pl))
        return set_error(ROSAR_ERR_UNSUPPORTED, "sparse_azimuth_migrating_fft: n_az=%d is not 2^a 3^b 5^c in [2, %d]",
                         n_az, AF_MAX_N);
    const MigCall c{S, Planes{X, H, n_bins, n_rng, d_lo, n_d}, X, out, n_az, s};
    const bool few = n_rng <= kFewRows;
    if (Row3600::is(n_az, pl)) return launch_fixed<256, 4, 3600, 16, 15, 15>(c);
    if (Row1800::is(n_az, pl))
        return few ? launch_fixed<256, 4, 1800, 8, 15, 15>(c) : launch_fixed<128, 8, 1800, 8, 15, 15>(c);
    if (Row7200::is(n_az, pl)) return launch_fixed<256, 3, 7200, 8, 4, 15, 15>(c);
    if (Row360::is(n_az, pl)) return launch_fixed<128, 8, 360, 8, 3, 15>(c);
    // 128 threads up to 2048: 480 x 256 9.7 us against 12.2 on 256, 1024 x 256 10.1 against 12.3, 1125 x 512 17.0 each.
    if (n_az <= 4096) return launch_runtime<256, 3>(c, pl, n_az <= 2048 ? 128 : 256);
    if (n_az <= 8192 && !few) return launch_runtime<256, 3>(c, pl, 256);
    return launch_runtime<512, 1>(c, pl, 512);
}

}  // namespace rosar
