// K2b: the sparse-aperture azimuth filter of Eq. (43) evaluated exactly as a circular
// convolution in the azimuth-frequency domain (arXiv 2309.08038, Sec. III-D; the
// pixel-parallel form of Remark 2, here per range row):
//
//   out[r][.] = sum_k w[r][k] * S[r][(. + o_k) mod N] = g_r (*) S[r][.],   g_r[(-o_k) mod N] += w[r][k]
//            = IFFT_N( FFT_N(g_r)/N . FFT_N(S[r][.]) )
//
// The same taps, the same circular modulo; only the summation order differs from the
// gather form.  Work per pixel is O(log N) instead of O(K), so at K >= 32 the
// azimuth stage turns from shared-memory/FMA bound to HBM bound (24 B/px: S, H, out).
//
// One CTA owns one range row, staged in shared memory (one pad element per 16
// against bank conflicts).  The forward transform is an in-place mixed-radix
// decimation-in-frequency FFT (radices 16, 8, 4, 2, 5, 3 and a prime-factor 15; N = 2^a 3^b 5^c <= 16384;
// a planner picks the sequence with the fewest passes, e.g. 3600 = 16*15*15).
// Every butterfly reads and writes the same R slots, so only its own R values are
// live and passes need one barrier each; its twiddles are powers of one table entry.  It leaves the spectrum in digit-reversed
// order; H is produced by the same transform (so it is stored in that order), the
// pointwise product needs no reordering, and the inverse is the transposed
// (decimation-in-time) pass sequence between two conjugations, which restores the
// natural order.  Twiddles exp(-2*pi*i*q/N) come from a two-level shared table
// (q >> 6, q & 63) built per CTA with sincospif.

#include "azimuth_layout.cuh"
#include "batch_rows.cuh"

namespace rosar {
namespace {

using namespace rowfft;

// What one CTA filters: a row of S through a row of H (conj_h: conj(H), the adjoint filter) into a row of out, which
// may be the row of S itself.  phase (optional): [N] per-column factors applied as the row is loaded.  spec (optional):
// [N] receives the row's forward transform (digit-reversed order, before the product with H), for the weight gradient.
struct RowRef {
    const float2 *S, *H;
    float2 *out;
    bool conj_h;
    const float2 *phase;
    float2 *spec;
};

// Rows of a stack: row b of S and out uses row (b mod h_rows) of H (a stack of scans sharing one plan) and phase row
// b / h_rows (each scan its own phase correction); phase [n_rows / h_rows][N], spec [n_rows][N].
struct StackRows {
    const float2 *S, *H;
    float2 *out;
    int h_rows, conj_h;
    const float2 *phase;
    float2 *spec;

    __device__ __forceinline__ RowRef at(int b, int N) const {
        const size_t row = (size_t)b * N;
        return RowRef{S + row, H + (size_t)(b % h_rows) * N, out + row, conj_h != 0,
                      phase ? phase + (size_t)(b / h_rows) * N : nullptr, spec ? spec + row : nullptr};
    }
};

// Rows of the scans of a batch that have this length, each scan with its own plan.
struct BatchRows {
    ScanGroup g;

    __device__ __forceinline__ RowRef at(int b, int N) const {
        int r;
        const ScanDev &sc = g.find(b, r);
        const size_t row = (size_t)r * N;
        return RowRef{sc.S + row, sc.H + row, sc.out + row, false, nullptr, nullptr};
    }
};

// The row filter on one CTA with a run-time plan: stage the twiddle table and (few rows) the H row, wait for S, then
// forward DIF, product with H (digit-reversed order, carries 1/N) between conjugations, DIT.
template <typename ROWS, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB)
azimuth_fft_kernel(ROWS rows, int N, RowPlan pl, Layout lay) {
    extern __shared__ float2 sm[];
    const int T = blockDim.x;
    const int pad_shift = pl.pad_shift;
    float2 *x = sm;
    float2 *hb = x + padded_len(N);
    float2 *tw = lay.stage_h ? hb + padded_len(N) : hb;
    const RowRef ref = rows.at(blockIdx.x, N);
    const float hs = ref.conj_h ? -1.f : 1.f;
    // prologue independent of S
    if (lay.stage_h)
        for (int n = threadIdx.x; n < N; n += T) cp_async8(hb + rpad(n, pad_shift), ref.H + n);
    cp_async_commit();
    const float2 *tc, *tf;
    build_twiddles(N, lay.full_tab != 0, tw, &tc, &tf);
    __syncthreads();
    griddep_wait();                          // S is complete (no-op unless launched to overlap its producer)
    if (pl.npass == 1) {                     // one butterfly: N itself a radix
        cp_async_wait<0>();
        for (int n = threadIdx.x; n < N; n += T) {
            const float2 v = __ldcg(ref.S + n);
            x[rpad(n, pad_shift)] = ref.phase ? cmul(v, __ldg(ref.phase + n)) : v;
        }
        __syncthreads();
        row_dif(x, N, pl, tc, tf);
        for (int n = threadIdx.x; n < N; n += T) {
            float2 h = __ldg(ref.H + n);
            h.y *= hs;
            if (ref.spec) ref.spec[n] = x[rpad(n, pad_shift)];
            const float2 y = cmul(h, x[rpad(n, pad_shift)]);
            x[rpad(n, pad_shift)] = make_float2(y.x, -y.y);
        }
        __syncthreads();
        row_dit(x, N, pl, tc, tf);
        for (int n = threadIdx.x; n < N; n += T) {
            const float2 y = x[rpad(n, pad_shift)];
            ref.out[n] = make_float2(y.x, -y.y);
        }
        return;
    }
    const float2 *h = lay.stage_h ? hb : ref.H;
    if (pad_shift == 4)
        row_filter_runtime<true>(ref.S, h, lay.stage_h, hs, x, ref.out, N, pl, tc, tf, ref.phase, ref.spec);
    else
        row_filter_runtime<false>(ref.S, h, lay.stage_h, hs, x, ref.out, N, pl, tc, tf, ref.phase, ref.spec);
}

// Compile-time plan for one row length (T threads, no padding: N has an odd factor): the first pass reads S from
// global memory, the last writes the image, and the last forward pass, the product with H and the first inverse pass
// run as one step (row_filter_fused): four barriers for 16.15.15.  H_FROM: where H is read (HSource).  PAIRED:
// the two outermost passes of each transform in registers (row_filter_paired).
template <typename ROWS, int T, int MINB, int N, int H_FROM, bool PAIRED, int... R>
__global__ void __launch_bounds__(T, MINB)
azimuth_fft_fixed_kernel(ROWS rows) {
    extern __shared__ float2 sm[];
    const RowRef ref = rows.at(blockIdx.x, N);
    filter_row_cta<T, N, H_FROM, PAIRED, R...>(ref.S, ref.H, ref.conj_h, ref.out, sm, ref.phase, ref.spec);
}

}  // namespace

namespace {

template <typename K, typename... A>
cudaError_t launch_overlapped(K kernel, int grid, int threads, size_t smem, bool overlap, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// One launch of a row filter over n_rng rows; `only_prepare`: set the kernel's shared-memory limit and launch nothing.
struct RowLaunch {
    int n_az, n_rng;
    bool overlap, only_prepare;
    cudaStream_t s;
};

template <typename ROWS, int T, int MINB, int N, int H_FROM, bool PAIRED, int... R>
rosar_status launch_fixed(const RowLaunch &l, const ROWS &rows) {
    static int done[kMaxDevices] = {};
    constexpr size_t smem = filter_row_smem<N, H_FROM>();
    static_assert(smem <= 200 * 1024, "the staged rows exceed the shared-memory cap");
    const auto kernel = azimuth_fft_fixed_kernel<ROWS, T, MINB, N, H_FROM, PAIRED, R...>;
    rosar_status st = ensure_smem((const void *)kernel, smem, done, "azimuth_fft");
    if (st != ROSAR_OK || l.only_prepare) return st;
    const cudaError_t e = launch_overlapped(kernel, l.n_rng, T, smem, l.overlap, l.s, rows);
    if (e != cudaSuccess) return set_error(ROSAR_ERR_CUDA, "azimuth_fft: launch failed: %s", cudaGetErrorString(e));
    return check_launch("azimuth_fft");
}

template <typename ROWS, int MAXT, int MINB>
rosar_status launch_runtime(const RowLaunch &l, const ROWS &rows, const RowPlan &pl, const Layout &lay, int T) {
    static int done[kMaxDevices] = {};
    const auto kernel = azimuth_fft_kernel<ROWS, MAXT, MINB>;
    rosar_status st = ensure_smem((const void *)kernel, lay.bytes, done, "azimuth_fft");
    if (st != ROSAR_OK || l.only_prepare) return st;
    const cudaError_t e = launch_overlapped(kernel, l.n_rng, T, lay.bytes, l.overlap, l.s, rows, l.n_az, pl, lay);
    if (e != cudaSuccess) return set_error(ROSAR_ERR_CUDA, "azimuth_fft: launch failed: %s", cudaGetErrorString(e));
    return check_launch("azimuth_fft");
}

// The run-time plan: the staged H row pays where a row's own latency counts, up to two rows an SM.  Against loading the
// row, the passes, the product and the store as steps of their own: 800 pulses, 256 rows 8.3 -> 7.1 us, 2048 rows 47 ->
// 22; 4500: 23.9 -> 19.7 and 165 -> 89; 16384: 76 -> 51 (256 rows).
template <typename ROWS>
rosar_status launch_rows_runtime(const RowLaunch &l, const ROWS &rows, const RowPlan &pl) {
    const bool few = l.n_rng <= 304;
    const Layout lay = layout_for(l.n_az, few);
    if (l.n_az <= 4096) return launch_runtime<ROWS, 256, 3>(l, rows, pl, lay, !few && l.n_az <= 2048 ? 128 : 256);
    if (l.n_az <= 8192 && !few) return launch_runtime<ROWS, 256, 3>(l, rows, pl, lay, 256);
    // two rows an SM up to about 14200: 1024 rows of 9000 120 -> 92 us, of 12000 152 -> 121, of 13500 158 -> 156
    if (!few && 2 * (lay.bytes + 1024) <= 228 * 1024) return launch_runtime<ROWS, 512, 2>(l, rows, pl, lay, 512);
    return launch_runtime<ROWS, 512, 1>(l, rows, pl, lay, 512);
}

// Up to three rows an SM, a row's own latency counts: 256 threads and H staged while S is awaited.  With more the SM's
// rows in flight count: one row of shared memory and at most 64 registers hold 4 CTAs of 3600 pulses (46 % of the warps
// instead of 30) or 8 of 1800, and H is read in the fused step.  4096 rows of 3600 pulses 82 -> 77 us, 8192 of 1800 97 ->
// 76; 305 rows of 360 3.50 and 3.69, 400 rows of 1800 6.38 and 6.61, but 457 rows 5.13 and 3.82, 8.43 and 7.61.
// 7200-pulse rows hold one CTA an SM with H staged: 152 rows 10.2 us (11.3 not staged).  With more rows three CTAs an SM
// and the passes of radix 8 and 4 together in registers (PAIRED): 256 rows 18.4 -> 15.8 -> 13.8, 1024 rows 72 -> 54 ->
// 47, 4096 rows 271 -> 186 -> 159 (176 on two CTAs).
constexpr int kFewRows = 456;

template <typename ROWS>
rosar_status launch_rows_of(const RowLaunch &l, const ROWS &rows) {
    RowPlan pl;
    if (!make_plan(l.n_az, &pl))
        return set_error(ROSAR_ERR_UNSUPPORTED, "azimuth_fft: n_az=%d is not 2^a 3^b 5^c in [2, %d]", l.n_az, AF_MAX_N);
    const bool few = l.n_rng <= kFewRows;
    if (stored_radix(l.n_az, pl) == 0) return launch_rows_runtime<ROWS>(l, rows, pl);
    if (Row3600::is(l.n_az, pl))
        return few ? launch_fixed<ROWS, 256, 2, 3600, kStaged, false, 16, 15, 15>(l, rows)
                   : launch_fixed<ROWS, 256, 4, 3600, kFused, false, 16, 15, 15>(l, rows);
    if (Row1800::is(l.n_az, pl))
        return few ? launch_fixed<ROWS, 256, 2, 1800, kStaged, false, 8, 15, 15>(l, rows)
                   : launch_fixed<ROWS, 128, 8, 1800, kFused, false, 8, 15, 15>(l, rows);
    if (Row7200::is(l.n_az, pl))
        return l.n_rng <= 152 ? launch_fixed<ROWS, 512, 1, 7200, kStaged, false, 8, 4, 15, 15>(l, rows)
                              : launch_fixed<ROWS, 256, 3, 7200, kFused, true, 8, 4, 15, 15>(l, rows);
    // 14400: one row an SM on 1024 threads, or two on 512 each.  152 rows 15.8 us (17.0 streamed); 256 rows 32.8 -> 28.9,
    // 1024 rows 130 -> 115 (two rows an SM with the fused step 133, one with the streamed step 140).
    if (Row14400::is(l.n_az, pl))
        return l.n_rng <= 152 ? launch_fixed<ROWS, 1024, 1, 14400, kFused, false, 8, 8, 15, 15>(l, rows)
                              : launch_fixed<ROWS, 512, 2, 14400, kStreamed, false, 8, 8, 15, 15>(l, rows);
    return few ? launch_fixed<ROWS, 256, 2, 360, kStaged, false, 8, 3, 15>(l, rows)
               : launch_fixed<ROWS, 64, 8, 360, kFused, false, 8, 3, 15>(l, rows);
}

}  // namespace

rosar_status launch_azimuth_fft(const float2 *S, const float2 *H, int n_rng, int n_az, float2 *out, cudaStream_t s,
                                bool overlap_predecessor, int h_rows, bool conj_h, const float2 *phase, float2 *spec) {
    return launch_rows_of(RowLaunch{n_az, n_rng, overlap_predecessor, false, s},
                          StackRows{S, H, out, h_rows > 0 ? h_rows : n_rng, conj_h ? 1 : 0, phase, spec});
}

rosar_status launch_azimuth_group(int n_az, const ScanGroup &g, int total, cudaStream_t s, bool prepare) {
    return launch_rows_of(RowLaunch{n_az, total, false, prepare, s}, BatchRows{g});
}

}  // namespace rosar
