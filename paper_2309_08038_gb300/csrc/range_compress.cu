// K1: range compression of every pulse (arXiv 2309.08038, Sec. III-D, Eq. (38)).
//
//   S[l][n] = c_l * sum_m win[m] * raw[n][m] * exp(-j*2*pi*l*m/L),  c_l = exp(+j*pi*l*(L-1)/L)
//
// One CTA transforms P consecutive pulses.  Each pulse uses T = L/16 threads that
// hold 16 complex samples each in registers; the FFT is a Stockham auto-sort
// sequence of radix-16 passes (plus one radix-2/4/8 pass when log2(L) is not a
// multiple of 4), each an in-register DFT followed by an exchange through shared
// memory.  The window is applied as samples are loaded from HBM; the centring
// phase c_l is applied in the last pass, which writes the tile transposed
// ([l][p]) so that the store to the range-major S[l][n0..n0+P) is coalesced
// along azimuth.  Twiddles come from a two-level per-CTA table of exp(-j*pi*q/L)
// (32 + 2L/32 entries, built with sincospif), one lookup per butterfly raised to
// powers.  (fft_tile.cuh holds the tile itself.)
//
// Memory-bound: 16 algorithmic bytes per sample (8 read, 8 written).

#include "batch_rows.cuh"
#include "fft_tile.cuh"

namespace rosar {
namespace {

// Pulses per CTA for the standalone kernel: small tiles give enough CTAs to cover
// the memory latency at the scan sizes of interest.  L = 1024 takes 8 pulses (stores of 64 bytes instead of 32) on 512
// threads at 64 registers, two CTAs an SM: 14400 pulses 55.0 -> 52.2 us, or HALF of them (half_tiles below).
template <int L, bool HALF = false>
struct Plan : fft::Tile<L, (L <= 16 ? 32 : L <= 64 ? 16 : L <= 256 ? 8 : L == 512 || (L == 1024 && HALF) ? 4
                            : L == 1024 ? 8 : 2)> {
    // 0: none asked for.  A minimum of one lets the compiler spend 98 registers on L = 256 where it takes 80: 16 scans of
    // 3600 pulses 39.8 -> 45.7 us.
    static constexpr int MINB = L == 1024 && !HALF ? 2 : 0;
};

template <int L, bool HALF>
__global__ void __launch_bounds__(Plan<L, HALF>::THREADS, Plan<L, HALF>::MINB)
range_compress_kernel(const float2 *__restrict__ raw, const float *__restrict__ win, int n_az, int centred,
                      float2 *__restrict__ S, int vec_store) {
    extern __shared__ float2 smem[];
    const size_t scan = (size_t)blockIdx.y * n_az * L;      // grid.y: scans of a stack
    constexpr int P = Plan<L, HALF>::P;
    fft::range_tile<L, P>(raw + scan, win, n_az, centred != 0, S + scan, blockIdx.x * P, smem, true, vec_store != 0);
}

// The same over the scans of a batch that have this length.
template <int L>
__global__ void __launch_bounds__(Plan<L>::THREADS, Plan<L>::MINB)
range_group_kernel(ScanGroup g) {
    extern __shared__ float2 smem[];
    int tile;
    const ScanDev &sc = g.find(blockIdx.x, tile);
    fft::range_tile<L, Plan<L>::P>(sc.raw, sc.win, sc.n_az, true, sc.S, tile * Plan<L>::P, smem, true, sc.vec_store != 0);
}

template <int L>
rosar_status launch_group_L(const ScanGroup &g, int total, cudaStream_t s, bool prepare) {
    using PL = Plan<L>;
    static int done[kMaxDevices] = {};
    rosar_status st = ensure_smem((const void *)range_group_kernel<L>, PL::SMEM, done, "batch range compression");
    if (st != ROSAR_OK || prepare) return st;
    range_group_kernel<L><<<total, PL::THREADS, PL::SMEM, s>>>(g);
    return check_launch("batch range compression");
}

// Pulses a CTA of the adjoint: 8 are a 64-byte segment of a bin's row (from L = 1024 on 4 run faster), and 4 consecutive
// samples of a pulse's are a sector.  Bound by memory: 16 scans of 3600 x 256 82 -> 54.6 us (of 35 at the copy rate),
// x 128 49 -> 28.7, 8 scans of x 512 109 -> 66 (75 on two CTAs an SM), 14400 x 1024 102 -> 63 (72 with 8 pulses a CTA),
// against bins staged pulse by pulse in shared memory before the first pass and after the last.
template <int L>
struct AdjointPlan : fft::Tile<L, (L <= 16 ? 32 : L <= 32 ? 16 : L <= 512 ? 8 : L <= 2048 ? 4 : 2)> {
    using Base = fft::Tile<L, (L <= 16 ? 32 : L <= 32 ? 16 : L <= 512 ? 8 : L <= 2048 ? 4 : 2)>;
    static constexpr size_t SMEM = sizeof(float2) * (size_t)(Base::TAB + Base::P * Base::LP);
};

template <int L>
__global__ void __launch_bounds__(AdjointPlan<L>::THREADS, L == 512 ? 3 : 0)
range_adjoint_kernel(const float2 *__restrict__ g, const float *__restrict__ win, int n_az, int centred,
                     float2 *__restrict__ grad_raw) {
    extern __shared__ float2 smem[];
    const size_t scan = (size_t)blockIdx.y * n_az * L;      // grid.y: scans of a stack
    constexpr int P = AdjointPlan<L>::P;
    fft::range_adjoint_tile<L, P>(g + scan, win, n_az, centred != 0, grad_raw + scan, blockIdx.x * P, smem);
}

template <int L>
rosar_status launch_adjoint_L(const float2 *g, const float *win, int n_az, int centred, float2 *grad_raw,
                              cudaStream_t s, int n_scans) {
    using PL = AdjointPlan<L>;
    static_assert(PL::SMEM <= 227 * 1024, "range-adjoint tile exceeds shared memory");
    if (PL::SMEM > 48 * 1024) {
        static int done[kMaxDevices] = {};
        rosar_status st = ensure_smem((const void *)range_adjoint_kernel<L>, PL::SMEM, done, "range_compress_adjoint");
        if (st != ROSAR_OK) return st;
    }
    const dim3 grid((n_az + PL::P - 1) / PL::P, n_scans);
    range_adjoint_kernel<L><<<grid, PL::THREADS, PL::SMEM, s>>>(g, win, n_az, centred, grad_raw);
    return check_launch("range_compress_adjoint");
}

template <int L, bool HALF>
rosar_status launch_plan(const float2 *raw, const float *win, int n_az, int centred, float2 *S, cudaStream_t s,
                         int n_scans, bool vec) {
    using PL = Plan<L, HALF>;
    static_assert(PL::SMEM <= 227 * 1024, "range-compress tile exceeds shared memory");
    if (PL::SMEM > 48 * 1024) {
        static int done[kMaxDevices] = {};
        rosar_status st = ensure_smem((const void *)range_compress_kernel<L, HALF>, PL::SMEM, done, "range_compress");
        if (st != ROSAR_OK) return st;
    }
    const dim3 grid((n_az + PL::P - 1) / PL::P, n_scans);
    range_compress_kernel<L, HALF><<<grid, PL::THREADS, PL::SMEM, s>>>(raw, win, n_az, centred, S, vec ? 1 : 0);
    return check_launch("range_compress");
}

// L = 1024: tiles of 4 pulses instead of 8 where the fullest SM would hold half of a last tile of 8 (an odd number of
// tiles of 4 on it), and for rows of an odd stride, whose stores are single: 360 pulses 5.7 against 4.1 us, 1000 6.0 and
// 6.0, 1800 8.9 and 7.7, 2000 9.3 and 10.3, 2800 13.2 and 12.6, 3600 13.5 and 14.7, 7200 28.0 and 29.3; 1501 9.5 and 7.5,
// 3607 13.9 and 13.3, 10001 38.8 and 38.5.
bool half_tiles(int n_az, int n_scans, bool vec) {
    const long long tiles = (long long)n_scans * ((n_az + 3) / 4);
    return !vec || ((tiles + 151) / 152) % 2 == 1;
}

template <int L>
rosar_status launch_L(const float2 *raw, const float *win, int n_az, int centred, float2 *S, cudaStream_t s,
                      int n_scans) {
    const bool vec = n_az % 2 == 0 && (reinterpret_cast<uintptr_t>(S) & 15) == 0;
    if constexpr (L == 1024)
        if (half_tiles(n_az, n_scans, vec)) return launch_plan<L, true>(raw, win, n_az, centred, S, s, n_scans, vec);
    return launch_plan<L, false>(raw, win, n_az, centred, S, s, n_scans, vec);
}

}  // namespace

rosar_status launch_range_compress(const float2 *raw, const float *win, int n_az, int L, int centred, float2 *S,
                                   cudaStream_t s, int n_scans) {
    if (n_scans < 1 || n_scans > 65535)
        return set_error(ROSAR_ERR_UNSUPPORTED, "range_compress: n_scans=%d not in [1, 65535]", n_scans);
    switch (L) {
        case 8: return launch_L<8>(raw, win, n_az, centred, S, s, n_scans);
        case 16: return launch_L<16>(raw, win, n_az, centred, S, s, n_scans);
        case 32: return launch_L<32>(raw, win, n_az, centred, S, s, n_scans);
        case 64: return launch_L<64>(raw, win, n_az, centred, S, s, n_scans);
        case 128: return launch_L<128>(raw, win, n_az, centred, S, s, n_scans);
        case 256: return launch_L<256>(raw, win, n_az, centred, S, s, n_scans);
        case 512: return launch_L<512>(raw, win, n_az, centred, S, s, n_scans);
        case 1024: return launch_L<1024>(raw, win, n_az, centred, S, s, n_scans);
        case 2048: return launch_L<2048>(raw, win, n_az, centred, S, s, n_scans);
        case 4096: return launch_L<4096>(raw, win, n_az, centred, S, s, n_scans);
        default: return set_error(ROSAR_ERR_UNSUPPORTED, "range_compress: L=%d is not a power of two in [8, 4096]", L);
    }
}

int range_group_pulses(int L) {
    switch (L) {
        case 16: return Plan<16>::P;
        case 32: return Plan<32>::P;
        case 64: return Plan<64>::P;
        case 128: return Plan<128>::P;
        case 256: return Plan<256>::P;
        case 512: return Plan<512>::P;
        case 1024: return Plan<1024>::P;
        default: return Plan<2048>::P;
    }
}

rosar_status launch_range_group(int L, const ScanGroup &g, int total, cudaStream_t s, bool prepare) {
    switch (L) {
        case 16: return launch_group_L<16>(g, total, s, prepare);
        case 32: return launch_group_L<32>(g, total, s, prepare);
        case 64: return launch_group_L<64>(g, total, s, prepare);
        case 128: return launch_group_L<128>(g, total, s, prepare);
        case 256: return launch_group_L<256>(g, total, s, prepare);
        case 512: return launch_group_L<512>(g, total, s, prepare);
        case 1024: return launch_group_L<1024>(g, total, s, prepare);
        default: return launch_group_L<2048>(g, total, s, prepare);
    }
}

rosar_status launch_range_compress_adjoint(const float2 *g, const float *win, int n_az, int L, int centred,
                                           float2 *grad_raw, cudaStream_t s, int n_scans) {
    if (n_scans < 1 || n_scans > 65535)
        return set_error(ROSAR_ERR_UNSUPPORTED, "range_compress_adjoint: n_scans=%d not in [1, 65535]", n_scans);
    switch (L) {
        case 8: return launch_adjoint_L<8>(g, win, n_az, centred, grad_raw, s, n_scans);
        case 16: return launch_adjoint_L<16>(g, win, n_az, centred, grad_raw, s, n_scans);
        case 32: return launch_adjoint_L<32>(g, win, n_az, centred, grad_raw, s, n_scans);
        case 64: return launch_adjoint_L<64>(g, win, n_az, centred, grad_raw, s, n_scans);
        case 128: return launch_adjoint_L<128>(g, win, n_az, centred, grad_raw, s, n_scans);
        case 256: return launch_adjoint_L<256>(g, win, n_az, centred, grad_raw, s, n_scans);
        case 512: return launch_adjoint_L<512>(g, win, n_az, centred, grad_raw, s, n_scans);
        case 1024: return launch_adjoint_L<1024>(g, win, n_az, centred, grad_raw, s, n_scans);
        case 2048: return launch_adjoint_L<2048>(g, win, n_az, centred, grad_raw, s, n_scans);
        case 4096: return launch_adjoint_L<4096>(g, win, n_az, centred, grad_raw, s, n_scans);
        default:
            return set_error(ROSAR_ERR_UNSUPPORTED, "range_compress_adjoint: L=%d is not a power of two in [8, 4096]", L);
    }
}

}  // namespace rosar
