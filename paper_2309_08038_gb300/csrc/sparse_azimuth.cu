// K2: sparse-aperture azimuth matched filter (arXiv 2309.08038, Sec. III-D, Eq. (43); Algorithm 2).
//
//   out[r][theta] = sum_{k<K} w[r][k] * S[r][(theta + o_k) mod n_az]
//
// Grid: (azimuth tiles of 256 J outputs, range rows, scans); each CTA runs one
// gather-MAC tile (azimuth_tile.cuh): the row's circular window staged in shared
// memory, J outputs per thread, taps broadcast from shared memory.  The same
// kernel with conjugated weights and negated offsets is the adjoint in S.
//
// Bound by shared memory: an 8-byte read for every product, and a tap's weight and offset once for a thread's J.  A
// tile's lanes past the row's end read and multiply for nothing, and a grid of a few CTAs an SM ends with its fullest
// SM: J is chosen for the row length and the number of rows.

#include "azimuth_tile.cuh"

namespace rosar {
namespace {

constexpr int SA_J = 4;      // migrating taps

// CTAs an SM that the registers are held to.  At J = 4 none is asked for: five (48 registers for 40) lose 5 to 13 % at up to
// 16 taps (7200 x 1024, K = 8: 42 -> 47 us) and up to 7 % with offsets over the whole ring; but MANY taps after range
// compression's tail gain (image of 3607 x 256, K = 128: 45.9 -> 41.8).
template <int J, bool MANY>
constexpr int gather_min_blocks() { return J <= 3 ? 8 : MANY ? 5 : 0; }

// blockIdx = (azimuth tile, range row, scan); scans are stacked [n_scans][n_rng][n_az] and share w, o.  A launch that
// overlaps nothing reads S by the non-coherent path and without the wait: 7200 x 1024 with 1 to 16 taps is 8 to 15 %
// slower otherwise.
template <bool ADJ, int J, bool OVERLAP, bool MANY>
__global__ void __launch_bounds__(az::THREADS, (gather_min_blocks<J, MANY>()))
sparse_azimuth_kernel(const float2 *__restrict__ S, const float2 *__restrict__ w, const int32_t *__restrict__ o,
                      int o_row_stride, int n_rng, int n_az, int K, float2 *__restrict__ out) {
    extern __shared__ __align__(16) char sm[];
    __shared__ int red[4 * az::THREADS / 32];
    const size_t scan = (size_t)blockIdx.z * n_rng * n_az;
    az::azimuth_tile<J, OVERLAP ? az::kOverlapped : az::kEnded, ADJ>(S + scan, w, o, o_row_stride, n_az, K, out + scan,
                                                                     blockIdx.y, blockIdx.x * az::Geo<J>::TW, sm, red);
}

// Time of a launch of J outputs a thread over `rows` rows of n_az: about l + s * (CTAs of the fullest SM) us at 64 taps (the
// order of the J is the same at 4 to 128).
struct GatherCost { int J; double l, s; };
constexpr GatherCost kGather[] = {{4, 3.5, 2.72}, {1, 3.3, 1.07}, {2, 3.7, 1.57}, {3, 4.4, 2.12}};
long long gather_ctas(int n_az, long long rows, int J) {
    return rows * ((n_az - 1) / (az::THREADS * J) + 1);
}

// Four outputs a thread unless another J is better by an eighth, since offsets spread over more than a window read S
// through L2 and gain less.  Five and six outputs are up to 1.4 times slower there and are not taken.  Measured against
// J = 4 for every row, 2890 sizes with offsets over a sixth and the whole of the ring: 1.13 times as fast on average, 0.90
// at the least (four taps, wide); 541 x 1024, K = 64: 20.8 -> 17.7 us; 1031 x 512, K = 48: 18.2 -> 15.
const GatherCost &gather_cost(int n_az, long long rows) {
    const GatherCost *best = kGather;
    double least = 1e30;
    for (const GatherCost &c : kGather) {
        const double t = c.l + c.s * (double)((gather_ctas(n_az, rows, c.J) + 151) / 152);
        if (t < least) {
            least = c.J == 4 ? 0.88 * t : t;
            best = &c;
        }
    }
    return *best;
}

// Whether to launch over the tail of range compression.  CTAs that all fit beside it settle where it leaves room first
// and stay there: between one and five an SM, the fullest SM gets one more than its share (2047 x 256, K = 128: 27.1
// us one after the other, 33.7 overlapped), which costs more than the microsecond gained unless a CTA is shorter.
bool gather_overlaps(int n_az, long long rows, int K) {
    const GatherCost &c = gather_cost(n_az, rows);
    const long long ctas = gather_ctas(n_az, rows, c.J);
    return ctas <= 152 || ctas > 5 * 152 || c.s * K <= 64.0;
}

template <bool ADJ, int J, bool OVERLAP, bool MANY = false>
rosar_status launch_gather_j(const float2 *S, const float2 *w, const int32_t *o, int o_row_stride, int n_scans,
                             int n_rng, int n_az, int K, float2 *out, cudaStream_t s) {
    static int done[kMaxDevices] = {};
    constexpr int smem = az::Geo<J>::SMEM_BYTES;
    rosar_status st = ensure_smem((const void *)sparse_azimuth_kernel<ADJ, J, OVERLAP, MANY>, smem, done, "sparse_azimuth");
    if (st != ROSAR_OK) return st;
    const dim3 grid((n_az + az::Geo<J>::TW - 1) / az::Geo<J>::TW, n_rng, n_scans);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(az::THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = OVERLAP ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, sparse_azimuth_kernel<ADJ, J, OVERLAP, MANY>, S, w, o, o_row_stride, n_rng,
                                             n_az, K, out);
    if (e != cudaSuccess) return set_error(ROSAR_ERR_CUDA, "sparse_azimuth: launch failed: %s", cudaGetErrorString(e));
    return check_launch(ADJ ? "sparse_azimuth_adjoint" : "sparse_azimuth");
}

template <bool ADJ, bool OVERLAP = false>
rosar_status launch_gather(const float2 *S, const float2 *w, const int32_t *o, int o_row_stride, int n_scans,
                           int n_rng, int n_az, int K, float2 *out, cudaStream_t s) {
    if (n_rng > 65535 || n_scans > 65535)
        return set_error(ROSAR_ERR_UNSUPPORTED, "sparse_azimuth: n_rng=%d or n_scans=%d exceeds 65535", n_rng, n_scans);
    switch (gather_cost(n_az, (long long)n_rng * n_scans).J) {
        case 1: return launch_gather_j<ADJ, 1, OVERLAP>(S, w, o, o_row_stride, n_scans, n_rng, n_az, K, out, s);
        case 2: return launch_gather_j<ADJ, 2, OVERLAP>(S, w, o, o_row_stride, n_scans, n_rng, n_az, K, out, s);
        case 3: return launch_gather_j<ADJ, 3, OVERLAP>(S, w, o, o_row_stride, n_scans, n_rng, n_az, K, out, s);
        default: break;
    }
    if constexpr (OVERLAP)
        if (K >= 48)
            return launch_gather_j<ADJ, 4, OVERLAP, true>(S, w, o, o_row_stride, n_scans, n_rng, n_az, K, out, s);
    return launch_gather_j<ADJ, 4, OVERLAP>(S, w, o, o_row_stride, n_scans, n_rng, n_az, K, out, s);
}

using MigGeo = az::GeoMig<SA_J>;

__global__ void __launch_bounds__(az::THREADS)
sparse_azimuth_mig_kernel(const float2 *__restrict__ S, int n_bins, const float2 *__restrict__ w,
                          const int32_t *__restrict__ o, int o_row_stride, const int32_t *__restrict__ dl, int n_az,
                          int K, float2 *__restrict__ out) {
    extern __shared__ __align__(16) char sm[];
    __shared__ int red[4 * az::THREADS / 32];
    az::azimuth_tile<SA_J, az::kEnded, false, true>(S, w, o, o_row_stride, n_az, K, out, blockIdx.y,
                                               blockIdx.x * MigGeo::TW, sm, red, dl, n_bins);
}

}  // namespace

rosar_status launch_sparse_azimuth_migrating(const float2 *S, int n_bins, const float2 *w, const int32_t *o,
                                             int o_row_stride, const int32_t *dl, int n_rng, int n_az, int K,
                                             float2 *out, cudaStream_t s) {
    static int done[kMaxDevices] = {};
    rosar_status st = ensure_smem((const void *)sparse_azimuth_mig_kernel, MigGeo::SMEM_BYTES, done,
                                  "sparse_azimuth_migrating");
    if (st != ROSAR_OK) return st;
    if (n_rng > 65535) return set_error(ROSAR_ERR_UNSUPPORTED, "sparse_azimuth_migrating: n_rng=%d exceeds 65535", n_rng);
    dim3 grid((n_az + MigGeo::TW - 1) / MigGeo::TW, n_rng);
    sparse_azimuth_mig_kernel<<<grid, az::THREADS, MigGeo::SMEM_BYTES, s>>>(S, n_bins, w, o, o_row_stride, dl, n_az,
                                                                           K, out);
    return check_launch("sparse_azimuth_migrating");
}

rosar_status launch_sparse_azimuth(const float2 *S, const float2 *w, const int32_t *o, int o_row_stride, int n_rng,
                                   int n_az, int K, float2 *out, cudaStream_t s, bool overlap_predecessor) {
    return overlap_predecessor && gather_overlaps(n_az, n_rng, K)
               ? launch_gather<false, true>(S, w, o, o_row_stride, 1, n_rng, n_az, K, out, s)
               : launch_gather<false>(S, w, o, o_row_stride, 1, n_rng, n_az, K, out, s);
}

rosar_status launch_sparse_azimuth_scans(const float2 *S, const float2 *w, const int32_t *o, int o_row_stride,
                                         int n_scans, int n_rng, int n_az, int K, bool adjoint, float2 *out,
                                         cudaStream_t s) {
    return adjoint ? launch_gather<true>(S, w, o, o_row_stride, n_scans, n_rng, n_az, K, out, s)
                   : launch_gather<false>(S, w, o, o_row_stride, n_scans, n_rng, n_az, K, out, s);
}

}  // namespace rosar
