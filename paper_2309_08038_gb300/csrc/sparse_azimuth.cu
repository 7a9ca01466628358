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

// CTAs an SM that the registers are held to.  Left to the compiler, 40 to 47 a thread: 7200 x 1024, K = 16 (J = 6)
// 69 -> 62 us; 3600 x 256, K = 64 (J = 4) 23.5 -> 21.8 with five, 22.8 with six.
template <int J>
constexpr int gather_min_blocks() { return J <= 3 ? 8 : J == 5 ? 6 : 5; }

// blockIdx = (azimuth tile, range row, scan); scans are stacked [n_scans][n_rng][n_az] and share w, o.
template <bool ADJ, int J>
__global__ void __launch_bounds__(az::THREADS, gather_min_blocks<J>())
sparse_azimuth_kernel(const float2 *__restrict__ S, const float2 *__restrict__ w, const int32_t *__restrict__ o,
                      int o_row_stride, int n_rng, int n_az, int K, float2 *__restrict__ out) {
    extern __shared__ __align__(16) char sm[];
    __shared__ int red[4 * az::THREADS / 32];
    const size_t scan = (size_t)blockIdx.z * n_rng * n_az;
    az::azimuth_tile<J, false, ADJ>(S + scan, w, o, o_row_stride, n_az, K, out + scan, blockIdx.y,
                                    blockIdx.x * az::Geo<J>::TW, sm, red);
}

// Outputs per thread for `rows` rows of n_az: the least (CTAs of the fullest SM) J (measured time of one product at J
// against J = 4: fewer or more products share a tap's weight and offset).  Against J = 4 for every row: 360 x 256, K =
// 64 (J = 2) 7.8 -> 5.8 us; 1031 x 512, K = 48 (5) 18.2 -> 13.0; 541 x 1024, K = 64 (3) 20.8 -> 17.7; 7196 x 512,
// K = 128 (6) 139.8 -> 125.8; J = 8 is never less than J = 4 by this count.
int outputs_per_thread(int n_az, long long rows) {
    static const struct { int J; double rate; } js[] = {{1, 1.50}, {2, 1.15}, {3, 1.05}, {4, 1.00},
                                                        {5, 0.99}, {6, 0.94}};
    int best = 4;
    double least = 1e30;
    for (const auto &c : js) {
        const long long tiles = (n_az + az::THREADS * c.J - 1) / (az::THREADS * c.J);
        const double cost = (double)((tiles * rows + 151) / 152) * c.J * c.rate;
        if (cost < least) {
            least = cost;
            best = c.J;
        }
    }
    return best;
}

template <bool ADJ, int J>
rosar_status launch_gather_j(const float2 *S, const float2 *w, const int32_t *o, int o_row_stride, int n_scans,
                             int n_rng, int n_az, int K, float2 *out, cudaStream_t s, bool overlap) {
    static int done[kMaxDevices] = {};
    constexpr int smem = az::Geo<J>::SMEM_BYTES;
    rosar_status st = ensure_smem((const void *)sparse_azimuth_kernel<ADJ, J>, smem, done, "sparse_azimuth");
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
    cfg.numAttrs = overlap ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, sparse_azimuth_kernel<ADJ, J>, S, w, o, o_row_stride, n_rng, n_az, K, out);
    if (e != cudaSuccess) return set_error(ROSAR_ERR_CUDA, "sparse_azimuth: launch failed: %s", cudaGetErrorString(e));
    return check_launch(ADJ ? "sparse_azimuth_adjoint" : "sparse_azimuth");
}

template <bool ADJ>
rosar_status launch_gather(const float2 *S, const float2 *w, const int32_t *o, int o_row_stride, int n_scans,
                           int n_rng, int n_az, int K, float2 *out, cudaStream_t s, bool overlap = false) {
    if (n_rng > 65535 || n_scans > 65535)
        return set_error(ROSAR_ERR_UNSUPPORTED, "sparse_azimuth: n_rng=%d or n_scans=%d exceeds 65535", n_rng, n_scans);
    switch (outputs_per_thread(n_az, (long long)n_rng * n_scans)) {
        case 1: return launch_gather_j<ADJ, 1>(S, w, o, o_row_stride, n_scans, n_rng, n_az, K, out, s, overlap);
        case 2: return launch_gather_j<ADJ, 2>(S, w, o, o_row_stride, n_scans, n_rng, n_az, K, out, s, overlap);
        case 3: return launch_gather_j<ADJ, 3>(S, w, o, o_row_stride, n_scans, n_rng, n_az, K, out, s, overlap);
        case 4: return launch_gather_j<ADJ, 4>(S, w, o, o_row_stride, n_scans, n_rng, n_az, K, out, s, overlap);
        case 5: return launch_gather_j<ADJ, 5>(S, w, o, o_row_stride, n_scans, n_rng, n_az, K, out, s, overlap);
        default: return launch_gather_j<ADJ, 6>(S, w, o, o_row_stride, n_scans, n_rng, n_az, K, out, s, overlap);
    }
}

using MigGeo = az::GeoMig<SA_J>;

__global__ void __launch_bounds__(az::THREADS)
sparse_azimuth_mig_kernel(const float2 *__restrict__ S, int n_bins, const float2 *__restrict__ w,
                          const int32_t *__restrict__ o, int o_row_stride, const int32_t *__restrict__ dl, int n_az,
                          int K, float2 *__restrict__ out) {
    extern __shared__ __align__(16) char sm[];
    __shared__ int red[4 * az::THREADS / 32];
    az::azimuth_tile<SA_J, false, false, true>(S, w, o, o_row_stride, n_az, K, out, blockIdx.y,
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
    return launch_gather<false>(S, w, o, o_row_stride, 1, n_rng, n_az, K, out, s, overlap_predecessor);
}

rosar_status launch_sparse_azimuth_scans(const float2 *S, const float2 *w, const int32_t *o, int o_row_stride,
                                         int n_scans, int n_rng, int n_az, int K, bool adjoint, float2 *out,
                                         cudaStream_t s) {
    return adjoint ? launch_gather<true>(S, w, o, o_row_stride, n_scans, n_rng, n_az, K, out, s)
                   : launch_gather<false>(S, w, o, o_row_stride, n_scans, n_rng, n_az, K, out, s);
}

}  // namespace rosar
