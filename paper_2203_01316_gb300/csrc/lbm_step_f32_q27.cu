// Kernel instantiations for FP32 storage, D3Q27 h.
#define LBM_KERNEL_TU
#include "lbm_kernels.cuh"

namespace lbmd {
template cudaError_t launch_step<float, 27>(const Buffers&, const DevParams&, cudaStream_t, bool, cudaStream_t);
template cudaError_t launch_objective<float, 27>(const Buffers&, const DevParams&, AdjObjective, double*, double*,
                                              cudaStream_t);
template cudaError_t launch_init<float, 27>(const Buffers&, const DevParams&, const double*, const double*,
                                         const double*, cudaStream_t);
template cudaError_t launch_macros<float, 27>(const Buffers&, const DevParams&, double*, double*, double*,
                                           cudaStream_t);
template cudaError_t launch_populations<float, 27>(const Buffers&, const DevParams&, double*, double*, cudaStream_t);
template cudaError_t launch_record_h<float, 27>(const Buffers&, const DevParams&, void*, cudaStream_t);
template cudaError_t launch_mirror<float, 27>(const Buffers&, const DevParams&, cudaStream_t);
template cudaError_t launch_inlet<float, 27>(const Buffers&, const DevParams&, cudaStream_t, bool);
template cudaError_t launch_balances<float, 27>(const Buffers&, const DevParams&, double*, double*, cudaStream_t);
template cudaError_t launch_surface_flux<float, 27>(const Buffers&, const DevParams&, int, double*, double*,
                                                 cudaStream_t);
template cudaError_t launch_wall_force<float, 27>(const Buffers&, const DevParams&, int, double*, double*,
                                               cudaStream_t);

// streaming map of the step kernels (storage independent)
__global__ void k_stream_map(const uint8_t* __restrict__ flags, const int32_t* __restrict__ wnode,
                             const uint32_t* __restrict__ wmask, int nw, int32_t* __restrict__ src,
                             const DevParams p) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= p.N) return;
    const size_t N = (size_t)p.N;
    const int type = flags[n] & 3;
    if (type == T_SOLID || type == T_INLET) {
        for (int a = 0; a < 27; ++a) src[a * N + n] = -2;
        return;
    }
    uint32_t mask = 0;
    if (flags[n] & F_WALL) {
        int lo = 0, hi = nw - 1;
        while (lo <= hi) {
            const int mid = (lo + hi) >> 1;
            const int v = wnode[mid];
            if (v == n) { mask = wmask[mid]; break; }
            if (v < n) lo = mid + 1; else hi = mid - 1;
        }
    }
    int x, y, z;
    node_xyz(n, p, x, y, z);
    const Nbr nb = make_nbr(x, y, z, p);
#pragma unroll
    for (int a = 0; a < 27; ++a) src[a * N + n] = (mask & (1u << OPP(a))) ? -1 : src_of(nb, a);
}

cudaError_t launch_stream_map(const Buffers& b, const DevParams& p, int qh, int32_t* src, cudaStream_t s) {
    (void)qh;
    const int grid = (p.N + kBlock - 1) / kBlock;
    k_stream_map<<<grid, kBlock, 0, s>>>(b.flags, b.wnode, b.wmask, b.nw, src, p);
    return cudaGetLastError();
}

__global__ void __launch_bounds__(kRedThreads) k_reduce3(const double* __restrict__ acc, int n, int parts,
                                                         double* __restrict__ part, const RedOut o) {
    __shared__ double sh[32 * 3];
    double v[3] = {0.0, 0.0, 0.0};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
#pragma unroll
        for (int k = 0; k < 3; ++k)
            for (int j = 0; j < parts; ++j) v[k] += acc[((size_t)i * 3 + k) * parts + j];
    if (reduce_in_last_block<3>(v, sh, part, red_counter(part))) write_totals<3>(v, o);
}

cudaError_t launch_reduce3(const double* acc, int n, int parts, double* out, double* scratch, cudaStream_t s) {
    const int grid = std::min((n + kRedThreads - 1) / kRedThreads, kRedBlocks);
    k_reduce3<<<grid, kRedThreads, 0, s>>>(acc, n, parts, scratch, RedOut{out, nullptr, 0.0, 0});
    return cudaGetLastError();
}

// per-wall sums of the links' accumulators: blockIdx.y is the wall, a block
// takes a stripe of the links (in a fixed order, so the sums are reproducible).
// Copying the accumulators to pageable host memory and adding them there took
// 0.3 ms per call at 147k links (every gradient calls it twice).
__global__ void __launch_bounds__(kRedThreads) k_wall_sums(const double* __restrict__ dlink,
                                                           const int32_t* __restrict__ lwall, int64_t nl,
                                                           double* __restrict__ part) {
    __shared__ double sh[32];
    double v[1] = {0.0};
    for (int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; l < nl; l += (int64_t)gridDim.x * blockDim.x)
        if (lwall[l] == (int)blockIdx.y) v[0] += dlink[l];
    block_sum<1>(v, sh);
    if (threadIdx.x == 0) part[blockIdx.y * gridDim.x + blockIdx.x] = v[0];
}
__global__ void k_wall_sums_total(const double* __restrict__ part, int nb, double* __restrict__ out) {
    __shared__ double sh[32];
    double v[1] = {(int)threadIdx.x < nb ? part[blockIdx.x * nb + threadIdx.x] : 0.0};
    block_sum<1>(v, sh);
    if (threadIdx.x == 0) out[blockIdx.x] = v[0];
}
static_assert(kWallSumBlocks <= 64, "one thread per partial sum");

cudaError_t launch_wall_sums(const double* dlink, const int32_t* lwall, int64_t nl, int n_walls, double* part,
                             double* out, cudaStream_t s) {
    const int nb = (int)std::min<int64_t>((nl + kRedThreads - 1) / kRedThreads, kWallSumBlocks);
    k_wall_sums<<<dim3(nb, n_walls), kRedThreads, 0, s>>>(dlink, lwall, nl, part);
    k_wall_sums_total<<<n_walls, 64, 0, s>>>(part, nb, out);
    return cudaGetLastError();
}
}  // namespace lbmd
