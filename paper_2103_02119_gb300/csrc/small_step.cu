// small_step.cu -- many steps of one small lattice in one launch of one
// thread-block cluster (the work is in small_step.cuh).
#include "small_step.cuh"

#include <algorithm>

namespace lbm {

namespace {

template <typename T>
__global__ void __launch_bounds__(kSmallMaxThreads<T>)
small_run_kernel(T* f0, T* f1, const uint8_t* __restrict__ bits,
                 const __grid_constant__ KParams<T> p, int from, int nsteps) {
    extern __shared__ __align__(16) unsigned char smem[];
    small_run<T>(p, f0, f1, bits, p.nx, from, nsteps, smem, (int)blockIdx.x, (int)gridDim.x);
}

int small_cluster_size(int ny) { return ny < kSmallCluster ? ny : kSmallCluster; }

template <typename T>
cudaLaunchConfig_t small_config(const KParams<T>& p, cudaStream_t s, cudaLaunchAttribute* attr) {
    const int C = small_cluster_size(p.ny);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C, 1, 1);
    cfg.blockDim = dim3(small_threads<T>(p.nx, p.ny, C), 1, 1);
    cfg.dynamicSmemBytes = small_smem_bytes<T>(p.nx, p.ny, C);
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// Allows the kernel its clusters and shared memory on the current device (of the
// largest CTA: one row of 1365 FP64 cells, 3 x 1365 cells on three CTAs).
template <typename T>
cudaError_t configure_small() {
    cudaError_t e = cudaFuncSetAttribute(small_run_kernel<T>,
                                         cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(small_run_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kSmallSmemMax);
}

}  // namespace

// CTAs per lattice of a batch: as many (1, 2, 4, 8) as shared memory asks for,
// and more while the batch makes at most two CTAs per SM and the tallest lattice has
// two rows for each.  Us a step with a
// target of one / two / four CTAs per SM (and of the band kernel, one launch a
// step): 64 lattices of 16-32 cells a side 1.89 / 1.83 / 1.94 (11.0), 32 of 60-64
// 2.80 / 2.64 / 2.64 (11.9), 128 of 16-64 4.34 / 4.35 / 6.55 (24.5).
SmallBatch small_batch_shape(const int* nx, const int* ny, int n, int sms) {
    SmallBatch best;
    // (a CTA past a lattice's last row has none and only joins the barriers)
    const int tallest = n ? *std::max_element(ny, ny + n) : 0;
    for (int C = 1; C <= 8; C *= 2) {
        SmallBatch b;
        b.cluster = C;
        for (int k = 0; k < n; ++k) {
            const size_t m = small_smem_bytes<float>(nx[k], ny[k], C);
            const int t = small_threads<float>(nx[k], ny[k], C);
            if (m > b.smem) b.smem = m;
            if (t > b.threads) b.threads = t;
        }
        if (b.smem > (size_t)kSmallSmemMax) continue;
        if (best.cluster && ((long long)n * C > 2LL * sms || 2 * C > tallest)) break;
        best = b;
    }
    best.queues = (long long)n * best.cluster > sms && 2 * best.smem > (size_t)kSmallSmemMax;
    return best;
}

template <typename T>
cudaError_t launch_small_run(T* f0, T* f1, const uint8_t* bits, const KParams<T>& p, int from,
                             int nsteps, cudaStream_t s) {
    if (nsteps <= 0) return cudaSuccess;
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = small_config<T>(p, s, attr);
    return cudaLaunchKernelEx(&cfg, small_run_kernel<T>, f0, f1, bits, p, from, nsteps);
}

template <typename T>
bool small_run_fits(const KParams<T>& p) {
    if (configure_small<T>() != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = small_config<T>(p, nullptr, attr);
    if (cfg.dynamicSmemBytes > (size_t)kSmallSmemMax) return false;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, small_run_kernel<T>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return n >= 1;
}
template bool small_run_fits<float>(const KParams<float>&);
template bool small_run_fits<double>(const KParams<double>&);

template cudaError_t launch_small_run<float>(float*, float*, const uint8_t*, const KParams<float>&,
                                             int, int, cudaStream_t);
template cudaError_t launch_small_run<double>(double*, double*, const uint8_t*,
                                              const KParams<double>&, int, int, cudaStream_t);

}  // namespace lbm
