// band_run.cu -- many steps of a middle-sized FP32 lattice in one cooperative
// launch (the work is in band_run.cuh): shape and launch.
#include "band_run.cuh"

namespace lbm {

namespace {

constexpr int kBandSmemMax = kSmallSmemMax - 1024;  // (the kernel has a word of its own)

size_t band_smem(int nx, int ny, int C) {
    const int R = (ny + C - 1) / C, P = small_row<float>(nx);
    return band_cells(R, P) + 16 + (size_t)kSmallTable * 4 * R * (P / 2) + (size_t)(R + 2) * P;
}

// Whether the current device takes `ctas` such CTAs at once.  Allows the kernel
// its shared memory on this device as well: the setting belongs to the device, so it
// is made with every lattice, not once for the process.
template <int SCH>
bool band_fits(int ctas, int threads, size_t smem, int sms) {
    int n = 0;
    if (cudaFuncSetAttribute(band_run_kernel<SCH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kBandSmemMax) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, band_run_kernel<SCH>, threads, smem) !=
            cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return (long long)n * sms >= ctas;
}

template <int SCH>
cudaError_t launch_band(float* f0, float* f1, const KParams<float>& p, int from, int nsteps,
                        const BandRun& b, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(b.flags, 0, (size_t)b.ctas * 32 * sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(b.ctas, 1, 1);
    cfg.blockDim = dim3(b.threads, 1, 1);
    cfg.dynamicSmemBytes = band_smem(p.nx, p.ny, b.ctas);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, band_run_kernel<SCH>, f0, f1, p, from, nsteps, b.mail, b.flags);
}

}  // namespace

BandRun band_run_shape(int nx, int ny, int sms) {
    BandRun b;
    const int C = ny / 2 < sms ? ny / 2 : sms;  // at least two rows each
    if (nx < 4 || C < 1 || band_smem(nx, ny, C) > (size_t)kBandSmemMax) return b;
    const int R = (ny + C - 1) / C, G = (nx + 1) / 2;
    if ((long long)(R + 2) * G >= 65536 || 2LL * kMailRows * G >= 65536) return b;
    const int n = ((R + 2) * G + 31) / 32 * 32;
    const int threads = n < 64 ? 64 : n < kBandThreads ? n : kBandThreads;
    const size_t smem = band_smem(nx, ny, C);
    if (!(band_fits<0>(C, threads, smem, sms) && band_fits<1>(C, threads, smem, sms) &&
          band_fits<3>(C, threads, smem, sms)))
        return b;
    b.ctas = C;
    b.threads = threads;
    b.mail_bytes = (size_t)C * 4 * kMailRows * small_row<float>(nx) * sizeof(float);
    return b;
}

cudaError_t launch_band_run(float* f0, float* f1, const KParams<float>& p, int from, int nsteps,
                            const BandRun& b, cudaStream_t s) {
    return p.raw      ? launch_band<1>(f0, f1, p, from, nsteps, b, s)
           : p.forced ? launch_band<0>(f0, f1, p, from, nsteps, b, s)
                      : launch_band<3>(f0, f1, p, from, nsteps, b, s);
}

}  // namespace lbm
