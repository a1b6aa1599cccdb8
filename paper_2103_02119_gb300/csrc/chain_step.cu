// chain_step.cu -- two fused steps of a large FP32 lattice (the work is in
// chain_step.cuh): launch and launch shape.
#include "chain_step.cuh"

namespace lbm {

namespace {

constexpr int kSteps = 2;
constexpr int kValid = kStrip - 4 * kSteps;  // columns of a strip that are stored
static_assert(kValid == kChainColumns);

template <int SCH, bool MASK>
cudaError_t launch_chain_mask(const float* fin, float* fout, const KParams<float>& p,
                              int nbands, cudaStream_t s) {
    constexpr size_t smem = chain_smem_bytes<kSteps>();
    static bool configured = false;
    if (!configured) {
        cudaError_t e = cudaFuncSetAttribute(chain_kernel<SCH, MASK, kSteps>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    const dim3 grid((p.nx + kValid - 1) / kValid, nbands);
    chain_kernel<SCH, MASK, kSteps><<<grid, 32 * kSteps, smem, s>>>(fin, fout, p, nbands);
    return cudaGetLastError();
}

template <int SCH>
cudaError_t launch_chain_scheme(const float* fin, float* fout, const KParams<float>& p,
                                int nbands, cudaStream_t s) {
    return p.lmask ? launch_chain_mask<SCH, true>(fin, fout, p, nbands, s)
                   : launch_chain_mask<SCH, false>(fin, fout, p, nbands, s);
}

}  // namespace

cudaError_t launch_chain2(const float* fin, float* fout, const KParams<float>& p,
                          int nbands, cudaStream_t s) {
    return p.raw      ? launch_chain_scheme<1>(fin, fout, p, nbands, s)
           : p.forced ? launch_chain_scheme<0>(fin, fout, p, nbands, s)
                      : launch_chain_scheme<3>(fin, fout, p, nbands, s);
}

int chain2_bands(int nx, int ny, int pitch, int sms) {
    if (!chain2_takes(nx, ny, pitch)) return 0;
    const double strips = (nx + kValid - 1) / kValid;
    int best = 0;
    double cost = 0.0;
    for (int nb = 1; nb <= ny / 8 && nb <= 4096; ++nb) {
        const double rows = (ny + nb - 1) / nb + 10;  // rows that a chain takes for a band
        const double per_sm = strips * nb / sms, waves = per_sm / 8;
        // clocks a row: 1310 of a chain alone on an SM, 2800 of eight
        const double clocks = 1100.0 + 212.0 * (per_sm < 1 ? 1 : per_sm < 8 ? per_sm : 8);
        const double c = rows * clocks * (waves <= 1 ? 1.18 : waves + 0.25);
        if (best == 0 || c < cost) {
            best = nb;
            cost = c;
        }
    }
    return best;
}

}  // namespace lbm
