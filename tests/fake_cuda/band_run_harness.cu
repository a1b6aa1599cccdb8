// Runs the host side of band_run.cu on the fake CUDA runtime's devices: 0 and 1 take
// every launch that has been allowed its shared memory there, 2 and 3 take none, 4 has
// fewer SMs (the shape then has fewer blocks).
#include <cstdio>

#include "lbm_launch.h"

extern int fake_device, fake_launches;

int main() {
    int bad = 0;
    for (int dev = 0; dev < 5; ++dev) {
        fake_device = dev;
        const int sms = dev == 4 ? 100 : 152;
        const lbm::BandRun b = lbm::band_run_shape(256, 256, sms);
        lbm::KParams<float> p{};
        p.nx = p.ny = 256;
        std::printf("device %d: %d blocks", dev, b.ctas);
        if (b.ctas) {
            for (int scheme = 0; scheme < 3; ++scheme) {
                p.raw = scheme == 1;
                p.forced = scheme == 2;
                const cudaError_t e = lbm::launch_band_run(nullptr, nullptr, p, 0, 3, b, nullptr);
                std::printf(" launch %d", (int)e);
                bad += e != cudaSuccess;
            }
            bad += (dev == 2 || dev == 3) || b.ctas > sms;
        } else {
            bad += dev < 2 || dev == 4;
        }
        std::printf("\n");
    }
    std::printf("%s, %d launches\n", bad ? "failed" : "ok", fake_launches);
    return bad != 0;
}
