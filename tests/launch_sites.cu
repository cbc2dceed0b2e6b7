// Calls every launch site that needs function attributes on several devices of
// the stand-in runtime (fake_cudart.cpp) and prints what was refused.
#include <stdio.h>

#include "vefd_internal.cuh"
#include "vefd_nn.h"

extern "C" {
void fake_set_device(int d);
void fake_counts(int* launches, int* refused);
}

using namespace vefd;

int main() {
    alignas(64) CUtensorMap tm{};
    alignas(16) static char mem[4096];
    StepBufs b{};
    int bad = 0;
    auto check = [&](const char* what, int dev, cudaError_t e, cudaError_t want) {
        int n, refused;
        fake_counts(&n, &refused);
        if (e != want || refused || (want == cudaSuccess && n != 1)) {
            printf("%s on device %d: error %d, %d launches, %d refused\n", what, dev, (int)e, n, refused);
            ++bad;
        }
    };
    const int order[] = {0, 1, 0, 2, 1};
    for (int dev : order) {
        fake_set_device(dev);
        for (int prec = 0; prec < 3; ++prec)
            for (int ncomp = 1; ncomp <= 2; ++ncomp)
                for (int fd = 0; fd < 2; ++fd) {
                    StepParams p{};
                    p.prec = prec, p.nx = 64, p.ny = 32, p.nz = 1, p.N = 2048, p.yhi = 32;
                    for (p.collision = 0; p.collision < 2; ++p.collision)
                        check("launch_small", dev, launch_small(ncomp, fd, p, b, 8, nullptr),
                              dev == 2 ? cudaErrorNotSupported : cudaSuccess);
                    p.nz = 16, p.N *= 16, p.collision = 0;
                    Parts parts{};
                    check("launch_post_zm", dev, launch_post_zm(ncomp, fd, p, b, &tm, nullptr, 0, parts), cudaSuccess);
                    parts.part = reinterpret_cast<float*>(mem), parts.by = 4, parts.bz = 2;
                    check("launch_post_zm parts", dev, launch_post_zm(ncomp, fd, p, b, &tm, nullptr, 0, parts), cudaSuccess);
                    check("launch_post_zm_fused", dev, launch_post_zm_fused(ncomp, fd, p, b, nullptr, 4, 0), cudaSuccess);
                    check("launch_post_batch", dev,
                          launch_post_batch(ncomp, prec, fd, nullptr, nullptr, 1, 8, 0, true, nullptr), cudaSuccess);
                    for (int tile = 0; tile < 6; ++tile)
                        check("launch_lattice", dev, launch_lattice(1, ncomp, true, p, b, nullptr, &tm, 0, tile, Parts{}),
                              cudaSuccess);
                    for (p.collision = 0; p.collision < 2; ++p.collision)
                        check("launch_lattice_zm", dev, launch_lattice_zm(ncomp, p, b, nullptr, &tm, 4, 0), cudaSuccess);
                }
        for (int n : {16, 64, 128, 256}) {
            const int r = vefd_nn_gemm_bf16(mem, 64, mem, 64, reinterpret_cast<float*>(mem), n, 128, n, 64, 0,
                                            reinterpret_cast<unsigned*>(mem), nullptr);
            check("vefd_nn_gemm_bf16", dev, r == VEFD_NN_OK ? cudaSuccess : cudaErrorUnknown, cudaSuccess);
        }
        int conv_launches = 0, refused = 0;
        for (int cin : {8, 48}) {
            vefd_nn_conv3d_forward(reinterpret_cast<float*>(mem), 1, 8, 8, 8, cin, 1, mem, nullptr, 16, 0, mem,
                                   reinterpret_cast<float*>(mem), nullptr, reinterpret_cast<unsigned*>(mem), nullptr);
            vefd_nn_conv3d_backward(mem, reinterpret_cast<float*>(mem), reinterpret_cast<float*>(mem), 1, 8, 8, 8, cin, 1, mem, 16,
                                    0, reinterpret_cast<float*>(mem), reinterpret_cast<float*>(mem),
                                    reinterpret_cast<float*>(mem), 0, reinterpret_cast<float*>(mem),
                                    reinterpret_cast<unsigned*>(mem), nullptr);
        }
        fake_counts(&conv_launches, &refused);
        if (refused || conv_launches < 8) {
            printf("convolutions on device %d: %d launches, %d refused\n", dev, conv_launches, refused);
            ++bad;
        }
    }
    printf(bad ? "%d wrong\n" : "ok\n", bad);
    return bad != 0;
}
