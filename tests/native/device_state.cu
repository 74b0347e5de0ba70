// device_state.cu -- every launcher on four devices of a stand-in for the CUDA runtime
// (fake_cudart.cpp; no GPU).
#include <cstdio>

#include "batch_internal.h"
#include "fake_cudart.h"
#include "mlp_internal.h"

using namespace gals;

namespace {

int failures = 0;

void expect(bool ok, const char *what)
{
    if (ok) return;
    ++failures;
    std::printf("device %d: %s\n", fake_device, what);
}

// every launcher once on the current device
void all_launchers()
{
    Geom g{};
    g.n0 = g.n1 = 64; g.n2 = 64; g.pitch = 64; g.plane = 64 * 64 * 64;
    VelParams vp{};
    static CUtensorMap map;
    static float data[8];
    static int err;
    static StageCoef coef;
    const int before = fake_refused;

    SmallLaunch sl{};
    sl.in = data; sl.out = data; sl.geom = g; sl.vp = vp; sl.coef = &coef; sl.dt = 0.1; sl.nsteps = 8;
    sl.vp.kind = VK_VORTEX2D; sl.trace = TR_RK3; sl.write_cross = sl.planes = 1;
    bool done = false;
    fake_cluster = 0;
    const cudaError_t e = launch_step2d_small(sl, nullptr, &done);
    expect(e == cudaSuccess, "small-grid run failed");
    expect(done == (fake_placeable[fake_device] > 0), "small-grid run: wrong report of whether it was queued");
    expect(fake_cluster == fake_placeable[fake_device], "small-grid run: not the cluster that the device can place");

    StepLaunch a{};
    a.in = data; a.out = data; a.geom = g; a.vp = vp; a.coef = &coef; a.dt = 0.1; a.err = &err; a.trace = TR_RK3;
    for (auto &row : a.tmap) for (auto &m : row) m = &map;
    a.tmap_cross = &map;
    a.vp.kind = VK_VORTEX2D;
    for (int n1 : {64, 100000})  // short and tall tiles
        for (int wc = 0; wc < 2; ++wc)
            for (int ci : {CROSS_PLANE, CROSS_RECON}) {
                a.geom.n1 = n1;
                a.write_cross = wc;
                a.cross_in = ci;
                expect(launch_step2d(a, nullptr) == cudaSuccess, "2D step failed");
            }
    a.geom = g;
    a.vp.kind = VK_DEFORM3D;
    for (int ci : {CROSS_PLANE, CROSS_RECON, CROSS_CELL}) {
        a.cross_in = ci;
        a.write_cross = ci == CROSS_PLANE;
        expect(launch_step3d(a, nullptr) == cudaSuccess, "3D step failed");
    }

    BatchLaunch b{};
    b.nitems = 4;
    for (int variant = 0; variant < 2; ++variant)
        for (int kind : {VK_FOURIER2D, VK_VORTEX2D})
            for (int ci : {CROSS_PLANE, CROSS_RECON})
                for (int wc = 0; wc < 2; ++wc) {
                    b.variant = variant; b.kind = kind; b.cross_in = ci; b.write_cross = wc;
                    expect(launch_batch2d(b, nullptr) == cudaSuccess, "batched step failed");
                }
    BatchRunLaunch br{};
    br.nitems = 4; br.nprob = 1; br.nsteps = 2; br.variant = 1; br.kind = VK_FOURIER2D;
    expect(launch_batch2d_run(br, nullptr) == cudaSuccess, "batched run failed");

    mlp::InferParams ip{};
    expect(mlp::infer_points(ip, data, data, 4, &err, nullptr) == cudaSuccess, "network failed");
    mlp::Check chk{};
    for (int kind : {VK_FOURIER2D, VK_WAVES2D}) {
        vp.kind = kind;
        expect(mlp::launch_mlp_trace(ip, g, vp, &coef, nullptr, 0, 0.1, data, chk, nullptr) == cudaSuccess,
               "learned trace failed");
    }
    expect(mlp::launch_train_tiles(data, nullptr, data, data, 128, data, data, nullptr, &err, nullptr) == cudaSuccess,
           "training step failed");
    expect(fake_refused == before, "a launch was refused");
}

}  // namespace

int main()
{
    for (int round = 0; round < 2; ++round)
        for (fake_device = 0; fake_device < 4; ++fake_device) all_launchers();
    std::printf("%d launches, %d refused, %d failures\n", fake_launches, fake_refused, failures);
    return failures || fake_refused || fake_launches == 0;
}
