// kernels_brick.cu -- the brick sweeps of brick_pass.cuh: planner and launches.
#include <algorithm>
#include <cstddef>

#include "kernels.h"
#include "brick_pass.cuh"

namespace mcgb {
namespace {

template <int LAW, int FACES, int ODD, int MEASURE>
cudaError_t launch(const BrickArgs& a, const float* cone, cudaStream_t s) {
    static const bool ok = [] {
        int dev = 0, optin = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        return cudaFuncSetAttribute(brick_sweep_kernel<LAW, FACES, ODD, MEASURE>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    optin - int(kResStaticSmem)) == cudaSuccess;
    }();
    if (!ok) return cudaErrorInvalidConfiguration;
    // cooperative: the launch fails rather than run with a block not resident
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.nyc * a.nzc);
    cfg.blockDim = dim3(kBrickThreads);
    cfg.dynamicSmemBytes = a.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, brick_sweep_kernel<LAW, FACES, ODD, MEASURE>, a, cone);
}

template <int LAW, int FACES, int ODD>
cudaError_t launch_m(const BrickArgs& a, const float* cone, int measure, cudaStream_t s) {
    if (measure >= 2) return launch<LAW, FACES, ODD, 2>(a, cone, s);
    if (measure == 1) return launch<LAW, FACES, ODD, 1>(a, cone, s);
    return launch<LAW, FACES, ODD, 0>(a, cone, s);
}

cudaError_t launch_any(const BrickArgs& a, uint32_t Lh, const float* cone, int measure, cudaStream_t s) {
    if (a.law == 0) return a.faces ? launch_m<0, 1, 0>(a, cone, measure, s) : launch_m<0, 0, 0>(a, cone, measure, s);
    if (Lh & 1u) return a.faces ? launch_m<1, 1, 1>(a, cone, measure, s) : launch_m<1, 0, 1>(a, cone, measure, s);
    return a.faces ? launch_m<1, 1, 0>(a, cone, measure, s) : launch_m<1, 0, 0>(a, cone, measure, s);
}

}  // namespace

bool brick_plan(const LatParams& p, BrickArgs* out) {
    int dev = 0, sms = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const uint32_t cap = uint32_t(std::max(0, optin - int(kResStaticSmem)));
    const uint32_t most = uint32_t(std::min(sms, kBrickMaxBlocks));
    const uint32_t Lh = uint32_t(p.Lh), Ly = uint32_t(p.Ly), Lz = uint32_t(p.Lz);
    const bool odd = Lh & 1u;
    bool found = false;
    double best = 0;
    auto consider = [&](uint32_t nyc, uint32_t nzc, uint32_t rows, uint32_t halo) {
        const uint32_t smem = brick_smem_bytes(rows, Lh), G = nyc * nzc;
        if (smem > cap) return;
        const uint32_t tiles = ((rows * Lh + 1) / 2 + 31) / 32, rounds = (tiles + kBrickWarps - 1) / kBrickWarps;
        // us a pass, fitted to 8^3 ... 96^3 at 1 ... 152 blocks: the exchange
        // and up to two tiles a scheduler 1.45 (one block 1.15), 0.105 a tile
        // beyond; among equals fewer rounds, face rows and blocks
        const double cost = std::max(G > 1 ? 1.45 : 1.15, 0.3 + 0.105 * tiles) + 0.1 * rounds + 1e-3 * double(halo) +
                            1e-3 * G;
        if (found && cost >= best) return;
        found = true;
        best = cost;
        out->nyc = nyc;
        out->nzc = nzc;
        out->rows = rows;
        out->smem = smem;
    };
    if (odd) {
        const uint32_t pairs = (Ly * Lz + 1) / 2;
        for (uint32_t G = 1; G <= most && G <= pairs; ++G) consider(G, 1, 2 * ((pairs + G - 1) / G), 0);
    } else {
        for (uint32_t nyc = 1; nyc <= Ly && nyc <= most; ++nyc)
            for (uint32_t nzc = 1; nzc <= Lz && nyc * nzc <= most; ++nzc) {
                const uint32_t by = (Ly + nyc - 1) / nyc, bz = (Lz + nzc - 1) / nzc;
                consider(nyc, nzc, by * bz, (nyc > 1 ? 2 * bz : 0) + (nzc > 1 ? 2 * by : 0));
            }
    }
    if (!found) return false;
    out->div_half = make_fastdiv(std::max(1u, Lh / 2));
    out->law = p.colour_kernel == kColourRow || p.colour_kernel == kColourRowFaces ? 0 : 1;
    out->faces = p.bc[0] || p.bc[1] || p.bc[2] ? 1 : 0;
    return true;
}

cudaError_t brick_sweeps(const BrickArgs& b, uint32_t Lh, const void* cone, int n, int measure, cudaStream_t s) {
    for (int done = 0; done < n;) {
        BrickArgs a = b;
        a.n_sweeps = std::min(n - done, measure ? kBrickMaxMeasured : kResMaxSweeps);
        cudaError_t e = cudaMemsetAsync(a.ctl, 0, offsetof(BrickCtl, epoch), s);
        if (e == cudaSuccess && measure)
            e = cudaMemsetAsync(a.record, 0, size_t(a.n_sweeps) * kRecordWords * sizeof(long long), s);
        if (e == cudaSuccess) e = launch_any(a, Lh, static_cast<const float*>(cone), measure, s);
        if (e == cudaSuccess && measure) {
            brick_close_kernel<4><<<(a.n_sweeps + 3) / 4, 128, 0, s>>>(a.lat, a.ctl, a.record, a.n_sweeps);
            e = cudaGetLastError();
        }
        if (e != cudaSuccess) return e;
        done += a.n_sweeps;
    }
    return cudaSuccess;
}

}  // namespace mcgb
