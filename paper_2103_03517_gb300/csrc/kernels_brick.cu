// kernels_brick.cu -- the brick sweeps of brick_pass.cuh: planner and launches.
#include <algorithm>
#include <cstddef>
#include <vector>

#include "kernels.h"
#include "brick_pass.cuh"

namespace mcgb {
namespace {

template <int LAW, int FACES, int ODD, int MEASURE, int GROUP>
cudaError_t launch(const BrickArgs& a, const BrickGroup& g, uint32_t blocks, uint32_t smem, const float* cone,
                   cudaStream_t s) {
    if ((GROUP ? g.n_sweeps : a.n_sweeps) < a.refuse) return cudaErrorInvalidValue;
    if (smem + kResStaticSmem > 48u * 1024u) {  // what any kernel may take
        const cudaError_t opt = opt_in_smem(brick_sweep_kernel<LAW, FACES, ODD, MEASURE, GROUP>);
        if (opt != cudaSuccess) return opt;
    }
    // cooperative: the launch fails rather than run with a block not resident
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(kBrickThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, brick_sweep_kernel<LAW, FACES, ODD, MEASURE, GROUP>, a, g, cone);
}

template <int LAW, int FACES, int ODD, int GROUP = 0>
cudaError_t launch_m(const BrickArgs& a, const BrickGroup& g, uint32_t blocks, uint32_t smem, const float* cone,
                     int measure, cudaStream_t s) {
    if (measure >= 2) return launch<LAW, FACES, ODD, 2, GROUP>(a, g, blocks, smem, cone, s);
    if (measure == 1) return launch<LAW, FACES, ODD, 1, GROUP>(a, g, blocks, smem, cone, s);
    return launch<LAW, FACES, ODD, 0, GROUP>(a, g, blocks, smem, cone, s);
}

cudaError_t launch_any(const BrickArgs& a, uint32_t Lh, const float* cone, int measure, cudaStream_t s) {
    const BrickGroup g{};
    const uint32_t b = a.nyc * a.nzc;
    if (a.law == 0)
        return a.faces ? launch_m<0, 1, 0>(a, g, b, a.smem, cone, measure, s)
                       : launch_m<0, 0, 0>(a, g, b, a.smem, cone, measure, s);
    if (Lh & 1u)
        return a.faces ? launch_m<1, 1, 1>(a, g, b, a.smem, cone, measure, s)
                       : launch_m<1, 0, 1>(a, g, b, a.smem, cone, measure, s);
    return a.faces ? launch_m<1, 1, 0>(a, g, b, a.smem, cone, measure, s)
                   : launch_m<1, 0, 0>(a, g, b, a.smem, cone, measure, s);
}

// What comes before a launch: brick_prep_kernel on lattice `one`, or on `many`;
// n measured sweeps.
cudaError_t prep(const BrickArgs& one, const BrickArgs* many, int lattices, int n, cudaStream_t s) {
    brick_prep_kernel<256><<<dim3(uint32_t(n * kRecordWords / 256 + 1), uint32_t(lattices)), 256, 0, s>>>(one, many, n);
    return cudaGetLastError();
}

struct Device {
    uint32_t most, cap;  // blocks at once, shared memory of a block
};

Device device() {
    int dev = 0, sms = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return Device{uint32_t(std::min(sms, kBrickMaxBlocks)), uint32_t(std::max(0, optin - int(kResStaticSmem)))};
}

// A split and its estimated us a pass, fitted to 8^3 ... 96^3 at 1 ... 152
// blocks: the exchange and up to two tiles a scheduler 1.45 (one block 1.15),
// 0.105 a tile beyond; among equals fewer rounds, face rows and blocks.
struct Split {
    uint32_t nyc = 0, nzc = 0, rows = 0, smem = 0;
    double cost = 0;
};

// The best split of lattice p over exactly G blocks or fewer, for G = 1 ...
// most (nyc = 0: none fits).
std::vector<Split> splits(const LatParams& p, const Device& d) {
    const uint32_t Lh = uint32_t(p.Lh), Ly = uint32_t(p.Ly), Lz = uint32_t(p.Lz);
    std::vector<Split> best(d.most + 1);
    auto consider = [&](uint32_t nyc, uint32_t nzc, uint32_t rows, uint32_t halo) {
        const uint32_t smem = brick_smem_bytes(rows, Lh), G = nyc * nzc;
        if (smem > d.cap) return;
        const uint32_t tiles = ((rows * Lh + 1) / 2 + 31) / 32, rounds = (tiles + kBrickWarps - 1) / kBrickWarps;
        const double cost = std::max(G > 1 ? 1.45 : 1.15, 0.3 + 0.105 * tiles) + 0.1 * rounds + 1e-3 * double(halo) +
                            1e-3 * G;
        if (best[G].nyc == 0 || cost < best[G].cost) best[G] = Split{nyc, nzc, rows, smem, cost};
    };
    if (Lh & 1u) {
        const uint32_t pairs = (Ly * Lz + 1) / 2;
        for (uint32_t G = 1; G <= d.most && G <= pairs; ++G) consider(G, 1, 2 * ((pairs + G - 1) / G), 0);
    } else {
        for (uint32_t nyc = 1; nyc <= Ly && nyc <= d.most; ++nyc)
            for (uint32_t nzc = 1; nzc <= Lz && nyc * nzc <= d.most; ++nzc) {
                const uint32_t by = (Ly + nyc - 1) / nyc, bz = (Lz + nzc - 1) / nzc;
                consider(nyc, nzc, by * bz, (nyc > 1 ? 2 * bz : 0) + (nzc > 1 ? 2 * by : 0));
            }
    }
    for (uint32_t G = 1; G <= d.most; ++G)
        if (best[G - 1].nyc && (best[G].nyc == 0 || best[G - 1].cost <= best[G].cost)) best[G] = best[G - 1];
    return best;
}

void take(const LatParams& p, const Split& b, BrickArgs* out) {
    out->nyc = b.nyc;
    out->nzc = b.nzc;
    out->rows = b.rows;
    out->smem = b.smem;
    out->div_half = make_fastdiv(std::max(1u, uint32_t(p.Lh) / 2));
    out->law = p.colour_kernel == kColourRow || p.colour_kernel == kColourRowFaces ? 0 : 1;
    out->faces = p.bc[0] || p.bc[1] || p.bc[2] ? 1 : 0;
}

}  // namespace

bool brick_plan(const LatParams& p, BrickArgs* out) {
    const std::vector<Split> best = splits(p, device());
    if (best.back().nyc == 0) return false;
    take(p, best.back(), out);
    return true;
}

double brick_group_plan(const std::vector<const LatParams*>& lats, std::vector<BrickArgs>* out) {
    const Device d = device();
    const size_t n = lats.size();
    if (n > d.most) return 0.0;
    std::vector<std::vector<Split>> s;  // of each size once
    std::vector<size_t> kind(n);
    std::vector<const LatParams*> seen;
    std::vector<uint32_t> G(n);
    uint32_t total = 0;
    for (size_t i = 0; i < n; ++i) {
        const LatParams& p = *lats[i];
        for (kind[i] = 0; kind[i] < seen.size(); ++kind[i]) {
            const LatParams& q = *seen[kind[i]];
            if (q.Lh == p.Lh && q.Ly == p.Ly && q.Lz == p.Lz) break;
        }
        if (kind[i] == seen.size()) {
            seen.push_back(&p);
            s.push_back(splits(p, d));
        }
        for (G[i] = 1; G[i] <= d.most && s[kind[i]][G[i]].nyc == 0;) ++G[i];
        if (G[i] > d.most) return 0.0;
        total += G[i];
    }
    if (total > d.most) return 0.0;
    for (;;) {  // more blocks for the slowest, while they make it faster and there are any
        size_t i = 0;
        for (size_t j = 1; j < n; ++j)
            if (s[kind[j]][G[j]].cost > s[kind[i]][G[i]].cost) i = j;
        uint32_t g = G[i] + 1;
        while (g <= d.most && s[kind[i]][g].cost >= s[kind[i]][G[i]].cost) ++g;
        if (g > d.most || total + (g - G[i]) > d.most) break;
        total += g - G[i];
        G[i] = g;
    }
    double slowest = 0.0;
    for (size_t i = 0; i < n; ++i) {
        take(*lats[i], s[kind[i]][G[i]], &(*out)[i]);
        slowest = std::max(slowest, s[kind[i]][G[i]].cost);
    }
    return 2.0 * slowest;
}

cudaError_t brick_sweeps(const BrickArgs& b, uint32_t Lh, const void* cone, int n, int measure, bool* ran,
                         cudaStream_t s) {
    BrickArgs a = b;
    a.n_sweeps = n;
    cudaError_t e = prep(a, nullptr, 1, measure ? n : 0, s);
    if (e == cudaSuccess) e = launch_any(a, Lh, static_cast<const float*>(cone), measure, s);
    *ran = e == cudaSuccess;
    if (*ran && measure) {
        e = brick_close(a, static_cast<const BrickArgs*>(nullptr), 1, n, s);
    }
    return e;
}

cudaError_t brick_group_sweeps(const BrickClass& c, const void* cone, int n, int measure, bool* ran, cudaStream_t s) {
    const float* c32 = static_cast<const float*>(cone);
    const BrickGroup g{c.args, c.first, c.n, n};
    BrickArgs none{};
    none.refuse = c.refuse;
    cudaError_t e = prep(none, c.args, c.n, measure ? n : 0, s);
    if (e == cudaSuccess)
        e = c.law == 0 ? launch_m<0, 0, 0, 1>(none, g, c.blocks, c.smem, c32, measure, s)
            : c.odd    ? launch_m<1, 0, 1, 1>(none, g, c.blocks, c.smem, c32, measure, s)
                       : launch_m<1, 0, 0, 1>(none, g, c.blocks, c.smem, c32, measure, s);
    *ran = e == cudaSuccess;
    if (*ran && measure) {
        e = brick_close(none, static_cast<const BrickArgs*>(c.args), c.n, n, s);
    }
    return e;
}

}  // namespace mcgb
