// kernels_f64.cu -- double instances of the libmc kernels and their launchers.
// Built with -fmad=false: no multiply-add contraction, so every FP64
// expression is evaluated as one IEEE operation at a time, left to right.
#include "kernels.h"
#include "pass_impl.cuh"

namespace mcgb {
namespace {

using R = double;
constexpr int MINB = 1;  // minimum resident blocks per SM of the colour pass
constexpr int V = kSitesPerThreadF64;
constexpr int kPairChunk = 4;   // consecutive pair tiles per grid-stride step of the pair pass
constexpr int kFieldChunk = 4;  // the same for the neighbour-field kernel

#include "launchers_common.cuh"

template <int C>
void pair_pass_t(const GroupArgs& g, uint32_t ntiles, const R* cone, int colour, int sub, uint32_t cap,
                 cudaStream_t s) {
    const Spread sp = spread_warps((ntiles + C - 1) / C, cap);
    launch_chained_if(chain_small(sp, cap), pair_pass_kernel<R, 1, C, false>, sp.blocks, sp.threads, s, g, ntiles, cone, colour, sub);
}

// launch shapes: at most {default, 8, 2} tiles per grid-stride step; FP64
// lattices always take pair order (LatParams::pair_leader)
void pair_pass(const GroupArgs& g, uint32_t ntiles, const void* cone, int colour, int leader, int shape, int sub,
               cudaStream_t s) {
    (void)leader;
    static const uint32_t cap = resident_blocks(pair_pass_kernel<R, 1, kPairChunk, false>);
    const R* c64 = static_cast<const R*>(cone);
    const int c = tiles_per_step(ntiles, cap * (kBlock / 32), shape == 1 ? 8 : shape == 2 ? 2 : kPairChunk);
    if (c == 8) pair_pass_t<8>(g, ntiles, c64, colour, sub, cap, s);
    else if (c == 4) pair_pass_t<4>(g, ntiles, c64, colour, sub, cap, s);
    else if (c == 2) pair_pass_t<2>(g, ntiles, c64, colour, sub, cap, s);
    else pair_pass_t<1>(g, ntiles, c64, colour, sub, cap, s);
}

}  // namespace

const KernelSet& kernels_f64() {
    static const KernelSet k{colour_pass, nullptr,     pair_pass,   sweep_end,         pair_field,
                             ml_reset,    mlong,       measure,     nullptr,           grain_sample,
                             profile,     init_spins,  sample_close, nullptr, "f64",
                             nullptr,     nullptr,     nullptr,           nullptr,      nullptr,
                             nullptr,     nullptr,     nullptr};
    return k;
}

}  // namespace mcgb
